// lines32.cu -- launches of the FP32 line solves (lines32.cuh): one grid, and batches.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstring>

#include "df.cuh"
#include "eos.cuh"
#include "lines32.cuh"

namespace cplbm {
namespace {

constexpr int kC = kC32, kW = 32 * kC;
constexpr int kMaxT = 512;
constexpr double kEps = 1e-8;  // what the recursions are cut at

double lambda(int order) {
    const double alpha = order == 6 ? 1.0 / 3.0 : 0.25;
    return (1.0 - std::sqrt(1.0 - 4.0 * alpha * alpha)) / (2.0 * alpha);
}

}  // namespace

Line32 line32_constants(int order) {
    const double alpha = order == 6 ? 1.0 / 3.0 : 0.25, lam = lambda(order);
    const double a = 2.0 / 3.0 * (alpha + 2.0), b = (4.0 * alpha - 1.0) / 3.0;  // Eq. 38
    Line32 k;
    k.c1 = (float)(lam / alpha * a / 2.0);
    k.c2 = (float)(lam / alpha * b / 4.0);
    k.nlam = (float)-lam;
    double p = 1.0;
    for (int j = 0; j < kC; ++j) k.pw[j] = (float)(p *= -lam);
    const double m = std::pow(-lam, kC);
    k.m1 = (float)m;
    k.m2 = (float)(m * m);
    k.Cm1 = (float)(kC * m);
    k.Cm2 = (float)(2.0 * kC * m * m);
    return k;
}

// eps1, eps2: what the recursions of the first and second derivative are cut at (eps2 0: no
// second).  Halo: lam^H (single recursion) or (H+1) lam^H (double) below them, rounded up to
// a multiple of 4 so that windows start on 16-byte boundaries.
Geo32 line32_geometry(int nx, int ny, int axis, int order, double eps1, double eps2,
                      bool walls_y) {
    const double lam = lambda(order);
    int h1 = 1, h2 = 0;
    for (double p = lam; p >= eps1; p *= lam) ++h1;
    if (eps2 > 0.0)
        for (double p = 1.0; (h2 + 1) * p >= eps2; p *= lam) ++h2;
    Geo32 g;
    g.n = axis == 0 ? nx : ny;
    g.nlines = axis == 0 ? ny : nx;
    g.ps = axis == 0 ? 1 : nx;
    g.ls = axis == 0 ? nx : 1;
    g.H = (std::max(h1, h2) + 1 + 3) / 4 * 4;
    g.own = kW - 2 * g.H;
    if (g.own > g.n) g.own = g.n;
    g.nwin = (g.n + g.own - 1) / g.own;
    g.vec = nx % 4 == 0;
    g.mirror = axis == 1 && walls_y;
    g.period = g.mirror ? 2 * g.n : g.n;
    g.lift = (g.H + 4 + g.period - 1) / g.period * g.period;
    g.magic = g.period < kW + 8
                  ? (unsigned)(((1ull << 32) + g.period - 1) / (unsigned long long)g.period)
                  : 0u;
    // chunks up to four past the last owned one (a multiple of 4: whole 16-byte pieces)
    const int nch = (g.H + g.own - 1) / kC + 1 + 4;
    g.nch = nch >= 32 ? 32 : (nch + 3) / 4 * 4;
    return g;
}

namespace {

Geo32 geometry(int nx, int ny, int axis, int order, bool second, bool walls_y) {
    return line32_geometry(nx, ny, axis, order, kEps, second ? kEps : 0.0, walls_y);
}

// lines a block of T threads takes; y-lines: a power of two of adjacent columns
void divide(Geo32& g, int axis, int T) {
    g.nl = T / g.nch;
    if (axis == 1) {
        int nl = 1;
        while (2 * nl <= g.nl && nl < 32) nl *= 2;
        g.nl = nl;
    }
    g.ngroups = (g.nlines + g.nl - 1) / g.nl;
}

// Threads a block: 256 (8 full windows or 8 columns, 32-byte row pieces).  Measured steps
// with 64 / 128 / 256 / 512: 512^2 22.5 / 17.7 / 16.0 / 18.2 us, 128^2 12.9 / 11.4 / 11.6 /
// 13.5.  Rows that are not whole 16-byte pieces are staged four bytes at a time, which
// wants more blocks: 333 x 277 18.0 / 17.2 / 18.1 / 21.2.
constexpr int kLoneT = 256;
int pick_threads(int nx) { return nx % 4 == 0 ? kLoneT : 128; }

size_t smem_of(const Geo32& gx, int T, bool second) {
    return ((size_t)6 * T + (size_t)gx.nl * l32::line_stride(gx.nch) * (second ? 2 : 1)) *
           sizeof(float);
}
// the most that a block of up to T threads can need: the shortest windows (8 chunks) stage
// the most lines
size_t most_smem(int T, bool second) {
    size_t most = 0;
    for (int nch = 8; nch <= 32; nch += 4) {
        Geo32 g{};
        g.nl = T / nch;
        g.nch = nch;
        most = std::max(most, smem_of(g, T, second));
    }
    return most;
}
int blocks_of(const Geo32& g) { return g.ngroups * g.nwin; }

template <int MODE, bool SIXTH>
__global__ void __launch_bounds__(kMaxT, 2)
    k_lines32(Dir32 x, Dir32 y, const __grid_constant__ Line32 k, DevState* st,
              int bump, int nbx) {
    pdl_prologue();
    extern __shared__ __align__(16) float sh32[];
    if (bump && blockIdx.x == 0 && threadIdx.x == 0) st->t += 1;
    // y-lines first: their windows take longer
    const int nby = (int)gridDim.x - nbx, b = blockIdx.x;
    if (b < nby)
        l32::block<MODE, SIXTH, 1>(y, k, b, sh32);
    else
        l32::block<MODE, SIXTH, 0>(x, k, b - nby, sh32);
}

// block b belongs to instance map[b]; each instance bumps its own time level
template <int MODE, bool SIXTH>
__global__ void __launch_bounds__(kMaxT, 2)
    k_lines32_batch(const Lines32Inst* __restrict__ d, const int* __restrict__ map,
                    const __grid_constant__ Line32 k, int bump) {
    extern __shared__ __align__(16) float sh32[];
    const Lines32Inst& D = d[map[blockIdx.x]];
    const int local = (int)blockIdx.x - D.blk0;
    if (bump && local == 0 && threadIdx.x == 0) D.st->t += 1;
    if (local < D.nbx)
        l32::block<MODE, SIXTH, 0>(D.x, k, local, sh32);
    else
        l32::block<MODE, SIXTH, 1>(D.y, k, local - D.nbx, sh32);
}

Dir32 density_dir(const float* rh, float* d1, float* d2) {
    Dir32 d{};
    d.u = rh;
    d.o1 = d1;
    d.o2 = d2;
    return d;
}
Dir32 force_dir(const float* mu, const float* rh, const float* dr, float* F) {
    Dir32 d{};
    d.u = mu;
    d.rho = rh;
    d.dr = dr;
    d.o1 = F;
    return d;
}

// geometry of both directions for blocks of T threads (T <= 0: chosen here); returns T
int lay_out(Dir32& x, Dir32& y, int nx, int ny, int order, bool second, bool walls_y, int T) {
    x.g = geometry(nx, ny, 0, order, second, false);
    y.g = geometry(nx, ny, 1, order, second, walls_y);
    if (T <= 0) T = pick_threads(nx);
    divide(x.g, 0, T);
    divide(y.g, 1, T);
    return T;
}

template <int MODE>
cudaError_t run(Dir32 x, Dir32 y, int nx, int ny, int order, bool walls_y, DevState* st, int bump,
                cudaStream_t s) {
    constexpr bool SECOND = MODE == l32::RHO;
    const int T = lay_out(x, y, nx, ny, order, SECOND, walls_y, 0);
    if ((long long)nx * ny > kLines32Nodes)
        return lines32_wide(x, y, nx, ny, order, SECOND, st, bump, s);
    const int nbx = blocks_of(x.g), nby = blocks_of(y.g);
    const size_t smem = smem_of(x.g, T, SECOND);
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, most_smem(kLoneT, SECOND));
        if (e != cudaSuccess) return e;
        return launch_pdl(kern, dim3(nbx + nby), dim3(T), smem, s, x, y, line32_constants(order),
                          st, bump, nbx);
    };
    return order == 6 ? go(k_lines32<MODE, true>) : go(k_lines32<MODE, false>);
}

}  // namespace

cudaError_t lines32_rho(const float* rh, float* dxr, float* dxx, float* dyr, float* dyy, int nx,
                        int ny, int order, DevState* st, int bump, cudaStream_t s, bool walls_y) {
    return run<l32::RHO>(density_dir(rh, dxr, dxx), density_dir(rh, dyr, dyy), nx, ny, order,
                         walls_y, st, bump, s);
}

cudaError_t lines32_force(const float* mu, const float* rh, const float* dxr, const float* dyr,
                          float* Fx, float* Fy, int nx, int ny, int order, DevState* st,
                          cudaStream_t s, bool walls_y) {
    return run<l32::FORCE>(force_dir(mu, rh, dxr, Fx), force_dir(mu, rh, dyr, Fy), nx, ny, order,
                           walls_y, st, 0, s);
}

// ---- batches ----
void lines32_window_use(int nx, int ny, int order, long long& chunks, long long& windows) {
    for (int axis = 0; axis < 2; ++axis) {
        const Geo32 g = geometry(nx, ny, axis, order, true, false);
        windows += (long long)g.nlines * g.nwin;
        chunks += (long long)g.nlines * g.nwin * g.nch;
    }
}

int lines32_batch_blocks(int nx, int ny, int order, bool second, int nl, bool wide) {
    Dir32 x{}, y{};
    lay_out(x, y, nx, ny, order, second, false, 32 * nl);
    if (wide) lines32_wide_divide(x, y, nl);
    return blocks_of(x.g) + blocks_of(y.g);
}

Lines32Inst lines32_batch_inst(const MixedLinesView& v, int order, bool second, int blk0, int nl,
                               bool wide) {
    Lines32Inst d{};
    if (second) {
        d.x = density_dir(v.rh, v.dxr, v.dxx);
        d.y = density_dir(v.rh, v.dyr, v.dyy);
    } else {
        d.x = force_dir(v.dxx, v.rh, v.dxr, v.Fx);
        d.y = force_dir(v.dxx, v.rh, v.dyr, v.Fy);
    }
    lay_out(d.x, d.y, v.nx, v.ny, order, second, false, 32 * nl);
    if (wide) lines32_wide_divide(d.x, d.y, nl);
    d.nbx = blocks_of(d.x.g);
    d.blk0 = blk0;
    d.st = v.st;
    return d;
}

cudaError_t lines32_batch_launch(const Lines32Inst* d, const int* map, int nblocks, int order,
                                 bool second, int bump, int nl, bool wide, cudaStream_t s) {
    if (nblocks <= 0) return cudaSuccess;
    if (wide) return lines32_wide_batch(d, map, nblocks, order, second, bump, nl, s);
    const int T = 32 * nl;
    const size_t smem = most_smem(T, second);  // (of any of the batch's grids)
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, most_smem(kMaxT, second));
        if (e != cudaSuccess) return e;
        kern<<<nblocks, T, smem, s>>>(d, map, line32_constants(order), bump);
        return cudaGetLastError();
    };
    if (second)
        return order == 6 ? go(k_lines32_batch<l32::RHO, true>)
                          : go(k_lines32_batch<l32::RHO, false>);
    return order == 6 ? go(k_lines32_batch<l32::FORCE, true>)
                      : go(k_lines32_batch<l32::FORCE, false>);
}

namespace {
// ---------------------------------------------------------------------------
// Small grids: whole time steps in one launch of one cluster of kCl CTAs.  A step of the
// four passes on a few thousand nodes is four launches of about 3 us each, most of it
// latency; here the passes are separated by the cluster's hardware barrier and a launch
// runs many steps.  Fields stay in global memory (L2): the barrier's release / acquire
// orders them, so nothing here may be read through the non-coherent path (no __restrict__
// const pointers).  An 8 x 400 step 11.7 -> 9.4 us, 32^2 8.5,
// 128 x 64 10.5; 128^2 11.7 -> 12.5, so up to kSmallNodes.
// ---------------------------------------------------------------------------
constexpr int kCl = 16, kSmallT = 256;
struct SmallArgs {
    float* f[2];
    float *Fx, *Fy, *rh, *dxx, *dyy;
    int nx, ny;
    size_t plane;
    float omega, se, seps, sq;
    Dir32 rx, ry, fx, fy;
    int nb_rx, nb_r, nb_fx, nb_f;  // x-line blocks and all blocks of the two line passes
    Line32 k;
    MuConstF mu;
    DevState* st;
    int from, steps;
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

template <bool MRT, bool SIXTH>
__global__ void __launch_bounds__(kSmallT, 1) k_small(const __grid_constant__ SmallArgs a) {
    extern __shared__ __align__(16) float sh32[];
    const int rank = blockIdx.x, t = threadIdx.x;  // the grid is one cluster
    const int nx = a.nx, ny = a.ny;
    const int64_t t0 = a.st->t;
    const int y0 = ny * rank / kCl, y1 = ny * (rank + 1) / kCl;
    const int nn = (y1 - y0) * nx, nh = nn + 2 * nx;  // own nodes, and with a halo row each side
    for (int i = 0; i < a.steps; ++i) {
        const float* fin = a.f[(a.from + i) & 1];
        float* fout = a.f[1 - ((a.from + i) & 1)];
        bool bad_rho = false, bad_mu = false;
        // collide-stream: own rows and the halo rows collided into shared memory, then pulled
        for (int n = t; n < nh; n += kSmallT) {
            const int yl = n / nx, x = n - yl * nx;
            int y = y0 - 1 + yl;
            y += y < 0 ? ny : (y >= ny ? -ny : 0);
            const size_t o = (size_t)y * nx + x;
            float f[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) f[q] = fin[q * a.plane + o];
            const float fx = a.Fx[o], fy = a.Fy[o];
            if constexpr (MRT)
                bad_rho |= !collide_mrt<float>(f, fx, fy, a.omega, FLT_MAX, a.se, a.seps, a.sq);
            else
                bad_rho |= !collide_pairs(f, fx, fy, a.omega, FLT_MAX);
#pragma unroll
            for (int q = 0; q < 9; ++q) sh32[q * nh + n] = f[q];
        }
        __syncthreads();
        for (int n = t; n < nn; n += kSmallT) {
            const int x = n % nx, m = n + nx;  // m: its slot among the halo's rows
            const int xw = x > 0 ? -1 : nx - 1, xe = x + 1 < nx ? 1 : 1 - nx;
            float g[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const int dx = q_ex(q) > 0 ? xw : (q_ex(q) < 0 ? xe : 0);
                g[q] = sh32[q * nh + m - q_ey(q) * nx + dx];
            }
            const size_t o = (size_t)y0 * nx + n;
#pragma unroll
            for (int q = 0; q < 9; ++q) fout[q * a.plane + o] = g[q];
            a.rh[o] = sum9_exact(g).hi;
        }
        cluster_sync();
        for (int b = rank; b < a.nb_r; b += kCl) {
            if (b < a.nb_rx) l32::block<l32::RHO, SIXTH, 0>(a.rx, a.k, b, sh32);
            else l32::block<l32::RHO, SIXTH, 1>(a.ry, a.k, b - a.nb_rx, sh32);
            __syncthreads();
        }
        cluster_sync();
        const bool capped = t0 + i + 1 < a.mu.cap_steps;
        for (int n = t; n < nn; n += kSmallT) {
            const size_t o = (size_t)y0 * nx + n;
            a.dxx[o] = mu_node(a.rh[o], a.dxx[o], a.dyy[o], a.mu, capped, bad_mu);
        }
        cluster_sync();
        for (int b = rank; b < a.nb_f; b += kCl) {
            if (b < a.nb_fx) l32::block<l32::FORCE, SIXTH, 0>(a.fx, a.k, b, sh32);
            else l32::block<l32::FORCE, SIXTH, 1>(a.fy, a.k, b - a.nb_fx, sh32);
            __syncthreads();
        }
        if (bad_rho || bad_mu) {
            atomicOr(&a.st->flag, (bad_rho ? FLAG_RHO : 0u) | (bad_mu ? FLAG_EOS : 0u));
            atomicMin(&a.st->failed_t, (unsigned long long)(t0 + i + (bad_rho ? 0 : 1)));
        }
        cluster_sync();
    }
    if (rank == 0 && t == 0) a.st->t = t0 + a.steps;
}

size_t small_smem(const SmallArgs& a) {
    const size_t tile = (size_t)((a.ny + kCl - 1) / kCl + 2) * a.nx * 9 * sizeof(float);
    const size_t rho = smem_of(a.rx.g, kSmallT, true), force = smem_of(a.fx.g, kSmallT, false);
    return std::max(tile, std::max(rho, force));
}

SmallArgs small_args(const SmallStep& p) {
    SmallArgs a{};
    a.f[0] = p.f[0];
    a.f[1] = p.f[1];
    a.Fx = p.v.Fx;
    a.Fy = p.v.Fy;
    a.rh = const_cast<float*>(p.v.rh);
    a.dxx = p.v.dxx;
    a.dyy = p.v.dyy;
    a.nx = p.v.nx;
    a.ny = p.v.ny;
    a.plane = p.plane;
    a.omega = (float)p.phys.omega;
    if (p.mrt) {
        a.se = (float)p.mrt->se;
        a.seps = (float)p.mrt->seps;
        a.sq = (float)p.mrt->sq;
    }
    a.rx = density_dir(p.v.rh, p.v.dxr, p.v.dxx);
    a.ry = density_dir(p.v.rh, p.v.dyr, p.v.dyy);
    a.fx = force_dir(p.v.dxx, p.v.rh, p.v.dxr, p.v.Fx);
    a.fy = force_dir(p.v.dxx, p.v.rh, p.v.dyr, p.v.Fy);
    lay_out(a.rx, a.ry, a.nx, a.ny, p.order, true, false, kSmallT);
    lay_out(a.fx, a.fy, a.nx, a.ny, p.order, false, false, kSmallT);
    a.nb_rx = blocks_of(a.rx.g);
    a.nb_r = a.nb_rx + blocks_of(a.ry.g);
    a.nb_fx = blocks_of(a.fx.g);
    a.nb_f = a.nb_fx + blocks_of(a.fy.g);
    a.k = line32_constants(p.order);
    a.mu = mu_mixed_const(p.phys);
    a.st = p.v.st;
    return a;
}

template <class F>
cudaError_t with_small_kernel(bool mrt, int order, F f) {
    if (mrt) return order == 6 ? f(k_small<true, true>) : f(k_small<true, false>);
    return order == 6 ? f(k_small<false, true>) : f(k_small<false, false>);
}

cudaLaunchConfig_t small_config(cudaLaunchAttribute* attr, size_t smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kCl);
    cfg.blockDim = dim3(kSmallT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = kCl;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

bool small_steps_fit(const SmallStep& p) {
    if ((long long)p.v.nx * p.v.ny > kSmallNodes) return false;
    const SmallArgs a = small_args(p);
    const size_t smem = small_smem(a);
    // one round of blocks in each line pass (with two, 8 x 500 takes 13.3 us against 11.7 by
    // separate launches), and rows in whole 16-byte pieces unless there are few of them
    // (90 x 45: 12.2)
    if (a.nb_r > kCl || a.nb_f > kCl || smem > 220 * 1024) return false;
    if (!a.rx.g.vec && (long long)a.nx * a.ny > kSmallNodes / 4) return false;
    int clusters = 0;
    const cudaError_t e = with_small_kernel(p.mrt != nullptr, p.order, [&](auto kern) {
        cudaError_t r =
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(220 * 1024));
        if (r != cudaSuccess) return r;
        cudaLaunchAttribute attr[1];
        const cudaLaunchConfig_t cfg = small_config(attr, smem, nullptr);
        return cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
    });
    if (e != cudaSuccess) {
        cudaGetLastError();  // not an error of the caller's
        return false;
    }
    return clusters >= 1;
}

cudaError_t launch_small_steps(const SmallStep& p, int from, int64_t steps, cudaStream_t s) {
    SmallArgs a = small_args(p);
    const size_t smem = small_smem(a);
    while (steps > 0) {
        a.from = from;
        a.steps = (int)(steps < kSmallSteps ? steps : kSmallSteps);
        const cudaError_t e = with_small_kernel(p.mrt != nullptr, p.order, [&](auto kern) {
            cudaLaunchAttribute attr[1];
            const cudaLaunchConfig_t cfg = small_config(attr, smem, s);
            return cudaLaunchKernelEx(&cfg, kern, a);
        });
        if (e != cudaSuccess) return e;
        from = (from + a.steps) & 1;
        steps -= a.steps;
    }
    return cudaSuccess;
}

}  // namespace cplbm
