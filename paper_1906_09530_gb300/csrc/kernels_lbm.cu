// kernels_lbm.cu -- lattice kernels of the FP64 path: collide-stream (Eqs. 1, 2, 5),
// equilibrium initialisation, output velocity and diagnostics.
//
// Populations are structure-of-arrays, f[i*plane + y*nx + x], i in the velocity
// order of Sec. 2.
#include <cfloat>
#include <climits>

#include "cplbm_internal.cuh"
#include "fp64_math.cuh"
#include "lattice.cuh"

namespace cplbm {
namespace {

// Second-order equilibrium of Eq. 2 with c_s^2 = 1/3:
//   f_i^eq = w_i rho (1 + 3 e.u + 9/2 (e.u)^2 - 3/2 u.u).
__device__ __forceinline__ double feq(int i, double rho, double ux, double uy, double uu) {
    const double w = i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
    const double eu = q_ex(i) * ux + q_ey(i) * uy;
    return w * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu);
}

__device__ __forceinline__ void raise_flag(DevState* st, unsigned bits, int64_t t) {
    atomicOr(&st->flag, bits);
    atomicMin(&st->failed_t, (unsigned long long)t);
}

// In-place BGK collision with exact-difference forcing (Eqs. 1, 2, 5), with j = rho u,
// m = j + F, keep = 1 - 1/tau, g = m - keep j and P = (m m - keep j j)/rho:
//   f_i* = keep f_i + w_i [omega rho + 3 e.g + 9/2 (e e : P) - 3/2 tr P],
// in moments, so that the velocity is never formed and opposite directions share all but
// the sign of one term: 60 FP64 instructions.  (Pair by pair in u and v it is 84.)
__device__ __forceinline__ void collide_bgk(double (&f)[9], double rho, double Fx, double Fy,
                                            double omega) {
    const double keep = rn_sub(1.0, omega);
    const double d57 = rn_sub(f[5], f[7]), d68 = rn_sub(f[6], f[8]);
    const double jx = rn_add(rn_sub(f[1], f[3]), rn_sub(d57, d68));
    const double jy = rn_add(rn_sub(f[2], f[4]), rn_add(d57, d68));
    const double inv = rcp64(rho);
    const double mx = rn_add(jx, Fx), my = rn_add(jy, Fy);
    const double kx = rn_mul(keep, jx), ky = rn_mul(keep, jy);
    double pxx, pyy, pxy;
    if (__double2hiint(rho) >= (1023 - 400) << 20) {  // 2^-400, without an FP64 comparison
        pxx = rn_mul(rn_fma(mx, mx, -rn_mul(kx, jx)), inv);
        pyy = rn_mul(rn_fma(my, my, -rn_mul(ky, jy)), inv);
        pxy = rn_mul(rn_fma(mx, my, -rn_mul(kx, jy)), inv);
    } else {  // m m would underflow
        const double vx = rn_mul(mx, inv), vy = rn_mul(my, inv);
        const double ux = rn_mul(kx, inv), uy = rn_mul(ky, inv);
        pxx = rn_fma(mx, vx, -rn_mul(ux, jx));
        pyy = rn_fma(my, vy, -rn_mul(uy, jy));
        pxy = rn_fma(mx, vy, -rn_mul(ux, jy));
    }
    const double s = rn_add(pxx, pyy);
    const double e1 = rn_mul(rn_fma(-1.5, s, rn_mul(omega, rho)), 1.0 / 9.0);
    f[0] = rn_fma(keep, f[0], rn_mul(4.0, e1));
    const double bx = rn_mul(rn_sub(mx, kx), 1.0 / 3.0), by = rn_mul(rn_sub(my, ky), 1.0 / 3.0);
    auto pair = [&](int i, int j, double even, double c, double odd) {
        f[i] = rn_fma(c, odd, rn_fma(keep, f[i], even));
        f[j] = rn_fma(-c, odd, rn_fma(keep, f[j], even));
    };
    pair(1, 3, rn_fma(0.5, pxx, e1), 1.0, bx);
    pair(2, 4, rn_fma(0.5, pyy, e1), 1.0, by);
    const double e2 = rn_fma(0.125, s, rn_mul(0.25, e1));
    pair(5, 7, rn_fma(0.25, pxy, e2), 0.25, rn_add(bx, by));
    pair(6, 8, rn_fma(-0.25, pxy, e2), 0.25, rn_sub(by, bx));
}

// ---------------------------------------------------------------------------
// Pass 1, FP64: collide a node and push its populations to its neighbours.  A thread
// per node; each plane is written by a warp as one row piece shifted by e_i.  What bounds
// it is the FP64 pipe, so no node is collided twice: a tile pulling from a collided halo
// (32 x 16 nodes, 1.2 collisions a node) took 251 us at 1024^2, this takes 123.  The new
// density is summed by the pass that needs it first (the x-lines).
// ---------------------------------------------------------------------------
constexpr int kCsT = 128;

template <bool MRT, bool WALLS>
__global__ void __launch_bounds__(kCsT)
    k_collide_stream(const double* __restrict__ fin, double* __restrict__ fout,
                     const double* __restrict__ Fx, const double* __restrict__ Fy,
                     const double* __restrict__ rho, int nx, int ny, size_t plane, double omega,
                     double se, double seps, double sq, double uwb6, double uwt6,
                     DevState* __restrict__ st) {
    const long long n = blockIdx.x * (long long)kCsT + threadIdx.x;
    if (n >= (long long)nx * ny) return;
    const int y = (int)(n / nx), x = (int)(n - (long long)y * nx);
    double f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = fin[i * plane + n];
    const double r = rho[n];
    bool ok = positive64(r);
    if constexpr (MRT)
        ok &= collide_mrt<double>(f, Fx[n], Fy[n], omega, (double)FLT_MAX, se, seps, sq);
    else
        collide_bgk(f, r, Fx[n], Fy[n], omega);
    const int xs[3] = {x > 0 ? x - 1 : nx - 1, x, x + 1 < nx ? x + 1 : 0};
    const int ys[3] = {y > 0 ? y - 1 : ny - 1, y, y + 1 < ny ? y + 1 : 0};
    // the node's density, for the momentum a moving wall gives
    const bool bottom = WALLS && y == 0, top = WALLS && y == ny - 1;
    double rw = 0.0;
    if (WALLS && (bottom || top)) {
#pragma unroll
        for (int i = 0; i < 9; ++i) rw += f[i];
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        // halfway bounce-back at walls: the node keeps the population, reversed, plus
        // e_x rho U / 6 on the diagonals from a wall moving at U (Ladd)
        if (WALLS && ((q_ey(i) < 0 && bottom) || (q_ey(i) > 0 && top)))
            fout[q_opp(i) * plane + n] =
                f[i] - (double)q_ex(i) * rw * (q_ey(i) < 0 ? uwb6 : uwt6);
        else
            fout[i * plane + (size_t)ys[q_ey(i) + 1] * nx + xs[q_ex(i) + 1]] = f[i];
    }
    if (!ok) raise_flag(st, FLAG_RHO, st->t);
}

// f_i = f_i^eq(rho, u) (Eq. 2).
__global__ void k_init_feq(const double* __restrict__ rho, const double* __restrict__ ux,
                           const double* __restrict__ uy, double* __restrict__ f, size_t N,
                           size_t plane) {
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N;
         n += (size_t)gridDim.x * blockDim.x) {
        const double r = rho[n];
        const double u = ux ? ux[n] : 0.0, v = uy ? uy[n] : 0.0;
        const double uu = u * u + v * v;
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i * plane + n] = feq(i, r, u, v, uu);
    }
}

// Output velocity v = u + F/(2 rho) (Sec. 2, after Eq. 5).
__device__ __forceinline__ void node_velocity(const double* __restrict__ f, size_t plane, size_t n,
                                              double rho, double Fx, double Fy, double& vx,
                                              double& vy) {
    double g[9];
#pragma unroll
    for (int i = 1; i < 9; ++i) g[i] = f[i * plane + n];
    const double jx = (g[1] + g[5] + g[8]) - (g[3] + g[6] + g[7]);
    const double jy = (g[2] + g[5] + g[6]) - (g[4] + g[7] + g[8]);
    vx = jx + 0.5 * Fx;
    vy = jy + 0.5 * Fy;
    quotients64(vx, vy, rho);
}

__global__ void k_macro(const double* __restrict__ f, const double* __restrict__ rho,
                        const double* __restrict__ Fx, const double* __restrict__ Fy,
                        double* __restrict__ vx, double* __restrict__ vy, size_t N,
                        size_t plane) {
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N;
         n += (size_t)gridDim.x * blockDim.x) {
        double u, v;
        node_velocity(f, plane, n, rho[n], Fx[n], Fy[n], u, v);
        if (vx) vx[n] = u;
        if (vy) vy[n] = v;
    }
}

// Diagnostics, two deterministic stages: per-block partials, then one block.
constexpr int kDiagThreads = 256;

__global__ void __launch_bounds__(kDiagThreads)
    k_diag_partial(const double* __restrict__ f, const double* __restrict__ rho,
                   const double* __restrict__ Fx, const double* __restrict__ Fy, size_t N,
                   size_t plane, double* __restrict__ partials) {
    double s = 0.0, vmax = 0.0, rmin = DBL_MAX, rmax = -DBL_MAX;
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N;
         n += (size_t)gridDim.x * blockDim.x) {
        double u, v;
        const double rf = rho[n];
        node_velocity(f, plane, n, rf, Fx[n], Fy[n], u, v);
        s += rf;
        vmax = fmax(vmax, u * u + v * v);  // the square: one root a thread
        rmin = fmin(rmin, rf);
        rmax = fmax(rmax, rf);
    }
    __shared__ double sh[4][kDiagThreads];
    sh[0][threadIdx.x] = s;
    sh[1][threadIdx.x] = sqrt(vmax);
    sh[2][threadIdx.x] = rmin;
    sh[3][threadIdx.x] = rmax;
    __syncthreads();
    for (int w = kDiagThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
            sh[1][threadIdx.x] = fmax(sh[1][threadIdx.x], sh[1][threadIdx.x + w]);
            sh[2][threadIdx.x] = fmin(sh[2][threadIdx.x], sh[2][threadIdx.x + w]);
            sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        for (int q = 0; q < 4; ++q) partials[4 * blockIdx.x + q] = sh[q][0];
    }
}

__global__ void __launch_bounds__(kDiagThreads)
    k_diag_final(const double* __restrict__ partials, int nparts, DevState* __restrict__ st) {
    double s = 0.0, vmax = 0.0, rmin = DBL_MAX, rmax = -DBL_MAX;
    for (int b = threadIdx.x; b < nparts; b += blockDim.x) {
        s += partials[4 * b];
        vmax = fmax(vmax, partials[4 * b + 1]);
        rmin = fmin(rmin, partials[4 * b + 2]);
        rmax = fmax(rmax, partials[4 * b + 3]);
    }
    __shared__ double sh[4][kDiagThreads];
    sh[0][threadIdx.x] = s;
    sh[1][threadIdx.x] = vmax;
    sh[2][threadIdx.x] = rmin;
    sh[3][threadIdx.x] = rmax;
    __syncthreads();
    for (int w = kDiagThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
            sh[1][threadIdx.x] = fmax(sh[1][threadIdx.x], sh[1][threadIdx.x + w]);
            sh[2][threadIdx.x] = fmin(sh[2][threadIdx.x], sh[2][threadIdx.x + w]);
            sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        for (int q = 0; q < 4; ++q) st->diag[q] = sh[q][0];
    }
}

__global__ void k_f_to_double(const float* __restrict__ f, double* __restrict__ out, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        out[i] = widen(f[i]);
}

__global__ void k_f_from_double(const double* __restrict__ in, float* __restrict__ f, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        f[i] = (float)in[i];
}

inline unsigned grid_for(size_t n, int threads) {
    size_t b = (n + threads - 1) / threads;
    return (unsigned)(b < 65535 * 16 ? (b ? b : 1) : 65535 * 16);
}

}  // namespace

cudaError_t launch_collide_stream(const double* fin, double* fout, const double* Fx,
                                  const double* Fy, const double* rho, int nx, int ny,
                                  size_t plane, double omega, const MrtRates* mrt, DevState* st,
                                  cudaStream_t s, const Walls& walls) {
    const unsigned grid = (unsigned)(((long long)nx * ny + kCsT - 1) / kCsT);
    const double se = mrt ? mrt->se : 0.0, seps = mrt ? mrt->seps : 0.0, sq = mrt ? mrt->sq : 0.0;
    auto go = [&](auto kern) {
        kern<<<grid, kCsT, 0, s>>>(fin, fout, Fx, Fy, rho, nx, ny, plane, omega, se, seps, sq,
                                   walls.u[0] / 6.0, walls.u[1] / 6.0, st);
        return cudaGetLastError();
    };
    if (mrt)
        return walls.on ? go(k_collide_stream<true, true>) : go(k_collide_stream<true, false>);
    return walls.on ? go(k_collide_stream<false, true>) : go(k_collide_stream<false, false>);
}

cudaError_t launch_init_feq(const double* rho, const double* ux, const double* uy, double* f,
                            int nx, int ny, size_t plane, cudaStream_t s) {
    const size_t N = (size_t)nx * ny;
    k_init_feq<<<grid_for(N, 256), 256, 0, s>>>(rho, ux, uy, f, N, plane);
    return cudaGetLastError();
}

cudaError_t launch_macro(const double* f, const double* rho, const double* Fx, const double* Fy,
                         double* vx, double* vy, int nx, int ny, size_t plane, cudaStream_t s) {
    const size_t N = (size_t)nx * ny;
    k_macro<<<grid_for(N, 256), 256, 0, s>>>(f, rho, Fx, Fy, vx, vy, N, plane);
    return cudaGetLastError();
}

cudaError_t launch_diag(const double* f, const double* rho, const double* Fx, const double* Fy,
                        int nx, int ny, size_t plane, double* partials, int nparts,
                        DevState* st, cudaStream_t s) {
    const size_t N = (size_t)nx * ny;
    k_diag_partial<<<nparts, kDiagThreads, 0, s>>>(f, rho, Fx, Fy, N, plane, partials);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_diag_final(partials, nparts, st, s);
}

cudaError_t launch_diag_final(const double* partials, int nparts, DevState* st, cudaStream_t s) {
    k_diag_final<<<1, kDiagThreads, 0, s>>>(partials, nparts, st);
    return cudaGetLastError();
}

cudaError_t launch_f_to_double(const float* f, double* out, size_t n, cudaStream_t s) {
    k_f_to_double<<<grid_for(n, 256), 256, 0, s>>>(f, out, n);
    return cudaGetLastError();
}

cudaError_t launch_f_from_double(const double* in, float* f, size_t n, cudaStream_t s) {
    k_f_from_double<<<grid_for(n, 256), 256, 0, s>>>(in, f, n);
    return cudaGetLastError();
}

}  // namespace cplbm
