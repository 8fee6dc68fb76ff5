// kernels_lines.cu -- warp-cooperative compact-FD line solves (Eqs. 37-39) of the mixed
// path, with the fused force (Eq. 12) epilogue.  (The FP64 path's are in lines64.cu.)
//
// The periodic compact scheme is the circulant system A d = B u with
//   (A d)_i = alpha d_{i-1} + d_i + alpha d_{i+1},
//   (B u)_i = a/2 (u_{i+1} - u_{i-1}) + b/4 (u_{i+2} - u_{i-2})   (a, b: Eq. 38).
// A = (alpha/lam)(1 + lam S^-1)(1 + lam S), lam = (1 - sqrt(1 - 4 alpha^2))/(2 alpha),
// so d follows from two first-order recursions on r = (lam/alpha) B u:
//   forward  w_i = r_i - lam w_{i-1},    backward  z_i = w_i - lam z_{i+1},   d = z.
// |lam| < 1 (0.382 at alpha = 1/3, 0.268 at alpha = 1/4), so a value's influence
// decays as lam^distance and each recursion is exact to rounding once started a
// few dozen positions away; positions are taken mod n, so any line length works.
//
// Parallel form.  A block stages a window of W = 32 C consecutive positions of
// NL lines in shared memory (loads and stores coalesced whichever axis the lines
// run along).  Warp w owns line w; lane l owns positions [l C, l C + C).  Each
// lane runs both recursions over its chunk from a zero state, then the chunk
// boundary states are joined by a two-level shuffle scan: the state entering
// chunk l is T_{l-1} with T_l = E_l + m T_{l-1}, m = (-lam)^C (|m| = 1.1e-8 for
// C = 19), and each position adds (-lam)^{j+1} times that carry.  The window
// starts H positions before the first owned position and ends H after the last,
// H chosen so that lam^H (or (H+1) lam^H for the double recursion) is below the
// arithmetic's rounding.  The second derivative D(D u) ("applying CFM twice",
// Sec. 4.3) uses that the circulant operators commute: D D u = F_b F_b F_f F_f B B u,
// a double recursion in each direction whose chunk-joining map is
// (v, w) -> (m v, m (C v + w)).
//
// Arithmetic policies: PolF (FP32), PolDF (double-float pairs).
// The mixed path uses PolDF for the first derivative of the density and PolF for
// everything else (see kernels_mixed.cu for why).
#include <cuda.h>  // CUtensorMap and its encoder's types (the encoder is fetched at run time)

#include <cfloat>
#include <cmath>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "cplbm_internal.cuh"
#include "df.cuh"
#include "eos.cuh"
#include "lattice.cuh"

namespace cplbm {
namespace {

constexpr unsigned kFull = 0xffffffffu;

struct PolF {
    using V = float;
    using K = float;
    using O = float;
    static __device__ __forceinline__ V zero() { return 0.0f; }
    static __device__ __forceinline__ V sub(V a, V b) { return a - b; }
    static __device__ __forceinline__ V mulc(V a, K c) { return a * c; }
    static __device__ __forceinline__ V fmac(V a, K c, V b) { return fmaf(a, c, b); }
    static __device__ __forceinline__ V up(V a, int o) { return __shfl_up_sync(kFull, a, o); }
    static __device__ __forceinline__ V down(V a, int o) { return __shfl_down_sync(kFull, a, o); }
    static __device__ __forceinline__ O out(V a) { return a; }
    static K konst(double v) { return (float)v; }
    using S = float;
    static constexpr int kPlanes = 1;
    static __device__ __forceinline__ V sget(const S* t, int i, int) { return t[i]; }
    static __device__ __forceinline__ void sput(S* t, int i, int, V v) { t[i] = v; }
};

struct PolDF {
    using V = df;
    using K = df;
    using O = float;  // the derivative is rounded once, relative to itself
    static __device__ __forceinline__ V zero() { return df{0.0f, 0.0f}; }
    static __device__ __forceinline__ V sub(V a, V b) { return df_sub(a, b); }
    static __device__ __forceinline__ V mulc(V a, K c) { return df_mul(a, c.hi, c.lo); }
    static __device__ __forceinline__ V fmac(V a, K c, V b) { return df_fma(a, c.hi, c.lo, b); }
    static __device__ __forceinline__ V up(V a, int o) {
        return df{__shfl_up_sync(kFull, a.hi, o), __shfl_up_sync(kFull, a.lo, o)};
    }
    static __device__ __forceinline__ V down(V a, int o) {
        return df{__shfl_down_sync(kFull, a.hi, o), __shfl_down_sync(kFull, a.lo, o)};
    }
    static __device__ __forceinline__ O out(V a) { return df_round(a); }
    static K konst(double v) {
        df r;
        r.hi = (float)v;
        r.lo = (float)(v - (double)r.hi);
        return r;
    }
    // hi and lo in two planes, `ps` floats apart (no bank conflicts for 4-byte words)
    using S = float;
    static constexpr int kPlanes = 2;
    static __device__ __forceinline__ V sget(const S* t, int i, int ps) {
        return df{t[i], t[i + ps]};
    }
    static __device__ __forceinline__ void sput(S* t, int i, int ps, V v) {
        t[i] = v.hi;
        t[i + ps] = v.lo;
    }
};

// value of the second-derivative arithmetic from the first's right-hand side
template <class P2>
__device__ __forceinline__ typename P2::V to2(float v) { return (typename P2::V)v; }
template <class P2>
__device__ __forceinline__ typename P2::V to2(df v) { return (typename P2::V)v.hi; }

constexpr int kC = 19;         // positions per lane (odd: chunk starts hit distinct banks)
constexpr int kW = 32 * kC;    // window length
constexpr int kNL = 8;         // lines (warps) per block
// Shared-memory stride of one line, in the staged input (window + margin 4 on
// each side) and in the outputs, which take over the staged rows once the
// solve has read them (each warp reads and writes only its own line's rows).
// It is 4 mod 32: lanes reading chunk starts (odd stride) and the y-line
// staging/epilogue (8 lines x 4 positions per warp) then touch 32 distinct banks.
constexpr int kLW = 644;
constexpr int kSO = kLW;
static_assert(kLW >= kW + 8 && kLW % 32 == 4, "strides");
static_assert((kW + 8) % 88 == 0, "y-line windows split into whole tensor-copy boxes");

template <class P>
struct LineConst {
    typename P::K c1, c2, nlam;  // (lam/alpha) a/2, (lam/alpha) b/4, -lam
    typename P::K pw[kC];        // (-lam)^(j+1)
    typename P::K m1, m2;        // (-lam)^C, (-lam)^(2C)
    typename P::K Cm1, Cm2;      // C (-lam)^C, 2C (-lam)^(2C)  (double-recursion joins)
};

struct LineGeo {
    int n;          // line length
    int nlines;
    long long ps;   // stride along a line
    long long ls;   // stride between lines
    int H;          // window positions before the first owned one
    int own;        // owned positions per window
    int nwin;       // windows per line
    int ngroups;    // line groups of kNL
    int vec;        // nx % 4 == 0: 16-byte staging (x-lines) and epilogue (float fields)
    int period;     // n (periodic line), or 2 n (y-line between walls, extended evenly)
    int mirror;     // positions n .. 2n-1 of the period read position 2n-1-p
};

// Asynchronous global -> shared copies (cp.async): the staging loads need no
// registers, so a thread's whole share of the window is in flight at once.
__device__ __forceinline__ void cp_async4(void* sdst, const void* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// ---- tensor-memory-access (TMA) staging of y-line windows -------------------
// A y-line window of 8 adjacent columns is 8 floats (32 bytes) of each of kRows
// consecutive rows: one 2-D tensor copy box of 8 x kBoxRows elements per piece,
// kRows / kBoxRows pieces, all issued by one thread and completed on one
// mbarrier.  The wait is bounded: a window that never arrives raises
// FLAG_STAGE and the block gives up instead of spinning forever.
constexpr int kBoxRows = 88;
constexpr unsigned kWaitSpins = 1u << 22;  // ~ tens of milliseconds of polling

__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// bounded wait for phase `parity` of the barrier; false when it gave up
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned parity) {
    for (unsigned i = 0; i < kWaitSpins; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ void tma_load_2d(void* sdst, const CUtensorMap* map, int x, int y,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];\n" ::"r"(smem_u32(sdst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Input fields: stage(t, i, ps, o) copies the element at global offset o into
// staging slot i (planes `ps` apart).
struct InF {
    const float* p;
    __device__ __forceinline__ void init(const DevState*) {}
    __device__ __forceinline__ void stage(float* t, int i, int, size_t o) {
        cp_async4(t + i, p + o);
    }
    // four consecutive elements, 16-byte aligned on both sides
    __device__ __forceinline__ void stage4(float* t, int i, int, size_t o) {
        cp_async16(t + i, p + o);
    }
    __device__ __forceinline__ bool flagged() const { return false; }
};
struct InDF {
    const float* h;
    const float* l;
    __device__ __forceinline__ void init(const DevState*) {}
    __device__ __forceinline__ void stage(float* t, int i, int ps, size_t o) {
        cp_async4(t + i, h + o);
        cp_async4(t + i + ps, l + o);
    }
    __device__ __forceinline__ void stage4(float* t, int i, int ps, size_t o) {
        cp_async16(t + i, h + o);
        cp_async16(t + i + ps, l + o);
    }
    __device__ __forceinline__ bool flagged() const { return false; }
};

__device__ __forceinline__ int wrapi(long long v, int n) {
    long long r = v % n;
    return (int)(r < 0 ? r + n : r);
}

__device__ __forceinline__ void raise_flag(DevState* st, unsigned bits, int64_t t) {
    atomicOr(&st->flag, bits);
    atomicMin(&st->failed_t, (unsigned long long)t);
}

// ---------------------------------------------------------------------------
// The kernel.  AXIS 0: lines along x (rows, stride 1); AXIS 1: lines along y.
// ---------------------------------------------------------------------------
// Reader of the staged window in the arithmetic Q of a solve: the full value,
// or only the hi plane when an FP32 solve runs on a double-float staging.
template <class Q, class P1>
struct Rd {
    static __device__ __forceinline__ typename Q::V get(const typename P1::S* t, int i, int ps) {
        return P1::sget(t, i, ps);
    }
};
template <>
struct Rd<PolF, PolDF> {
    static __device__ __forceinline__ float get(const float* t, int i, int) { return t[i]; }
};

// One window, one warp per line: right-hand sides, chunked recursions joined by
// shuffle scans, results to tout1 (first derivative) and tout2 (second).
template <class Q, class P1, class P2, bool SIXTH, bool SECOND, int NL>
__device__ __forceinline__ void solve_window(const typename P1::S* tin, typename Q::O* tout1,
                                             typename P2::V* tout2, const LineConst<Q>& kq,
                                             const LineConst<P2>& k2) {
    using VQ = typename Q::V;
    using V2 = typename P2::V;
    constexpr int kPS = NL * kLW;
    const int tid = threadIdx.x;
    const int w = tid >> 5, lane = tid & 31;
    const int tb = w * kLW + 4;  // slot of window position 0 of this warp's line
    auto tl = [&](int q) { return Rd<Q, P1>::get(tin, tb + q, kPS); };  // q in [-4, kW+4)
    const int q0 = lane * kC;

    VQ r[kC];  // right-hand side, then forward states, then the result
    {
        VQ u[kC + 4];
#pragma unroll
        for (int k = 0; k < kC + 4; ++k) u[k] = tl(q0 - 2 + k);
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            VQ b = Q::mulc(Q::sub(u[j + 3], u[j + 1]), kq.c1);
            if (SIXTH) b = Q::fmac(Q::sub(u[j + 4], u[j]), kq.c2, b);
            r[j] = b;
        }
    }
    V2 r2[kC];
    if (SECOND) {
        // b1 at positions q0-2 .. q0+kC+1 in the second arithmetic; the two
        // extra on each side are recomputed from the staged field
        V2 bx[kC + 4];
#pragma unroll
        for (int k = 0; k < kC + 4; ++k) {
            if (k >= 2 && k < kC + 2) {
                bx[k] = to2<P2>(r[k - 2]);
            } else {
                const int qc = q0 - 2 + k;  // in [-2, kW+2)
                V2 t = (to2<P2>(tl(qc + 1)) - to2<P2>(tl(qc - 1))) * k2.c1;
                if (SIXTH) t = P2::fmac(to2<P2>(tl(qc + 2)) - to2<P2>(tl(qc - 2)), k2.c2, t);
                bx[k] = t;
            }
        }
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            V2 t = (bx[j + 3] - bx[j + 1]) * k2.c1;
            if (SIXTH) t = P2::fmac(bx[j + 4] - bx[j], k2.c2, t);
            r2[j] = t;
        }
    }

    // forward recursions over the chunk from a zero state
    VQ wv = Q::zero();
#pragma unroll
    for (int j = 0; j < kC; ++j) {
        wv = Q::fmac(wv, kq.nlam, r[j]);
        r[j] = wv;
    }
    V2 vv = 0, ww = 0;
    if (SECOND) {
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            vv = P2::fmac(vv, k2.nlam, r2[j]);
            ww = P2::fmac(ww, k2.nlam, vv);
            r2[j] = ww;
        }
    }
    // join the chunks (forward): state entering this lane's chunk
    {
        VQ T = wv;
        VQ t = Q::up(T, 1);
        if (lane >= 1) T = Q::fmac(t, kq.m1, T);
        t = Q::up(T, 2);
        if (lane >= 2) T = Q::fmac(t, kq.m2, T);
        VQ c = Q::up(T, 1);
        if (lane == 0) c = Q::zero();
#pragma unroll
        for (int j = 0; j < kC; ++j) r[j] = Q::fmac(c, kq.pw[j], r[j]);
    }
    if (SECOND) {
        V2 TV = vv, TW = ww;
        V2 tv = P2::up(TV, 1), tw = P2::up(TW, 1);
        if (lane >= 1) {
            TW = TW + k2.m1 * tw + k2.Cm1 * tv;
            TV = TV + k2.m1 * tv;
        }
        tv = P2::up(TV, 2);
        tw = P2::up(TW, 2);
        if (lane >= 2) {
            TW = TW + k2.m2 * tw + k2.Cm2 * tv;
            TV = TV + k2.m2 * tv;
        }
        V2 cv = P2::up(TV, 1), cw = P2::up(TW, 1);
        if (lane == 0) cv = cw = 0;
#pragma unroll
        for (int j = 0; j < kC; ++j) r2[j] = r2[j] + k2.pw[j] * ((V2)(j + 1) * cv + cw);
    }

    // backward recursions over the chunk from a zero state
    VQ zv = Q::zero();
#pragma unroll
    for (int j = kC - 1; j >= 0; --j) {
        zv = Q::fmac(zv, kq.nlam, r[j]);
        r[j] = zv;
    }
    V2 yv = 0, zz = 0;
    if (SECOND) {
#pragma unroll
        for (int j = kC - 1; j >= 0; --j) {
            yv = P2::fmac(yv, k2.nlam, r2[j]);
            zz = P2::fmac(zz, k2.nlam, yv);
            r2[j] = zz;
        }
    }
    {
        VQ T = zv;
        VQ t = Q::down(T, 1);
        if (lane <= 30) T = Q::fmac(t, kq.m1, T);
        t = Q::down(T, 2);
        if (lane <= 29) T = Q::fmac(t, kq.m2, T);
        VQ c = Q::down(T, 1);
        if (lane == 31) c = Q::zero();
#pragma unroll
        for (int j = 0; j < kC; ++j) r[j] = Q::fmac(c, kq.pw[kC - 1 - j], r[j]);
    }
    if (SECOND) {
        V2 TY = yv, TZ = zz;
        V2 ty = P2::down(TY, 1), tz = P2::down(TZ, 1);
        if (lane <= 30) {
            TZ = TZ + k2.m1 * tz + k2.Cm1 * ty;
            TY = TY + k2.m1 * ty;
        }
        ty = P2::down(TY, 2);
        tz = P2::down(TZ, 2);
        if (lane <= 29) {
            TZ = TZ + k2.m2 * tz + k2.Cm2 * ty;
            TY = TY + k2.m2 * ty;
        }
        V2 cy = P2::down(TY, 1), cz = P2::down(TZ, 1);
        if (lane == 31) cy = cz = 0;
#pragma unroll
        for (int j = 0; j < kC; ++j)
            r2[j] = r2[j] + k2.pw[kC - 1 - j] * ((V2)(kC - j) * cy + cz);
    }
#pragma unroll
    for (int j = 0; j < kC; ++j) {
        tout1[w * kSO + q0 + j] = Q::out(r[j]);
        if (SECOND) tout2[w * kSO + q0 + j] = r2[j];
    }
}

// y-lines of FP32 fields, window staged row by row: slot r of the window
// (position r - 4) holds the NL adjacent columns of one grid row,
// tin[r * NL + line].  A lane owns chunk c = (32 / NL) warp + lane / NL (kC
// positions from q0 = c kC) of line lane % NL; the lanes of a warp read 32 / NL
// chunks x NL lines at one row offset per access, in 32 distinct banks (kC is
// odd).  The chunks of a line sit in different warps, so their boundary states
// are joined through shared memory: the state entering chunk c is
// E_{c-1} + m E_{c-2} + m^2 E_{c-3} (m = (-lam)^kC), the same three terms the
// shuffle scan of solve_window keeps.  Results go to tout1 / tout2 in the same
// row layout, position q at [q * NL + line].
template <bool SIXTH, bool SECOND, int NL>
__device__ __forceinline__ void solve_window_y(const float* tin, float* tout1, float* tout2,
                                               const LineConst<PolF>& kq,
                                               const LineConst<PolF>& k2) {
    __shared__ float xa[32][NL], xb[32][NL], xc[32][NL];  // forward states
    __shared__ float ya[32][NL], yb[32][NL], yc[32][NL];  // backward states
    const int tid = threadIdx.x;
    const int w = tid >> 5, lane = tid & 31;
    static_assert(32 % NL == 0, "a warp holds whole rows of the window");
    const int l = lane % NL, c = (32 / NL) * w + lane / NL;  // NL warps: 32 chunks
    const int q0 = c * kC;
    auto tl = [&](int q) { return tin[(q + 4) * NL + l]; };  // q in [-4, kW+4)

    float r[kC];
    {
        float u[kC + 4];
#pragma unroll
        for (int k = 0; k < kC + 4; ++k) u[k] = tl(q0 - 2 + k);
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            float b = (u[j + 3] - u[j + 1]) * kq.c1;
            if (SIXTH) b = fmaf(u[j + 4] - u[j], kq.c2, b);
            r[j] = b;
        }
    }
    float r2[kC];
    if (SECOND) {
        float bx[kC + 4];
#pragma unroll
        for (int k = 0; k < kC + 4; ++k) {
            if (k >= 2 && k < kC + 2) {
                bx[k] = r[k - 2];
            } else {
                const int qc = q0 - 2 + k;
                float t = (tl(qc + 1) - tl(qc - 1)) * k2.c1;
                if (SIXTH) t = fmaf(tl(qc + 2) - tl(qc - 2), k2.c2, t);
                bx[k] = t;
            }
        }
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            float t = (bx[j + 3] - bx[j + 1]) * k2.c1;
            if (SIXTH) t = fmaf(bx[j + 4] - bx[j], k2.c2, t);
            r2[j] = t;
        }
    }
    // forward recursions over the chunk from a zero state
    float wv = 0.0f;
#pragma unroll
    for (int j = 0; j < kC; ++j) {
        wv = fmaf(wv, kq.nlam, r[j]);
        r[j] = wv;
    }
    float vv = 0.0f, ww = 0.0f;
    if (SECOND) {
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            vv = fmaf(vv, k2.nlam, r2[j]);
            ww = fmaf(ww, k2.nlam, vv);
            r2[j] = ww;
        }
    }
    xa[c][l] = wv;
    if (SECOND) {
        xb[c][l] = vv;
        xc[c][l] = ww;
    }
    __syncthreads();  // also: every staged value this block reads has been read
    {
        float cf = 0.0f;
        if (c >= 1) cf = xa[c - 1][l];
        if (c >= 2) cf = fmaf(xa[c - 2][l], kq.m1, cf);
        if (c >= 3) cf = fmaf(xa[c - 3][l], kq.m2, cf);
#pragma unroll
        for (int j = 0; j < kC; ++j) r[j] = fmaf(cf, kq.pw[j], r[j]);
    }
    if (SECOND) {
        float cv = 0.0f, cw = 0.0f;
        if (c >= 1) {
            cv = xb[c - 1][l];
            cw = xc[c - 1][l];
        }
        if (c >= 2) {
            cw = cw + k2.m1 * xc[c - 2][l] + k2.Cm1 * xb[c - 2][l];
            cv = cv + k2.m1 * xb[c - 2][l];
        }
        if (c >= 3) {
            cw = cw + k2.m2 * xc[c - 3][l] + k2.Cm2 * xb[c - 3][l];
            cv = cv + k2.m2 * xb[c - 3][l];
        }
#pragma unroll
        for (int j = 0; j < kC; ++j) r2[j] = r2[j] + k2.pw[j] * ((float)(j + 1) * cv + cw);
    }
    // backward recursions over the chunk from a zero state
    float zv = 0.0f;
#pragma unroll
    for (int j = kC - 1; j >= 0; --j) {
        zv = fmaf(zv, kq.nlam, r[j]);
        r[j] = zv;
    }
    float yv = 0.0f, zz = 0.0f;
    if (SECOND) {
#pragma unroll
        for (int j = kC - 1; j >= 0; --j) {
            yv = fmaf(yv, k2.nlam, r2[j]);
            zz = fmaf(zz, k2.nlam, yv);
            r2[j] = zz;
        }
    }
    ya[c][l] = zv;
    if (SECOND) {
        yb[c][l] = yv;
        yc[c][l] = zz;
    }
    __syncthreads();
    {
        float cb = 0.0f;
        if (c <= 30) cb = ya[c + 1][l];
        if (c <= 29) cb = fmaf(ya[c + 2][l], kq.m1, cb);
        if (c <= 28) cb = fmaf(ya[c + 3][l], kq.m2, cb);
#pragma unroll
        for (int j = 0; j < kC; ++j) r[j] = fmaf(cb, kq.pw[kC - 1 - j], r[j]);
    }
    if (SECOND) {
        float cy = 0.0f, cz = 0.0f;
        if (c <= 30) {
            cy = yb[c + 1][l];
            cz = yc[c + 1][l];
        }
        if (c <= 29) {
            cz = cz + k2.m1 * yc[c + 2][l] + k2.Cm1 * yb[c + 2][l];
            cy = cy + k2.m1 * yb[c + 2][l];
        }
        if (c <= 28) {
            cz = cz + k2.m2 * yc[c + 3][l] + k2.Cm2 * yb[c + 3][l];
            cy = cy + k2.m2 * yb[c + 3][l];
        }
#pragma unroll
        for (int j = 0; j < kC; ++j)
            r2[j] = r2[j] + k2.pw[kC - 1 - j] * ((float)(kC - j) * cy + cz);
    }
#pragma unroll
    for (int j = 0; j < kC; ++j) {
        tout1[(q0 + j) * NL + l] = r[j];
        if (SECOND) tout2[(q0 + j) * NL + l] = r2[j];
    }
}

template <int AXIS, class P1, class P2, bool SIXTH, bool SECOND, int NL, class In, class Epi>
__device__ __forceinline__ void lines_body(In& in, const LineGeo& g, const LineConst<P1>& k1,
                                           const LineConst<PolF>& k1f,
                                           const LineConst<P2>& k2, Epi& epi, DevState* st,
                                           int bid, const CUtensorMap* tmap = nullptr) {
    // FP32 y-lines stage their window row by row ([slot][NL lines]); the rest
    // stage it line by line ([line][slot])
    constexpr bool kRowY = AXIS == 1 && std::is_same<P1, PolF>::value &&
                           std::is_same<P2, PolF>::value;
    using V1 = typename P1::V;
    using V2 = typename P2::V;
    using O1 = typename P1::O;
    using S1 = typename P1::S;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int kPS = NL * kLW;                                   // plane stride
    // the outputs reuse the staged planes: the first derivative plane 0, the
    // second plane 1 (double-float input) or a plane of its own
    S1* tin = reinterpret_cast<S1*>(smem_raw);                      // [planes][NL][kLW]
    static_assert(sizeof(O1) == sizeof(S1), "first derivative over the staged plane 0");
    O1* tout1 = reinterpret_cast<O1*>(tin);                         // [NL][kSO]
    V2* tout2 = P1::kPlanes >= 2 ? reinterpret_cast<V2*>(tin + kPS)
                                 : reinterpret_cast<V2*>(tin + P1::kPlanes * kPS);

    const int grp = bid % g.ngroups;
    const int win = bid / g.ngroups;
    const int line0 = grp * NL;
    const int s = win * g.own;                      // first owned position
    const int e = min(s + g.own, g.n);              // one past the last
    const int tid = threadIdx.x;

    // ---- stage the window: positions s-H-4 .. s-H+kW+3 of NL lines ----
    constexpr int LWIN = kW + 8;
    const int p0 = wrapi((long long)s - g.H - 4, g.period);  // period position of slot 0
    const bool short_line = g.period < LWIN;
    if constexpr (kRowY) {
        // row layout: slot q holds columns line0 .. line0 + 7 of period position p0 + q
        const long long p_end = (long long)s - g.H - 4 + LWIN;  // one past the last slot
        const bool interior = (long long)s - g.H - 4 >= 0 && p_end <= g.n;
        if (tmap && st && g.vec && interior && line0 + NL <= g.nlines &&
            (smem_u32(tin) & 127u) == 0) {
            // one elected thread moves the window with tensor copies
            __shared__ __align__(8) uint64_t bar;
            if (tid == 0) mbar_init(&bar, 1);
            __syncthreads();
            if (tid == 0) {
                mbar_expect_tx(&bar, (unsigned)(LWIN * NL * sizeof(float)));
#pragma unroll 1
                for (int b = 0; b < LWIN / kBoxRows; ++b)
                    tma_load_2d(tin + b * kBoxRows * NL, tmap, line0, p0 + b * kBoxRows, &bar);
            }
            const bool arrived = mbar_wait_bounded(&bar, 0);
            if (__syncthreads_or(!arrived)) {
                // not arrived in time: flag the run; wait once more (bounded) for
                // the copies in flight before the block leaves its shared memory
                if (tid == 0) raise_flag(st, FLAG_STAGE, st->t);
                mbar_wait_bounded(&bar, 0);
                return;
            }
        } else if (g.vec) {
            // 16-byte pieces: slot q, piece h covers columns line0 + 4h .. + 3
            constexpr int PR = NL / 4;  // pieces per row
            for (int idx = tid; idx < PR * LWIN; idx += NL * 32) {
                const int q = idx / PR, h = idx % PR;
                const int col = line0 + 4 * h;
                S1* dst = tin + q * NL + 4 * h;
                if (col < g.nlines) {
                    int p = p0 + q;
                    if (short_line) p %= g.period;
                    else if (p >= g.period) p -= g.period;
                    if (g.mirror && p >= g.n) p = 2 * g.n - 1 - p;
                    in.stage4(dst, 0, kPS, (size_t)p * g.ps + (size_t)col);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) dst[k] = 0.0f;
                }
            }
        } else {
            for (int idx = tid; idx < NL * LWIN; idx += NL * 32) {
                const int q = idx / NL, ll = idx % NL;
                const int col = line0 + ll;
                if (col < g.nlines) {
                    int p = p0 + q;
                    if (short_line) p %= g.period;
                    else if (p >= g.period) p -= g.period;
                    if (g.mirror && p >= g.n) p = 2 * g.n - 1 - p;
                    in.stage(tin, q * NL + ll, kPS, (size_t)p * g.ps + (size_t)col);
                } else {
                    tin[q * NL + ll] = 0.0f;
                }
            }
        }
    } else if (AXIS == 0 && g.vec) {
        // rows: warp w stages line line0 + w in 16-byte chunks (p0, H and own are
        // multiples of 4, and so is the line length, so no chunk straddles the
        // periodic wrap)
        constexpr int CW = LWIN / 4;
        const int l = tid >> 5, lane = tid & 31;
        const int line = line0 + l;
        if (line < g.nlines) {
            const size_t lbase = (size_t)line * g.ls;
            for (int c = lane; c < CW; c += 32) {
                int p = p0 + 4 * c;
                if (short_line) p %= g.period;
                else if (p >= g.period) p -= g.period;
                in.stage4(tin, l * kLW + 4 * c, kPS, lbase + (size_t)p);
            }
        } else {
            for (int c = lane; c < CW; c += 32) {
#pragma unroll
                for (int k = 0; k < 4; ++k) P1::sput(tin, l * kLW + 4 * c + k, kPS, P1::zero());
            }
        }
    } else {
        for (int idx = tid; idx < NL * LWIN; idx += NL * 32) {
            int l, q;
            if (AXIS == 0) {
                l = idx / LWIN;
                q = idx - l * LWIN;
            } else {
                q = idx / NL;
                l = idx - q * NL;
            }
            const int line = line0 + l;
            if (line < g.nlines) {
                int p = p0 + q;
                if (short_line) p %= g.period;
                else if (p >= g.period) p -= g.period;
                if (g.mirror && p >= g.n) p = 2 * g.n - 1 - p;
                in.stage(tin, l * kLW + q, kPS, (size_t)line * g.ls + (size_t)p * g.ps);
            } else {
                P1::sput(tin, l * kLW + q, kPS, P1::zero());
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();

    // ---- solve: double-float only where the window spans a large range ----
    // With all staged densities within a factor 32, FP32 rounding stays below
    // ~2e-6 of the local values, as accurate as the FP32 result that is stored;
    // only windows reaching across an interface need the double-float solve.
    if constexpr (kRowY) {
        solve_window_y<SIXTH, SECOND, NL>(tin, tout1, tout2, k1, k2);
    } else if constexpr (std::is_same<P1, PolDF>::value) {
        __shared__ float red[2][NL];
        float mn = FLT_MAX, mx = 0.0f;
        for (int idx = tid; idx < NL * LWIN; idx += NL * 32) {
            const int l = idx / LWIN, q = idx - l * LWIN;
            const float v = tin[l * kLW + q];
            mn = fminf(mn, v);
            mx = fmaxf(mx, v);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mn = fminf(mn, __shfl_xor_sync(kFull, mn, o));
            mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
        }
        if ((tid & 31) == 0) {
            red[0][tid >> 5] = mn;
            red[1][tid >> 5] = mx;
        }
        __syncthreads();
        mn = red[0][0];
        mx = red[1][0];
#pragma unroll
        for (int k = 1; k < NL; ++k) {
            mn = fminf(mn, red[0][k]);
            mx = fmaxf(mx, red[1][k]);
        }
        if (mn > 0.0f && mx <= 32.0f * mn)
            solve_window<PolF, P1, P2, SIXTH, SECOND, NL>(tin, tout1, tout2, k1f, k2);
        else
            solve_window<P1, P1, P2, SIXTH, SECOND, NL>(tin, tout1, tout2, k1, k2);
    } else {
        solve_window<P1, P1, P2, SIXTH, SECOND, NL>(tin, tout1, tout2, k1, k2);
    }
    __syncthreads();

    // ---- epilogue over the owned positions, coalesced ----
    // Each thread takes elements tid, tid + 256, ...; operands are fetched in
    // groups of kB before any of the group's results is written.
    constexpr int kB = Epi::kBatch;
    const int nown = e - s;
    const int lmax = min(NL, g.nlines - line0);
    bool bad = false;
    if constexpr (kRowY) {
        // outputs in the row layout: position q of line l at [q * NL + l]
        if (g.vec) {
            // 16-byte pieces: one row, four adjacent lines (columns line0 + 4h ..)
            constexpr int PR = NL / 4;  // pieces per row
            const int total = PR * nown;
            for (int base = tid; base < total; base += kB * NL * 32) {
                int sl[kB];
                size_t off[kB];
                typename Epi::Ops4 ops[kB];
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    const int idx = base + k * NL * 32;
                    const int qq = idx / PR, h4 = 4 * (idx % PR);
                    sl[k] = (g.H + qq) * NL + h4;
                    off[k] = (size_t)(line0 + h4) + (size_t)(s + qq) * g.ps;
                    if (!(idx < total && h4 < lmax)) sl[k] = -1;
                    else ops[k] = epi.fetch4(off[k]);
                }
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    if (sl[k] < 0) continue;
                    const float4 a = *reinterpret_cast<const float4*>(tout1 + sl[k]);
                    float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (SECOND) b = *reinterpret_cast<const float4*>(tout2 + sl[k]);
                    bad |= epi.put4(off[k], a, b, ops[k]);
                }
            }
        } else {
            const int total = NL * nown;
            for (int base = tid; base < total; base += kB * NL * 32) {
                int slot[kB];
                size_t off[kB];
                typename Epi::Ops ops[kB];
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    const int idx = base + k * NL * 32;
                    const int qq = idx / NL, ll = idx % NL;
                    const bool live = idx < total && ll < lmax;
                    slot[k] = live ? (g.H + qq) * NL + ll : -1;
                    off[k] = (size_t)(line0 + ll) + (size_t)(s + qq) * g.ps;
                    if (live) ops[k] = epi.fetch(off[k]);
                }
#pragma unroll
                for (int k = 0; k < kB; ++k)
                    if (slot[k] >= 0)
                        bad |= epi(off[k], tout1[slot[k]], SECOND ? tout2[slot[k]] : (V2)0,
                                   ops[k]);
            }
        }
        bad |= in.flagged();
        if (bad) raise_flag(st, FLAG_EOS, st->t);
        return;
    }
    if constexpr (AXIS == 0 && sizeof(O1) == 4 && sizeof(V2) == 4) {
        if (g.vec) {
            // float fields, nx % 4 == 0: warp w writes line line0 + w in chunks
            // of four outputs, 16-byte loads from the staged plane and stores
            const int ll = tid >> 5, lane = tid & 31;
            if (ll < lmax) {
                const size_t lbase = (size_t)(line0 + ll) * g.ls + (size_t)s;
                const int sbase = ll * kSO + g.H;
                for (int q4 = 4 * lane; q4 < nown; q4 += 4 * 32 * kB) {
                    typename Epi::Ops4 ops[kB];
#pragma unroll
                    for (int k = 0; k < kB; ++k) {
                        const int qq = q4 + 4 * 32 * k;
                        if (qq < nown) ops[k] = epi.fetch4(lbase + qq);
                    }
#pragma unroll
                    for (int k = 0; k < kB; ++k) {
                        const int qq = q4 + 4 * 32 * k;
                        if (qq >= nown) continue;
                        const float4 a = *reinterpret_cast<const float4*>(tout1 + sbase + qq);
                        float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (SECOND) b = *reinterpret_cast<const float4*>(tout2 + sbase + qq);
                        bad |= epi.put4(lbase + qq, a, b, ops[k]);
                    }
                }
            }
            bad |= in.flagged();
            if (bad) raise_flag(st, FLAG_EOS, st->t);
            return;
        }
    }
    if constexpr (sizeof(O1) == 4 && sizeof(V2) == 4) {
        if (g.vec) {
            // float fields, nx % 4 == 0: chunks of four outputs, 16-byte stores.
            // x-lines: four consecutive positions of one line; y-lines: one
            // position of four adjacent lines (columns line0 + 4h .. + 3).
            const int cpl = AXIS == 0 ? nown / 4 : 2;  // chunks per line / per position
            const int total = AXIS == 0 ? NL * cpl : 2 * nown;
            for (int base = tid; base < total; base += kB * NL * 32) {
                int sl[kB];
                size_t off[kB];
                typename Epi::Ops4 ops[kB];
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    const int idx = base + k * NL * 32;
                    bool live;
                    if (AXIS == 0) {
                        const int ll = idx / cpl;
                        const int qq = 4 * (idx - ll * cpl);
                        live = idx < total && ll < lmax;
                        sl[k] = ll * kSO + g.H + qq;
                        off[k] = (size_t)(line0 + ll) * g.ls + (size_t)(s + qq);
                    } else {
                        const int qq = idx >> 1, h4 = 4 * (idx & 1);
                        live = idx < total && h4 < lmax;
                        sl[k] = h4 * kSO + g.H + qq;
                        off[k] = (size_t)(line0 + h4) + (size_t)(s + qq) * g.ps;
                    }
                    if (!live) sl[k] = -1;
                    else ops[k] = epi.fetch4(off[k]);
                }
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    if (sl[k] < 0) continue;
                    float4 a, b = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (AXIS == 0) {
                        a = *reinterpret_cast<const float4*>(tout1 + sl[k]);
                        if (SECOND) b = *reinterpret_cast<const float4*>(tout2 + sl[k]);
                    } else {
                        a = make_float4(tout1[sl[k]], tout1[sl[k] + kSO], tout1[sl[k] + 2 * kSO],
                                        tout1[sl[k] + 3 * kSO]);
                        if (SECOND)
                            b = make_float4(tout2[sl[k]], tout2[sl[k] + kSO],
                                            tout2[sl[k] + 2 * kSO], tout2[sl[k] + 3 * kSO]);
                    }
                    bad |= epi.put4(off[k], a, b, ops[k]);
                }
            }
            bad |= in.flagged();
            if (bad) raise_flag(st, FLAG_EOS, st->t);
            return;
        }
    }
    const int total = NL * nown;
    int l0 = 0, q0e = tid;  // AXIS 0 walk: position q0e within line l0
    if (AXIS == 0) {
        while (q0e >= nown && l0 < NL) { q0e -= nown; ++l0; }
    }
    for (int base = tid; base < total; base += kB * NL * 32) {
        int slot[kB];
        size_t off[kB];
        typename Epi::Ops ops[kB];
#pragma unroll
        for (int k = 0; k < kB; ++k) {
            int ll, qq;
            if (AXIS == 0) {
                ll = l0;
                qq = q0e;
                q0e += NL * 32;
                while (q0e >= nown && l0 < NL) { q0e -= nown; ++l0; }
            } else {
                const int idx = base + k * NL * 32;
                qq = idx / NL;
                ll = idx - qq * NL;
            }
            const bool live = ll < lmax && qq < nown;
            slot[k] = live ? ll * kSO + g.H + qq : -1;
            off[k] = AXIS == 0 ? (size_t)(line0 + ll) * g.ls + (size_t)(s + qq)
                               : (size_t)(line0 + ll) + (size_t)(s + qq) * g.ps;
            if (live) ops[k] = epi.fetch(off[k]);
        }
#pragma unroll
        for (int k = 0; k < kB; ++k)
            if (slot[k] >= 0)
                bad |= epi(off[k], tout1[slot[k]], SECOND ? tout2[slot[k]] : (V2)0, ops[k]);
    }
    bad |= in.flagged();
    if (bad) raise_flag(st, FLAG_EOS, st->t);
}

template <int AXIS, class P1, class P2, bool SIXTH, bool SECOND, class In, class Epi>
__global__ void __launch_bounds__(kNL * 32)
    k_lines(In in, LineGeo g, LineConst<P1> k1, LineConst<PolF> k1f, LineConst<P2> k2, Epi epi,
            DevState* st, int bump) {
    if (bump && blockIdx.x == 0 && threadIdx.x == 0) st->t += 1;
    epi.init(st);
    in.init(st);
    lines_body<AXIS, P1, P2, SIXTH, SECOND, kNL>(in, g, k1, k1f, k2, epi, st, (int)blockIdx.x);
}

// x-lines and y-lines of two independent solves in one launch: blocks below
// nbx take the x windows, the rest the y windows.
// Blocks of NL lines (NL warps); the launch bounds keep 32 warps per SM.
template <int NL, bool SECOND, class P1>
constexpr int xy_min_blocks() {
    return NL == 8 ? (SECOND && P1::kPlanes >= 2 ? 3 : 4) : 8 * 4 / NL;
}

template <class P1, class P2, bool SIXTH, bool SECOND, int NL, class InX, class EpiX,
          class InY, class EpiY>
__global__ void __launch_bounds__(NL * 32, (xy_min_blocks<NL, SECOND, P1>()))
    k_lines_xy(InX inx, LineGeo gx, EpiX ex, InY iny, LineGeo gy, EpiY ey, LineConst<P1> k1,
               LineConst<PolF> k1f, LineConst<P2> k2, DevState* st, int bump, int nbx,
               const __grid_constant__ CUtensorMap tmy, int use_tma, int y_first) {
    pdl_prologue();
    if (bump && blockIdx.x == 0 && threadIdx.x == 0) st->t += 1;
    // y_first: the y-line blocks take the low block indices, so they are
    // dispatched first (in a launch of about one wave the slower y-windows then
    // do not form the tail); otherwise by tiles
    const int nby = (int)gridDim.x - nbx;
    bool x;
    int local;
    if (y_first) {
        x = (int)blockIdx.x >= nby;
        local = x ? (int)blockIdx.x - nby : (int)blockIdx.x;
    } else {
        // line groups across a tile (windows of a longer line own a multiple of NL)
        const int gr = gy.nwin == 1 ? gx.ngroups : gy.own / NL;
        const int gc = gx.nwin == 1 ? gy.ngroups : gx.own / NL;
        const int row = gx.nwin * gr + gy.ngroups;     // blocks of a full row of tiles
        const int ty = min((int)blockIdx.x / row, gy.nwin - 1);
        int r = (int)blockIdx.x - ty * row;
        const int cx = min(gr, gx.ngroups - ty * gr);
        const int tx = min(r / (cx + gc), gx.nwin - 1);
        r -= tx * (cx + gc);
        x = r < cx;
        local = x ? tx * gx.ngroups + ty * gr + r : ty * gy.ngroups + tx * gc + r - cx;
    }
    if (x) {
        ex.init(st);
        inx.init(st);
        lines_body<0, P1, P2, SIXTH, SECOND, NL>(inx, gx, k1, k1f, k2, ex, st, local);
    } else {
        ey.init(st);
        iny.init(st);
        lines_body<1, P1, P2, SIXTH, SECOND, NL>(iny, gy, k1, k1f, k2, ey, st, local,
                                             use_tma ? &tmy : nullptr);
    }
}

// Batched x|y lines: block b belongs to instance map[b]; within the instance the
// blocks are those of k_lines_xy for its grid.  Each instance bumps its own
// time level.
template <class InX, class EpiX, class InY, class EpiY>
struct LinesXYInst {
    InX inx;
    EpiX ex;
    InY iny;
    EpiY ey;
    LineGeo gx, gy;
    int nbx;   // x-line blocks of this instance
    int blk0;  // first block of this instance in the launch
    DevState* st;
};

template <class P1, class P2, bool SIXTH, bool SECOND, int NL, class InX, class EpiX, class InY,
          class EpiY>
__global__ void __launch_bounds__(NL * 32, NL == 8 ? 3 : 2)
    k_lines_xy_batch(const LinesXYInst<InX, EpiX, InY, EpiY>* __restrict__ d,
                     const int* __restrict__ map, LineConst<P1> k1, LineConst<PolF> k1f,
                     LineConst<P2> k2, int bump) {
    const LinesXYInst<InX, EpiX, InY, EpiY>& D = d[map[blockIdx.x]];
    DevState* st = D.st;
    const int local = (int)blockIdx.x - D.blk0;
    if (bump && local == 0 && threadIdx.x == 0) st->t += 1;
    if (local < D.nbx) {
        InX in = D.inx;
        EpiX epi = D.ex;
        const LineGeo g = D.gx;
        epi.init(st);
        in.init(st);
        lines_body<0, P1, P2, SIXTH, SECOND, NL>(in, g, k1, k1f, k2, epi, st, local);
    } else {
        InY in = D.iny;
        EpiY epi = D.ey;
        const LineGeo g = D.gy;
        epi.init(st);
        in.init(st);
        lines_body<1, P1, P2, SIXTH, SECOND, NL>(in, g, k1, k1f, k2, epi, st, local - D.nbx);
    }
}

// ---- epilogues: return true when a value is bad (flags the run) ----
template <class O, class V2>
struct EpiStore {
    static constexpr int kBatch = 4;  // outputs fetched per thread before any is written
    O* d1;
    V2* d2;
    struct Ops {};
    struct Ops4 {};
    __device__ __forceinline__ void init(const DevState*) {}
    __device__ __forceinline__ Ops fetch(size_t) const { return Ops{}; }
    __device__ __forceinline__ bool operator()(size_t o, O a, V2 b, const Ops&) {
        d1[o] = a;
        if (d2) d2[o] = b;
        return false;
    }
    // four consecutive outputs (float fields only)
    __device__ __forceinline__ Ops4 fetch4(size_t) const { return Ops4{}; }
    __device__ __forceinline__ bool put4(size_t o, float4 a, float4 b, const Ops4&) {
        *reinterpret_cast<float4*>(d1 + o) = a;
        if (d2) *reinterpret_cast<float4*>(d2 + o) = b;
        return false;
    }
};

// F = -rho d(mu-hat) + c_s^2 d(rho), Eq. 12.  In FP32, c_s^2 = 1/3 as a constant is 3e-8
// too large, a bias that the populations' pressure does not share and that moves the dilute
// gas at high density ratios.  So c_s^2 = hi + lo, and the sum is rounded once.
__device__ __forceinline__ float force_term(float r, float dmu, float d) {
    constexpr float hi = 1.0f / 3.0f;
    constexpr float lo = (float)(1.0 / 3.0 - (double)hi);
    return rn_fma(d, hi, rn_fma(-r, dmu, rn_mul(d, lo)));
}

template <class O, class RhoT>
struct EpiForce {
    static constexpr int kBatch = 4;  // its operands are float4 pairs: four in flight
    O* F;
    const RhoT* __restrict__ rho;
    const O* __restrict__ dr;
    struct Ops {
        RhoT r;
        O d;
    };
    __device__ __forceinline__ void init(const DevState*) {}
    __device__ __forceinline__ Ops fetch(size_t o) const { return Ops{__ldg(rho + o), __ldg(dr + o)}; }
    __device__ __forceinline__ bool operator()(size_t o, O dmu, O, const Ops& op) {
        // explicit rounding: the epilogue is inlined in several kernels
        F[o] = force_term((O)op.r, dmu, op.d);
        return false;
    }
    struct Ops4 {
        float4 r, d;
    };
    __device__ __forceinline__ Ops4 fetch4(size_t o) const {
        return Ops4{__ldg(reinterpret_cast<const float4*>(rho + o)),
                    __ldg(reinterpret_cast<const float4*>(dr + o))};
    }
    __device__ __forceinline__ bool put4(size_t o, float4 dmu, float4, const Ops4& op) {
        float4 f;
        f.x = force_term(op.r.x, dmu.x, op.d.x);
        f.y = force_term(op.r.y, dmu.y, op.d.y);
        f.z = force_term(op.r.z, dmu.z, op.d.z);
        f.w = force_term(op.r.w, dmu.w, op.d.w);
        *reinterpret_cast<float4*>(F + o) = f;
        return false;
    }
};

// ---------------------------------------------------------------------------
// Host side: constants, geometry, launch
// ---------------------------------------------------------------------------
struct Scheme {
    double alpha, a, b, lam, c1, c2;
};
Scheme scheme(int order) {
    Scheme s;
    s.alpha = order == 6 ? 1.0 / 3.0 : 0.25;
    s.a = 2.0 / 3.0 * (s.alpha + 2.0);  // Eq. 38
    s.b = (4.0 * s.alpha - 1.0) / 3.0;  // Eq. 38
    s.lam = (1.0 - std::sqrt(1.0 - 4.0 * s.alpha * s.alpha)) / (2.0 * s.alpha);
    s.c1 = s.lam / s.alpha * s.a / 2.0;
    s.c2 = s.lam / s.alpha * s.b / 4.0;
    return s;
}

template <class P>
LineConst<P> make_const(int order) {
    const Scheme sc = scheme(order);
    LineConst<P> k;
    k.c1 = P::konst(sc.c1);
    k.c2 = P::konst(sc.c2);
    k.nlam = P::konst(-sc.lam);
    double p = 1.0;
    for (int j = 0; j < kC; ++j) {
        p *= -sc.lam;
        k.pw[j] = P::konst(p);
    }
    const double m = std::pow(-sc.lam, kC);
    k.m1 = P::konst(m);
    k.m2 = P::konst(m * m);
    k.Cm1 = P::konst(kC * m);
    k.Cm2 = P::konst(2.0 * kC * m * m);
    return k;
}

// Halo: lam^H (single recursion) or (H+1) lam^H (double) below eps.
int halo(int order, double eps1, bool second, double eps2) {
    const double lam = scheme(order).lam;
    int h1 = 1;
    while (std::pow(lam, h1) >= eps1) ++h1;
    int h2 = 0;
    if (second) {
        h2 = 1;
        while ((h2 + 1) * std::pow(lam, h2) >= eps2) ++h2;
    }
    return (h1 > h2 ? h1 : h2) + 1;
}

// Walls in y (walls_y): the y-lines are extended evenly about both walls, a
// periodic line of period 2 ny whose first ghost equals its fluid neighbour
// (the wall rule of Sec. 5.5); only the ny fluid positions are owned.
LineGeo make_geo(int nx, int ny, int axis, int H, bool walls_y = false, int nl = kNL) {
    LineGeo g;
    if (axis == 0) {
        g.n = nx; g.nlines = ny; g.ps = 1; g.ls = nx;
    } else {
        g.n = ny; g.nlines = nx; g.ps = nx; g.ls = 1;
    }
    // the halo is rounded up to a multiple of 4 so that windows start on
    // 16-byte boundaries (own = kW - 2H is then a multiple of 4 too)
    H = (H + 3) / 4 * 4;
    g.H = H;
    g.own = kW - 2 * H;
    if (g.own > g.n) g.own = g.n;
    g.nwin = (g.n + g.own - 1) / g.own;
    g.ngroups = (g.nlines + nl - 1) / nl;
    g.vec = nx % 4 == 0;
    g.mirror = axis == 1 && walls_y;
    g.period = g.mirror ? 2 * g.n : g.n;
    return g;
}

template <class P1, class P2, bool SECOND, int NL = kNL>
size_t smem_bytes() {
    return (size_t)P1::kPlanes * NL * kLW * sizeof(typename P1::S) +
           (SECOND && P1::kPlanes < 2 ? (size_t)NL * kSO * sizeof(typename P2::V) : 0);
}

template <int AXIS, class P1, class P2, bool SIXTH, bool SECOND, class In, class Epi>
cudaError_t launch_lines_t(In in, const LineGeo& g, int order, Epi epi, DevState* st, int bump,
                           cudaStream_t s) {
    auto kern = k_lines<AXIS, P1, P2, SIXTH, SECOND, In, Epi>;
    const size_t smem = smem_bytes<P1, P2, SECOND>();
    static bool attr = false;  // one flag per kernel instantiation
    if (!attr) {
        cudaError_t e =
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const unsigned blocks = (unsigned)((long long)g.ngroups * g.nwin);
    kern<<<blocks, kNL * 32, smem, s>>>(in, g, make_const<P1>(order), make_const<PolF>(order),
                                        make_const<P2>(order), epi, st, bump);
    return cudaGetLastError();
}

// Tensor map of an FP32 field [ny][nx] for the y-line windows: boxes of 8
// columns x kBoxRows rows, no swizzle.  The encoder is the driver's
// cuTensorMapEncodeTiled, looked up once through the runtime (no link to the
// driver library); without it, or for fields it cannot describe (nx not a
// multiple of 4), the windows are staged by cp.async instead.
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn tensor_map_encoder() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

bool y_tensor_map(const float* field, int nx, int ny, int nl, CUtensorMap* m) {
    if (!field || nx % 4 != 0 || nx < nl || ny < kW + 8) return false;
    const EncodeTiledFn enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)nx, (cuuint64_t)ny};
    const cuuint64_t strides[1] = {(cuuint64_t)nx * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)nl, (cuuint32_t)kBoxRows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(field), dims, strides,
               box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

template <class In>
const float* y_field(const In&) { return nullptr; }
const float* y_field(const InF& in) { return in.p; }

// Lines per block of a merged launch.  16 lines make the FP32 y-line windows
// move 64-byte row pieces (32-byte pieces lose about a quarter of the DRAM
// bandwidth: 2.5 against 3.35 TB/s measured for windows read alone), but halve
// the blocks resident per SM.  Measured on the merged density lines: 16 lines
// win on grids up to 1024^2 (13.3 against 14.8 us), 8 from 2048^2 up (30 against
// 32 us; 95 against 107 us at 4096^2).  Double-float and FP64 solves keep 8.
// The choice moves no result: every line is solved the same way either way.
constexpr long long kWideLinesMaxNodes = 1LL << 21;

template <class P1, class P2, bool SIXTH, bool SECOND, int NL, class InX, class EpiX,
          class InY, class EpiY>
cudaError_t launch_xy_t(InX inx, EpiX ex, InY iny, EpiY ey, int nx, int ny, int order, int H,
                        DevState* st, int bump, bool walls_y, cudaStream_t s) {
    auto kern = k_lines_xy<P1, P2, SIXTH, SECOND, NL, InX, EpiX, InY, EpiY>;
    const size_t smem = smem_bytes<P1, P2, SECOND, NL>();
    static bool attr = false;  // one flag per kernel instantiation
    if (!attr) {
        cudaError_t e =
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const LineGeo gx = make_geo(nx, ny, 0, H, false, NL),
                  gy = make_geo(nx, ny, 1, H, walls_y, NL);
    const int nbx = gx.ngroups * gx.nwin;
    const unsigned blocks = (unsigned)(nbx + gy.ngroups * gy.nwin);
    // FP32 y-lines take their interior windows by tensor copies (a state block
    // is needed to report a copy that never arrives)
    CUtensorMap tmy;
    std::memset(&tmy, 0, sizeof(tmy));
    int use_tma = 0;
    if (std::is_same<P1, PolF>::value && std::is_same<P2, PolF>::value && st)
        use_tma = y_tensor_map(y_field(iny), nx, ny, NL, &tmy) ? 1 : 0;
    // y-line blocks first in the launches of 16 lines a block (grids up to 2^21
    // nodes, about one wave): at 1024^2 the density lines 14.3 -> 12.7 us, the
    // force lines 12.3 -> 12.0; at 4096^2 (8 lines a block, many waves) no gain
    const int y_first = NL == 16 ? 1 : 0;
    return launch_pdl(kern, blocks, NL * 32, smem, s, inx, gx, ex, iny, gy, ey,
                      make_const<P1>(order), make_const<PolF>(order), make_const<P2>(order), st,
                      bump, nbx, tmy, use_tma, y_first);
}

template <class P1, class P2, bool SECOND, class InX, class EpiX, class InY, class EpiY>
cudaError_t launch_xy(InX inx, EpiX ex, InY iny, EpiY ey, int nx, int ny, int order,
                      double eps1, double eps2, DevState* st, int bump, cudaStream_t s,
                      bool walls_y = false) {
    const int H = halo(order, eps1, SECOND, eps2);
    constexpr bool kF32 = std::is_same<P1, PolF>::value && std::is_same<P2, PolF>::value;
    if constexpr (kF32) {
        if ((long long)nx * ny <= kWideLinesMaxNodes) {
            if (order == 6)
                return launch_xy_t<P1, P2, true, SECOND, 16>(inx, ex, iny, ey, nx, ny, order, H,
                                                             st, bump, walls_y, s);
            return launch_xy_t<P1, P2, false, SECOND, 16>(inx, ex, iny, ey, nx, ny, order, H, st,
                                                          bump, walls_y, s);
        }
    }
    if (order == 6)
        return launch_xy_t<P1, P2, true, SECOND, kNL>(inx, ex, iny, ey, nx, ny, order, H, st,
                                                      bump, walls_y, s);
    return launch_xy_t<P1, P2, false, SECOND, kNL>(inx, ex, iny, ey, nx, ny, order, H, st, bump,
                                                   walls_y, s);
}

// dispatch on axis and scheme order
template <class P1, class P2, bool SECOND, class In, class Epi>
cudaError_t launch_lines(In in, int nx, int ny, int axis, int order, double eps1, double eps2,
                         Epi epi, DevState* st, int bump, cudaStream_t s, bool walls_y = false) {
    const LineGeo g = make_geo(nx, ny, axis, halo(order, eps1, SECOND, eps2), walls_y);
    if (axis == 0) {
        if (order == 6)
            return launch_lines_t<0, P1, P2, true, SECOND>(in, g, order, epi, st, bump, s);
        return launch_lines_t<0, P1, P2, false, SECOND>(in, g, order, epi, st, bump, s);
    }
    if (order == 6) return launch_lines_t<1, P1, P2, true, SECOND>(in, g, order, epi, st, bump, s);
    return launch_lines_t<1, P1, P2, false, SECOND>(in, g, order, epi, st, bump, s);
}

// rounding levels the recursions are cut at
constexpr double kEpsDF = 1e-15, kEpsF = 1e-8;

// ---- batched mixed line passes ----
using RhoInst = LinesXYInst<InDF, EpiStore<float, float>, InDF, EpiStore<float, float>>;
using RhoF32Inst = LinesXYInst<InF, EpiStore<float, float>, InF, EpiStore<float, float>>;
using ForceInst = LinesXYInst<InF, EpiForce<float, float>, InF, EpiForce<float, float>>;

int halo_of(LineBatchKind kind, int order) {
    switch (kind) {
        case LineBatchKind::kRhoDF: return halo(order, kEpsDF, true, kEpsF);
        case LineBatchKind::kRhoF32: return halo(order, kEpsF, true, kEpsF);
        default: return halo(order, kEpsF, false, kEpsF);
    }
}

template <class P1, class P2, bool SIXTH, bool SECOND, int NL, class Inst>
cudaError_t launch_batch_t(const Inst* d, const int* map, int nblocks, int order, int bump,
                           cudaStream_t s) {
    auto kern = k_lines_xy_batch<P1, P2, SIXTH, SECOND, NL, decltype(Inst::inx),
                                 decltype(Inst::ex), decltype(Inst::iny), decltype(Inst::ey)>;
    const size_t smem = smem_bytes<P1, P2, SECOND, NL>();
    static bool attr = false;  // one flag per kernel instantiation
    if (!attr) {
        cudaError_t e =
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    kern<<<nblocks, NL * 32, smem, s>>>(d, map, make_const<P1>(order), make_const<PolF>(order),
                                        make_const<P2>(order), bump);
    return cudaGetLastError();
}

}  // namespace

// ---- mixed path ----
cudaError_t lines_mixed_rho_xy(const float* rh, const float* rl, float* dxr, float* dxx,
                               float* dyr, float* dyy, int nx, int ny, int order, DevState* st,
                               int bump, cudaStream_t s, bool walls_y) {
    return launch_xy<PolDF, PolF, true>(InDF{rh, rl}, EpiStore<float, float>{dxr, dxx},
                                        InDF{rh, rl}, EpiStore<float, float>{dyr, dyy}, nx, ny,
                                        order, kEpsDF, kEpsF, st, bump, s, walls_y);
}
cudaError_t lines_mixed_rho_xy_f32(const float* rh, float* dxr, float* dxx, float* dyr,
                                   float* dyy, int nx, int ny, int order, DevState* st, int bump,
                                   cudaStream_t s, bool walls_y) {
    return launch_xy<PolF, PolF, true>(InF{rh}, EpiStore<float, float>{dxr, dxx}, InF{rh},
                                       EpiStore<float, float>{dyr, dyy}, nx, ny, order, kEpsF,
                                       kEpsF, st, bump, s, walls_y);
}
cudaError_t lines_mixed_force_xy(const float* mu, const float* rh, const float* dxr,
                                 const float* dyr, float* Fx, float* Fy, int nx, int ny,
                                 int order, cudaStream_t s, bool walls_y, DevState* st) {
    return launch_xy<PolF, PolF, false>(InF{mu}, EpiForce<float, float>{Fx, rh, dxr}, InF{mu},
                                        EpiForce<float, float>{Fy, rh, dyr}, nx, ny, order,
                                        kEpsF, kEpsF, st, 0, s, walls_y);
}
cudaError_t lines_mixed_plain(const float* uh, const float* ul, float* d1, float* d2, int nx,
                              int ny, int axis, int order, cudaStream_t s) {
    if (d2)
        return launch_lines<PolDF, PolF, true>(InDF{uh, ul}, nx, ny, axis, order, kEpsDF, kEpsF,
                                               EpiStore<float, float>{d1, d2}, nullptr, 0, s);
    return launch_lines<PolDF, PolF, false>(InDF{uh, ul}, nx, ny, axis, order, kEpsDF, kEpsF,
                                            EpiStore<float, float>{d1, nullptr}, nullptr, 0, s);
}

// ---- batched mixed path ----
size_t lines_batch_desc_bytes(LineBatchKind kind) {
    switch (kind) {
        case LineBatchKind::kRhoDF: return sizeof(RhoInst);
        case LineBatchKind::kRhoF32: return sizeof(RhoF32Inst);
        default: return sizeof(ForceInst);
    }
}

// Lines per block of a batch launch: 8 or 16 for the FP32 kinds; the
// double-float density lines always 8 (16 would spill).
int batch_nl(LineBatchKind kind, int nl) { return kind == LineBatchKind::kRhoDF ? kNL : nl; }

int lines_batch_blocks(int nx, int ny, int order, LineBatchKind kind, int nl) {
    const int H = halo_of(kind, order);
    nl = batch_nl(kind, nl);
    const LineGeo gx = make_geo(nx, ny, 0, H, false, nl), gy = make_geo(nx, ny, 1, H, false, nl);
    return gx.ngroups * gx.nwin + gy.ngroups * gy.nwin;
}

void lines_batch_fill(LineBatchKind kind, const MixedLinesView& v, int order, int blk0,
                      void* host_dst, int nl) {
    const int H = halo_of(kind, order);
    nl = batch_nl(kind, nl);
    const LineGeo gx = make_geo(v.nx, v.ny, 0, H, false, nl),
                  gy = make_geo(v.nx, v.ny, 1, H, false, nl);
    const int nbx = gx.ngroups * gx.nwin;
    if (kind == LineBatchKind::kRhoDF) {
        RhoInst d{InDF{v.rh, v.rl}, EpiStore<float, float>{v.dxr, v.dxx},
                  InDF{v.rh, v.rl}, EpiStore<float, float>{v.dyr, v.dyy}, gx, gy, nbx, blk0, v.st};
        std::memcpy(host_dst, &d, sizeof(d));
    } else if (kind == LineBatchKind::kRhoF32) {
        RhoF32Inst d{InF{v.rh}, EpiStore<float, float>{v.dxr, v.dxx},
                     InF{v.rh}, EpiStore<float, float>{v.dyr, v.dyy}, gx, gy, nbx, blk0, v.st};
        std::memcpy(host_dst, &d, sizeof(d));
    } else {
        ForceInst d{InF{v.dxx}, EpiForce<float, float>{v.Fx, v.rh, v.dxr},
                    InF{v.dxx}, EpiForce<float, float>{v.Fy, v.rh, v.dyr}, gx, gy, nbx, blk0, v.st};
        std::memcpy(host_dst, &d, sizeof(d));
    }
}

cudaError_t lines_batch_launch(LineBatchKind kind, const void* d_desc, const int* map,
                               int nblocks, int order, int bump, cudaStream_t s, int nl) {
    if (nblocks <= 0) return cudaSuccess;
    const bool six = order == 6;
    if (kind == LineBatchKind::kRhoDF) {
        const RhoInst* d = static_cast<const RhoInst*>(d_desc);
        return six ? launch_batch_t<PolDF, PolF, true, true, kNL>(d, map, nblocks, order, bump, s)
                   : launch_batch_t<PolDF, PolF, false, true, kNL>(d, map, nblocks, order, bump, s);
    }
    if (kind == LineBatchKind::kRhoF32) {
        const RhoF32Inst* d = static_cast<const RhoF32Inst*>(d_desc);
        if (nl == 16)
            return six ? launch_batch_t<PolF, PolF, true, true, 16>(d, map, nblocks, order, bump, s)
                       : launch_batch_t<PolF, PolF, false, true, 16>(d, map, nblocks, order, bump,
                                                                     s);
        return six ? launch_batch_t<PolF, PolF, true, true, kNL>(d, map, nblocks, order, bump, s)
                   : launch_batch_t<PolF, PolF, false, true, kNL>(d, map, nblocks, order, bump, s);
    }
    const ForceInst* d = static_cast<const ForceInst*>(d_desc);
    if (nl == 16)
        return six ? launch_batch_t<PolF, PolF, true, false, 16>(d, map, nblocks, order, 0, s)
                   : launch_batch_t<PolF, PolF, false, false, 16>(d, map, nblocks, order, 0, s);
    return six ? launch_batch_t<PolF, PolF, true, false, kNL>(d, map, nblocks, order, 0, s)
               : launch_batch_t<PolF, PolF, false, false, kNL>(d, map, nblocks, order, 0, s);
}

}  // namespace cplbm
