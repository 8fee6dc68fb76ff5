// lines32.cuh -- FP32 compact-FD line solves of the mixed path (Eqs. 37-39): the density's
// first and second derivatives, and the derivative of mu-hat with the force (Eq. 12).
//
// The periodic compact scheme is the circulant system A d = B u with
//   (A d)_i = alpha d_{i-1} + d_i + alpha d_{i+1},
//   (B u)_i = a/2 (u_{i+1} - u_{i-1}) + b/4 (u_{i+2} - u_{i-2})   (a, b: Eq. 38).
// A = (alpha/lam)(1 + lam S^-1)(1 + lam S), lam = (1 - sqrt(1 - 4 alpha^2))/(2 alpha),
// so d follows from two first-order recursions on r = (lam/alpha) B u:
//   forward  w_i = r_i - lam w_{i-1},    backward  z_i = w_i - lam z_{i+1},   d = z.
// |lam| < 1 (0.382 at alpha = 1/3, 0.268 at 1/4): each recursion is exact to rounding once
// started a few dozen positions away.  The second derivative D(D u) ("applying CFM twice",
// Sec. 4.3) uses that the circulant operators commute: D D u = F_b F_b F_f F_f B B u, a
// double recursion in each direction.
//
// A line is cut into windows of 32 chunks of kC positions, H of them (24) before the first
// owned position, the last H after it.  A thread runs one chunk of one line in registers,
// both recursions from a zero state; the chunks' end states are joined through shared
// memory with m = (-lam)^kC (|m| = 1.1e-8): three or four of them are all that FP32 sees.
// So a window with few owned positions needs only the chunks up to four past its last
// owned one, and a block takes any number of lines: the threads of a block are its
// (line, chunk) pairs.  Short lines (a 64-line: 12 chunks, an 8-line: 8) then cost what they
// need, and small grids spread over more SMs.
//
// x-lines are staged in shared memory in 16-byte pieces and written back through it;
// y-lines need no staging: the threads of a warp are adjacent columns of one chunk, so each
// reads its 23 (27) rows straight into registers and writes its rows, coalesced as they are.
// Against full windows for every line (lines32_wide.cu): steps of 128^2 12.2 -> 11.6 us, 512^2
// 17.2 -> 16.0, 333 x 277 20.8 -> 17.2.  On large grids, where every chunk is needed and rows
// come from DRAM, those windows stay ahead.
#pragma once

#include "cplbm_internal.cuh"
#include "lattice.cuh"

namespace cplbm {

struct Line32 {
    float c1, c2, nlam;  // (lam/alpha) a/2, (lam/alpha) b/4, -lam
    float pw[kC32];      // (-lam)^(j+1)
    float m1, m2;        // (-lam)^C, (-lam)^(2C)
    float Cm1, Cm2;      // C (-lam)^C, 2C (-lam)^(2C)  (double-recursion joins)
};

Line32 line32_constants(int order);
Geo32 line32_geometry(int nx, int ny, int axis, int order, double eps1, double eps2,
                      bool walls_y);

namespace l32 {

constexpr int kC = kC32;
enum Mode : int {
    RHO,       // u -> first and second derivative
    FORCE,     // u = mu-hat -> F = -rho du + c_s^2 dr
};

__device__ __forceinline__ void cp4(void* s, const void* g) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(
                     (unsigned)__cvta_generic_to_shared(s)),
                 "l"(g)
                 : "memory");
}
__device__ __forceinline__ void cp16(void* s, const void* g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                     (unsigned)__cvta_generic_to_shared(s)),
                 "l"(g)
                 : "memory");
}

// F = -rho d(mu-hat) + c_s^2 d(rho), Eq. 12.  c_s^2 = 1/3 as an FP32 constant is 3e-8 too
// large, a bias that the populations' pressure does not share and that moves the dilute
// gas at high density ratios.  So c_s^2 = hi + lo, and the sum is rounded once.
__device__ __forceinline__ float force_term(float r, float dmu, float d) {
    constexpr float hi = 1.0f / 3.0f;
    constexpr float lo = (float)(1.0 / 3.0 - (double)hi);
    return rn_fma(d, hi, rn_fma(-r, dmu, rn_mul(d, lo)));
}

// Right-hand sides of a chunk from u at chunk positions -4 .. kC + 3 (first derivative
// alone: -2 .. kC + 1), and the recursions forward from a zero state.
// Explicitly rounded, as everything here: with contraction left to the compiler, the same
// line could have other bits in another kernel.  At 4th order the chunk's two outermost
// right-hand sides have one use each, and go into it as a multiply-add (EDGE; not in
// lines_df.cu).
template <bool SIXTH, bool SECOND, bool EDGE = true, class U>
__device__ __forceinline__ void chunk_forward(U u, const Line32& k, float (&r)[kC],
                                              float (&r2)[kC], float& w1, float& v2, float& w2) {
    auto rhs = [&](float am2, float am1, float ap1, float ap2) {
        float b = rn_mul(rn_sub(ap1, am1), k.c1);
        if (SIXTH) b = rn_fma(rn_sub(ap2, am2), k.c2, b);
        return b;
    };
#pragma unroll
    for (int j = 0; j < kC; ++j) r[j] = rhs(u(j - 2), u(j - 1), u(j + 1), u(j + 2));
    if (SECOND) {
        // the first right-hand side at j - 2, without its factor (4th order)
        auto dif = [&](int j) { return rn_sub(u(j - 1), u(j - 3)); };
        float b[kC + 4];  // the first right-hand side at -2 .. kC + 1
#pragma unroll
        for (int j = 0; j < kC + 4; ++j)
            b[j] = j >= 2 && j < kC + 2 ? r[j - 2] : rhs(u(j - 4), u(j - 3), u(j - 1), u(j));
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            if (SIXTH) r2[j] = rhs(b[j], b[j + 1], b[j + 3], b[j + 4]);
            else if (EDGE && j == 0) r2[j] = rn_mul(rn_fma(-dif(1), k.c1, b[3]), k.c1);
            else if (EDGE && j == kC - 1) r2[j] = rn_mul(rn_fma(dif(kC + 2), k.c1, -b[kC]), k.c1);
            else r2[j] = rn_mul(rn_sub(b[j + 3], b[j + 1]), k.c1);
        }
    }
    w1 = 0.0f;
#pragma unroll
    for (int j = 0; j < kC; ++j) r[j] = w1 = rn_fma(w1, k.nlam, r[j]);
    v2 = w2 = 0.0f;
    if (SECOND) {
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            v2 = rn_fma(v2, k.nlam, r2[j]);
            r2[j] = w2 = rn_fma(w2, k.nlam, v2);
        }
    }
}

// add the state entering the chunk, then the recursions backward from a zero state
template <bool SECOND>
__device__ __forceinline__ void chunk_backward(const Line32& k, float cf, float cv, float cw,
                                               float (&r)[kC], float (&r2)[kC], float& z1,
                                               float& y2, float& z2) {
#pragma unroll
    for (int j = 0; j < kC; ++j) r[j] = rn_fma(cf, k.pw[j], r[j]);
    if (SECOND) {
#pragma unroll
        for (int j = 0; j < kC; ++j)
            r2[j] = rn_fma(k.pw[j], rn_fma((float)(j + 1), cv, cw), r2[j]);
    }
    z1 = 0.0f;
#pragma unroll
    for (int j = kC - 1; j >= 0; --j) r[j] = z1 = rn_fma(z1, k.nlam, r[j]);
    y2 = z2 = 0.0f;
    if (SECOND) {
#pragma unroll
        for (int j = kC - 1; j >= 0; --j) {
            y2 = rn_fma(y2, k.nlam, r2[j]);
            r2[j] = z2 = rn_fma(z2, k.nlam, y2);
        }
    }
}
template <bool SECOND>
__device__ __forceinline__ void chunk_finish(const Line32& k, float cb, float cy, float cz,
                                             float (&r)[kC], float (&r2)[kC]) {
#pragma unroll
    for (int j = 0; j < kC; ++j) r[j] = rn_fma(cb, k.pw[kC - 1 - j], r[j]);
    if (SECOND) {
#pragma unroll
        for (int j = 0; j < kC; ++j)
            r2[j] = rn_fma(k.pw[kC - 1 - j], rn_fma((float)(kC - j), cy, cz), r2[j]);
    }
}

// The state entering a chunk from the end states of the chunks before it (the k-th one
// before: e[-k s]; `have` of them exist): forward with s > 0, backward with s < 0.  x-lines
// pair them first, (e1 + m e2) + m^2 (e3 + m e4); y-lines add them one by one.
template <int AXIS>
__device__ __forceinline__ float join1(const Line32& k, const float* e, int s, int have) {
    if (have < 1) return 0.0f;
    float c = e[-s];
    if (AXIS == 0) {
        if (have >= 2) c = rn_fma(e[-2 * s], k.m1, c);
        if (have >= 3) {
            float d = e[-3 * s];
            if (have >= 4) d = rn_fma(e[-4 * s], k.m1, d);
            c = rn_fma(d, k.m2, c);
        }
    } else {
        if (have >= 2) c = rn_fma(e[-2 * s], k.m1, c);
        if (have >= 3) c = rn_fma(e[-3 * s], k.m2, c);
    }
    return c;
}
template <int AXIS>
__device__ __forceinline__ void join2(const Line32& k, const float* v, const float* w, int s,
                                      int have, float& cv, float& cw) {
    cv = cw = 0.0f;
    if (have < 1) return;
    cv = v[-s];
    cw = w[-s];
    if (have >= 2) {
        cw = rn_fma(k.Cm1, v[-2 * s], rn_fma(k.m1, w[-2 * s], cw));
        cv = rn_fma(k.m1, v[-2 * s], cv);
    }
    if (have >= 3) {
        float dv = v[-3 * s], dw = w[-3 * s];
        if (AXIS == 0 && have >= 4) {
            dw = rn_fma(k.Cm1, v[-4 * s], rn_fma(k.m1, w[-4 * s], dw));
            dv = rn_fma(k.m1, v[-4 * s], dv);
        }
        cw = rn_fma(k.Cm2, dv, rn_fma(k.m2, dw, cw));
        cv = rn_fma(k.m2, dv, cv);
    }
}

// Shared memory of a block of T threads: six join arrays of T floats, then (x-lines) one or
// two planes of [lines][LW].
__host__ __device__ constexpr int line_stride(int nch) { return kC * nch + 32; }

// One block: window `bid / ngroups` of line group `bid % ngroups`.  Every thread of the block
// calls it; threads beyond the block's (line, chunk) pairs only keep the barriers.
template <int MODE, bool SIXTH, int AXIS>
__device__ __forceinline__ void block(const Dir32& d, const Line32& k, int bid, float* sh) {
    constexpr bool SECOND = MODE == RHO;
    const Geo32& g = d.g;
    const int T = blockDim.x, t = threadIdx.x;
    const int grp = bid % g.ngroups, win = bid / g.ngroups;
    const int s0 = win * g.own, nown = min(g.own, g.n - s0);
    const int nch = g.nch, H = g.H;
    const int ln = AXIS == 0 ? t / nch : t & (g.nl - 1);
    const int c = AXIS == 0 ? t - ln * nch : t / g.nl;
    const int line = grp * g.nl + ln;
    const bool mine = ln < g.nl && c < nch, live = mine && line < g.nlines;
    // end states of the chunks: forward, forward double (v, w), backward likewise
    float *ea = sh + t, *ev = ea + T, *ew = ev + T, *za = ew + T, *zv = za + T, *zw = zv + T;
    const int js = AXIS == 0 ? 1 : g.nl;  // from a chunk's state to the next one's
    // position of the period: p in [0, period + window)
    auto wrap = [&](int p) {
        if (g.magic) p -= g.period * (int)__umulhi((unsigned)p, g.magic);
        else if (p >= g.period) p -= g.period;
        return p;
    };
    const int p0 = wrap(s0 - H - 4 + g.lift);  // period position of window position -4

    float r[kC], r2[kC];
    float w1, v2, w2;
    if constexpr (AXIS == 0) {
        const int LW = line_stride(nch);
        float* plane = sh + 6 * T;
        float* row = plane + ln * LW;                 // staged: window position q at row[q + 4]
        const size_t lo = (size_t)line * g.ls;
        const int nq = kC * nch + 8;
        if (live) {
            if (g.vec) {
                for (int q = 4 * c; q < nq; q += 4 * nch)
                    cp16(row + q, d.u + lo + (size_t)wrap(p0 + q));
            } else {
                for (int q = c; q < nq; q += nch) cp4(row + q, d.u + lo + (size_t)wrap(p0 + q));
            }
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
        if (live) {
            const float* u0 = row + 4 + c * kC;
            chunk_forward<SIXTH, SECOND>([&](int j) { return u0[j]; }, k, r, r2, w1, v2, w2);
        }
    } else {
        if (live) {
            constexpr int M = SECOND ? 4 : 2;  // rows read before and after the chunk
            float u[kC + 2 * M];
            int p = wrap(p0 + 4 + c * kC - M);
#pragma unroll
            for (int j = 0; j < kC + 2 * M; ++j) {
                const int y = g.mirror && p >= g.n ? 2 * g.n - 1 - p : p;
                u[j] = d.u[(size_t)line + (size_t)y * g.ps];
                p = p + 1 == g.period ? 0 : p + 1;
            }
            chunk_forward<SIXTH, SECOND>([&](int j) { return u[j + M]; }, k, r, r2, w1, v2, w2);
        }
    }
    if (live) {
        *ea = w1;
        if (SECOND) {
            *ev = v2;
            *ew = w2;
        }
    }
    __syncthreads();  // also: every staged value has been read
    float z1, y2, z2;
    if (live) {
        const float cf = join1<AXIS>(k, ea, js, c);
        float cv = 0.0f, cw = 0.0f;
        if (SECOND) join2<AXIS>(k, ev, ew, js, c, cv, cw);
        chunk_backward<SECOND>(k, cf, cv, cw, r, r2, z1, y2, z2);
        *za = z1;
        if (SECOND) {
            *zv = y2;
            *zw = z2;
        }
    }
    __syncthreads();
    if (live) {
        const int after = nch - 1 - c;
        const float cb = join1<AXIS>(k, za, -js, after);
        float cy = 0.0f, cz = 0.0f;
        if (SECOND) join2<AXIS>(k, zv, zw, -js, after, cy, cz);
        chunk_finish<SECOND>(k, cb, cy, cz, r, r2);
    }
    if constexpr (AXIS == 0) {
        const int LW = line_stride(nch);
        float* row = sh + 6 * T + ln * LW;
        float* row2 = row + (size_t)g.nl * LW;
        if (live) {
#pragma unroll
            for (int j = 0; j < kC; ++j) {
                row[c * kC + j] = r[j];
                if (SECOND) row2[c * kC + j] = r2[j];
            }
        }
        __syncthreads();
        if (live) {
            const size_t lo = (size_t)line * g.ls + (size_t)s0;
            if (g.vec) {
                for (int q = 4 * c; q < nown; q += 4 * nch) {
                    const float4 a = *reinterpret_cast<const float4*>(row + H + q);
                    if constexpr (SECOND) {
                        *reinterpret_cast<float4*>(d.o1 + lo + q) = a;
                        *reinterpret_cast<float4*>(d.o2 + lo + q) =
                            *reinterpret_cast<const float4*>(row2 + H + q);
                    } else {
                        const float4 p = *reinterpret_cast<const float4*>(d.rho + lo + q);
                        const float4 e = *reinterpret_cast<const float4*>(d.dr + lo + q);
                        *reinterpret_cast<float4*>(d.o1 + lo + q) =
                            make_float4(force_term(p.x, a.x, e.x), force_term(p.y, a.y, e.y),
                                        force_term(p.z, a.z, e.z), force_term(p.w, a.w, e.w));
                    }
                }
            } else {
                for (int q = c; q < nown; q += nch) {
                    if constexpr (SECOND) {
                        d.o1[lo + q] = row[H + q];
                        d.o2[lo + q] = row2[H + q];
                    } else {
                        d.o1[lo + q] = force_term(d.rho[lo + q], row[H + q], d.dr[lo + q]);
                    }
                }
            }
        }
    } else if (live) {
        const int q0 = c * kC - H;  // owned index of the chunk's first position
        const size_t o0 = (size_t)line + (size_t)(s0 + q0) * g.ps;
        if constexpr (SECOND) {
#pragma unroll
            for (int j = 0; j < kC; ++j)
                if ((unsigned)(q0 + j) < (unsigned)nown) {
                    d.o1[o0 + (size_t)j * g.ps] = r[j];
                    d.o2[o0 + (size_t)j * g.ps] = r2[j];
                }
        } else {
            constexpr int kB = 5;  // operands fetched before any of them is used
#pragma unroll
            for (int b = 0; b < kC; b += kB) {
                float p[kB], e[kB];
#pragma unroll
                for (int j = 0; j < kB; ++j)
                    if (b + j < kC && (unsigned)(q0 + b + j) < (unsigned)nown) {
                        p[j] = d.rho[o0 + (size_t)(b + j) * g.ps];
                        e[j] = d.dr[o0 + (size_t)(b + j) * g.ps];
                    }
#pragma unroll
                for (int j = 0; j < kB; ++j)
                    if (b + j < kC && (unsigned)(q0 + b + j) < (unsigned)nown)
                        d.o1[o0 + (size_t)(b + j) * g.ps] = force_term(p[j], r[b + j], e[j]);
            }
        }
    }
}

}  // namespace l32
}  // namespace cplbm
