// lines_df.cu -- line solves of the density in double-float (df.cuh): first derivatives in
// double-float wherever a window crosses an interface, second derivatives in FP32 (see
// kernels_mixed.cu for why), for the mixed path above a density ratio of 1e4 and the
// stand-alone lbm_cfd_df.
//
// Windows, chunks and joins are those of lines32.cuh, with a halo of 40 (6th order) so that
// the double-float recursions are cut at 1e-15.  A block takes groups of eight lines; a
// group whose staged densities all lie within a factor 32 is solved in FP32 on the hi part
// (FP32 rounding then stays below ~2e-6 of the local values, as accurate as the FP32 result
// that is stored).  Both axes are staged by 16-byte copies, x-lines line by line, y-lines
// row by row ([slot][lines]).
//
// A chunk is in registers from its right-hand side to its result, unrolled over its 19
// positions, 128 registers and two blocks an SM.  In launches of many blocks (kManyBlocks) the
// double-float chunks stay in shared memory, in place of the staged window, as loops: 80
// registers and three blocks, for the groups solved in FP32, which are most of a large grid.
// With those as loops too, density lines of 1000^2 at ratio 8e4 took 25.2 us and a step 47.2;
// so it is 44.6.  (The chunk in registers within one kernel templated over all number types:
// 33.4 and 54.4.)
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <type_traits>

#include "df.cuh"
#include "lines32.cuh"

namespace cplbm {
namespace {

constexpr int kC = kC32, kT = 256, kGroup = 8;
constexpr double kEpsDF = 1e-15, kEpsF = 1e-8;

struct LineDF {
    Line32 f;
    df c1, c2, nlam, pw[kC], m1, m2;
};

__device__ __forceinline__ df fma_df(df x, df c, df y) { return df_fma(x, c.hi, c.lo, y); }

// join1<0> in double-float: forward s > 0, backward s < 0, `have` chunks on that side
__device__ __forceinline__ df join_df(const LineDF& k, const float* h, const float* l, int s,
                                      int have) {
    auto at = [&](int i) { return df{h[-i * s], l[-i * s]}; };
    if (have < 1) return df{0.0f, 0.0f};
    df c = at(1);
    if (have >= 2) c = fma_df(at(2), k.m1, c);
    if (have >= 3) {
        df d = at(3);
        if (have >= 4) d = fma_df(at(4), k.m1, d);
        c = fma_df(d, k.m2, c);
    }
    return c;
}

// Shared memory: eight join arrays of kT floats, the two planes of the staged window (hi, lo),
// whose places the first derivative takes, and the second derivative's plane.
// LOOPS: double-float chunks are loops in shared memory (see kManyBlocks).
template <bool SIXTH, bool SECOND, bool LOOPS>
__device__ __forceinline__ void block_df(const Dir32& d, const LineDF& k, int axis, int bid,
                                         float* sh) {
    const Geo32& g = d.g;
    const int t = threadIdx.x;
    const int grp = bid % g.ngroups, win = bid / g.ngroups;
    const int s0 = win * g.own, nown = min(g.own, g.n - s0);
    const int nch = g.nch, nl = g.nl;
    const int ln = axis == 0 ? t / nch : t % nl;
    const int c = axis == 0 ? t - ln * nch : t / nl;
    const int line = grp * nl + ln;
    const bool live = ln < nl && c < nch && line < g.nlines;
    const int js = axis == 0 ? 1 : nl;
    // end states: first derivative (hi, lo) and second (v, w), forward and backward
    float *eh = sh + t, *el = eh + kT, *ev = el + kT, *ew = ev + kT;
    float *zh = ew + kT, *zl = zh + kT, *zv = zl + kT, *zw = zv + kT;
    const int LW = l32::line_stride(nch), nq = kC * nch + 8;
    float* hi = sh + 8 * kT;
    float* lo = hi + nl * LW;
    float* p2 = lo + nl * LW;
    __shared__ int lowest[kT / 8 / kGroup], highest[kT / 8 / kGroup];
    if (t < kT / 8 / kGroup) {
        lowest[t] = __float_as_int(FLT_MAX);
        highest[t] = 0;
    }
    auto wrap = [&](int p) {
        if (g.magic) p -= g.period * (int)__umulhi((unsigned)p, g.magic);
        else if (p >= g.period) p -= g.period;
        return g.period == 1 ? 0 : p;
    };
    const int p0 = wrap(s0 - g.H - 4 + g.lift);
    // ---- stage ----
    if (axis == 0) {
        if (live) {
            const size_t base = (size_t)line * g.ls;
            const int w = g.vec ? 4 : 1;
            for (int q = w * c; q < nq; q += w * nch) {
                const size_t o = base + (size_t)wrap(p0 + q);
                if (g.vec) {
                    l32::cp16(hi + ln * LW + q, d.u + o);
                    l32::cp16(lo + ln * LW + q, d.ul + o);
                } else {
                    l32::cp4(hi + ln * LW + q, d.u + o);
                    l32::cp4(lo + ln * LW + q, d.ul + o);
                }
            }
        }
    } else {
        // pieces of four columns (one where rows are not whole 16-byte pieces)
        const int w = g.vec ? 4 : 1, pr = nl / w;
        for (int i = t; i < nq * pr; i += kT) {
            const int q = i / pr, x = w * (i - q * pr), col = grp * nl + x;
            if (col >= g.nlines) continue;  // (whole pieces: nlines is a multiple of w)
            int p = wrap(p0 + q);
            if (g.mirror && p >= g.n) p = 2 * g.n - 1 - p;
            const size_t o = (size_t)p * g.ps + (size_t)col;
            if (g.vec) {
                l32::cp16(hi + q * nl + x, d.u + o);
                l32::cp16(lo + q * nl + x, d.ul + o);
            } else {
                l32::cp4(hi + q * nl + x, d.u + o);
                l32::cp4(lo + q * nl + x, d.ul + o);
            }
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    // chunk position j at base + j ps
    const int ps = axis == 0 ? 1 : nl;
    const int base = axis == 0 ? ln * LW + c * kC + 4 : (c * kC + 4) * nl + ln;
    float *uh = hi + base, *ul = lo + base, *q2 = p2 + base;
    // ---- which groups need double-float ----
    if (live) {
        float mn = FLT_MAX, mx = 0.0f;
#pragma unroll 9
        for (int j = -4; j < kC + 4; ++j) {
            mn = fminf(mn, uh[j * ps]);
            mx = fmaxf(mx, uh[j * ps]);
        }
        // non-negative floats order as integers
        atomicMin(&lowest[ln / kGroup], __float_as_int(fmaxf(mn, 0.0f)));
        atomicMax(&highest[ln / kGroup], __float_as_int(mx));
    }
    __syncthreads();
    bool wide = true;
    if (live) {
        const float mn = __int_as_float(lowest[ln / kGroup]),
                    mx = __int_as_float(highest[ln / kGroup]);
        // (a group cut short by the grid's edge is always solved in double-float)
        const bool whole = (line / kGroup + 1) * kGroup <= g.nlines;
        wide = !(whole && mn > 0.0f && mx <= 32.0f * mn);
    }
    auto U = [&](int j) { return df{uh[j * ps], ul[j * ps]}; };
    auto rhs = [&](df am2, df am1, df ap1, df ap2) {
        df b = df_mul(df_sub(ap1, am1), k.c1.hi, k.c1.lo);
        if (SIXTH) b = fma_df(df_sub(ap2, am2), k.c2, b);
        return b;
    };
    auto rhs_f = [&](float am2, float am1, float ap1, float ap2) {
        float b = (ap1 - am1) * k.f.c1;
        if (SIXTH) b = rn_fma(ap2 - am2, k.f.c2, b);
        return b;
    };
    auto at_f = [&](int j) {
        return rhs_f(uh[(j - 2) * ps], uh[(j - 1) * ps], uh[(j + 1) * ps], uh[(j + 2) * ps]);
    };
    // What the chunk needs of its neighbours, before they overwrite it: the window two
    // positions either side, and the first right-hand side there (FP32), in r; or the chunk
    // itself.
    float r[kC], r2[kC], rl[LOOPS ? 1 : kC];
    if (live && !wide) {
        float w1, v2, w2;
        l32::chunk_forward<SIXTH, SECOND, false>([&](int j) { return uh[j * ps]; }, k.f, r, r2, w1,
                                                 v2, w2);
        *eh = w1;
        if (SECOND) {
            *ev = v2;
            *ew = w2;
        }
    } else if (live) {
        if constexpr (!LOOPS) {
            df w{0.0f, 0.0f};
            float b[kC + 4];  // the right-hand side's hi part at -2 .. kC + 1
#pragma unroll
            for (int j = 0; j < kC; ++j) {
                const df h = rhs(U(j - 2), U(j - 1), U(j + 1), U(j + 2));
                b[j + 2] = h.hi;
                w = fma_df(w, k.nlam, h);
                r[j] = w.hi;
                rl[j] = w.lo;
            }
            *eh = w.hi;
            *el = w.lo;
            if (SECOND) {
                b[0] = at_f(-2);
                b[1] = at_f(-1);
                b[kC + 2] = at_f(kC);
                b[kC + 3] = at_f(kC + 1);
                float v = 0.0f, w2 = 0.0f;
#pragma unroll
                for (int j = 0; j < kC; ++j) {
                    float y = rn_mul(rn_sub(b[j + 3], b[j + 1]), k.f.c1);
                    if (SIXTH) y = rn_fma(rn_sub(b[j + 4], b[j]), k.f.c2, y);
                    v = rn_fma(v, k.f.nlam, y);
                    r2[j] = w2 = rn_fma(w2, k.f.nlam, v);
                }
                *ev = v;
                *ew = w2;
            }
        } else {
            auto keep = [&](int i, df x) {
                r[i] = x.hi;
                r[i + 1] = x.lo;
            };
            keep(0, U(-2));
            keep(2, U(-1));
            keep(4, U(kC));
            keep(6, U(kC + 1));
            if (SECOND) {
                r[8] = at_f(-2);
                r[9] = at_f(-1);
                r[10] = at_f(kC);
                r[11] = at_f(kC + 1);
            }
        }
    }
    const int after = nch - 1 - c;
    // ---- forward, in place of the staged window ----
    if constexpr (LOOPS) {
        __syncthreads();
        if (live && wide) {
            df a{r[0], r[1]}, b{r[2], r[3]}, e = U(0), f = U(1), w{0.0f, 0.0f};
            float *ph = uh, *pl = ul, *p = q2;  // at position j
            auto step = [&](df h) {
                const df x = rhs(a, b, f, h);
                w = fma_df(w, k.nlam, x);
                *p = x.hi;
                *ph = w.hi;
                *pl = w.lo;
                p += ps;
                ph += ps;
                pl += ps;
                a = b;
                b = e;
                e = f;
                f = h;
            };
#pragma unroll 4
            for (int j = 0; j < kC - 3; ++j) step(df{ph[2 * ps], pl[2 * ps]});
            step(df{ph[2 * ps], pl[2 * ps]});
            step(df{r[4], r[5]});
            step(df{r[6], r[7]});
            *eh = w.hi;
            *el = w.lo;
            if (SECOND) {
                float p = r[8], q = r[9], u = q2[0], x = q2[ps], v = 0.0f, w = 0.0f;
                float* o = q2;
                auto step = [&](float h) {
                    float y = rn_mul(rn_sub(x, q), k.f.c1);
                    if (SIXTH) y = rn_fma(rn_sub(h, p), k.f.c2, y);
                    v = rn_fma(v, k.f.nlam, y);
                    *o = w = rn_fma(w, k.f.nlam, v);
                    o += ps;
                    p = q;
                    q = u;
                    u = x;
                    x = h;
                };
#pragma unroll 8
                for (int j = 0; j < kC - 3; ++j) step(o[2 * ps]);
                step(o[2 * ps]);
                step(r[10]);
                step(r[11]);
                *ev = v;
                *ew = w;
            }
        }
    }
    __syncthreads();
    // ---- backward ----
    if (live && !wide) {
        const float cf = l32::join1<0>(k.f, eh, js, c);
        float cv = 0.0f, cw = 0.0f, y, z;
        if (SECOND) l32::join2<0>(k.f, ev, ew, js, c, cv, cw);
        l32::chunk_backward<SECOND>(k.f, cf, cv, cw, r, r2, *zh, y, z);
        if (SECOND) {
            *zv = y;
            *zw = z;
        }
    } else if (live) {
        const df cf = join_df(k, eh, el, js, c);
        df z{0.0f, 0.0f};
        if constexpr (!LOOPS) {
#pragma unroll
            for (int j = kC - 1; j >= 0; --j) {
                z = fma_df(z, k.nlam, fma_df(cf, k.pw[j], df{r[j], rl[j]}));
                r[j] = z.hi;
                rl[j] = z.lo;
            }
        } else {
            float *ph = uh + (kC - 1) * ps, *pl = ul + (kC - 1) * ps;
#pragma unroll 4
            for (int j = kC - 1; j >= 0; --j) {
                z = fma_df(z, k.nlam, fma_df(cf, k.pw[j], df{*ph, *pl}));
                *ph = z.hi;
                *pl = z.lo;
                ph -= ps;
                pl -= ps;
            }
        }
        *zh = z.hi;
        *zl = z.lo;
        if (SECOND) {
            float cv, cw, y = 0.0f, x = 0.0f;
            l32::join2<0>(k.f, ev, ew, js, c, cv, cw);
            auto step = [&](int j, float& v) {
                y = rn_fma(y, k.f.nlam, rn_fma(k.f.pw[j], rn_fma((float)(j + 1), cv, cw), v));
                v = x = rn_fma(x, k.f.nlam, y);
            };
            if constexpr (!LOOPS) {
#pragma unroll
                for (int j = kC - 1; j >= 0; --j) step(j, r2[j]);
            } else {
#pragma unroll 5
                for (int j = kC - 1; j >= 0; --j) step(j, q2[j * ps]);
            }
            *zv = y;
            *zw = x;
        }
    }
    __syncthreads();
    // ---- the state entering from after the chunk ----
    if (live && !wide) {
        const float cb = l32::join1<0>(k.f, zh, -js, after);
        float cy = 0.0f, cz = 0.0f;
        if (SECOND) l32::join2<0>(k.f, zv, zw, -js, after, cy, cz);
        l32::chunk_finish<SECOND>(k.f, cb, cy, cz, r, r2);
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            uh[j * ps] = r[j];
            if (SECOND) q2[j * ps] = r2[j];
        }
    } else if (live) {
        const df cb = join_df(k, zh, zl, -js, after);
        float cy = 0.0f, cz = 0.0f;
        if (SECOND) l32::join2<0>(k.f, zv, zw, -js, after, cy, cz);
        auto second = [&](int j, float v) {
            return rn_fma(k.f.pw[kC - 1 - j], rn_fma((float)(kC - j), cy, cz), v);
        };
        if constexpr (!LOOPS) {
#pragma unroll
            for (int j = 0; j < kC; ++j) {
                uh[j * ps] = df_round(fma_df(cb, k.pw[kC - 1 - j], df{r[j], rl[j]}));
                if (SECOND) q2[j * ps] = second(j, r2[j]);
            }
        } else {
            float *ph = uh, *pl = ul;
#pragma unroll 4
            for (int j = 0; j < kC; ++j) {
                *ph = df_round(fma_df(cb, k.pw[kC - 1 - j], df{*ph, *pl}));
                ph += ps;
                pl += ps;
            }
            if (SECOND) {
#pragma unroll 5
                for (int j = 0; j < kC; ++j) q2[j * ps] = second(j, q2[j * ps]);
            }
        }
    }
    __syncthreads();
    // ---- out: window position q at slot q + 4 ----
    const int H4 = g.H + 4;
    if (axis == 0) {
        if (live) {
            const size_t o = (size_t)line * g.ls + (size_t)s0;
            const float *r1 = hi + ln * LW + H4, *r2 = p2 + ln * LW + H4;
            if (g.vec) {
                for (int q = 4 * c; q < nown; q += 4 * nch) {
                    *reinterpret_cast<float4*>(d.o1 + o + q) =
                        *reinterpret_cast<const float4*>(r1 + q);
                    if (SECOND)
                        *reinterpret_cast<float4*>(d.o2 + o + q) =
                            *reinterpret_cast<const float4*>(r2 + q);
                }
            } else {
                for (int q = c; q < nown; q += nch) {
                    d.o1[o + q] = r1[q];
                    if (SECOND) d.o2[o + q] = r2[q];
                }
            }
        }
    } else {
        const int w = g.vec ? 4 : 1, pr = nl / w;
        for (int i = t; i < nown * pr; i += kT) {
            const int q = i / pr, x = w * (i - q * pr), col = grp * nl + x;
            if (col >= g.nlines) continue;
            const size_t o = (size_t)(s0 + q) * g.ps + (size_t)col;
            const int m = (q + H4) * nl + x;
            if (g.vec) {
                *reinterpret_cast<float4*>(d.o1 + o) = *reinterpret_cast<const float4*>(hi + m);
                if (SECOND)
                    *reinterpret_cast<float4*>(d.o2 + o) = *reinterpret_cast<const float4*>(p2 + m);
            } else {
                d.o1[o] = hi[m];
                if (SECOND) d.o2[o] = p2[m];
            }
        }
    }
}

template <bool SIXTH, bool SECOND, bool LOOPS>
__global__ void __launch_bounds__(kT, LOOPS ? 3 : 2)
    k_lines_df(Dir32 x, Dir32 y, const __grid_constant__ LineDF k, DevState* st, int bump,
               int nbx) {
    pdl_prologue();
    extern __shared__ __align__(16) float shdf[];
    if (bump && blockIdx.x == 0 && threadIdx.x == 0) st->t += 1;
    const int nby = (int)gridDim.x - nbx, b = blockIdx.x;
    const bool is_y = b < nby;
    const Dir32& d = is_y ? y : x;
    block_df<SIXTH, SECOND, LOOPS>(d, k, is_y, is_y ? b : b - nby, shdf);
}

template <bool SIXTH, bool LOOPS>
__global__ void __launch_bounds__(kT, LOOPS ? 3 : 2)
    k_lines_df_batch(const Lines32Inst* __restrict__ d, const int* __restrict__ map,
                     const __grid_constant__ LineDF k, int bump) {
    extern __shared__ __align__(16) float shdf[];
    const Lines32Inst& D = d[map[blockIdx.x]];
    const int local = (int)blockIdx.x - D.blk0;
    if (bump && local == 0 && threadIdx.x == 0) D.st->t += 1;
    const bool is_y = local >= D.nbx;
    block_df<SIXTH, true, LOOPS>(is_y ? D.y : D.x, k, is_y, is_y ? local - D.nbx : local, shdf);
}

// ---- host side ----
df split(double v) {
    df r;
    r.hi = (float)v;
    r.lo = (float)(v - (double)r.hi);
    return r;
}
LineDF constants_df(int order) {
    const double alpha = order == 6 ? 1.0 / 3.0 : 0.25;
    const double lam = (1.0 - std::sqrt(1.0 - 4.0 * alpha * alpha)) / (2.0 * alpha);
    const double a = 2.0 / 3.0 * (alpha + 2.0), b = (4.0 * alpha - 1.0) / 3.0;  // Eq. 38
    LineDF k;
    k.f = line32_constants(order);
    k.c1 = split(lam / alpha * a / 2.0);
    k.c2 = split(lam / alpha * b / 4.0);
    k.nlam = split(-lam);
    double p = 1.0;
    for (int j = 0; j < kC; ++j) k.pw[j] = split(p *= -lam);
    const double m = std::pow(-lam, kC);
    k.m1 = split(m);
    k.m2 = split(m * m);
    return k;
}

// Lines a block: groups of eight, as many as the block's threads hold.
void divide_df(Geo32& g) {
    g.nl = std::max(kGroup, kT / g.nch / kGroup * kGroup);
    g.ngroups = (g.nlines + g.nl - 1) / g.nl;
}
Dir32 dir_df(const float* h, const float* l, float* d1, float* d2, int nx, int ny, int axis,
             int order, bool second, bool walls_y) {
    Dir32 d{};
    d.u = h;
    d.ul = l;
    d.o1 = d1;
    d.o2 = d2;
    d.g = line32_geometry(nx, ny, axis, order, kEpsDF, second ? kEpsF : 0.0, walls_y);
    // 16-byte pieces want 16-byte pointers as well as whole pieces a row: lbm_cfd_df takes any
    // that hold floats.  (The fields of contexts and batches are 256-byte aligned.)
    for (const float* p : {h, l, (const float*)d1, (const float*)d2})
        if ((uintptr_t)p % 16 != 0) d.g.vec = 0;
    divide_df(d.g);
    return d;
}
int blocks_of(const Geo32& g) { return g.ngroups * g.nwin; }
size_t smem_df(const Geo32& g) {
    return ((size_t)8 * kT + 3 * (size_t)g.nl * l32::line_stride(g.nch)) * sizeof(float);
}
// the most that a block stages, of any grid
size_t most_smem_df() {
    size_t most = 0;
    for (int nch = 8; nch <= 32; nch += 4) {
        Geo32 g{};
        g.nch = nch;
        divide_df(g);
        most = std::max(most, smem_df(g));
    }
    return most;
}
// Steps at ratio 8e4 with double-float chunks in registers and as loops: 512^2 20.4 and 22.5
// us, 1000^2 44.6 and 47.0, 1500^2 91.7 and 94.2, a batch of 4 x 1024^2 (2048 blocks) 177.6 and
// 185.1, 2 x 2048^2 (4096) 335.5 and 335.0, 4096^2 (8192) 553.9 and 537.6.
constexpr int kManyBlocks = 15 * 2 * 152;
cudaError_t run_df(const Dir32& x, const Dir32& y, int nbx, int nby, int order, DevState* st,
                   int bump, cudaStream_t s) {
    const size_t smem = std::max(smem_df(x.g), smem_df(y.g));
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, most_smem_df());
        if (e != cudaSuccess) return e;
        return launch_pdl(kern, dim3(nbx + nby), dim3(kT), smem, s, x, y, constants_df(order), st,
                          bump, nbx);
    };
    const bool loops = nbx + nby > kManyBlocks;
    auto pick = [&](auto sixth, auto second) {
        constexpr bool S = decltype(sixth)::value, D = decltype(second)::value;
        return loops ? go(k_lines_df<S, D, true>) : go(k_lines_df<S, D, false>);
    };
    using T = std::true_type;
    using F = std::false_type;
    if (x.o2) return order == 6 ? pick(T(), T()) : pick(F(), T());
    return order == 6 ? pick(T(), F()) : pick(F(), F());
}

}  // namespace

cudaError_t lines_df_rho(const float* rh, const float* rl, float* dxr, float* dxx, float* dyr,
                         float* dyy, int nx, int ny, int order, DevState* st, int bump,
                         cudaStream_t s, bool walls_y) {
    const Dir32 x = dir_df(rh, rl, dxr, dxx, nx, ny, 0, order, true, false),
                y = dir_df(rh, rl, dyr, dyy, nx, ny, 1, order, true, walls_y);
    return run_df(x, y, blocks_of(x.g), blocks_of(y.g), order, st, bump, s);
}

cudaError_t lines_df_plain(const float* uh, const float* ul, float* d1, float* d2, int nx, int ny,
                           int axis, int order, cudaStream_t s) {
    const Dir32 d = dir_df(uh, ul, d1, d2, nx, ny, axis, order, d2 != nullptr, false);
    const int nb = blocks_of(d.g);
    return run_df(d, d, axis == 0 ? nb : 0, axis == 0 ? 0 : nb, order, nullptr, 0, s);
}

int lines_df_batch_blocks(int nx, int ny, int order) {
    return blocks_of(dir_df(nullptr, nullptr, nullptr, nullptr, nx, ny, 0, order, true, false).g) +
           blocks_of(dir_df(nullptr, nullptr, nullptr, nullptr, nx, ny, 1, order, true, false).g);
}

Lines32Inst lines_df_batch_inst(const MixedLinesView& v, int order, int blk0) {
    Lines32Inst d{};
    d.x = dir_df(v.rh, v.rl, v.dxr, v.dxx, v.nx, v.ny, 0, order, true, false);
    d.y = dir_df(v.rh, v.rl, v.dyr, v.dyy, v.nx, v.ny, 1, order, true, false);
    d.nbx = blocks_of(d.x.g);
    d.blk0 = blk0;
    d.st = v.st;
    return d;
}

size_t lines_df_batch_smem(const Lines32Inst& d) {
    return std::max(smem_df(d.x.g), smem_df(d.y.g));
}

cudaError_t lines_df_batch_launch(const Lines32Inst* d, const int* map, int nblocks, int order,
                                  size_t smem, bool beside, int bump, cudaStream_t s) {
    if (nblocks <= 0) return cudaSuccess;
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, most_smem_df());
        if (e != cudaSuccess) return e;
        kern<<<nblocks, kT, smem, s>>>(d, map, constants_df(order), bump);
        return cudaGetLastError();
    };
    // (beside the FP32 lines of other members the registers are shared: 24 members, 232 of the
    // blocks these, 83.0 us a step in registers and 81.3 as loops; 17 members, 34 of the blocks,
    // 35.7 and 37.5; 8, 164, 36.6 and 39.1)
    constexpr int kManyBeside = 200;
    if (nblocks > (beside ? kManyBeside : kManyBlocks))
        return order == 6 ? go(k_lines_df_batch<true, true>) : go(k_lines_df_batch<false, true>);
    return order == 6 ? go(k_lines_df_batch<true, false>) : go(k_lines_df_batch<false, false>);
}

}  // namespace cplbm
