// lines32_wide.cu -- FP32 line solves (Eqs. 37-39) of large grids, with the fused force
// (Eq. 12) epilogue: full windows of 32 chunks, NL lines (NL warps) a block.  Windows,
// chunks, joins and rounding are those of lines32.cuh, so both give the same bits; on grids
// above kLines32Nodes these are faster (1024^2 33.9 us a step against 36.6, 4096^2 454
// against 487), and in batches by the rule in capi_batch.cu.
//
//   x-lines  warp w owns line w and lane l chunk l, staged in 16-byte pieces line by line;
//            chunk states are joined by warp shuffles.
//   y-lines  staged row by row ([slot][NL columns]): an interior window arrives by tensor
//            copies of NL columns x kBoxRows rows, issued by one thread and completed on one
//            mbarrier; wrapping or mirrored ones by 16-byte pieces.  Lane l of warp w owns
//            chunk (32 / NL) w + l / NL of column l mod NL, so a warp reads whole rows in 32
//            distinct banks; chunk states are joined through shared memory.
// Results take the staged rows' places and go out in 16-byte pieces.
#include <cuda.h>  // CUtensorMap and its encoder's types (the encoder is fetched at run time)

#include <cstring>
#include <mutex>
#include <type_traits>

#include "lines32.cuh"

namespace cplbm {
namespace {

using l32::kC;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kW = 32 * kC, kLWin = kW + 8;  // window, and staged slots (4 more each side)
constexpr int kLW = 644;  // stride of a staged x-line: 16-byte aligned, odd number of banks x 4
static_assert(kLW >= kLWin && kLW % 4 == 0, "strides");
constexpr int kBoxRows = 88;
static_assert(kLWin % kBoxRows == 0, "y windows split into whole tensor-copy boxes");
constexpr unsigned kWaitSpins = 1u << 22;  // ~ tens of milliseconds of polling

// ---- tensor copies ----
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

// x-lines: joins by shuffles, the pairs of l32::join1<0> and join2<0> (DIR 1: forward, from
// the lanes before; -1: backward)
template <int DIR>
__device__ __forceinline__ float lane_at(float v, int o) {
    return DIR > 0 ? __shfl_up_sync(kFull, v, o) : __shfl_down_sync(kFull, v, o);
}
template <int DIR>
__device__ __forceinline__ float shuffle_join1(const Line32& k, float e, int have) {
    float t = lane_at<DIR>(e, 1);
    if (have >= 1) e = rn_fma(t, k.m1, e);
    t = lane_at<DIR>(e, 2);
    if (have >= 2) e = rn_fma(t, k.m2, e);
    t = lane_at<DIR>(e, 1);
    return have >= 1 ? t : 0.0f;
}
template <int DIR>
__device__ __forceinline__ void shuffle_join2(const Line32& k, float v, float w, int have,
                                              float& cv, float& cw) {
    float tv = lane_at<DIR>(v, 1), tw = lane_at<DIR>(w, 1);
    if (have >= 1) {
        w = rn_fma(k.Cm1, tv, rn_fma(k.m1, tw, w));
        v = rn_fma(k.m1, tv, v);
    }
    tv = lane_at<DIR>(v, 2);
    tw = lane_at<DIR>(w, 2);
    if (have >= 2) {
        w = rn_fma(k.Cm2, tv, rn_fma(k.m2, tw, w));
        v = rn_fma(k.m2, tv, v);
    }
    cv = lane_at<DIR>(v, 1);
    cw = lane_at<DIR>(w, 1);
    if (have < 1) cv = cw = 0.0f;
}

__device__ __forceinline__ float4 force4(float4 p, float4 a, float4 e) {
    return make_float4(l32::force_term(p.x, a.x, e.x), l32::force_term(p.y, a.y, e.y),
                       l32::force_term(p.z, a.z, e.z), l32::force_term(p.w, a.w, e.w));
}
__device__ __forceinline__ float force4(float p, float a, float e) {
    return l32::force_term(p, a, e);
}

// The owned positions of a solved window in pieces of W floats: a warp walks its x-line, the
// block walks rows of y-lines.  Operands are fetched in groups of kB before any result of
// the group is written.
template <int AXIS, bool SECOND, int NL, int W>
__device__ __forceinline__ void write_out(const Dir32& d, const float* plane, const float* plane2,
                                          int line0, int s0, int nown) {
    using V = typename std::conditional<W == 4, float4, float>::type;
    const Geo32& g = d.g;
    constexpr int kB = 4, PR = NL / W;  // pieces of a row
    const int t = threadIdx.x;
    const int first = AXIS == 0 ? W * (t & 31) : t, step = AXIS == 0 ? 32 * W : 32 * NL;
    const int count = AXIS == 0 ? nown : PR * nown;
    if (AXIS == 0 && line0 + (t >> 5) >= g.nlines) return;
    auto ok = [&](int i) { return i < count && (AXIS == 0 || line0 + W * (i % PR) < g.nlines); };
    auto field = [&](int i) {
        return AXIS == 0 ? (size_t)(line0 + (t >> 5)) * g.ls + (size_t)(s0 + i)
                         : (size_t)(line0 + W * (i % PR)) + (size_t)(s0 + i / PR) * g.ps;
    };
    auto slot = [&](int i) {
        return AXIS == 0 ? (t >> 5) * kLW + g.H + i : (g.H + i / PR) * NL + W * (i % PR);
    };
    auto at = [](const float* p) { return *reinterpret_cast<const V*>(p); };
    for (int i0 = first; i0 < count; i0 += kB * step) {
        if constexpr (SECOND) {
#pragma unroll
            for (int b = 0; b < kB; ++b) {
                const int i = i0 + b * step;
                if (!ok(i)) continue;
                *reinterpret_cast<V*>(d.o1 + field(i)) = at(plane + slot(i));
                *reinterpret_cast<V*>(d.o2 + field(i)) = at(plane2 + slot(i));
            }
        } else {
            V p[kB], e[kB];
#pragma unroll
            for (int b = 0; b < kB; ++b) {
                const int i = i0 + b * step;
                if (!ok(i)) continue;
                p[b] = __ldg(reinterpret_cast<const V*>(d.rho + field(i)));
                e[b] = __ldg(reinterpret_cast<const V*>(d.dr + field(i)));
            }
#pragma unroll
            for (int b = 0; b < kB; ++b) {
                const int i = i0 + b * step;
                if (!ok(i)) continue;
                *reinterpret_cast<V*>(d.o1 + field(i)) = force4(p[b], at(plane + slot(i)), e[b]);
            }
        }
    }
}

// One window of NL lines; d.g.nl == NL.
template <int AXIS, bool SIXTH, bool SECOND, int NL>
__device__ __forceinline__ void window(const Dir32& d, const Line32& k, DevState* st, int bid,
                                       float* sh, const CUtensorMap* tmap) {
    const Geo32& g = d.g;
    const int grp = bid % g.ngroups, win = bid / g.ngroups;
    const int line0 = grp * NL, s0 = win * g.own, nown = min(g.own, g.n - s0), H = g.H;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    float* plane = sh;                                       // staged, then first derivatives
    float* plane2 = sh + NL * (AXIS == 0 ? kLW : kLWin);     // second derivatives
    auto wrap = [&](int p) {
        if (g.magic) p -= g.period * (int)__umulhi((unsigned)p, g.magic);
        else if (p >= g.period) p -= g.period;
        return p;
    };
    const int p0 = wrap(s0 - H - 4 + g.lift);  // period position of slot 0
    constexpr int PR = NL / 4;                 // 16-byte pieces of a row
    // ---- stage ----
    if constexpr (AXIS == 0) {
        const int line = line0 + warp;
        float* row = plane + warp * kLW;
        if (line < g.nlines) {
            const float* src = d.u + (size_t)line * g.ls;
            if (g.vec)
                for (int q = 4 * lane; q < kLWin; q += 128) l32::cp16(row + q, src + wrap(p0 + q));
            else
                for (int q = lane; q < kLWin; q += 32) l32::cp4(row + q, src + wrap(p0 + q));
        } else {
            for (int q = lane; q < kLWin; q += 32) row[q] = 0.0f;
        }
    } else {
        const bool interior = s0 - H - 4 >= 0 && s0 - H - 4 + kLWin <= g.n;
        if (tmap && interior && line0 + NL <= g.nlines) {
            __shared__ __align__(8) uint64_t bar;
            if (t == 0) mbar_init(&bar, 1);
            __syncthreads();
            if (t == 0) {
                mbar_expect_tx(&bar, (unsigned)(kLWin * NL * sizeof(float)));
#pragma unroll 1
                for (int b = 0; b < kLWin / kBoxRows; ++b)
                    tma_load_2d(plane + b * kBoxRows * NL, tmap, line0, p0 + b * kBoxRows, &bar);
            }
            const bool arrived = mbar_wait_bounded(&bar, 0);
            if (__syncthreads_or(!arrived)) {
                // not arrived in time: flag the run; wait once more (bounded) for the copies
                // in flight before the block leaves its shared memory
                if (t == 0) {
                    atomicOr(&st->flag, (unsigned)FLAG_STAGE);
                    atomicMin(&st->failed_t, (unsigned long long)st->t);
                }
                mbar_wait_bounded(&bar, 0);
                return;
            }
        } else {
            const int w = g.vec ? 4 : 1, pr = g.vec ? PR : NL;
            for (int i = t; i < kLWin * pr; i += NL * 32) {
                const int q = i / pr, x = w * (i - q * pr);
                float* dst = plane + q * NL + x;
                if (line0 + x >= g.nlines) {
                    for (int b = 0; b < w; ++b) dst[b] = 0.0f;
                    continue;
                }
                int p = wrap(p0 + q);
                if (g.mirror && p >= g.n) p = 2 * g.n - 1 - p;
                const float* src = d.u + (size_t)p * g.ps + (size_t)(line0 + x);
                if (g.vec) l32::cp16(dst, src);
                else l32::cp4(dst, src);
            }
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    // ---- solve ----
    const int c = AXIS == 0 ? lane : (32 / NL) * warp + lane / NL;
    float r[kC], r2[kC];
    float w1, v2, w2, z1, y2, z2, cv = 0.0f, cw = 0.0f;
    if constexpr (AXIS == 0) {
        float* row = plane + warp * kLW;
        const float* u0 = row + 4 + c * kC;
        l32::chunk_forward<SIXTH, SECOND>([&](int j) { return u0[j]; }, k, r, r2, w1, v2, w2);
        const float cf = shuffle_join1<1>(k, w1, c);
        if (SECOND) shuffle_join2<1>(k, v2, w2, c, cv, cw);
        l32::chunk_backward<SECOND>(k, cf, cv, cw, r, r2, z1, y2, z2);
        const float cb = shuffle_join1<-1>(k, z1, 31 - c);
        if (SECOND) shuffle_join2<-1>(k, y2, z2, 31 - c, cv, cw);
        l32::chunk_finish<SECOND>(k, cb, cv, cw, r, r2);
        __syncwarp();
        float* row2 = plane2 + warp * kLW;
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            row[c * kC + j] = r[j];
            if (SECOND) row2[c * kC + j] = r2[j];
        }
    } else {
        __shared__ float ea[32 * NL], ev[SECOND ? 32 * NL : 1], ew[SECOND ? 32 * NL : 1];
        __shared__ float za[32 * NL], zv[SECOND ? 32 * NL : 1], zw[SECOND ? 32 * NL : 1];
        const int l = lane % NL, e = c * NL + l;
        const float* u0 = plane + (c * kC + 4) * NL + l;
        l32::chunk_forward<SIXTH, SECOND>([&](int j) { return u0[j * NL]; }, k, r, r2, w1, v2,
                                          w2);
        ea[e] = w1;
        if (SECOND) {
            ev[e] = v2;
            ew[e] = w2;
        }
        __syncthreads();  // also: every staged value this block reads has been read
        const float cf = l32::join1<1>(k, ea + e, NL, c);
        if (SECOND) l32::join2<1>(k, ev + e, ew + e, NL, c, cv, cw);
        l32::chunk_backward<SECOND>(k, cf, cv, cw, r, r2, z1, y2, z2);
        za[e] = z1;
        if (SECOND) {
            zv[e] = y2;
            zw[e] = z2;
        }
        __syncthreads();
        const float cb = l32::join1<1>(k, za + e, -NL, 31 - c);
        if (SECOND) l32::join2<1>(k, zv + e, zw + e, -NL, 31 - c, cv, cw);
        l32::chunk_finish<SECOND>(k, cb, cv, cw, r, r2);
        float *o1 = plane + c * kC * NL + l, *o2 = plane2 + c * kC * NL + l;
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            o1[j * NL] = r[j];
            if (SECOND) o2[j * NL] = r2[j];
        }
    }
    __syncthreads();
    // ---- out ----
    if (g.vec) write_out<AXIS, SECOND, NL, 4>(d, plane, plane2, line0, s0, nown);
    else write_out<AXIS, SECOND, NL, 1>(d, plane, plane2, line0, s0, nown);
}

// x- and y-lines in one launch; 32 warps an SM
template <bool SIXTH, bool SECOND, int NL>
__global__ void __launch_bounds__(NL * 32, 32 / NL)
    k_lines_wide(Dir32 dx, Dir32 dy, const __grid_constant__ Line32 k, DevState* st, int bump,
                 int nbx, const __grid_constant__ CUtensorMap tmy, int use_tma) {
    pdl_prologue();
    extern __shared__ __align__(128) float shw[];
    if (bump && blockIdx.x == 0 && threadIdx.x == 0) st->t += 1;
    const Geo32 &gx = dx.g, &gy = dy.g;
    const int nby = (int)gridDim.x - nbx;
    bool x;
    int local;
    if (NL == 16) {
        // about one wave: the y-line blocks first, so that the slower y-windows do not form
        // the tail (1024^2: density lines 14.3 -> 12.7 us, force lines 12.3 -> 12.0)
        x = (int)blockIdx.x >= nby;
        local = x ? (int)blockIdx.x - nby : (int)blockIdx.x;
    } else {
        // many waves: by tiles of one x-window by one y-window, so that the second axis finds
        // in L2 what the first has read (4096^2 force lines 100 -> 92 us)
        // (windows of a longer line own a multiple of NL)
        const int gr = gy.nwin == 1 ? gx.ngroups : gy.own / NL;  // line groups across a tile
        const int gc = gx.nwin == 1 ? gy.ngroups : gx.own / NL;
        const int row = gx.nwin * gr + gy.ngroups;  // blocks of a full row of tiles
        const int ty = min((int)blockIdx.x / row, gy.nwin - 1);
        int r = (int)blockIdx.x - ty * row;
        const int cx = min(gr, gx.ngroups - ty * gr);
        const int tx = min(r / (cx + gc), gx.nwin - 1);
        r -= tx * (cx + gc);
        x = r < cx;
        local = x ? tx * gx.ngroups + ty * gr + r : ty * gy.ngroups + tx * gc + r - cx;
    }
    if (x)
        window<0, SIXTH, SECOND, NL>(dx, k, st, local, shw, nullptr);
    else
        window<1, SIXTH, SECOND, NL>(dy, k, st, local, shw, use_tma ? &tmy : nullptr);
}

// batched: block b belongs to instance map[b]; each instance bumps its own time level
template <bool SIXTH, bool SECOND, int NL>
__global__ void __launch_bounds__(NL * 32, NL == 8 ? 3 : 2)
    k_lines_wide_batch(const Lines32Inst* __restrict__ d, const int* __restrict__ map,
                       const __grid_constant__ Line32 k, int bump) {
    extern __shared__ __align__(128) float shw[];
    const Lines32Inst& D = d[map[blockIdx.x]];
    const int local = (int)blockIdx.x - D.blk0;
    if (bump && local == 0 && threadIdx.x == 0) D.st->t += 1;
    if (local < D.nbx) {
        const Dir32 x = D.x;
        window<0, SIXTH, SECOND, NL>(x, k, D.st, local, shw, nullptr);
    } else {
        const Dir32 y = D.y;
        window<1, SIXTH, SECOND, NL>(y, k, D.st, local - D.nbx, shw, nullptr);
    }
}

// ---- host side ----
// Tensor map of an FP32 field [ny][nx] for the y windows: boxes of nl columns x kBoxRows
// rows, no swizzle.  The encoder is the driver's cuTensorMapEncodeTiled, looked up once
// through the runtime (no link to the driver library); without it, or for fields it cannot
// describe, the windows are staged by cp.async instead.
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
    if (nx % 4 != 0 || nx < nl || ny < kLWin) return false;
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

// Lines a block.  16 lines make the y windows move 64-byte row pieces (32-byte pieces lose
// about a quarter of the DRAM bandwidth: 2.5 against 3.35 TB/s measured for windows read
// alone), but halve the blocks resident per SM.  Merged density lines: 16 win at 1024^2
// (13.3 against 14.8 us), 8 from 2048^2 up (30 against 32; 95 against 107 at 4096^2).  The
// choice moves no result.
constexpr long long kWide16Nodes = 1LL << 21;

template <bool SECOND, int NL>
constexpr size_t smem_wide() {
    return (size_t)(SECOND ? 2 : 1) * NL * kLW * sizeof(float);
}
void divide_wide(Dir32& d, int nl) {
    d.g.nl = nl;
    d.g.ngroups = (d.g.nlines + nl - 1) / nl;
}
int blocks_of(const Geo32& g) { return g.ngroups * g.nwin; }

template <bool SECOND, int NL>
cudaError_t run_wide(Dir32 x, Dir32 y, int nx, int ny, int order, DevState* st, int bump,
                     cudaStream_t s) {
    divide_wide(x, NL);
    divide_wide(y, NL);
    const int nbx = blocks_of(x.g), nby = blocks_of(y.g);
    CUtensorMap tmy;
    std::memset(&tmy, 0, sizeof(tmy));
    // (a state block is needed to report a copy that never arrives)
    const int use_tma = st && y_tensor_map(y.u, nx, ny, NL, &tmy) ? 1 : 0;
    constexpr size_t smem = smem_wide<SECOND, NL>();
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
        return launch_pdl(kern, dim3(nbx + nby), dim3(NL * 32), smem, s, x, y,
                          line32_constants(order), st, bump, nbx, tmy, use_tma);
    };
    return order == 6 ? go(k_lines_wide<true, SECOND, NL>) : go(k_lines_wide<false, SECOND, NL>);
}

template <bool SECOND, int NL>
cudaError_t run_wide_batch(const Lines32Inst* d, const int* map, int nblocks, int order, int bump,
                           cudaStream_t s) {
    constexpr size_t smem = smem_wide<SECOND, NL>();
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
        kern<<<nblocks, NL * 32, smem, s>>>(d, map, line32_constants(order), bump);
        return cudaGetLastError();
    };
    return order == 6 ? go(k_lines_wide_batch<true, SECOND, NL>)
                      : go(k_lines_wide_batch<false, SECOND, NL>);
}

}  // namespace

cudaError_t lines32_wide(Dir32 x, Dir32 y, int nx, int ny, int order, bool second, DevState* st,
                         int bump, cudaStream_t s) {
    const bool wide16 = (long long)nx * ny <= kWide16Nodes;
    if (second)
        return wide16 ? run_wide<true, 16>(x, y, nx, ny, order, st, bump, s)
                      : run_wide<true, 8>(x, y, nx, ny, order, st, bump, s);
    return wide16 ? run_wide<false, 16>(x, y, nx, ny, order, st, bump, s)
                  : run_wide<false, 8>(x, y, nx, ny, order, st, bump, s);
}

void lines32_wide_divide(Dir32& x, Dir32& y, int nl) {
    divide_wide(x, nl);
    divide_wide(y, nl);
}

cudaError_t lines32_wide_batch(const Lines32Inst* d, const int* map, int nblocks, int order,
                               bool second, int bump, int nl, cudaStream_t s) {
    if (second)
        return nl == 16 ? run_wide_batch<true, 16>(d, map, nblocks, order, bump, s)
                        : run_wide_batch<true, 8>(d, map, nblocks, order, bump, s);
    return nl == 16 ? run_wide_batch<false, 16>(d, map, nblocks, order, bump, s)
                    : run_wide_batch<false, 8>(d, map, nblocks, order, bump, s);
}

}  // namespace cplbm
