// mlp.cu -- the surrogate network of the warm start (lbm_mlp_* of
// include/cplbm.h): a 4-256-256-256-256 multilayer perceptron with tanh hidden
// layers that maps (T_r, kappa-hat, k, 1/R) to a 256-point equilibrium interface
// profile (R the radius of a drop; 0 for flat interfaces), trained and evaluated
// by the kernels of this file.
//
// Arithmetic: every matrix product runs on the tensor cores in BF16 with FP32
// accumulation; master weights, Adam moments, biases, activations kept for the
// backward pass, and the loss are FP32 (the loss sum FP64).  The products:
//   forward            Z_l   = A_{l-1} W_l          [B x fan_in] [fan_in x fan_out]
//   weight gradient    dW_l  = A_{l-1}^T D_l        [fan_in x B] [B x fan_out]
//   input gradient     D_{l-1} = (D_l W_l^T) (1 - A_{l-1}^2)
// with fused epilogues (bias + tanh, tanh derivative).  All of them run as
// tcgen05 MMAs with the accumulator in tensor memory: the forward and input-gradient
// products of a batch of rows one after another in k_umma_chain, the weight gradient
// (K = the batch) split over K in k_umma_wgrad, its operands brought in by tensor copies.  The strided mma.sync tile kernel
// (k_gemm) is kept as the comparison point, selected by lbm_mlp_set_tcgen05, and
// runs a call whose tensor maps cannot be made.
#include <cuda.h>  // CUtensorMap and its encoder's types (the encoder is fetched at run time)
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "cplbm_internal.cuh"

namespace cplbm {
namespace {

constexpr int kIn = 4, kW = 256, kOut = 256, kLayers = 4;
constexpr int kInPad = 16;  // the first product's K on mma.sync, padded to one k-step
constexpr int kK0 = 64;     // row stride of the BF16 input and K of its tcgen05 product
                            // (zero-padded to one 128-byte swizzle row)
constexpr int kFanIn[kLayers] = {kIn, kW, kW, kW};
constexpr int kFanOut[kLayers] = {kW, kW, kW, kOut};

// offset of W_l in the parameter vector (W_l then b_l, layer after layer);
// closed form on scalar constants, so device code can evaluate it too
__host__ __device__ constexpr long long param_offset(int l) {
    static_assert(kOut == kW, "the output layer has the hidden width");
    return l == 0 ? 0 : (long long)(kIn * kW + kW) + (long long)(l - 1) * (kW * kW + kW);
}
constexpr long long kParams = param_offset(kLayers);

// ---------------------------------------------------------------------------
// GEMM: C[m][n] = sum_k A(m, k) B(k, n), A(m, k) = A[m sam + k sak],
// B(k, n) = B[k sbk + n sbn], BF16 operands, FP32 accumulation.  Block tile
// 64 x 64 x 16, four warps of 32 x 32 (2 x 4 mma tiles of 16 x 8).
// ---------------------------------------------------------------------------
constexpr int BM = 64, BN = 64, BK = 16, KP = BK + 8;  // KP: padded shared row

enum Epi : int {
    EPI_STORE = 0,      // out32[m][n] = acc
    EPI_BIAS_TANH = 1,  // a = tanh(acc + bias[n]): out32 = a, out16 = bf16(a)
    EPI_BIAS = 2,       // out32 = acc + bias[n]
    EPI_TANH_BACK = 3,  // d = acc (1 - aprev[m][n]^2): out32 = d, out16 = bf16(d)
    EPI_LOSS = 4,       // y = acc + bias[n], e = y - target[m][n]: d = e scale, sum e^2
};

struct GemmArgs {
    const __nv_bfloat16* A;
    long long sam, sak;
    const __nv_bfloat16* B;
    long long sbk, sbn;
    int M, N, K;
    int epi;
    const float* bias;   // [N]
    const float* aprev;  // [M][N] (EPI_TANH_BACK)
    float* out32;        // [M][N], row-major, leading dimension N
    __nv_bfloat16* out16;
    int ld16;            // leading dimension of out16
};

__device__ __forceinline__ void mma_bf16(float c[4], const unsigned a[4], const unsigned b[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// tanh(x) = 1 - 2 / (1 + exp(2x)) with the fast exponential and division
// intrinsics: six instructions, exact limits at +-inf, NaN in NaN out.  Its
// absolute error stays below about 3e-7 at every x (relative error grows only
// where |tanh x| < 1e-3, where the BF16 rounding that every activation gets,
// 2^-9 relative, is still larger in absolute terms above |x| ~ 1.5e-4).
__device__ __forceinline__ float tanh_act(float x) {
    return 1.0f - __fdividef(2.0f, 1.0f + __expf(2.0f * x));
}

__global__ void __launch_bounds__(128) k_gemm(GemmArgs g) {
    __shared__ __align__(16) __nv_bfloat16 As[BM][KP];  // [m][k]
    __shared__ __align__(16) __nv_bfloat16 Bs[BN][KP];  // [n][k]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp >> 1, wn = warp & 1;
    const int gq = lane >> 2, tq = lane & 3;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
    const __nv_bfloat16 zero = __float2bfloat16_rn(0.0f);
    for (int k0 = 0; k0 < g.K; k0 += BK) {
        // stage: 64 x 16 of A and of B, element by element (out of range: 0)
        for (int e = tid; e < BM * BK; e += 128) {
            const int r = e / BK, k = e - r * BK;
            const int m = m0 + r, kk = k0 + k;
            As[r][k] = (m < g.M && kk < g.K) ? g.A[m * g.sam + kk * g.sak] : zero;
            const int n = n0 + r;
            Bs[r][k] = (n < g.N && kk < g.K) ? g.B[kk * g.sbk + n * g.sbn] : zero;
        }
        __syncthreads();
        unsigned a[2][4], b[4][2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = wm * 32 + i * 16 + gq;
            a[i][0] = *reinterpret_cast<const unsigned*>(&As[r][2 * tq]);
            a[i][1] = *reinterpret_cast<const unsigned*>(&As[r + 8][2 * tq]);
            a[i][2] = *reinterpret_cast<const unsigned*>(&As[r][2 * tq + 8]);
            a[i][3] = *reinterpret_cast<const unsigned*>(&As[r + 8][2 * tq + 8]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = wn * 32 + j * 8 + gq;
            b[j][0] = *reinterpret_cast<const unsigned*>(&Bs[n][2 * tq]);
            b[j][1] = *reinterpret_cast<const unsigned*>(&Bs[n][2 * tq + 8]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], b[j]);
        __syncthreads();
    }
    // epilogue: accumulator (i, j, q) is row m0 + wm 32 + i 16 + gq (+8 for
    // q >= 2), column n0 + wn 32 + j 8 + 2 tq (+1 for odd q)
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int m = m0 + wm * 32 + i * 16 + gq + (q >= 2 ? 8 : 0);
                const int n = n0 + wn * 32 + j * 8 + 2 * tq + (q & 1);
                if (m >= g.M || n >= g.N) continue;
                float v = acc[i][j][q];
                const long long o = (long long)m * g.N + n;
                if (g.epi == EPI_BIAS_TANH) {
                    v = tanh_act(v + g.bias[n]);
                    g.out16[(long long)m * g.ld16 + n] = __float2bfloat16_rn(v);
                } else if (g.epi == EPI_BIAS) {
                    v += g.bias[n];
                } else if (g.epi == EPI_TANH_BACK) {
                    const float ap = g.aprev[o];
                    v *= 1.0f - ap * ap;
                    g.out16[(long long)m * g.ld16 + n] = __float2bfloat16_rn(v);
                }
                g.out32[o] = v;
            }
}

// ---------------------------------------------------------------------------
// Tensor-core products on tcgen05 (5th-generation tensor cores, accumulator in
// tensor memory), BF16 operands, FP32 accumulation.  Operands move in K chunks
// of 64 elements: a tensor copy (TMA) of a box of 64 x rows with 128-byte
// swizzling writes each row's 128 bytes with its 16-byte pieces permuted by the
// row index mod 8, which is the tensor cores' K-major 128-byte-swizzle layout
// (8-row groups 1024 bytes apart); the MMA of the k-th 16-wide step starts
// 32 k bytes into the chunk.  Every wait on an mbarrier is
// bounded: one that runs out sets the error word and a shared abort flag, the
// other roles see the flag and leave their loops, and the CTA waits (bounded)
// for its copies and MMAs in flight before it frees its tensor memory.
//
// k_umma_chain (described beside it): the forward products and the input gradients.
//
// k_umma_wgrad: the weight gradients dW[fi x 256] = A^T D over the batch, of all four
// layers in one launch.  Both operands are read as the chain kernel left them, [batch][256],
// so K (the batch) is their slow dimension: the MN-major 128-byte-swizzle layout, 64
// columns a row of 128 bytes, 8 batch rows a group of 1024 bytes, the next 64 columns one
// box further.  K is split into slices (grid.y); each CTA streams its
// slice through a four-stage ring of 64-row chunks (warp 4 loads, warp 5 issues the MMAs)
// and writes an FP32 partial; k_gradient adds the partials in a fixed order
// (deterministic) and, in training, applies Adam to each entry as it gets it.
//
// The kernels of a call are launched with programmatic serialization: each sets up its
// barriers and tensor memory while the one before it finishes.  An Adam step at batch 256
// takes 27 us (174 with products of 2 CTAs and eighteen launches), at 32768 118 us (297).
// ---------------------------------------------------------------------------
constexpr int UM = 128, UN = 256;
constexpr unsigned kUmmaSpins = 1u << 22;
constexpr int kS32 = 36;  // padded rows of the epilogue's staging blocks
constexpr int kKC = 64;              // K chunk of the streamed operands
// k_umma_wgrad: 4 epilogue warps, a loader warp and an MMA warp; 4-stage ring
constexpr int kWgEpi = 4, kStages = 4;
constexpr int kWgThreads = 32 * (kWgEpi + 2);
constexpr int kChainCap = 1024;  // most CTAs of a k_umma_chain launch
constexpr int kBox = 64;                              // rows of a tensor-copy box
constexpr unsigned kBoxBytes = kBox * kKC * 2;        // 64 x 64 BF16
// the stages are aligned to 1024 bytes inside the dynamic allocation (hence + 1024)
constexpr size_t kWChunk = (size_t)UM * kKC * 2;             // 128 features of a row product
constexpr size_t kChunkBytes = (size_t)(UM + UN) * kKC * 2;  // of the weight gradient
constexpr size_t kWgSmem = 1024 + kStages * kChunkBytes + (size_t)kWgEpi * 32 * kS32 * 4;
static_assert(kWgSmem <= 227 * 1024 - 1024, "weight-gradient kernel shared memory");

struct RowArgs {
    int M;
    int epi;
    const float* bias;   // [256] (EPI_BIAS_TANH, EPI_BIAS, EPI_LOSS)
    const float* t;      // [M][256]: the targets (EPI_LOSS)
    float scale;         // EPI_LOSS: dL/dy = scale (y - target)
    double* sse;         // EPI_LOSS: sums of (y - target)^2, [grid]
    float* bpart;        // or null: column sums of the result, [grid][256]
    float* out32;        // [M][256] (EPI_BIAS) or null
    __nv_bfloat16* out16;   // [M][256] or null
    int* err;
};

// 128-row tiles of dW: one of layer 0 (its 4 rows padded), two of each further layer
constexpr int kWgTiles = 7;
__host__ __device__ constexpr int wg_row0(int l) { return l == 0 ? 0 : UM + (l - 1) * kW; }
struct WgMaps {
    CUtensorMap a[kLayers], d[kLayers];  // layer inputs and signals, [batch][K or 256]
};
struct WgArgs {
    int chunks;       // K chunks (64 batch rows) in all
    int per_slice;    // K chunks per slice
    float* part;      // [slices][kWgTiles * 128][256]
    const double* sse_part;  // squared-error sums of the chain's CTAs
    int nsse;                // how many
    double* sse;             // their sum
    int* err;
};

__device__ __forceinline__ unsigned su32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ bool mb_try(uint64_t* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait for the phase of the given parity; gives up early when another
// role has raised the abort flag (null: no early exit)
__device__ __forceinline__ bool mb_wait(uint64_t* bar, unsigned parity,
                                        const volatile int* abort_flag) {
    for (unsigned i = 0; i < kUmmaSpins; ++i) {
        if (mb_try(bar, parity)) return true;
        if (abort_flag && *abort_flag) return false;
    }
    return false;
}
__device__ __forceinline__ void mb_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(su32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void mb_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(su32(bar)) : "memory");
}
__device__ __forceinline__ void mb_expect(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(bar)),
                 "r"(bytes)
                 : "memory");
}
// 2-D tensor copy global -> shared of the box at (k, row), completing on bar
__device__ __forceinline__ void tma2(void* dst, const CUtensorMap* map, int k, int row,
                                     uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];\n" ::"r"(su32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(k), "r"(row), "r"(su32(bar))
        : "memory");
}
// shared-memory matrix descriptor of a K-major operand in the 128-byte swizzle
// layout: start address, leading byte offset 16 (unused by this layout), stride
// byte offset 1024 (one 8-row group), descriptor version 1, layout type 2
__device__ __forceinline__ uint64_t umma_desc(unsigned addr) {  // K-major
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// the same of an MN-major operand: 64 columns a 128-byte row, leading byte offset from one
// 64-column box to the next, stride byte offset from one group of 8 K rows to the next
__device__ __forceinline__ uint64_t umma_desc_mn(unsigned addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(kBoxBytes >> 4) << 16) |
           ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// instruction descriptor: D f32 (bits 4-5), A and B bf16 (7-9, 10-12), A and B
// MN-major (15, 16), N >> 3 at bit 17, M >> 4 at bit 24
constexpr uint32_t idesc(int n, bool mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? 3u << 15 : 0u) |
           ((uint32_t)(n >> 3) << 17) | ((uint32_t)(UM >> 4) << 24);
}
// The MMA issuer is a whole warp that stays together, in which one elected lane issues: with
// operands that the compiler sees to be the same in every lane, four MMAs and a commit take
// half the time that they do from one lane of a divergent branch (650 -> 390 cycles a
// chunk of the chain kernel).
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t r;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(r));
    return r;
}
template <uint32_t IDESC>
__device__ __forceinline__ void umma(uint32_t lead, uint32_t tmem, uint64_t da, uint64_t db,
                                     bool acc) {
    asm volatile(
        "{\n .reg .pred p, e;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 e, %5, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(da), "l"(db), "r"(IDESC), "r"(acc ? 1u : 0u), "r"(lead)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t lead, uint64_t* bar) {
    asm volatile(
        "{\n .reg .pred e;\n setp.ne.b32 e, %1, 0;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::
            "r"(su32(bar)),
        "r"(lead)
        : "memory");
}
// mb_wait by a whole warp, with one answer for all of it
__device__ __forceinline__ bool mb_wait_warp(uint64_t* bar, unsigned parity,
                                             const volatile int* abort_flag) {
    return __all_sync(0xffffffffu, mb_wait(bar, parity, abort_flag));
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}
// kNC consecutive accumulator columns of this warp's 32 lanes (one row a thread).  32, so
// that the FP32 row pieces of the epilogue are 128 bytes: in 64-byte pieces the hidden
// layers of a batch of 32768 wrote 2.8 TB/s (Adam step there 205 -> 179 us).
constexpr int kNC = 32;
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float* x) {
    uint32_t v[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
        "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
          "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
          "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),
          "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < kNC; ++j) x[j] = __uint_as_float(v[j]);
}

// this warp's 32 rows [r0, r0 + 32) x kNC columns [c, c + kNC) of a row-major
// FP32 matrix (row stride ld): thread `lane` holds row r0 + lane in x.  Stores
// and loads go through the warp's staging block s (32 rows of kS32 floats), so
// that the global accesses are 128-byte row pieces, four rows an instruction.
__device__ __forceinline__ void rows_store32(float* s, const float* x, float* out, long long ld,
                                             int r0, int c, int M, int lane) {
#pragma unroll
    for (int j = 0; j < kNC / 4; ++j)
        *reinterpret_cast<float4*>(s + lane * kS32 + 4 * j) =
            make_float4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int rr = 4 * j + (lane >> 3), q = lane & 7;
        if (r0 + rr < M)
            *reinterpret_cast<float4*>(out + (long long)(r0 + rr) * ld + c + 4 * q) =
                *reinterpret_cast<const float4*>(s + rr * kS32 + 4 * q);
    }
    __syncwarp();
}

// entries k .. k + 7 of row b of the input: x [B][4] FP32 -> BF16 [B][kK0], zero-padded
__device__ __forceinline__ uint4 input_piece(const float* x, int b, int k) {
    __align__(16) __nv_bfloat16 h[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        h[j] = __float2bfloat16_rn(k + j < kIn ? x[b * kIn + k + j] : 0.0f);
    return *reinterpret_cast<uint4*>(h);
}

// ---------------------------------------------------------------------------
// The chain of row products of ROWS (32 or 64) batch rows in one CTA, tile after tile: the
// input conversion, the four layers and, in training, the three input gradients.  The
// products are transposed, D^T = W^T A^T: 256 features are two 128-row tiles of weights,
// streamed through a ring, the batch rows the narrow operand, which stays in shared memory
// from one stage to the next, so that no CTA needs another's results.  A thread of the
// epilogue has one feature of ROWS / 2 rows: targets, outputs and biases are read and written
// in rows without staging; the hidden activations that the backward stages need stay in
// tensor memory.  Global memory gets what the weight gradient reads, written while the next
// products run.
// Roles: warps 0..15 epilogue, then the loader and the MMA issuer.  A wait that runs out sets
// the abort flag, on which every later wait gives up: the CTA goes through its stages
// without waiting, and its results are void.
// Bound by a stage's latency: of 2.5 us, the MMA issuer's waits and MMAs are 1.6 and the
// second feature tile's epilogue the rest.  A training pass of 256 rows takes 17 us, 33 in
// clusters of four CTAs that each had a quarter of the features of 128 rows, 39 as eight
// launches; one of 32768 rows 90 us, 130 as eight launches.  (Issuing the products of the
// first half of K before the second half's epilogue, and a converged loader warp, were
// slower: 496 and 516 us a fit epoch of 16 x 256 against 481.)
// ---------------------------------------------------------------------------
constexpr int kChainStages = 2 * kLayers - 1;
constexpr int kChainEpi = 16, kChainThreads = 32 * (kChainEpi + 2);
constexpr size_t act_chunk(int rows) { return (size_t)rows * kKC * 2; }  // a K chunk of rows
constexpr size_t act_bytes(int rows) { return (kW / kKC) * act_chunk(rows); }
// The weights' ring is of units of two K chunks: a wait, even for what is there, and the
// commit that frees the place cost the MMA issuer some 300 cycles.
constexpr size_t kWUnit = 2 * kWChunk;
constexpr int chain_ring(int rows) { return rows == 32 ? 5 : 4; }
constexpr size_t chain_smem(int rows) {
    return 1024 + chain_ring(rows) * kWUnit + 2 * act_bytes(rows) +
           (size_t)kLayers * kChainEpi * 32 * 4;
}
static_assert(chain_smem(32) <= 226 * 1024 - 1024, "chain kernel shared memory");
static_assert(chain_smem(64) <= 226 * 1024 - 1024, "chain kernel shared memory");
// tensor memory: [feature tile][row] of the accumulators, then of each hidden layer
constexpr int chain_cols(int rows) { return kLayers * 2 * rows; }
static_assert(chain_cols(32) == 256 && chain_cols(64) == 512, "a power of two, at most 512");
static_assert(kK0 == kKC && kKC * 2 == 128 && UM == 2 * kBox && kW == 2 * UM, "chain layout");
struct ChainMaps {
    CUtensorMap w[kChainStages];  // each stage's weights, [feature][K]
};
struct ChainArgs {
    const float* x;
    __nv_bfloat16* x16;
    int tiles;                 // of ROWS batch rows
    int n;                     // stages: 4 (inference) or 7
    RowArgs st[kChainStages];  // layers 0..3, then the signals of layers 2, 1, 0
};

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* x) {
    uint32_t v[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
        "%13,%14,%15}, [%16];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
          "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) x[j] = __uint_as_float(v[j]);
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* x) {
    uint32_t v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __float_as_uint(x[j]);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"
        "%12,%13,%14,%15};\n" ::"r"(v[0]),
        "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
        "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
}

template <int ROWS>
__global__ void __launch_bounds__(kChainThreads, 1)
    k_umma_chain(const __grid_constant__ ChainMaps m, const __grid_constant__ ChainArgs g) {
    constexpr int RING = chain_ring(ROWS), kCR = ROWS / 2;  // rows of an epilogue thread
    constexpr size_t CH = act_chunk(ROWS);
    extern __shared__ __align__(1024) unsigned char usm_raw[];
    unsigned char* usm = usm_raw + ((1024u - (su32(usm_raw) & 1023u)) & 1023u);
    // the weights' ring, two stages of the rows ([K chunk][row][128 bytes], swizzled), the
    // column sums of each layer's signals ([layer][epilogue thread])
    unsigned char* act = usm + RING * kWUnit;
    float* bsum = reinterpret_cast<float*>(act + 2 * act_bytes(ROWS));
    // units there, units free, feature tile 0/1 done, rows there, all products done
    constexpr int F0 = 0, E0 = RING, TF = 2 * RING, RF = TF + 2, DN = RF + 1;
    __shared__ __align__(8) uint64_t bar[DN + 1];
    __shared__ uint32_t tbase;
    __shared__ int abort_s;
    __shared__ double wsse[kChainEpi];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int M = g.st[0].M;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         su32(&tbase)),
                     "r"(chain_cols(ROWS))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int q = 0; q <= DN; ++q) mb_init(&bar[q], q == RF ? kChainEpi : 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        abort_s = 0;
    }
    for (int i = tid; i < kLayers * kChainEpi * 32; i += kChainThreads) bsum[i] = 0.0f;
    pdl_prologue();  // what follows reads what the kernels before this one wrote
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tbase;
    volatile int* abort_v = &abort_s;
    auto give_up = [&] {
        atomicExch(g.st[0].err, 1);
        *abort_v = 1;
    };
    // k: stages so far, over all tiles; the rows of stage k are in buffer k & 1
    if (warp == kChainEpi) {
        if (lane == 0) {
            // loader: each stage's weights, feature tile after feature tile, through the ring
            int q = 0;  // units issued
            bool ok = true;
            for (int t = blockIdx.x; ok && t < g.tiles; t += gridDim.x)
                for (int s = 0; ok && s < g.n; ++s) {
                    const int nkc = s == 0 ? 1 : kW / kKC;  // K: kK0 in the first layer
                    for (int tile = 0; ok && tile < 2; ++tile)
                        for (int j = 0; j < nkc; j += 2, ++q) {
                            const int st = q % RING;
                            if (q >= RING)
                                ok = mb_wait(&bar[E0 + st], ((q / RING) - 1) & 1, abort_v);
                            if (!ok) break;
                            const int sub = nkc - j < 2 ? nkc - j : 2;
                            mb_expect(&bar[F0 + st], sub * (unsigned)kWChunk);
                            for (int r = 0; r < sub * UM; r += kBox)
                                tma2(usm + st * kWUnit + r * kKC * 2, &m.w[s],
                                     (j + r / UM) * kKC, tile * UM + r % UM, &bar[F0 + st]);
                        }
                }
            if (!ok) give_up();
            // the copies issued last complete before the CTA leaves (bounded)
            for (int r = (q > RING ? q - RING : 0); r < q; ++r)
                mb_wait(&bar[F0 + r % RING], (r / RING) & 1, nullptr);
        }
    } else if (warp == kChainEpi + 1) {
        const uint32_t lead = elect_one();
        int st = 0, k = 0;
        unsigned phase = 0;
        bool ok = true;
        for (int t = blockIdx.x; ok && t < g.tiles; t += gridDim.x)
            for (int s = 0; ok && s < g.n; ++s, ++k) {
                const int nkc = s == 0 ? 1 : kW / kKC;
                const uint64_t rows = umma_desc(su32(act + (k & 1) * act_bytes(ROWS)));
                ok = mb_wait_warp(&bar[RF], k & 1, abort_v);
                for (int tile = 0; ok && tile < 2; ++tile) {
                    for (int j = 0; j < nkc; j += 2) {
                        ok = mb_wait_warp(&bar[F0 + st], phase, abort_v);
                        if (!ok) break;
                        tc_fence_after();
                        for (int h = j; h < j + 2 && h < nkc; ++h) {
                            const uint64_t A =
                                umma_desc(su32(usm + st * kWUnit + (h - j) * kWChunk));
                            const uint64_t B = rows + (uint64_t)h * (CH >> 4);
#pragma unroll
                            for (int kk = 0; kk < kKC / 16; ++kk)
                                umma<idesc(ROWS, false)>(lead, tmem + (uint32_t)(tile * ROWS),
                                                         A + kk * 2, B + kk * 2,
                                                         h > 0 || kk > 0);
                        }
                        umma_commit(lead, &bar[E0 + st]);
                        if (++st == RING) {
                            st = 0;
                            phase ^= 1u;
                        }
                    }
                    if (ok) umma_commit(lead, &bar[TF + tile]);
                }
            }
        if (!ok && lead) give_up();
        umma_commit(lead, &bar[DN]);
        mb_wait_warp(&bar[DN], 0, nullptr);
    } else {
        const int quarter = warp & 3, tile = (warp >> 2) & 1, half = warp >> 3;
        const int f0 = tile * UM + quarter * 32, f = f0 + lane;
        const uint32_t col = tmem + ((uint32_t)(quarter * 32) << 16) +
                             (uint32_t)(tile * ROWS + half * kCR);
        // element f of the rows; 16-byte pieces of this warp's 32 features
        unsigned char* af = act + (f >> 6) * CH + (f & 7) * 2;
        unsigned char* aw = act + (f0 >> 6) * CH;
        const int piece = (f & 63) >> 3, piece0 = (f0 & 63) >> 3;
        // this warp's rows of tile t of the input into the buffer of stage k: those of its
        // features (kK0 in all), by the warps that have them
        auto input = [&](int t, int k) {
            if (f0 < kK0) {
#pragma unroll
                for (int i = 0; i < kCR / 8; ++i) {
                    const int rr = half * kCR + ((lane + 32 * i) >> 2), p = piece0 + (lane & 3);
                    const int b = t * ROWS + rr;
                    const uint4 v =
                        b < M ? input_piece(g.x, b, 8 * p) : make_uint4(0u, 0u, 0u, 0u);
                    *reinterpret_cast<uint4*>(aw + (k & 1) * act_bytes(ROWS) + rr * 128 +
                                              ((p ^ (rr & 7)) << 4)) = v;
                    if (b < M && g.n > kLayers)
                        *reinterpret_cast<uint4*>(g.x16 + (long long)b * kK0 + 8 * p) = v;
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mb_arrive(&bar[RF]);
        };
        double sse = 0.0;
        int k = 0;
        input(blockIdx.x, 0);
        for (int t = blockIdx.x; t < g.tiles; t += gridDim.x) {
            const int r0 = t * ROWS + half * kCR;  // this thread's rows r0 .. of feature f
            const int nr = M - r0;                 // those below it are live
            for (int s = 0; s < g.n; ++s, ++k) {
                const RowArgs& r = g.st[s];
                const unsigned next = (unsigned)(((k + 1) & 1) * act_bytes(ROWS));
                const float bias = r.bias ? r.bias[f] : 0.0f;
                float pre[kCR];
                if (r.epi == EPI_LOSS) {
#pragma unroll
                    for (int j = 0; j < kCR; ++j)
                        pre[j] = j < nr ? __ldg(r.t + (long long)(r0 + j) * UN + f) : 0.0f;
                }
                if (!mb_wait_warp(&bar[TF + tile], k & 1, abort_v) && lane == 0) give_up();
                __syncwarp();
                tc_fence_after();
                float bs = 0.0f;
#pragma unroll
                for (int h = 0; h < kCR; h += 16) {
                    float a[16], x[16];
                    tmem_ld16(col + (uint32_t)h, x);
                    if (r.epi == EPI_TANH_BACK) {
                        tmem_ld16(col + (uint32_t)((kChainStages - s) * 2 * ROWS + h), a);
#pragma unroll
                        for (int j = 0; j < 16; ++j) x[j] *= 1.0f - a[j] * a[j];
                    } else if (r.epi == EPI_BIAS_TANH) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) x[j] = tanh_act(x[j] + bias);
                    } else if (r.epi == EPI_BIAS) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) x[j] += bias;
                    } else {
                        float e2 = 0.0f;
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float e = h + j < nr ? x[j] + bias - pre[h + j] : 0.0f;
                            e2 = fmaf(e, e, e2);
                            x[j] = 2.0f * e * r.scale;
                        }
                        sse += (double)e2;
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (h + j >= nr) x[j] = 0.0f;  // rows past M add nothing to the sums
                    if (r.out16) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const int rr = half * kCR + h + j;
                            *reinterpret_cast<__nv_bfloat16*>(af + next + rr * 128 +
                                                              ((piece ^ (rr & 7)) << 4)) =
                                __float2bfloat16_rn(x[j]);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (h + j < nr) r.out32[(long long)(r0 + h + j) * kW + f] = x[j];
                    }
                    if (r.epi == EPI_BIAS_TANH && g.n > kLayers)
                        tmem_st16(col + (uint32_t)((s + 1) * 2 * ROWS + h), x);
                    if (r.bpart) {
                        float cs = 0.0f;
#pragma unroll
                        for (int j = 0; j < 16; ++j) cs += x[j];
                        bs += cs;
                    }
                }
                if (s + 1 < g.n) {
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mb_arrive(&bar[RF]);
                }
                __syncwarp();
                // what the weight gradient reads, while the next products run
                if (r.out16 && g.n > kLayers) {
#pragma unroll
                    for (int i = 0; i < kCR / 8; ++i) {
                        const int j = (lane + 32 * i) >> 2, p = lane & 3, rr = half * kCR + j;
                        if (j < nr)
                            *reinterpret_cast<uint4*>(r.out16 + (long long)(r0 + j) * kW + f0 +
                                                      8 * p) =
                                *reinterpret_cast<const uint4*>(
                                    aw + next + rr * 128 + (((piece0 + p) ^ (rr & 7)) << 4));
                    }
                }
                const int layer = s < kLayers ? s : kChainStages - 1 - s;
                if (r.bpart) bsum[layer * kChainEpi * 32 + tid] += bs;
                __syncwarp();
            }
            if (t + gridDim.x < g.tiles) input(t + gridDim.x, k);
        }
        if (g.n > kLayers) {
            for (int i = 16; i > 0; i >>= 1) sse += __shfl_down_sync(0xffffffffu, sse, i);
            if (lane == 0) wsse[warp] = sse;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (g.n > kLayers && tid < kW)
        // (threads f and f + kW have feature f's halves of the rows)
        for (int s = kLayers - 1; s < g.n; ++s) {
            const int layer = s < kLayers ? s : kChainStages - 1 - s;
            const float* b = bsum + layer * kChainEpi * 32;
            g.st[s].bpart[(long long)blockIdx.x * UN + tid] = b[tid] + b[tid + kW];
        }
    if (g.n > kLayers && warp == kW / 32) {
        double sse = lane < kChainEpi ? wsse[lane] : 0.0;
        for (int i = kChainEpi / 2; i > 0; i >>= 1) sse += __shfl_down_sync(0xffffffffu, sse, i);
        if (lane == 0) g.st[kLayers - 1].sse[blockIdx.x] = sse;
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                     "r"(chain_cols(ROWS))
                     : "memory");
}

__global__ void __launch_bounds__(kWgThreads, 1)
    k_umma_wgrad(const __grid_constant__ WgMaps maps, WgArgs g) {
    extern __shared__ __align__(1024) unsigned char usm_raw[];
    unsigned char* usm = usm_raw + ((1024u - (su32(usm_raw) & 1023u)) & 1023u);
    // stage s: A chunk (UM x kKC) then B chunk (UN x kKC)
    constexpr unsigned kAbytes = UM * kKC * 2, kBbytes = UN * kKC * 2;
    static_assert(kAbytes + kBbytes == kChunkBytes, "chunk layout");
    float* st32 = reinterpret_cast<float*>(usm + (size_t)kStages * (kAbytes + kBbytes));
    // [0..3] stage full, [4..7] stage free, [8] all MMAs done
    __shared__ __align__(8) uint64_t bar[2 * kStages + 1];
    __shared__ uint32_t tbase;
    __shared__ int abort_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mt = blockIdx.x, slice = blockIdx.y;
    const int layer = (mt + 1) / 2, m0 = mt == 0 ? 0 : ((mt - 1) & 1) * UM;
    const int j0 = slice * g.per_slice;
    const int nk = min(g.per_slice, g.chunks - j0);  // >= 1 by the host's choice of slices
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         su32(&tbase)),
                     "r"(UN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < 2 * kStages + 1; ++s) mb_init(&bar[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        abort_s = 0;
    }
    pdl_prologue();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tbase;
    volatile int* abort_v = &abort_s;
    if (warp == kWgEpi) {
        if (lane == 0) {
            // loader
            int loaded = 0;  // chunks whose copies were issued
            bool ok = true;
            for (int j = 0; j < nk; ++j) {
                const int s = j % kStages;
                if (j >= kStages) ok = mb_wait(&bar[kStages + s], ((j / kStages) - 1) & 1, abort_v);
                if (!ok) break;
                unsigned char* A = usm + (size_t)s * (kAbytes + kBbytes);
                mb_expect(&bar[s], kAbytes + kBbytes);
                for (int c = 0; c < UM; c += kKC)
                    tma2(A + c * kBox * 2, &maps.a[layer], m0 + c, (j0 + j) * kBox, &bar[s]);
                for (int c = 0; c < UN; c += kKC)
                    tma2(A + kAbytes + c * kBox * 2, &maps.d[layer], c, (j0 + j) * kBox, &bar[s]);
                loaded = j + 1;
            }
            if (!ok) {
                atomicExch(g.err, 1);
                *abort_v = 1;
            }
            // every issued copy completes before the CTA leaves (bounded)
            for (int j = (loaded > kStages ? loaded - kStages : 0); j < loaded; ++j)
                mb_wait(&bar[j % kStages], (j / kStages) & 1, nullptr);
        }
    } else if (warp == kWgEpi + 1) {
        // MMA issuer
        const uint32_t lead = elect_one();
        bool ok = true;
        int issued = 0;
        for (int j = 0; j < nk; ++j) {
            const int s = j % kStages;
            ok = mb_wait_warp(&bar[s], (j / kStages) & 1, abort_v);
            if (!ok) break;
            tc_fence_after();
            const unsigned A = su32(usm + (size_t)s * (kAbytes + kBbytes));
            const uint64_t da = umma_desc_mn(A), db = umma_desc_mn(A + kAbytes);
#pragma unroll
            for (int kk = 0; kk < kKC / 16; ++kk)
                umma<idesc(UN, true)>(lead, tmem, da + kk * (2048 >> 4), db + kk * (2048 >> 4),
                                      j > 0 || kk > 0);
            umma_commit(lead, &bar[kStages + s]);
            issued = j + 1;
        }
        if (ok) {
            umma_commit(lead, &bar[2 * kStages]);
        } else {
            if (lead) {
                atomicExch(g.err, 1);
                *abort_v = 1;
            }
            if (issued > 0)
                mb_wait_warp(&bar[kStages + (issued - 1) % kStages],
                             ((issued - 1) / kStages) & 1, nullptr);
        }
    } else {
        if (mt == 0 && slice == 0 && warp == 0) {
            // the call's squared-error sum, in a fixed order, while the products run
            double sse = 0.0;
            for (int q = lane; q < g.nsse; q += 32) sse += g.sse_part[q];
            for (int o = 16; o > 0; o >>= 1) sse += __shfl_down_sync(0xffffffffu, sse, o);
            if (lane == 0) *g.sse = sse;
        }
        bool ok = mb_wait(&bar[2 * kStages], 0, abort_v);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
            tc_fence_after();
            float* s32 = st32 + warp * 32 * kS32;
            const uint32_t acc = tmem + ((uint32_t)(warp * 32) << 16);
            const int r0 = mt * UM + warp * 32;
            float* out = g.part + (long long)slice * kWgTiles * UM * UN;
            for (int c = 0; c < UN; c += kNC) {
                float x[kNC];
                tmem_ld(acc + (uint32_t)c, x);
                rows_store32(s32, x, out, UN, r0, c, kWgTiles * UM, lane);
            }
        } else if (lane == 0) {
            atomicExch(g.err, 1);
            *abort_v = 1;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                     "r"(UN)
                     : "memory");
}

// One Adam step of one parameter.
__device__ __forceinline__ float adam(float p, float gi, float* m, float* v, float lr, float c1,
                                      float c2) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float mi = b1 * *m + (1.0f - b1) * gi;
    const float vi = b2 * *v + (1.0f - b2) * gi * gi;
    *m = mi;
    *v = vi;
    return p - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// where the BF16 copies of parameter k of layer l's weights (k = row * 256 + column) go
__device__ __forceinline__ void store_w16(int l, int k, float p, __nv_bfloat16* w16,
                                          __nv_bfloat16* w16t) {
    const __nv_bfloat16 h = __float2bfloat16_rn(p);
    const int row = k / kW, n = k - row * kW;
    if (l == 0) {
        w16[k] = h;
        w16t[n * kK0 + row] = h;
    } else {
        w16[kInPad * kW + (l - 1) * kW * kW + k] = h;
        w16t[kK0 * kW + (l - 1) * kW * kW + n * kW + row] = h;
    }
}

struct GradArgs {
    const float* part;    // [slices][kWgTiles * 128][256]
    int slices;
    const float* bpart;   // [layers][kChainCap][256]: column sums of each signal
    int nb;               // rows of it in use
    float* grad;          // !ADAM: the gradient
    float *p, *m, *v;     // ADAM: parameters and moments
    float lr, c1, c2;
    __nv_bfloat16 *w16, *w16t;
};

// The parameter's new value from its gradient, or the gradient itself.
template <bool ADAM>
__device__ __forceinline__ void take_gradient(const GradArgs& g, int l, int k, bool weight,
                                              float t) {
    const int i = (int)param_offset(l) + k;
    if constexpr (ADAM) {
        const float p = adam(g.p[i], t, g.m + i, g.v + i, g.lr, g.c1, g.c2);
        g.p[i] = p;
        if (weight) store_w16(l, k, p, g.w16, g.w16t);
    } else {
        g.grad[i] = t;
    }
}

// The gradient: dW[k][n] = sum of part[s][row][n] over the slices, db[n] = sum of the
// column-sum rows.  Eight running sums (rows q, q + 8, ...) added in order at the end, so
// the result does not depend on timing: a weight's in one thread (the first kGradW blocks),
// a bias's in eight (a large batch has 152 rows to add; in one thread they set the kernel's
// time).  ADAM: the parameter and its BF16 copies are updated with it, which a launch of
// its own would read back.  65 us at batch 32768 with a bias in one thread, 6.4 so.
constexpr int kGradW = (kIn * kW + (kLayers - 1) * kW * kW) / 256;  // blocks of weights
constexpr int kGradB = kLayers * kW / 32;                           // blocks of biases
template <bool ADAM>
__global__ void __launch_bounds__(256) k_gradient(GradArgs g) {
    pdl_prologue();
    if ((int)blockIdx.x < kGradW) {
        int k = blockIdx.x * 256 + threadIdx.x, l = 0;
        if (k >= kIn * kW) {
            k -= kIn * kW;
            l = 1 + k / (kW * kW);
            k -= (l - 1) * kW * kW;
        }
        const float* src = g.part + (long long)wg_row0(l) * UN + k;
        constexpr long long stride = (long long)kWgTiles * UM * UN;
        float acc[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 2
        for (int q = 0; q < g.slices; q += 8) {
            float r[8];
#pragma unroll
            for (int y = 0; y < 8; ++y) r[y] = q + y < g.slices ? src[(q + y) * stride] : 0.0f;
#pragma unroll
            for (int y = 0; y < 8; ++y) acc[y] += r[y];
        }
        float t = acc[0];
#pragma unroll
        for (int y = 1; y < 8; ++y) t += acc[y];
        take_gradient<ADAM>(g, l, k, true, t);
        return;
    }
    __shared__ float acc[8][33];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int o = ((int)blockIdx.x - kGradW) * 32 + x, l = o / kW, n = o - l * kW;
    const float* src = g.bpart + (long long)l * kChainCap * UN + n;
    float s = 0.0f;
#pragma unroll 8
    for (int q = y; q < g.nb; q += 8) s += src[q * UN];
    acc[y][x] = s;
    __syncthreads();
    if (y == 0) {
        float t = acc[0][x];
#pragma unroll
        for (int p = 1; p < 8; ++p) t += acc[p][x];
        take_gradient<ADAM>(g, l, (l == 0 ? kIn : kW) * kW + n, false, t);
    }
}

// x [B][4] FP32 -> BF16 [B][kK0], zero-padded
__global__ void k_input(const float* __restrict__ x, __nv_bfloat16* __restrict__ x16, int B) {
    pdl_prologue();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    // eight of a row's kK0 entries a thread
    if (i < B * (kK0 / 8))
        reinterpret_cast<uint4*>(x16)[i] = input_piece(x, i / (kK0 / 8), 8 * (i % (kK0 / 8)));
}

// FP32 master weights -> BF16 copies ([fan_in padded][fan_out] for layer 0; the
// padding stays zero), and the same transposed ([fan_out][fan_in padded]) for the
// tensor-core products, whose second operand is K-major
__global__ void k_weights16(const float* __restrict__ p, __nv_bfloat16* __restrict__ w16,
                            __nv_bfloat16* __restrict__ w16t) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kParams) return;
    int l = 0;
    while (l + 1 < kLayers && i >= param_offset(l + 1)) ++l;
    const int k = i - (int)param_offset(l);
    if (k < (l == 0 ? kIn : kW) * kW) store_w16(l, k, p[i], w16, w16t);
}

// dL/dy = 2 (y - t) / (B N) (FP32 and BF16), and the squared-error sum
__global__ void k_loss_grad(const float* __restrict__ y, const float* __restrict__ t, int total,
                            float scale, float* __restrict__ d32, __nv_bfloat16* __restrict__ d16,
                            double* __restrict__ sse) {
    __shared__ double red[256];
    double s = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const float e = y[i] - t[i];
        const float d = 2.0f * e * scale;
        d32[i] = d;
        d16[i] = __float2bfloat16_rn(d);
        s += (double)e * e;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(sse, red[0]);
}

// column sums: db[n] = sum_b d[b][n]
__global__ void k_bias_grad(const float* __restrict__ d, int B, int N, float* __restrict__ db) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    float s = 0.0f;
    for (int b = 0; b < B; ++b) s += d[(long long)b * N + n];
    db[n] = s;
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, long long n, float lr, float c1, float c2) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        p[i] = adam(p[i], g[i], m + i, v + i, lr, c1, c2);
}

}  // namespace
}  // namespace cplbm

using namespace cplbm;

struct lbm_mlp;

namespace {

// tensor maps of the tcgen05 products for one batch size (they depend on the
// batch through the row extents), all with boxes of 64 x 64
struct TcMaps {
    int B = -1;
    WgMaps wg;               // a: x16, a16[0..2], also the forward A operands;
                             // d: the backward signals, also the input gradients' A
    CUtensorMap wt[kLayers]; // w16t of each layer: [256][K]
    CUtensorMap w[kLayers];  // w16 of layers 1..3 ([fi][fo] = [256][K = fo])
};

}  // namespace

struct lbm_mlp {
    int dev, max_batch, R, nsm;  // R: rows of the batch-sized buffers (max_batch rounded to 8)
    cudaStream_t stream;
    float *p, *g, *m, *v;        // FP32 parameters, gradient, Adam moments
    __nv_bfloat16* w16;          // BF16 weight copies, layer by layer ([fan_in][fan_out])
    __nv_bfloat16* w16t;         // the same transposed ([fan_out][fan_in]; fan_in kK0 for layer 0)
    int* err;                    // device word: a tensor-core product's wait ran out
    int* h_err;                  // pinned mirror
    __nv_bfloat16* x16;          // [R][kK0]
    float* a32[kLayers];         // layer outputs, FP32 [R][256]
    __nv_bfloat16* a16[kLayers - 1];   // hidden outputs, BF16 (inputs of the next product)
    __nv_bfloat16* sig[kLayers]; // backward signal at each layer's output, BF16 [R][256]
    float *d32, *e32;            // the same in FP32 (mma.sync kernel only), alternating
    float* part;                 // weight-gradient partials [slices][kWgTiles * 128][256]
    float* bpart;                // bias-gradient partials [layers][kChainCap][256]
    double* sse;                 // squared-error sum of the call
    double* sse_part;            // those of the chain's CTAs, [kChainCap]
    double* h_sse;               // pinned mirror of the sum and err
    long long step;
    bool tensor_cores;           // forward and input-gradient products by tcgen05
    TcMaps maps;
};

namespace {

size_t al(size_t v) { return (v + 255) / 256 * 256; }

struct MlpLayout {
    size_t p, g, m, v, w16, w16t, x16, a32, a16, sig, d32, e32, part, bpart, sse, sse_part,
        total;
};

int rows_of(int B) { return (B + 7) / 8 * 8; }  // rows of the batch-sized buffers

// K slices of the weight gradients for a batch of B: 64-row chunks, one a slice up to
// kWgSlices; larger batches take as many as make one wave of the launch's CTAs, kWgTiles
// a slice, which also keeps the partials small (at 32768: 21 slices, 19 MB for all layers).
constexpr int kWgSlices = 74, kWgWave = 21;
struct Slicing {
    int chunks, per_slice, slices;
};
Slicing slicing(int B) {
    Slicing s;
    s.chunks = (B + kBox - 1) / kBox;
    s.per_slice = s.chunks <= kWgSlices ? 1 : (s.chunks + kWgWave - 1) / kWgWave;
    s.slices = (s.chunks + s.per_slice - 1) / s.per_slice;
    return s;
}

MlpLayout mlp_layout(int B0) {
    const size_t B = (size_t)rows_of(B0);
    // slices of any batch up to B0: at most kWgSlices, and at most its chunks
    const int chunks = slicing(B0).chunks;
    const size_t S = (size_t)(chunks < kWgSlices ? chunks : kWgSlices);
    MlpLayout L;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += al(bytes);
        return at;
    };
    L.p = take(kParams * 4);
    L.g = take(kParams * 4);
    L.m = take(kParams * 4);
    L.v = take(kParams * 4);
    L.w16 = take(((size_t)kInPad * kW + 3ull * kW * kW) * 2);
    L.w16t = take(((size_t)kK0 * kW + 3ull * kW * kW) * 2);
    L.x16 = take(B * kK0 * 2);
    L.a32 = take((size_t)kLayers * B * kW * 4);
    L.a16 = take((size_t)(kLayers - 1) * B * kW * 2);
    L.sig = take((size_t)kLayers * B * kW * 2);
    L.d32 = take(B * kW * 4);
    L.e32 = take(B * kW * 4);
    L.part = take(S * kWgTiles * UM * UN * 4);
    L.bpart = take((size_t)kLayers * kChainCap * UN * 4);
    L.sse = take(16);  // the squared-error sum and the error word, read back together
    L.sse_part = take(kChainCap * sizeof(double));
    L.total = o;
    return L;
}

#define CK(call)                                  \
    do {                                          \
        cudaError_t e_ = (call);                  \
        if (e_ != cudaSuccess) return LBM_ECUDA;  \
    } while (0)

cudaError_t gemm(const GemmArgs& g, cudaStream_t s) {
    dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM);
    k_gemm<<<grid, 128, 0, s>>>(g);
    return cudaGetLastError();
}

const __nv_bfloat16* w16_of(const lbm_mlp* n, int l) {
    return l == 0 ? n->w16 : n->w16 + (size_t)kInPad * kW + (size_t)(l - 1) * kW * kW;
}
const __nv_bfloat16* w16t_of(const lbm_mlp* n, int l) {
    return l == 0 ? n->w16t : n->w16t + (size_t)kK0 * kW + (size_t)(l - 1) * kW * kW;
}

// Drain the stream; a tensor-core product whose bounded wait ran out since the
// last check makes this LBM_ETIMEOUT (and the word is cleared).
lbm_status sync(lbm_mlp* n) {
    if (cudaMemcpyAsync(n->h_sse, n->sse, 16, cudaMemcpyDeviceToHost, n->stream) !=
            cudaSuccess ||
        cudaStreamSynchronize(n->stream) != cudaSuccess)
        return LBM_ECUDA;
    if (*n->h_err) {
        *n->h_err = 0;
        if (cudaMemsetAsync(n->err, 0, sizeof(int), n->stream) != cudaSuccess) return LBM_ECUDA;
        return LBM_ETIMEOUT;
    }
    return LBM_OK;
}

// ---- tensor-core products: host side ----
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                   const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encoder() {
    static EncodeTiledFn fn = nullptr;
    static bool looked = false;
    if (!looked) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        looked = true;
    }
    return fn;
}

// Tensor map of a BF16 matrix [rows][cols] (cols a multiple of 8) whose boxes of 64
// columns x 64 rows land in shared memory in the 128-byte-swizzle layout; parts of a
// box outside the matrix arrive as zeros.
bool sw128_map(const __nv_bfloat16* A, int rows, int cols, CUtensorMap* m) {
    const EncodeTiledFn enc = encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kKC, (cuuint32_t)kBox};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(A), dims,
               strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

// every tensor map of the tcgen05 path for a batch of B; false if one cannot
// be made (the call then runs on the mma.sync kernel)
bool prepare_maps(lbm_mlp* n, int B) {
    TcMaps& t = n->maps;
    if (t.B == B) return true;
    t.B = -1;
    bool ok = true;
    for (int l = 0; l < kLayers; ++l) {
        const int K = l == 0 ? kK0 : kW;
        ok = ok && sw128_map(l == 0 ? n->x16 : n->a16[l - 1], B, K, &t.wg.a[l]);
        ok = ok && sw128_map(n->sig[l], B, kW, &t.wg.d[l]);
        ok = ok && sw128_map(w16t_of(n, l), UN, K, &t.wt[l]);
        if (l > 0) ok = ok && sw128_map(w16_of(n, l), UN, kW, &t.w[l]);
    }
    if (ok) t.B = B;
    return ok;
}

cudaError_t set_smem_attrs(int dev) {
    static unsigned long long done = 0;  // one bit per device
    const unsigned long long bit = 1ull << (dev & 63);
    if (done & bit) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(
        k_umma_chain<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chain_smem(32));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_umma_chain<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)chain_smem(64));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_umma_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kWgSmem);
    if (e == cudaSuccess) done |= bit;
    return e;
}

// a launch with programmatic serialization (every kernel here starts with pdl_prologue)
template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kern)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t s,
                   Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

float* bpart_of(const lbm_mlp* n, int l) { return n->bpart + (size_t)l * kChainCap * UN; }

// The row products of a pass on tcgen05, in order: the four layers and, where there are
// targets t (training), the signals of layers 2, 1, 0.  t null: inference, only the output
// (written to y).  In training the last layer's epilogue turns its output straight into the loss
// signal dL/dy (BF16, column sums) and the squared-error sum, without storing y.
int row_stages(lbm_mlp* n, int B, const float* t, float* y, RowArgs* st) {
    for (int l = 0; l < kLayers; ++l) {
        RowArgs& g = st[l];
        g = RowArgs{};
        g.M = B;
        g.bias = n->p + param_offset(l) + (long long)kFanIn[l] * kFanOut[l];
        g.err = n->err;
        if (l < kLayers - 1) {
            g.epi = EPI_BIAS_TANH;
            g.out16 = n->a16[l];
        } else if (t) {
            g.epi = EPI_LOSS;
            g.t = t;
            g.scale = 1.0f / ((float)B * kOut);
            g.sse = n->sse_part;
            g.out16 = n->sig[l];
            g.bpart = bpart_of(n, l);
        } else {
            g.epi = EPI_BIAS;
            g.out32 = y;
        }
    }
    if (!t) return kLayers;
    for (int l = kLayers - 1; l > 0; --l) {
        // D_{l-1} = (D_l W_l^T) (1 - A_{l-1}^2): the weights' K-major operand is W_l itself
        // ([fi][fo])
        RowArgs& g = st[2 * kLayers - 1 - l];
        g = RowArgs{};
        g.M = B;
        g.epi = EPI_TANH_BACK;
        g.out16 = n->sig[l - 1];
        g.bpart = bpart_of(n, l - 1);
        g.err = n->err;
    }
    return kChainStages;
}

// Rows of a chain CTA's tile: 32 while those tiles are at most one round of CTAs, where the
// latency of a tile is what counts (17 us against 22 of 64 rows, by the stages' timings),
// else 64, for half the weights' traffic a row.
int chain_rows(const lbm_mlp* n, int B) {
    return (B + UM - 1) / UM * (UM / 32) <= n->nsm ? 32 : 64;
}
// (of whole 128-row tiles)
int chain_tiles(const lbm_mlp* n, int B) { return (B + UM - 1) / UM * (UM / chain_rows(n, B)); }
// CTAs, each of which leaves one row of column sums per layer
int chain_ctas(const lbm_mlp* n, int B) {
    const int cap = n->nsm < kChainCap ? n->nsm : kChainCap, tiles = chain_tiles(n, B);
    return tiles < cap ? tiles : cap;
}

// the row products of a pass (row_stages), one launch
lbm_status rows_pass(lbm_mlp* n, const float* x, int B, const float* t, float* y) {
    ChainArgs c;
    c.x = x;
    c.x16 = n->x16;
    c.tiles = chain_tiles(n, B);
    c.n = row_stages(n, B, t, y, c.st);
    ChainMaps m;
    for (int s = 0; s < kChainStages; ++s)
        m.w[s] = s < kLayers ? n->maps.wt[s] : n->maps.w[2 * kLayers - 1 - s];
    const int rows = chain_rows(n, B);
    CK(launch(rows == 32 ? k_umma_chain<32> : k_umma_chain<64>, dim3(chain_ctas(n, B)),
              kChainThreads, chain_smem(rows), n->stream, m, c));
    return LBM_OK;
}

// the partial weight gradients, after rows_pass with targets, and the squared-error sum from
// those of the chain's CTAs: each is stored, so that nothing is left of an earlier call, a
// captured one or a replay
lbm_status wgrad_tc(lbm_mlp* n, int B) {
    const Slicing sl = slicing(B);
    const WgArgs w{sl.chunks, sl.per_slice, n->part, n->sse_part, chain_ctas(n, B), n->sse,
                   n->err};
    CK(launch(k_umma_wgrad, dim3(kWgTiles, sl.slices), kWgThreads, kWgSmem, n->stream,
              n->maps.wg, w));
    return LBM_OK;
}

// the gradient from the partial sums of wgrad_tc: into grad, or (grad null) into one
// Adam step of the parameters
lbm_status gradient_tc(lbm_mlp* n, int B, float* grad, float lr, float c1, float c2) {
    const GradArgs g{n->part, slicing(B).slices, n->bpart, chain_ctas(n, B), grad,
                     n->p, n->m, n->v, lr, c1, c2, n->w16, n->w16t};
    CK(launch(grad ? k_gradient<false> : k_gradient<true>, dim3(kGradW + kGradB), 256, 0,
              n->stream, g));
    return LBM_OK;
}

// the mma.sync forward pass (every layer's FP32 output kept)
lbm_status forward_ms(lbm_mlp* n, const float* x, int B) {
    cudaStream_t s = n->stream;
    CK(launch(k_input, dim3((B * (kK0 / 8) + 255) / 256), 256, 0, s, x, n->x16, B));
    for (int l = 0; l < kLayers; ++l) {
        GemmArgs g{};
        g.A = l == 0 ? n->x16 : n->a16[l - 1];
        g.sam = l == 0 ? kK0 : kW;
        g.sak = 1;
        g.B = w16_of(n, l);
        g.sbk = kFanOut[l];
        g.sbn = 1;
        g.M = B;
        g.N = kFanOut[l];
        g.K = l == 0 ? kInPad : kW;
        g.epi = l < kLayers - 1 ? EPI_BIAS_TANH : EPI_BIAS;
        g.bias = n->p + param_offset(l) + (long long)kFanIn[l] * kFanOut[l];
        g.out32 = n->a32[l];
        g.out16 = l < kLayers - 1 ? n->a16[l] : nullptr;
        g.ld16 = kW;
        CK(gemm(g, s));
    }
    return LBM_OK;
}

// whether this call runs on tcgen05 (maps for batch B made, attributes set)
bool use_tc(lbm_mlp* n, int B, lbm_status* st) {
    *st = LBM_OK;
    if (!n->tensor_cores) return false;
    if (!prepare_maps(n, B)) {
        n->tensor_cores = false;  // no tensor map: the mma.sync kernel from here on
        return false;
    }
    if (set_smem_attrs(n->dev) != cudaSuccess) *st = LBM_ECUDA;
    return true;
}


// loss and gradient into n->g (device) on the mma.sync kernel, after forward_ms()
lbm_status backward_ms(lbm_mlp* n, const float* t, int B) {
    cudaStream_t s = n->stream;
    CK(cudaMemsetAsync(n->sse, 0, sizeof(double), s));
    const int total = B * kOut;
    k_loss_grad<<<(total + 255) / 256 < 1024 ? (total + 255) / 256 : 1024, 256, 0, s>>>(
        n->a32[kLayers - 1], t, total, 1.0f / (float)total, n->d32, n->sig[1], n->sse);
    CK(cudaGetLastError());
    float* d32 = n->d32;
    __nv_bfloat16* d16 = n->sig[1];
    float* e32 = n->e32;
    __nv_bfloat16* e16 = n->sig[0];
    for (int l = kLayers - 1; l >= 0; --l) {
        const int fi = kFanIn[l], fo = kFanOut[l];
        float* gw = n->g + param_offset(l);
        float* gb = gw + (long long)fi * fo;
        // dW = A_{l-1}^T D (the input layer's padded columns are not kept)
        GemmArgs g{};
        g.A = l == 0 ? n->x16 : n->a16[l - 1];
        g.sam = 1;
        g.sak = l == 0 ? kK0 : kW;
        g.B = d16;
        g.sbk = fo;
        g.sbn = 1;
        g.M = fi;
        g.N = fo;
        g.K = B;
        g.epi = EPI_STORE;
        g.out32 = gw;
        CK(gemm(g, s));
        k_bias_grad<<<(fo + 127) / 128, 128, 0, s>>>(d32, B, fo, gb);
        CK(cudaGetLastError());
        if (l == 0) break;
        // D_{l-1} = (D W_l^T) (1 - A_{l-1}^2)
        GemmArgs h{};
        h.A = d16;
        h.sam = fo;
        h.sak = 1;
        h.B = w16_of(n, l);
        h.sbk = 1;
        h.sbn = fo;
        h.M = B;
        h.N = fi;
        h.K = fo;
        h.epi = EPI_TANH_BACK;
        h.aprev = n->a32[l - 1];
        h.out32 = e32;
        h.out16 = e16;
        h.ld16 = fi;
        CK(gemm(h, s));
        std::swap(d32, e32);
        std::swap(d16, e16);
    }
    return LBM_OK;
}

lbm_status refresh_w16(lbm_mlp* n) {
    k_weights16<<<(unsigned)((kParams + 255) / 256), 256, 0, n->stream>>>(n->p, n->w16, n->w16t);
    CK(cudaGetLastError());
    return LBM_OK;
}

// Forward and backward pass of a batch, then one of: the gradient into d_grad, the
// gradient kept inside (d_grad null), an Adam step (lr > 0); and the loss (h_loss not
// null, which waits).
lbm_status train(lbm_mlp* n, const float* x, const float* t, int B, float lr, float* d_grad,
                 double* h_loss) {
    if (!n || !x || !t || B < 1 || B > n->max_batch) return LBM_EINVAL;
    CK(cudaSetDevice(n->dev));
    lbm_status st = LBM_OK;
    const bool tc = use_tc(n, B, &st);
    if (st) return st;
    auto loss = [&]() -> lbm_status {
        if (!h_loss) return LBM_OK;
        const lbm_status w = sync(n);
        if (w) return w;
        *h_loss = *n->h_sse / ((double)B * kOut);
        return LBM_OK;
    };
    float c1 = 0.0f, c2 = 0.0f;
    auto corrections = [&] {
        n->step += 1;
        c1 = (float)(1.0 - std::pow(0.9, (double)n->step));
        c2 = (float)(1.0 - std::pow(0.999, (double)n->step));
    };
    if (tc) {
        st = rows_pass(n, x, B, t, nullptr);
        if (!st) st = wgrad_tc(n, B);
        if (!st && !(lr > 0)) st = gradient_tc(n, B, d_grad ? d_grad : n->g, 0.0f, 0.0f, 0.0f);
        if (!st) st = loss();  // (a wait that ran out is reported before the step is taken)
        if (st || !(lr > 0)) return st;
        corrections();
        return gradient_tc(n, B, nullptr, lr, c1, c2);
    }
    st = forward_ms(n, x, B);
    if (!st) st = backward_ms(n, t, B);
    if (st) return st;
    if (d_grad)
        CK(cudaMemcpyAsync(d_grad, n->g, kParams * 4, cudaMemcpyDeviceToDevice, n->stream));
    st = loss();
    if (st || !(lr > 0)) return st;
    corrections();
    k_adam<<<592, 256, 0, n->stream>>>(n->p, n->g, n->m, n->v, kParams, lr, c1, c2);
    CK(cudaGetLastError());
    return refresh_w16(n);
}

}  // namespace

extern "C" {

int64_t lbm_mlp_param_count(void) { return kParams; }

size_t lbm_mlp_workspace_bytes(int32_t max_batch) {
    if (max_batch < 1 || max_batch > (1 << 20)) return 0;
    return mlp_layout(max_batch).total;
}

lbm_status lbm_mlp_init(lbm_mlp** out, int32_t max_batch, void* d_ws, size_t bytes,
                        void* stream) {
    if (!out) return LBM_EINVAL;
    *out = nullptr;
    if (max_batch < 1 || max_batch > (1 << 20) || !d_ws || ((uintptr_t)d_ws % 256))
        return LBM_EINVAL;
    const MlpLayout L = mlp_layout(max_batch);
    if (bytes < L.total) return LBM_ENOMEM;
    lbm_mlp* n = new (std::nothrow) lbm_mlp();
    if (!n) return LBM_ENOMEM;
    if (cudaGetDevice(&n->dev) != cudaSuccess) {
        delete n;
        return LBM_ECUDA;
    }
    char* w = (char*)d_ws;
    n->max_batch = max_batch;
    n->stream = (cudaStream_t)stream;
    n->p = (float*)(w + L.p);
    n->g = (float*)(w + L.g);
    n->m = (float*)(w + L.m);
    n->v = (float*)(w + L.v);
    n->w16 = (__nv_bfloat16*)(w + L.w16);
    n->w16t = (__nv_bfloat16*)(w + L.w16t);
    n->x16 = (__nv_bfloat16*)(w + L.x16);
    n->R = rows_of(max_batch);
    const size_t R = (size_t)n->R;
    for (int l = 0; l < kLayers; ++l) n->a32[l] = (float*)(w + L.a32) + (size_t)l * R * kW;
    for (int l = 0; l < kLayers - 1; ++l)
        n->a16[l] = (__nv_bfloat16*)(w + L.a16) + (size_t)l * R * kW;
    for (int l = 0; l < kLayers; ++l) n->sig[l] = (__nv_bfloat16*)(w + L.sig) + (size_t)l * R * kW;
    n->d32 = (float*)(w + L.d32);
    n->e32 = (float*)(w + L.e32);
    n->part = (float*)(w + L.part);
    n->bpart = (float*)(w + L.bpart);
    n->sse = (double*)(w + L.sse);
    n->err = (int*)(n->sse + 1);
    n->sse_part = (double*)(w + L.sse_part);
    n->step = 0;
    n->tensor_cores = true;
    if (cudaDeviceGetAttribute(&n->nsm, cudaDevAttrMultiProcessorCount, n->dev) != cudaSuccess ||
        n->nsm < 1) {
        delete n;
        return LBM_ECUDA;
    }
    if (cudaMallocHost((void**)&n->h_sse, 16) != cudaSuccess) {
        delete n;
        return LBM_ECUDA;
    }
    n->h_err = (int*)(n->h_sse + 1);
    if (cudaMemsetAsync(w, 0, L.total, n->stream) != cudaSuccess) {
        lbm_mlp_free(n);
        return LBM_ECUDA;
    }
    *out = n;
    return LBM_OK;
}

lbm_status lbm_mlp_set_tcgen05(lbm_mlp* n, int32_t on) {
    if (!n || (on != 0 && on != 1)) return LBM_EINVAL;
    n->tensor_cores = on == 1;
    return LBM_OK;
}

int32_t lbm_mlp_tcgen05(const lbm_mlp* n) { return n ? (n->tensor_cores ? 1 : 0) : -1; }

void lbm_mlp_free(lbm_mlp* n) {
    if (!n) return;
    cudaSetDevice(n->dev);
    if (n->h_sse) cudaFreeHost(n->h_sse);
    delete n;
}

lbm_status lbm_mlp_set_params(lbm_mlp* n, const float* h_params) {
    if (!n || !h_params) return LBM_EINVAL;
    CK(cudaSetDevice(n->dev));
    CK(cudaMemcpyAsync(n->p, h_params, kParams * 4, cudaMemcpyHostToDevice, n->stream));
    CK(cudaMemsetAsync(n->m, 0, kParams * 4, n->stream));
    CK(cudaMemsetAsync(n->v, 0, kParams * 4, n->stream));
    n->step = 0;
    lbm_status st = refresh_w16(n);
    if (st) return st;
    return sync(n);
}

lbm_status lbm_mlp_get_params(lbm_mlp* n, float* h_params) {
    if (!n || !h_params) return LBM_EINVAL;
    CK(cudaSetDevice(n->dev));
    CK(cudaMemcpyAsync(h_params, n->p, kParams * 4, cudaMemcpyDeviceToHost, n->stream));
    return sync(n);
}

lbm_status lbm_mlp_forward(lbm_mlp* n, const float* d_x, int32_t batch, float* d_y) {
    if (!n || !d_x || !d_y || batch < 1 || batch > n->max_batch) return LBM_EINVAL;
    CK(cudaSetDevice(n->dev));
    lbm_status st = LBM_OK;
    if (use_tc(n, batch, &st)) return st ? st : rows_pass(n, d_x, batch, nullptr, d_y);
    if (st) return st;
    st = forward_ms(n, d_x, batch);
    if (st) return st;
    CK(cudaMemcpyAsync(d_y, n->a32[kLayers - 1], (size_t)batch * kOut * 4,
                       cudaMemcpyDeviceToDevice, n->stream));
    return LBM_OK;
}

lbm_status lbm_mlp_loss_grad(lbm_mlp* n, const float* d_x, const float* d_t, int32_t batch,
                             double* h_loss, float* d_grad) {
    return train(n, d_x, d_t, batch, 0.0f, d_grad, h_loss);
}

lbm_status lbm_mlp_train_step(lbm_mlp* n, const float* d_x, const float* d_t, int32_t batch,
                              float lr, double* h_loss) {
    if (!n || !(lr > 0)) return LBM_EINVAL;
    return train(n, d_x, d_t, batch, lr, nullptr, h_loss);
}

}  // extern "C"
