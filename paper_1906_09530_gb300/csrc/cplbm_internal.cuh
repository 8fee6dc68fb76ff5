// cplbm_internal.cuh -- shared declarations of the CUDA library (device
// kernels, launchers and the context).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/cplbm.h"

#include <utility>

namespace cplbm {

// ---- programmatic dependent launch (the single-instance mixed step) --------
// The kernels of a mixed step are each about one wave at small grids, so the gap
// between one kernel's last blocks and the next kernel's first is a visible part
// of the step.  Launched with the programmatic-serialization attribute, a kernel
// lets the next one be scheduled once all of its own blocks have started
// (launch_dependents), and waits, before touching memory, until the previous
// kernel has completed and its writes are visible (wait).  The next kernel's
// blocks thus become resident during this one's tail instead of after it.  Both
// instructions are no-ops for a kernel launched without the attribute.
__device__ __forceinline__ void pdl_prologue() {
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

// Whether launch_pdl sets the attribute: chosen per context by whoever enqueues
// (the host thread that enqueues a step sets it first; enqueueing is synchronous).
bool& launch_pdl_on();

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = launch_pdl_on() ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// Lets launches of a kernel have up to `most` bytes of dynamic shared memory.  The limit is
// state of the device, which the launches of all grids, contexts and host threads share: every
// caller gives the most that any grid needs of that kernel, never its own grid's size, so that
// no thread lowers the limit between another's call and its launch.  (Also below 48 KB, which
// need no telling only if the kernel's static arrays fit in them too.)
template <class K>
cudaError_t allow_smem(K kern, size_t most) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// Device-resident state block (one per context, inside the workspace).
struct DevState {
    int64_t t;              // time level of the populations in f[cur]
    unsigned int flag;      // error bits, see FLAG_*
    unsigned int pad0;
    unsigned long long failed_t;  // smallest flagged time level (ULLONG_MAX: none)
    double diag[4];         // mass, max|v|, rho_min, rho_max
};

enum : unsigned int {
    FLAG_RHO = 1u,   // collide-stream: rho <= 0 or not finite
    FLAG_EOS = 2u,   // EOS pass: rho <= 0, the EOS pole with the upper limit off,
                     // or mu not finite
    FLAG_STAGE = 4u, // a line window's tensor copy did not arrive within the
                     // bounded wait (the block gave up; the step is void)
};

// Physical parameters the kernels need.
struct PhysParams {
    int eos;             // LBM_EOS_* (Sec. 3.2)
    double alpha;        // alpha(T) of Eqs. 16-19 at this T (1 for CS and VDW)
    double T, a, b, R;   // EOS constants, T absolute
    double k2;           // k^2 (Eq. 33)
    double kappa;        // kappa-hat (Eq. 33)
    double omega;        // 1 / tau (Eq. 1)
    double mu_cap;       // k^2 * mu_max (mesh-space limit, Sec. 5.6)
    int64_t cap_steps;   // limit active while t < cap_steps
};

// MRT relaxation rates of Eq. 4 other than s_v = 1/tau (NULL pointer: BGK).
struct MrtRates {
    double se, seps, sq;
};

// Solid walls below row 0 and above row ny-1 (Sec. 5.5), halfway bounce-back;
// u: the x-velocities of the bottom and the top wall (a moving frame).
struct Walls {
    bool on = false;
    double u[2] = {0.0, 0.0};
};

// Launchers (all asynchronous on `s`).  FP64 path: fields are [ny][nx], populations
// [9][plane] with plane >= nx*ny.
cudaError_t launch_collide_stream(const double* fin, double* fout, const double* Fx,
                                  const double* Fy, const double* rho, int nx, int ny,
                                  size_t plane, double omega, const MrtRates* mrt, DevState* st,
                                  cudaStream_t s, const Walls& walls = Walls());
cudaError_t launch_init_feq(const double* rho, const double* ux, const double* uy, double* f,
                            int nx, int ny, size_t plane, cudaStream_t s);
cudaError_t launch_macro(const double* f, const double* rho, const double* Fx, const double* Fy,
                         double* vx, double* vy, int nx, int ny, size_t plane, cudaStream_t s);
cudaError_t launch_diag(const double* f, const double* rho, const double* Fx, const double* Fy,
                        int nx, int ny, size_t plane, double* partials, int nparts,
                        DevState* st, cudaStream_t s);
// FP32 populations <-> FP64 host layout
cudaError_t launch_f_to_double(const float* f, double* out, size_t n, cudaStream_t s);
cudaError_t launch_f_from_double(const double* in, float* f, size_t n, cudaStream_t s);

cudaError_t launch_diag_final(const double* partials, int nparts, DevState* st, cudaStream_t s);

// ---- mixed precision path (kernels_mixed.cu) ------------------------------
// ring_rows: -1 = the sliding-window kernel; 0 = the row-ring kernel where the
// grid allows it (periodic, nx a multiple of 4 and >= 128, aligned planes), with
// its default rows a block; > 0 = the row-ring kernel with that many rows a block
cudaError_t launch_cs_mixed(const float* fin, float* fout, const float* Fx, const float* Fy,
                            float* rh, float* rl, int nx, int ny, size_t plane, double omega,
                            const MrtRates* mrt, DevState* st, cudaStream_t s,
                            const Walls& walls = Walls(), int ring_rows = -1);
// whether launch_cs_mixed with these arguments runs the row-ring kernel
bool cs_ring_used(int nx, int ny, size_t plane, const void* fin, const void* Fx,
                  const void* Fy, bool walls, int ring_rows);
cudaError_t launch_init_mixed(const double* rho, const double* ux, const double* uy, float* f,
                              float* rh, float* rl, int nx, int ny, size_t plane,
                              cudaStream_t s);
cudaError_t launch_rho_from_f_mixed(const float* f, float* rh, float* rl, int nx, int ny,
                                    size_t plane, cudaStream_t s);
cudaError_t launch_macro_mixed(const float* f, const float* rh, const float* rl,
                               const float* Fx, const float* Fy, const float* mu, double* rho,
                               double* vx, double* vy, double* mu_out, int nx, int ny,
                               size_t plane, cudaStream_t s);
cudaError_t launch_diag_mixed(const float* f, const float* rh, const float* rl, const float* Fx,
                              const float* Fy, int nx, int ny, size_t plane, double* partials,
                              int nparts, DevState* st, cudaStream_t s);

// ---- batched mixed path: per-instance argument blocks -----------------------
// A batch runs many independent instances (each its own grid, temperature,
// tau, k, kappa and state block) through the same four passes, one launch per
// pass for the whole batch.  Every launch reads, per block, the instance index
// from a block map and that instance's argument block; inside an instance the
// work is the single-instance kernel's, block for block.

// Collide-stream arguments of one instance (mixed path).
struct CsArgs {
    const float* fin;
    float* fout;
    const float* Fx;
    const float* Fy;
    float* rh;
    float* rl;
    int nx, ny;
    size_t plane;
    float omega;
    int nstrips, nseg, rows;  // warp strips of 30 columns x `rows` rows
    DevState* st;
    int mrt;                  // 0: BGK (Eq. 1); 1: MRT (Eq. 4) with the rates below
    float se, seps, sq;
    int walls;                // 1: halfway bounce-back below row 0 and above row ny-1
    float uw6[2];             // bottom / top wall x-velocity over 6 (moving walls)
};
struct CsBatchInst {
    CsArgs a;      // fin / fout are taken from f[] by the launch's `from`
    float* f[2];
    int blk0;      // first block of this instance in the launch
};
// FP32 constants of the chemical potential, converted on the host: FP64 -> FP32
// conversions run on the FP64 pipe, which a per-thread conversion would make the
// bottleneck of the pointwise kernel.
template <class T>
struct EosC {
    int kind;   // LBM_EOS_*
    T rt;       // R T
    T a2;       // 2 a (CS, VDW)
    T b;        // b (cubic EOSs) or b / 4 (CS)
    T aal;      // a alpha(T) (RK, RKS, PR)
    T clog;     // a alpha / b (RK, RKS) or a alpha / (2 sqrt 2 b) (PR)
};
struct MuConstF {
    EosC<float> e;
    float k2, kappa, cap;
    long long cap_steps;
};
// The EOS constants of PhysParams in arithmetic T (host).
template <class T>
EosC<T> eos_const(const PhysParams& p) {
    EosC<T> c;
    c.kind = p.eos;
    c.rt = (T)(p.R * p.T);
    c.a2 = (T)(2 * p.a);
    c.b = (T)(p.eos == LBM_EOS_CS ? 0.25 * p.b : p.b);
    c.aal = (T)(p.a * p.alpha);
    c.clog = (T)(p.eos == LBM_EOS_PR ? p.a * p.alpha / (2 * 1.4142135623730951 * p.b)
                                     : p.a * p.alpha / p.b);
    return c;
}
constexpr int kMuBatchT = 128;  // threads per block of the batched mu-hat pass (4 nodes each)
struct MuBatchInst {
    const float* rh;
    float* mu;  // holds d_xx rho on entry
    const float* dyy;
    size_t N;
    MuConstF c;
    DevState* st;
    int blk0;
};
// Pointers and sizes of one instance's mixed fields, for the batched line passes.
struct MixedLinesView {
    const float* rh;
    const float* rl;
    float *dxr, *dyr, *dxx, *dyy;  // dxx holds mu-hat after the mu pass
    float *Fx, *Fy;
    int nx, ny;
    DevState* st;
};

CsArgs cs_mixed_args(const float* fin, float* fout, const float* Fx, const float* Fy,
                     float* rh, float* rl, int nx, int ny, size_t plane, double omega,
                     const MrtRates* mrt, DevState* st,
                     int rows,  // 0: the default of a batch member, < 0: of a lone grid
                     const Walls& walls = Walls());
int cs_mixed_blocks(const CsArgs& a);
cudaError_t launch_cs_mixed_args(const CsArgs& a, cudaStream_t s);
cudaError_t launch_cs_mixed_batch(const CsBatchInst* d, const int* map, int nblocks, int from,
                                  bool mrt, cudaStream_t s);
MuConstF mu_mixed_const(const PhysParams& p);
cudaError_t launch_mu_mixed_batch(const MuBatchInst* d, const int* map, int nblocks,
                                  cudaStream_t s);
// ---- FP32 line solves (lines32.cuh, lines32.cu) ----
constexpr int kC32 = 19;  // positions of a chunk (odd: chunk starts hit distinct banks)
// One direction's windows; see lines32.cuh.
struct Geo32 {
    int n, nlines;            // line length, lines
    long long ps, ls;         // stride along a line, between lines
    int H, own, nwin;         // halo, owned positions of a window, windows a line
    int nch;                  // chunks solved of a window's 32
    int nl, ngroups;          // lines a block, line groups
    int vec;                  // nx a multiple of 4: 16-byte pieces
    int period, mirror;       // n, or 2 n with positions n .. 2n-1 reading 2n-1-p (walls)
    int lift;                 // multiple of the period that makes window starts positive
    unsigned magic;           // ceil(2^32 / period) for periods shorter than a window, else 0
};
struct Dir32 {
    Geo32 g;
    const float* u;           // the field solved (density, or mu-hat)
    const float* ul;          // its low part (double-float solves)
    const float *rho, *dr;    // force: density and its derivative along the line
    float *o1, *o2;           // first and second derivative, or the force
};
struct Lines32Inst {          // one instance of a batch
    Dir32 x, y;
    int nbx, blk0;            // x-line blocks, first block in the launch
    DevState* st;
};
cudaError_t lines32_rho(const float* rh, float* dxr, float* dxx, float* dyr, float* dyy, int nx,
                        int ny, int order, DevState* st, int bump, cudaStream_t s,
                        bool walls_y = false);
cudaError_t lines32_force(const float* mu, const float* rh, const float* dxr, const float* dyr,
                          float* Fx, float* Fy, int nx, int ny, int order, DevState* st,
                          cudaStream_t s, bool walls_y = false);
// Grids whose FP32 lines are solved by (line, chunk) pairs; larger ones take full windows
// (lines32_wide.cu), which lines32_rho and lines32_force dispatch to.
constexpr long long kLines32Nodes = 1LL << 19;
cudaError_t lines32_wide(Dir32 x, Dir32 y, int nx, int ny, int order, bool second, DevState* st,
                         int bump, cudaStream_t s);
// adds the windows (one line each) of a grid's density lines, and the chunks of them, of 32 a
// window, that (line, chunk) pairs solve
void lines32_window_use(int nx, int ny, int order, long long& chunks, long long& windows);
// Batches: nl (8 or 16): blocks of 32 nl threads; wide: full windows, nl lines a block
int lines32_batch_blocks(int nx, int ny, int order, bool second, int nl, bool wide);
Lines32Inst lines32_batch_inst(const MixedLinesView& v, int order, bool second, int blk0, int nl,
                               bool wide);
cudaError_t lines32_batch_launch(const Lines32Inst* d, const int* map, int nblocks, int order,
                                 bool second, int bump, int nl, bool wide, cudaStream_t s);
void lines32_wide_divide(Dir32& x, Dir32& y, int nl);
cudaError_t lines32_wide_batch(const Lines32Inst* d, const int* map, int nblocks, int order,
                               bool second, int bump, int nl, cudaStream_t s);

// Double-float density lines (lines_df.cu): x and y in one launch, stand-alone, batches.
cudaError_t lines_df_rho(const float* rh, const float* rl, float* dxr, float* dxx, float* dyr,
                         float* dyy, int nx, int ny, int order, DevState* st, int bump,
                         cudaStream_t s, bool walls_y = false);
cudaError_t lines_df_plain(const float* uh, const float* ul, float* d1, float* d2, int nx, int ny,
                           int axis, int order, cudaStream_t s);
int lines_df_batch_blocks(int nx, int ny, int order);
Lines32Inst lines_df_batch_inst(const MixedLinesView& v, int order, int blk0);
// smem: the largest lines_df_batch_smem of the batch's instances.  (Short lines stage the most,
// 79 KB a block, of which an SM holds two: 16 x 256^2 at ratio 8e4 took 77 us a step with it and
// 69 with the 70 of their own.)  beside: FP32 density lines run at the same time.
size_t lines_df_batch_smem(const Lines32Inst& d);
cudaError_t lines_df_batch_launch(const Lines32Inst* d, const int* map, int nblocks, int order,
                                  size_t smem, bool beside, int bump, cudaStream_t s);

// Whole steps of a small periodic grid in one launch (FP32 density lines).
struct SmallStep {
    float* f[2];
    MixedLinesView v;
    size_t plane;
    PhysParams phys;
    const MrtRates* mrt;
    int order;
};
constexpr long long kSmallNodes = 1 << 13;  // largest grid it is used for
constexpr int64_t kSmallSteps = 512;        // steps a launch (a few milliseconds)
// whether the grid and the device allow it (also makes the kernel ready to launch)
bool small_steps_fit(const SmallStep& p);
cudaError_t launch_small_steps(const SmallStep& p, int from, int64_t steps, cudaStream_t s);

// Below this Maxwell density ratio the mixed path solves the density's lines in
// FP32 (measured: coexistence densities within 2e-4 of the FP64 path); at and
// above it, in double-float wherever a window spans more than a factor 32.
constexpr double kDfRatio = 1e4;

// Compact-FD line solves.  With walls_y the y-lines are extended evenly about both
// walls (a periodic line of period 2 ny, the first ghost equal to its fluid neighbour,
// Sec. 5.5).  axis 0: lines along x, 1: along y.
// FP64 path (lines64.cu).  z: a derivative without its factor c1 (c1^2 for a second one).
// The x-lines take the density as the sum of the populations and store it.
cudaError_t lines_fp64_rho_x(const double* f, size_t plane, double* rho, double* zx, double* zxx,
                             int nx, int ny, int order, DevState* st, int bump, cudaStream_t s);
cudaError_t lines_fp64_rho_y_mu(const double* rho, const double* zxx, double* zy, double* mu,
                                int nx, int ny, int order, const PhysParams& p, DevState* st,
                                cudaStream_t s, bool walls_y = false);
// the x- and y-lines of mu-hat in one launch; zx or zy null: the other direction alone
cudaError_t lines_fp64_force(const double* mu, const double* rho, const double* zx,
                             const double* zy, double* Fx, double* Fy, int nx, int ny, int order,
                             cudaStream_t s, bool walls_y = false);
cudaError_t lines_fp64_plain(const double* u, double* d1, double* d2, int nx, int ny, int axis,
                             int order, cudaStream_t s);
// mu-hat = k^2 mu0(rho) - kappa (d_xx + d_yy) rho (Eqs. 21, 33, Sec. 5.6), FP32,
// written over d_xx rho (`dxx_mu`); flags bad values.
cudaError_t launch_mu_mixed(const float* rh, float* dxx_mu, const float* dyy, int nx, int ny,
                            const PhysParams& p, DevState* st, cudaStream_t s);
// Host thermodynamics of the product library (independent of the oracle), for
// the EOS kinds LBM_EOS_* (Sec. 3.2).  Return 0 or -1 (invalid arguments, or
// T outside (0, T_c) for the Maxwell pair).
int eos_critical(int kind, double a, double b, double R, double* Tc, double* rhoc);
double eos_alpha(int kind, double a, double b, double R, double omega, double T);
int eos_maxwell(int kind, double a, double b, double R, double omega, double T,
                double* rho_g, double* rho_l);

}  // namespace cplbm
