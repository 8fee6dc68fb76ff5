// capi_batch.cu -- the batched C ABI (lbm_batch_* of include/cplbm.h): many
// independent periodic instances of the mixed path, each with its own grid and
// physical parameters, advanced together.
//
// Each instance keeps the single-instance layout (two FP32 population buffers,
// eight FP32 field planes, reduction partials) in its own region of the
// caller's workspace; a table region follows with, per pass, one argument block
// per instance and a block map (block -> instance), plus the instances' device
// state blocks side by side.  A time step is four launches for the whole batch:
//   collide-stream | x|y lines of rho | mu-hat | x|y lines of mu-hat + force
// and lbm_batch_step replays two steps as one CUDA graph.  Blocks are assigned
// to instances in decreasing order of instance size, so the long-running work
// of the large grids starts first.
#include <algorithm>
#include <chrono>
#include <climits>
#include <cmath>
#include <cstring>
#include <map>
#include <new>
#include <thread>
#include <utility>
#include <vector>

#include "cplbm_internal.cuh"

using namespace cplbm;

namespace {

constexpr size_t kAlign = 256;
constexpr int kParts = 256;  // diagnostic partial records per instance
constexpr int kRowChoices[] = {4, 8, 16, 32};  // collide-stream strip heights

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct InstHost {
    int nx, ny;
    size_t N, plane;
    PhysParams phys;
    size_t off;  // region offset in the workspace
    float* f[2];
    float *rh, *rl, *dxr, *dyr, *dxx, *dyy, *Fx, *Fy;
    double* partials;
    int64_t t;
    bool ready;
    bool rho_df;  // density lines in double-float (else FP32), as for a lone context
    int rows;     // collide-stream strip height (0: the single-instance default)
};

// the density's low part, where the line solves read it (null: not kept by the steps)
float* rl_of(const InstHost& h) { return h.rho_df ? h.rl : nullptr; }

struct Region {
    size_t plane, f_bytes, field_bytes, parts_off, total;
};

Region region(int nx, int ny) {
    Region r;
    r.plane = align_up((size_t)nx * ny, 64);
    r.f_bytes = align_up(9 * r.plane * sizeof(float), kAlign);
    r.field_bytes = align_up(r.plane * sizeof(float), kAlign);
    r.parts_off = 2 * r.f_bytes + 8 * r.field_bytes;
    r.total = r.parts_off + align_up(4 * kParts * sizeof(double), kAlign);
    return r;
}

// Block counts of each pass for one instance.
int cs_blocks_for(int nx, int ny, int rows) {
    return cs_mixed_blocks(cs_mixed_args(nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                                         nx, ny, 0, 1.0, nullptr, nullptr, rows));
}
int mu_blocks_for(size_t N) { return (int)(((N + 3) / 4 + kMuBatchT - 1) / kMuBatchT); }

// Whether a batch solves its FP32 lines in full windows (lines32_wide.cu) instead of by (line,
// chunk) pairs, which saves chunks and spreads over more threads: with a grid above
// kLines32Nodes; and where all rows are whole 16-byte pieces (else it always lost: 24 odd
// members up to 400^2 63 us a step against 73), if most chunks are needed (16 of 512^2 147 us
// by pairs and 140 in windows, 24 members up to 512^2 that use 84 of 100 chunks 111 and 109;
// 24 that use 67 of 100 64 and 66, 256 of 128^2 174 and 233), or if the launch is about one
// round of blocks, where a full window is done no later than a part of one (one 700^2 28.2
// and 26.1, 8 members up to 400^2 28.4 and 25.3, 4 up to 256^2 20.2 and 18.0).
bool wide_lines(const lbm_instance* inst, int n, int order) {
    constexpr long long kRound = 4 * 152 * 8;  // windows of one line
    long long chunks = 0, windows = 0;
    bool vec = true;
    for (int i = 0; i < n; ++i) {
        const int nx = inst[i].grid.nx, ny = inst[i].grid.ny;
        if ((long long)nx * ny > kLines32Nodes) return true;
        vec = vec && nx % 4 == 0;
        lines32_window_use(nx, ny, order, chunks, windows);
    }
    return vec && (windows <= kRound || 10 * chunks >= 8 * 32 * windows);
}

// Offsets of the table region, sized for the largest block counts (the
// smallest strip height) so that autotuning never needs more room.
struct Tables {
    size_t cs, mu, rho_df, rho_f32, force, state;
    size_t map_cs, map_mu, map_rho_df, map_rho_f32, map_force, end;
    int nb_cs, nb_mu, nb_rho_df, nb_rho_f32, nb_force;  // current counts
    size_t smem_df;  // shared memory of a block of the double-float density lines
};

Tables table_layout(const lbm_instance* inst, int n, int order, size_t base) {
    // each density map is sized for every instance in it (the double-float
    // windows are the shorter ones, so their count bounds both kinds)
    long long cs_max = 0, mu = 0, rho = 0, force = 0;
    const bool wide = wide_lines(inst, n, order);
    for (int i = 0; i < n; ++i) {
        const int nx = inst[i].grid.nx, ny = inst[i].grid.ny;
        cs_max += cs_blocks_for(nx, ny, kRowChoices[0]);
        mu += mu_blocks_for((size_t)nx * ny);
        rho += std::max(lines_df_batch_blocks(nx, ny, order),
                        lines32_batch_blocks(nx, ny, order, true, 8, wide));
        force += lines32_batch_blocks(nx, ny, order, false, 8, wide);
    }
    Tables t;
    size_t o = base;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = align_up(o + bytes, kAlign);
        return at;
    };
    t.cs = take(n * sizeof(CsBatchInst));
    t.mu = take(n * sizeof(MuBatchInst));
    t.rho_df = take(n * sizeof(Lines32Inst));
    t.rho_f32 = take(n * sizeof(Lines32Inst));
    t.force = take(n * sizeof(Lines32Inst));
    t.state = take(n * sizeof(DevState));
    t.map_cs = take(cs_max * sizeof(int));
    t.map_mu = take(mu * sizeof(int));
    t.map_rho_df = take(rho * sizeof(int));
    t.map_rho_f32 = take(rho * sizeof(int));
    t.map_force = take(force * sizeof(int));
    t.end = o;
    t.nb_cs = t.nb_mu = t.nb_rho_df = t.nb_rho_f32 = t.nb_force = 0;
    t.smem_df = 0;
    return t;
}

bool instance_ok(const lbm_instance& in) {
    return in.grid.nx >= 8 && in.grid.ny >= 8 && in.T_r > 0 && in.T_r < 1 && in.kappa > 0 &&
           in.tau > 0.5 && in.mesh_coeff > 0 && in.mesh_coeff <= 1 && !std::isnan(in.mu_max) &&
           (size_t)in.grid.nx * in.grid.ny <= (size_t)1 << 31;
}

#define CK(call)                                  \
    do {                                          \
        cudaError_t e_ = (call);                  \
        if (e_ != cudaSuccess) return LBM_ECUDA;  \
    } while (0)

}  // namespace

struct lbm_batch {
    int dev, n, order;
    bool mrt;  // MRT collision (Eq. 4) for every instance
    bool wide;  // FP32 lines in full windows
    MrtRates rates;
    cudaStream_t stream, cap_stream, side_stream;  // the last two for graph capture only
    cudaEvent_t ev, tev[5], fork_ev, join_ev;
    char* ws;
    std::vector<InstHost> inst;
    std::vector<int> order_by_size;  // instance indices, largest grid first
    Tables tb;
    DevState* dst;  // n state blocks, device
    DevState* hst;  // pinned host mirror
    int cur;
    int line_nl;  // lines per block of the FP32 line launches (8 or 16)
    cudaGraphExec_t graph[2];
    double timeout_s;
    int failed_inst;
    int64_t failed_step;
};

namespace {

lbm_status wait_stream(lbm_batch* b) {
    CK(cudaEventRecord(b->ev, b->stream));
    const auto t0 = std::chrono::steady_clock::now();
    for (;;) {
        cudaError_t q = cudaEventQuery(b->ev);
        if (q == cudaSuccess) return LBM_OK;
        if (q != cudaErrorNotReady) return LBM_ECUDA;
        const double el =
            std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        if (el > b->timeout_s) return LBM_ETIMEOUT;
        // a sleep of 5 us takes about 60: short waits are polled through
        if (el > 3e-4)
            std::this_thread::sleep_for(std::chrono::microseconds(el < 0.01 ? 5 : 200));
    }
}

void drop_graphs(lbm_batch* b) {
    for (int i = 0; i < 2; ++i)
        if (b->graph[i]) {
            cudaGraphExecDestroy(b->graph[i]);
            b->graph[i] = nullptr;
        }
}

MixedLinesView view_of(const lbm_batch* b, int i) {
    const InstHost& h = b->inst[i];
    return MixedLinesView{h.rh, h.rl, h.dxr, h.dyr, h.dxx, h.dyy, h.Fx, h.Fy, h.nx, h.ny,
                          b->dst + i};
}

// Write every pass's argument blocks and block maps to the workspace.
lbm_status upload_tables(lbm_batch* b) {
    Tables& t = b->tb;
    const int n = b->n;
    std::vector<CsBatchInst> cs(n);
    std::vector<MuBatchInst> mu(n);
    std::vector<Lines32Inst> rdf(n), rf(n), force(n);
    std::vector<int> mcs, mmu, mrdf, mrf, mforce;
    for (int i : b->order_by_size) {
        const InstHost& h = b->inst[i];
        DevState* st = b->dst + i;
        CsBatchInst c;
        c.a = cs_mixed_args(h.f[0], h.f[1], h.Fx, h.Fy, h.rh, rl_of(h), h.nx, h.ny, h.plane,
                            h.phys.omega, b->mrt ? &b->rates : nullptr, st, h.rows);
        c.f[0] = h.f[0];
        c.f[1] = h.f[1];
        c.blk0 = (int)mcs.size();
        mcs.insert(mcs.end(), cs_mixed_blocks(c.a), i);
        cs[i] = c;

        MuBatchInst m{h.rh, h.dxx, h.dyy, h.N, mu_mixed_const(h.phys), st, (int)mmu.size()};
        mmu.insert(mmu.end(), mu_blocks_for(h.N), i);
        mu[i] = m;

        const MixedLinesView v = view_of(b, i);
        if (h.rho_df) {
            rdf[i] = lines_df_batch_inst(v, b->order, (int)mrdf.size());
            t.smem_df = std::max(t.smem_df, lines_df_batch_smem(rdf[i]));
            mrdf.insert(mrdf.end(), lines_df_batch_blocks(h.nx, h.ny, b->order), i);
        } else {
            rf[i] = lines32_batch_inst(v, b->order, true, (int)mrf.size(), b->line_nl, b->wide);
            mrf.insert(mrf.end(),
                       lines32_batch_blocks(h.nx, h.ny, b->order, true, b->line_nl, b->wide), i);
        }
        force[i] = lines32_batch_inst(v, b->order, false, (int)mforce.size(), b->line_nl, b->wide);
        mforce.insert(mforce.end(),
                      lines32_batch_blocks(h.nx, h.ny, b->order, false, b->line_nl, b->wide), i);
    }
    // the table region was sized for the largest counts
    const size_t cap_cs = (t.map_mu - t.map_cs) / sizeof(int);
    if (mcs.size() > cap_cs) return LBM_ENOMEM;
    t.nb_cs = (int)mcs.size();
    t.nb_mu = (int)mmu.size();
    t.nb_rho_df = (int)mrdf.size();
    t.nb_rho_f32 = (int)mrf.size();
    t.nb_force = (int)mforce.size();
    cudaStream_t s = b->stream;
    char* ws = b->ws;
    auto put = [&](size_t off, const void* src, size_t bytes) {
        return bytes ? cudaMemcpyAsync(ws + off, src, bytes, cudaMemcpyHostToDevice, s)
                     : cudaSuccess;
    };
    CK(put(t.cs, cs.data(), n * sizeof(CsBatchInst)));
    CK(put(t.mu, mu.data(), n * sizeof(MuBatchInst)));
    CK(put(t.rho_df, rdf.data(), n * sizeof(Lines32Inst)));
    CK(put(t.rho_f32, rf.data(), n * sizeof(Lines32Inst)));
    CK(put(t.force, force.data(), n * sizeof(Lines32Inst)));
    CK(put(t.map_cs, mcs.data(), mcs.size() * sizeof(int)));
    CK(put(t.map_mu, mmu.data(), mmu.size() * sizeof(int)));
    CK(put(t.map_rho_df, mrdf.data(), mrdf.size() * sizeof(int)));
    CK(put(t.map_rho_f32, mrf.data(), mrf.size() * sizeof(int)));
    CK(put(t.map_force, mforce.data(), mforce.size() * sizeof(int)));
    // the host vectors are pageable: the copies have completed when this returns
    return wait_stream(b);
}

template <class T>
const T* at(const lbm_batch* b, size_t off) {
    return reinterpret_cast<const T*>(b->ws + off);
}

// one FP32 line pass of the whole batch: the density's, or the force's
cudaError_t f32_lines(const lbm_batch* b, bool rho, int bump, cudaStream_t s) {
    const Tables& t = b->tb;
    return lines32_batch_launch(at<Lines32Inst>(b, rho ? t.rho_f32 : t.force),
                                at<int>(b, rho ? t.map_rho_f32 : t.map_force),
                                rho ? t.nb_rho_f32 : t.nb_force, b->order, rho, bump, b->line_nl,
                                b->wide, s);
}

// `side` (while capturing): another stream, on which the double-float density lines run
// beside the FP32 ones (they are other instances'; one after the other they took 17 and 15
// us of the 24-instance batch's 92)
lbm_status enqueue_step(lbm_batch* b, cudaStream_t s, int from, cudaEvent_t* ev = nullptr,
                        cudaStream_t side = nullptr) {
    const Tables& t = b->tb;
    auto mark = [&](int i) { return ev ? cudaEventRecord(ev[i], s) : cudaSuccess; };
    CK(launch_cs_mixed_batch(at<CsBatchInst>(b, t.cs), at<int>(b, t.map_cs), t.nb_cs, from,
                             b->mrt, s));
    CK(mark(1));
    // every instance is in exactly one of the two density launches
    const bool fork = side && t.nb_rho_df > 0 && t.nb_rho_f32 > 0;
    cudaStream_t sd = fork ? side : s;
    if (fork) {
        CK(cudaEventRecord(b->fork_ev, s));
        CK(cudaStreamWaitEvent(side, b->fork_ev, 0));
    }
    CK(lines_df_batch_launch(at<Lines32Inst>(b, t.rho_df), at<int>(b, t.map_rho_df), t.nb_rho_df,
                             b->order, t.smem_df, t.nb_rho_f32 > 0, 1, sd));
    CK(f32_lines(b, true, 1, s));
    if (fork) {
        CK(cudaEventRecord(b->join_ev, side));
        CK(cudaStreamWaitEvent(s, b->join_ev, 0));
    }
    CK(mark(2));
    CK(launch_mu_mixed_batch(at<MuBatchInst>(b, t.mu), at<int>(b, t.map_mu), t.nb_mu, s));
    CK(mark(3));
    CK(f32_lines(b, false, 0, s));
    CK(mark(4));
    return LBM_OK;
}

lbm_status build_graph(lbm_batch* b, int from) {
    if (b->graph[from]) return LBM_OK;
    cudaGraph_t g = nullptr;
    CK(cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal));
    lbm_status st = enqueue_step(b, b->cap_stream, from, nullptr, b->side_stream);
    if (st == LBM_OK) st = enqueue_step(b, b->cap_stream, 1 - from, nullptr, b->side_stream);
    cudaError_t e = cudaStreamEndCapture(b->cap_stream, &g);
    if (st != LBM_OK) {
        if (g) cudaGraphDestroy(g);
        return st;
    }
    if (e != cudaSuccess) return LBM_ECUDA;
    e = cudaGraphInstantiate(&b->graph[from], g, 0);
    cudaGraphDestroy(g);
    return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

// Read all state blocks back; translate the error flags.  A flagged instance
// becomes not ready (its state is undefined until it is set again) and is not
// reported again; `include` is an instance being set, checked although not ready.
lbm_status read_states(lbm_batch* b, int include = -1) {
    CK(cudaMemcpyAsync(b->hst, b->dst, b->n * sizeof(DevState), cudaMemcpyDeviceToHost,
                       b->stream));
    lbm_status w = wait_stream(b);
    if (w != LBM_OK) return w;
    int bad = -1;
    unsigned long long bad_t = ULLONG_MAX;
    for (int i = 0; i < b->n; ++i) {
        const DevState& h = b->hst[i];
        if (!h.flag || (!b->inst[i].ready && i != include)) continue;
        b->inst[i].ready = false;
        const unsigned long long ft = h.failed_t == ULLONG_MAX ? (unsigned long long)b->inst[i].t
                                                               : h.failed_t;
        if (bad < 0 || ft < bad_t) {
            bad = i;
            bad_t = ft;
        }
    }
    if (bad >= 0) {
        b->failed_inst = bad;
        b->failed_step = (int64_t)bad_t;
        return LBM_EUNSTABLE;
    }
    return LBM_OK;
}

bool all_ready(const lbm_batch* b) {
    for (const auto& h : b->inst)
        if (!h.ready) return false;
    return true;
}

lbm_status reset_state(lbm_batch* b, int i) {
    DevState h;
    std::memset(&h, 0, sizeof(h));
    h.failed_t = ULLONG_MAX;
    b->hst[i] = h;
    CK(cudaMemcpyAsync(b->dst + i, b->hst + i, sizeof(DevState), cudaMemcpyHostToDevice,
                       b->stream));
    b->inst[i].t = 0;
    return wait_stream(b);  // the pinned mirror is reused by read_states
}

// Passes 2-4 of one instance alone (its force at its current density).
lbm_status instance_force(lbm_batch* b, int i) {
    const InstHost& h = b->inst[i];
    DevState* st = b->dst + i;
    cudaStream_t s = b->stream;
    if (h.rho_df)
        CK(lines_df_rho(h.rh, h.rl, h.dxr, h.dxx, h.dyr, h.dyy, h.nx, h.ny, b->order, st, 0, s));
    else
        CK(lines32_rho(h.rh, h.dxr, h.dxx, h.dyr, h.dyy, h.nx, h.ny, b->order, st, 0, s));
    CK(launch_mu_mixed(h.rh, h.dxx, h.dyy, h.nx, h.ny, h.phys, st, s));
    CK(lines32_force(h.dxx, h.rh, h.dxr, h.dyr, h.Fx, h.Fy, h.nx, h.ny, b->order, st, s));
    return LBM_OK;
}

}  // namespace

extern "C" {

size_t lbm_batch_workspace_bytes(const lbm_instance* inst, int32_t n, const lbm_opts* opts) {
    if (!inst || n < 1 || !opts ||
        (opts->prec != LBM_PREC_MIXED && opts->prec != LBM_PREC_MIXED_DF) ||
        (opts->fd_order != 4 && opts->fd_order != 6))
        return 0;
    size_t o = 0;
    for (int i = 0; i < n; ++i) {
        if (!instance_ok(inst[i])) return 0;
        o += region(inst[i].grid.nx, inst[i].grid.ny).total;
    }
    return table_layout(inst, n, opts->fd_order, o).end;
}

lbm_status lbm_batch_init(lbm_batch** out, const lbm_instance* inst, int32_t n,
                          const lbm_eos* eos, const lbm_opts* opts, void* d_workspace,
                          size_t ws_bytes, void* cuda_stream) {
    if (!out) return LBM_EINVAL;
    *out = nullptr;
    if (!inst || n < 1 || !opts || !eos) return LBM_EINVAL;
    if (opts->fd_order != 4 && opts->fd_order != 6) return LBM_EINVAL;
    if (opts->prec != LBM_PREC_MIXED && opts->prec != LBM_PREC_MIXED_DF) return LBM_ENOTIMPL;
    auto rate_ok = [](double r) { return r > 0 && r < 2; };
    if (!(opts->collision == LBM_COLLIDE_BGK ||
          (opts->collision == LBM_COLLIDE_MRT && rate_ok(opts->s_e) && rate_ok(opts->s_eps) &&
           rate_ok(opts->s_q))))
        return LBM_EINVAL;
    if (!(eos->kind >= LBM_EOS_CS && eos->kind <= LBM_EOS_PR && eos->a > 0 && eos->b > 0 &&
          eos->R > 0 && std::isfinite(eos->omega)))
        return LBM_EINVAL;
    for (int i = 0; i < n; ++i) {
        if (!inst[i].grid.periodic_x || !inst[i].grid.periodic_y) return LBM_ENOTIMPL;
        if (!instance_ok(inst[i])) return LBM_EINVAL;
    }
    if (!d_workspace || ((uintptr_t)d_workspace % kAlign)) return LBM_EINVAL;
    const size_t need = lbm_batch_workspace_bytes(inst, n, opts);
    if (need == 0) return LBM_EINVAL;
    if (ws_bytes < need) return LBM_ENOMEM;
    double Tc, rc;
    if (eos_critical(eos->kind, eos->a, eos->b, eos->R, &Tc, &rc)) return LBM_EINVAL;

    lbm_batch* b = new (std::nothrow) lbm_batch();
    if (!b) return LBM_ENOMEM;
    b->n = n;
    b->order = opts->fd_order;
    b->wide = wide_lines(inst, n, b->order);
    b->line_nl = 8;
    b->mrt = opts->collision == LBM_COLLIDE_MRT;
    b->rates = MrtRates{opts->s_e, opts->s_eps, opts->s_q};
    b->stream = (cudaStream_t)cuda_stream;
    b->ws = (char*)d_workspace;
    b->timeout_s = 600.0;
    b->failed_inst = -1;
    b->failed_step = -1;
    b->cur = 0;
    b->graph[0] = b->graph[1] = nullptr;
    b->cap_stream = b->side_stream = nullptr;
    b->ev = b->fork_ev = b->join_ev = nullptr;
    for (auto& e : b->tev) e = nullptr;
    b->hst = nullptr;
    if (cudaGetDevice(&b->dev) != cudaSuccess) {
        delete b;
        return LBM_ECUDA;
    }
    b->inst.resize(n);
    size_t o = 0;
    for (int i = 0; i < n; ++i) {
        InstHost& h = b->inst[i];
        const lbm_instance& in = inst[i];
        const Region r = region(in.grid.nx, in.grid.ny);
        h.nx = in.grid.nx;
        h.ny = in.grid.ny;
        h.N = (size_t)h.nx * h.ny;
        h.plane = r.plane;
        h.off = o;
        char* base = b->ws + o;
        h.f[0] = (float*)base;
        h.f[1] = (float*)(base + r.f_bytes);
        float* fields = (float*)(base + 2 * r.f_bytes);
        const size_t fs = r.field_bytes / sizeof(float);
        float** slots[8] = {&h.rh, &h.rl, &h.dxr, &h.dyr, &h.dxx, &h.dyy, &h.Fx, &h.Fy};
        for (int q = 0; q < 8; ++q) *slots[q] = fields + q * fs;
        h.partials = (double*)(base + r.parts_off);
        PhysParams& p = h.phys;
        p.eos = eos->kind;
        p.T = in.T_r * Tc;
        p.alpha = eos_alpha(eos->kind, eos->a, eos->b, eos->R, eos->omega, p.T);
        p.a = eos->a;
        p.b = eos->b;
        p.R = eos->R;
        p.k2 = in.mesh_coeff * in.mesh_coeff;
        p.kappa = in.kappa;
        p.omega = 1.0 / in.tau;
        p.mu_cap = std::isinf(in.mu_max) ? HUGE_VAL : p.k2 * in.mu_max;
        p.cap_steps = in.mu_cap_steps;
        h.t = 0;
        h.ready = false;
        h.rows = 0;
        h.rho_df = opts->prec == LBM_PREC_MIXED_DF;
        if (!h.rho_df) {
            double rg, rl;
            h.rho_df = eos_maxwell(eos->kind, eos->a, eos->b, eos->R, eos->omega, p.T, &rg,
                                   &rl) != 0 ||
                       !(rl < kDfRatio * rg);
        }
        o += r.total;
    }
    b->tb = table_layout(inst, n, b->order, o);
    b->dst = (DevState*)(b->ws + b->tb.state);
    b->order_by_size.resize(n);
    for (int i = 0; i < n; ++i) b->order_by_size[i] = i;
    std::stable_sort(b->order_by_size.begin(), b->order_by_size.end(),
                     [&](int x, int y) { return b->inst[x].N > b->inst[y].N; });

    if (cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&b->side_stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->fork_ev, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->join_ev, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->ev, cudaEventDisableTiming) != cudaSuccess ||
        cudaMallocHost((void**)&b->hst, n * sizeof(DevState)) != cudaSuccess) {
        lbm_batch_free(b);
        return LBM_ECUDA;
    }
    for (auto& e : b->tev)
        if (cudaEventCreate(&e) != cudaSuccess) {
            lbm_batch_free(b);
            return LBM_ECUDA;
        }
    lbm_status st = LBM_OK;
    for (int i = 0; i < n && st == LBM_OK; ++i) st = reset_state(b, i);
    if (st == LBM_OK) st = upload_tables(b);
    if (st != LBM_OK) {
        lbm_batch_free(b);
        return st;
    }
    *out = b;
    return LBM_OK;
}

void lbm_batch_free(lbm_batch* b) {
    if (!b) return;
    cudaSetDevice(b->dev);
    drop_graphs(b);
    for (cudaEvent_t e : {b->ev, b->fork_ev, b->join_ev})
        if (e) cudaEventDestroy(e);
    for (auto& e : b->tev)
        if (e) cudaEventDestroy(e);
    for (cudaStream_t x : {b->cap_stream, b->side_stream})
        if (x) cudaStreamDestroy(x);
    if (b->hst) cudaFreeHost(b->hst);
    delete b;
}

lbm_status lbm_batch_set_timeout(lbm_batch* b, double seconds) {
    if (!b || !(seconds > 0)) return LBM_EINVAL;
    b->timeout_s = seconds;
    return LBM_OK;
}

int64_t lbm_batch_time(const lbm_batch* b, int32_t i) {
    if (!b || i < 0 || i >= b->n) return -1;
    return b->inst[i].t;
}

int32_t lbm_batch_tile_rows(const lbm_batch* b, int32_t i) {
    if (!b || i < 0 || i >= b->n) return -1;
    const InstHost& h = b->inst[i];
    return cs_mixed_args(nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, h.nx, h.ny, 0,
                         1.0, nullptr, nullptr, h.rows)
        .rows;
}

lbm_status lbm_batch_failed(const lbm_batch* b, int32_t* inst, int64_t* step) {
    if (!b) return LBM_EINVAL;
    if (inst) *inst = b->failed_inst;
    if (step) *step = b->failed_step;
    return LBM_OK;
}

lbm_status lbm_batch_set_fields(lbm_batch* b, int32_t i, const double* h_rho,
                                const double* h_ux, const double* h_uy) {
    if (!b || i < 0 || i >= b->n || !h_rho) return LBM_EINVAL;
    CK(cudaSetDevice(b->dev));
    lbm_status st = wait_stream(b);
    if (st) return st;
    InstHost& h = b->inst[i];
    h.ready = false;
    // stage in this instance's idle population buffer (>= 3 N doubles)
    double* sg = (double*)h.f[1 - b->cur];
    const size_t B = h.N * sizeof(double);
    CK(cudaMemcpyAsync(sg, h_rho, B, cudaMemcpyHostToDevice, b->stream));
    if (h_ux) CK(cudaMemcpyAsync(sg + h.N, h_ux, B, cudaMemcpyHostToDevice, b->stream));
    if (h_uy) CK(cudaMemcpyAsync(sg + 2 * h.N, h_uy, B, cudaMemcpyHostToDevice, b->stream));
    st = reset_state(b, i);
    if (st) return st;
    CK(launch_init_mixed(sg, h_ux ? sg + h.N : nullptr, h_uy ? sg + 2 * h.N : nullptr,
                         h.f[b->cur], h.rh, h.rl, h.nx, h.ny, h.plane, b->stream));
    st = instance_force(b, i);
    if (st) return st;
    st = read_states(b, i);
    if (st) return st;
    h.ready = true;
    return LBM_OK;
}

lbm_status lbm_batch_step(lbm_batch* b, int64_t n) {
    if (!b || n < 0) return LBM_EINVAL;
    if (!all_ready(b)) return LBM_EINVAL;
    CK(cudaSetDevice(b->dev));
    int64_t left = n;
    if (left >= 2) {
        lbm_status st = build_graph(b, b->cur);
        if (st) return st;
        for (; left >= 2; left -= 2) CK(cudaGraphLaunch(b->graph[b->cur], b->stream));
    }
    if (left == 1) {
        lbm_status st = enqueue_step(b, b->stream, b->cur);
        if (st) return st;
        b->cur = 1 - b->cur;
    }
    for (auto& h : b->inst) h.t += n;
    return read_states(b);
}

lbm_status lbm_batch_step_timed(lbm_batch* b, float* pass_ms) {
    if (!b || !pass_ms) return LBM_EINVAL;
    if (!all_ready(b)) return LBM_EINVAL;
    CK(cudaSetDevice(b->dev));
    CK(cudaEventRecord(b->tev[0], b->stream));
    lbm_status st = enqueue_step(b, b->stream, b->cur, b->tev);
    if (st) return st;
    b->cur = 1 - b->cur;
    for (auto& h : b->inst) h.t += 1;
    st = read_states(b);
    if (st) return st;
    for (int i = 0; i < 4; ++i) CK(cudaEventElapsedTime(&pass_ms[i], b->tev[i], b->tev[i + 1]));
    return LBM_OK;
}

lbm_status lbm_batch_fields(lbm_batch* b, int32_t i, double* h_rho, double* h_vx,
                            double* h_vy, double* h_mu) {
    if (!b || i < 0 || i >= b->n) return LBM_EINVAL;
    InstHost& h = b->inst[i];
    if (!h.ready) return LBM_EINVAL;
    CK(cudaSetDevice(b->dev));
    double* sg = (double*)h.f[1 - b->cur];  // idle buffer: >= 4 N doubles
    const size_t N = h.N;
    CK(launch_macro_mixed(h.f[b->cur], h.rh, rl_of(h), h.Fx, h.Fy, h.dxx /* holds mu-hat */,
                          h_rho ? sg : nullptr, h_vx ? sg + N : nullptr,
                          h_vy ? sg + 2 * N : nullptr, h_mu ? sg + 3 * N : nullptr, h.nx, h.ny,
                          h.plane, b->stream));
    lbm_status st = wait_stream(b);
    if (st) return st;
    const size_t B = N * sizeof(double);
    if (h_rho) CK(cudaMemcpyAsync(h_rho, sg, B, cudaMemcpyDeviceToHost, b->stream));
    if (h_vx) CK(cudaMemcpyAsync(h_vx, sg + N, B, cudaMemcpyDeviceToHost, b->stream));
    if (h_vy) CK(cudaMemcpyAsync(h_vy, sg + 2 * N, B, cudaMemcpyDeviceToHost, b->stream));
    if (h_mu) CK(cudaMemcpyAsync(h_mu, sg + 3 * N, B, cudaMemcpyDeviceToHost, b->stream));
    return wait_stream(b);
}

lbm_status lbm_batch_diag(lbm_batch* b, double* mass, double* max_v, double* rho_min,
                          double* rho_max) {
    if (!b) return LBM_EINVAL;
    if (!all_ready(b)) return LBM_EINVAL;
    CK(cudaSetDevice(b->dev));
    for (int i = 0; i < b->n; ++i) {
        const InstHost& h = b->inst[i];
        CK(launch_diag_mixed(h.f[b->cur], h.rh, rl_of(h), h.Fx, h.Fy, h.nx, h.ny, h.plane,
                             h.partials, kParts, b->dst + i, b->stream));
    }
    lbm_status st = read_states(b);
    if (st) return st;
    for (int i = 0; i < b->n; ++i) {
        const double* d = b->hst[i].diag;
        if (mass) mass[i] = d[0];
        if (max_v) max_v[i] = d[1];
        if (rho_min) rho_min[i] = d[2];
        if (rho_max) rho_max[i] = d[3];
    }
    return LBM_OK;
}

lbm_status lbm_batch_autotune(lbm_batch* b, int32_t reps) {
    if (!b || reps < 1) return LBM_EINVAL;
    if (!all_ready(b)) return LBM_EINVAL;
    CK(cudaSetDevice(b->dev));
    lbm_status st = wait_stream(b);
    if (st) return st;
    // one representative instance per distinct grid size
    std::map<std::pair<int, int>, int> rep;
    for (int i = 0; i < b->n; ++i) rep.emplace(std::make_pair(b->inst[i].nx, b->inst[i].ny), i);
    cudaStream_t s = b->stream;
    for (const auto& kv : rep) {
        const InstHost& h = b->inst[kv.second];
        DevState* dst = b->dst + kv.second;
        float best = 0.0f;
        int best_rows = 0;
        for (int rows : kRowChoices) {
            const CsArgs a =
                cs_mixed_args(h.f[b->cur], h.f[1 - b->cur], h.Fx, h.Fy, h.rh, rl_of(h), h.nx, h.ny,
                              h.plane, h.phys.omega, b->mrt ? &b->rates : nullptr, dst, rows);
            CK(launch_cs_mixed_args(a, s));  // warm-up
            CK(cudaEventRecord(b->tev[0], s));
            for (int r = 0; r < reps; ++r) CK(launch_cs_mixed_args(a, s));
            CK(cudaEventRecord(b->tev[1], s));
            st = wait_stream(b);
            if (st) return st;
            float ms = 0.0f;
            CK(cudaEventElapsedTime(&ms, b->tev[0], b->tev[1]));
            if (best_rows == 0 || ms < best) {
                best = ms;
                best_rows = rows;
            }
        }
        for (auto& x : b->inst)
            if (x.nx == h.nx && x.ny == h.ny) x.rows = best_rows;
    }
    // the timing launches overwrote the idle buffer and the density planes
    // with the next time level: recompute the density of the current state
    for (const auto& h : b->inst)
        CK(launch_rho_from_f_mixed(h.f[b->cur], h.rh, h.rl, h.nx, h.ny, h.plane, s));
    // lines per block of the FP32 line launches: the whole FP32 density launch
    // and the force launch of the batch, timed at 8 and 16
    {
        float best = 0.0f;
        int best_nl = 8;
        for (int nl : {8, 16}) {
            b->line_nl = nl;
            st = upload_tables(b);
            if (st) return st;
            auto pass = [&]() -> cudaError_t {
                const cudaError_t e = f32_lines(b, true, 0, s);
                return e != cudaSuccess ? e : f32_lines(b, false, 0, s);
            };
            CK(pass());  // warm-up
            CK(cudaEventRecord(b->tev[0], s));
            for (int r = 0; r < reps; ++r) CK(pass());
            CK(cudaEventRecord(b->tev[1], s));
            st = wait_stream(b);
            if (st) return st;
            float ms = 0.0f;
            CK(cudaEventElapsedTime(&ms, b->tev[0], b->tev[1]));
            if (nl == 8 || ms < best) {
                best = ms;
                best_nl = nl;
            }
        }
        b->line_nl = best_nl;
    }
    // the density lines overwrote mu-hat (it shares its plane with d_xx rho) and
    // the force lines then read that: recompute the force stage of the state
    for (int i = 0; i < b->n; ++i) {
        st = instance_force(b, i);
        if (st) return st;
    }
    drop_graphs(b);
    st = upload_tables(b);
    if (st) return st;
    return read_states(b);
}

int32_t lbm_batch_lines_per_block(const lbm_batch* b) { return b ? b->line_nl : -1; }

lbm_status lbm_batch_set_lines_per_block(lbm_batch* b, int32_t nl) {
    if (!b || (nl != 8 && nl != 16)) return LBM_EINVAL;
    CK(cudaSetDevice(b->dev));
    b->line_nl = nl;
    drop_graphs(b);
    return upload_tables(b);
}

}  // extern "C"
