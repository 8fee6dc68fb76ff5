// lines64.cu -- compact-FD line solves of the FP64 path (Eqs. 37-39), with the
// moment sum (Eq. 3), chemical-potential (Eqs. 21, 33, Sec. 5.6) and force (Eq. 12) work
// of the pass each belongs to.
//
// The scheme is A d = B u along a periodic line, A = (alpha, 1, alpha).  A splits into the
// two recursions w_i = r_i - lam w_{i-1} and z_i = w_i - lam z_{i+1} (lam = 0.382 at
// alpha = 1/3, 0.268 at 1/4), and B u is c1 times r_i = (u_{i+1} - u_{i-1}) + gamma (u_{i+2} -
// u_{i-2}), so d = c1 z.  The factor c1 (and c1^2 of the second derivative, which is the
// solve applied to z) is left to whoever uses the result, where it folds into a constant.
//
// What bounds it: the FP64 pipe, 2 lanes a clock and SM.  So the solve is arranged for the
// fewest FP64 instructions a position, 7 and a share of the joins: 3 for r, one for each
// recursion, one for each join.  A warp takes a line; each lane runs a contiguous chunk of
// about L/32 positions in place in shared memory and the chunk ends are joined by a
// circular shuffle scan, which is exact for a periodic line of any length: no window, no
// halo.  (Windows of 608 positions with halos of 44-48, chunks of 19 and a double recursion
// for the second derivative took 70 us for the x-lines of a 1024^2 grid and 190 for the
// y-lines with mu-hat; this takes 55, the moment sum included, and 106.)  A join
// reaches kPw positions into a chunk: beyond, lam^k is below 4e-24.
//
// Lines longer than kLWhole are cut into overlapping windows (whole, a line of 4096 leaves four
// warps an SM: a 4096^2 step took 8.5 ms, in windows 5.3; on 1536^2 it is the same either
// way), shorter ones too where a launch has few of them (geo64), and lines between walls
// (the even extension of period 2 n, Sec. 5.5) of more than 2 kHalo positions are one window
// with a mirrored halo.  A window is solved as if it were periodic: what that gets wrong at
// its ends has decayed by the owned positions.
#include "cplbm_internal.cuh"
#include "eos.cuh"
#include "fp64_math.cuh"
#include "lattice.cuh"

namespace cplbm {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kT = 128;       // threads a block; warps 0 .. nl-1 solve a line each
constexpr int kPw = 57;       // powers (-lam)^0 .. (-lam)^56
constexpr int kHalo = 96;     // two solves of kPw - 9 positions: lam^48 < 1e-20
constexpr int kLWhole = 1600; // longest line solved whole
constexpr int kLOwn = 1100;   // most positions a window of a longer one owns
// in launches of few lines (see geo64): most positions a window owns where there is room for
// more of them, and the longest lines solved whole, with such room and without
constexpr int kLOwnRoom = 512, kLRoom = 1024, kLFew = kLOwn + 2 * kHalo;
constexpr int kSMs = 152;

struct Geo {
    int n, nlines;       // line length, lines
    long long ps, ls;    // stride along a line, between lines
    int axis;            // 0: x-lines, 1: y-lines
    int L, H, own;       // window length, halo before the owned positions, owned positions
    int nwin, period;    // windows a line; n, or 2 n where the line is mirrored
    int nl, ngroups;     // lines a block, line groups
    int base, rem;       // lane chunks: rem of base + 1 positions, the others of base
    int steps;           // doubling steps of the chunk scan
};
struct Scheme64 {
    double gamma, nlam, c1;
    double pw[kPw];   // (-lam)^k
    double periodic;  // 1 / (1 - (-lam)^L): the line seen through its own period
};

// slot of window position q in shared memory: one spare slot in 32, so that lanes whose
// chunks start a power of two apart do not meet in one bank
__device__ __forceinline__ int slot(int q) { return q + (q >> 5); }
__host__ __device__ constexpr int line_slots(int L) { return L + (L >> 5) + 1; }

// One line, one warp: s holds u on entry and z on return.
template <bool SIXTH>
__device__ __forceinline__ void solve_line(double* s, const Geo& g, const double* pw, double gamma,
                                           double nlam, double periodic) {
    const int lane = threadIdx.x & 31, L = g.L;
    auto start = [&](int l) { return l * g.base + min(l, g.rem); };
    const int q0 = start(lane), q1 = start(lane + 1), len = q1 - q0;
    auto at = [&](int q) {
        while (q < 0) q += L;
        while (q >= L) q -= L;
        return s[slot(q)];
    };
    // the two values on either side of the chunk, before its neighbours overwrite them
    double a = at(q0 - 2), b = at(q0 - 1);
    const double r1 = at(q1), r2 = at(q1 + 1);
    __syncwarp();
    double T = 0.0;
    if (len > 0) {
        double c = s[slot(q0)], d = len > 1 ? s[slot(q0 + 1)] : r1;
#pragma unroll 4
        for (int j = 0; j < len; ++j) {
            const int q = q0 + j;
            const double e = j + 2 < len ? s[slot(q + 2)] : (j + 2 == len ? r1 : r2);
            double r = __dadd_rn(d, -b);
            if (SIXTH) r = __fma_rn(gamma, __dadd_rn(e, -a), r);
            T = __fma_rn(nlam, T, r);
            s[slot(q)] = T;
            a = b;
            b = c;
            c = d;
            d = e;
        }
    }
    // state leaving chunk l: its own end, plus (-lam)^(span) times the state before it
    for (int k = 0; k < g.steps; ++k) {
        const int o = 1 << k;
        int span = q1 - start((lane - o + 1) & 31);
        if (span < 0) span += L;
        const double t = __shfl_sync(kFull, T, (lane - o) & 31);
        if (span < kPw) T = __fma_rn(pw[span], t, T);
    }
    double carry = __dmul_rn(__shfl_sync(kFull, T, (lane - 1) & 31), periodic);
    T = 0.0;
#pragma unroll 4
    for (int j = len - 1; j >= 0; --j) {
        double w = s[slot(q0 + j)];
        if (j < kPw - 1) w = __fma_rn(pw[j + 1], carry, w);
        T = __fma_rn(nlam, T, w);
        s[slot(q0 + j)] = T;
    }
    for (int k = 0; k < g.steps; ++k) {
        const int o = 1 << k;
        int span = start(((lane + o - 1) & 31) + 1) - q0;
        if (span < 0) span += L;
        const double t = __shfl_sync(kFull, T, (lane + o) & 31);
        if (span < kPw) T = __fma_rn(pw[span], t, T);
    }
    carry = __dmul_rn(__shfl_sync(kFull, T, (lane + 1) & 31), periodic);
    const int j0 = max(0, len - (kPw - 1));
#pragma unroll 4
    for (int j = len - 1; j >= j0; --j)
        s[slot(q0 + j)] = __fma_rn(pw[len - j], carry, s[slot(q0 + j)]);
}

struct MuArgs {
    EosC<double> e;
    double k2, kappa_c2, cap;  // kappa_c2: kappa c1^2 (the second derivatives arrive as z)
    int64_t cap_steps;
};

enum Mode : int { RHO_X, RHO_Y, FORCE, PLAIN };

struct Args {
    const double* u;      // the field solved (not RHO_X)
    const double* f;      // RHO_X: populations, whose sum is the density
    size_t plane;
    double* rho_out;      // RHO_X
    double* d1;           // RHO_X, RHO_Y: z; PLAIN: the derivative; FORCE: the force
    double* d2;           // RHO_X: z of z; RHO_Y: mu-hat; PLAIN: the second derivative or null
    const double* rho;    // RHO_Y, FORCE
    const double* dr;     // RHO_Y: z of z along x; FORCE: z of the density
    DevState* st;
    int bump;
};

__device__ __forceinline__ void raise_flag(DevState* st, unsigned bits, int64_t t) {
    atomicOr(&st->flag, bits);
    atomicMin(&st->failed_t, (unsigned long long)t);
}

template <int MODE, bool SIXTH>
__device__ __forceinline__ void lines_block(const Args& a, const Geo& g, const Scheme64& sc,
                                            const MuArgs* mu, const LogTable* tab, int bid) {
    extern __shared__ __align__(16) double sh[];
    __shared__ double pw[kPw];
    __shared__ double2 logs[MODE == RHO_Y ? LogTable::kN : 1];
    const int tid = threadIdx.x;
    if (tid < kPw) pw[tid] = sc.pw[tid];
    if constexpr (MODE == RHO_Y) {
        if (tid < LogTable::kN) logs[tid] = tab->e[tid];
    }
    const int grp = bid % g.ngroups, win = bid / g.ngroups;
    const int first = win * g.own;                  // first owned position
    const int own = min(g.own, g.n - first);
    const int LS = line_slots(g.L);
    // thread -> (line, position): x-lines by whole rows, y-lines by adjacent columns
    const int tpl = kT / g.nl;
    const int ln = g.axis == 0 ? tid / tpl : tid & (g.nl - 1);
    const int qs = g.axis == 0 ? tid - ln * tpl : tid / g.nl;
    const int line = grp * g.nl + ln;
    const bool live = line < g.nlines;
    double* s = sh + ln * LS;
    const size_t lo = (size_t)line * g.ls;
    if (live) {
#pragma unroll 2
        for (int q = qs; q < g.L; q += tpl) {
            int p = first - g.H + q;
            if (p < 0 || p >= g.period) {
                p %= g.period;
                if (p < 0) p += g.period;
            }
            if (p >= g.n) p = 2 * g.n - 1 - p;  // between walls: the even extension
            const size_t o = lo + (size_t)p * g.ps;
            double v;
            if constexpr (MODE == RHO_X) {
                double f[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) f[i] = a.f[i * a.plane + o];
                v = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
                if (q >= g.H && q < g.H + own) a.rho_out[o] = v;
            } else {
                v = a.u[o];
            }
            s[slot(q)] = v;
        }
    } else {
        for (int q = qs; q < g.L; q += tpl) s[slot(q)] = 0.0;
    }
    __syncthreads();
    const int warp = tid >> 5;
    if (warp < g.nl) solve_line<SIXTH>(sh + warp * LS, g, pw, sc.gamma, sc.nlam, sc.periodic);
    __syncthreads();
    if constexpr (MODE == FORCE) {
        if (live)
            for (int q = qs; q < own; q += tpl) {
                const size_t o = lo + (size_t)(first + q) * g.ps;
                // F = c1 (-rho z(mu) + c_s^2 z(rho)), Eq. 12
                a.d1[o] = __fma_rn(-__dmul_rn(a.rho[o], sc.c1), s[slot(g.H + q)],
                                   __dmul_rn(a.dr[o], sc.c1 / 3.0));
            }
        return;
    }
    const bool second = MODE != PLAIN || a.d2;
    if (live)
        for (int q = qs; q < own; q += tpl) {
            const double z = s[slot(g.H + q)];
            a.d1[lo + (size_t)(first + q) * g.ps] = MODE == PLAIN ? __dmul_rn(z, sc.c1) : z;
        }
    if (!second) return;
    __syncthreads();
    if (warp < g.nl) solve_line<SIXTH>(sh + warp * LS, g, pw, sc.gamma, sc.nlam, sc.periodic);
    __syncthreads();
    if (!live) return;
    if constexpr (MODE == RHO_Y) {
        const int64_t t = a.st->t;
        const bool capped = t < mu->cap_steps;
        const Math64 M{logs};
        bool bad = false;
        for (int q = qs; q < own; q += tpl) {
            const size_t o = lo + (size_t)(first + q) * g.ps;
            const double r = a.rho[o], lap = __dadd_rn(a.dr[o], s[slot(g.H + q)]);
            bool b0 = false;
            const double mu0 = eos_mu0(mu->e, r, b0, M);
            double m = __fma_rn(mu->k2, mu0, -__dmul_rn(mu->kappa_c2, lap));
            if (capped) {
                if (eos_at_pole(mu->e, r)) {  // mu0 = +infinity: the limit takes the node
                    m = mu->cap;
                    b0 = false;
                } else {
                    m = m < mu->cap ? m : mu->cap;
                }
            }
            a.d2[o] = m;
            // |m| < 1e30 (and not NaN) by the high word
            bad |= b0 || ((unsigned)__double2hiint(m) & 0x7fffffffu) >= 0x46293e59u;
        }
        if (bad) raise_flag(a.st, FLAG_EOS, t);
    } else {
        for (int q = qs; q < own; q += tpl) {
            const double z = s[slot(g.H + q)];
            a.d2[lo + (size_t)(first + q) * g.ps] =
                MODE == PLAIN ? __dmul_rn(z, __dmul_rn(sc.c1, sc.c1)) : z;
        }
    }
}

template <int MODE, bool SIXTH>
__global__ void __launch_bounds__(kT)
    k_lines64(Args a, Geo g, const __grid_constant__ Scheme64 sc) {
    if (a.bump && blockIdx.x == 0 && threadIdx.x == 0) a.st->t += 1;
    lines_block<MODE, SIXTH>(a, g, sc, nullptr, nullptr, (int)blockIdx.x);
}

template <bool SIXTH>
__global__ void __launch_bounds__(kT)
    k_lines64_mu(Args a, Geo g, const __grid_constant__ Scheme64 sc,
                 const __grid_constant__ MuArgs mu, const __grid_constant__ LogTable tab) {
    lines_block<RHO_Y, SIXTH>(a, g, sc, &mu, &tab, (int)blockIdx.x);
}

// the x- and y-lines of mu-hat in one launch: the first nbx blocks take x-lines
template <bool SIXTH>
__global__ void __launch_bounds__(kT)
    k_lines64_force(Args ax, Geo gx, const __grid_constant__ Scheme64 sx, Args ay, Geo gy,
                    const __grid_constant__ Scheme64 sy, int nbx) {
    if ((int)blockIdx.x < nbx)
        lines_block<FORCE, SIXTH>(ax, gx, sx, nullptr, nullptr, (int)blockIdx.x);
    else
        lines_block<FORCE, SIXTH>(ay, gy, sy, nullptr, nullptr, (int)blockIdx.x - nbx);
}

// ---- host side ----
Scheme64 scheme64(int order, int L) {
    const double alpha = order == 6 ? 1.0 / 3.0 : 0.25;
    const double a = 2.0 / 3.0 * (alpha + 2.0), b = (4.0 * alpha - 1.0) / 3.0;  // Eq. 38
    const double lam = (1.0 - std::sqrt(1.0 - 4.0 * alpha * alpha)) / (2.0 * alpha);
    Scheme64 s;
    s.c1 = lam / alpha * a / 2.0;
    s.gamma = (b / 4.0) / (a / 2.0);
    s.nlam = -lam;
    double p = 1.0;
    for (int k = 0; k < kPw; ++k, p *= -lam) s.pw[k] = p;
    s.periodic = 1.0 / (1.0 - std::pow(-lam, L));
    return s;
}

// lines_all: the lines of the whole launch (both directions of a merged one)
Geo geo64(int nx, int ny, int axis, bool walls_y, int lines_all) {
    Geo g;
    g.axis = axis;
    g.n = axis == 0 ? nx : ny;
    g.nlines = axis == 0 ? ny : nx;
    g.ps = axis == 0 ? 1 : nx;
    g.ls = axis == 0 ? nx : 1;
    const bool mirror = axis == 1 && walls_y;
    g.period = mirror ? 2 * g.n : g.n;
    g.H = 0;
    g.own = g.n;
    g.L = g.period;
    if (mirror && g.n > 2 * kHalo) {
        g.H = kHalo;
        g.L = g.n + 2 * kHalo;
    }
    g.nwin = 1;
    // Where an SM has one or two lines a line's length is the time, and windows are shorter:
    // 100 and 200 stand-alone lines of 1500, both derivatives, 37.1 and 41.2 us whole and 28.9
    // and 26.8 in two windows (300: 41.2 and 35.0, but steps of 1600 x 304 205 and 207); where
    // no SM gets two, short ones: 7 of 1500 37.2 and 20.7.
    const int room = (g.n + kLOwnRoom - 1) / kLOwnRoom;
    const bool has_room = (long long)lines_all * room <= kSMs;
    if (g.L > (has_room ? kLRoom : 2 * lines_all <= 3 * kSMs ? kLFew : kLWhole)) {
        g.nwin = has_room ? room : (g.n + kLOwn - 1) / kLOwn;
        g.own = ((g.n + g.nwin - 1) / g.nwin + 3) / 4 * 4;
        g.H = kHalo;
        g.L = g.own + 2 * kHalo;
    }
    // Lines a block: the pipe is shared by all warps of an SM, so a launch takes as long as
    // the SM with most lines; 4 (32-byte pieces of the rows for y-lines) unless fewer
    // spread the lines better by more than a tenth (1024 lines: 7 an SM with one a block,
    // 8 with four; 128 lines: 1 instead of 4)
    double best = 0.0;
    for (int nl : {4, 2, 1}) {
        const long long blocks = (long long)((lines_all + nl - 1) / nl) * g.nwin;
        const double most = (double)((blocks + kSMs - 1) / kSMs) * nl;
        if (nl == 4 || most < 0.9 * best) {
            best = most;
            g.nl = nl;
        }
    }
    g.ngroups = (g.nlines + g.nl - 1) / g.nl;
    g.base = g.L / 32;
    g.rem = g.L % 32;
    g.steps = 0;
    while (g.steps < 5 && (g.base << g.steps) < kPw) ++g.steps;
    return g;
}

// (windows of longer lines, and windows with a mirrored halo, are no longer than kLWhole)
constexpr size_t kMostSmem = 4 * (size_t)line_slots(kLWhole) * sizeof(double);
static_assert(kLOwn % 4 == 0 && kLOwn + 2 * kHalo <= kLWhole, "the longest window");
size_t smem64(const Geo& g) { return (size_t)g.nl * line_slots(g.L) * sizeof(double); }
unsigned blocks64(const Geo& g) { return (unsigned)((long long)g.ngroups * g.nwin); }

template <int MODE>
cudaError_t launch64(const Args& a, const Geo& g, int order, cudaStream_t s) {
    const size_t smem = smem64(g);
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, kMostSmem);
        if (e != cudaSuccess) return e;
        kern<<<blocks64(g), kT, smem, s>>>(a, g, scheme64(order, g.L));
        return cudaGetLastError();
    };
    return order == 6 ? go(k_lines64<MODE, true>) : go(k_lines64<MODE, false>);
}

}  // namespace

cudaError_t lines_fp64_rho_x(const double* f, size_t plane, double* rho, double* zx, double* zxx,
                             int nx, int ny, int order, DevState* st, int bump, cudaStream_t s) {
    Args a{};
    a.f = f;
    a.plane = plane;
    a.rho_out = rho;
    a.d1 = zx;
    a.d2 = zxx;
    a.st = st;
    a.bump = bump;
    return launch64<RHO_X>(a, geo64(nx, ny, 0, false, ny), order, s);
}

cudaError_t lines_fp64_rho_y_mu(const double* rho, const double* zxx, double* zy, double* mu,
                                int nx, int ny, int order, const PhysParams& p, DevState* st,
                                cudaStream_t s, bool walls_y) {
    Args a{};
    a.u = a.rho = rho;
    a.dr = zxx;
    a.d1 = zy;
    a.d2 = mu;
    a.st = st;
    const Geo g = geo64(nx, ny, 1, walls_y, nx);
    const Scheme64 sc = scheme64(order, g.L);
    const MuArgs m{eos_const<double>(p), p.k2, p.kappa * sc.c1 * sc.c1, p.mu_cap, p.cap_steps};
    const size_t smem = smem64(g);
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, kMostSmem);
        if (e != cudaSuccess) return e;
        kern<<<blocks64(g), kT, smem, s>>>(a, g, sc, m, log_table());
        return cudaGetLastError();
    };
    return order == 6 ? go(k_lines64_mu<true>) : go(k_lines64_mu<false>);
}

cudaError_t lines_fp64_force(const double* mu, const double* rho, const double* zx,
                             const double* zy, double* Fx, double* Fy, int nx, int ny, int order,
                             cudaStream_t s, bool walls_y) {
    auto args = [&](const double* z, double* F) {
        Args a{};
        a.u = mu;
        a.rho = rho;
        a.dr = z;
        a.d1 = F;
        return a;
    };
    const int lines = (zx ? ny : 0) + (zy ? nx : 0);
    const Geo gx = geo64(nx, ny, 0, false, lines), gy = geo64(nx, ny, 1, walls_y, lines);
    const unsigned nbx = zx ? blocks64(gx) : 0, nby = zy ? blocks64(gy) : 0;
    const size_t sx = smem64(gx), sy = smem64(gy), smem = sx > sy ? sx : sy;
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, kMostSmem);
        if (e != cudaSuccess) return e;
        kern<<<nbx + nby, kT, smem, s>>>(args(zx, Fx), gx, scheme64(order, gx.L),
                                                  args(zy, Fy), gy, scheme64(order, gy.L),
                                                  (int)nbx);
        return cudaGetLastError();
    };
    return order == 6 ? go(k_lines64_force<true>) : go(k_lines64_force<false>);
}

cudaError_t lines_fp64_plain(const double* u, double* d1, double* d2, int nx, int ny, int axis,
                             int order, cudaStream_t s) {
    Args a{};
    a.u = u;
    a.d1 = d1;
    a.d2 = d2;
    return launch64<PLAIN>(a, geo64(nx, ny, axis, false, axis ? nx : ny), order, s);
}

}  // namespace cplbm
