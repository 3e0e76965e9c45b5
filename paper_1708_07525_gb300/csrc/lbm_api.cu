// C ABI of liblbm (declared in include/lbm.h): context management, parameter
// mapping, stepping with CUDA-graph replay, read-outs, checkpoints.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_launch.h"

using namespace lbm;

namespace {

thread_local std::string g_last_error = "";

void set_global_error(const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_last_error = buf;
}

size_t storage_size(int prec) {
    switch (prec) {
        case LBM_F64: return 8;
        case LBM_F32: return 4;
        default: return 2;
    }
}


}  // namespace

namespace lbm {
namespace {
template <int B>
void set_const(FxConst<B>& k, long double c) {
    k.c = (unsigned long long)llrintl(ldexpl(fabsl(c), 63 + B)) & ~1ull;
}
// What fx_plus / fx_minus / fx_one take off: half the constants (the offset of the products'
// arguments) less the rounding of quarters, which makes up for the floors of a sum (two
// quarters' halves down), of a difference (none) or of one product.
template <int B, int D>
long long less_plus(FxConst<B> c, FxConst<D> d) { return (long long)(c.c / 2 + d.c / 2) - 2; }
template <int B, int D>
long long less_minus(FxConst<B> c, FxConst<D> d) { return (long long)(c.c / 2 - d.c / 2) - 1; }
template <int B>
long long less_one(FxConst<B> c) { return (long long)(c.c / 2) - 2; }

FixedScalar fixed_scalar(const double r[5], long double nc3_over_cap) {
    FixedScalar k;
    set_const(k.b1, 0.5L * r[1]);
    set_const(k.q1, 0.5L - 0.25L * r[1]);
    set_const(k.b2, 0.5L * r[2]);
    set_const(k.q2, 0.5L - 0.25L * r[2]);
    set_const(k.b3, r[3] / 20.0L);
    set_const(k.b4, 0.25L * r[4]);
    set_const(k.p, r[3] / 20.0L * nc3_over_cap);
    k.p_neg = nc3_over_cap < 0.0L;
    k.less1 = less_minus(k.b1, k.q1);
    k.less2 = less_minus(k.b2, k.q2);
    k.less3 = less_plus(k.b3, k.p);
    k.less4 = less_one(k.b4);
    return k;
}
void set_fixed(NoFixed&, const lbm_params&) {}
void set_fixed(FixedCoef& k, const lbm_params& P) {
    // the rates lie in (0, 2), which bounds every factor but the last one's
    const long double pT = P.model_a ? 4.0L - 5.0L * P.varpi : 4.0L - 5.0L * P.varpi / P.sigma;
    const long double pC = P.model_a ? 4.0L - 5.0L * P.varpi : 4.0L - 5.0L * P.varpi / P.eps;
    k.on = fabsl(pT * P.zeta[3] / 20.0L) < 1.0L && fabsl(pC * P.eta[3] / 20.0L) < 1.0L;
    if (!k.on) return;
    auto h = [](double s) { return 1.0L - 0.5L * s; };
    set_const(k.k1, P.s[1] / 36.0L);
    set_const(k.k1F, h(P.s[1]) / 6.0L);
    set_const(k.k2, P.s[2] / 12.0L);
    set_const(k.k2F, h(P.s[2]) / 6.0L);
    set_const(k.k4, P.s[4] / 12.0L);
    set_const(k.k4F, h(P.s[4]) / 12.0L);
    set_const(k.k6, P.s[6] / 12.0L);
    set_const(k.k6F, h(P.s[6]) / 12.0L);
    set_const(k.k7, P.s[7] / 4.0L);
    set_const(k.k7F, h(P.s[7]) / 2.0L);
    set_const(k.k8, P.s[8] / 4.0L);
    set_const(k.k8F, h(P.s[8]) / 4.0L);
    set_const(k.sixth, 1.0L / 6.0L);
    k.less1 = less_minus(k.k1, k.k1F);
    k.less2 = less_plus(k.k2, k.k2F);
    k.less4 = less_plus(k.k4, k.k4F);
    k.less6 = less_plus(k.k6, k.k6F);
    k.less7 = less_minus(k.k7, k.k7F);
    k.less8 = less_minus(k.k8, k.k8F);
    k.less_sixth = less_one(k.sixth);
    k.zs = fixed_scalar(P.zeta, pT);
    k.es = fixed_scalar(P.eta, pC);
}
}  // namespace

template <typename R>
Coef<R> make_coef(const lbm_params& P) {
    Coef<R> c;
    std::memset(&c, 0, sizeof c);
    const double eps = P.eps;
    c.T0 = (R)P.T0;
    c.C0 = (R)P.C0;
    c.inv_sigma = (R)(1.0 / P.sigma);
    c.inv_eps = (R)(1.0 / eps);
    c.eps = (R)eps;
    c.half_eps = (R)(0.5 * eps);
    c.inv_eps_f = (R)(1.0 / eps);
    c.gbT = (R)P.gbT;
    c.gbC = (R)P.gbC;
    c.Gx = (R)P.Gx;
    // Eq. 19 with delta_t = 1
    const double l0 = 0.5 * (1.0 + eps * 0.5 * P.nu / P.K);
    const double l1 = eps * 0.5 * P.Feps / std::sqrt(P.K);
    c.l0 = (R)l0;
    c.l0sq = (R)(l0 * l0);
    c.l1 = (R)l1;
    c.ndrag_lin = (R)(-eps * P.nu / P.K);                   // Eq. 5
    c.ndrag_quad = (R)(-eps * P.Feps / std::sqrt(P.K));
    c.half_epsGx = (R)(0.5 * eps * P.Gx);
    c.epsGx = (R)(eps * P.Gx);
    // relaxation rates s and forcing factors 1 - s / 2 (Eqs. 10, 21, 22) with the factors of
    // M^-1 and N^-1, in the compute precision (collide_flow, collide_d2q5)
    auto h = [](double s) { return 1.0 - 0.5 * s; };
    c.k1 = (R)(P.s[1] / 36.0);  c.k1F = (R)(-h(P.s[1]) / 6.0);
    c.k2 = (R)(P.s[2] / 12.0);  c.k2F = (R)(h(P.s[2]) / 6.0);
    c.k4 = (R)(P.s[4] / 12.0);  c.k4F = (R)(h(P.s[4]) / 12.0);
    c.k6 = (R)(P.s[6] / 12.0);  c.k6F = (R)(h(P.s[6]) / 12.0);
    c.k7 = (R)(P.s[7] / 4.0);   c.k7F = (R)(-h(P.s[7]) / 2.0);
    c.k8 = (R)(P.s[8] / 4.0);   c.k8F = (R)(-h(P.s[8]) / 4.0);
    auto scalar = [&](const double r[5]) {
        CoefScalar<R> k;
        k.b1 = (R)(r[1] / 2.0);  k.q1 = (R)(-h(r[1]) / 2.0);
        k.b2 = (R)(r[2] / 2.0);  k.q2 = (R)(-h(r[2]) / 2.0);
        k.b3 = (R)(r[3] / 20.0);
        k.b4 = (R)(r[4] / 4.0);
        return k;
    };
    c.zs = scalar(P.zeta);
    c.es = scalar(P.eta);
    // Eqs. 24 / 25 (model A: Eqs. 30 / 31): n_eq,3 = c3 Phi
    c.nc3T = (R)(P.model_a ? (4.0 - 5.0 * P.varpi) * P.sigma : 4.0 * P.sigma - 5.0 * P.varpi);
    c.nc3C = (R)(P.model_a ? (4.0 - 5.0 * P.varpi) * eps : 4.0 * eps - 5.0 * P.varpi);
    const double w = 0.25 * P.varpi;                        // w~_1..4 (Sec. 3.2)
    // anti-bounce-back constant g_q^eq + g_opp^eq at the wall value: 2 w~ Phi_w (Eq. 28),
    // 2 w~ sigma T_w / 2 w~ eps C_w for model A; in deviations from Phi0
    const double kg = P.model_a ? P.sigma : 1.0, kh = P.model_a ? eps : 1.0;
    for (int s = 0; s < 4; ++s) {
        c.wallT[s] = (R)(2.0 * w * kg * (P.Tw[s] - P.T0));
        c.wallC[s] = (R)(2.0 * w * kh * (P.Cw[s] - P.C0));
    }
    c.dirichlet_mask = (P.wall_lr == LBM_WALL_DIRICHLET ? 3 : 0) |
                       (P.wall_tb == LBM_WALL_DIRICHLET ? 12 : 0);
    c.sr = 1;
    c.poro = nullptr;
    c.nu = (R)P.nu;
    c.varpi5 = (R)(5.0 * P.varpi);
    c.moving = 0;
    for (int s = 0; s < 4; ++s)
        for (int d = 0; d < 2; ++d) {
            c.wmom[s][d] = (R)(2.0 * 1.0 * P.uw[s][d] / (1.0 / 3.0));   // 2 rho0 u_w / c_s^2
            if (P.uw[s][d] != 0.0) c.moving = 1;
        }
    // walls with nodes on them (Sec. 3.3)
    c.nee = P.nee;
    const double L = P.nx - 1.0;
    for (int s = 0; s < 4; ++s) {
        c.TwP[s] = (R)(P.Tw[s] - P.T0);
        c.CwP[s] = (R)(P.Cw[s] - P.C0);
        c.bT[s] = (R)(P.nee ? P.BiT[s] / L : 0.0);
        c.bC[s] = (R)(P.nee ? P.BiC[s] / L : 0.0);
        c.uwall[s][0] = (R)P.uw[s][0];
        c.uwall[s][1] = (R)P.uw[s][1];
    }
    const double c3T = P.model_a ? (5.0 * P.varpi - 4.0) * P.sigma : 5.0 * P.varpi - 4.0 * P.sigma;
    const double c3C = P.model_a ? (5.0 * P.varpi - 4.0) * eps : 5.0 * P.varpi - 4.0 * eps;
    c.aT0 = (R)((P.sigma - c3T) / 5.0);
    c.aT1 = (R)(P.sigma / 5.0 + c3T / 20.0);
    c.aC0 = (R)((eps - c3C) / 5.0);
    c.aC1 = (R)(eps / 5.0 + c3C / 20.0);
    set_fixed(c.fx, P);
    return c;
}
template Coef<float> make_coef<float>(const lbm_params&);
template Coef<double> make_coef<double>(const lbm_params&);
}  // namespace lbm

namespace {

bool rate_ok(double s) { return s > 0.0 && s < 2.0; }

const char* check_params(const lbm_params& P) {
    if (P.nx < 3 || P.ny < 3) return "nx and ny must be >= 3";
    if (!(P.eps > 0.0 && P.eps <= 1.0)) return "porosity eps must lie in (0, 1]";
    if (!(P.sigma > 0.0)) return "sigma must be positive";
    if (!(P.varpi > 0.0 && P.varpi < 1.0)) return "varpi must lie in (0, 1)";
    if (!(P.K > 0.0)) return "permeability K must be positive";
    if (!(P.nu >= 0.0) || !(P.Feps >= 0.0)) return "nu and F_eps must be non-negative";
    for (int k = 0; k < 9; ++k)
        if (!rate_ok(P.s[k])) return "a flow relaxation rate lies outside (0, 2)";
    for (int k = 0; k < 5; ++k)
        if (!rate_ok(P.zeta[k]) || !rate_ok(P.eta[k]))
            return "a scalar relaxation rate lies outside (0, 2)";
    if (P.wall_lr != LBM_WALL_DIRICHLET && P.wall_lr != LBM_WALL_ADIABATIC) return "bad wall_lr";
    if (P.wall_tb != LBM_WALL_DIRICHLET && P.wall_tb != LBM_WALL_ADIABATIC) return "bad wall_tb";
    if (P.model_a != 0 && P.model_a != 1) return "model_a must be 0 or 1";
    if (P.nee != 0 && P.nee != 1) return "nee must be 0 or 1";
    if (P.nee && (P.nx < 5 || P.ny < 5)) return "walls with nodes on them need nx, ny >= 5";
    for (int k = 0; k < 4; ++k) {
        if (!(P.BiT[k] >= 0.0) || !(P.BiC[k] >= 0.0) || !std::isfinite(P.BiT[k]) ||
            !std::isfinite(P.BiC[k]))
            return "Biot numbers must be finite and >= 0";
        if (!P.nee && (P.BiT[k] > 0.0 || P.BiC[k] > 0.0))
            return "convective (Robin) walls need walls with nodes on them (nee = 1)";
    }
    if ((double)P.nx * (double)P.ny > 4.0e9) return "grid too large";
    return nullptr;
}

}  // namespace

// Pinned host memory that kernels write a context's few read-out numbers to (32 doubles a
// context), so that a read-out waits for its kernel and for no copy behind it: a copy of
// 32 bytes to pageable memory took 8 of the 29 us of a call.  One block of the process
// serves up to 256 contexts; it is taken with the first and given back with the last, as
// whole pages of ordinary memory that are registered: 15 us for both (cudaHostAlloc and
// cudaFreeHost take 250: a program with one cavity at a time waited 517 us for a cavity of
// 64 x 64 and its end, 124 without the block).
// A context without a slot copies its results as before.
struct HostSlots {
    static constexpr int kSlots = 256, kDoubles = 32;
    static constexpr size_t kBytes = sizeof(double) * kSlots * kDoubles;   // 64 KiB: whole pages of any size
    std::mutex mu;
    double* block = nullptr;
    int used = 0;
    bool taken[kSlots] = {};
    // the block, or NULL; another thread may be capturing, whose streams this does not touch
    static double* pin() {
        void *p = std::aligned_alloc(kBytes, kBytes), *dev = nullptr;
        if (!p) return nullptr;
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        cudaThreadExchangeStreamCaptureMode(&mode);
        cudaError_t e = cudaHostRegister(p, kBytes, cudaHostRegisterPortable | cudaHostRegisterMapped);
        const bool pinned = e == cudaSuccess;
        if (pinned) e = cudaHostGetDevicePointer(&dev, p, 0);
        const bool usable = e == cudaSuccess && dev == p;      // kernels take the host's address
        if (pinned && !usable) cudaHostUnregister(p);
        if (e != cudaSuccess) cudaGetLastError();
        cudaThreadExchangeStreamCaptureMode(&mode);
        if (!usable) {
            std::free(p);
            p = nullptr;
        }
        return (double*)p;
    }
    static void unpin(double* p) {
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        cudaThreadExchangeStreamCaptureMode(&mode);
        const cudaError_t e = cudaHostUnregister(p);
        cudaThreadExchangeStreamCaptureMode(&mode);
        if (e == cudaSuccess) std::free(p);                    // else the pages stay: the GPU may hold them
        else cudaGetLastError();
    }
    double* take() {
        std::lock_guard<std::mutex> lk(mu);
        if (!block) block = pin();
        if (!block) return nullptr;
        for (int k = 0; k < kSlots; ++k)
            if (!taken[k]) {
                taken[k] = true;
                ++used;
                return block + (size_t)k * kDoubles;
            }
        return nullptr;
    }
    void give(double* p) {
        if (!p) return;
        std::lock_guard<std::mutex> lk(mu);
        taken[(p - block) / kDoubles] = false;
        if (--used == 0) {
            unpin(block);
            block = nullptr;
        }
    }
};
HostSlots g_host_slots;

// d_out: Nu/Sh of the side walls at 0, residual maxima at 8, Nu/Sh of bottom and top at
// 20, scratch of the Nu/Sh pass at 64, behind it the slots of the residual pass.  Both are
// zero at create, and every pass leaves them so.
constexpr int SMALL_CHUNK = 8;      // steps of the smaller captured chunk (even)
constexpr int OUT_SCRATCH = 64, OUT_SLOTS = OUT_SCRATCH + NUSH_SCRATCH, OUT_DOUBLES = OUT_SLOTS + RES_SCRATCH;

struct lbm_ctx {
    lbm_params P;
    int prec = LBM_F64, layout = LBM_AB_PULL;
    Geom G{};
    size_t esz = 8, rsz = 8;
    void* buf[2] = {nullptr, nullptr};
    void* hist = nullptr;           // history of the current level
    void* hist_alt = nullptr;       // second history buffer (two steps per launch), or NULL
    int hcur = 0;                   // swaps of hist and hist_alt so far, mod 2
    double* d_out = nullptr;        // OUT_DOUBLES: Nu/Sh and residual results, the passes' scratch
    double* h_out = nullptr;        // HostSlots::kDoubles of pinned memory laid out as d_out, or NULL
    double* d_fields = nullptr;     // lazily allocated [5][h][w] read-out window
    size_t fields_cap = 0;          // nodes d_fields holds
    void* d_snap = nullptr;         // lazily allocated [4][ny][nx] in the compute precision
    double* d_stage = nullptr;      // lazily allocated [2][ny][nx] initial-field staging
    void* poro = nullptr;           // optional [2][ny][pitch] (eps, K) in the compute precision
    bool snap_valid = false;
    int cur = 0;                    // two-buffer layout: buffer holding the state
    int64_t t = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    cudaStream_t aux = nullptr;           // second stream for the ring launches of split steps
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    int device = 0;
    int slab_y0 = 0;                // global row of the first updated row (0 for a cavity)
    bool slab = false;              // a slab of a cavity split along y (lbm_create_slab)
    Coef<double> cd{};
    Coef<float> cf{};
    LaunchCfg L{};
    int graph_chunk = 0;
    bool round_nearest = false;     // 16-bit storage: nearest-even instead of stochastic
    // captured chunks of graph_chunk steps and of a few (small_chunk), by the buffers they start
    // from: [2 * cur + hcur], and the buffers they end on
    cudaGraphExec_t graph[2][4] = {};
    int graph_end[2][4] = {};
    int64_t launched = 0;           // steps taken by launches of their own
    // the caller has captured steps (or a reset) of this context: from then on every call and
    // chunk takes an even number of two-step launches, so that an even number of steps ends on
    // the buffers it began with and the graph can be replayed, with or without other steps, a
    // reset or a load in between
    bool caller_graph = false, stale_graphs = false;
    lbm_alloc_fn alloc = nullptr;
    lbm_free_fn free_fn = nullptr;
    void* alloc_user = nullptr;
    size_t bytes = 0;
    std::string err;

    lbm_status fail(lbm_status s, const char* fmt, ...) {
        char b[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(b, sizeof b, fmt, ap);
        va_end(ap);
        err = b;
        g_last_error = b;
        return s;
    }
    lbm_status cuda_fail(cudaError_t e, const char* where) {
        return fail(LBM_ERR_CUDA, "%s: %s", where, cudaGetErrorString(e));
    }

    void* dalloc(size_t n) {
        void* p = nullptr;
        if (alloc) {
            p = alloc(n, alloc_user, (void*)stream);
            if (p && ((uintptr_t)p & 255u)) {   // the kernels assume 256-byte alignment
                free_fn(p, alloc_user, (void*)stream);
                p = nullptr;
            }
        } else if (cudaMalloc(&p, n) != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        if (p) bytes += n;
        return p;
    }
    void dfree(void* p, size_t n) {
        if (!p) return;
        if (alloc)
            free_fn(p, alloc_user, (void*)stream);
        else
            cudaFree(p);
        bytes -= n;
    }

    size_t state_bytes() const { return (size_t)NQ * G.plane * esz; }
    size_t hist_bytes() const { return (size_t)4 * G.plane * rsz; }
    size_t nodes() const { return (size_t)G.nx * G.ny; }
    int read_mode() const {
        if (layout == LBM_AB_PULL) return P.nee ? GATHER_NEE_AB : GATHER_PULL_AB;
        return (t & 1) ? GATHER_PULL_AA : GATHER_LOCAL;
    }
};

namespace {

inline const Coef<double>& coef_of(const lbm_ctx* c, double*) { return c->cd; }
inline const Coef<float>& coef_of(const lbm_ctx* c, float*) { return c->cf; }

template <typename S>
cudaError_t dispatch_step(lbm_ctx* c) {
    using R = typename Real<S>::type;
    const Coef<R>& k = coef_of(c, (R*)nullptr);
    if (c->layout == LBM_AB_PULL) {
        cudaError_t e = launch_step_ab<S>(c->buf[c->cur], c->buf[c->cur ^ 1], c->hist, c->G, k, c->L);
        c->cur ^= 1;
        return e;
    }
    return launch_step_aa<S>(c->buf[0], c->hist, c->G, k, (c->t & 1) != 0, c->L);
}

cudaError_t one_step(lbm_ctx* c) {
    cudaError_t e;
    switch (c->prec) {
        case LBM_F64: e = dispatch_step<double>(c); break;
        case LBM_F32: e = dispatch_step<float>(c); break;
        case LBM_BF16: e = dispatch_step<__nv_bfloat16>(c); break;
        default: e = dispatch_step<__half>(c); break;
    }
    c->t += 1;
    return e;
}

// Two steps in one launch (lbm_march.cuh): FP32, two buffers, halfway walls, a second
// history buffer, which only cavities that take them have.
bool can_march(const lbm_ctx* c) { return c->hist_alt != nullptr && !c->P.nee; }

// The caller is capturing the context's stream (the legacy stream cannot be captured).
bool captured_by_caller(const lbm_ctx* c) {
    if (c->stream == nullptr || c->stream == cudaStreamLegacy) return false;
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(c->stream, &s) == cudaSuccess && s != cudaStreamCaptureStatusNone;
}

// Notes a call that is being captured.
void note_capture(lbm_ctx* c, bool outer) {
    if (outer && can_march(c) && !c->caller_graph) c->caller_graph = c->stale_graphs = true;
}

// The buffer for a state of level t that replaces the present one: the one in which a run of
// single steps would hold it, so that launches which the caller has captured find it.  (t
// mod 2, until two steps per launch have swapped the buffers an odd number of times.)
int slot_for(const lbm_ctx* c, int64_t t) {
    return c->layout == LBM_AB_PULL ? c->cur ^ (int)((c->t ^ t) & 1) : 0;
}

void drop_graphs(lbm_ctx* c) {
    for (auto& kind : c->graph)
        for (cudaGraphExec_t& g : kind) {
            if (g) cudaGraphExecDestroy(g);
            g = nullptr;
        }
}

cudaError_t two_steps(lbm_ctx* c) {
    cudaError_t e = launch_step2_ab(c->buf[c->cur], c->buf[c->cur ^ 1], c->hist, c->hist_alt, c->G, c->cf, c->L);
    c->cur ^= 1;
    std::swap(c->hist, c->hist_alt);
    c->hcur ^= 1;
    c->t += 2;
    return e;
}

// Enqueues n steps; stops at the first error.
cudaError_t enqueue(lbm_ctx* c, int64_t n) {
    cudaError_t e = cudaSuccess;
    c->launched += n;
    // n mod 4 single steps instead of n mod 2 keep the number of two-step launches even
    int64_t pairs = !can_march(c) ? 0 : c->caller_graph ? n / 4 * 2 : n / 2;
    for (n -= 2 * pairs; pairs > 0 && e == cudaSuccess; --pairs) e = two_steps(c);
    for (; n > 0 && e == cudaSuccess; --n) e = one_step(c);
    return e;
}

#define LBM_DISPATCH(c, CALL_D, CALL_F, CALL_B, CALL_H) \
    ((c)->prec == LBM_F64 ? (CALL_D) : (c)->prec == LBM_F32 ? (CALL_F) : (c)->prec == LBM_BF16 ? (CALL_B) : (CALL_H))

cudaError_t run_init(lbm_ctx* c, const InitSpec& I, int slot) {
    const bool pull = c->layout == LBM_AB_PULL;
    void* b = c->buf[slot];
    return LBM_DISPATCH(c, launch_init<double>(b, c->hist, c->G, c->cd, I, pull, c->stream),
                        launch_init<float>(b, c->hist, c->G, c->cf, I, pull, c->stream),
                        launch_init<__nv_bfloat16>(b, c->hist, c->G, c->cf, I, pull, c->stream),
                        launch_init<__half>(b, c->hist, c->G, c->cf, I, pull, c->stream));
}

const void* cur_buf(const lbm_ctx* c) { return c->layout == LBM_AB_PULL ? c->buf[c->cur] : c->buf[0]; }

// Where the results at d_out + at go: the pinned slot, or device memory to copy from.
inline double* out_at(const lbm_ctx* c, int at) { return (c->h_out ? c->h_out : c->d_out) + at; }
// Fetches n of them after their kernel; waits for the stream.
cudaError_t fetch(lbm_ctx* c, cudaError_t e, int at, int n, double* to) {
    if (e == cudaSuccess && !c->h_out)
        e = cudaMemcpyAsync(to, c->d_out + at, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e == cudaSuccess && c->h_out) std::memcpy(to, c->h_out + at, n * sizeof(double));
    return e;
}

// (Re)initialise the state at t = 0 from host T / C fields or from the noise.
lbm_status do_init(lbm_ctx* c, const double* T_host, const double* C_host, uint64_t seed,
                   double noise) {
    InitSpec I;
    std::memset(&I, 0, sizeof I);
    I.seed = seed;
    I.noise = noise < 0 ? 0.0 : (noise == 0 ? 1e-3 : noise);
    I.T0 = c->P.T0;
    I.C0 = c->P.C0;
    I.sigma = c->P.sigma;
    I.eps = c->P.eps;
    I.varpi = c->P.varpi;
    I.model_a = c->P.model_a;
    // noise keys of the whole cavity: a slab draws the values its rows have in it
    I.key_ny = c->P.ny;
    I.key_j0 = c->slab_y0 - c->G.jb;
    const size_t n = (size_t)c->G.nx * step_rows(c->G);
    cudaError_t e = cudaSuccess;
    if (T_host) {
        if (!c->d_stage) {
            c->d_stage = (double*)c->dalloc(2 * c->nodes() * sizeof(double));
            if (!c->d_stage) return c->fail(LBM_ERR_NOMEM, "no device memory for initial fields");
        }
        e = cudaMemcpyAsync(c->d_stage, T_host, n * sizeof(double), cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(c->d_stage + n, C_host, n * sizeof(double), cudaMemcpyHostToDevice,
                                c->stream);
        I.T_init = c->d_stage;
        I.C_init = c->d_stage + n;
    }
    note_capture(c, captured_by_caller(c));
    const int slot = slot_for(c, 0);
    if (e == cudaSuccess) e = run_init(c, I, slot);
    if (e != cudaSuccess) return c->cuda_fail(e, "init");
    c->t = 0;
    c->cur = slot;
    c->snap_valid = false;
    return LBM_OK;
}

}  // namespace

bool lbm_ctx_view(const lbm_ctx* c, CtxView* v) {
    if (!c || !v) return false;
    v->prec = c->prec;
    v->buf = cur_buf(c);
    v->G = c->G;
    v->cd = &c->cd;
    v->cf = &c->cf;
    v->mode = c->read_mode();
    v->stream = c->stream;
    v->device = c->device;
    v->slots = c->d_out + OUT_SLOTS;
    v->out = out_at(c, 8);
    v->out_on_host = c->h_out != nullptr;
    return true;
}

void lbm_set_error(lbm_ctx* c, const char* msg) {
    if (c) c->err = msg;
    g_last_error = msg;
}

extern "C" {

namespace {

// The mapping of Sec. 4 / 4.1 for a characteristic length of N_x spacings
// (L = nx for halfway walls, nx - 1 with nodes on the walls).
lbm_status derive_core(lbm_grid grid, int nee, double Ra, double Da, double eps, double Pr,
                       double Le, double N, double J, double sigma, double Ma, double varpi,
                       lbm_params* out) {
    if (!out) {
        set_global_error("lbm_derive_params: out is NULL");
        return LBM_ERR_INVALID;
    }
    if (grid.nx < 3 || grid.ny < 3) {
        set_global_error("lbm_derive_params: nx and ny must be >= 3 (got %d x %d)", grid.nx, grid.ny);
        return LBM_ERR_INVALID;
    }
    if (!(eps > 0.0 && eps <= 1.0) || !(Da > 0.0) || !(Ra > 0.0) || !(Pr > 0.0) || !(Le > 0.0) ||
        !(J > 0.0) || !(sigma > 0.0) || !std::isfinite(N)) {
        set_global_error("lbm_derive_params: need eps in (0,1], Da, Ra, Pr, Le, J, sigma > 0");
        return LBM_ERR_INVALID;
    }
    if (!(Ma > 0.0)) Ma = 0.1;
    if (!(varpi > 0.0)) varpi = 0.4;
    lbm_params P;
    std::memset(&P, 0, sizeof P);
    P.nx = grid.nx;
    P.ny = grid.ny;
    P.nee = nee;
    // characteristic length = N_x spacings (Sec. 4.1): nx halfway cells, or the nx - 1
    // spacings between wall nodes
    const double L = nee ? grid.nx - 1.0 : (double)grid.nx;
    const double cs2 = 1.0 / 3.0, cs = std::sqrt(cs2);
    const double U = Ma * cs;                       // Ma = U / c_s
    const double nu_e = J * U * L * std::sqrt(Pr / Ra);
    const double nu = nu_e / J;
    const double alpha_e = nu / Pr;
    const double D_e = alpha_e / Le;
    const double csT2 = 0.5 * varpi;
    const double s_nu = 1.0 / (0.5 + nu_e / cs2);   // nu_e = c_s^2 (1/s_nu - 1/2)
    const double za = 1.0 / (0.5 + alpha_e / csT2); // Eq. 29
    const double eD = 1.0 / (0.5 + D_e / csT2);
    P.eps = eps;
    P.sigma = sigma;
    P.varpi = varpi;
    P.nu = nu;
    P.K = Da * L * L;                               // Da = K / L^2
    P.Feps = 1.75 / std::sqrt(150.0 * eps * eps * eps);   // Eq. 7
    P.gbT = U * U / L;                              // U^2 = g beta_T dT L with dT = 1
    P.gbC = N * P.gbT;                              // N = beta_C dC / (beta_T dT)
    P.Gx = 0.0;
    P.T0 = 0.5;
    P.C0 = 0.5;
    const double s[9] = {1.0, 1.1, 1.1, 1.0, 1.2, 1.0, 1.2, s_nu, s_nu};   // Sec. 4
    const double z[5] = {1.0, za, za, 1.5, 1.5};
    const double e[5] = {1.0, eD, eD, 1.5, 1.5};
    std::memcpy(P.s, s, sizeof s);
    std::memcpy(P.zeta, z, sizeof z);
    std::memcpy(P.eta, e, sizeof e);
    const double Tw[4] = {1.0, 0.0, 0.5, 0.5};
    std::memcpy(P.Tw, Tw, sizeof Tw);
    std::memcpy(P.Cw, Tw, sizeof Tw);
    P.wall_lr = LBM_WALL_DIRICHLET;
    P.wall_tb = LBM_WALL_ADIABATIC;
    const char* bad = check_params(P);
    if (bad) {
        set_global_error("lbm_derive_params: %s (s_nu=%g zeta_a=%g eta_D=%g)", bad, s_nu, za, eD);
        return LBM_ERR_INVALID;
    }
    *out = P;
    return LBM_OK;
}

}  // namespace

lbm_status lbm_derive_params(lbm_grid grid, double Ra, double Da, double eps, double Pr,
                             double Le, double N, double J, double sigma, double Ma,
                             double varpi, lbm_params* out) {
    return derive_core(grid, 0, Ra, Da, eps, Pr, Le, N, J, sigma, Ma, varpi, out);
}

lbm_status lbm_derive_params_nee(lbm_grid grid, double Ra, double Da, double eps, double Pr,
                                 double Le, double N, double J, double sigma, double Ma,
                                 double varpi, lbm_params* out) {
    return derive_core(grid, 1, Ra, Da, eps, Pr, Le, N, J, sigma, Ma, varpi, out);
}

lbm_status lbm_derive_params_convective(int Nx, double Ra, double Da, double eps, double Pr,
                                        double Le, double N, double BiT, double BiC, double J,
                                        double sigma, double Ma, double varpi, lbm_params* out) {
    if (!(BiT >= 0.0) || !(BiC >= 0.0) || !std::isfinite(BiT) || !std::isfinite(BiC) || Nx < 4) {
        set_global_error("lbm_derive_params_convective: need Nx >= 4 and finite Bi >= 0");
        return LBM_ERR_INVALID;
    }
    lbm_grid g;
    g.nx = g.ny = Nx + 1;
    lbm_status st = derive_core(g, 1, Ra, Da, eps, Pr, Le, N, J, sigma, Ma, varpi, out);
    if (st != LBM_OK) return st;
    out->BiT[1] = BiT;                  // the right wall: ambient T = C = 0 (Tw[1], Cw[1])
    out->BiC[1] = BiC;
    return LBM_OK;
}

namespace {

lbm_status derive_lid_core(lbm_grid grid, int nee, double Re, double Gr, double Da, double eps,
                           double Pr, double Le, double N, double J, double sigma, double U0,
                           double varpi, lbm_params* out) {
    if (!out || grid.nx < 3 || grid.ny < 3 || !(Re > 0.0) || !(Gr >= 0.0) || !(Da > 0.0) ||
        !(eps > 0.0 && eps <= 1.0) || !(Pr > 0.0) || !(Le > 0.0) || !(J > 0.0) || !(sigma > 0.0)) {
        set_global_error("lbm_derive_params_lid: invalid arguments");
        return LBM_ERR_INVALID;
    }
    if (!(U0 > 0.0)) U0 = 0.1;
    if (!(varpi > 0.0)) varpi = 0.4;
    // reuse the cavity mapping for everything but the flow scales, then set those (Sec. 4.3)
    lbm_status st = derive_core(grid, nee, 1e4, Da, eps, Pr, Le, N, J, sigma, 0.1, varpi, out);
    if (st != LBM_OK) return st;
    lbm_params P = *out;
    const double L = nee ? grid.nx - 1.0 : (double)grid.nx, cs2 = 1.0 / 3.0, csT2 = 0.5 * varpi;
    const double nu_e = J * L * U0 / Re;             // 1/s_nu = 1/2 + J L U0 / (c_s^2 Re)
    const double nu = nu_e / J;
    const double alpha_e = nu / Pr, D_e = alpha_e / Le;
    const double s_nu = 1.0 / (0.5 + nu_e / cs2);
    P.nu = nu;
    P.s[7] = P.s[8] = s_nu;
    P.zeta[1] = P.zeta[2] = 1.0 / (0.5 + alpha_e / csT2);   // Eq. 29
    P.eta[1] = P.eta[2] = 1.0 / (0.5 + D_e / csT2);
    P.gbT = Gr * nu * nu / (L * L * L);                       // Gr = g beta_T dT L^3 / nu^2
    P.gbC = N * P.gbT;
    const double Tw[4] = {0.5, 0.5, 0.0, 1.0};               // bottom cold, top hot
    std::memcpy(P.Tw, Tw, sizeof Tw);
    std::memcpy(P.Cw, Tw, sizeof Tw);
    P.wall_lr = LBM_WALL_ADIABATIC;
    P.wall_tb = LBM_WALL_DIRICHLET;
    std::memset(P.uw, 0, sizeof P.uw);
    P.uw[3][0] = U0;                                          // the lid
    const char* bad = check_params(P);
    if (bad) {
        set_global_error("lbm_derive_params_lid: %s", bad);
        return LBM_ERR_INVALID;
    }
    *out = P;
    return LBM_OK;
}

}  // namespace

lbm_status lbm_derive_params_lid(lbm_grid grid, double Re, double Gr, double Da, double eps,
                                 double Pr, double Le, double N, double J, double sigma,
                                 double U0, double varpi, lbm_params* out) {
    return derive_lid_core(grid, 0, Re, Gr, Da, eps, Pr, Le, N, J, sigma, U0, varpi, out);
}

lbm_status lbm_derive_params_lid_nee(lbm_grid grid, double Re, double Gr, double Da, double eps,
                                     double Pr, double Le, double N, double J, double sigma,
                                     double U0, double varpi, lbm_params* out) {
    return derive_lid_core(grid, 1, Re, Gr, Da, eps, Pr, Le, N, J, sigma, U0, varpi, out);
}

lbm_status lbm_params_model_a(lbm_params* p) {
    if (!p || p->model_a) {
        set_global_error("lbm_params_model_a: NULL parameters, or already model A");
        return LBM_ERR_INVALID;
    }
    // Eq. 29 -> alpha_e, D_e; Eq. 32 -> the model-A rates
    const double csT2 = 0.5 * p->varpi;
    const double alpha_e = csT2 * (1.0 / p->zeta[1] - 0.5);
    const double D_e = csT2 * (1.0 / p->eta[1] - 0.5);
    lbm_params q = *p;
    q.zeta[1] = q.zeta[2] = 1.0 / (0.5 + alpha_e / (p->sigma * csT2));
    q.eta[1] = q.eta[2] = 1.0 / (0.5 + D_e / (p->eps * csT2));
    q.model_a = 1;
    const char* bad = check_params(q);
    if (bad) {
        set_global_error("lbm_params_model_a: %s", bad);
        return LBM_ERR_INVALID;
    }
    *p = q;
    return LBM_OK;
}

namespace {

// A cavity (slab_h = 0), or the slab of rows [slab_y0, slab_y0 + slab_h) of it.
lbm_status create_core(const lbm_params* params, const lbm_options* opt, int slab_y0, int slab_h,
                       lbm_ctx** out) {
    if (!params || !out) {
        set_global_error("lbm_create_raw: params and out must be non-NULL");
        return LBM_ERR_INVALID;
    }
    *out = nullptr;
    const char* bad = check_params(*params);
    if (bad) {
        set_global_error("lbm_create_raw: %s", bad);
        return LBM_ERR_INVALID;
    }
    const bool slab = slab_h > 0;
    if (slab) {
        if (slab_y0 < 0 || slab_y0 + slab_h > params->ny) {
            set_global_error("lbm_create_slab: rows [%d, %d) outside the %d rows of the cavity",
                             slab_y0, slab_y0 + slab_h, params->ny);
            return LBM_ERR_INVALID;
        }
        if (params->nee || (opt && (opt->layout != LBM_AB_PULL || opt->eps_field || opt->K_field))) {
            set_global_error("lbm_create_slab: slabs take halfway walls, the two-buffer layout "
                             "and a uniform porous medium");
            return LBM_ERR_INVALID;
        }
    }
    lbm_options O;
    std::memset(&O, 0, sizeof O);
    if (opt) O = *opt;
    if (O.precision < LBM_F64 || O.precision > LBM_F16) {
        set_global_error("lbm_create: unknown precision %d", O.precision);
        return LBM_ERR_INVALID;
    }
    if (O.layout != LBM_AB_PULL && O.layout != LBM_AA) {
        set_global_error("lbm_create: unknown layout %d", O.layout);
        return LBM_ERR_INVALID;
    }
    if ((O.alloc == nullptr) != (O.free == nullptr)) {
        set_global_error("lbm_create: alloc and free hooks must be given together");
        return LBM_ERR_INVALID;
    }
    if (params->nee && O.layout != LBM_AB_PULL) {
        set_global_error("lbm_create: walls with nodes on them (nee) need the two-buffer layout");
        return LBM_ERR_INVALID;
    }
    // the step kernels are compiled for blocks of at most 256 threads; the shape after
    // the defaults below (block_x 0 -> 128 or 32, block_y 0 -> 128 / block_x) must fit
    if (O.block_x < 0 || O.block_y < 0 || O.block_x > 256 || O.block_y > 256 ||
        (O.block_x && O.block_x % 32) ||
        (O.block_x ? O.block_x : (params->nx >= 128 ? 128 : 32)) *
                (O.block_y ? O.block_y : 1) > 256) {
        set_global_error("lbm_create: block_x must be a multiple of 32 and block_x*block_y <= 256");
        return LBM_ERR_INVALID;
    }
    lbm_ctx* c = new (std::nothrow) lbm_ctx();
    if (!c) {
        set_global_error("lbm_create: out of host memory");
        return LBM_ERR_NOMEM;
    }
    c->P = *params;
    c->prec = O.precision;
    c->layout = O.layout;
    c->esz = storage_size(c->prec);
    c->rsz = c->prec == LBM_F64 ? 8 : 4;
    c->alloc = O.alloc;
    c->free_fn = O.free;
    c->alloc_user = O.alloc_user;
    cudaGetDevice(&c->device);
    if (O.stream) {
        c->stream = (cudaStream_t)O.stream;
    } else {
        cudaError_t e = cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) {
            lbm_status s = c->cuda_fail(e, "cudaStreamCreate");
            delete c;
            return s;
        }
        c->own_stream = true;
    }
    const int nx = params->nx;
    // a slab holds a ghost row beside each side that is a cut rather than a wall
    const int glo = slab && slab_y0 > 0 ? 1 : 0;
    const int ghi = slab && slab_y0 + slab_h < params->ny ? 1 : 0;
    const int rows = slab ? slab_h : params->ny;
    const int ny = rows + glo + ghi;
    const int per128 = (int)(128 / c->esz);
    c->slab = slab;
    c->slab_y0 = slab ? slab_y0 : 0;
    c->G.nx = nx;
    c->G.ny = ny;
    c->G.jb = glo;
    c->G.je = glo + rows;
    c->G.pitch = (nx + per128 - 1) / per128 * per128;
    c->G.plane = (size_t)ny * c->G.pitch;
    c->cd = make_coef<double>(c->P);
    c->cf = make_coef<float>(c->P);
    c->round_nearest = O.round_nearest != 0;
    c->cf.sr = c->round_nearest ? 0 : 1;
    // rounding streams keyed by the node's index in the undivided cavity
    c->cf.seed_off = (long long)(c->slab_y0 - c->G.jb) * c->G.pitch;
    int bx = O.block_x, by = O.block_y;
    if (bx == 0) bx = nx >= 128 ? 128 : 32;
    if (by == 0) by = bx >= 128 ? 1 : 128 / bx;
    if ((ny + by - 1) / by > 65535) {   // the launch grid's y extent
        lbm_status s = c->fail(LBM_ERR_INVALID, "lbm_create: ny = %d needs block_y >= %d", ny,
                               (ny + 65534) / 65535);
        g_last_error = c->err;
        lbm_destroy(c);
        return s;
    }
    c->L.bx = bx;
    c->L.by = by;
    c->L.stream = c->stream;
    c->L.aux = nullptr;
    c->L.sms = 152;
    cudaDeviceGetAttribute(&c->L.sms, cudaDevAttrMultiProcessorCount, c->device);
    // 16-bit storage takes the two-nodes-per-thread kernels, except on slabs, whose rows
    // all run the one-node kernel (the same arithmetic as a one-node whole cavity)
    c->L.pair = (c->prec == LBM_BF16 || c->prec == LBM_F16) && !slab;
    // a second stream lets the small ring launch of a split step run beside the inner one;
    // without it both go to the context's stream
    if (cudaStreamCreateWithFlags(&c->aux, cudaStreamNonBlocking) == cudaSuccess &&
        cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming) == cudaSuccess &&
        cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming) == cudaSuccess) {
        c->L.aux = c->aux;
        c->L.fork = c->ev_fork;
        c->L.join = c->ev_join;
    } else {
        cudaGetLastError();
    }
    c->graph_chunk = O.graph_chunk == 0 ? 64 : (O.graph_chunk < 0 ? 0 : O.graph_chunk);
    if (c->graph_chunk & 1) c->graph_chunk += 1;   // a chunk must return to the same parity
    if (c->stream == nullptr || c->stream == cudaStreamLegacy || c->stream == cudaStreamPerThread)
        c->graph_chunk = 0;                        // the legacy stream cannot be captured

    c->buf[0] = c->dalloc(c->state_bytes());
    if (c->layout == LBM_AB_PULL) c->buf[1] = c->dalloc(c->state_bytes());
    c->hist = c->dalloc(c->hist_bytes());
    if (c->prec == LBM_F32 && c->layout == LBM_AB_PULL && !c->P.nee && !slab && !O.eps_field && !O.K_field &&
        !O.block_x && !O.block_y && march_fits(c->G)) {
        // two steps per launch write a second history buffer; without it (no memory for it, or
        // a state of more than a quarter of the device, which leaves the rest to the
        // caller) every step is a launch
        size_t free_b = 0, total_b = 0;
        if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess && 2 * c->state_bytes() < total_b / 4)
            c->hist_alt = c->dalloc(c->hist_bytes());
    }
    c->d_out = (double*)c->dalloc(OUT_DOUBLES * sizeof(double));
    c->h_out = g_host_slots.take();
    if (O.eps_field || O.K_field) {
        if (c->P.model_a) {
            lbm_status s = c->fail(LBM_ERR_INVALID, "lbm_create: porous fields are not supported with model_a");
            g_last_error = c->err;
            lbm_destroy(c);
            return s;
        }
        // both planes in the compute precision, row pitch of the state
        const size_t plane = c->G.plane, n2 = 2 * plane;
        std::vector<double> hv(n2, 0.0);
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i) {
                const size_t k = (size_t)j * nx + i, d = (size_t)j * c->G.pitch + i;
                const double e = O.eps_field ? O.eps_field[k] : c->P.eps;
                const double K = O.K_field ? O.K_field[k] : c->P.K;
                if (!(e > 0.0 && e <= 1.0) || !(K > 0.0)) {
                    lbm_status s = c->fail(LBM_ERR_INVALID,
                                           "lbm_create: porous field at (%d, %d): eps %g, K %g", i, j, e, K);
                    g_last_error = c->err;
                    lbm_destroy(c);
                    return s;
                }
                hv[d] = e;
                hv[plane + d] = K;
            }
        // padding columns: copies of a valid value, never read by the kernels
        for (size_t d = 0; d < n2; ++d)
            if (hv[d] == 0.0) hv[d] = d < plane ? c->P.eps : c->P.K;
        c->poro = c->dalloc(n2 * c->rsz);
        if (!c->poro) {
            lbm_status s = c->fail(LBM_ERR_NOMEM, "lbm_create: no device memory for the porous field");
            g_last_error = c->err;
            lbm_destroy(c);
            return s;
        }
        cudaError_t e;
        if (c->rsz == 8) {
            e = cudaMemcpy(c->poro, hv.data(), n2 * 8, cudaMemcpyHostToDevice);
        } else {
            std::vector<float> hf(hv.begin(), hv.end());
            e = cudaMemcpy(c->poro, hf.data(), n2 * 4, cudaMemcpyHostToDevice);
        }
        if (e != cudaSuccess) {
            lbm_status s = c->cuda_fail(e, "lbm_create: porous field upload");
            g_last_error = c->err;
            lbm_destroy(c);
            return s;
        }
        c->cd.poro = c->rsz == 8 ? (const double*)c->poro : nullptr;
        c->cf.poro = c->rsz == 4 ? (const float*)c->poro : nullptr;
    }
    if (!c->buf[0] || (c->layout == LBM_AB_PULL && !c->buf[1]) || !c->hist || !c->d_out) {
        lbm_status s = c->fail(LBM_ERR_NOMEM, "lbm_create: device allocation of %.3f GB failed",
                               (2.0 * c->state_bytes() + c->hist_bytes()) / 1e9);
        lbm_destroy(c);
        return s;
    }
    // padding columns are never read, but keep them defined
    cudaMemsetAsync(c->buf[0], 0, c->state_bytes(), c->stream);
    if (c->buf[1]) cudaMemsetAsync(c->buf[1], 0, c->state_bytes(), c->stream);
    cudaMemsetAsync(c->hist, 0, c->hist_bytes(), c->stream);
    if (c->hist_alt) cudaMemsetAsync(c->hist_alt, 0, c->hist_bytes(), c->stream);
    // the block counts of the Nu/Sh and residual passes; here, where the stream is waited for, and
    // not at the first read-out, which may be refused for a stream that is being captured
    cudaMemsetAsync(c->d_out, 0, OUT_DOUBLES * sizeof(double), c->stream);

    if ((O.T_init == nullptr) != (O.C_init == nullptr)) {
        lbm_status s = c->fail(LBM_ERR_INVALID, "lbm_create: give both T_init and C_init");
        lbm_destroy(c);
        return s;
    }
    lbm_status s = do_init(c, O.T_init, O.C_init, O.seed, O.noise);
    if (s == LBM_OK) {   // the caller may release T_init / C_init once create returns
        cudaError_t e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) s = c->cuda_fail(e, "lbm_create: init");
    }
    if (s != LBM_OK) {
        g_last_error = c->err;
        lbm_destroy(c);
        return s;
    }
    *out = c;
    return LBM_OK;
}

}  // namespace

lbm_status lbm_create_raw(const lbm_params* params, const lbm_options* opt, lbm_ctx** out) {
    return create_core(params, opt, 0, 0, out);
}

lbm_status lbm_create_slab(const lbm_params* params, int y0, int h, const lbm_options* opt,
                           lbm_ctx** out) {
    if (h < 1) {
        if (out) *out = nullptr;
        set_global_error("lbm_create_slab: a slab needs at least one row");
        return LBM_ERR_INVALID;
    }
    return create_core(params, opt, y0, h, out);
}

lbm_status lbm_create(lbm_grid grid, double Ra, double Da, double eps, double Pr, double Le,
                      double N, double J, double sigma, const lbm_options* opt, lbm_ctx** out) {
    lbm_params P;
    const double Ma = opt ? opt->Ma : 0.0, varpi = opt ? opt->varpi : 0.0;
    lbm_status s = lbm_derive_params(grid, Ra, Da, eps, Pr, Le, N, J, sigma, Ma, varpi, &P);
    if (s != LBM_OK) return s;
    return lbm_create_raw(&P, opt, out);
}

lbm_status lbm_reset(lbm_ctx* c, const double* T_init, const double* C_init, uint64_t seed,
                     double noise) {
    if (!c || ((T_init == nullptr) != (C_init == nullptr))) {
        set_global_error("lbm_reset: NULL context, or only one of T_init / C_init given");
        return LBM_ERR_INVALID;
    }
    DeviceGuard dg(c->device);
    return do_init(c, T_init, C_init, seed, noise);
}

lbm_status lbm_step(lbm_ctx* c, int64_t n) {
    if (!c || n < 0) {
        set_global_error("lbm_step: invalid context or negative step count");
        return LBM_ERR_INVALID;
    }
    DeviceGuard dg(c->device);
    cudaError_t e = cudaSuccess;
    const bool outer = captured_by_caller(c);
    note_capture(c, outer);
    if (!outer && c->stale_graphs) {
        drop_graphs(c);
        c->stale_graphs = false;
    }
    // the in-place layout replays its graph from even levels
    while (n > 0 && c->layout == LBM_AA && (c->t & 1) && e == cudaSuccess) {
        e = one_step(c);
        --n;
    }
    // chunks of graph_chunk steps; and, in a loop that takes a few steps at a time, of
    // SMALL_CHUNK: a replay of those costs the host 6 us, their launches 33 (a capture, about
    // 150 us, once a context has made 64 launches of its own)
    for (int kind = 0; kind < 2 && c->graph_chunk > 0; ++kind) {
        const int chunk = kind == 0 ? c->graph_chunk : SMALL_CHUNK;
        if (kind == 1 && (c->launched < 64 || chunk >= c->graph_chunk || outer)) break;
        while (n >= chunk && e == cudaSuccess) {
            // a chunk is captured once per pair of buffers it can start from, and may end
            // on the others
            const int k0 = 2 * c->cur + c->hcur;
            cudaGraphExec_t& graph = c->graph[kind][k0];
            if (!graph) {
                const int64_t t0 = c->t, launched0 = c->launched;
                const int cur0 = c->cur, hcur0 = c->hcur;
                void *h0 = c->hist, *h1 = c->hist_alt;
                cudaGraph_t g = nullptr;
                e = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal);
                if (e == cudaSuccess) {
                    const cudaError_t le = enqueue(c, chunk);
                    c->graph_end[kind][k0] = 2 * c->cur + c->hcur;
                    c->t = t0;   // capture records, it does not run
                    c->launched = launched0;
                    c->cur = cur0;
                    c->hcur = hcur0;
                    c->hist = h0;
                    c->hist_alt = h1;
                    e = cudaStreamEndCapture(c->stream, &g);
                    if (le != cudaSuccess) e = le;
                }
                if (e == cudaSuccess) e = cudaGraphInstantiate(&graph, g, 0);
                if (g) cudaGraphDestroy(g);
                if (e != cudaSuccess) {
                    graph = nullptr;
                    return c->cuda_fail(e, "lbm_step: graph capture");
                }
            }
            e = cudaGraphLaunch(graph, c->stream);
            if (e == cudaSuccess) {
                const int k1 = c->graph_end[kind][k0];
                c->cur = k1 >> 1;
                if ((k1 & 1) != c->hcur) {
                    std::swap(c->hist, c->hist_alt);
                    c->hcur ^= 1;
                }
                c->t += chunk;
                n -= chunk;
            }
        }
    }
    if (e == cudaSuccess) e = enqueue(c, n);
    if (e != cudaSuccess) return c->cuda_fail(e, "lbm_step");
    return LBM_OK;
}

int64_t lbm_time(const lbm_ctx* c) { return c ? c->t : -1; }

int lbm_steps_per_launch(const lbm_ctx* c) { return !c ? 0 : can_march(c) ? 2 : 1; }

lbm_status lbm_fields_window(lbm_ctx* c, int x0, int y0, int w, int h, double* ux, double* uy,
                             double* T, double* C, double* rho) {
    if (!c) {
        set_global_error("lbm_fields_window: NULL context");
        return LBM_ERR_INVALID;
    }
    const int rows = step_rows(c->G);
    if (x0 < 0 || y0 < 0 || w < 1 || h < 1 || x0 + w > c->G.nx || y0 + h > rows || h > 65535)
        return c->fail(LBM_ERR_INVALID, "lbm_fields_window: window (%d, %d, %d x %d) outside the %d x %d grid",
                       x0, y0, w, h, c->G.nx, rows);
    y0 += c->G.jb;   // a slab's rows start after its lower ghost row
    DeviceGuard dg(c->device);
    const size_t n = (size_t)w * h;
    if (n > c->fields_cap) {
        c->dfree(c->d_fields, 5 * c->fields_cap * sizeof(double));
        c->fields_cap = 0;
        c->d_fields = (double*)c->dalloc(5 * n * sizeof(double));
        if (!c->d_fields) return c->fail(LBM_ERR_NOMEM, "lbm_fields: no device memory for read-out");
        c->fields_cap = n;
    }
    const int mode = c->read_mode();
    const void* b = cur_buf(c);
    cudaError_t e = LBM_DISPATCH(c, launch_fields<double>(b, c->G, c->cd, mode, x0, y0, w, h, c->d_fields, c->stream),
                                 launch_fields<float>(b, c->G, c->cf, mode, x0, y0, w, h, c->d_fields, c->stream),
                                 launch_fields<__nv_bfloat16>(b, c->G, c->cf, mode, x0, y0, w, h, c->d_fields, c->stream),
                                 launch_fields<__half>(b, c->G, c->cf, mode, x0, y0, w, h, c->d_fields, c->stream));
    double* outs[5] = {ux, uy, T, C, rho};
    for (int k = 0; k < 5 && e == cudaSuccess; ++k)
        if (outs[k])
            e = cudaMemcpyAsync(outs[k], c->d_fields + k * n, n * sizeof(double),
                                cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return c->cuda_fail(e, "lbm_fields");
    return LBM_OK;
}

lbm_status lbm_fields(lbm_ctx* c, double* ux, double* uy, double* T, double* C, double* rho) {
    if (!c) {
        set_global_error("lbm_fields: NULL context");
        return LBM_ERR_INVALID;
    }
    // whole grid, in row bands of at most 65535 rows and about 2^26 nodes (2.7 GB of read-out)
    const int band = (int)std::max<size_t>(1, std::min<size_t>(65535, ((size_t)1 << 26) / c->G.nx));
    const int rows = step_rows(c->G);
    if (rows <= band) return lbm_fields_window(c, 0, 0, c->G.nx, rows, ux, uy, T, C, rho);
    for (int y0 = 0; y0 < rows; y0 += band) {
        const int h = std::min(band, rows - y0);
        const size_t off = (size_t)y0 * c->G.nx;
        lbm_status s = lbm_fields_window(c, 0, y0, c->G.nx, h, ux ? ux + off : nullptr, uy ? uy + off : nullptr,
                                         T ? T + off : nullptr, C ? C + off : nullptr, rho ? rho + off : nullptr);
        if (s != LBM_OK) return s;
    }
    return LBM_OK;
}

lbm_status lbm_nusselt_sherwood(lbm_ctx* c, double out[4]) {
    if (!c || !out) {
        set_global_error("lbm_nusselt_sherwood: NULL argument");
        return LBM_ERR_INVALID;
    }
    DeviceGuard dg(c->device);
    WallSpec W;
    W.Tw[0] = c->P.Tw[0];
    W.Tw[1] = c->P.Tw[1];
    W.Cw[0] = c->P.Cw[0];
    W.Cw[1] = c->P.Cw[1];
    W.T0 = c->P.T0;
    W.C0 = c->P.C0;
    W.dT = c->P.Tw[0] - c->P.Tw[1];
    W.dC = c->P.Cw[0] - c->P.Cw[1];
    W.nee = c->P.nee;
    W.L = c->P.nee ? c->P.nx - 1.0 : (double)c->P.nx;
    const int mode = c->read_mode();
    const void* b = cur_buf(c);
    cudaError_t e = LBM_DISPATCH(c, launch_nush<double>(b, c->G, c->cd, mode, W, c->d_out + OUT_SCRATCH, out_at(c, 0), c->stream),
                                 launch_nush<float>(b, c->G, c->cf, mode, W, c->d_out + OUT_SCRATCH, out_at(c, 0), c->stream),
                                 launch_nush<__nv_bfloat16>(b, c->G, c->cf, mode, W, c->d_out + OUT_SCRATCH, out_at(c, 0), c->stream),
                                 launch_nush<__half>(b, c->G, c->cf, mode, W, c->d_out + OUT_SCRATCH, out_at(c, 0), c->stream));
    e = fetch(c, e, 0, 4, out);
    if (e != cudaSuccess) return c->cuda_fail(e, "lbm_nusselt_sherwood");
    for (int k = 0; k < 4; ++k)
        if (!std::isfinite(out[k]))
            return c->fail(LBM_ERR_DIVERGED, "lbm_nusselt_sherwood: non-finite result at t=%lld",
                           (long long)c->t);
    return LBM_OK;
}

lbm_status lbm_nusselt_sherwood_tb(lbm_ctx* c, double out[4]) {
    if (!c || !out) {
        set_global_error("lbm_nusselt_sherwood_tb: NULL argument");
        return LBM_ERR_INVALID;
    }
    if (c->slab) return c->fail(LBM_ERR_INVALID, "lbm_nusselt_sherwood_tb: not defined on a slab");
    DeviceGuard dg(c->device);
    WallSpec W;
    W.Tw[0] = c->P.Tw[2];
    W.Tw[1] = c->P.Tw[3];
    W.Cw[0] = c->P.Cw[2];
    W.Cw[1] = c->P.Cw[3];
    W.T0 = c->P.T0;
    W.C0 = c->P.C0;
    W.dT = c->P.Tw[3] - c->P.Tw[2];
    W.dC = c->P.Cw[3] - c->P.Cw[2];
    W.nee = c->P.nee;
    W.L = c->P.nee ? c->P.ny - 1.0 : (double)c->P.ny;
    const int mode = c->read_mode();
    const void* b = cur_buf(c);
    cudaError_t e = LBM_DISPATCH(c, launch_nush_tb<double>(b, c->G, c->cd, mode, W, c->d_out + OUT_SCRATCH, out_at(c, 20), c->stream),
                                 launch_nush_tb<float>(b, c->G, c->cf, mode, W, c->d_out + OUT_SCRATCH, out_at(c, 20), c->stream),
                                 launch_nush_tb<__nv_bfloat16>(b, c->G, c->cf, mode, W, c->d_out + OUT_SCRATCH, out_at(c, 20), c->stream),
                                 launch_nush_tb<__half>(b, c->G, c->cf, mode, W, c->d_out + OUT_SCRATCH, out_at(c, 20), c->stream));
    e = fetch(c, e, 20, 4, out);
    if (e != cudaSuccess) return c->cuda_fail(e, "lbm_nusselt_sherwood_tb");
    for (int k = 0; k < 4; ++k)
        if (!std::isfinite(out[k]))
            return c->fail(LBM_ERR_DIVERGED, "lbm_nusselt_sherwood_tb: non-finite result");
    return LBM_OK;
}

namespace {

// The residual pass over the updated rows: h[0..3] = max |phi_now - phi_snap|,
// h[4..7] = max |phi_now| (phi = u_x, u_y, T, C), h[8] != 0 if a value is not finite;
// the snapshot is replaced by phi_now.
lbm_status residual_maxima(lbm_ctx* c, const char* who, double h[9]) {
    DeviceGuard dg(c->device);
    const size_t n = c->nodes();
    if (!c->d_snap) {
        c->d_snap = c->dalloc(4 * n * c->rsz);
        if (!c->d_snap) return c->fail(LBM_ERR_NOMEM, "%s: no device memory", who);
    }
    const int mode = c->read_mode();
    const void* b = cur_buf(c);
    double *o = out_at(c, 8), *slots = c->d_out + OUT_SLOTS;
    cudaError_t e = LBM_DISPATCH(
        c, launch_residual<double>(b, c->G, c->cd, mode, c->d_snap, slots, o, c->stream),
        launch_residual<float>(b, c->G, c->cf, mode, c->d_snap, slots, o, c->stream),
        launch_residual<__nv_bfloat16>(b, c->G, c->cf, mode, c->d_snap, slots, o, c->stream),
        launch_residual<__half>(b, c->G, c->cf, mode, c->d_snap, slots, o, c->stream));
    e = fetch(c, e, 8, 9, h);
    if (e != cudaSuccess) return c->cuda_fail(e, who);
    if (h[8] != 0.0) return c->fail(LBM_ERR_DIVERGED, "%s: non-finite field at t=%lld", who, (long long)c->t);
    if (!c->snap_valid)   // no earlier fields: the changes are unknown
        for (int q = 0; q < 4; ++q) h[q] = INFINITY;
    c->snap_valid = true;
    return LBM_OK;
}

}  // namespace

lbm_status lbm_residual(lbm_ctx* c, double* r) {
    if (!c || !r) {
        set_global_error("lbm_residual: NULL argument");
        return LBM_ERR_INVALID;
    }
    double h[9];
    lbm_status st = residual_maxima(c, "lbm_residual", h);
    if (st != LBM_OK) return st;
    double res = 0.0;
    for (int q = 0; q < 4; ++q) {
        double rq = h[4 + q] > 0 ? h[q] / h[4 + q] : (h[q] > 0 ? INFINITY : 0.0);
        res = rq > res ? rq : res;
    }
    *r = res;
    return LBM_OK;
}

lbm_status lbm_residual_parts(lbm_ctx* c, double parts[8]) {
    if (!c || !parts) {
        set_global_error("lbm_residual_parts: NULL argument");
        return LBM_ERR_INVALID;
    }
    double h[9];
    lbm_status st = residual_maxima(c, "lbm_residual_parts", h);
    if (st != LBM_OK) return st;
    for (int q = 0; q < 8; ++q) parts[q] = h[q];
    return LBM_OK;
}

lbm_status lbm_halo_bytes(const lbm_ctx* c, size_t* bytes) {
    if (!c || !bytes) {
        set_global_error("lbm_halo_bytes: NULL argument");
        return LBM_ERR_INVALID;
    }
    *bytes = 5 * (size_t)c->G.nx * c->esz;
    return LBM_OK;
}

namespace {

// side 0: the cut below the slab, 1: the cut above it.  Export reads the populations of
// the slab's outermost updated row that cross the cut; import writes the neighbour's into
// the ghost row on that side.
lbm_status halo_copy(lbm_ctx* c, int side, void* face, bool pack, const char* who) {
    if (!c || !face || (side != 0 && side != 1)) {
        set_global_error("%s: NULL argument or side not 0 / 1", who);
        return LBM_ERR_INVALID;
    }
    const bool cut = side == 0 ? c->G.jb > 0 : c->G.je < c->G.ny;
    if (!cut) return c->fail(LBM_ERR_INVALID, "%s: side %d of this context is a wall, not a cut", who, side);
    DeviceGuard dg(c->device);
    // export below: the bottom row's downward populations; export above: the top row's
    // upward ones; import below fills the lower ghost row with the upward populations of
    // the slab beneath, import above the upper ghost row with the downward ones
    const int row = pack ? (side == 0 ? c->G.jb : c->G.je - 1) : (side == 0 ? c->G.jb - 1 : c->G.je);
    const int up = pack ? side : 1 - side;
    void* b = c->layout == LBM_AB_PULL ? c->buf[c->cur] : c->buf[0];
    const int pk = pack ? 1 : 0;
    cudaError_t e = LBM_DISPATCH(c, launch_halo<double>(b, c->G, row, up, face, pk, c->stream),
                                 launch_halo<float>(b, c->G, row, up, face, pk, c->stream),
                                 launch_halo<__nv_bfloat16>(b, c->G, row, up, face, pk, c->stream),
                                 launch_halo<__half>(b, c->G, row, up, face, pk, c->stream));
    if (e != cudaSuccess) return c->cuda_fail(e, who);
    return LBM_OK;
}

}  // namespace

lbm_status lbm_halo_export(lbm_ctx* c, int side, void* face) {
    return halo_copy(c, side, face, true, "lbm_halo_export");
}

lbm_status lbm_halo_import(lbm_ctx* c, int side, const void* face) {
    return halo_copy(c, side, const_cast<void*>(face), false, "lbm_halo_import");
}

// Checkpoint layout: header, then the 19 state planes, then the 4 history planes.
namespace {
// A stored deviation as FP64: element k of a state array of precision prec (FP16 holds
// the deviation scaled by 2^12), and the reverse (rounded to nearest for narrower types).
double decode_value(int prec, const char* base, size_t k) {
    switch (prec) {
        case LBM_F64: return ((const double*)base)[k];
        case LBM_F32: return (double)((const float*)base)[k];
        case LBM_BF16: return (double)__bfloat162float(((const __nv_bfloat16*)base)[k]);
        default: return (double)__half2float(((const __half*)base)[k]) / 4096.0;
    }
}
void encode_value(int prec, char* base, size_t k, double v) {
    switch (prec) {
        case LBM_F64: ((double*)base)[k] = v; break;
        case LBM_F32: ((float*)base)[k] = (float)v; break;
        case LBM_BF16: ((__nv_bfloat16*)base)[k] = __float2bfloat16_rn((float)v); break;
        default: ((__half*)base)[k] = __float2half_rn((float)(v * 4096.0)); break;
    }
}
}  // namespace

namespace {
struct CkptHeader {
    char magic[8];
    int32_t version, nx, ny, prec, layout, pitch;
    int64_t t;
    lbm_params P;
};
}  // namespace

lbm_status lbm_save(lbm_ctx* c, void* buf, size_t* len) {
    if (!c || !len) {
        set_global_error("lbm_save: NULL argument");
        return LBM_ERR_INVALID;
    }
    const size_t need = sizeof(CkptHeader) + c->state_bytes() + c->hist_bytes();
    if (!buf) {
        *len = need;
        return LBM_OK;
    }
    if (*len < need) return c->fail(LBM_ERR_INVALID, "lbm_save: buffer of %zu bytes, need %zu", *len, need);
    DeviceGuard dg(c->device);
    CkptHeader h;
    std::memset(&h, 0, sizeof h);
    std::memcpy(h.magic, "LBMDDC1", 8);
    h.version = 2;   // 2: lbm_params carries the wall-node fields (nee, BiT, BiC)
    h.nx = c->G.nx;
    h.ny = c->G.ny;
    h.prec = c->prec;
    h.layout = c->layout;
    h.pitch = c->G.pitch;
    h.t = c->t;
    h.P = c->P;
    std::memcpy(buf, &h, sizeof h);
    char* p = (char*)buf + sizeof h;
    cudaError_t e = cudaMemcpyAsync(p, cur_buf(c), c->state_bytes(), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p + c->state_bytes(), c->hist, c->hist_bytes(), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return c->cuda_fail(e, "lbm_save");
    *len = need;
    return LBM_OK;
}

lbm_status lbm_load(lbm_ctx* c, const void* buf, size_t len) {
    if (!c || !buf) {
        set_global_error("lbm_load: NULL argument");
        return LBM_ERR_INVALID;
    }
    CkptHeader h;
    if (len < sizeof h) return c->fail(LBM_ERR_INVALID, "lbm_load: truncated checkpoint");
    std::memcpy(&h, buf, sizeof h);
    if (std::memcmp(h.magic, "LBMDDC1", 8) != 0 || h.version != 2)
        return c->fail(LBM_ERR_INVALID, "lbm_load: not a checkpoint of this library version");
    if (const char* bad = check_params(h.P))
        return c->fail(LBM_ERR_INVALID, "lbm_load: checkpoint parameters: %s", bad);
    if (h.P.nee && c->layout != LBM_AB_PULL)
        return c->fail(LBM_ERR_INVALID, "lbm_load: walls with nodes on them need the two-buffer layout");
    if (h.nx != c->G.nx || h.ny != c->G.ny || h.layout != c->layout)
        return c->fail(LBM_ERR_INVALID, "lbm_load: checkpoint does not match this context");
    if (h.prec < LBM_F64 || h.prec > LBM_F16)
        return c->fail(LBM_ERR_INVALID, "lbm_load: checkpoint of unknown precision %d", h.prec);
    const size_t src_esz = storage_size(h.prec), src_rsz = h.prec == LBM_F64 ? 8 : 4;
    const size_t src_plane = (size_t)h.ny * (size_t)h.pitch;
    const size_t src_state = (size_t)NQ * src_plane * src_esz, src_hist = 4 * src_plane * src_rsz;
    if (h.pitch < h.nx || len < sizeof h + src_state + src_hist)
        return c->fail(LBM_ERR_INVALID, "lbm_load: truncated checkpoint");
    DeviceGuard dg(c->device);
    const int slot = slot_for(c, h.t);
    const char* p = (const char*)buf + sizeof h;
    cudaError_t e;
    if (h.prec == c->prec && h.pitch == c->G.pitch) {
        e = cudaMemcpyAsync(c->buf[slot], p, c->state_bytes(), cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(c->hist, p + c->state_bytes(), c->hist_bytes(), cudaMemcpyHostToDevice,
                                c->stream);
    } else {
        // another storage precision: every stored deviation and history value is decoded
        // to FP64 and encoded in this context's precision (exact when widening, rounded to
        // nearest when narrowing), row by row into this context's row pitch
        std::vector<char> st;
        try {
            st.assign(c->state_bytes() + c->hist_bytes(), 0);
        } catch (...) {
            return c->fail(LBM_ERR_NOMEM, "lbm_load: no host memory to convert the checkpoint");
        }
        const size_t plane = c->G.plane;
        for (int q = 0; q < NQ; ++q)
            for (int j = 0; j < h.ny; ++j)
                for (int i = 0; i < h.nx; ++i) {
                    const size_t a = (size_t)q * src_plane + (size_t)j * h.pitch + i;
                    const size_t b = (size_t)q * plane + (size_t)j * c->G.pitch + i;
                    encode_value(c->prec, st.data(), b, decode_value(h.prec, p, a));
                }
        const char* ph = p + src_state;
        char* dh = st.data() + c->state_bytes();
        for (int k = 0; k < 4; ++k)
            for (int j = 0; j < h.ny; ++j)
                for (int i = 0; i < h.nx; ++i) {
                    const size_t a = (size_t)k * src_plane + (size_t)j * h.pitch + i;
                    const size_t b = (size_t)k * plane + (size_t)j * c->G.pitch + i;
                    const double v = src_rsz == 8 ? ((const double*)ph)[a] : (double)((const float*)ph)[a];
                    if (c->rsz == 8)
                        ((double*)dh)[b] = v;
                    else
                        ((float*)dh)[b] = (float)v;
                }
        e = cudaMemcpyAsync(c->buf[slot], st.data(), c->state_bytes(), cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(c->hist, dh, c->hist_bytes(), cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);   // before st is released
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return c->cuda_fail(e, "lbm_load");
    c->P = h.P;
    c->cd = make_coef<double>(c->P);
    c->cf = make_coef<float>(c->P);
    c->cf.sr = c->round_nearest ? 0 : 1;
    c->cf.seed_off = (long long)(c->slab_y0 - c->G.jb) * c->G.pitch;
    c->cd.poro = (c->poro && c->rsz == 8) ? (const double*)c->poro : nullptr;
    c->cf.poro = (c->poro && c->rsz == 4) ? (const float*)c->poro : nullptr;
    drop_graphs(c);                         // constants are baked into the captured launches
    c->t = h.t;
    c->cur = slot;
    c->snap_valid = false;
    return LBM_OK;
}

lbm_status lbm_get_params(const lbm_ctx* c, lbm_params* out) {
    if (!c || !out) {
        set_global_error("lbm_get_params: NULL argument");
        return LBM_ERR_INVALID;
    }
    *out = c->P;
    return LBM_OK;
}

size_t lbm_device_bytes(const lbm_ctx* c) { return c ? c->bytes : 0; }

void lbm_destroy(lbm_ctx* c) {
    if (!c) return;
    DeviceGuard dg(c->device);
    if (c->stream) cudaStreamSynchronize(c->stream);
    drop_graphs(c);
    c->dfree(c->buf[0], c->state_bytes());
    c->dfree(c->buf[1], c->state_bytes());
    c->dfree(c->hist, c->hist_bytes());
    c->dfree(c->hist_alt, c->hist_bytes());
    c->dfree(c->d_out, OUT_DOUBLES * sizeof(double));
    g_host_slots.give(c->h_out);
    c->dfree(c->d_fields, 5 * c->fields_cap * sizeof(double));
    c->dfree(c->d_snap, 4 * c->nodes() * c->rsz);
    c->dfree(c->d_stage, 2 * c->nodes() * sizeof(double));
    c->dfree(c->poro, 2 * c->G.plane * c->rsz);
    if (c->ev_fork) cudaEventDestroy(c->ev_fork);
    if (c->ev_join) cudaEventDestroy(c->ev_join);
    if (c->aux) cudaStreamDestroy(c->aux);
    if (c->own_stream) cudaStreamDestroy(c->stream);
    delete c;
}

const char* lbm_last_error(const lbm_ctx* c) {
    if (c) return c->err.c_str();
    return g_last_error.c_str();
}

}  // extern "C"
