// Steady-state residual without any device allocation.
//
// lbm_residual() allocates its snapshot on the first call.  Some callers cannot allocate
// device memory at that point: a host framework that has reserved the device memory for its
// own pool, or a loop that must not stall on cudaMalloc / cudaFree, which can synchronise
// the device.  lbm_residual_noalloc() computes the same residual with the caller's
// snapshot buffer; the pass's slots belong to the context, so that calls on different
// contexts do not meet.  There is no counterpart in the paper; this is plumbing.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>

#include "../../include/lbm.h"
#include "lbm_kernels.cuh"

using namespace lbm;

namespace {

inline const Coef<double>& coef_of(const CtxView& v, double*) { return *v.cd; }
inline const Coef<float>& coef_of(const CtxView& v, float*) { return *v.cf; }

template <typename S>
cudaError_t launch(const CtxView& v, double* snap) {
    using R = typename Real<S>::type;
    return launch_residual_pass<S, double>((const S*)v.buf, v.G, coef_of(v, (R*)nullptr), v.mode, snap, v.slots,
                                           v.out, v.stream);
}

lbm_status fail(lbm_ctx* ctx, lbm_status s, const char* m, const char* detail = "") {
    char msg[256];
    std::snprintf(msg, sizeof msg, "lbm_residual_noalloc: %s%s", m, detail);
    lbm_set_error(ctx, msg);
    return s;
}

}  // namespace

extern "C" {

lbm_status lbm_residual_noalloc(lbm_ctx* ctx, double* snapshot, int have_snapshot, double* r) {
    CtxView v;
    if (!ctx || !snapshot || !r || !lbm_ctx_view(ctx, &v))
        return fail(ctx, LBM_ERR_INVALID, "ctx, snapshot and r must be non-NULL");
    if (v.G.jb != 0 || v.G.je != v.G.ny)   // a slab: its snapshot would include ghost rows
        return fail(ctx, LBM_ERR_INVALID, "not defined on a slab (use lbm_residual_parts)");
    DeviceGuard dg(v.device);      // the launches on the context's stream and the copy belong to it
    cudaError_t e;
    switch (v.prec) {
        case LBM_F64: e = launch<double>(v, snapshot); break;
        case LBM_F32: e = launch<float>(v, snapshot); break;
        case LBM_BF16: e = launch<__nv_bfloat16>(v, snapshot); break;
        default: e = launch<__half>(v, snapshot); break;
    }
    double h[9];
    if (e == cudaSuccess && !v.out_on_host)
        e = cudaMemcpyAsync(h, v.out, sizeof h, cudaMemcpyDeviceToHost, v.stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(v.stream);
    if (e == cudaSuccess && v.out_on_host) std::memcpy(h, v.out, sizeof h);
    if (e != cudaSuccess) return fail(ctx, LBM_ERR_CUDA, "", cudaGetErrorString(e));
    if (h[8] != 0.0) return fail(ctx, LBM_ERR_DIVERGED, "non-finite field value");
    double res = 0.0;
    for (int q = 0; q < 4; ++q) {
        const double rq = h[4 + q] > 0 ? h[q] / h[4 + q] : (h[q] > 0 ? INFINITY : 0.0);
        res = rq > res ? rq : res;
    }
    *r = have_snapshot ? res : INFINITY;
    return LBM_OK;
}

}  // extern "C"
