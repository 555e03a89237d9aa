// sg_tune (declared in include/smolyak.h): measured choice of the row kernels'
// plan for one context.
//
// Three knobs, searched one after another (coordinate descent: each in turn
// over its candidates with the others at their best so far), every candidate
// timed on real applies of the caller's block size:
//   1. vectors per lane (1, 2, 4): wider loads of the input copy and fewer
//      lanes per row, against more rows in flight (FP64 with one vector per
//      lane makes no copy: rows_direct);
//   2. rows per window, in units of 16 (1, 2, 4): how many rows a block takes;
//   3. the shared memory that SG_ROW_SHARE resident blocks may use: a window
//      ends early where its entries would exceed its part.
// A row's sum does not depend on the plan, so results do not either.
#include <algorithm>
#include <cmath>
#include <limits>
#include <string>
#include <vector>

#include "sg_internal.h"

namespace {

struct Plan {
    int slice_vt, warp_vt, smem_kb;
};

struct Tuner {
    sg_ctx *ctx;
    cudaStream_t s;
    const double *x;
    double *y;
    int nvec;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t err = cudaSuccess;

    // Cuts the row operator into the windows of p.  False when that fails: the
    // operator in force, and the plan that it was cut by, stay.  The new operator
    // is formed beside the old one; without the memory for both, p is not taken
    // (no error of the tuner's: err stays clear).
    bool install(const Plan &p)
    {
        sg::HostTables &T = ctx->host;
        const int vt = T.slice_vt, units = T.warp_vt, budget = T.fbudget;
        const bool same = sg::row_window_units(T) == p.warp_vt && sg::row_budget(T, ctx->prob.prec) == p.smem_kb * 1024;
        T.slice_vt = p.slice_vt;
        T.warp_vt = p.warp_vt;
        T.fbudget = p.smem_kb * 1024;
        const cudaError_t e = same ? cudaSuccess : sg::build_rows(ctx);
        if (e != cudaSuccess) {
            T.slice_vt = vt;
            T.warp_vt = units;
            T.fbudget = budget;
            if (e != cudaErrorMemoryAllocation) err = e;
            return false;
        }
        ctx->plan_version++;
        return true;
    }

    // Median of three timed applies after one untimed; negative on failure.
    double time_apply(sg_status *st)
    {
        std::vector<float> t;
        for (int k = 0; k < 4 && *st == SG_OK; k++) {
            if ((err = cudaEventRecord(e0, s)) != cudaSuccess) { *st = SG_ECUDA; break; }
            *st = sg_apply_H(ctx, x, y, nvec, s);
            if (*st == SG_OK && (err = cudaEventRecord(e1, s)) != cudaSuccess) *st = SG_ECUDA;
            if (*st == SG_OK && (err = cudaEventSynchronize(e1)) != cudaSuccess) *st = SG_ECUDA;
            float ms = 0.f;
            if (*st == SG_OK) cudaEventElapsedTime(&ms, e0, e1);
            if (k > 0) t.push_back(ms);
        }
        if (*st != SG_OK) return -1.0;
        std::sort(t.begin(), t.end());
        return t[1];
    }
};

}  // namespace

extern "C" sg_status sg_tune(sg_ctx *ctx, int nvec, int *slice_vt, double *ms_out, void *stream)
{
    if (!ctx) return SG_EINVAL;
    if (!ctx->has_device) { ctx->last_error = "sg_tune: context was made by sg_plan"; return SG_EINVAL; }
    if (!sg_on_ctx_device(ctx)) { ctx->last_error = std::string("sg_tune: ") + "the current CUDA device is not the one the context was made on"; return SG_EINVAL; }
    if (nvec < 1 || nvec > 64) { ctx->last_error = "sg_tune: need 1 <= nvec <= 64"; return SG_EINVAL; }
    sg::HostTables &T = ctx->host;
    if (!T.rows || !T.pairs) {  // not a pair potential: the default plan
        if (slice_vt) *slice_vt = 0;
        if (ms_out) *ms_out = 0.0;
        return SG_OK;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaStreamSynchronize(s) != cudaSuccess) { ctx->last_error = "sg_tune: stream synchronize"; return SG_ECUDA; }
    const size_t n = (size_t)T.n_cs * nvec;
    double *x = nullptr, *y = nullptr;
    cudaError_t e;
    if ((e = cudaMalloc(&x, n * sizeof(double))) != cudaSuccess || (e = cudaMalloc(&y, n * sizeof(double))) != cudaSuccess) {
        if (x) cudaFree(x);
        ctx->last_error = std::string("sg_tune: cudaMalloc: ") + cudaGetErrorString(e);
        return SG_ENOMEM;
    }
    {
        std::vector<double> h(n);
        for (size_t i = 0; i < n; i++) h[i] = 1.0 / (1.0 + (double)(i % 977)) - 0.25;
        e = cudaMemcpy(x, h.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    }
    Tuner tu{ctx, s, x, y, nvec};
    if (e == cudaSuccess) e = cudaEventCreate(&tu.e0);
    if (e == cudaSuccess) e = cudaEventCreate(&tu.e1);
    sg_status st = e == cudaSuccess ? SG_OK : SG_ECUDA;
    const sg_precision prec = ctx->prob.prec;
    const Plan original{sg::row_vt(T, prec), sg::row_window_units(T), sg::row_budget(T, prec) / 1024};
    Plan best = original;
    double best_ms = std::numeric_limits<double>::infinity();
    std::vector<Plan> tried;
    auto evaluate = [&](const Plan &p) {
        for (const Plan &q : tried)
            if (q.slice_vt == p.slice_vt && q.warp_vt == p.warp_vt && q.smem_kb == p.smem_kb) return;
        tried.push_back(p);
        if (st != SG_OK || !tu.install(p)) {
            if (tu.err != cudaSuccess) st = SG_ECUDA;
            return;
        }
        const double ms = tu.time_apply(&st);
        if (st == SG_OK && ms >= 0.0 && ms < best_ms) { best_ms = ms; best = p; }
    };
    evaluate(original);
    for (int v : {1, 2, 4}) evaluate(Plan{v, best.warp_vt, best.smem_kb});
    for (int v : {1, 2, 4}) evaluate(Plan{best.slice_vt, v, best.smem_kb});
    for (int kb : ctx->fp32 ? std::vector<int>{52, 70, 104} : std::vector<int>{70, 104})
        evaluate(Plan{best.slice_vt, best.warp_vt, kb});
    // keep the fastest plan (the original one if none could be timed)
    const bool ok = std::isfinite(best_ms);
    const cudaError_t keep_err = tu.err;
    tu.err = cudaSuccess;
    if (!tu.install(ok ? best : original) && st == SG_OK) {
        st = tu.err != cudaSuccess ? SG_ECUDA : SG_ENOMEM;
        if (st == SG_ENOMEM)
            ctx->last_error = "sg_tune: no memory to install the fastest plan; the plan in force (sg_tune_plan) stays";
    }
    if (tu.e0) cudaEventDestroy(tu.e0);
    if (tu.e1) cudaEventDestroy(tu.e1);
    cudaFree(x);
    cudaFree(y);
    if (st != SG_OK) {
        // a failed apply has set its own message; CUDA errors of the tuner set this one
        const cudaError_t ce = tu.err != cudaSuccess ? tu.err : keep_err != cudaSuccess ? keep_err : e;
        if (st == SG_ECUDA && ce != cudaSuccess) ctx->last_error = std::string("sg_tune: ") + cudaGetErrorString(ce);
        return st;
    }
    if (slice_vt) *slice_vt = ok ? best.slice_vt : 0;
    if (ms_out) *ms_out = ok ? best_ms : 0.0;
    return SG_OK;
}

extern "C" sg_status sg_tune_plan(const sg_ctx *ctx, int *slice_vt, int *warp_vt, int *smem_kb)
{
    if (!ctx) return SG_EINVAL;
    const sg::HostTables &T = ctx->host;
    const bool plan = T.rows && T.pairs;
    if (slice_vt) *slice_vt = plan ? sg::row_vt(T, ctx->prob.prec) : 0;
    if (warp_vt) *warp_vt = plan ? sg::row_window_units(T) : 0;
    if (smem_kb) *smem_kb = plan ? sg::row_budget(T, ctx->prob.prec) / 1024 : 0;
    return SG_OK;
}
