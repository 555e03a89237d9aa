// Many Smolyak problems per apply (declared in include/smolyak.h): the row
// windows of all problems go to the device in one launch, so a batch of small
// and large problems keeps every SM busy until the end.
#include <algorithm>
#include <new>
#include <string>
#include <vector>

#include "sg_arena.h"
#include "sg_internal.h"

// A problem with at least this many rows fills the GPU for several waves by
// itself: it runs as its own launches (parameters in the kernel's parameter
// bank, windows of its own plan) inside the batch's sequence, and only the
// smaller problems share the packed launches.  Two FP32 vectors each, packed
// and on its own: 646,646 rows 47.8 and 46.3 us; 293,930 rows with eight small
// problems 22.9 and 26.9.
constexpr int64_t kSoloRows = 524288;

struct sg_batch {
    std::vector<sg_ctx *> ctxs;
    std::vector<int> plan_versions;    // of the contexts when the batch was made
    int device = 0;
    bool fp32 = false;
    std::vector<long long> cs_prefix;  // host copy
    int64_t n_terms = 0;
    const long long *d_cs_prefix = nullptr;
    const sg::RowOp *d_ops = nullptr;  // one per problem
    const int2 *items = nullptr;       // (problem, window) of the packed problems, most entries first
    const int2 *stage_items = nullptr; // (problem, chunk of 256 rows) of the packed problems
    int n_items = 0, n_stage = 0, cap = 0, wrows = 16;
    const int2 *all_items = nullptr, *all_stage = nullptr;  // the same over every row-form problem
    int n_all = 0, n_all_stage = 0, all_cap = 0;
    std::vector<int> packed, solo;     // row-form problems: shared launches, launches of their own
    std::vector<int> generic;          // problems applied term by term
    std::vector<void *> allocations;
    // workspace: input copies and flags of the row-form problems, accumulators
    // and exponents of the others (all from the start of the problem's vectors)
    void *xs = nullptr;
    unsigned *flags = nullptr;
    unsigned long long *acc = nullptr;
    long long *maxbits = nullptr;
    int acc_nvec = 0;
    // the apply's launch sequence captured as a graph, for the last (x, y, nvec, stream)
    cudaGraphExec_t graph = nullptr;
    const double *gx = nullptr;
    double *gy = nullptr;
    int gnvec = 0;
    cudaStream_t gstream = nullptr;
    int64_t graph_launches = 0;
    std::string last_error;
};

namespace {

sg_status bfail(sg_batch *b, sg_status st, const std::string &msg)
{
    if (b) b->last_error = msg;
    return st;
}

void drop_graph(sg_batch *b)
{
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
    b->gx = nullptr;
    b->gy = nullptr;
    b->gnvec = 0;
    b->gstream = nullptr;
}

void free_workspace(sg_batch *b)
{
    if (b->acc) cudaFree(b->acc);
    if (b->maxbits) cudaFree(b->maxbits);
    if (b->xs) cudaFree(b->xs);
    if (b->flags) cudaFree(b->flags);
    b->acc = nullptr;
    b->maxbits = nullptr;
    b->xs = nullptr;
    b->flags = nullptr;
    b->acc_nvec = 0;
}

void free_all(sg_batch *b)
{
    drop_graph(b);
    for (void *p : b->allocations) cudaFree(p);
    b->allocations.clear();
    free_workspace(b);
}

}  // namespace

extern "C" sg_status sg_batch_create(sg_ctx *const *ctxs, int n, sg_batch **out)
{
    if (!out) return SG_EINVAL;
    *out = nullptr;
    if (!ctxs || n < 1 || n > 65535) return SG_EINVAL;
    sg_batch *b = new (std::nothrow) sg_batch;
    if (!b) return SG_ENOMEM;
    for (int j = 0; j < n; j++) {
        sg_ctx *c = ctxs[j];
        if (!c || !c->has_device) { delete b; return SG_EINVAL; }
        if (c->prob.prec == SG_DF64) { delete b; return SG_EUNSUPPORTED; }  // double-float contexts are applied one by one
        if (j > 0 && (c->device != b->device || c->fp32 != b->fp32)) { delete b; return SG_EINVAL; }
        b->device = c->device;
        b->fp32 = c->fp32;
        b->ctxs.push_back(c);
        b->plan_versions.push_back(c->plan_version);
    }
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess || cur != b->device) { delete b; return SG_EINVAL; }

    b->cs_prefix.assign(n + 1, 0);
    std::vector<sg::RowOp> ops(n);
    struct Item { int nent, j, w; };
    std::vector<Item> it, all;
    std::vector<int2> stage, all_stage;
    for (int j = 0; j < n; j++) {
        const sg_ctx *c = ctxs[j];
        b->cs_prefix[j + 1] = b->cs_prefix[j] + c->host.n_cs;
        b->n_terms += c->host.n_terms;
        ops[j] = c->rop;
        if (!c->host.rows) { b->generic.push_back(j); continue; }
        b->all_cap = std::max(b->all_cap, c->rop.cap);
        for (int w = 0; w < c->rop.nwin; w++) all.push_back({c->win_entries[w], j, w});
        for (int q = 0; q * (int64_t)256 < c->host.n_cs; q++) all_stage.push_back(make_int2(j, q));
        if (c->host.n_cs >= kSoloRows) { b->solo.push_back(j); continue; }
        b->packed.push_back(j);
        b->cap = std::max(b->cap, c->rop.cap);
        b->wrows = std::max(b->wrows, c->rop.wrows);
        for (int w = 0; w < c->rop.nwin; w++) it.push_back({c->win_entries[w], j, w});
        for (int q = 0; q * (int64_t)256 < c->host.n_cs; q++) stage.push_back(make_int2(j, q));
    }
    if (all.size() > (size_t)0x7FFFFFFF) { delete b; return SG_EUNSUPPORTED; }
    auto largest_first = [](std::vector<Item> &v) {
        std::stable_sort(v.begin(), v.end(), [](const Item &a, const Item &c) { return a.nent > c.nent; });
        std::vector<int2> out(v.size());
        for (size_t q = 0; q < v.size(); q++) out[q] = make_int2(v[q].j, v[q].w);
        return out;
    };
    const std::vector<int2> items = largest_first(it), all_items = largest_first(all);
    b->n_items = (int)items.size();
    b->n_stage = (int)stage.size();
    b->n_all = (int)all_items.size();
    b->n_all_stage = (int)all_stage.size();
    sg::Arena A;
    const size_t o[6] = {A.add(ops), A.add(b->cs_prefix), A.add(items), A.add(stage), A.add(all_items), A.add(all_stage)};
    unsigned char *base = nullptr;
    const cudaError_t e = A.put(&base);
    if (base) b->allocations.push_back(base);
    if (e != cudaSuccess) {
        const sg_status st = e == cudaErrorMemoryAllocation ? SG_ENOMEM : SG_ECUDA;
        free_all(b);
        delete b;
        return st;
    }
    b->d_ops = reinterpret_cast<const sg::RowOp *>(base + o[0]);
    b->d_cs_prefix = reinterpret_cast<const long long *>(base + o[1]);
    b->items = reinterpret_cast<const int2 *>(base + o[2]);
    b->stage_items = reinterpret_cast<const int2 *>(base + o[3]);
    b->all_items = reinterpret_cast<const int2 *>(base + o[4]);
    b->all_stage = reinterpret_cast<const int2 *>(base + o[5]);
    *out = b;
    return SG_OK;
}

extern "C" sg_status sg_batch_size(const sg_batch *b, int64_t *n_cs_total, int64_t *n_terms_total,
                                   int *launches_per_apply)
{
    if (!b) return SG_EINVAL;
    if (n_cs_total) *n_cs_total = b->cs_prefix.back();
    if (n_terms_total) *n_terms_total = b->n_terms;
    if (launches_per_apply) {
        // at most; row form: input copies (where made), rows, settle; term by term: max|x|, terms, finalisation
        const int l = (b->packed.empty() ? 0 : 3) + 3 * (int)(b->solo.size() + b->generic.size());
        *launches_per_apply = l;
    }
    return SG_OK;
}

sg_status enqueue_apply(sg_batch *b, const double *x, double *y, int nvec, cudaStream_t s);

extern "C" sg_status sg_apply_H_batch(sg_batch *b, const double *x, double *y, int nvec, void *stream)
{
    if (!b) return SG_EINVAL;
    if (!x || !y) return bfail(b, SG_EINVAL, "x or y is NULL");
    if (nvec < 1) return bfail(b, SG_EINVAL, "nvec must be >= 1");
    const int nprob = (int)b->ctxs.size();
    const size_t total = (size_t)b->cs_prefix.back() * (size_t)nvec;
    if ((x < y + total) && (y < x + total)) return bfail(b, SG_EINVAL, "x and y overlap");
    if ((size_t)nprob * nvec > 65535u * 65535u) return bfail(b, SG_EUNSUPPORTED, "too many vectors");
    if (nvec > 65535) return bfail(b, SG_EUNSUPPORTED, "nvec > 65535");
    for (int j = 0; j < nprob; j++)
        if (b->ctxs[j]->plan_version != b->plan_versions[j])
            return bfail(b, SG_EINVAL, "problem " + std::to_string(j) +
                                           " was re-planned by sg_tune after the batch was made: recreate the batch");
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e;
    if (nvec > b->acc_nvec) {
        drop_graph(b);  // it names the old workspace
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess)
            return bfail(b, SG_ECUDA, std::string("stream synchronize: ") + cudaGetErrorString(e));
        free_workspace(b);
        if (!b->packed.empty() || !b->solo.empty()) {
            const size_t rb = b->fp32 ? 4 : 8, nf = (size_t)nprob * nvec * sizeof(unsigned);
            if ((e = cudaMalloc(&b->xs, (size_t)b->cs_prefix.back() * sg::xs_stride(nvec) * rb)) != cudaSuccess ||
                (e = cudaMalloc(&b->flags, nf)) != cudaSuccess)
                return bfail(b, SG_ENOMEM, std::string("workspace cudaMalloc: ") + cudaGetErrorString(e));
            if ((e = cudaMemsetAsync(b->flags, 0, nf, s)) != cudaSuccess)
                return bfail(b, SG_ECUDA, std::string("workspace memset: ") + cudaGetErrorString(e));
        }
        if (!b->generic.empty()) {
            const size_t words = total * sg::acc_words(b->fp32);
            if ((e = cudaMalloc(&b->acc, words * sizeof(unsigned long long))) != cudaSuccess ||
                (e = cudaMalloc(&b->maxbits, sizeof(long long) * (size_t)nprob * nvec)) != cudaSuccess)
                return bfail(b, SG_ENOMEM, std::string("workspace cudaMalloc: ") + cudaGetErrorString(e));
            if ((e = cudaMemsetAsync(b->acc, 0, words * sizeof(unsigned long long), s)) != cudaSuccess)
                return bfail(b, SG_ECUDA, std::string("workspace memset: ") + cudaGetErrorString(e));
        }
        b->acc_nvec = nvec;
    }
    // Replay the captured launch sequence when the same buffers, block size and
    // stream come back; capture it on first use.  Not on the legacy default
    // stream (it cannot be captured) nor while the caller is capturing the
    // stream itself (the launches then go into the caller's graph).
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (s != nullptr && (e = cudaStreamIsCapturing(s, &cs)) != cudaSuccess)
        return bfail(b, SG_ECUDA, std::string("stream capture query: ") + cudaGetErrorString(e));
    if (s != nullptr && cs == cudaStreamCaptureStatusNone) {
        if (!(b->graph && b->gx == x && b->gy == y && b->gnvec == nvec && b->gstream == s)) {
            drop_graph(b);
            cudaGraph_t g = nullptr;
            if ((e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal)) != cudaSuccess)
                return bfail(b, SG_ECUDA, std::string("begin capture: ") + cudaGetErrorString(e));
            const sg_status st = enqueue_apply(b, x, y, nvec, s);
            e = cudaStreamEndCapture(s, &g);
            if (st != SG_OK) { if (g) cudaGraphDestroy(g); return st; }
            if (e != cudaSuccess) return bfail(b, SG_ECUDA, std::string("end capture: ") + cudaGetErrorString(e));
            e = cudaGraphInstantiate(&b->graph, g, 0);
            cudaGraphDestroy(g);
            if (e != cudaSuccess) { b->graph = nullptr; return bfail(b, SG_ECUDA, std::string("graph instantiate: ") + cudaGetErrorString(e)); }
            b->gx = x; b->gy = y; b->gnvec = nvec; b->gstream = s;
        }
        if ((e = cudaGraphLaunch(b->graph, s)) != cudaSuccess)
            return bfail(b, SG_ECUDA, std::string("graph launch: ") + cudaGetErrorString(e));
        b->graph_launches++;
        return SG_OK;
    }
    return enqueue_apply(b, x, y, nvec, s);
}

// The launch sequence of one batched apply.
sg_status enqueue_apply(sg_batch *b, const double *x, double *y, int nvec, cudaStream_t s)
{
    const sg_precision prec = b->fp32 ? SG_MIXED : SG_FP64;
    const size_t rb = b->fp32 ? 4 : 8;
    cudaError_t e;
    sg::RowIO io{};
    io.x = x;
    io.y = y;
    io.xs = b->xs;
    io.flags = b->flags;
    io.nvec = nvec;
    io.stride = sg::xs_stride(nvec);
    io.nparts = 1;
    for (int j : b->solo) {
        const size_t c0 = (size_t)b->cs_prefix[j];
        sg::RowIO o = io;
        o.x += c0 * nvec;
        o.y += c0 * nvec;
        o.xs = static_cast<unsigned char *>(b->xs) + c0 * io.stride * rb;
        o.flags += (size_t)j * nvec;
        const sg_ctx *c = b->ctxs[j];
        const int vt = sg::row_vt(c->host, prec);
        if (sg::rows_direct(prec, vt, nvec)) o.xs = nullptr;
        if ((o.xs && (e = sg::launch_row_stage(c->rop, o, prec, s)) != cudaSuccess) ||
            (e = sg::launch_rows(c->rop, o, prec, vt, s)) != cudaSuccess ||
            (e = sg::launch_row_settle(o, c->rop.n, s)) != cudaSuccess)
            return bfail(b, SG_ECUDA, std::string("row launch: ") + cudaGetErrorString(e));
    }
    if (!b->packed.empty()) {
        const int vt = b->fp32 ? SG_F32_VT : SG_F64_VT;
        if (sg::rows_direct(prec, vt, nvec)) io.xs = nullptr;
        if ((io.xs &&
             (e = sg::launch_row_stage_batch(io, prec, b->d_cs_prefix, b->stage_items, b->n_stage, s)) != cudaSuccess) ||
            (e = sg::launch_rows_batch(b->d_ops, b->items, b->n_items, b->cap, b->wrows, io, prec, vt,
                                       b->d_cs_prefix, s)) != cudaSuccess ||
            (e = sg::launch_row_settle_batch(io, b->d_cs_prefix, (int)b->ctxs.size(), s)) != cudaSuccess)
            return bfail(b, SG_ECUDA, std::string("batched row launch: ") + cudaGetErrorString(e));
    }
    for (int j : b->generic) {
        sg::KParams kp = b->ctxs[j]->kp;
        const size_t off = (size_t)nvec * (size_t)b->cs_prefix[j];
        kp.acc = b->acc + off * sg::acc_words(b->fp32);
        if ((e = sg::launch_apply(kp, b->fp32, x + off, y + off, nvec, b->maxbits + (size_t)j * nvec, s)) != cudaSuccess)
            return bfail(b, SG_ECUDA, std::string("term launch: ") + cudaGetErrorString(e));
    }
    return SG_OK;
}

namespace sg {

sg_status batch_cheb(sg_batch *b, const ChebIO &io, const ChebState *st, bool restage, cudaStream_t s)
{
    if (!b->generic.empty()) return SG_EUNSUPPORTED;
    const sg_precision prec = b->fp32 ? SG_MIXED : SG_FP64;
    cudaError_t e = cudaSuccess;
    if (restage) {
        RowIO r{};
        r.x = io.X;
        r.xs = io.xs;
        r.nvec = 2;
        r.stride = xs_stride(2);
        e = launch_row_stage_batch(r, prec, b->d_cs_prefix, b->all_stage, b->n_all_stage, s);
    }
    if (e == cudaSuccess)
        e = launch_cheb_rows_batch(b->d_ops, b->all_items, b->n_all, b->all_cap, io, st, prec, b->d_cs_prefix, s);
    return e == cudaSuccess ? SG_OK : bfail(b, SG_ECUDA, std::string("recurrence launch: ") + cudaGetErrorString(e));
}

}  // namespace sg

extern "C" const char *sg_batch_last_error(const sg_batch *b)
{
    return b ? b->last_error.c_str() : "";
}

extern "C" void sg_batch_destroy(sg_batch *b)
{
    if (!b) return;
    free_all(b);
    delete b;
}
