// C ABI of libsmolyak (declared in include/smolyak.h).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "sg_arena.h"
#include "sg_internal.h"

namespace {

thread_local std::string g_create_error;

sg_status fail(sg_ctx *ctx, sg_status st, const std::string &msg)
{
    if (ctx) ctx->last_error = msg; else g_create_error = msg;
    return st;
}

sg_status cuda_fail(sg_ctx *ctx, cudaError_t e, const char *where)
{
    return fail(ctx, SG_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

template <typename T>
sg_status upload(sg_ctx *ctx, const std::vector<T> &v, const T **dst)
{
    void *p = nullptr;
    size_t bytes = std::max<size_t>(1, v.size()) * sizeof(T);
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();  // reported here; not by a later launch
        return fail(ctx, SG_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    }
    ctx->allocations.push_back(p);
    ctx->bytes_device += (int64_t)bytes;
    if (!v.empty()) {
        e = cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaMemcpy");
    }
    *dst = static_cast<const T *>(p);
    return SG_OK;
}

void free_workspace(sg_ctx *ctx)
{
    if (ctx->acc) cudaFree(ctx->acc);
    if (ctx->maxbits) cudaFree(ctx->maxbits);
    if (ctx->xs) cudaFree(ctx->xs);
    ctx->acc = nullptr;
    ctx->maxbits = nullptr;
    ctx->xs = nullptr;
    ctx->flags = nullptr;
    ctx->acc_nvec = 0;
}

void free_tables(sg_ctx *ctx)
{
    for (void *p : ctx->allocations) cudaFree(p);
    ctx->allocations.clear();
    sg::free_rows(ctx);
    ctx->bytes_device = 0;
}

void free_all(sg_ctx *ctx)
{
    free_tables(ctx);
    if (ctx->stage_x) cudaFree(ctx->stage_x);
    if (ctx->stage_y) cudaFree(ctx->stage_y);
    ctx->stage_x = ctx->stage_y = nullptr;
    if (ctx->pin) cudaFreeHost(ctx->pin);
    ctx->pin = nullptr;
    free_workspace(ctx);
}

// What the row form's set-up kernels and the index map read, and the harmonic energies.
cudaError_t upload_row_tables(sg_ctx *ctx)
{
    const sg::HostTables &T = ctx->host;
    sg::KParams &kp = ctx->kp;
    sg::Arena A;
    const int zero = 0;
    const size_t rank = A.add(T.rank_tab), lmin = A.add(T.lmin_tab), lvl = A.add(T.lvl), tab = A.add(T.tabd),
                 es = A.add(T.esplit), err = A.add(&zero, 1);
    unsigned char *base = nullptr;
    const cudaError_t e = A.put(&base);
    if (base) ctx->allocations.push_back(base);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();  // reported here; not by a later launch
        return e;
    }
    ctx->bytes_device += (int64_t)A.host.size();
    kp.rank_tab = reinterpret_cast<const int *>(base + rank);
    kp.lmin_tab = base + lmin;
    kp.lvl = reinterpret_cast<const sg::LevelInfo *>(base + lvl);
    kp.tabd = reinterpret_cast<const double *>(base + tab);
    kp.esplit = reinterpret_cast<const double *>(base + es);
    kp.err = reinterpret_cast<int *>(base + err);
    return cudaSuccess;
}

// The tables of the term-by-term kernel.
sg_status upload_term_tables(sg_ctx *ctx)
{
    const sg::HostTables &T = ctx->host;
    const sg::Problem &p = ctx->prob;
    sg::KParams &kp = ctx->kp;
    const std::vector<float> tabf(T.tabd.begin(), T.tabd.end());
    const std::vector<int> zero(1, 0);
    const int *errp = nullptr;
    sg_status st;
    if ((st = upload(ctx, T.levels, &kp.levels)) != SG_OK ||
        (st = upload(ctx, T.coefs, &kp.coefs)) != SG_OK ||
        (st = upload(ctx, T.order, &kp.order)) != SG_OK ||
        (st = upload(ctx, T.rank_tab, &kp.rank_tab)) != SG_OK ||
        (st = upload(ctx, T.lmin_tab, &kp.lmin_tab)) != SG_OK ||
        (st = upload(ctx, T.lvl, &kp.lvl)) != SG_OK ||
        (st = upload(ctx, T.tabd, &kp.tabd)) != SG_OK ||
        (st = upload(ctx, tabf, &kp.tabf)) != SG_OK ||
        (st = upload(ctx, p.mcoef, &kp.mcoef)) != SG_OK ||
        (st = upload(ctx, p.mnfac, &kp.mnfac)) != SG_OK ||
        (st = upload(ctx, p.mfoff, &kp.mfoff)) != SG_OK ||
        (st = upload(ctx, p.mfmode, &kp.mfmode)) != SG_OK ||
        (st = upload(ctx, p.mfpow, &kp.mfpow)) != SG_OK ||
        (st = upload(ctx, T.harm_mono, &kp.harm_mono)) != SG_OK ||
        (st = upload(ctx, T.esplit, &kp.esplit)) != SG_OK ||
        (st = upload(ctx, zero, &errp)) != SG_OK)
        return st;
    kp.err = const_cast<int *>(errp);
    return SG_OK;
}

// Apply workspace for nvec vectors.  Row form: per-vector flags (zero between
// applies) and the entry-major input copy.  Term-by-term kernel: fixed-point
// accumulators (zeroed here and left zeroed by every apply) and the
// per-vector max|x| words.
sg_status ensure_workspace(sg_ctx *ctx, int nvec, cudaStream_t s)
{
    if (nvec <= ctx->acc_nvec) return SG_OK;
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "stream synchronize");
    free_workspace(ctx);
    if (ctx->host.rows) {
        const size_t xs_bytes =
            (((size_t)ctx->host.n_cs * sg::xs_stride(nvec) * sg::row_value_bytes(ctx->prob.prec)) + 15) & ~(size_t)15;
        if ((e = cudaMalloc(&ctx->xs, xs_bytes + sizeof(unsigned) * (nvec + 1))) != cudaSuccess)
            return fail(ctx, SG_ENOMEM, std::string("workspace cudaMalloc: ") + cudaGetErrorString(e));
        ctx->flags = reinterpret_cast<unsigned *>(static_cast<unsigned char *>(ctx->xs) + xs_bytes);
        if ((e = cudaMemsetAsync(ctx->flags, 0, sizeof(unsigned) * (nvec + 1), s)) != cudaSuccess)
            return cuda_fail(ctx, e, "workspace memset");
    } else {
        const size_t words = (size_t)ctx->host.n_cs * nvec * sg::acc_words(ctx->fp32);
        if ((e = cudaMalloc(&ctx->acc, words * sizeof(unsigned long long))) != cudaSuccess ||
            (e = cudaMalloc(&ctx->maxbits, sizeof(long long) * nvec)) != cudaSuccess)
            return fail(ctx, SG_ENOMEM, std::string("workspace cudaMalloc: ") + cudaGetErrorString(e));
        if ((e = cudaMemsetAsync(ctx->acc, 0, words * sizeof(unsigned long long), s)) != cudaSuccess)
            return cuda_fail(ctx, e, "workspace memset");
        ctx->kp.acc = ctx->acc;
    }
    ctx->acc_nvec = nvec;
    return SG_OK;
}

sg::RowIO row_io(const sg_ctx *ctx, const double *x, double *y, int nvec)
{
    sg::RowIO io{};
    io.x = x;
    io.xs = ctx->xs;
    io.y = y;
    io.flags = ctx->flags;
    io.ticket = ctx->flags + ctx->acc_nvec;
    io.nvec = nvec;
    io.stride = sg::xs_stride(nvec);
    io.words = sg::acc_words(ctx->fp32);
    io.part = 0;
    io.nparts = 1;
    return io;
}

// The launches of one apply (workspace ready).
cudaError_t enqueue_apply(sg_ctx *ctx, const double *x, double *y, int nvec, cudaStream_t s)
{
    if (!ctx->host.rows) return sg::launch_apply(ctx->kp, ctx->fp32, x, y, nvec, ctx->maxbits, s);
    return sg::apply_rows(ctx, row_io(ctx, x, y, nvec), s);
}

// Device shared-memory opt-in limit of sm_100-class GPUs, used to size plans
// made without a device (sg_plan).
constexpr int kPlanSmemOptin = 232448;

sg_status plan(int D, int L, const sg_basis *basis, const sg_grid *grids,
                     const sg_hamiltonian *H, sg_precision prec, int smem_optin, sg_ctx **out)
{
    using namespace sg;
    if (!out) return fail(nullptr, SG_EINVAL, "out is NULL");
    *out = nullptr;
    if (D < 1) return fail(nullptr, SG_EINVAL, "D must be >= 1");
    if (D > kMaxD) return fail(nullptr, SG_EUNSUPPORTED, "D > 32");
    if (L < 0) return fail(nullptr, SG_EINVAL, "L must be >= 0");
    if (!basis || !grids || !H || !H->omega) return fail(nullptr, SG_EINVAL, "NULL basis/grids/H/omega");
    if (prec != SG_FP64 && prec != SG_MIXED && prec != SG_DF64) return fail(nullptr, SG_EINVAL, "unknown precision");
    for (int i = 0; i < D; i++) {
        const sg_basis &b = basis[i];
        const sg_grid &g = grids[i];
        if (b.nb_A < 1 || b.nb_B < 0 || g.nq_A < b.nb_A || g.nq_B < b.nb_B)
            return fail(nullptr, SG_EINVAL, "mode rules need nb_A>=1, nb_B>=0, nq_A>=nb_A, nq_B>=nb_B");
        if (!(b.scale > 0) || !std::isfinite(b.scale) || !std::isfinite(b.q0))
            return fail(nullptr, SG_EINVAL, "scale must be finite and > 0, q0 finite");
        if ((int64_t)g.nq_A + (int64_t)g.nq_B * L > kMaxLevelSize)
            return fail(nullptr, SG_EUNSUPPORTED, "nq(L) > 32");
        if (!std::isfinite(H->omega[i])) return fail(nullptr, SG_EINVAL, "omega not finite");
    }
    const sg_poly &V = H->V;
    if (V.nterms < 0) return fail(nullptr, SG_EINVAL, "V.nterms < 0");
    if (V.nterms > kMaxMono) return fail(nullptr, SG_EUNSUPPORTED, "more than 256 monomials");
    if (V.nterms > 0 && (!V.coef || !V.nfac)) return fail(nullptr, SG_EINVAL, "NULL V arrays");

    sg_ctx *ctx = new (std::nothrow) sg_ctx();
    if (!ctx) return fail(nullptr, SG_ENOMEM, "host allocation failed");
    Problem &p = ctx->prob;
    p.D = D; p.L = L; p.prec = prec;
    p.basis.assign(basis, basis + D);
    p.grids.assign(grids, grids + D);
    p.omega.assign(H->omega, H->omega + D);
    p.mfoff.push_back(0);
    for (int m = 0; m < V.nterms; m++) {
        if (V.nfac[m] < 0 || V.nfac[m] > kMaxFac) { delete ctx; return fail(nullptr, SG_EUNSUPPORTED, "monomial with more than 8 factors"); }
        if (!std::isfinite(V.coef[m])) { delete ctx; return fail(nullptr, SG_EINVAL, "V coefficient not finite"); }
        if (V.nfac[m] > 0 && (!V.mode || !V.power)) { delete ctx; return fail(nullptr, SG_EINVAL, "NULL V factor arrays"); }
        p.mcoef.push_back(V.coef[m]);
        p.mnfac.push_back(V.nfac[m]);
        int tot[kMaxD] = {0};
        for (int f = p.mfoff[m]; f < p.mfoff[m] + V.nfac[m]; f++) {
            if (V.mode[f] < 0 || V.mode[f] >= D) { delete ctx; return fail(nullptr, SG_EINVAL, "factor mode out of range"); }
            if (V.power[f] < 1 || V.power[f] > kMaxPow) { delete ctx; return fail(nullptr, SG_EUNSUPPORTED, "factor power outside 1..16"); }
            tot[V.mode[f]] += V.power[f];
            if (tot[V.mode[f]] > kMaxPow) { delete ctx; return fail(nullptr, SG_EUNSUPPORTED, "total power of a mode > 16"); }
            p.mfmode.push_back(V.mode[f]);
            p.mfpow.push_back(V.power[f]);
        }
        p.mfoff.push_back(p.mfoff[m] + V.nfac[m]);
    }
    ctx->fp32 = (prec == SG_MIXED);
    const int budget = std::min(smem_optin - 4096, ctx->fp32 ? 72 * 1024 : 110 * 1024);
    std::string err = build_tables(p, budget, ctx->fp32 ? 4 : 8, &ctx->host);
    if (!err.empty()) { delete ctx; return fail(nullptr, SG_EUNSUPPORTED, err); }
    HostTables &T = ctx->host;
    KParams &kp = ctx->kp;
    kp.D = D; kp.L = L; kp.Dpad = T.Dpad;
    kp.nmono = (int)p.mcoef.size(); kp.pmax = T.pmax; kp.kw = T.kw;
    kp.n_cs = (int)T.n_cs; kp.n_terms = T.n_terms;
    kp.part = 0; kp.nparts = 1;
    kp.cap = T.cap; kp.maxnb = T.maxnb; kp.matcap = T.matcap; kp.vtabcap = T.vtabcap;
    *out = ctx;
    return SG_OK;
}

}  // namespace

namespace sg {

// Entry-major copies of x of at most this many values are not made: the row
// kernel gathers from x itself, which stays in the caches, and a launch is saved
// (mixed, 24,024 values 9.1 us without the copy and 11.4 with it; 64,350 12.4
// and 11.7; 97,240 14.3 and 11.1).
constexpr int64_t kDirectElems = 65536;
// The last block settles the vectors up to this many windows, a launch beyond
// (403 windows 9.4 us by the block and 11.8 by a launch, 684 11.1 and 13.8,
// about 2,000 22.5 and 20.0, 10,104 86.3 and 81.5: the blocks meet at the counter).
constexpr int kTicketBlocks = 1024;

cudaError_t apply_rows(sg_ctx *ctx, RowIO io, cudaStream_t s)
{
    if (ctx->rop.nwin <= 0) return cudaErrorInvalidValue;  // nothing would write y
    const sg_precision prec = ctx->prob.prec;
    cudaError_t e = cudaSuccess;
    const int vt = row_vt(ctx->host, prec);
    if (!io.xs || ctx->host.n_cs * (int64_t)io.nvec <= kDirectElems || rows_direct(prec, vt, io.nvec)) io.xs = nullptr;
    else e = launch_row_stage(ctx->rop, io, prec, s);
    if (!io.y || ctx->rop.nwin > kTicketBlocks) io.ticket = nullptr;
    if (e == cudaSuccess) e = launch_rows(ctx->rop, io, prec, vt, s);
    if (e == cudaSuccess && io.y && !io.ticket) e = launch_row_settle(io, ctx->rop.n, s);
    return e;
}

void free_rows(sg_ctx *ctx)
{
    for (void *p : ctx->row_allocs) cudaFree(p);
    ctx->row_allocs.clear();
    ctx->bytes_device -= ctx->row_bytes;
    ctx->row_bytes = 0;
    ctx->rop = RowOp{};
}

// The earlier operator is released once the new one is complete: a failure leaves it in force.
cudaError_t build_rows(sg_ctx *ctx)
{
    const HostTables &T = ctx->host;
    const KParams &kp = ctx->kp;
    const sg_precision prec = ctx->prob.prec;
    const size_t n = (size_t)T.n_cs;
    // set-up tables (released below) and the row lengths
    Arena A;
    const size_t o[9] = {A.add(T.sh_off), A.add(T.sh_mode), A.add(T.sh_d), A.add(T.sh_src_off), A.add(T.sh_src),
                         A.add(T.pr_off), A.add(T.pr_mode), A.add(T.pr_op), A.add(T.pr_coef)};
    unsigned char *set = nullptr, *plan = nullptr, *own = nullptr;
    size_t at = 0;
    cudaError_t e = A.put(&set, n * sizeof(int), &at);
    RowShifts S{};
    S.nshift = (int)T.sh_off.size() - 1;
    auto ints = [&](int q) { return reinterpret_cast<const int *>(set + o[q]); };
    if (e == cudaSuccess) {
        S.off = ints(0); S.mode = ints(1); S.d = ints(2); S.src_off = ints(3); S.src = ints(4);
        S.prod_off = ints(5); S.fmode = ints(6); S.fop = ints(7);
        S.coef = reinterpret_cast<const double *>(set + o[8]);
        e = launch_row_count(kp, S, reinterpret_cast<int *>(set + at), 0);
    }
    std::vector<int> hc(n);
    if (e == cudaSuccess) e = cudaMemcpy(hc.data(), set + at, n * sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) {
        const RowWindows W = cut_rows(hc, row_window_rows((int64_t)n, row_window_units(T)), row_budget(T, prec),
                                      row_value_bytes(prec));
        Arena B, C;  // for the fill kernel; kept: the windows and their records
        const size_t meta = B.add(W.meta), win = B.add(W.win), start = B.add(W.start);
        size_t rec = 0;
        C.add(W.wins);
        e = B.put(&plan);
        if (e == cudaSuccess) e = C.put(&own, (size_t)W.bytes, &rec);
        RowOp R{};
        if (e == cudaSuccess) {
            R.wins = reinterpret_cast<const RowWin *>(own);
            R.blob = own + rec;
            int most = 0;
            for (const RowWin &w : W.wins) most = std::max(most, w.nent);
            e = launch_row_fill(kp, S, prec, R.wins, (int)W.wins.size(), most, reinterpret_cast<const int *>(plan + win),
                                reinterpret_cast<const int *>(plan + start), reinterpret_cast<const uint2 *>(plan + meta),
                                own + rec, 0);
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(0);
        R.esplit = kp.esplit;
        R.err = kp.err;
        R.nwin = (int)W.wins.size();
        R.n = (int)n;
        R.cap = W.cap;
        R.wrows = W.wrows;
        if (e == cudaSuccess) {
            ctx->plan_version++;  // before anything that a batch may still point to is released
            free_rows(ctx);
            ctx->row_allocs.push_back(own);
            ctx->rop = R;
            ctx->win_entries.resize(W.wins.size());
            ctx->win_rows.resize(W.wins.size());
            for (size_t w = 0; w < W.wins.size(); w++) {
                ctx->win_entries[w] = W.wins[w].nent;
                ctx->win_rows[w] = W.wins[w].nrows;
            }
            ctx->row_bytes = (int64_t)(rec + W.bytes);
            ctx->bytes_device += ctx->row_bytes;
        }
    }
    if (set) cudaFree(set);
    if (plan) cudaFree(plan);
    if (e != cudaSuccess) {
        if (own) cudaFree(own);
        (void)cudaGetLastError();  // reported here; not by a later launch
    }
    return e;
}

int64_t planned_device_bytes(const sg_ctx *ctx)
{
    const HostTables &T = ctx->host;
    const Problem &p = ctx->prob;
    auto b = [](const auto &v) { return std::max<int64_t>(1, (int64_t)v.size()) * (int64_t)sizeof(v[0]); };
    const int64_t terms = b(T.levels) + b(T.coefs) + b(T.order) + b(T.rank_tab) + b(T.lmin_tab) + b(T.lvl) +
                          b(T.tabd) * 3 / 2 + b(p.mcoef) + b(p.mnfac) + b(p.mfoff) + b(p.mfmode) + b(p.mfpow) +
                          b(T.harm_mono) + b(T.esplit) + (int64_t)sizeof(int);
    if (!T.rows) return terms;
    // every table in the arenas of upload_row_tables and build_rows starts at a multiple of 256 bytes
    const int64_t rows = b(T.rank_tab) + b(T.lmin_tab) + b(T.lvl) + b(T.tabd) + b(T.esplit) + (int64_t)sizeof(int) +
                         7 * 256 + row_form_bytes(T, p.prec);
    return std::max(terms, rows);
}

}  // namespace sg

extern "C" {

sg_status sg_plan(int D, int L, const sg_basis *basis, const sg_grid *grids,
                  const sg_hamiltonian *H, sg_precision prec, sg_ctx **out)
{
    return plan(D, L, basis, grids, H, prec, kPlanSmemOptin, out);
}

sg_status sg_create(int D, int L, const sg_basis *basis, const sg_grid *grids,
                    const sg_hamiltonian *H, sg_precision prec, sg_ctx **out)
{
    using namespace sg;
    if (!out) return fail(nullptr, SG_EINVAL, "out is NULL");
    *out = nullptr;
    int device = 0, smem_optin = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaGetDevice");
    e = cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaDeviceGetAttribute");
    sg_ctx *ctx = nullptr;
    sg_status st0 = plan(D, L, basis, grids, H, prec, smem_optin, &ctx);
    if (st0 != SG_OK) return st0;
    ctx->device = device;
    auto give_up = [&](sg_status st) {
        free_all(ctx);
        delete ctx;
        return st;
    };
    ctx->has_device = true;
    HostTables &T = ctx->host;
    if (prec == SG_DF64 && (!T.rows || !T.pairs))
        return give_up(fail(nullptr, SG_EUNSUPPORTED,
                            "SG_DF64 needs the row form of a potential with monomials of one and two modes (at most 64 pairs)"));
    if (T.rows) {
        e = upload_row_tables(ctx);
        if (e == cudaSuccess) e = build_rows(ctx);
        if (e == cudaSuccess) e = configure_rows();
        if (e == cudaErrorMemoryAllocation && prec == SG_DF64)
            return give_up(fail(nullptr, SG_ENOMEM, std::string("cudaMalloc (row operator): ") + cudaGetErrorString(e)));
        if (e == cudaErrorMemoryAllocation) {
            // no room for the rows: term by term, whose tables are a small part of them
            T.rows = false;
            free_tables(ctx);
        } else if (e != cudaSuccess) {
            return give_up(cuda_fail(nullptr, e, "context set-up"));
        }
    }
    if (!T.rows) {
        const sg_status st = upload_term_tables(ctx);
        if (st != SG_OK) {
            g_create_error = ctx->last_error;
            return give_up(st);
        }
        ctx->smem_bytes = apply_smem_bytes(ctx->kp, ctx->fp32);
        e = configure_kernels(ctx->smem_bytes, ctx->fp32);
        if (e != cudaSuccess) return give_up(cuda_fail(nullptr, e, "context set-up"));
    }
    *out = ctx;
    return SG_OK;
}

sg_status sg_size(const sg_ctx *ctx, int64_t *n_cs, int64_t *n_terms, int64_t *n_s,
                  int64_t *n_grid, int64_t *bytes_device)
{
    if (!ctx) return SG_EINVAL;
    if (n_cs) *n_cs = ctx->host.n_cs;
    if (n_terms) *n_terms = ctx->host.n_terms;
    if (n_s) *n_s = ctx->host.n_s;
    if (n_grid) *n_grid = ctx->host.n_grid;
    // a context made by sg_plan holds nothing on the device: report what
    // sg_create would allocate for the same problem
    if (bytes_device) *bytes_device = ctx->has_device ? ctx->bytes_device : sg::planned_device_bytes(ctx);
    return SG_OK;
}

sg_status sg_apply_H(sg_ctx *ctx, const double *x, double *y, int nvec, void *stream)
{
    if (!ctx) return SG_EINVAL;
    if (!ctx->has_device) return fail(ctx, SG_EINVAL, "context was made by sg_plan (no device state)");
    if (!sg_on_ctx_device(ctx)) return fail(ctx, SG_EINVAL, "the current CUDA device is not the one the context was made on");
    if (!x || !y) return fail(ctx, SG_EINVAL, "x or y is NULL");
    if (nvec < 1) return fail(ctx, SG_EINVAL, "nvec must be >= 1");
    const size_t n = (size_t)ctx->host.n_cs * nvec;
    if ((x < y + n) && (y < x + n)) return fail(ctx, SG_EINVAL, "x and y overlap");
    sg_status st = ensure_workspace(ctx, nvec, (cudaStream_t)stream);
    if (st != SG_OK) return st;
    cudaError_t e = enqueue_apply(ctx, x, y, nvec, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "apply launch");
    return SG_OK;
}

sg_status sg_apply_H_part(sg_ctx *ctx, const double *x, int nvec, int part, int nparts, int64_t *acc, void *stream)
{
    if (!ctx) return SG_EINVAL;
    if (!ctx->has_device) return fail(ctx, SG_EINVAL, "context was made by sg_plan (no device state)");
    if (!sg_on_ctx_device(ctx)) return fail(ctx, SG_EINVAL, "the current CUDA device is not the one the context was made on");
    if (!x || !acc) return fail(ctx, SG_EINVAL, "x or acc is NULL");
    if (nvec < 1) return fail(ctx, SG_EINVAL, "nvec must be >= 1");
    if (nparts < 1 || part < 0 || part >= nparts) return fail(ctx, SG_EINVAL, "need 0 <= part < nparts");
    sg_status st = ensure_workspace(ctx, nvec, (cudaStream_t)stream);
    if (st != SG_OK) return st;
    if (ctx->host.rows) {
        sg::RowIO io = row_io(ctx, x, nullptr, nvec);
        io.acc = reinterpret_cast<unsigned long long *>(acc);
        io.part = part;
        io.nparts = nparts;
        const cudaError_t er = sg::apply_rows(ctx, io, (cudaStream_t)stream);
        if (er != cudaSuccess) return cuda_fail(ctx, er, "partial apply launch");
        return SG_OK;
    }
    sg::KParams kp = ctx->kp;
    kp.acc = reinterpret_cast<unsigned long long *>(acc);
    kp.part = part;
    kp.nparts = nparts;
    cudaError_t e = sg::launch_maxabs(kp, x, nvec, ctx->maxbits, (cudaStream_t)stream);
    if (e == cudaSuccess) e = sg::launch_apply_terms(kp, ctx->fp32, x, ctx->maxbits, nvec, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "partial apply launch");
    return SG_OK;
}

sg_status sg_apply_H_finish(sg_ctx *ctx, const double *x, int64_t *acc, double *y, int nvec, void *stream)
{
    if (!ctx) return SG_EINVAL;
    if (!ctx->has_device) return fail(ctx, SG_EINVAL, "context was made by sg_plan (no device state)");
    if (!sg_on_ctx_device(ctx)) return fail(ctx, SG_EINVAL, "the current CUDA device is not the one the context was made on");
    if (!x || !y || !acc) return fail(ctx, SG_EINVAL, "x, y or acc is NULL");
    if (nvec < 1) return fail(ctx, SG_EINVAL, "nvec must be >= 1");
    const size_t n = (size_t)ctx->host.n_cs * nvec;
    if ((x < y + n) && (y < x + n)) return fail(ctx, SG_EINVAL, "x and y overlap");
    sg_status st = ensure_workspace(ctx, nvec, (cudaStream_t)stream);
    if (st != SG_OK) return st;
    if (ctx->host.rows) {
        sg::RowIO io = row_io(ctx, x, y, nvec);
        io.acc = reinterpret_cast<unsigned long long *>(acc);
        cudaError_t er = sg::launch_row_finish(ctx->rop, io, (cudaStream_t)stream);
        if (er == cudaSuccess) er = sg::launch_row_settle(io, ctx->rop.n, (cudaStream_t)stream);
        if (er != cudaSuccess) return cuda_fail(ctx, er, "finish launch");
        return SG_OK;
    }
    sg::KParams kp = ctx->kp;
    kp.acc = reinterpret_cast<unsigned long long *>(acc);
    cudaError_t e = sg::launch_maxabs(kp, x, nvec, ctx->maxbits, (cudaStream_t)stream);
    if (e == cudaSuccess) e = sg::launch_finalize(kp, ctx->fp32, x, y, nvec, ctx->maxbits, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "finish launch");
    return SG_OK;
}

sg_status sg_part_size(const sg_ctx *ctx, int part, int nparts, int64_t *n_items, int64_t *cost)
{
    if (!ctx || nparts < 1 || part < 0 || part >= nparts) return SG_EINVAL;
    const sg::HostTables &T = ctx->host;
    int64_t c = 0, k = 0;
    if (T.rows && ctx->has_device) {
        for (size_t w = part; w < ctx->win_entries.size(); w += nparts) {
            c += ctx->win_entries[w];
            k += ctx->win_rows[w];
        }
    } else if (T.rows) {  // not cut yet: whole windows, their rows of the mean length
        const int64_t rows = sg::row_window_rows(T.n_cs, sg::row_window_units(T));
        for (int64_t r = part * rows; r < T.n_cs; r += nparts * rows) k += std::min(rows, T.n_cs - r);
        c = (int64_t)((double)T.row_nnz * k / T.n_cs);
    } else {
        for (int64_t p = part; p < T.n_terms; p += nparts) {
            c += T.pcost[(size_t)p];
            k++;
        }
    }
    if (n_items) *n_items = k;
    if (cost) *cost = c;
    return SG_OK;
}

sg_status sg_apply_H_host(sg_ctx *ctx, const double *x_host, double *y_host, int nvec, void *stream)
{
    if (!ctx) return SG_EINVAL;
    if (!ctx->has_device) return fail(ctx, SG_EINVAL, "context was made by sg_plan (no device state)");
    if (!sg_on_ctx_device(ctx)) return fail(ctx, SG_EINVAL, "the current CUDA device is not the one the context was made on");
    if (!x_host || !y_host) return fail(ctx, SG_EINVAL, "x_host or y_host is NULL");
    if (nvec < 1) return fail(ctx, SG_EINVAL, "nvec must be >= 1");
    const int64_t n = ctx->host.n_cs * (int64_t)nvec;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e;
    if (n > ctx->stage_elems) {
        if (ctx->stage_x) cudaFree(ctx->stage_x);
        if (ctx->stage_y) cudaFree(ctx->stage_y);
        ctx->stage_x = ctx->stage_y = nullptr;
        ctx->stage_elems = 0;
        if ((e = cudaMalloc(&ctx->stage_x, n * sizeof(double))) != cudaSuccess ||
            (e = cudaMalloc(&ctx->stage_y, n * sizeof(double))) != cudaSuccess)
            return fail(ctx, SG_ENOMEM, std::string("staging cudaMalloc: ") + cudaGetErrorString(e));
        ctx->stage_elems = n;
    }
    if ((e = cudaMemcpyAsync(ctx->stage_x, x_host, n * sizeof(double), cudaMemcpyHostToDevice, s)) != cudaSuccess)
        return cuda_fail(ctx, e, "H2D copy");
    sg_status st = ensure_workspace(ctx, nvec, s);
    if (st != SG_OK) return st;
    if ((e = enqueue_apply(ctx, ctx->stage_x, ctx->stage_y, nvec, s)) != cudaSuccess)
        return cuda_fail(ctx, e, "apply launch");
    if ((e = cudaMemcpyAsync(y_host, ctx->stage_y, n * sizeof(double), cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        return cuda_fail(ctx, e, "D2H copy");
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return cuda_fail(ctx, e, "stream synchronize");
    return SG_OK;
}

sg_status sg_term_levels(const sg_ctx *ctx, int64_t t0, int64_t nt, int *levels_host, int *coef_host)
{
    if (!ctx) return SG_EINVAL;
    const sg::HostTables &T = ctx->host;
    if (t0 < 0 || nt < 0 || t0 + nt > T.n_terms || (nt > 0 && !levels_host)) return SG_EINVAL;
    const int D = ctx->prob.D;
    for (int64_t t = 0; t < nt; t++) {
        for (int i = 0; i < D; i++) levels_host[t * D + i] = T.levels[(size_t)(t0 + t) * T.Dpad + i];
        if (coef_host) coef_host[t] = T.coefs[t0 + t];
    }
    return SG_OK;
}

sg_status sg_index_map(sg_ctx *ctx, int64_t t0, int64_t nt, int64_t *offsets_host,
                       int64_t *cs_index_dev, void *stream)
{
    if (!ctx) return SG_EINVAL;
    const sg::HostTables &T = ctx->host;
    if (t0 < 0 || nt < 0 || t0 + nt > T.n_terms || !offsets_host)
        return fail(ctx, SG_EINVAL, "bad term range or NULL offsets");
    const int D = ctx->prob.D, L = ctx->prob.L;
    offsets_host[0] = 0;
    for (int64_t t = 0; t < nt; t++) {
        int64_t nb = 1;
        for (int i = 0; i < D; i++) nb *= T.lvl[(size_t)i * (L + 1) + T.levels[(size_t)(t0 + t) * T.Dpad + i]].nb;
        offsets_host[t + 1] = offsets_host[t] + nb;
    }
    if (!cs_index_dev || nt == 0) return SG_OK;
    if (!ctx->has_device) return fail(ctx, SG_EINVAL, "context was made by sg_plan (no device state)");
    if (!sg_on_ctx_device(ctx)) return fail(ctx, SG_EINVAL, "the current CUDA device is not the one the context was made on");
    // the offsets and the levels of the range
    cudaStream_t s = (cudaStream_t)stream;
    sg::Arena A;
    const size_t off = A.add(offsets_host, (size_t)nt + 1);
    const size_t lev = A.add(T.levels.data() + (size_t)t0 * T.Dpad, (size_t)nt * T.Dpad);
    unsigned char *base = nullptr;
    cudaError_t e = A.put(&base);
    if (!base) return fail(ctx, SG_ENOMEM, "cudaMalloc offsets");
    sg::KParams kp = ctx->kp;
    kp.levels = base + lev;
    if (e == cudaSuccess)
        e = sg::launch_index_map(kp, 0, nt, reinterpret_cast<const int64_t *>(base + off), cs_index_dev, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(base);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "index map");
    return SG_OK;
}

sg_status sg_device_error(sg_ctx *ctx, int *code)
{
    if (!ctx || !code) return SG_EINVAL;
    if (!ctx->has_device) return fail(ctx, SG_EINVAL, "context was made by sg_plan (no device state)");
    if (!sg_on_ctx_device(ctx)) return fail(ctx, SG_EINVAL, "the current CUDA device is not the one the context was made on");
    int v = 0;
    cudaError_t e = cudaMemcpy(&v, ctx->kp.err, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "read error word");
    *code = v;
    if (v) {  // reported once: clear it for the next apply
        int z = 0;
        e = cudaMemcpy(ctx->kp.err, &z, sizeof(int), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "clear error word");
    }
    return SG_OK;
}

sg_status sg_compact_rank(const sg_ctx *ctx, const int *k, int64_t n, int64_t *rank)
{
    if (!ctx || n < 0 || (n > 0 && (!k || !rank))) return SG_EINVAL;
    const sg::HostTables &T = ctx->host;
    const int D = ctx->prob.D, L = ctx->prob.L;
    for (int64_t q = 0; q < n; q++) {
        const int *kq = k + q * D;
        int64_t r = 0;
        int s = 0;
        bool ok = true;
        for (int i = 0; i < D && ok; i++) {
            if (kq[i] < 0 || kq[i] >= T.kw) { ok = false; break; }
            const int lm = T.lmin_tab[(size_t)i * T.kw + kq[i]];
            if (lm > L || s + lm > L) { ok = false; break; }
            r += T.rank_tab[((size_t)i * (L + 1) + s) * T.kw + kq[i]];
            s += lm;
        }
        rank[q] = ok ? r : -1;
    }
    return SG_OK;
}

sg_status sg_mode_tables(const sg_ctx *ctx, int mode, int level, int *nb, int *nq,
                         double *B, double *BW, double *K, double *Q)
{
    if (!ctx || mode < 0 || mode >= ctx->prob.D || level < 0 || level > ctx->prob.L) return SG_EINVAL;
    const sg::HostTables &T = ctx->host;
    const sg::LevelInfo &li = T.lvl[(size_t)mode * (ctx->prob.L + 1) + level];
    if (nb) *nb = li.nb;
    if (nq) *nq = li.nq;
    const double *t = T.tabd.data();
    if (B) std::copy(t + li.offB, t + li.offB + li.nb * li.nq, B);
    if (BW) std::copy(t + li.offBW, t + li.offBW + li.nb * li.nq, BW);
    if (K) std::copy(t + li.offK, t + li.offK + li.nb * li.nb, K);
    if (Q) std::copy(t + li.offQ, t + li.offQ + li.nq, Q);
    return SG_OK;
}

const char *sg_last_error(const sg_ctx *ctx)
{
    return ctx ? ctx->last_error.c_str() : g_create_error.c_str();
}

void sg_destroy(sg_ctx *ctx)
{
    if (!ctx) return;
    free_all(ctx);
    delete ctx;
}

}  // extern "C"
