// A stand-in for the CUDA runtime and the kernels' launchers, in host memory,
// for tests of the library's host code: allocations are counted and can be made
// to fail, freed memory is overwritten and kept (so that a stale pointer reads
// garbage instead of faulting), and the row form does a simple product: row r
// holds its count times the entry (r, 1), so y = (count + esplit) x whatever the
// windows are.
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "sg_internal.h"

namespace {

struct State {
    std::map<void *, size_t> live;
    size_t bytes = 0, peak = 0, largest = 0;
    long allowed = -1;      // allocations of at least min_bytes that still succeed (-1: all)
    size_t min_bytes = 0;
    long matching = 0;      // allocations of at least min_bytes asked for
    std::map<std::string, long> launches;
    int event = 0;
    long entries = 0;       // of the windows that launch_rows has been given
} g;
std::mutex lock;  // eigen requests of a server run on threads of their own

cudaError_t allocate(void **p, size_t n)
{
    std::lock_guard<std::mutex> lk(lock);
    *p = nullptr;
    if (n >= g.min_bytes) {
        g.matching++;
        if (g.allowed == 0) return cudaErrorMemoryAllocation;
        if (g.allowed > 0) g.allowed--;
    }
    *p = std::calloc(1, n ? n : 1);
    if (!*p) return cudaErrorMemoryAllocation;
    g.live[*p] = n;
    g.bytes += n;
    if (g.bytes > g.peak) g.peak = g.bytes;
    if (n > g.largest) g.largest = n;
    return cudaSuccess;
}

cudaError_t launched(const char *name)
{
    std::lock_guard<std::mutex> lk(lock);
    g.launches[name]++;
    return cudaSuccess;
}

}  // namespace

extern "C" {

void fake_reset() { g = State(); }
void fake_fail_after(long n, size_t min_bytes)
{
    g.allowed = n;
    g.min_bytes = min_bytes;
    g.matching = 0;
}
long fake_matching() { return g.matching; }
size_t fake_live() { return g.bytes; }
size_t fake_peak() { return g.peak; }
void fake_clear_peak() { g.peak = g.bytes; g.largest = 0; }
size_t fake_largest() { return g.largest; }
long fake_entries() { return g.entries; }
long fake_launches(const char *name) { return g.launches.count(name) ? g.launches[name] : 0; }

// ---------------------------------------------------------------- runtime
cudaError_t cudaMalloc(void **p, size_t n) { return allocate(p, n); }
cudaError_t cudaFree(void *p)
{
    std::lock_guard<std::mutex> lk(lock);
    auto f = g.live.find(p);
    if (f == g.live.end()) return p ? cudaErrorInvalidValue : cudaSuccess;
    std::memset(p, 0xFF, f->second);  // kept: see above
    g.bytes -= f->second;
    g.live.erase(f);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 232448; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "an error"; }
// every timing is longer than the one before it
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = (float)++g.event; return cudaSuccess; }
// no capture: calls with a stream of their own are outside these tests
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

}  // extern "C"

namespace sg {

// ---------------------------------------------------------------- row form
// Entries per row as the operator has them: shifts that stay inside the basis.
cudaError_t launch_row_count(const KParams &P, const RowShifts &S, int *cnt, cudaStream_t)
{
    std::vector<int> k(P.D);
    for (int r = 0; r < P.n_cs; r++) {
        int s = 0, left = r;
        for (int i = 0; i < P.D; i++) {
            const int *t = P.rank_tab + (size_t)(i * (P.L + 1) + s) * P.kw;
            int v = 0;
            while (v + 1 < P.kw && t[v + 1] <= left) v++;
            k[i] = v;
            left -= t[v];
            s += P.lmin_tab[i * P.kw + v];
        }
        cnt[r] = 0;
        for (int q = 0; q < S.nshift; q++) {
            int u = s;
            for (int e = S.off[q]; e < S.off[q + 1] && u <= P.L; e++) {
                const int i = S.mode[e], k2 = k[i] + S.d[e];
                if (k2 < 0 || k2 >= P.kw || P.lmin_tab[i * P.kw + k2] > P.L) u = P.L + 1;
                else if (S.d[e] > 0) u += P.lmin_tab[i * P.kw + k2] - P.lmin_tab[i * P.kw + k[i]];
            }
            cnt[r] += u <= P.L;
        }
    }
    return launched("row_count");
}
cudaError_t launch_row_fill(const KParams &P, const RowShifts &, sg_precision, const RowWin *wins, int, int, const int *win,
                            const int *start, const uint2 *meta, unsigned char *blob, cudaStream_t)
{
    for (int r = 0; r < P.n_cs; r++) {
        const RowWin w = wins[win[r]];
        reinterpret_cast<uint2 *>(blob + w.off)[r - w.row0] = meta[r];
        int *cols = reinterpret_cast<int *>(blob + w.off + row_meta_bytes(w.nrows));
        const int next = r + 1 < w.row0 + w.nrows ? start[r + 1] : w.nent;
        for (int e = start[r]; e < next; e++) cols[e] = r;
    }
    return launched("row_fill");
}
cudaError_t configure_rows() { return cudaSuccess; }
// y, or a 1 into the accumulator of every row of the part
static void product(const RowOp &R, const RowIO &io)
{
    for (int w = io.part; w < R.nwin; w += io.nparts) {
        const RowWin W = R.wins[w];
        g.entries += W.nent;
        if (!io.y) {
            for (int r = W.row0; r < W.row0 + W.nrows; r++)
                for (int v = 0; v < io.nvec; v++) io.acc[((size_t)r * io.nvec + v) * io.words]++;
            continue;
        }
        const uint2 *meta = reinterpret_cast<const uint2 *>(R.blob + W.off);
        const int *cols = reinterpret_cast<const int *>(R.blob + W.off + row_meta_bytes(W.nrows));
        for (int q = 0; q < W.nrows; q++) {
            const int r = W.row0 + (int)(meta[q].x >> 24);
            for (int v = 0; v < io.nvec; v++) {
                double s = 0.0;
                for (unsigned e = 0; e < meta[q].y; e++) s += io.x[(size_t)v * R.n + cols[(meta[q].x & 0xFFFFFFu) + e]];
                io.y[(size_t)v * R.n + r] = s + R.esplit[r] * io.x[(size_t)v * R.n + r];
            }
        }
    }
}
cudaError_t launch_rows(const RowOp &R, const RowIO &io, sg_precision, int, cudaStream_t)
{
    product(R, io);
    return launched("rows");
}
cudaError_t launch_rows_batch(const RowOp *, const int2 *, int, int, int, const RowIO &, sg_precision, int,
                              const long long *, cudaStream_t)
{
    return launched("rows_batch");
}
cudaError_t launch_row_stage(const RowOp &, const RowIO &, sg_precision, cudaStream_t) { return launched("stage"); }
cudaError_t launch_row_stage_batch(const RowIO &, sg_precision, const long long *, const int2 *, int, cudaStream_t)
{
    return launched("stage_batch");
}
cudaError_t launch_row_settle(const RowIO &, int, cudaStream_t) { return launched("settle"); }
cudaError_t launch_row_settle_batch(const RowIO &, const long long *, int, cudaStream_t) { return launched("settle_batch"); }
cudaError_t launch_row_finish(const RowOp &, const RowIO &, cudaStream_t) { return launched("finish"); }
cudaError_t launch_cheb_rows(const RowOp &, const ChebIO &, const ChebTerm &, sg_precision, cudaStream_t)
{
    return launched("cheb_rows");
}
cudaError_t launch_cheb_rows_batch(const RowOp *, const int2 *, int, int, const ChebIO &, const ChebState *, sg_precision,
                                   const long long *, cudaStream_t)
{
    return launched("cheb_rows_batch");
}
cudaError_t launch_cheb_iteration(ChebState *, const long long *, int, int64_t, const double *, const double *, double *,
                                  double *, cudaStream_t)
{
    return launched("cheb_iteration");
}
cudaError_t launch_cheb_log_advance(ChebState *, const long long *, int, const double *, const double *, cudaStream_t)
{
    return launched("cheb_log_advance");
}

// ---------------------------------------------------------------- term-by-term form
size_t apply_smem_bytes(const KParams &, bool) { return 1024; }
cudaError_t configure_kernels(size_t, bool) { return cudaSuccess; }
static cudaError_t terms(const KParams &P)
{
    // every table that the kernels read is there
    const void *need[] = {P.levels, P.coefs, P.order, P.rank_tab, P.lmin_tab, P.lvl, P.tabd, P.tabf, P.mcoef, P.mnfac,
                          P.mfoff, P.mfmode, P.mfpow, P.harm_mono, P.esplit, P.acc, P.err};
    for (const void *p : need)
        if (!g.live.count(const_cast<void *>(p))) return cudaErrorInvalidValue;
    return launched("terms");
}
cudaError_t launch_apply(const KParams &P, bool, const double *, double *, int, long long *, cudaStream_t) { return terms(P); }
cudaError_t launch_maxabs(const KParams &, const double *, int, long long *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_apply_terms(const KParams &P, bool, const double *, const long long *, int, cudaStream_t) { return terms(P); }
cudaError_t launch_finalize(const KParams &, bool, const double *, double *, int, const long long *, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_index_map(const KParams &, int64_t, int64_t, const int64_t *, int64_t *, cudaStream_t) { return cudaSuccess; }

// ---------------------------------------------------------------- solvers (no arithmetic: rank 0 everywhere)
cudaError_t dev_gram(const double *, int, const double *, int, int64_t, double *, double *, cudaStream_t) { return launched("gram"); }
size_t gram_partial_doubles(int64_t n, int ka)
{
    return (size_t)std::min<int64_t>(64, (n + 16383) / 16384) * ka * 8;
}
cudaError_t dev_combine(const double *, int, const double *, int, double, const double *, double *, int64_t, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t dev_chol_inverse(const double *, int, double *, int *, cudaStream_t) { return cudaSuccess; }
cudaError_t dev_residual(const double *, const double *, double *, int rows, int64_t, double *, double *, cudaStream_t)
{
    return rows < 1 ? cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t dev_direction(const double *, const double *, const double *, int, int64_t, double *, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t dev_unit_vectors(double *, int64_t, const double *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t dev_normalise(double *, int64_t, double *, double *, cudaStream_t) { return cudaSuccess; }
cudaError_t dev_project_normalise(const double *, int, const double *, double *, int64_t, double *, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t dev_axpby(int64_t, double, const double *, double, double *, cudaStream_t) { return cudaSuccess; }
void sym_eig(int n, std::vector<double>, std::vector<double> &w, std::vector<double> &Z)
{
    w.resize(n);
    for (int i = 0; i < n; i++) w[i] = i;
    Z.assign((size_t)n * n, 0.0);
}
int chol_inverse(int, std::vector<double> &) { return 0; }
std::vector<double> bessel_j(int kmax, double) { return std::vector<double>(kmax + 1, 1.0); }

}  // namespace sg
