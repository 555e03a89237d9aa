// C ABI of the solvers: sg_eigs, sg_eigs_refine, sg_propagate, sg_product_state.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "sg_internal.h"

namespace sg {
cudaError_t dev_gram(const double *A, int ka, const double *B, int kb, int64_t n, double *C_dev, double *partial,
                     cudaStream_t s);
size_t gram_partial_doubles(int64_t n, int ka);
cudaError_t dev_combine(const double *V, int k, const double *S_dev, int r, double alpha, const double *base,
                        double *out, int64_t n, cudaStream_t s);
cudaError_t dev_chol_inverse(const double *G, int b, double *Ri, int *rank, cudaStream_t s);
cudaError_t dev_residual(const double *X, const double *theta, double *HX, int rows, int64_t n, double *norms2,
                         double *partial, cudaStream_t s);
cudaError_t dev_direction(const double *R, const double *d, const double *sel, int rows, int64_t n, double *T,
                          cudaStream_t s);
cudaError_t dev_unit_vectors(double *X, int64_t n, const double *at, int r, cudaStream_t s);
cudaError_t dev_normalise(double *x, int64_t n, double *nn, double *partial, cudaStream_t s);
cudaError_t dev_project_normalise(const double *V, int k, const double *c, double *x, int64_t n, double *nn,
                                  cudaStream_t s);
cudaError_t dev_axpby(int64_t len, double a, const double *x, double b, double *y, cudaStream_t s);
void sym_eig(int n, std::vector<double> A, std::vector<double> &w, std::vector<double> &Z);
int chol_inverse(int b, std::vector<double> &G);
std::vector<double> bessel_j(int kmax, double x);
}  // namespace sg

namespace {

using namespace sg;

constexpr int kBlk = 8;  // largest block size of the eigensolvers

struct SolverError {
    sg_status st;
    std::string msg;
};

void ck(cudaError_t e, const char *where)
{
    if (e != cudaSuccess) throw SolverError{SG_ECUDA, std::string(where) + ": " + cudaGetErrorString(e)};
}

void ckst(sg_status st, sg_ctx *ctx)
{
    if (st != SG_OK) throw SolverError{st, sg_last_error(ctx)};
}

// device buffer owned by a solver call
struct DBuf {
    double *p = nullptr;
    explicit DBuf(size_t n) { ck(cudaMalloc(&p, std::max<size_t>(1, n) * sizeof(double)), "solver cudaMalloc"); }
    ~DBuf() { if (p) cudaFree(p); }
    DBuf(const DBuf &) = delete;
    DBuf &operator=(const DBuf &) = delete;
};

uint64_t splitmix(uint64_t &s)
{
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Solver context: the apply, scratch, and small dense helpers.  Small matrices
// go to the device, and results come back, through the context's pinned host
// memory: the kernels write inner products there, and one stream
// synchronisation makes several of them readable.
struct Solver {
    sg_ctx *ctx;
    cudaStream_t s;
    int64_t n;
    DBuf mem;  // Gram scratch, then the small device matrices
    struct { double *p; } partial, small;
    double *pin = nullptr;
    size_t cap, used = 0;  // doubles of pin and small; handed out since the last synchronisation
    std::vector<double> pageable;
    const ApplyFn *apply_fn = nullptr;  // when set, applications of H_S go through it
    // kmax: largest basis; cols: largest number of columns combined at once.
    // pinned: results may be written to pin (a solver with many round trips);
    // without, pin only stages uploads.
    Solver(sg_ctx *c, cudaStream_t st, int kmax, int cols, bool pinned = true)
        : ctx(c), s(st), n(c->host.n_cs), mem(scratch(c->host.n_cs, kmax, cols) + capacity(kmax, cols)),
          cap(capacity(kmax, cols))
    {
        partial.p = mem.p;
        small.p = mem.p + scratch(n, kmax, cols);
        if (!pinned) {
            pageable.resize(cap);
            pin = pageable.data();
            return;
        }
        if (ctx->pin_doubles < cap) {
            if (ctx->pin) cudaFreeHost(ctx->pin);
            ctx->pin = nullptr;
            ctx->pin_doubles = 0;
            ck(cudaMallocHost(&ctx->pin, cap * sizeof(double)), "solver cudaMallocHost");
            ctx->pin_doubles = cap;
        }
        pin = ctx->pin;
    }
    static size_t scratch(int64_t n, int kmax, int cols)
    {
        return gram_partial_doubles(n, std::max({kmax, cols, 2 * kBlk}));
    }
    static size_t capacity(int kmax, int cols) { return (size_t)(kmax + 16) * (2 * cols + 6 * kBlk) + 1024; }

    // a range of pin and of small, free until the next synchronisation
    size_t take(size_t k)
    {
        if (used + k > cap) throw SolverError{SG_ECUDA, "solver scratch too small"};
        used += k;
        return used - k;
    }
    void sync(const char *where)
    {
        ck(cudaStreamSynchronize(s), where);
        used = 0;
    }

    void apply(const double *x, double *y, int r)
    {
        if (!apply_fn) { ckst(sg_apply_H(ctx, x, y, r, s), ctx); return; }
        // the routed apply reads x and writes y outside this stream: order both
        ck(cudaStreamSynchronize(s), "apply sync");
        const sg_status st = (*apply_fn)(x, y, r);
        if (st != SG_OK) throw SolverError{st, "routed apply failed"};
    }
    // Small matrix with its columns in groups of at most kBlk (each k x group, row-major).
    struct Mat {
        const double *d;
        int k, r;
    };
    Mat upload(const std::vector<double> &S, int k, int r)  // S: k x r row-major
    {
        const size_t o = take((size_t)k * r);
        double *q = pin + o;
        for (int j0 = 0; j0 < r; j0 += kBlk) {
            const int rr = std::min(kBlk, r - j0);
            for (int i = 0; i < k; i++)
                for (int j = 0; j < rr; j++) *q++ = S[(size_t)i * r + j0 + j];
        }
        ck(cudaMemcpyAsync(small.p + o, pin + o, sizeof(double) * k * r, cudaMemcpyHostToDevice, s), "small copy");
        return {small.p + o, k, r};
    }
    const double *upload(const double *v, int k)
    {
        const size_t o = take(k);
        std::copy(v, v + k, pin + o);
        ck(cudaMemcpyAsync(small.p + o, pin + o, sizeof(double) * k, cudaMemcpyHostToDevice, s), "small copy");
        return small.p + o;
    }
    // A^T B (A: ka vectors, B: kb) into C, columns in groups; C on the device or pinned
    void gram_to(const double *A, int ka, const double *B, int kb, double *C)
    {
        for (int j0 = 0; j0 < kb; j0 += kBlk) {
            const int r = std::min(kBlk, kb - j0);
            ck(dev_gram(A, ka, B + (size_t)j0 * n, r, n, C + (size_t)ka * j0, partial.p, s), "gram");
        }
    }
    static std::vector<double> ungroup(const double *C, int ka, int kb)
    {
        std::vector<double> out((size_t)ka * kb);
        for (int j0 = 0; j0 < kb; j0 += kBlk) {
            const int r = std::min(kBlk, kb - j0);
            const double *c = C + (size_t)ka * j0;
            for (int i = 0; i < ka; i++)
                for (int j = 0; j < r; j++) out[(size_t)i * kb + j0 + j] = c[(size_t)i * r + j];
        }
        return out;
    }
    // the same on the host (ka x kb, row-major)
    std::vector<double> gram(const double *A, int ka, const double *B, int kb)
    {
        double *C = pin + take((size_t)ka * kb);
        gram_to(A, ka, B, kb, C);
        sync("gram sync");
        return ungroup(C, ka, kb);
    }
    // out (S.r vectors) = base (or 0) + alpha * V S
    void combine(const double *V, const Mat &S, double alpha, const double *base, double *out)
    {
        for (int j0 = 0; j0 < S.r; j0 += kBlk) {
            const int rr = std::min(kBlk, S.r - j0);
            ck(dev_combine(V, S.k, S.d + (size_t)S.k * j0, rr, alpha, base ? base + (size_t)j0 * n : nullptr,
                           out + (size_t)j0 * n, n, s), "combine");
        }
    }
    // X (r vectors) <- X - V V^T X, twice (V: k orthonormal vectors)
    void orth_against(const double *V, int k, double *X, int r)
    {
        if (k <= 0) return;
        for (int pass = 0; pass < 2; pass++) {
            double *C = small.p + take((size_t)k * r);
            gram_to(V, k, X, r, C);
            combine(V, {C, k, r}, -1.0, X, X);
        }
    }
    // One pass of Cholesky QR: out = X R^{-1} (r <= kBlk vectors), the rank to *rank (pinned)
    void chol_pass(const double *X, int r, double *out, int *rank)
    {
        double *G = small.p + take((size_t)r * r), *Ri = small.p + take((size_t)r * r);
        ck(dev_gram(X, r, X, r, n, G, partial.p, s), "gram");
        ck(dev_chol_inverse(G, r, Ri, rank, s), "cholesky");
        combine(X, {Ri, r, r}, 1.0, nullptr, out);
    }
    // orthonormalise the r vectors of X (Cholesky QR twice, tmp: r vectors of
    // scratch); returns the rank kept
    int orthonormalise(double *X, int r, double *tmp)
    {
        int rank = r;
        for (int pass = 0; pass < 2; pass++) {
            std::vector<double> G = gram(X, rank, X, rank);
            const int rk = chol_inverse(rank, G), was = rank;
            rank = rk;
            if (rank == 0) break;
            // X <- X R^{-1} (first rk columns)
            std::vector<double> Gk((size_t)was * rk);
            for (int i = 0; i < was; i++)
                for (int j = 0; j < rk; j++) Gk[(size_t)i * rk + j] = G[(size_t)i * was + j];
            combine(X, upload(Gk, was, rk), 1.0, nullptr, tmp);
            ck(cudaMemcpyAsync(X, tmp, sizeof(double) * n * rk, cudaMemcpyDeviceToDevice, s), "orth copy");
        }
        return rank;
    }
    // Davidson start: unit vectors of the r lowest harmonic energies (the
    // preconditioner's diagonal; ties by index), so the subspace overlaps the
    // low-lying states from the first step; then, when `extra`, one vector with
    // random components of every function, weighted towards the low energies.
    // Symmetries of H leave sectors that no unit vector of the block lies in
    // (chained Henon-Heiles: the parity of mode 0), and the row operator keeps
    // them apart exactly: without that vector their states are never found.
    // False when no mode is split.
    bool lowest_diagonal_block(double *X, int r, bool extra)
    {
        const std::vector<double> &d = ctx->host.esplit;
        if ((int64_t)d.size() != n) return false;
        bool any = false;
        for (double v : d) any |= v != 0.0;
        if (!any) return false;
        std::vector<int64_t> idx(n);
        for (int64_t i = 0; i < n; i++) idx[i] = i;
        std::partial_sort(idx.begin(), idx.begin() + r, idx.end(),
                          [&](int64_t a, int64_t b) { return d[a] < d[b] || (d[a] == d[b] && a < b); });
        std::vector<double> at(r);  // positions, exact as doubles (N_cs < 2^31)
        for (int j = 0; j < r; j++) at[j] = (double)idx[j];
        ck(dev_unit_vectors(X, n, upload(at.data(), r), r, s), "start block");
        std::vector<double> h(extra ? n : 0);
        uint64_t st = 0x5eed4321ull;
        for (int64_t i = 0; extra && i < n; i++) {
            const double w = 1.0 + (d[i] - d[idx[0]]);
            h[i] = ((double)(splitmix(st) >> 11) * 0x1.0p-53 - 0.5) / (w * w);
        }
        if (extra)
            ck(cudaMemcpyAsync(X + (size_t)r * n, h.data(), sizeof(double) * n, cudaMemcpyHostToDevice, s), "start copy");
        ck(cudaStreamSynchronize(s), "start sync");
        return true;
    }
    void random_block(double *X, int r, uint64_t seed)
    {
        std::vector<double> h((size_t)r * n);
        uint64_t st = seed;
        for (auto &v : h) v = (double)(splitmix(st) >> 11) * 0x1.0p-53 - 0.5;
        ck(cudaMemcpyAsync(X, h.data(), sizeof(double) * h.size(), cudaMemcpyHostToDevice, s), "random copy");
        ck(cudaStreamSynchronize(s), "random sync");
    }
};

// Vectors of a run of block_eigs: basis V and images W = H V (kmax each), Ritz
// vectors X and their images and residuals HX (nx each), directions T (b),
// scratch Q (rmax, the largest block orthonormalised at once).  nx0: vectors to
// start from (0: none).
struct EigVectors {
    int kmax, guard, rmax;
    size_t nx, total;
    EigVectors(int64_t n, int nev, int b, bool davidson, int max_it, int nx0)
    {
        // basis size: Davidson restarts at max(3 nev, nev + 6 b); the Krylov (Lanczos)
        // form keeps at most 320 vectors (its projected problem is solved densely)
        kmax = (int)std::min<int64_t>(n, davidson ? std::max(3 * nev, nev + 6 * b)
                                                  : std::min<int64_t>((int64_t)max_it * b + b, 320));
        guard = davidson ? b : 0;
        nx = (size_t)std::max(nev + guard, b);
        rmax = std::min(kmax, std::max(nev + b, nx0) + 1);
        total = 2 * (size_t)kmax + 2 * nx + b + rmax;
    }
};

// Block Davidson (or, without preconditioner and without restart, a block
// Lanczos-type Krylov method with full reorthogonalisation and Rayleigh-Ritz).
// Returns the number of converged eigenpairs; evals/resid on the host, the
// Ritz vectors in evecs (device, nev x n) when not null.
// Davidson carries b Ritz pairs beyond the nev wanted ones (its start block
// and what it keeps at a restart hold them too), and expands once more along
// their residuals when the nev have converged: a state that the basis has
// missed so far, in a sector of its own or in a cluster closer than tol, then
// takes its place among the nev and the iteration goes on.
int block_eigs(Solver &S, int nev, int b, bool davidson, double tol, int max_it, const double *X0, int nx0,
               double *evals, double *evecs, double *resid)
{
    const int64_t n = S.n;
    const EigVectors size(n, nev, b, davidson, max_it, nx0);
    const int kmax = size.kmax, guard = size.guard;
    const size_t nx = size.nx;
    DBuf mem(size.total * n);
    double *const V = mem.p, *const W = V + (size_t)kmax * n, *const X = W + (size_t)kmax * n,
                 *const HX = X + nx * n, *const T = HX + nx * n, *const Q = T + (size_t)b * n;
    std::vector<double> Tm;  // projected matrix, k x k
    int k = 0;
    // initial block
    int r0 = davidson ? std::min(nev + b, kmax) : (int)std::min<int64_t>(b, n);
    if (X0 && nx0 > 0) {
        r0 = std::min(nx0, kmax);
        ck(cudaMemcpyAsync(V, X0, sizeof(double) * n * r0, cudaMemcpyDeviceToDevice, S.s), "x0 copy");
    } else if (const bool extra = r0 < kmax; davidson && S.lowest_diagonal_block(V, r0, extra)) {
        r0 += extra;
    } else {
        S.random_block(V, r0, 0x5eed1234ull);
    }
    r0 = S.orthonormalise(V, r0, Q);
    auto images = [&](int r) {  // W = H V for the new vectors V[k..k+r)
        for (int j0 = 0; j0 < r; j0 += kBlk)
            S.apply(V + (size_t)(k + j0) * n, W + (size_t)(k + j0) * n, std::min(kBlk, r - j0));
    };
    auto grow = [&](int r, const std::vector<double> &C) {  // C = V^T W of the new columns, (k+r) x r
        std::vector<double> Tn((size_t)(k + r) * (k + r));
        for (int i = 0; i < k; i++)
            for (int j = 0; j < k; j++) Tn[(size_t)i * (k + r) + j] = Tm[(size_t)i * k + j];
        for (int i = 0; i < k + r; i++)
            for (int j = 0; j < r; j++) {
                const double v = C[(size_t)i * r + j];
                Tn[(size_t)i * (k + r) + k + j] = v;
                Tn[(size_t)(k + j) * (k + r) + i] = v;
            }
        for (int i = k; i < k + r; i++)  // symmetrise the new diagonal block
            for (int j = i + 1; j < k + r; j++) {
                const double v = 0.5 * (Tn[(size_t)i * (k + r) + j] + Tn[(size_t)j * (k + r) + i]);
                Tn[(size_t)i * (k + r) + j] = Tn[(size_t)j * (k + r) + i] = v;
            }
        Tm.swap(Tn);
        k += r;
    };
    auto extend = [&](int r) {  // V[k..k+r) are new orthonormal vectors
        images(r);
        grow(r, S.gram(V, k + r, W + (size_t)k * n, r));
    };
    extend(r0);
    std::vector<double> theta, Z;
    int nconv = 0;
    bool checked = !davidson;  // the expansion after convergence has been made
    bool any = false;          // harmonic energies: a diagonal preconditioner
    for (int i = 0; davidson && i < S.ctx->prob.D; i++) any |= S.ctx->host.harm_mono[i] >= 0;
    const int ne = std::min<int64_t>(nev, n);
    for (int it = 0; it < max_it; it++) {
        sym_eig(k, Tm, theta, Z);
        const int nr = std::min(ne + guard, k);
        // Ritz vectors and their images, residuals
        std::vector<double> Zr((size_t)k * nr);
        for (int i = 0; i < k; i++)
            for (int j = 0; j < nr; j++) Zr[(size_t)i * nr + j] = Z[(size_t)i * k + j];
        const Solver::Mat Zd = S.upload(Zr, k, nr);
        const double *th = S.upload(theta.data(), nr);
        S.combine(V, Zd, 1.0, nullptr, X);
        S.combine(W, Zd, 1.0, nullptr, HX);
        double *rn2 = S.pin + S.take(nr);
        ck(dev_residual(X, th, HX, nr, n, rn2, S.partial.p, S.s), "resid");
        S.sync("residual sync");
        std::vector<double> rn(rn2, rn2 + nr);
        for (double &v : rn) v = std::sqrt(v);
        nconv = 0;
        while (nconv < nr && rn[nconv] <= tol * std::max(1.0, std::fabs(theta[nconv]))) nconv++;
        for (int j = 0; j < std::min(nr, ne); j++) { evals[j] = theta[j]; if (resid) resid[j] = rn[j]; }
        if (k >= n || (nconv >= ne && (checked || nconv >= nr))) break;
        checked = nconv >= ne || !davidson;
        // new directions: the residuals of the first unconverged Ritz pairs (of
        // the wanted ones, or of those beyond them when these have converged);
        // a converged pair among them would only add rounding noise
        std::vector<double> sel;
        const int upto = nconv >= ne ? nr : std::min(ne, k);
        for (int j = nconv; j < upto && (int)sel.size() < 2 * b; j++)
            if (rn[j] > tol * std::max(1.0, std::fabs(theta[j]))) { sel.push_back(j); sel.push_back(theta[j]); }
        if (sel.empty()) { sel.push_back(nr - 1); sel.push_back(theta[nr - 1]); }
        const int r = (int)sel.size() / 2;
        if (!davidson && k + r > kmax) break;
        ck(dev_direction(HX, any ? S.ctx->kp.esplit : nullptr, S.upload(sel.data(), 2 * r), r, n, T, S.s), "directions");
        if (davidson && k + r > kmax) {  // restart with the current Ritz vectors
            const int keep = std::min(nr, kmax - r);
            ck(cudaMemcpyAsync(V, X, sizeof(double) * n * keep, cudaMemcpyDeviceToDevice, S.s), "restart V");
            k = 0;
            Tm.clear();
            extend(S.orthonormalise(V, keep, Q));  // recomputes W = H V
        }
        S.orth_against(V, k, T, r);
        // The new vectors, their images and inner products on the assumption
        // that the r directions are independent; the ranks come with the results.
        int *rank = reinterpret_cast<int *>(S.pin + S.take(1));
        S.chol_pass(T, r, Q, rank);
        S.chol_pass(Q, r, V + (size_t)k * n, rank + 1);
        images(r);
        double *C = S.pin + S.take((size_t)(k + r) * r);
        S.gram_to(V, k + r, W + (size_t)k * n, r, C);
        S.sync("extend sync");
        if (rank[0] == r && rank[1] == r) {
            grow(r, Solver::ungroup(C, k + r, r));
            continue;
        }
        int rk = S.orthonormalise(T, r, Q);
        if (rk == 0) {  // the directions lie in the basis: add random ones
            S.random_block(T, r, 0x5eed0000ull + (uint64_t)it);
            S.orth_against(V, k, T, r);
            rk = S.orthonormalise(T, r, Q);
            if (rk == 0) break;
        }
        ck(cudaMemcpyAsync(V + (size_t)k * n, T, sizeof(double) * n * rk, cudaMemcpyDeviceToDevice, S.s), "append");
        extend(rk);
    }
    if (evecs) ck(cudaMemcpyAsync(evecs, X, sizeof(double) * n * std::min(ne, k), cudaMemcpyDeviceToDevice, S.s), "evecs");
    S.sync("eigs sync");
    return std::min(nconv, ne);
}

// Spectral interval of H_S for the Chebyshev propagator: a 40-vector Krylov
// run (Rayleigh-Ritz), the extreme Ritz values widened by their residual norms
// and by 5% of the range.  Deterministic (fixed start vector, ordered sums).
// The run stays on the device: a vector that vanishes against the basis
// becomes zero there, and the host ends the basis at it afterwards.
constexpr int kBoundVectors = 40;
void spectral_bounds(Solver &S, double &emin, double &emax)
{
    const int64_t n = S.n;
    const int ks = (int)std::min<int64_t>(n, kBoundVectors);
    DBuf mem((2 * (size_t)ks + 5) * n + (size_t)ks * (ks + 2));
    double *const V = mem.p, *const W = V + (size_t)(ks + 1) * n, *const X = W + (size_t)ks * n, *const HX = X + 2 * n,
                 *const cols = HX + 2 * n, *const nn = cols + (size_t)ks * (ks + 1);
    S.random_block(V, 1, 0xc4eb00ull);
    ck(dev_normalise(V, n, nn, S.partial.p, S.s), "krylov start");
    for (int k = 0; k < ks; k++) {
        S.apply(V + (size_t)k * n, W + (size_t)k * n, 1);
        // column k of the projected matrix, which is also the first projection of the next vector
        double *c = cols + (size_t)k * ks;
        ck(dev_gram(V, k + 1, W + (size_t)k * n, 1, n, c, S.partial.p, S.s), "krylov gram");
        if (k + 1 == ks) break;
        double *next = V + (size_t)(k + 1) * n, *c2 = S.small.p;
        ck(dev_combine(V, k + 1, c, 1, -1.0, W + (size_t)k * n, next, n, S.s), "krylov step");
        // the second projection, with next . next as its last product (next follows the basis)
        ck(dev_gram(V, k + 2, next, 1, n, c2, S.partial.p, S.s), "krylov gram");
        ck(dev_project_normalise(V, k + 1, c2, next, n, nn + k + 1, S.s), "krylov norm");
    }
    S.sync("krylov sync");
    std::vector<double> hc((size_t)ks * (ks + 2));
    ck(cudaMemcpy(hc.data(), cols, sizeof(double) * hc.size(), cudaMemcpyDeviceToHost), "krylov copy");
    const double *hn = &hc[(size_t)ks * (ks + 1)];
    int k = 1;
    while (k < ks && hn[k] > 1e-24) k++;
    std::vector<double> Tm((size_t)k * k), th, Z;
    for (int j = 0; j < k; j++)
        for (int i = 0; i <= j; i++) Tm[(size_t)i * k + j] = Tm[(size_t)j * k + i] = hc[(size_t)j * ks + i];
    sym_eig(k, Tm, th, Z);
    std::vector<double> z((size_t)k * 2);
    for (int i = 0; i < k; i++) { z[2 * i] = Z[(size_t)i * k]; z[2 * i + 1] = Z[(size_t)i * k + k - 1]; }
    const double ends[2] = {th[0], th[k - 1]};
    const Solver::Mat zd = S.upload(z, k, 2);
    const double *te = S.upload(ends, 2);
    S.combine(V, zd, 1.0, nullptr, X);
    S.combine(W, zd, 1.0, nullptr, HX);
    double *rn2d = S.small.p + S.take(2), rn2[2];
    ck(dev_residual(X, te, HX, 2, n, rn2d, S.partial.p, S.s), "bound resid");
    S.sync("bounds sync");
    ck(cudaMemcpy(rn2, rn2d, sizeof rn2, cudaMemcpyDeviceToHost), "bound copy");
    const double range = th[k - 1] - th[0];
    emin = th[0] - std::sqrt(rn2[0]) - 0.05 * range;
    emax = th[k - 1] + std::sqrt(rn2[1]) + 0.05 * range;
}

// The steps of sg_propagate on the row form: one launch per Chebyshev term.
void propagate_rows(Solver &S, double *psi, double Ebar, double dE, double dt, const std::vector<double> &J, int kend,
                    int nsteps, double *norm_log, double *energy_log)
{
    if (nsteps == 0) return;
    const size_t n = (size_t)S.n;
    const sg_precision prec = S.ctx->prob.prec;
    const size_t rb = (size_t)row_value_bytes(prec);
    const bool logs = norm_log || energy_log;
    const size_t ndots = logs ? 8 * (size_t)nsteps : 0;
    // T_k and T_{k-1}, the partial sum, H psi, the two entry-major copies, inner products of every logged step, flags
    DBuf mem(8 * n + 2 * (2 * n * rb + 7) / 8 + ndots + 4);
    double *x = mem.p, *p = x + 2 * n, *acc = p + 2 * n, *y = acc + 2 * n, *c0 = y + 2 * n;
    unsigned char *xs = reinterpret_cast<unsigned char *>(c0), *xn = xs + 2 * n * rb;
    double *dots = c0 + 2 * (2 * n * rb + 7) / 8;
    unsigned *flags = reinterpret_cast<unsigned *>(dots + ndots);
    ck(cudaMemsetAsync(flags, 0, 2 * sizeof(unsigned), S.s), "flags");
    ck(cudaMemcpyAsync(x, psi, sizeof(double) * 2 * n, cudaMemcpyDeviceToDevice, S.s), "psi copy");
    RowIO r{};
    r.x = x;
    r.xs = xs;
    r.nvec = 2;
    r.stride = xs_stride(2);
    ck(launch_row_stage(S.ctx->rop, r, prec, S.s), "psi stage");
    for (int step = 0; step < nsteps; step++) {
        for (int kn = 1; kn <= kend; kn++) {
            const ChebIO io{x, logs ? y : nullptr, p, acc, xs, xn, flags};
            const ChebTerm t{kn, kend, Ebar, 1.0 / dE, std::cos(Ebar * dt), -std::sin(Ebar * dt), J[0], 2.0 * J[kn]};
            ck(launch_cheb_rows(S.ctx->rop, io, t, prec, S.s), "chebyshev term");
            if (kn == 1 && logs) {  // <psi|psi> and <psi|H psi> of the parts: the diagonals of 2 x 2 products
                ck(dev_gram(x, 2, x, 2, (int64_t)n, dots + 8 * step, S.partial.p, S.s), "norm");
                ck(dev_gram(x, 2, y, 2, (int64_t)n, dots + 8 * step + 4, S.partial.p, S.s), "energy");
            }
            std::swap(x, p);
            std::swap(xs, xn);
        }
    }
    ck(cudaMemcpyAsync(psi, x, sizeof(double) * 2 * n, cudaMemcpyDeviceToDevice, S.s), "psi copy");
    RowIO f{};
    f.y = psi;
    f.flags = flags;
    f.nvec = 2;
    ck(launch_row_settle(f, (int)n, S.s), "settle");
    S.sync("propagate sync");
    if (!logs) return;
    std::vector<double> h(ndots);
    ck(cudaMemcpy(h.data(), dots, sizeof(double) * h.size(), cudaMemcpyDeviceToHost), "logs");
    for (int step = 0; step < nsteps; step++) {
        const double *q = &h[8 * (size_t)step];
        const double nn = q[0] + q[3];
        if (norm_log) norm_log[step] = nn;
        if (energy_log) energy_log[step] = (q[4] + q[7]) / nn;
    }
}

}  // namespace

extern "C" {

sg_status sg_eigs(sg_ctx *ctx, int nev, int method, int block, double tol, int max_it, double *evals,
                  double *evecs, double *resid, void *stream)
{
    if (!ctx) return SG_EINVAL;
    if (!ctx->has_device) { ctx->last_error = "context was made by sg_plan"; return SG_EINVAL; }
    if (!sg_on_ctx_device(ctx)) { ctx->last_error = "the current CUDA device is not the one the context was made on"; return SG_EINVAL; }
    if (nev < 1 || nev > ctx->host.n_cs || !evals || !(tol > 0) || max_it < 1 ||
        (method != SG_LANCZOS && method != SG_DAVIDSON)) {
        ctx->last_error = "sg_eigs: need 1 <= nev <= N_cs, tol > 0, max_it >= 1, a known method, evals";
        return SG_EINVAL;
    }
    const int b = block <= 0 ? std::min(nev, kBlk) : std::min(block, kBlk);
    try {
        Solver S(ctx, (cudaStream_t)stream, std::max({3 * nev, nev + 6 * b, 328}), nev + b + 1);
        const int nconv = block_eigs(S, nev, b, method == SG_DAVIDSON, tol, max_it, nullptr, 0, evals, evecs, resid);
        if (nconv < std::min<int64_t>(nev, ctx->host.n_cs)) {
            ctx->last_error = "sg_eigs: " + std::to_string(nconv) + " of " + std::to_string(nev) + " eigenpairs converged";
            return SG_ENOCONV;
        }
    } catch (const SolverError &e) {
        ctx->last_error = e.msg;
        return e.st;
    }
    return SG_OK;
}

sg_status sg_eigs_refine(sg_ctx *ctx, int nev, double *evecs, double *evals, double *resid, double tol, int max_it,
                         void *stream)
{
    if (!ctx) return SG_EINVAL;
    if (!ctx->has_device || nev < 1 || nev > ctx->host.n_cs || !evecs || !evals || !(tol > 0) || max_it < 1) {
        ctx->last_error = "sg_eigs_refine: invalid arguments";
        return SG_EINVAL;
    }
    if (!sg_on_ctx_device(ctx)) { ctx->last_error = "the current CUDA device is not the one the context was made on"; return SG_EINVAL; }
    const int b = std::min(nev, kBlk);
    try {
        Solver S(ctx, (cudaStream_t)stream, std::max(3 * nev, nev + 6 * b), nev + b + 1);
        const int nconv = block_eigs(S, nev, b, true, tol, max_it, evecs, nev, evals, evecs, resid);
        if (nconv < nev) {
            ctx->last_error = "sg_eigs_refine: " + std::to_string(nconv) + " of " + std::to_string(nev) + " converged";
            return SG_ENOCONV;
        }
    } catch (const SolverError &e) {
        ctx->last_error = e.msg;
        return e.st;
    }
    return SG_OK;
}

sg_status sg_product_state(const sg_ctx *ctx, const double *factors, int ld, double *out_host)
{
    if (!ctx || !factors || !out_host || ld < ctx->host.kw) return SG_EINVAL;
    const int D = ctx->prob.D, L = ctx->prob.L, kw = ctx->host.kw;
    const std::vector<uint8_t> &lmin = ctx->host.lmin_tab;
    std::vector<int> k(D, 0), c(D, 0);
    int sum = 0;
    int64_t r = 0;
    for (;;) {
        double v = 1.0;
        for (int i = 0; i < D; i++) v *= factors[(size_t)i * ld + k[i]];
        out_host[r++] = v;
        int i = D - 1;
        while (i >= 0) {
            k[i]++;
            const int lm = k[i] < kw ? lmin[(size_t)i * kw + k[i]] : 255;
            if (lm <= L && sum - c[i] + lm <= L) { sum += lm - c[i]; c[i] = lm; break; }
            sum -= c[i]; c[i] = 0; k[i] = 0; i--;
        }
        if (i < 0) break;
    }
    return r == ctx->host.n_cs ? SG_OK : SG_EINVAL;
}

sg_status sg_propagate(sg_ctx *ctx, double *psi, double dt, int nsteps, int order, double *norm_log,
                       double *energy_log, void *stream)
{
    if (!ctx) return SG_EINVAL;
    if (!ctx->has_device || !psi || nsteps < 0 || order < 1 || !std::isfinite(dt)) {
        ctx->last_error = "sg_propagate: invalid arguments";
        return SG_EINVAL;
    }
    if (!sg_on_ctx_device(ctx)) { ctx->last_error = "the current CUDA device is not the one the context was made on"; return SG_EINVAL; }
    try {
        Solver S(ctx, (cudaStream_t)stream, kBoundVectors, 2, !ctx->host.rows);
        const int64_t n = S.n;
        double emin, emax;
        spectral_bounds(S, emin, emax);
        const double Ebar = 0.5 * (emax + emin), dE = 0.5 * (emax - emin);
        const std::vector<double> J = bessel_j(order, dE * dt);
        int kend = order;  // skip terms whose Bessel weight is below double precision
        while (kend > 1 && kend > dE * dt && std::fabs(J[kend]) < 1e-17) kend--;
        if (ctx->host.rows) {
            propagate_rows(S, psi, Ebar, dE, dt, J, kend, nsteps, norm_log, energy_log);
            return SG_OK;
        }
        // phi buffers: 2 real vectors (re, im) each
        DBuf p0(2 * (size_t)n), p1(2 * (size_t)n), hp(2 * (size_t)n), acc(2 * (size_t)n);
        const double cph = std::cos(Ebar * dt), sph = -std::sin(Ebar * dt);  // e^{-i Ebar dt}
        for (int step = 0; step < nsteps; step++) {
            // phi_0 = psi, phi_1 = (H - Ebar) psi / dE
            ck(cudaMemcpyAsync(p0.p, psi, sizeof(double) * 2 * n, cudaMemcpyDeviceToDevice, S.s), "cheb copy");
            S.apply(p0.p, hp.p, 2);
            if (norm_log || energy_log) {
                std::vector<double> a = S.gram(psi, 1, psi, 1), bq = S.gram(psi + n, 1, psi + n, 1);
                std::vector<double> c1 = S.gram(psi, 1, hp.p, 1), c2 = S.gram(psi + n, 1, hp.p + n, 1);
                const double nn = a[0] + bq[0];
                if (norm_log) norm_log[step] = nn;
                if (energy_log) energy_log[step] = (c1[0] + c2[0]) / nn;
            }
            ck(cudaMemcpyAsync(p1.p, hp.p, sizeof(double) * 2 * n, cudaMemcpyDeviceToDevice, S.s), "cheb copy");
            ck(dev_axpby(2 * n, -Ebar / dE, p0.p, 1.0 / dE, p1.p, S.s), "cheb phi1");
            // acc = J0 phi0 + 2 J1 (-i) phi1
            ck(dev_axpby(2 * n, J[0], p0.p, 0.0, acc.p, S.s), "acc0");
            auto add_term = [&](int kk, const double *ph) {
                const double c = (kk == 0 ? 1.0 : 2.0) * J[kk];
                // (-i)^kk (x + i y): 0: x + iy; 1: y - ix; 2: -x - iy; 3: -y + ix
                const double *x = ph, *y = ph + n;
                double *ar = acc.p, *ai = acc.p + n;
                switch (kk % 4) {
                    case 0: ck(dev_axpby(n, c, x, 1.0, ar, S.s), "t"); ck(dev_axpby(n, c, y, 1.0, ai, S.s), "t"); break;
                    case 1: ck(dev_axpby(n, c, y, 1.0, ar, S.s), "t"); ck(dev_axpby(n, -c, x, 1.0, ai, S.s), "t"); break;
                    case 2: ck(dev_axpby(n, -c, x, 1.0, ar, S.s), "t"); ck(dev_axpby(n, -c, y, 1.0, ai, S.s), "t"); break;
                    default: ck(dev_axpby(n, -c, y, 1.0, ar, S.s), "t"); ck(dev_axpby(n, c, x, 1.0, ai, S.s), "t"); break;
                }
            };
            add_term(1, p1.p);
            double *a0 = p0.p, *a1 = p1.p;
            for (int kk = 2; kk <= kend; kk++) {
                // phi_{k} = 2 (H - Ebar)/dE phi_{k-1} - phi_{k-2}, written over phi_{k-2}
                S.apply(a1, hp.p, 2);
                ck(dev_axpby(2 * n, -2.0 * Ebar / dE, a1, -1.0, a0, S.s), "cheb rec");
                ck(dev_axpby(2 * n, 2.0 / dE, hp.p, 1.0, a0, S.s), "cheb rec");
                std::swap(a0, a1);
                add_term(kk, a1);
            }
            // psi = e^{-i Ebar dt} acc
            ck(dev_axpby(n, cph, acc.p, 0.0, psi, S.s), "phase");
            ck(dev_axpby(n, -sph, acc.p + n, 1.0, psi, S.s), "phase");
            ck(dev_axpby(n, sph, acc.p, 0.0, psi + n, S.s), "phase");
            ck(dev_axpby(n, cph, acc.p + n, 1.0, psi + n, S.s), "phase");
        }
        ck(cudaStreamSynchronize(S.s), "propagate sync");
    } catch (const SolverError &e) {
        ctx->last_error = e.msg;
        return e.st;
    }
    return SG_OK;
}

}  // extern "C"

namespace sg {

sg_status davidson_routed(sg_ctx *ctx, cudaStream_t stream, const ApplyFn &apply, int nev, int block, double tol,
                          int max_it, double *evals, double *resid, double *evecs, int *nconv, std::string *err)
{
    const int b = block <= 0 ? std::min(nev, kBlk) : std::min(block, kBlk);
    try {
        Solver S(ctx, stream, std::max(3 * nev, nev + 6 * b), nev + b + 1);
        S.apply_fn = &apply;
        *nconv = block_eigs(S, nev, b, true, tol, max_it, nullptr, 0, evals, evecs, resid);
    } catch (const SolverError &e) {
        if (err) *err = e.msg;
        return e.st;
    }
    return SG_OK;
}

int64_t davidson_device_bytes(int64_t n, int nev, int block)
{
    const int b = block <= 0 ? std::min(nev, kBlk) : std::min(block, kBlk);
    const int kmax = std::max(3 * nev, nev + 6 * b), cols = nev + b + 1;
    const size_t small = Solver::scratch(n, kmax, cols) + Solver::capacity(kmax, cols);
    return (int64_t)sizeof(double) * (int64_t)(small + EigVectors(n, nev, b, true, 1, 0).total * n);
}

sg_status chebyshev_bounds(sg_ctx *ctx, cudaStream_t stream, double *emin, double *emax)
{
    try {
        Solver S(ctx, stream, kBoundVectors, 2, false);
        spectral_bounds(S, *emin, *emax);
        ck(cudaStreamSynchronize(S.s), "bounds sync");
    } catch (const SolverError &e) {
        ctx->last_error = e.msg;
        return e.st;
    }
    return SG_OK;
}

}  // namespace sg
