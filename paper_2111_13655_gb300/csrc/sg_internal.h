// Internal declarations of libsmolyak (host setup <-> CUDA kernels <-> C ABI).
#pragma once

#include <cstdint>
#include <functional>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/smolyak.h"

namespace sg {

constexpr int kMaxD = 32;          // modes per problem
constexpr int kMaxLevelSize = 32;  // nb(l), nq(l) at any level
constexpr int kMaxMono = 256;      // monomials in V
constexpr int kMaxFac = 8;         // factors per monomial
constexpr int kMaxPow = 16;        // power of one factor
constexpr int kThreads = 128;      // threads per term-CTA

// Per (mode, level) entry: sizes and element offsets into the flat tables.
struct LevelInfo {
    int nb, nq;
    int offB;   // B[u*nb+k]   = b_k(Q_u)                 (nq x nb)
    int offBW;  // BW[k*nq+u]  = w_u b_k(Q_u)             (nb x nq)
    int offK;   // K[k*nb+k']  = -omega/2 <b_k|d2/dQ2|b_k'> on the grid (nb x nb)
    int offQ;   // Q[u]        = Q_u                      (nq)
    int offMu;  // mu[p]       = sum_u w_u b_0(Q_u)^2 Q_u^p, p = 0..pmax (pmax+1)
    int offM;   // M_p[k*nb+k'] = sum_u w_u b_k(Q_u) Q_u^p b_k'(Q_u), p = 1..pmax (pmax blocks nb x nb)
};

// Fixed-point accumulation of the compact result: every contribution D_l * y_l[k]
// is added exactly as an integer multiple of 2^E (E chosen per vector from
// max|x|), split into four signed 32-bit digits held in int64 words.
constexpr int kAccDigits = 4;
constexpr int kAccLsbBelowMax = 80;  // E = exponent(max|x|) - 80
// FP32 contexts: one signed 64-bit word per entry, unit 2^(exponent(max|x|) - 40)
constexpr int kAcc32LsbBelowMax = 40;
// 64-bit words per accumulated entry of a context's precision
__host__ __device__ constexpr int acc_words(bool fp32) { return fp32 ? 1 : kAccDigits; }

constexpr int kMaxPairs = 64;  // coupled mode pairs of a pair potential

// ---------------------------------------------------------------------------
// The row form of H_S (sg_rows.cu, sg_rows_setup.cpp).  With U_i(l) the
// operator of mode i on level l and Delta_i(l) = U_i(l) - U_i(l-1), Eq. (16)'s
// sum over the terms l in R(l) with the coefficients D_l of Eq. (8) is
//     H_S = sum_{|l| <= L} (x)_i Delta_i(l_i)
// for every product operator (x)_i U_i.  The potential is a sum of monomials,
// and a mode that a monomial does not touch contributes B^T W B = I on its
// nb(l) functions (nq >= nb), so Delta_i(l)[k] = 1 exactly for l = lmin_i(k).
// A monomial over the modes S therefore couples k and k' (equal outside S) by
//     c sum_{l_S: |l_S| <= T} prod_{i in S} Delta M_i(l_i)[k_i][k'_i],
//     T = L - sum_{i not in S} lmin_i(k_i),
// M_i(l) = B^T W diag(Q^p) B the quadrature matrix of the monomial's power on
// level l (the kinetic part: K).  These elements, quadrature errors included,
// are those of the term-by-term sum; M_i(l) is a power of the tridiagonal
// Jacobi matrix of the grid, so a monomial of power p couples k_i to
// k_i - p .. k_i + p only (every second one when q0 = 0), and few of these
// shifts stay inside the compact basis: 15 per row at D=12 L=10.  The
// elements are formed once per context in FP64 and stored row by row.

// One window: consecutive rows and their entries, stored together (a 16-byte
// aligned record that a bulk copy brings into shared memory):
//   per row, by decreasing length: {first entry | local row << 24, entries}
//   (8 bytes each, padded to 16), then the columns (int32 compact indices) and
//   the elements (float, double, or float2 = (hi, lo)) of the rows one after
//   another, each row filled to a multiple of four entries.
struct RowWin {
    long long off;    // byte offset of the record
    int row0, nrows;
    int nent, pad;    // entries, fillers included
};
__host__ __device__ inline int row_meta_bytes(int nrows) { return (8 * nrows + 15) & ~15; }
__host__ __device__ inline int row_win_bytes(const RowWin &w, int value_bytes)
{
    return row_meta_bytes(w.nrows) + w.nent * (4 + value_bytes);
}
// One problem's row operator on the device.
struct RowOp {
    const unsigned char *blob;  // the windows' records
    const RowWin *wins;
    const double *esplit;   // harmonic diagonal (FP64)
    int *err;
    int nwin, n;
    int cap;                // largest record that is staged (bytes); longer ones (a very long row) are read in place
    int wrows;              // rows per window (a power of two)
};
// What a row kernel reads and writes.
struct RowIO {
    const double *x;        // input vectors, column after column
    const void *xs;         // entry-major copy in the contraction type (rows of `stride`), or nullptr: gather from x
    double *y;              // result, or nullptr: the sums go to acc
    unsigned long long *acc;
    unsigned *flags;        // per vector: set when x holds a non-finite value
    unsigned *ticket;       // zero between launches; nullptr: launch_row_settle follows
    int nvec, stride, words;
    int part, nparts;       // windows w with w % nparts == part
};
// Largest level and number of distinct index shifts the row form is built for.
constexpr int kRowMaxL = 63;
constexpr int kRowMaxShifts = 65536;
// Largest row operator (bytes); larger ones use the term-by-term kernel.
constexpr int64_t kRowMaxBytes = (int64_t)64 << 30;

// Default plan of the row kernels (sg_tune measures the alternatives).
#ifndef SG_F32_VT
#define SG_F32_VT 4
#endif
#ifndef SG_F64_VT
#define SG_F64_VT 1
#endif
#ifndef SG_DF_VT
#define SG_DF_VT 2
#endif
#ifndef SG_ROW_WINDOW
#define SG_ROW_WINDOW 4  // rows per window, in units of 16
#endif
constexpr int kRowWindowMax = 64;  // rows per window at most
#ifndef SG_ROW_SHARE
#define SG_ROW_SHARE 4   // resident blocks that share the shared-memory budget
#endif
#ifndef SG_F32_SMEM_KB
#define SG_F32_SMEM_KB 52
#endif
#ifndef SG_F64_SMEM_KB
#define SG_F64_SMEM_KB 70
#endif

// Row length (elements) of the entry-major input copy for nvec vectors.
__host__ __device__ inline int xs_stride(int nvec) { return nvec <= 2 ? nvec : (nvec + 3) & ~3; }
// FP64 rows with one vector per lane gather from x itself at any size: the FP64
// pipe hides the extra sectors, and the copy is saved (8 vectors: D=10 L=8 24.2 us
// without the copy and 27.6 with it, D=12 L=8 41.0 and 42.5, D=12 L=9 87.5 and
// 89.9, D=12 L=10 202 and 203; 5 vectors 18.6 and 21.8, 31.0 and 33.0, 61.8 and
// 67.6, 147 and 154).  Other types convert what they gather: 2 to 3 times slower.
inline bool rows_direct(sg_precision prec, int vt, int nvec) { return prec == SG_FP64 && (vt == 1 || nvec == 1); }

// Everything the set-up kernels and the term-by-term kernel need.
struct alignas(16) KParams {
    int D, L, Dpad;
    int nmono, pmax, kw;
    int n_cs;
    int64_t n_terms;
    const uint8_t *levels;   // [n_terms][Dpad], Table-2 order
    const int *coefs;        // [n_terms] combination coefficient D_l
    const int *order;        // [n_terms] Table-2 index of the p-th processed term
    const int *rank_tab;     // [D][L+1][kw]: partial ranks T_i[s][k]
    const uint8_t *lmin_tab; // [D][kw]: smallest level holding function k
    const LevelInfo *lvl;    // [D][L+1]
    const double *tabd;      // flat FP64 tables
    const float *tabf;       // FP32 copies (same offsets)
    const double *mcoef;     // [nmono]
    const int *mnfac;        // [nmono]
    const int *mfoff;        // [nmono+1]
    const int *mfmode;       // [sum nfac]
    const int *mfpow;        // [sum nfac]
    const int *harm_mono;    // [D] monomial holding the harmonic part of mode i (-1: not split)
    const double *esplit;    // [n_cs] sum over split modes of omega_i s_i^2 (k_i + 1/2)
    unsigned long long *acc; // [n_cs][nvec][acc_words] fixed-point accumulators (entry-major)
    // capacities of the per-CTA shared-memory areas (elements)
    int cap;       // each of the two grid ping-pong buffers
    int maxnb;     // term basis tensor
    int matcap;    // per-term 1D matrices
    int vtabcap;   // per-term potential tables
    int *err;      // device error word (0 = fine)
    // term-sharded applies: only processing positions p with p % nparts == part
    int part, nparts;
};

// Shift tables of the row form (device copies of the HostTables arrays).
struct RowShifts {
    int nshift;
    const int *off;        // [nshift + 1] into mode / d
    const int *mode, *d;   // the modes a shift moves, and by how much
    const int *src_off;    // [nshift + 1] into src
    const int *src;        // products that contribute to the shift
    const int *prod_off;   // [nprod + 1] into fmode / fop
    const int *fmode, *fop;  // factors of a product: mode, power (0: the kinetic matrix)
    const double *coef;    // [nprod]
};

// Host-side description of a problem (after validation).
struct Problem {
    int D = 0, L = 0;
    std::vector<sg_basis> basis;
    std::vector<sg_grid> grids;
    std::vector<double> omega;
    std::vector<double> mcoef;
    std::vector<int> mnfac, mfoff, mfmode, mfpow;
    sg_precision prec = SG_FP64;
};

// Result of the host setup: everything that is uploaded.
struct HostTables {
    int Dpad = 0, pmax = 0, kw = 0;
    int64_t n_terms = 0, n_cs = 0, n_s = 0, n_grid = 0;
    std::vector<uint8_t> levels;     // [n_terms][Dpad]
    std::vector<int> coefs;          // [n_terms]
    std::vector<int> order;          // processing order (Table-2 indices)
    std::vector<int64_t> pcost;      // estimated cost of the p-th processed term
    std::vector<int> rank_tab;       // [D][L+1][kw]
    std::vector<uint8_t> lmin_tab;   // [D][kw]
    std::vector<LevelInfo> lvl;      // [D][L+1]
    std::vector<double> tabd;
    std::vector<int> harm_mono;      // [D]
    std::vector<double> esplit;      // [n_cs]
    bool pairs = false;  // every monomial touches at most two modes, in at most kMaxPairs pairs
    // row form (see RowShifts); rows = false: the term-by-term kernel applies H_S
    bool rows = false;
    int64_t row_nnz = 0;             // entries of the row operator
    std::vector<int> sh_off, sh_mode, sh_d, sh_src_off, sh_src, pr_off, pr_mode, pr_op;
    std::vector<double> pr_coef;
    // plan of the row kernels (0: default): vectors per lane, rows per window
    // in units of 16, shared memory that SG_ROW_SHARE blocks may use (bytes)
    int slice_vt = 0, warp_vt = 0, fbudget = 0;
    int cap = 0, maxnb = 0, matcap = 0, vtabcap = 0;
};

// Host setup (sg_setup.cpp).  Returns an empty string on success, else the error text.
std::string build_tables(const Problem &p, int smem_budget_bytes, int real_bytes, HostTables *out);

// One-mode Gauss-Hermite rule with Hermite-function-normalised weights.
std::string gauss_hermite(int n, std::vector<double> *x, std::vector<double> *wf);

// Term-by-term kernel (sg_apply.cu).  Return cudaSuccess or the launch error.
cudaError_t launch_apply(const KParams &kp, bool fp32, const double *x, double *y, int nvec,
                         long long *maxbits, cudaStream_t stream);
cudaError_t launch_index_map(const KParams &kp, int64_t t0, int64_t nt, const int64_t *offsets_dev,
                             int64_t *cs_index, cudaStream_t stream);
size_t apply_smem_bytes(const KParams &kp, bool fp32);
cudaError_t configure_kernels(size_t smem_bytes, bool fp32);
// The passes of launch_apply: per-vector max|x| bits (zeroed first), the terms,
// and y = (accumulated integer) * 2^E + esplit * x, which also clears kp.acc.
cudaError_t launch_maxabs(const KParams &kp, const double *x, int nvec, long long *maxbits, cudaStream_t stream);
cudaError_t launch_apply_terms(const KParams &kp, bool fp32, const double *x, const long long *maxbits, int nvec,
                               cudaStream_t stream);
cudaError_t launch_finalize(const KParams &kp, bool fp32, const double *x, double *y, int nvec,
                            const long long *maxbits, cudaStream_t stream);

// Row form, host half (sg_rows_setup.cpp).
void build_row_shifts(const Problem &p, HostTables *T);
int row_vt(const HostTables &T, sg_precision prec);      // vectors per lane of the plan
int row_window_units(const HostTables &T);               // rows per window / 16 of the plan
int row_budget(const HostTables &T, sg_precision prec);  // shared memory that SG_ROW_SHARE blocks may use (bytes)
int row_value_bytes(sg_precision prec);                  // bytes of a stored element
// Upper bounds of the row operator's windows and of its device bytes.
int64_t row_form_windows(const HostTables &T, sg_precision prec);
int64_t row_form_bytes(const HostTables &T, sg_precision prec);
struct RowWindows {
    std::vector<RowWin> wins;
    std::vector<uint2> meta;   // in the order of the records
    std::vector<int> win;      // window of each row
    std::vector<int> start;    // first entry of each row in its window
    int64_t bytes = 0;
    int cap = 0, wrows = 0;
};
// Cuts the rows (cnt[r] entries each) into windows of at most `wrows` rows and
// `budget` bytes, and orders the rows of each by decreasing length.
RowWindows cut_rows(const std::vector<int> &cnt, int wrows, int budget, int value_bytes);
int row_window_rows(int64_t n, int units);

// Row form, device half (sg_rows.cu).  prec selects the element type.
cudaError_t launch_row_count(const KParams &kp, const RowShifts &sh, int *cnt, cudaStream_t stream);
// The records of nwin windows of at most `most` entries each.
cudaError_t launch_row_fill(const KParams &kp, const RowShifts &sh, sg_precision prec, const RowWin *wins, int nwin,
                            int most, const int *win, const int *start, const uint2 *meta, unsigned char *blob,
                            cudaStream_t stream);
cudaError_t configure_rows();
// y = H_S x (io.y), or the sums of the windows of io.part into io.acc; vt: vectors per lane.
cudaError_t launch_rows(const RowOp &R, const RowIO &io, sg_precision prec, int vt, cudaStream_t stream);
// io.xs = the vectors entry-major in the contraction type; a batch: every problem's rows from cs_prefix[j] * stride.
cudaError_t launch_row_stage(const RowOp &R, const RowIO &io, sg_precision prec, cudaStream_t stream);
cudaError_t launch_row_stage_batch(const RowIO &io, sg_precision prec, const long long *cs_prefix, const int2 *items,
                                   int nitems, cudaStream_t stream);
// Vectors with a non-finite input become NaN; clears the flags (after launch_rows without a ticket).
cudaError_t launch_row_settle(const RowIO &io, int n, cudaStream_t stream);
cudaError_t launch_row_settle_batch(const RowIO &io, const long long *cs_prefix, int nprob, cudaStream_t stream);
// y from the summed accumulators of all parts; clears them.
cudaError_t launch_row_finish(const RowOp &R, const RowIO &io, cudaStream_t stream);
// Many problems: item = (problem, window); RowIO holds the batch's buffers.
cudaError_t launch_rows_batch(const RowOp *ops, const int2 *items, int nitems, int cap, int wrows, const RowIO &io,
                              sg_precision prec, int vt, const long long *cs_prefix, cudaStream_t stream);

// Propagation server (sg_server_api.cpp, sg_server.cu): device state of one
// active request's Chebyshev recurrence.  One iteration after Y = H X logs
// norm and energy for requests at k = 0, forms T_{k+1} (T_1 from T_0 when
// k = 0), adds c_{k+1} (-i)^{k+1} T_{k+1} to the partial sum and, on the
// step's last term (k + 1 = K), writes e^{-i Ebar dt} * sum; then k, step advance.
struct ChebState {
    int k, K, step, nsteps;
    double ebar, inv_de;   // (H - ebar) * inv_de maps the spectrum into [-1, 1]
    double cph, sph;       // e^{-i Ebar dt} = cph + i sph
    const double *c;       // device: (2 - delta_k0) J_k(dE dt), k = 0..K
    double *log;           // device: [nsteps][norm, energy]
};
cudaError_t launch_cheb_iteration(ChebState *st, const long long *prefix, int nitems, int64_t total,
                                  const double *X, const double *Y, double *P, double *A, cudaStream_t s);
// Logs the requests at the start of a step, then moves every request to its next term.
cudaError_t launch_cheb_log_advance(ChebState *st, const long long *prefix, int nitems, const double *X,
                                    const double *Y, cudaStream_t s);
// One recurrence term in one launch (sg_rows.cu): y = H T_k row by row, and the
// update of launch_cheb_iteration where the row sum ends.  Vectors as there
// (real parts, then imaginary parts); xs, xs_next: T_k and T_{k+1} entry-major
// in the contraction type; y is stored only at the start of a step (when not
// nullptr).  The term comes from `one` (host values) or, for a batch, from the
// requests' device states.
struct ChebTerm {
    int kn, K;             // forms T_kn; K: the step's last term
    double ebar, inv_de, cph, sph;
    double c0, cn;         // weights of T_0 (used when kn = 1) and of T_kn
};
struct ChebIO {
    const double *X;
    double *Y, *P, *A;
    const void *xs;
    void *xs_next;
    unsigned *flags;       // two words, set when X holds a non-finite value (nullptr: not kept)
};
cudaError_t launch_cheb_rows(const RowOp &R, const ChebIO &io, const ChebTerm &one, sg_precision prec,
                             cudaStream_t stream);
cudaError_t launch_cheb_rows_batch(const RowOp *ops, const int2 *items, int nitems, int cap, const ChebIO &io,
                                   const ChebState *st, sg_precision prec, const long long *cs_prefix,
                                   cudaStream_t stream);
// Chebyshev spectral interval of a context's H_S (Krylov, as sg_propagate); synchronous.
sg_status chebyshev_bounds(sg_ctx *ctx, cudaStream_t stream, double *emin, double *emax);
// Block Davidson of sg_eigs (method SG_DAVIDSON, same start block and
// iteration) with every application of H_S done by `apply` (x, y device, r
// vectors; x is ready when it is called, y must be complete when it returns).
// Vector algebra runs on `stream`.  nconv receives the converged pairs.
using ApplyFn = std::function<sg_status(const double *x, double *y, int r)>;
sg_status davidson_routed(sg_ctx *ctx, cudaStream_t stream, const ApplyFn &apply, int nev, int block, double tol,
                          int max_it, double *evals, double *resid, double *evecs, int *nconv, std::string *err);
// Device bytes that davidson_routed holds on n-entry vectors (eigenvectors and the routed apply's buffers apart).
int64_t davidson_device_bytes(int64_t n, int nev, int block);
// J_0..J_kmax at x (Miller's backward recurrence).
std::vector<double> bessel_j(int kmax, double x);
// Device bytes that sg_create keeps for a planned context, from above: the row
// operator and its tables, or the term-by-term tables where these are larger
// (a context may be made with them when the row operator does not fit).
int64_t planned_device_bytes(const sg_ctx *ctx);

}  // namespace sg

struct sg_ctx {
    sg::Problem prob;
    sg::HostTables host;
    sg::KParams kp{};
    int device = 0;
    bool fp32 = false;
    bool has_device = false;  // false for contexts made by sg_plan
    size_t smem_bytes = 0;
    int64_t bytes_device = 0;
    std::vector<void *> allocations;
    double *stage_x = nullptr, *stage_y = nullptr;  // host-API staging (device)
    int64_t stage_elems = 0;
    // row operator: its buffers, and the plan's vectors per lane
    sg::RowOp rop{};
    std::vector<void *> row_allocs;
    std::vector<int> win_entries, win_rows;  // entries and rows of each window
    int64_t row_bytes = 0;
    // apply workspace.  Row form: per-vector flags and the entry-major input
    // copy; term-by-term kernel: fixed-point accumulators and scale exponents
    void *xs = nullptr;
    unsigned *flags = nullptr;  // behind xs, in its allocation; after acc_nvec flags, the ticket
    unsigned long long *acc = nullptr;
    long long *maxbits = nullptr;
    int acc_nvec = 0;
    double *pin = nullptr;    // pinned host memory of the solvers' small matrices
    size_t pin_doubles = 0;
    int plan_version = 0;     // incremented whenever a plan or a row operator is installed
    std::string last_error;
};

// Calls with device work run on the device the context was made on: from any
// other current device its kernels would be handed another GPU's pointers.
inline bool sg_on_ctx_device(const sg_ctx *ctx)
{
    int cur = -1;
    return cudaGetDevice(&cur) == cudaSuccess && cur == ctx->device;
}

namespace sg {

// Row operator of a context (sg_api.cpp): forms it with the context's plan
// (then replacing an earlier one, which a failure leaves in force), releases
// it, and enqueues one apply or part.
cudaError_t build_rows(sg_ctx *ctx);
void free_rows(sg_ctx *ctx);
cudaError_t apply_rows(sg_ctx *ctx, RowIO io, cudaStream_t s);

// One recurrence term of every problem of a batch, two vectors each (sg_batch.cpp);
// `restage`: xs is made from X first.  SG_EUNSUPPORTED when a problem is applied term by term.
sg_status batch_cheb(sg_batch *b, const ChebIO &io, const ChebState *st, bool restage, cudaStream_t s);

}  // namespace sg
