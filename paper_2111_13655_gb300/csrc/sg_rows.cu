// Row form of H_S on the device (described in sg_internal.h): the kernels that
// form the row operator once per context, and those that apply it.
//
// One block applies one window of consecutive rows to all vectors:
//   1. the window's entries (column, element) come into shared memory by
//      16-byte asynchronous copies, as they lie;
//   2. a group of lanes takes a row, each lane `VT` vectors: per entry one
//      load of VT adjacent values of the entry-major copy xs and VT
//      multiply-adds.  The rows of a window go by decreasing length, so the
//      rows of a warp have about the same number of entries;
//   3. the row sums go through a shared-memory tile, so that y (column after
//      column) is written, and x read for the harmonic diagonal, in runs of
//      consecutive rows.
// A row's entries are summed in column order by one lane whatever the plan,
// the number of vectors or the batch, so every entry point gives the same bits.
// Sums: FP64 by fma; mixed precision rounds each product to FP32 and adds it
// to a pair of FP32 numbers without error (two-sum), so nothing is lost in the
// accumulation; double-float as df_fma.
#include <algorithm>
#include <cstring>

#include "sg_df.cuh"
#include "sg_internal.h"

namespace sg {

namespace {

constexpr int kRT = 128;    // threads per window block
constexpr int kTileV = 8;   // vectors per pass (the tile's columns)

// ---------------------------------------------------------------- set-up

// Multi-index of compact index r; returns the sum of its levels.
__device__ int unrank(const KParams &P, int r, int *k)
{
    int s = 0;
    const int Lp = P.L + 1;
    for (int i = 0; i < P.D; i++) {
        const int *t = P.rank_tab + (size_t)(i * Lp + s) * P.kw;
        int v = 0;
        while (v + 1 < P.kw && __ldg(t + v + 1) <= r) {
            // entries past the last admissible function repeat the total, which exceeds r
            v++;
        }
        k[i] = v;
        r -= __ldg(t + v);
        s += P.lmin_tab[i * P.kw + v];
    }
    return s;
}

// Whether k + shift q is a compact function and the pair couples (the levels
// of max(k_i, k_i + d_i) fit under L).
__device__ bool shift_fits(const KParams &P, const RowShifts &S, int q, const int *k, int sum)
{
    int s = sum;
    for (int e = S.off[q]; e < S.off[q + 1]; e++) {
        const int i = S.mode[e], d = S.d[e], k2 = k[i] + d;
        if (k2 < 0 || k2 >= P.kw) return false;
        if (d > 0) {
            const int lm = P.lmin_tab[i * P.kw + k2];
            if (lm > P.L) return false;
            s += lm - P.lmin_tab[i * P.kw + k[i]];
        }
    }
    return s <= P.L;
}

// M_i(l)[k][k'] of one factor: B^T W diag(Q^op) B, or the kinetic matrix (op 0)
__device__ double factor_elem(const KParams &P, int mode, int op, int l, int k, int k2)
{
    const LevelInfo li = P.lvl[mode * (P.L + 1) + l];
    if (k >= li.nb || k2 >= li.nb) return 0.0;
    const int off = op == 0 ? li.offK : li.offM + (op - 1) * li.nb * li.nb;
    return P.tabd[off + k * li.nb + k2];
}
__device__ double factor_diff(const KParams &P, int mode, int op, int l, int k, int k2)
{
    const double m = factor_elem(P, mode, op, l, k, k2);
    return l > 0 ? m - factor_elem(P, mode, op, l - 1, k, k2) : m;
}

// sum over |l_S| <= T of prod Delta M_i(l_i)[k_i][k'_i] over the factors of
// product q; the last factor's differences are summed in closed form
// (sum_{l <= t} Delta M(l) = M(t)).
__device__ double product_elem(const KParams &P, const RowShifts &S, int q, const int *k, const int *k2, int sum)
{
    const int f0 = S.prod_off[q], f1 = S.prod_off[q + 1];
    int T = P.L - sum;
    for (int f = f0; f < f1; f++) T += P.lmin_tab[S.fmode[f] * P.kw + k[S.fmode[f]]];
    if (f0 == f1) return 1.0;
    const int last = f1 - 1, ml = S.fmode[last], ol = S.fop[last];
    if (f1 - f0 == 1) return factor_elem(P, ml, ol, T, k[ml], k2[ml]);
    double a[kRowMaxL + 1], b[kRowMaxL + 1];
    {
        const int m = S.fmode[f0], o = S.fop[f0];
        for (int l = 0; l <= T; l++) a[l] = factor_diff(P, m, o, l, k[m], k2[m]);
    }
    for (int f = f0 + 1; f < last; f++) {
        const int m = S.fmode[f], o = S.fop[f];
        for (int t = 0; t <= T; t++) {
            double v = 0.0;
            for (int l = 0; l <= t; l++) v = fma(a[t - l], factor_diff(P, m, o, l, k[m], k2[m]), v);
            b[t] = v;
        }
        for (int t = 0; t <= T; t++) a[t] = b[t];
    }
    double v = 0.0;
    for (int l = 0; l <= T; l++)
        if (a[l] != 0.0) v = fma(a[l], factor_elem(P, ml, ol, T - l, k[ml], k2[ml]), v);
    return v;
}

// One warp per row, lanes over the shifts.
__global__ void __launch_bounds__(256) k_row_count(const KParams P, const RowShifts S, int *__restrict__ cnt)
{
    const int r = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (r >= P.n_cs) return;
    int k[kMaxD];
    const int sum = unrank(P, r, k);
    int c = 0;
    for (int q0 = 0; q0 < S.nshift; q0 += 32)
        c += __popc(__ballot_sync(0xffffffffu, q0 + lane < S.nshift && shift_fits(P, S, q0 + lane, k, sum)));
    if (lane == 0) cnt[r] = c;
}

template <typename T> struct Elem;
template <> struct Elem<float> { static __device__ float of(double v) { return (float)v; } };
template <> struct Elem<double> { static __device__ double of(double v) { return v; } };
template <> struct Elem<df2> { static __device__ df2 of(double v) { return df2(v); } };

template <typename T>
__global__ void __launch_bounds__(256) k_row_fill(const KParams P, const RowShifts S,
                                                  const long long *__restrict__ start, int *__restrict__ cols,
                                                  T *__restrict__ vals)
{
    const int r = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (r >= P.n_cs) return;
    int k[kMaxD], k2[kMaxD];
    const int sum = unrank(P, r, k);
    long long at = start[r];
    for (int q0 = 0; q0 < S.nshift; q0 += 32) {
        const int q = q0 + lane;
        const bool in = q < S.nshift && shift_fits(P, S, q, k, sum);
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) {
            for (int i = 0; i < P.D; i++) k2[i] = k[i];
            for (int e = S.off[q]; e < S.off[q + 1]; e++) k2[S.mode[e]] += S.d[e];
            int c = 0, s = 0;
            for (int i = 0; i < P.D; i++) {
                c += __ldg(P.rank_tab + (size_t)(i * (P.L + 1) + s) * P.kw + k2[i]);
                s += P.lmin_tab[i * P.kw + k2[i]];
            }
            double v = 0.0;
            for (int e = S.src_off[q]; e < S.src_off[q + 1]; e++)
                v = fma(S.coef[S.src[e]], product_elem(P, S, S.src[e], k, k2, sum), v);
            const long long p = at + __popc(m & ((1u << lane) - 1u));
            cols[p] = c;
            vals[p] = Elem<T>::of(v);
        }
        at += __popc(m);
    }
}

// ---------------------------------------------------------------- apply

template <typename T, int W>
struct alignas(sizeof(T) * W > 16 ? 16 : sizeof(T) * W) Vec {
    T v[W];
};

// W adjacent values through the read-only path, in accesses of at most 16 bytes
template <typename T, int W>
__device__ __forceinline__ Vec<T, W> load_vec(const T *p)
{
    Vec<T, W> r;
    constexpr int B = (int)sizeof(T) * W;
    if constexpr (B == 4) {
        const unsigned t = __ldg(reinterpret_cast<const unsigned *>(p));
        memcpy(&r, &t, 4);
    } else if constexpr (B == 8) {
        const uint2 t = __ldg(reinterpret_cast<const uint2 *>(p));
        memcpy(&r, &t, 8);
    } else {
#pragma unroll
        for (int i = 0; i < B / 16; i++) {
            const uint4 t = __ldg(reinterpret_cast<const uint4 *>(p) + i);
            memcpy(reinterpret_cast<char *>(&r) + 16 * i, &t, 16);
        }
    }
    return r;
}

// Row sum of one vector in each precision.
template <typename T> struct Sum;
template <> struct Sum<double> {
    double s;
    __device__ __forceinline__ void zero() { s = 0.0; }
    __device__ __forceinline__ void add(double a, double x) { s = fma(a, x, s); }
    __device__ __forceinline__ double value() const { return s; }
};
template <> struct Sum<float> {
    float hi, lo;
    __device__ __forceinline__ void zero() { hi = lo = 0.0f; }
    __device__ __forceinline__ void add(float a, float x)
    {
        float s, e;
        dfops::two_sum(hi, dfops::mul(a, x), s, e);
        hi = s;
        lo = dfops::add(lo, e);
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
template <> struct Sum<df2> {
    df2 s;
    __device__ __forceinline__ void zero() { s = df2(0.0f, 0.0f); }
    __device__ __forceinline__ void add(df2 a, df2 x) { s = df_fma(a, x, s); }
    __device__ __forceinline__ double value() const { return s.to_double(); }
};

__device__ __forceinline__ void copy16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
}

__device__ __forceinline__ bool finite(double v)
{
    return (__double2hiint(v) & 0x7FF00000) != 0x7FF00000;
}

// Bytes of shared memory of a window block.
__host__ __device__ inline size_t rows_smem(int cap, int wrows, size_t rb)
{
    return (size_t)cap * (4 + rb) + (size_t)kTileV * wrows * 8;
}

// One window.  ST: values come from the entry-major copy io.xs (VT adjacent
// ones per lane); else from x itself, converted (VT = 1).
template <typename T, int VT, bool ST>
__device__ __forceinline__ void rows_window(const RowOp &R, const RowIO &io, int w, int lgl, unsigned char *smem)
{
    const int tid = threadIdx.x;
    const RowWin win = R.wins[w];
    double *tile = reinterpret_cast<double *>(smem);
    T *sv = reinterpret_cast<T *>(smem + (size_t)kTileV * R.wrows * 8);
    int *sc = reinterpret_cast<int *>(sv + R.cap);
    const T *gv = static_cast<const T *>(R.vals) + win.ent0;
    const int *gc = R.cols + win.ent0;
    const int lane = tid & ((1 << lgl) - 1), slot = tid >> lgl, nslot = kRT >> lgl;
    const int vpass = VT << lgl;  // vectors per pass, at most kTileV
    const int lw = 31 - __clz(R.wrows);
    const bool once = win.nent <= R.cap;

    auto stage = [&](int e0, int n) {  // entries [e0, e0 + n) into shared memory
        constexpr int UV = 16 / (int)sizeof(T);
        for (int i = tid; i < (n + 3) / 4; i += kRT) copy16(sc + 4 * i, gc + e0 + 4 * i);
        for (int i = tid; i < (n + UV - 1) / UV; i += kRT) copy16(sv + UV * i, gv + e0 + UV * i);
        copy_wait();
    };
    if (once) {
        stage(0, win.nent);
        __syncthreads();
    }
    for (int v0 = 0; v0 < io.nvec; v0 += vpass) {
        const int v = v0 + lane * VT;
        for (int it = 0; it * nslot < win.nrows; it++) {
            // every second round in reverse: long and short rows on each slot
            const int q = it * nslot + (it & 1 ? nslot - 1 - slot : slot);
            const bool on = q < win.nrows && v < io.nvec;
            uint2 mt = make_uint2(0u, 0u);
            if (on) mt = __ldg(R.meta + win.row0 + q);
            const int start = (int)(mt.x & 0xFFFFFFu), len = (int)mt.y;
            Sum<T> acc[VT];
#pragma unroll
            for (int u = 0; u < VT; u++) acc[u].zero();
            auto run = [&](const int *cp, const T *vp, int n) {
                constexpr int UN = 4;
                int e = 0;
                for (; e + UN <= n; e += UN) {
                    Vec<T, VT> xv[UN];
#pragma unroll
                    for (int b = 0; b < UN; b++) {
                        const size_t c = (size_t)cp[e + b];
                        if constexpr (ST) xv[b] = load_vec<T, VT>(static_cast<const T *>(io.xs) + c * io.stride + v);
                        else xv[b].v[0] = Elem<T>::of(__ldg(io.x + (size_t)v * R.n + c));
                    }
#pragma unroll
                    for (int b = 0; b < UN; b++) {
                        const T a = vp[e + b];
#pragma unroll
                        for (int u = 0; u < VT; u++) acc[u].add(a, xv[b].v[u]);
                    }
                }
                for (; e < n; e++) {
                    const size_t c = (size_t)cp[e];
                    Vec<T, VT> xv;
                    if constexpr (ST) xv = load_vec<T, VT>(static_cast<const T *>(io.xs) + c * io.stride + v);
                    else xv.v[0] = Elem<T>::of(__ldg(io.x + (size_t)v * R.n + c));
                    const T a = vp[e];
#pragma unroll
                    for (int u = 0; u < VT; u++) acc[u].add(a, xv.v[u]);
                }
            };
            if (once) {
                run(sc + start, sv + start, len);
            } else {
                // a single row longer than the staging area: piece by piece
                for (int e0 = 0; e0 < win.nent; e0 += R.cap) {
                    const int n = min(R.cap, win.nent - e0);
                    __syncthreads();
                    stage(e0, n);
                    __syncthreads();
                    if (on) run(sc, sv, n);
                }
            }
            if (on) {
                const int lr = (int)(mt.x >> 24);
#pragma unroll
                for (int u = 0; u < VT; u++)
                    if (lane * VT + u < kTileV) tile[((lane * VT + u) << lw) + lr] = acc[u].value();
            }
        }
        __syncthreads();
        // y = sum + harmonic diagonal, or the sums' bits into the accumulators
        const int nv = min(vpass, io.nvec - v0);
        for (int i = tid; i < nv << lw; i += kRT) {
            const int u = i >> lw, r = i & (R.wrows - 1);
            if (r >= win.nrows) continue;
            const double s = tile[i];
            const size_t row = (size_t)win.row0 + r;
            if (io.y) {
                const size_t g = (size_t)(v0 + u) * R.n + row;
                const double xi = __ldg(io.x + g);
                io.y[g] = fma(__ldg(R.esplit + row), xi, s);
                if (!finite(xi)) atomicOr(io.flags + v0 + u, 1u);
                if (!finite(xi) || !finite(s)) atomicCAS(R.err, 0, 201);
            } else {
                io.acc[(row * io.nvec + v0 + u) * io.words] += (unsigned long long)__double_as_longlong(s);
                if (!finite(s)) atomicCAS(R.err, 0, 201);
            }
        }
        __syncthreads();
    }
}

template <typename T, int VT, bool ST>
__global__ void __launch_bounds__(kRT) k_rows(const RowOp R, const RowIO io, int lgl)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int w = blockIdx.x * io.nparts + io.part;
    if (w >= R.nwin) return;
    rows_window<T, VT, ST>(R, io, w, lgl, smem);
}

// Many problems: vectors of problem j from nvec * cs_prefix[j], its rows of xs from cs_prefix[j], flags from j * nvec.
template <typename T, int VT>
__global__ void __launch_bounds__(kRT) k_rows_batch(const RowOp *__restrict__ ops, const int2 *__restrict__ items,
                                                    const RowIO io, int lgl, const long long *__restrict__ cs_prefix)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int2 it = items[blockIdx.x];
    const RowOp R = ops[it.x];
    RowIO o = io;
    const size_t c0 = (size_t)cs_prefix[it.x];
    o.x += c0 * io.nvec;
    o.y += c0 * io.nvec;
    o.xs = static_cast<const T *>(io.xs) + c0 * io.stride;
    o.flags += (size_t)it.x * io.nvec;
    rows_window<T, VT, true>(R, o, it.y, lgl, smem);
}

// xs[r * stride + v] = x_v[r] in T (zero beyond nvec), rows r0 .. r0 + nr - 1
template <typename T>
__device__ __forceinline__ void stage_row(const double *__restrict__ x, size_t n, int nvec, int stride,
                                          T *__restrict__ xs, size_t r)
{
    T *row = xs + r * stride;
    if (stride < 4) {
        for (int v = 0; v < stride; v++) row[v] = Elem<T>::of(__ldg(x + (size_t)v * n + r));
        return;
    }
    constexpr int U = 16 / (int)sizeof(T);
    for (int v0 = 0; v0 < stride; v0 += 4) {
        Vec<T, 4> t;
#pragma unroll
        for (int u = 0; u < 4; u++) t.v[u] = v0 + u < nvec ? Elem<T>::of(__ldg(x + (size_t)(v0 + u) * n + r)) : Elem<T>::of(0.0);
#pragma unroll
        for (int u = 0; u < 4; u += U)
            *reinterpret_cast<Vec<T, U> *>(row + v0 + u) = *reinterpret_cast<const Vec<T, U> *>(t.v + u);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_row_stage(const RowOp R, const RowIO io)
{
    T *xs = const_cast<T *>(static_cast<const T *>(io.xs));
    for (size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x; r < (size_t)R.n; r += (size_t)gridDim.x * blockDim.x)
        stage_row<T>(io.x, R.n, io.nvec, io.stride, xs, r);
}

template <typename T>
__global__ void __launch_bounds__(256) k_row_stage_batch(const int2 *__restrict__ items, const RowIO io,
                                                         const long long *__restrict__ cs_prefix)
{
    const int2 it = items[blockIdx.x];  // (problem, chunk of 256 rows)
    const size_t c0 = (size_t)cs_prefix[it.x], n = (size_t)cs_prefix[it.x + 1] - c0;
    const size_t r = (size_t)it.y * 256 + threadIdx.x;
    if (r < n)
        stage_row<T>(io.x + c0 * io.nvec, n, io.nvec, io.stride,
                     const_cast<T *>(static_cast<const T *>(io.xs)) + c0 * io.stride, r);
}

// A vector that holds a non-finite value gives NaN everywhere; clears the
// flags.  Block j: problem j (its vectors from nvec * cs_prefix[j]).
__global__ void __launch_bounds__(1024) k_row_settle(const RowIO io, int n_one, const long long *__restrict__ cs_prefix)
{
    const int j = blockIdx.x;
    const size_t c0 = cs_prefix ? (size_t)cs_prefix[j] : 0;
    const size_t n = cs_prefix ? (size_t)cs_prefix[j + 1] - c0 : (size_t)n_one;
    unsigned *flags = io.flags + (size_t)j * io.nvec;
    for (int v = 0; v < io.nvec; v++) {
        const bool bad = flags[v] != 0u;  // the same for the whole block: written by earlier launches only
        if (!bad) continue;
        double *y = io.y + (c0 * io.nvec + (size_t)v * n);
        for (size_t i = threadIdx.x; i < n; i += blockDim.x) y[i] = __longlong_as_double(0x7FF8000000000000ll);
    }
    __syncthreads();
    for (int v = threadIdx.x; v < io.nvec; v += blockDim.x)
        if (flags[v]) flags[v] = 0u;
}

// y = the double whose bits the parts summed to, plus the harmonic diagonal; clears the accumulators.
__global__ void __launch_bounds__(256) k_row_finish(const RowOp R, const RowIO io)
{
    const size_t total = (size_t)R.n * io.nvec;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t v = i / R.n, r = i - v * R.n;
        unsigned long long *a = io.acc + (r * io.nvec + v) * io.words;
        const double s = __longlong_as_double((long long)a[0]), xi = io.x[i];
        for (int q = 0; q < io.words; q++) a[q] = 0ull;
        io.y[i] = fma(R.esplit[r], xi, s);
        if (!finite(xi)) atomicOr(io.flags + v, 1u);
        if (!finite(xi) || !finite(s)) atomicCAS(R.err, 0, 201);
    }
}

// lanes per row (log2): as many as cover the vectors of a pass
int lanes_log2(int nvec, int vt)
{
    int l = 0;
    while ((vt << (l + 1)) <= kTileV && (vt << l) < nvec) l++;
    return l;
}
// vectors per lane: the plan's, within the row length of the copy
int fit_vt(int vt, int stride)
{
    while (vt > stride) vt >>= 1;
    return std::max(1, vt);
}

template <typename K>
cudaError_t smem_limit(K kernel)
{
    int dev = 0, optin = 0;
    cudaFuncAttributes fa{};
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}
template <typename T>
cudaError_t smem_limits()
{
    cudaError_t e = smem_limit(k_rows<T, 1, false>);
    if (e == cudaSuccess) e = smem_limit(k_rows<T, 1, true>);
    if (e == cudaSuccess) e = smem_limit(k_rows<T, 2, true>);
    if (e == cudaSuccess) e = smem_limit(k_rows<T, 4, true>);
    if (e == cudaSuccess) e = smem_limit(k_rows_batch<T, 1>);
    if (e == cudaSuccess) e = smem_limit(k_rows_batch<T, 2>);
    if (e == cudaSuccess) e = smem_limit(k_rows_batch<T, 4>);
    return e;
}

template <typename T>
cudaError_t rows_t(const RowOp &R, const RowIO &io, int vt, cudaStream_t s)
{
    const unsigned blocks = (unsigned)((R.nwin - io.part + io.nparts - 1) / io.nparts);
    if (R.nwin <= io.part) return cudaSuccess;
    const size_t smem = rows_smem(R.cap, R.wrows, sizeof(T));
    if (!io.xs) {
        k_rows<T, 1, false><<<blocks, kRT, smem, s>>>(R, io, lanes_log2(io.nvec, 1));
        return cudaGetLastError();
    }
    vt = fit_vt(vt, io.stride);
    const int l = lanes_log2(io.nvec, vt);
    if (vt == 4) k_rows<T, 4, true><<<blocks, kRT, smem, s>>>(R, io, l);
    else if (vt == 2) k_rows<T, 2, true><<<blocks, kRT, smem, s>>>(R, io, l);
    else k_rows<T, 1, true><<<blocks, kRT, smem, s>>>(R, io, l);
    return cudaGetLastError();
}

template <typename T>
cudaError_t rows_batch_t(const RowOp *ops, const int2 *items, int nitems, size_t smem, const RowIO &io, int vt,
                         const long long *cs_prefix, cudaStream_t s)
{
    vt = fit_vt(vt, io.stride);
    const int l = lanes_log2(io.nvec, vt);
    if (vt == 4) k_rows_batch<T, 4><<<(unsigned)nitems, kRT, smem, s>>>(ops, items, io, l, cs_prefix);
    else if (vt == 2) k_rows_batch<T, 2><<<(unsigned)nitems, kRT, smem, s>>>(ops, items, io, l, cs_prefix);
    else k_rows_batch<T, 1><<<(unsigned)nitems, kRT, smem, s>>>(ops, items, io, l, cs_prefix);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_row_count(const KParams &kp, const RowShifts &sh, int *cnt, cudaStream_t stream)
{
    k_row_count<<<(unsigned)(((size_t)kp.n_cs * 32 + 255) / 256), 256, 0, stream>>>(kp, sh, cnt);
    return cudaGetLastError();
}

cudaError_t launch_row_fill(const KParams &kp, const RowShifts &sh, sg_precision prec, const long long *start,
                            int *cols, void *vals, cudaStream_t stream)
{
    const unsigned blocks = (unsigned)(((size_t)kp.n_cs * 32 + 255) / 256);
    if (prec == SG_MIXED) k_row_fill<float><<<blocks, 256, 0, stream>>>(kp, sh, start, cols, static_cast<float *>(vals));
    else if (prec == SG_DF64) k_row_fill<df2><<<blocks, 256, 0, stream>>>(kp, sh, start, cols, static_cast<df2 *>(vals));
    else k_row_fill<double><<<blocks, 256, 0, stream>>>(kp, sh, start, cols, static_cast<double *>(vals));
    return cudaGetLastError();
}

// The limits are a property of the kernels, shared by every context: the most the device allows.
cudaError_t configure_rows()
{
    cudaError_t e = smem_limits<float>();
    if (e == cudaSuccess) e = smem_limits<double>();
    if (e == cudaSuccess) e = smem_limits<df2>();
    return e;
}

cudaError_t launch_rows(const RowOp &R, const RowIO &io, sg_precision prec, int vt, cudaStream_t stream)
{
    if (prec == SG_MIXED) return rows_t<float>(R, io, vt, stream);
    if (prec == SG_DF64) return rows_t<df2>(R, io, vt, stream);
    return rows_t<double>(R, io, vt, stream);
}

cudaError_t launch_rows_batch(const RowOp *ops, const int2 *items, int nitems, int cap, int wrows, const RowIO &io,
                              sg_precision prec, int vt, const long long *cs_prefix, cudaStream_t stream)
{
    if (nitems <= 0) return cudaSuccess;
    const size_t smem = rows_smem(cap, wrows, (size_t)row_value_bytes(prec));
    if (prec == SG_MIXED) return rows_batch_t<float>(ops, items, nitems, smem, io, vt, cs_prefix, stream);
    return rows_batch_t<double>(ops, items, nitems, smem, io, vt, cs_prefix, stream);
}

cudaError_t launch_row_stage(const RowOp &R, const RowIO &io, sg_precision prec, cudaStream_t stream)
{
    const unsigned blocks = (unsigned)std::max(1, std::min((R.n + 255) / 256, 152 * 16));
    if (prec == SG_MIXED) k_row_stage<float><<<blocks, 256, 0, stream>>>(R, io);
    else if (prec == SG_DF64) k_row_stage<df2><<<blocks, 256, 0, stream>>>(R, io);
    else k_row_stage<double><<<blocks, 256, 0, stream>>>(R, io);
    return cudaGetLastError();
}

cudaError_t launch_row_stage_batch(const RowIO &io, sg_precision prec, const long long *cs_prefix, const int2 *items,
                                   int nitems, cudaStream_t stream)
{
    if (nitems <= 0) return cudaSuccess;
    if (prec == SG_MIXED) k_row_stage_batch<float><<<(unsigned)nitems, 256, 0, stream>>>(items, io, cs_prefix);
    else k_row_stage_batch<double><<<(unsigned)nitems, 256, 0, stream>>>(items, io, cs_prefix);
    return cudaGetLastError();
}

cudaError_t launch_row_settle(const RowIO &io, int n, cudaStream_t stream)
{
    k_row_settle<<<1, 1024, 0, stream>>>(io, n, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_row_settle_batch(const RowIO &io, const long long *cs_prefix, int nprob, cudaStream_t stream)
{
    k_row_settle<<<(unsigned)nprob, 1024, 0, stream>>>(io, 0, cs_prefix);
    return cudaGetLastError();
}

cudaError_t launch_row_finish(const RowOp &R, const RowIO &io, cudaStream_t stream)
{
    const size_t total = (size_t)R.n * io.nvec;
    const unsigned blocks = (unsigned)std::max<size_t>(1, std::min<size_t>((total + 255) / 256, 152 * 16));
    k_row_finish<<<blocks, 256, 0, stream>>>(R, io);
    return cudaGetLastError();
}

}  // namespace sg
