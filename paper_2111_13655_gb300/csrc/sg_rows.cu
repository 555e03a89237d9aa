// Row form of H_S on the device (described in sg_internal.h): the kernels that
// form the row operator once per context, and those that apply it.
//
// One block applies one window of consecutive rows to all vectors:
//   1. the window's record (columns, elements) comes into shared memory by one
//      bulk copy, as it lies;
//   2. a group of lanes takes a row, each lane `VT` vectors: per entry one
//      load of VT adjacent values of the entry-major copy xs and VT
//      multiply-adds.  The rows of a window go by decreasing length, so the
//      rows of a warp have about the same number of entries;
//   3. the row sums go through a shared-memory tile, so that y (column after
//      column) is written, and x read for the harmonic diagonal, in runs of
//      consecutive rows.
// A row's entries are summed in column order by one lane whatever the plan,
// the number of vectors or the batch, so every entry point gives the same bits.
// Sums: FP64 by fma; mixed precision adds four products in FP32 (a product and
// three multiply-adds, each rounded) and these groups by two-sum into a pair of
// FP32 numbers, whose low part collects the errors in FP32: a row's error is
// that of its products and groups, 6.1 * 2^-24 of the sum of its terms' sizes
// however long it is; double-float as df_fma.
//
// What bounds the row kernel (D=12 L=9, 8 vectors): FP64 its pipe, 81% busy;
// mixed and double-float the latency of the gathers, with 33% and 44% of the
// issue slots and a quarter of the DRAM bandwidth used.  Against the kernel
// that took every term through its grid: D=12 L=10 mixed 26.5 ms -> 80.6 us,
// D=12 L=9 FP64 39.9 ms -> 90.5 us, D=12 L=8 double-float 4.36 ms -> 28.8 us.
#include <algorithm>
#include <cstring>

#include "sg_cheb.cuh"
#include "sg_df.cuh"
#include "sg_launch.cuh"

namespace sg {

namespace {

// Two warps per block: with a window of 64 rows every slot takes a long and a
// short row, and few warps wait for the longest one.  Against 128 threads:
// 32 batched wavepackets 63.6 -> 52.0 us, D=12 L=10 mixed and FP64 within 3%.
constexpr int kRT = 64;
constexpr int kTileV = 8;  // vectors per pass (the tile's columns)
constexpr int kOut = kTileV * kRowWindowMax / kRT;  // outputs per thread and pass
// Resident blocks per SM the kernels are compiled for (80 / 128 registers).
// Sixteen FP32 blocks spill: D=12 L=10 83 -> 102 us.  Twelve FP64 blocks cost
// D=12 L=9 3% but are worth it for batches, whose windows are few and wait on
// memory: 12 FP64 wavepackets 22.9 -> 20.9 us.
template <typename T> constexpr int row_blocks() { return sizeof(T) == 4 ? 12 : 8; }
constexpr int kBatchBlocks = 12;

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
// sum over |l_S| <= T of prod Delta M_i(l_i)[k_i][k'_i] over the factors of
// product q; the last factor's differences are summed in closed form
// (sum_{l <= t} Delta M(l) = M(t)).  A factor's element is zero below the level
// that holds both functions, so the sums run over the levels that remain above
// these, `room` (of T).
__device__ double product_elem(const KParams &P, const RowShifts &S, int q, const int *k, const int *k2, int sum)
{
    const int f0 = S.prod_off[q], f1 = S.prod_off[q + 1];
    if (f0 == f1) return 1.0;
    auto first = [&](int f) {  // of the levels that hold both functions of factor f
        const int m = S.fmode[f];
        return (int)P.lmin_tab[m * P.kw + max(k[m], k2[m])];
    };
    int T = P.L - sum, low = 0;
    for (int f = f0; f < f1; f++) {
        T += P.lmin_tab[S.fmode[f] * P.kw + k[S.fmode[f]]];
        low += first(f);
    }
    const int last = f1 - 1, ml = S.fmode[last], ol = S.fop[last], room = T - low;
    if (f1 - f0 == 1) return factor_elem(P, ml, ol, T, k[ml], k2[ml]);
    double a[kRowMaxL + 1], d[kRowMaxL + 1];  // by level above the first
    for (int f = f0; f < last; f++) {
        const int m = S.fmode[f], o = S.fop[f], l0 = first(f);
        double below = 0.0;
        for (int j = 0; j <= room; j++) {
            const double e = factor_elem(P, m, o, l0 + j, k[m], k2[m]);
            d[j] = e - below;
            below = e;
        }
        for (int t = room; t >= 0; t--) {
            if (f == f0) {
                a[t] = d[t];
                continue;
            }
            double v = 0.0;
            for (int j = 0; j <= t; j++) v = fma(a[t - j], d[j], v);
            a[t] = v;
        }
    }
    double v = 0.0;
    for (int j = 0; j <= room; j++)
        if (a[j] != 0.0) v = fma(a[j], factor_elem(P, ml, ol, first(last) + room - j, k[ml], k2[ml]), v);
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
template <> struct Elem<df2> { static __device__ df2 of(double v) { return df_split(v); } };

// The record's row list, and the shift of every entry in the place of its
// column (~shift for the zero elements that fill a row's last group of four).
__global__ void __launch_bounds__(256) k_row_place(const KParams P, const RowShifts S, const RowWin *__restrict__ wins,
                                                   const int *__restrict__ win, const int *__restrict__ start,
                                                   const uint2 *__restrict__ meta, unsigned char *__restrict__ blob)
{
    const int r = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (r >= P.n_cs) return;
    int k[kMaxD];
    const int sum = unrank(P, r, k);
    const RowWin w = wins[win[r]];
    unsigned char *rec = blob + w.off;
    if (lane == 0) reinterpret_cast<uint2 *>(rec)[r - w.row0] = meta[r];
    int *cols = reinterpret_cast<int *>(rec + row_meta_bytes(w.nrows));
    int at = start[r];
    for (int q0 = 0; q0 < S.nshift; q0 += 32) {
        const int q = q0 + lane;
        const bool in = q < S.nshift && shift_fits(P, S, q, k, sum);
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) cols[at + __popc(m & ((1u << lane) - 1u))] = q;
        at += __popc(m);
    }
    const int pad = (4 - ((at - start[r]) & 3)) & 3;
    __syncwarp();
    if (lane < pad) cols[at + lane] = ~cols[at - 1];
}

// Columns and elements, a thread per entry; a block takes kElemChunk entries of
// a window and finds their rows' multi-indices once.  Bound by the FP64 pipe for
// products of many modes (their levels' convolutions).  Set-up of 64 six-mode
// products over 3,003 functions, and of the benchmark's operator (D=12 L=10):
// one kernel with a warp per row, its lanes over the shifts, most of them idle
// since few shifts fit a row, and sums over all levels 275 ms (the kernel there
// 2.6 ms); sums over the levels that remain 64; lanes filled from a list of the
// shifts that fit 27; a thread per entry 11 (0.5 + 0.8 ms), of which 6 are the
// plan.  Chunks of 1,024 entries: 14 (0.5 + 0.6).
constexpr int kElemThreads = 128, kElemChunk = 128;
template <typename T>
__global__ void __launch_bounds__(kElemThreads) k_row_elems(const KParams P, const RowShifts S,
                                                            const RowWin *__restrict__ wins,
                                                            const int *__restrict__ start,
                                                            unsigned char *__restrict__ blob)
{
    __shared__ unsigned char index[kRowWindowMax][kMaxD];
    __shared__ int level[kRowWindowMax];
    const RowWin w = wins[blockIdx.x];
    int *cols = reinterpret_cast<int *>(blob + w.off + row_meta_bytes(w.nrows));
    T *vals = reinterpret_cast<T *>(cols + w.nent);
    auto row_of = [&](int e) {  // the last row of the window that starts at or before entry e
        int lo = 0, hi = w.nrows;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (start[w.row0 + mid] <= e) lo = mid;
            else hi = mid;
        }
        return lo;
    };
    for (int e0 = blockIdx.y * kElemChunk; e0 < w.nent; e0 += gridDim.y * kElemChunk) {
        const int e1 = min(w.nent, e0 + kElemChunk), r1 = row_of(e1 - 1);
        int k[kMaxD], k2[kMaxD];
        for (int r = row_of(e0) + threadIdx.x; r <= r1; r += kElemThreads) {
            level[r] = unrank(P, w.row0 + r, k);
            for (int i = 0; i < P.D; i++) index[r][i] = (unsigned char)k[i];
        }
        __syncthreads();
        for (int e = e0 + threadIdx.x; e < e1; e += kElemThreads) {
            const int r = row_of(e);
            const bool fill = cols[e] < 0;
            const int q = fill ? ~cols[e] : cols[e];
            for (int i = 0; i < P.D; i++) k2[i] = k[i] = index[r][i];
            for (int d = S.off[q]; d < S.off[q + 1]; d++) k2[S.mode[d]] += S.d[d];
            int c = 0, s = 0;
            for (int i = 0; i < P.D; i++) {
                c += __ldg(P.rank_tab + (size_t)(i * (P.L + 1) + s) * P.kw + k2[i]);
                s += P.lmin_tab[i * P.kw + k2[i]];
            }
            double v = 0.0;
            for (int d = S.src_off[q]; d < S.src_off[q + 1] && !fill; d++)
                v = fma(S.coef[S.src[d]], product_elem(P, S, S.src[d], k, k2, level[r]), v);
            cols[e] = c;
            vals[e] = Elem<T>::of(v);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- apply

template <typename T, int W>
struct alignas(sizeof(T) * W > 16 ? 16 : sizeof(T) * W) Vec {
    T v[W];
};

// W adjacent values in accesses of at most 16 bytes.  Ordinary loads, not the
// read-only path: the launch may have begun before its predecessor ended, and
// only what is loaded after the wait on it is up to date.
template <typename T, int W>
__device__ __forceinline__ Vec<T, W> load_vec(const T *p)
{
    Vec<T, W> r;
    constexpr int B = (int)sizeof(T) * W;
    if constexpr (B == 4) {
        const unsigned t = *reinterpret_cast<const unsigned *>(p);
        memcpy(&r, &t, 4);
    } else if constexpr (B == 8) {
        const uint2 t = *reinterpret_cast<const uint2 *>(p);
        memcpy(&r, &t, 8);
    } else {
#pragma unroll
        for (int i = 0; i < B / 16; i++) {
            const uint4 t = *(reinterpret_cast<const uint4 *>(p) + i);
            memcpy(reinterpret_cast<char *>(&r) + 16 * i, &t, 16);
        }
    }
    return r;
}

// Two adjacent values written by an earlier launch that this one may overlap (not the read-only path)
template <typename T>
__device__ __forceinline__ Vec<T, 2> load_pair(const T *p)
{
    Vec<T, 2> r;
    if constexpr (sizeof(T) == 4) {
        const uint2 t = __ldcg(reinterpret_cast<const uint2 *>(p));
        memcpy(&r, &t, 8);
    } else {
        const uint4 t = __ldcg(reinterpret_cast<const uint4 *>(p));
        memcpy(&r, &t, 16);
    }
    return r;
}

// Two FP32 numbers per instruction (IEEE rounding, as the scalar forms)
__device__ __forceinline__ uint64_t pack2(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// a - b as one multiply-add: -1 * b is exact
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { return fma2(b, 0xBF800000BF800000ull, a); }

// hi + lo of a pair of FP32 numbers as a double.  The FP64 pipe is narrow (1/64
// of the FP32 rate): the conversions are made with integer instructions; pairs
// with a subnormal, an infinity or a NaN go through the conversion instruction.
__device__ __forceinline__ double widen(unsigned u)
{
    const unsigned m = u << 1;  // exponent and mantissa
    const unsigned hi = m ? (m >> 4) + 0x38000000u : 0u;
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}
__device__ __forceinline__ bool plain(unsigned u)  // a zero or a normal number
{
    return (u << 1) - 0x01000000u < 0xFE000000u || (u << 1) == 0u;
}
__device__ __forceinline__ double convert(unsigned u)  // volatile: stays on its (rare) branch
{
    double d;
    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(__uint_as_float(u)));
    return d;
}
__device__ __forceinline__ double widen_pair(uint64_t t)
{
    const unsigned h = (unsigned)t, l = (unsigned)(t >> 32);
    double a = widen(h), b = widen(l);
    if (!plain(h) || !plain(l)) {
        a = convert(h);
        b = convert(l);
    }
    return a + b;
}

// Row sums of VT vectors.  add4: the next four entries, n of them real (the
// others are zero elements).
template <typename T, int VT> struct Sum;
template <int VT> struct Sum<double, VT> {
    double s[VT];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int u = 0; u < VT; u++) s[u] = 0.0;
    }
    __device__ __forceinline__ void add4(const double *a, const Vec<double, VT> *x, int n)
    {
#pragma unroll
        for (int b = 0; b < 4; b++) {
            if (b < n) {
#pragma unroll
                for (int u = 0; u < VT; u++) s[u] = fma(a[b], x[b].v[u], s[u]);
            }
        }
    }
    __device__ __forceinline__ uint64_t bits(int u) const { return (uint64_t)__double_as_longlong(s[u]); }
    static __device__ __forceinline__ double value(uint64_t t) { return __longlong_as_double((long long)t); }
};
// FP32 sums of four products, each added without error (two-sum) to a pair of
// FP32 numbers; two vectors per instruction.
template <int VT> struct Sum<float, VT> {
    static constexpr int NP = (VT + 1) / 2;
    uint64_t hi[NP], lo[NP];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int q = 0; q < NP; q++) hi[q] = lo[q] = 0ull;
    }
    __device__ __forceinline__ void add4(const float *a, const Vec<float, VT> *x, int)
    {
        uint64_t p[NP];
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const uint64_t ab = pack2(a[b], a[b]);
#pragma unroll
            for (int q = 0; q < NP; q++) {
                const uint64_t xb = pack2(x[b].v[2 * q], 2 * q + 1 < VT ? x[b].v[2 * q + 1 < VT ? 2 * q + 1 : 0] : 0.0f);
                p[q] = b == 0 ? mul2(ab, xb) : fma2(ab, xb, p[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < NP; q++) {
            const uint64_t s = add2(hi[q], p[q]);
            const uint64_t ap = sub2(s, p[q]), bp = sub2(s, ap);
            const uint64_t e = add2(sub2(hi[q], ap), sub2(p[q], bp));
            hi[q] = s;
            lo[q] = add2(lo[q], e);
        }
    }
    __device__ __forceinline__ uint64_t bits(int u) const
    {
        float h[2], l[2];
        unpack2(hi[u >> 1], h[0], h[1]);
        unpack2(lo[u >> 1], l[0], l[1]);
        return pack2(h[u & 1], l[u & 1]);
    }
    static __device__ __forceinline__ double value(uint64_t t) { return widen_pair(t); }
};
template <int VT> struct Sum<df2, VT> {
    df2 s[VT];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int u = 0; u < VT; u++) s[u] = df2(0.0f, 0.0f);
    }
    __device__ __forceinline__ void add4(const df2 *a, const Vec<df2, VT> *x, int n)
    {
#pragma unroll
        for (int b = 0; b < 4; b++) {
            if (b < n) {
#pragma unroll
                for (int u = 0; u < VT; u++) s[u] = df_fma(a[b], x[b].v[u], s[u]);
            }
        }
    }
    __device__ __forceinline__ uint64_t bits(int u) const { return pack2(s[u].hi, s[u].lo); }
    static __device__ __forceinline__ double value(uint64_t t) { return widen_pair(t); }
};

// Bulk copy of a record into shared memory, completing on an mbarrier.
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t *bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, unsigned bytes, uint64_t *bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
// Waits for phase `parity` of the barrier, a bounded number of polls (false: not reached).
constexpr int kBarPolls = 1 << 20;
__device__ __forceinline__ bool bar_wait(uint64_t *bar, unsigned parity)
{
    for (int q = 0; q < kBarPolls; q++) {
        unsigned done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done)
                     : "r"(smem_addr(bar)), "r"(parity)
                     : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ bool finite(double v)
{
    return (__double2hiint(v) & 0x7FF00000) != 0x7FF00000;
}

// Shared memory of a block: the window's record, and a tile of kTileV vectors by
// wrows rows for the sums on their way to y.
__host__ __device__ inline size_t rows_smem(int cap, int wrows)
{
    return (size_t)((cap + 15) & ~15) + (size_t)kTileV * wrows * 8;
}

// One window of problem R, whose vectors start at io.x, io.y, io.xs.  ST:
// values come from the entry-major copy io.xs (VT adjacent ones per lane);
// else from x itself, converted (VT = 1).  True in a thread that found a
// non-finite input value.
template <typename T, int VT, bool ST>
__device__ __forceinline__ bool rows_window(const RowOp &R, const RowIO &io, const RowWin &win, int lanes, int cap,
                                            unsigned char *smem, uint64_t *bar)
{
    const int tid = threadIdx.x, n = R.n;
    const int bytes = row_win_bytes(win, (int)sizeof(T));
    const bool staged = bytes <= cap;
    if (staged && tid == 0) {
        bar_init(bar);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        bulk_copy(smem, R.blob + win.off, (unsigned)bytes, bar);
    }
    // the thread's row of the tile, its first vector and its step over the vectors
    const int lw = 31 - __clz(R.wrows);
    const int tr = tid & (R.wrows - 1), tv = tid >> lw, tvs = kRT >> lw;
    const bool own = tr < win.nrows;
    const double es = own && io.y ? __ldg(R.esplit + win.row0 + tr) : 0.0;
    uint64_t *tile = reinterpret_cast<uint64_t *>(smem + ((cap + 15) & ~15));

    const unsigned char *rec = staged ? smem : R.blob + win.off;
    const uint2 *meta = reinterpret_cast<const uint2 *>(rec);
    const int *cols = reinterpret_cast<const int *>(rec + row_meta_bytes(win.nrows));
    const T *vals = reinterpret_cast<const T *>(cols + win.nent);
    const T *xs = static_cast<const T *>(io.xs);
    const int slot = tid / lanes, lane = tid - slot * lanes, nslot = kRT / lanes;  // slots from nslot on are idle
    const int vpass = VT * lanes;  // vectors per pass, at most kTileV
    __syncthreads();  // the barrier is initialised
    const bool late = staged && !bar_wait(bar, 0);
    // everything above reads the operator only; x, y and the flags belong to earlier launches until here
    grid_wait();
    if (__syncthreads_or(late)) {
        if (tid == 0) atomicCAS(R.err, 0, 120);
        bar_wait(bar, 0);
        return false;
    }
    bool odd = false;  // a non-finite value was found
    // (the passes of few windows go to blocks of their own: gridDim.y)
    for (int v0 = blockIdx.y * vpass; v0 < io.nvec; v0 += gridDim.y * vpass) {
        const int nv = min(vpass, io.nvec - v0);
        // x of the thread's outputs is on its way during the sums, unless these
        // take all registers (FP32, four vectors per lane; D=12 L=10, 8 vectors:
        // 88.8 us with the loads up front, 82.9 after the sums; one or two
        // vectors per lane: batches 46.2 and 46.6, FP64 91.7 and 92.7)
        const size_t g0 = (size_t)(v0 + tv) * n + win.row0 + tr, gs = (size_t)tvs * n;
        double xi[kOut];
        auto fetch = [&] {
#pragma unroll
            for (int q = 0; q < kOut; q++)
                if (io.y && own && tv + q * tvs < nv) xi[q] = io.x[g0 + q * gs];
        };
        constexpr bool early = !(sizeof(T) == 4 && VT == 4);
        if (early) fetch();
        const int v = v0 + lane * VT;
        for (int it = 0; it * nslot < win.nrows; it++) {
            // every second round in reverse: long and short rows on each slot
            const int q = it * nslot + (it & 1 ? nslot - 1 - slot : slot);
            if (slot >= nslot || q >= win.nrows || v >= io.nvec) continue;
            const uint2 mt = meta[q];
            Sum<T, VT> acc;
            acc.zero();
            // groups of four entries, the loads of two groups ahead of their sums
            auto load4 = [&](const int *cp, Vec<T, VT> *xv) {
                const int4 c = *reinterpret_cast<const int4 *>(cp);
                const int cc[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    if constexpr (ST) xv[u] = load_vec<T, VT>(xs + (size_t)cc[u] * io.stride + v);
                    else xv[u].v[0] = Elem<T>::of(io.x[(size_t)v * n + cc[u]]);
                }
            };
            auto sum4 = [&](const T *vp, const Vec<T, VT> *xv, int m) {
                const Vec<T, 4> a = *reinterpret_cast<const Vec<T, 4> *>(vp);
                acc.add4(a.v, xv, m);
            };
            const int *cp = cols + (mt.x & 0xFFFFFFu);
            const T *vp = vals + (mt.x & 0xFFFFFFu);
            const int m = (int)mt.y;
            int e = 0;
            for (; e + 4 < m; e += 8) {
                Vec<T, VT> x0[4], x1[4];
                load4(cp + e, x0);
                load4(cp + e + 4, x1);
                sum4(vp + e, x0, 4);
                sum4(vp + e + 4, x1, m - e - 4);
            }
            if (e < m) {
                Vec<T, VT> x0[4];
                load4(cp + e, x0);
                sum4(vp + e, x0, m - e);
            }
            uint64_t *t = tile + ((lane * VT) << lw) + (mt.x >> 24);
#pragma unroll
            for (int u = 0; u < VT; u++) t[u << lw] = acc.bits(u);
        }
        if (!early) fetch();
        __syncthreads();
        // y = sum + harmonic diagonal, or the sums' bits into the accumulators
        if (own) {
#pragma unroll
            for (int q = 0; q < kOut; q++) {
                const int u = tv + q * tvs;
                if (u >= nv) break;
                double s = Sum<T, VT>::value(tile[tid + q * kRT]);
                if (io.y) {
                    s = fma(es, xi[q], s);
                    io.y[g0 + q * gs] = s;
                    if (!finite(s) && !finite(xi[q])) {
                        atomicOr(io.flags + v0 + u, 1u);
                        odd = true;
                    }
                } else {
                    io.acc[((size_t)(win.row0 + tr) * io.nvec + v0 + u) * io.words] +=
                        (unsigned long long)__double_as_longlong(s);
                }
                if (!finite(s)) atomicCAS(R.err, 0, 201);
            }
        }
        if (v0 + (int)gridDim.y * vpass < io.nvec) __syncthreads();
    }
    return odd;
}

// A vector of n entries that holds a non-finite value gives NaN everywhere;
// clears its flag.  By a whole block.
__device__ __forceinline__ void settle_vectors(unsigned *flags, int nvec, double *y, size_t n)
{
    // the flags all at once: one after another their latencies made 5 us of a launch that finds none
    bool any = false;
    for (int v = threadIdx.x; v < nvec; v += blockDim.x) any |= __ldcg(flags + v) != 0u;
    if (!__syncthreads_or(any)) return;
    for (int v = 0; v < nvec; v++) {
        if (__ldcg(flags + v) == 0u) continue;
        for (size_t i = threadIdx.x; i < n; i += blockDim.x) y[(size_t)v * n + i] = __longlong_as_double(0x7FF8000000000000ll);
    }
    __syncthreads();
    for (int v = threadIdx.x; v < nvec; v += blockDim.x)
        if (__ldcg(flags + v)) flags[v] = 0u;
}

template <typename T, int VT, bool ST>
__global__ void __launch_bounds__(kRT, row_blocks<T>()) k_rows(const RowOp R, const RowIO io, int lanes)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t bar;
    grid_trigger();
    const bool odd =
        rows_window<T, VT, ST>(R, io, R.wins[blockIdx.x * io.nparts + io.part], lanes, R.cap, smem, &bar);
    if (!io.ticket) return;
    // the block that ends last settles the vectors (instead of a launch of its
    // own) if any block found one: the high half of the ticket counts those
    __shared__ unsigned tickets;
    const bool any = __syncthreads_or(odd);
    if (threadIdx.x == 0) {
        __threadfence();
        tickets = atomicAdd(io.ticket, any ? 0x10001u : 1u) + (any ? 0x10001u : 1u);
        if ((tickets & 0xFFFFu) == gridDim.x * gridDim.y) *io.ticket = 0u;
    }
    __syncthreads();
    if ((tickets & 0xFFFFu) != gridDim.x * gridDim.y || tickets < 0x10000u) return;
    __threadfence();
    settle_vectors(io.flags, io.nvec, io.y, (size_t)R.n);
}

// Many problems: item = (problem, window); vectors of problem j from
// nvec * cs_prefix[j], its rows of xs from cs_prefix[j], flags from j * nvec.
template <typename T, int VT, bool ST>
__global__ void __launch_bounds__(kRT, kBatchBlocks) k_rows_batch(const RowOp *__restrict__ ops,
                                                                const int2 *__restrict__ items, const RowIO io,
                                                                int lanes, const long long *__restrict__ cs_prefix,
                                                                int cap)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t bar;
    grid_trigger();
    const int2 it = items[blockIdx.x];
    const RowOp &R = ops[it.x];
    RowIO o = io;
    const size_t c0 = (size_t)cs_prefix[it.x];
    o.x += c0 * io.nvec;
    o.y += c0 * io.nvec;
    if (ST) o.xs = static_cast<const T *>(io.xs) + c0 * io.stride;
    o.flags += (size_t)it.x * io.nvec;
    rows_window<T, VT, ST>(R, o, R.wins[it.y], lanes, cap, smem, &bar);
}

// One Chebyshev term of a window: a thread takes a row, both vectors (the real
// and the imaginary part), and updates the row's entry where its sum ends.
// The record does not depend on the previous term: it is fetched while that
// term still runs.  term_of(done): the term, asked for after the wait.
template <typename T, typename F>
__device__ __forceinline__ void cheb_window(const RowOp &R, const ChebIO &io, const F &term_of, const RowWin &win,
                                            int cap, unsigned char *smem, uint64_t *bar)
{
    const int tid = threadIdx.x;
    const size_t n = (size_t)R.n;
    const int bytes = row_win_bytes(win, (int)sizeof(T));
    const bool staged = bytes <= cap;
    if (staged && tid == 0) {
        bar_init(bar);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        bulk_copy(smem, R.blob + win.off, (unsigned)bytes, bar);
    }
    __syncthreads();  // the barrier is initialised
    const bool late = staged && !bar_wait(bar, 0);
    grid_wait();
    if (__syncthreads_or(late)) {
        if (tid == 0) atomicCAS(R.err, 0, 120);
        bar_wait(bar, 0);
        return;
    }
    if (tid >= win.nrows) return;
    bool done = false;
    const ChebTerm term = term_of(done);
    const unsigned char *rec = staged ? smem : R.blob + win.off;
    const uint2 mt = reinterpret_cast<const uint2 *>(rec)[tid];
    const int *cols = reinterpret_cast<const int *>(rec + row_meta_bytes(win.nrows));
    const T *vals = reinterpret_cast<const T *>(cols + win.nent);
    const T *xs = static_cast<const T *>(io.xs);
    const size_t re = (size_t)win.row0 + (mt.x >> 24), im = re + n;
    // (state of an earlier launch that this one may overlap: read past the L1 cache)
    const double xr = __ldcg(io.X + re), xi = __ldcg(io.X + im);
    double pr = 0.0, pi = 0.0, ar = 0.0, ai = 0.0;
    if (!done && term.kn > 1) {
        pr = __ldcg(io.P + re);
        pi = __ldcg(io.P + im);
        ar = __ldcg(io.A + re);
        ai = __ldcg(io.A + im);
    }
    Sum<T, 2> acc;
    acc.zero();
    auto load4 = [&](const int *cp, Vec<T, 2> *xv) {
        const int4 c = *reinterpret_cast<const int4 *>(cp);
        const int cc[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int u = 0; u < 4; u++) xv[u] = load_pair<T>(xs + 2 * (size_t)cc[u]);
    };
    auto sum4 = [&](const T *vp, const Vec<T, 2> *xv, int m) {
        const Vec<T, 4> a = *reinterpret_cast<const Vec<T, 4> *>(vp);
        acc.add4(a.v, xv, m);
    };
    const int *cp = cols + (mt.x & 0xFFFFFFu);
    const T *vp = vals + (mt.x & 0xFFFFFFu);
    const int m = (int)mt.y;
    int e = 0;
    for (; e + 4 < m; e += 8) {
        Vec<T, 2> x0[4], x1[4];
        load4(cp + e, x0);
        load4(cp + e + 4, x1);
        sum4(vp + e, x0, 4);
        sum4(vp + e + 4, x1, m - e - 4);
    }
    if (e < m) {
        Vec<T, 2> x0[4];
        load4(cp + e, x0);
        sum4(vp + e, x0, m - e);
    }
    const double es = __ldg(R.esplit + re);
    const double yr = fma(es, xr, Sum<T, 2>::value(acc.bits(0))), yi = fma(es, xi, Sum<T, 2>::value(acc.bits(1)));
    if (!finite(yr) || !finite(yi)) {
        if (io.flags && (!finite(xr) || !finite(xi))) {  // one non-finite value makes both parts NaN at the end
            atomicOr(io.flags, 1u);
            atomicOr(io.flags + 1, 1u);
        }
        atomicCAS(R.err, 0, 201);
    }
    if (done) {  // past its last step: psi passes through
        pr = xr;
        pi = xi;
    } else {
        if (term.kn == 1 && io.Y) {
            io.Y[re] = yr;
            io.Y[im] = yi;
        }
        if (!cheb_entry(term, xr, xi, yr, yi, pr, pi, ar, ai)) {
            io.A[re] = ar;
            io.A[im] = ai;
        }
    }
    io.P[re] = pr;
    io.P[im] = pi;
    Vec<T, 2> o;
    o.v[0] = Elem<T>::of(pr);
    o.v[1] = Elem<T>::of(pi);
    *reinterpret_cast<Vec<T, 2> *>(static_cast<T *>(io.xs_next) + 2 * re) = o;
}

template <typename T>
__global__ void __launch_bounds__(kRT) k_cheb_rows(const RowOp R, const ChebIO io, const ChebTerm term)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t bar;
    grid_trigger();
    cheb_window<T>(R, io, [&](bool &) { return term; }, R.wins[blockIdx.x], R.cap, smem, &bar);
}

// Many problems: item = (problem, window); problem j's vectors from 2 * cs_prefix[j], its term from its state.
template <typename T>
__global__ void __launch_bounds__(kRT) k_cheb_rows_batch(const RowOp *__restrict__ ops,
                                                         const int2 *__restrict__ items, const ChebIO io,
                                                         const ChebState *st,
                                                         const long long *__restrict__ cs_prefix, int cap)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t bar;
    grid_trigger();
    const int2 it = items[blockIdx.x];
    const RowOp &R = ops[it.x];
    const size_t c0 = 2 * (size_t)cs_prefix[it.x];
    const ChebIO o{io.X + c0, io.Y + c0, io.P + c0, io.A + c0, static_cast<const T *>(io.xs) + c0,
                   static_cast<T *>(io.xs_next) + c0, nullptr};
    const ChebState *s = st + it.x;  // moved on by the launch before
    cheb_window<T>(
        R, o,
        [&](bool &done) {
            done = s->step >= s->nsteps;
            return done ? ChebTerm{} : cheb_term(*s);
        },
        R.wins[it.y], cap, smem, &bar);
}

// xs[r * stride + v] = x_v[r] in T (zero beyond nvec), rows r0 .. r0 + nr - 1
template <typename T>
__device__ __forceinline__ void stage_row(const double *x, size_t n, int nvec, int stride, T *xs, size_t r)
{
    T *row = xs + r * stride;
    if (stride < 4) {
        for (int v = 0; v < stride; v++) row[v] = Elem<T>::of(x[(size_t)v * n + r]);
        return;
    }
    constexpr int U = 16 / (int)sizeof(T);
    for (int v0 = 0; v0 < stride; v0 += 4) {
        Vec<T, 4> t;
#pragma unroll
        for (int u = 0; u < 4; u++) t.v[u] = v0 + u < nvec ? Elem<T>::of(x[(size_t)(v0 + u) * n + r]) : Elem<T>::of(0.0);
#pragma unroll
        for (int u = 0; u < 4; u += U)
            *reinterpret_cast<Vec<T, U> *>(row + v0 + u) = *reinterpret_cast<const Vec<T, U> *>(t.v + u);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_row_stage(const RowOp R, const RowIO io)
{
    grid_trigger();
    grid_wait();
    T *xs = const_cast<T *>(static_cast<const T *>(io.xs));
    for (size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x; r < (size_t)R.n; r += (size_t)gridDim.x * blockDim.x)
        stage_row<T>(io.x, R.n, io.nvec, io.stride, xs, r);
}

template <typename T>
__global__ void __launch_bounds__(256) k_row_stage_batch(const int2 *__restrict__ items, const RowIO io,
                                                         const long long *__restrict__ cs_prefix)
{
    grid_trigger();
    grid_wait();
    const int2 it = items[blockIdx.x];  // (problem, chunk of 256 rows)
    const size_t c0 = (size_t)cs_prefix[it.x], n = (size_t)cs_prefix[it.x + 1] - c0;
    const size_t r = (size_t)it.y * 256 + threadIdx.x;
    if (r < n)
        stage_row<T>(io.x + c0 * io.nvec, n, io.nvec, io.stride,
                     const_cast<T *>(static_cast<const T *>(io.xs)) + c0 * io.stride, r);
}

// Block j: problem j (its vectors from nvec * cs_prefix[j]).
__global__ void __launch_bounds__(1024) k_row_settle(const RowIO io, int n_one, const long long *__restrict__ cs_prefix)
{
    grid_wait();
    const int j = blockIdx.x;
    const size_t c0 = cs_prefix ? (size_t)cs_prefix[j] : 0;
    const size_t n = cs_prefix ? (size_t)cs_prefix[j + 1] - c0 : (size_t)n_one;
    settle_vectors(io.flags + (size_t)j * io.nvec, io.nvec, io.y + c0 * io.nvec, n);
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

// Lanes per row, of vt vectors each: the vectors are dealt out evenly over the
// fewest passes of at most kTileV.  An idle lane costs as much as a busy one, so
// the count is not rounded up to a power of two (D=12 L=9 FP64: 3, 5, 12 and 17
// vectors 52.5, 88.0, 166.9 and 249.4 us with powers of two, 45.8, 68.7, 144.9
// and 216.4 so; D=12 L=8 double-float, 5 vectors: 34.6 and 32.4).
int row_lanes(int nvec, int vt)
{
    const int need = (nvec + vt - 1) / vt, most = kTileV / vt, passes = (need + most - 1) / most;
    return (need + passes - 1) / passes;
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
    if constexpr (sizeof(T) == 8)
        if (e == cudaSuccess) e = smem_limit(k_rows_batch<T, 1, false>);
    if (e == cudaSuccess) e = smem_limit(k_rows_batch<T, 1, true>);
    if (e == cudaSuccess) e = smem_limit(k_rows_batch<T, 2, true>);
    if (e == cudaSuccess) e = smem_limit(k_rows_batch<T, 4, true>);
    if (e == cudaSuccess) e = smem_limit(k_cheb_rows<T>);
    if (e == cudaSuccess) e = smem_limit(k_cheb_rows_batch<T>);
    return e;
}

// Launched early: the blocks fetch their records, which nothing writes after
// set-up, while the preceding kernel runs (D=12 L=10, 5 vectors: 99.1 us with
// plain launches, 93.2 with these).
template <typename T>
cudaError_t rows_t(const RowOp &R, const RowIO &io, int vt, cudaStream_t s)
{
    if (R.nwin <= io.part) return cudaSuccess;
    const size_t smem = rows_smem(R.cap, R.wrows);
    const unsigned blocks = (unsigned)((R.nwin - io.part + io.nparts - 1) / io.nparts);
    vt = io.xs ? fit_vt(vt, io.stride) : 1;
    const int l = row_lanes(io.nvec, vt), vpass = vt * l;
    // several passes over the vectors: side by side while the windows are at
    // most two blocks per SM and leave SMs idle (D=2, 28 functions, 16 vectors:
    // 10.8 us one after another, 10.0 side by side, the rest is the call)
    const dim3 grid(blocks, blocks <= 304 ? std::min(16, (io.nvec + vpass - 1) / vpass) : 1);
    if (!io.xs) return launch_early(k_rows<T, 1, false>, grid, kRT, smem, s, R, io, l);
    if (vt == 4) return launch_early(k_rows<T, 4, true>, grid, kRT, smem, s, R, io, l);
    if (vt == 2) return launch_early(k_rows<T, 2, true>, grid, kRT, smem, s, R, io, l);
    return launch_early(k_rows<T, 1, true>, grid, kRT, smem, s, R, io, l);
}

template <typename T>
cudaError_t rows_batch_t(const RowOp *ops, const int2 *items, int nitems, int cap, int wrows, const RowIO &io, int vt,
                         const long long *cs_prefix, cudaStream_t s)
{
    const size_t smem = rows_smem(cap, wrows);
    const dim3 grid((unsigned)nitems);
    vt = io.xs ? fit_vt(vt, io.stride) : 1;
    const int l = row_lanes(io.nvec, vt);
    if constexpr (sizeof(T) == 8)
        if (!io.xs) return launch_early(k_rows_batch<T, 1, false>, grid, kRT, smem, s, ops, items, io, l, cs_prefix, cap);
    if (vt == 4) return launch_early(k_rows_batch<T, 4, true>, grid, kRT, smem, s, ops, items, io, l, cs_prefix, cap);
    if (vt == 2) return launch_early(k_rows_batch<T, 2, true>, grid, kRT, smem, s, ops, items, io, l, cs_prefix, cap);
    return launch_early(k_rows_batch<T, 1, true>, grid, kRT, smem, s, ops, items, io, l, cs_prefix, cap);
}

}  // namespace

cudaError_t launch_row_count(const KParams &kp, const RowShifts &sh, int *cnt, cudaStream_t stream)
{
    k_row_count<<<(unsigned)(((size_t)kp.n_cs * 32 + 255) / 256), 256, 0, stream>>>(kp, sh, cnt);
    return cudaGetLastError();
}

cudaError_t launch_row_fill(const KParams &kp, const RowShifts &sh, sg_precision prec, const RowWin *wins, int nwin,
                            int most, const int *win, const int *start, const uint2 *meta, unsigned char *blob,
                            cudaStream_t stream)
{
    k_row_place<<<(unsigned)(((size_t)kp.n_cs * 32 + 255) / 256), 256, 0, stream>>>(kp, sh, wins, win, start, meta, blob);
    const dim3 grid((unsigned)nwin, (unsigned)std::max(1, std::min(512, (most + kElemChunk - 1) / kElemChunk)));
    if (prec == SG_MIXED) k_row_elems<float><<<grid, kElemThreads, 0, stream>>>(kp, sh, wins, start, blob);
    else if (prec == SG_DF64) k_row_elems<df2><<<grid, kElemThreads, 0, stream>>>(kp, sh, wins, start, blob);
    else k_row_elems<double><<<grid, kElemThreads, 0, stream>>>(kp, sh, wins, start, blob);
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
    if (prec == SG_MIXED) return rows_batch_t<float>(ops, items, nitems, cap, wrows, io, vt, cs_prefix, stream);
    return rows_batch_t<double>(ops, items, nitems, cap, wrows, io, vt, cs_prefix, stream);
}

namespace {

template <typename T>
cudaError_t cheb_rows_t(const RowOp &R, const ChebIO &io, const ChebTerm &term, cudaStream_t s)
{
    if (R.nwin <= 0) return cudaSuccess;
    return launch_early(k_cheb_rows<T>, dim3((unsigned)R.nwin), kRT, (size_t)((R.cap + 15) & ~15), s, R, io, term);
}

}  // namespace

cudaError_t launch_cheb_rows(const RowOp &R, const ChebIO &io, const ChebTerm &one, sg_precision prec,
                             cudaStream_t stream)
{
    if (prec == SG_MIXED) return cheb_rows_t<float>(R, io, one, stream);
    if (prec == SG_DF64) return cheb_rows_t<df2>(R, io, one, stream);
    return cheb_rows_t<double>(R, io, one, stream);
}

cudaError_t launch_cheb_rows_batch(const RowOp *ops, const int2 *items, int nitems, int cap, const ChebIO &io,
                                   const ChebState *st, sg_precision prec, const long long *cs_prefix,
                                   cudaStream_t stream)
{
    if (nitems <= 0) return cudaSuccess;
    const size_t smem = (size_t)((cap + 15) & ~15);
    if (prec == SG_MIXED)
        return launch_early(k_cheb_rows_batch<float>, dim3((unsigned)nitems), kRT, smem, stream, ops, items, io, st,
                            cs_prefix, cap);
    return launch_early(k_cheb_rows_batch<double>, dim3((unsigned)nitems), kRT, smem, stream, ops, items, io, st,
                        cs_prefix, cap);
}

cudaError_t launch_row_stage(const RowOp &R, const RowIO &io, sg_precision prec, cudaStream_t stream)
{
    const unsigned blocks = (unsigned)std::max(1, std::min((R.n + 255) / 256, 152 * 16));
    if (prec == SG_MIXED) return launch_early(k_row_stage<float>, dim3(blocks), 256, 0, stream, R, io);
    if (prec == SG_DF64) return launch_early(k_row_stage<df2>, dim3(blocks), 256, 0, stream, R, io);
    return launch_early(k_row_stage<double>, dim3(blocks), 256, 0, stream, R, io);
}

cudaError_t launch_row_stage_batch(const RowIO &io, sg_precision prec, const long long *cs_prefix, const int2 *items,
                                   int nitems, cudaStream_t stream)
{
    if (nitems <= 0) return cudaSuccess;
    const dim3 grid((unsigned)nitems);
    if (prec == SG_MIXED) return launch_early(k_row_stage_batch<float>, grid, 256, 0, stream, items, io, cs_prefix);
    return launch_early(k_row_stage_batch<double>, grid, 256, 0, stream, items, io, cs_prefix);
}

cudaError_t launch_row_settle(const RowIO &io, int n, cudaStream_t stream)
{
    return launch_early(k_row_settle, dim3(1), 1024, 0, stream, io, n, nullptr);
}

cudaError_t launch_row_settle_batch(const RowIO &io, const long long *cs_prefix, int nprob, cudaStream_t stream)
{
    return launch_early(k_row_settle, dim3((unsigned)nprob), 1024, 0, stream, io, 0, cs_prefix);
}

cudaError_t launch_row_finish(const RowOp &R, const RowIO &io, cudaStream_t stream)
{
    const size_t total = (size_t)R.n * io.nvec;
    const unsigned blocks = (unsigned)std::max<size_t>(1, std::min<size_t>((total + 255) / 256, 152 * 16));
    k_row_finish<<<blocks, 256, 0, stream>>>(R, io);
    return cudaGetLastError();
}

}  // namespace sg
