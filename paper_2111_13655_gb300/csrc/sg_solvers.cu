// Solvers around the Smolyak action (Sec. 3, last paragraph: the Davidson
// method for stationary states, the Chebyshev method for wave-packet
// propagation): block Lanczos and block Davidson eigensolvers, Chebyshev
// propagation.  Recurrence vectors, inner products and orthogonalisation are
// FP64 on the device; the small projected problems are solved on the host.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "sg_internal.h"
#include "sg_launch.cuh"

namespace sg {

namespace {

constexpr int kMaxCols = 8;    // columns of B (block size) per call

// One block per inner product and chunk, one column per block of 64 entries:
// the products go to as many SMs as there are, since the narrow FP64 pipe (1/64
// of the FP32 rate) sets the time and sharing loads between products saves
// none of it.  Blocks that made 8 x 8 products over 304 chunks reduced 64 sums
// each through that pipe, and the 304 partial sums one after another: six
// Davidson pairs at n = 12,870 22.2 ms, now 4.0; eight at n = 646,646 85.9 and
// 40.9, and two propagation steps there 55.5 and 10.2 ms (most of it bounds).
// A product of n = 646,646 in one block instead of 40: 78.6 and 38.6 ms.
constexpr int64_t kChunk = 16384;  // entries per block; a product of more is summed in chunk order
constexpr int kMaxChunks = 64;
int chunks(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>(kMaxChunks, (n + kChunk - 1) / kChunk)); }
constexpr int kDotThreads = 256;

// Sum over the block, in a fixed order, to every thread.  The last step is made
// by one warp: the FP64 pipe serves one warp instruction in about 19 cycles, and
// letting every thread add the warps' sums took 10 us of a 1,024-thread block.
template <int THREADS>
__device__ __forceinline__ double block_sum(double v)
{
    constexpr int NW = THREADS / 32;
    __shared__ double red[NW];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double t = threadIdx.x < NW ? red[threadIdx.x] : 0.0;
        for (int o = NW / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) red[0] = t;
    }
    __syncthreads();
    return red[0];
}

// C[z][i][j] = sum over chunk z of A_i[e] B_j[e], block (i, j, z)
__global__ void __launch_bounds__(kDotThreads) k_gram(const double *A, const double *B, int n, int chunk, double *C)
{
    grid_trigger();
    grid_wait();
    const size_t e0 = (size_t)blockIdx.z * chunk;
    const double *a = A + (size_t)blockIdx.x * n + e0, *b = B + (size_t)blockIdx.y * n + e0;
    const int len = min(chunk, n - (int)e0);
    double v = 0.0;
#pragma unroll 8
    for (int e = threadIdx.x; e < len; e += kDotThreads) v = fma(a[e], b[e], v);
    v = block_sum<kDotThreads>(v);
    if (threadIdx.x == 0) C[((size_t)blockIdx.z * gridDim.x + blockIdx.x) * gridDim.y + blockIdx.y] = v;
}
// C[q] = sum_z partial[z][q], in chunk order
__global__ void __launch_bounds__(64) k_sum_chunks(const double *partial, int nchunk, int count, double *C)
{
    grid_trigger();
    grid_wait();
    const int q = blockIdx.x * 64 + threadIdx.x;
    if (q >= count) return;
    double v = 0.0;
#pragma unroll 16
    for (int z = 0; z < nchunk; z++) v += partial[(size_t)z * count + q];
    C[q] = v;
}

// sum_i V[i][e] s[i * stride] of the block's 64 columns e: G groups of threads
// take every G-th i, and their sums are added in order.  Four groups shorten the
// chain of loads while columns are few; many columns hide it, and one group
// saves the FP64 pipe the additions.  n = 3,003 propagation 1,918 us with one,
// 1,783 with four; n = 1,001 pairs 6,231 and 5,722; n = 50,388 5.87 and 5.78 ms;
// n = 125,970 9.9 and 10.5; n = 646,646 40.9 and 47.4.
constexpr int kColumns = 64;
constexpr int64_t kGroupedN = 65536;
template <int G>
__device__ __forceinline__ double column_sum(const double *V, int k, const double *s, int stride, unsigned e, unsigned n)
{
    double v = 0.0;
    if constexpr (G == 1) {
        if (e < n) {
#pragma unroll 16
            for (int i = 0; i < k; i++) v = fma(V[(size_t)i * n + e], s[i * stride], v);
        }
        return v;
    } else {
        __shared__ double part[G][kColumns];
        const int g = threadIdx.x / kColumns, c = threadIdx.x % kColumns;
        if (e < n) {
#pragma unroll 8
            for (int i = g; i < k; i += G) v = fma(V[(size_t)i * n + e], s[i * stride], v);
        }
        part[g][c] = v;
        __syncthreads();
        double t = part[0][c];
        for (int q = 1; q < G; q++) t += part[q][c];
        return t;
    }
}

// out[j][e] = base[j][e] + alpha * sum_i V[i][e] S[i][j] (base nullptr: 0), column j = blockIdx.y
template <int G>
__global__ void __launch_bounds__(kColumns * G) k_combine(const double *V, int k, const double *S, int r,
                                                                double alpha, const double *base, double *out,
                                                                unsigned n)
{
    grid_trigger();
    grid_wait();
    const unsigned e = blockIdx.x * kColumns + threadIdx.x % kColumns, j = blockIdx.y;
    const size_t o = (size_t)j * n + e;
    const bool own = threadIdx.x < kColumns && e < n;
    const double acc = column_sum<G>(V, k, S + j, r, e, n);
    if (own) out[o] = (base ? base[o] : 0.0) + alpha * acc;
}

// x <- (x - sum_i V_i c_i) / norm, norm^2 = c_k - sum_i c_i^2 (V orthonormal, c_i = V_i . x, c_k = x . x); x <- 0 when
// norm^2 <= 1e-24.  *nn = norm^2.
template <int G>
__global__ void __launch_bounds__(kColumns * G) k_project_normalise(const double *V, int k, const double *c,
                                                                          double *x, unsigned n, double *nn)
{
    grid_trigger();
    grid_wait();
    __shared__ double scale;
    if (threadIdx.x >= kColumns * G - 32) {
        double q = 0.0;
        for (int i = threadIdx.x % 32; i < k; i += 32) q = fma(c[i], c[i], q);
        for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        if (threadIdx.x % 32 == 0) {
            const double v = c[k] - q;
            scale = v > 1e-24 ? rsqrt(v) : 0.0;
            if (blockIdx.x == 0) *nn = v;
        }
    }
    const unsigned e = blockIdx.x * kColumns + threadIdx.x % kColumns;
    const bool own = threadIdx.x < kColumns && e < n;
    const double acc = column_sum<G>(V, k, c, 1, e, n);
    __syncthreads();  // scale
    if (own) x[e] = (x[e] - acc) * scale;
}

// Cholesky G = R^T R (b x b, row-major, b <= kMaxChol) to Ri = R^{-1}; columns
// after the first dependent one are zero, *rank the leading independent ones.
// A column is dependent when what the earlier ones leave of its squared norm is
// rounding: below 1e-13 of it (a Gram matrix resolves no more), or 1e-24.
constexpr int kMaxChol = 16;
constexpr double kDependent = 1e-13;
__global__ void __launch_bounds__(32) k_chol_inverse(const double *G, int b, double *Ri, int *rank)
{
    grid_trigger();
    grid_wait();
    __shared__ double R[kMaxChol][kMaxChol + 1], I[kMaxChol][kMaxChol + 1];
    const int i = threadIdx.x;
    for (int q = i; q < b * b; q += 32) { R[q / b][q % b] = 0.0; I[q / b][q % b] = 0.0; }
    __syncwarp();
    int rk = b;
    for (int j = 0; j < b; j++) {
        double v = 0.0;  // lane i >= j: entry (j, i) before the division
        if (i >= j && i < b) {
            v = G[j * b + i];
            for (int k = 0; k < j; k++) v = fma(-R[k][j], R[k][i], v);
        }
        const double d = __shfl_sync(0xffffffffu, v, j);
        if (!(d > fmax(1e-24, kDependent * G[j * b + j]))) { rk = j; break; }
        const double s = rsqrt(d);  // R[j][j] holds its reciprocal
        if (i == j) R[j][j] = s;
        else if (i > j && i < b) R[j][i] = v * s;
        __syncwarp();
    }
    // column i of the inverse of the leading rk x rk block
    if (i < rk) {
        I[i][i] = R[i][i];
        for (int r = i - 1; r >= 0; r--) {
            double v = 0.0;
            for (int k = r + 1; k <= i; k++) v = fma(R[r][k], I[k][i], v);
            I[r][i] = -v * R[r][r];
        }
    }
    __syncwarp();
    for (int q = i; q < b * b; q += 32) Ri[q] = I[q / b][q % b];
    if (i == 0) *rank = rk;
}

// Residuals: HX_j -= theta_j X_j, and their squared norms (partial[chunk][j], chunk = blockIdx.x)
__global__ void __launch_bounds__(256) k_residual(const double *X, const double *theta, double *HX, int64_t n,
                                                  int64_t chunk, double *partial)
{
    grid_trigger();
    grid_wait();
    const int j = blockIdx.y;
    const int64_t e0 = blockIdx.x * chunk, e1 = min(n, e0 + chunk);
    const double *x = X + (size_t)j * n;
    double *h = HX + (size_t)j * n;
    const double th = theta[j];
    double v = 0.0;
    for (int64_t e = e0 + threadIdx.x; e < e1; e += 256) {
        const double r = fma(-th, x[e], h[e]);
        h[e] = r;
        v = fma(r, r, v);
    }
    v = block_sum<256>(v);
    if (threadIdx.x == 0) partial[blockIdx.x * gridDim.y + j] = v;
}

// Directions: T_q = R_p / (d - theta_q) (guarded), or T_q = R_p without d; sel[2q] = p, sel[2q + 1] = theta_q
__global__ void __launch_bounds__(256) k_direction(const double *R, const double *d, const double *sel, int64_t n,
                                                   double *T)
{
    grid_trigger();
    grid_wait();
    const int q = blockIdx.y;
    const double *r = R + (size_t)sel[2 * q] * n;
    const double theta = sel[2 * q + 1];
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        double v = r[e];
        if (d) {
            const double den = d[e] - theta;
            v /= (fabs(den) < 1e-3 ? (den < 0 ? -1e-3 : 1e-3) : den);
        }
        T[(size_t)q * n + e] = v;
    }
}

// X_j = the unit vector of entry at[j]
__global__ void k_unit_vectors(double *__restrict__ X, int64_t n, const double *__restrict__ at, int r)
{
    const int64_t total = n * r;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = q / n;
        X[q] = q - j * n == (int64_t)at[j] ? 1.0 : 0.0;
    }
}

// x <- x / ||x|| by one block (0 when ||x||^2 <= 1e-24), the squared norm in *nn
__global__ void __launch_bounds__(1024) k_normalise(double *x, int64_t n, double *nn)
{
    grid_trigger();
    grid_wait();
    double v = 0.0;
    for (int64_t e = threadIdx.x; e < n; e += 1024) v = fma(x[e], x[e], v);
    v = block_sum<1024>(v);
    __shared__ double f;
    if (threadIdx.x == 0) f = v > 1e-24 ? 1.0 / sqrt(v) : 0.0;
    __syncthreads();
    for (int64_t e = threadIdx.x; e < n; e += 1024) x[e] *= f;
    if (threadIdx.x == 0) *nn = v;
}
// the same for longer vectors, from the squared norm
__global__ void __launch_bounds__(256) k_scale_norm(double *x, int64_t n, const double *xx, double *nn)
{
    const double v = *xx, f = v > 1e-24 ? 1.0 / sqrt(v) : 0.0;
    if (blockIdx.x == 0 && threadIdx.x == 0) *nn = v;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) x[e] *= f;
}

// y[j] = a * x[j] + b * y[j] over several vectors laid out contiguously
__global__ void k_axpby(int64_t len, double a, const double *__restrict__ x, double b, double *__restrict__ y)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < len; e += (int64_t)gridDim.x * blockDim.x)
        y[e] = a * x[e] + (b == 0.0 ? 0.0 : b * y[e]);
}

}  // namespace

// ---------------------------------------------------------------- device helpers
// C (ka x kb, row-major, device) = A^T B for column vectors A (ka x n), B (kb x n), kb <= kMaxCols.
// partial: gram_partial_doubles(n, ka) doubles of device scratch.  Deterministic.
cudaError_t dev_gram(const double *A, int ka, const double *B, int kb, int64_t n, double *C_dev,
                     double *partial, cudaStream_t s)
{
    if (kb > kMaxCols || kb < 1 || ka < 1) return cudaErrorInvalidValue;
    const int nz = chunks(n);
    cudaError_t e = launch_early(k_gram, dim3(ka, kb, nz), kDotThreads, 0, s, A, B, (int)n, (int)((n + nz - 1) / nz),
                                 nz == 1 ? C_dev : partial);
    if (e == cudaSuccess && nz > 1)
        e = launch_early(k_sum_chunks, dim3((ka * kb + 63) / 64), 64, 0, s, (const double *)partial, nz, ka * kb, C_dev);
    return e;
}

size_t gram_partial_doubles(int64_t n, int ka) { return (size_t)chunks(n) * ka * kMaxCols; }

// out (r x n) = base (r x n, or nullptr: zero; may be out) + alpha * V (k x n)^T-combination with S (k x r, device)
cudaError_t dev_combine(const double *V, int k, const double *S_dev, int r, double alpha, const double *base,
                        double *out, int64_t n, cudaStream_t s)
{
    if (r > kMaxCols || r < 1 || k < 1) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)((n + kColumns - 1) / kColumns), r);
    if (n <= kGroupedN)
        return launch_early(k_combine<4>, grid, kColumns * 4, 0, s, V, k, S_dev, r, alpha, base, out, (unsigned)n);
    return launch_early(k_combine<1>, grid, kColumns, 0, s, V, k, S_dev, r, alpha, base, out, (unsigned)n);
}

cudaError_t dev_chol_inverse(const double *G, int b, double *Ri, int *rank, cudaStream_t s)
{
    if (b < 1 || b > kMaxChol) return cudaErrorInvalidValue;
    return launch_early(k_chol_inverse, dim3(1), 32, 0, s, G, b, Ri, rank);
}

// HX_j -= theta_j X_j; norms2[j] = ||HX_j||^2 (device or pinned host).  partial: a double per row and chunk.
cudaError_t dev_residual(const double *X, const double *theta, double *HX, int rows, int64_t n, double *norms2,
                         double *partial, cudaStream_t s)
{
    if (rows < 1) return cudaErrorInvalidValue;
    const int nz = chunks(n);
    const int64_t chunk = (n + nz - 1) / nz;
    cudaError_t e =
        launch_early(k_residual, dim3(nz, rows), 256, 0, s, X, theta, HX, n, chunk, nz == 1 ? norms2 : partial);
    if (e == cudaSuccess && nz > 1)
        e = launch_early(k_sum_chunks, dim3((rows + 63) / 64), 64, 0, s, (const double *)partial, nz, rows, norms2);
    return e;
}

cudaError_t dev_direction(const double *R, const double *d, const double *sel, int rows, int64_t n, double *T,
                          cudaStream_t s)
{
    const unsigned bx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(608, (n + 255) / 256));
    return launch_early(k_direction, dim3(bx, rows), 256, 0, s, R, d, sel, n, T);
}

cudaError_t dev_unit_vectors(double *X, int64_t n, const double *at, int r, cudaStream_t s)
{
    const unsigned bx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(1216, (n * r + 255) / 256));
    k_unit_vectors<<<bx, 256, 0, s>>>(X, n, at, r);
    return cudaGetLastError();
}

// x <- x / ||x|| (zero when ||x||^2 <= 1e-24); nn: the squared norm (device)
cudaError_t dev_normalise(double *x, int64_t n, double *nn, double *partial, cudaStream_t s)
{
    if (chunks(n) == 1) return launch_early(k_normalise, dim3(1), 1024, 0, s, x, n, nn);
    double *xx = partial + gram_partial_doubles(n, 1);
    cudaError_t e = dev_gram(x, 1, x, 1, n, xx, partial, s);
    if (e != cudaSuccess) return e;
    k_scale_norm<<<608, 256, 0, s>>>(x, n, xx, nn);
    return cudaGetLastError();
}

// x <- (x - sum_{i<k} V_i c_i) / its norm, with c_i = V_i . x and c_k = x . x (device); nn: the squared norm
cudaError_t dev_project_normalise(const double *V, int k, const double *c, double *x, int64_t n, double *nn,
                                  cudaStream_t s)
{
    const dim3 grid((unsigned)((n + kColumns - 1) / kColumns));
    if (n <= kGroupedN)
        return launch_early(k_project_normalise<4>, grid, kColumns * 4, 0, s, V, k, c, x, (unsigned)n, nn);
    return launch_early(k_project_normalise<1>, grid, kColumns, 0, s, V, k, c, x, (unsigned)n, nn);
}

cudaError_t dev_axpby(int64_t len, double a, const double *x, double b, double *y, cudaStream_t s)
{
    k_axpby<<<608, 256, 0, s>>>(len, a, x, b, y);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- host dense algebra
// Symmetric eigenproblem: Householder reduction to tridiagonal form, then
// implicit QR steps with the Wilkinson shift (Golub & Van Loan, Matrix
// Computations, 8.3).  A: n x n, row-major; eigenvalues ascending in w,
// eigenvectors as columns of Z (row-major n x n).
void sym_eig(int n, std::vector<double> A, std::vector<double> &w, std::vector<double> &Z)
{
    std::vector<double> d(n), e(n, 0.0), p(n);
    std::vector<double> Q((size_t)n * n, 0.0);  // row i: the i-th column of the orthogonal factor
    auto a = [&](int i, int j) -> double & { return A[(size_t)i * n + j]; };
    std::vector<std::vector<double>> refl(n > 2 ? n - 2 : 0);
    for (int k = 0; k + 2 < n; k++) {
        // reflector v (unit) that takes column k below the diagonal to alpha e_1
        std::vector<double> &v = refl[k];
        v.assign(n - k - 1, 0.0);
        double nrm = 0.0;
        for (int i = k + 1; i < n; i++) { v[i - k - 1] = a(i, k); nrm = std::hypot(nrm, a(i, k)); }
        const double alpha = v[0] > 0.0 ? -nrm : nrm;
        e[k] = alpha;
        v[0] -= alpha;
        double vn = 0.0;
        for (double t : v) vn = std::hypot(vn, t);
        if (vn == 0.0) { v.clear(); continue; }
        for (double &t : v) t /= vn;
        // trailing block B <- B - 2 v q^T - 2 q v^T, q = B v - (v^T B v) v
        const int m = n - k - 1, o = k + 1;
        double vbv = 0.0;
        for (int i = 0; i < m; i++) {
            double t = 0.0;
            for (int j = 0; j < m; j++) t += a(o + i, o + j) * v[j];
            p[i] = t;
            vbv += v[i] * t;
        }
        for (int i = 0; i < m; i++) p[i] -= vbv * v[i];
        for (int i = 0; i < m; i++)
            for (int j = 0; j < m; j++) a(o + i, o + j) -= 2.0 * (v[i] * p[j] + p[i] * v[j]);
    }
    for (int i = 0; i < n; i++) { d[i] = a(i, i); Q[(size_t)i * n + i] = 1.0; }
    if (n > 1) e[n - 2] = a(n - 1, n - 2);
    // Q = H_0 H_1 ... : applied to the columns (rows of the array) from the last reflector on
    for (int k = n - 3; k >= 0; k--) {
        const std::vector<double> &v = refl[k];
        if (v.empty()) continue;
        const int o = k + 1, m = n - o;
        for (int c = 0; c < n; c++) {
            double *q = &Q[(size_t)c * n + o], t = 0.0;
            for (int i = 0; i < m; i++) t += v[i] * q[i];
            for (int i = 0; i < m; i++) q[i] -= 2.0 * t * v[i];
        }
    }
    // implicit QR on the unreduced block that ends at hi
    const double eps = 2.220446049250313e-16;
    int hi = n - 1, steps = 0;
    while (hi > 0 && steps < 60 * n) {
        for (int i = 0; i < hi; i++)
            if (std::fabs(e[i]) <= eps * (std::fabs(d[i]) + std::fabs(d[i + 1]))) e[i] = 0.0;
        if (e[hi - 1] == 0.0) { hi--; continue; }
        int lo = hi - 1;
        while (lo > 0 && e[lo - 1] != 0.0) lo--;
        steps++;
        const double half = 0.5 * (d[hi - 1] - d[hi]), b = e[hi - 1];
        const double shift = d[hi] - b * b / (half + std::copysign(std::hypot(half, b), half));
        double x = d[lo] - shift, z = e[lo];
        for (int k = lo; k < hi; k++) {
            // rotation of rows and columns k, k+1 that clears z against x
            const double r = std::hypot(x, z);
            const double c = r == 0.0 ? 1.0 : x / r, s = r == 0.0 ? 0.0 : z / r;
            if (k > lo) e[k - 1] = r;
            const double dk = d[k], dn = d[k + 1], ek = e[k];
            d[k] = c * c * dk + 2.0 * c * s * ek + s * s * dn;
            d[k + 1] = s * s * dk - 2.0 * c * s * ek + c * c * dn;
            e[k] = c * s * (dn - dk) + (c * c - s * s) * ek;
            if (k + 1 < hi) {
                x = e[k];
                z = s * e[k + 1];
                e[k + 1] *= c;
            }
            double *q0 = &Q[(size_t)k * n], *q1 = q0 + n;
            for (int i = 0; i < n; i++) {
                const double t0 = q0[i], t1 = q1[i];
                q0[i] = c * t0 + s * t1;
                q1[i] = c * t1 - s * t0;
            }
        }
    }
    std::vector<int> idx(n);
    for (int i = 0; i < n; i++) idx[i] = i;
    std::sort(idx.begin(), idx.end(), [&](int i, int j) { return d[i] < d[j]; });
    w.assign(n, 0.0);
    Z.assign((size_t)n * n, 0.0);
    for (int c = 0; c < n; c++) {
        w[c] = d[idx[c]];
        for (int i = 0; i < n; i++) Z[(size_t)i * n + c] = Q[(size_t)idx[c] * n + i];
    }
}

// Cholesky G = R^T R (G: b x b row-major, overwritten by R^{-1}, upper triangular).
// Returns the number of leading columns that were numerically independent.
int chol_inverse(int b, std::vector<double> &G)
{
    std::vector<double> R((size_t)b * b, 0.0);
    int rank = b;
    for (int j = 0; j < b; j++) {
        double d = G[(size_t)j * b + j];
        for (int k = 0; k < j; k++) d -= R[(size_t)k * b + j] * R[(size_t)k * b + j];
        if (!(d > std::max(1e-24, kDependent * G[(size_t)j * b + j]))) { rank = j; break; }
        R[(size_t)j * b + j] = std::sqrt(d);
        for (int i = j + 1; i < b; i++) {
            double v = G[(size_t)j * b + i];
            for (int k = 0; k < j; k++) v -= R[(size_t)k * b + j] * R[(size_t)k * b + i];
            R[(size_t)j * b + i] = v / R[(size_t)j * b + j];
        }
    }
    // inverse of the leading rank x rank block of R (upper triangular), zero elsewhere
    std::vector<double> Ri((size_t)b * b, 0.0);
    for (int j = 0; j < rank; j++) {
        Ri[(size_t)j * b + j] = 1.0 / R[(size_t)j * b + j];
        for (int i = j - 1; i >= 0; i--) {
            double v = 0.0;
            for (int k = i + 1; k <= j; k++) v += R[(size_t)i * b + k] * Ri[(size_t)k * b + j];
            Ri[(size_t)i * b + j] = -v / R[(size_t)i * b + i];
        }
    }
    G.swap(Ri);
    return rank;
}

// Bessel functions J_0..J_{kmax}(x), x > 0, by Miller's backward recurrence
// J_{k-1} = (2k/x) J_k - J_{k+1}, normalised with J_0 + 2 sum_{m>=1} J_{2m} = 1.
std::vector<double> bessel_j(int kmax, double x)
{
    std::vector<double> J(kmax + 1, 0.0);
    if (x == 0.0) { J[0] = 1.0; return J; }
    const int start = 2 * ((std::max(kmax, (int)x) + 30 + (int)(std::sqrt(40.0 * std::max(kmax, (int)x)))) / 2);
    std::vector<double> t(start + 2, 0.0);
    t[start + 1] = 0.0;
    t[start] = 1e-300;
    double norm = 0.0;
    for (int k = start; k >= 1; k--) {
        t[k - 1] = (2.0 * k / x) * t[k] - t[k + 1];
        if (std::fabs(t[k - 1]) > 1e250) {  // rescale to avoid overflow
            for (int q = k - 1; q <= start; q++) t[q] *= 1e-250;
        }
    }
    norm = t[0];
    for (int m = 2; m <= start; m += 2) norm += 2.0 * t[m];
    for (int k = 0; k <= kmax; k++) J[k] = t[k] / norm;
    return J;
}

}  // namespace sg
