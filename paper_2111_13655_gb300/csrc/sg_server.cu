// Device side of the propagation server (sg_server_api.cpp): one fused update of
// every active request's Chebyshev recurrence after a batched application of
// H_S, and the per-request norm / energy sums logged at the start of each step.
// The recurrence state (term index, step) lives on the device, so one
// iteration's launches are the same every time and can be replayed as a graph.
//
// Chebyshev propagator (Sec. 3, Sec. 5; Tal-Ezer-Kosloff form):
//   psi(t + dt) = e^{-i Ebar dt} sum_{k=0}^{K} c_k (-i)^k T_k,   c_k = (2 - delta_k0) J_k(dE dt),
//   T_0 = psi,  T_1 = (H - Ebar) psi / dE,  T_{k+1} = 2 (H - Ebar) T_k / dE - T_{k-1}.
// Vectors are complex, held as two real vectors (real part, then imaginary
// part) per request, requests one after another (the batch layout, nvec = 2).
#include <algorithm>

#include "sg_cheb.cuh"
#include "sg_launch.cuh"

namespace sg {

namespace {

// Which request owns complex entry g: the last j with prefix[j] <= g.
__device__ __forceinline__ int owner(const long long *__restrict__ prefix, int n, long long g)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// X = T_k, Y = H T_k, P = T_{k-1} (unused when forming T_1), A = partial sum;
// k, K and the weights come from the request's device state.  Writes T_{k+1}
// (or, on the step's last term, the new psi) into P's slot; the roles of X
// and P are then swapped for every request.  A request past its last step
// keeps psi: it is copied to P's slot.
__global__ void k_cheb_update(const ChebState *__restrict__ st, const long long *__restrict__ prefix, int nitems,
                              const double *__restrict__ X, const double *__restrict__ Y, double *P, double *A)
{
    const long long total = prefix[nitems];
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
         g += (long long)gridDim.x * blockDim.x) {
        const int j = owner(prefix, nitems, g);
        const ChebState &it = st[j];
        const long long n = prefix[j + 1] - prefix[j];
        const long long i = g - prefix[j];
        const long long re = 2 * prefix[j] + i, im = re + n;
        const double xr = X[re], xi = X[im];
        if (it.step >= it.nsteps) {
            P[re] = xr;
            P[im] = xi;
            continue;
        }
        const ChebTerm t = cheb_term(it);
        double pr = 0.0, pi = 0.0, ar = 0.0, ai = 0.0;
        if (t.kn > 1) {
            pr = P[re];
            pi = P[im];
            ar = A[re];
            ai = A[im];
        }
        const bool last = cheb_entry(t, xr, xi, Y[re], Y[im], pr, pi, ar, ai);
        P[re] = pr;
        P[im] = pi;
        if (!last) {
            A[re] = ar;
            A[im] = ai;
        }
    }
}

// One block per request, after the update: requests at the start of a step
// (k = 0) log <psi|psi> and <psi|H psi>/<psi|psi> over their own entries,
// summed in an order that depends on their size only; then every request moves
// to its next recurrence term.
constexpr int kLogThreads = 256;
__global__ void __launch_bounds__(kLogThreads) k_cheb_log_advance(ChebState *st,
                                                                  const long long *__restrict__ prefix,
                                                                  const double *X, const double *Y)
{
    grid_trigger();
    grid_wait();
    ChebState &S = st[blockIdx.x];
    const int k = S.k, step = S.step, K = S.K;
    __syncthreads();  // every thread has read the state that thread 0 moves on
    if (step >= S.nsteps) return;
    if (k != 0) {
        if (threadIdx.x == 0) {
            S.k = k + 1 == K ? 0 : k + 1;
            if (k + 1 == K) S.step = step + 1;
        }
        return;
    }
    const long long off = prefix[blockIdx.x], n = prefix[blockIdx.x + 1] - off;
    const double *xr = X + 2 * off, *xi = xr + n, *yr = Y + 2 * off, *yi = yr + n;
    double nn = 0.0, ee = 0.0;
    for (long long i = threadIdx.x; i < n; i += kLogThreads) {
        nn = fma(xr[i], xr[i], fma(xi[i], xi[i], nn));
        ee = fma(xr[i], yr[i], fma(xi[i], yi[i], ee));
    }
    __shared__ double sn[kLogThreads], se[kLogThreads];
    sn[threadIdx.x] = nn;
    se[threadIdx.x] = ee;
    __syncthreads();
    for (int h = kLogThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            sn[threadIdx.x] += sn[threadIdx.x + h];
            se[threadIdx.x] += se[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        S.log[2 * step] = sn[0];
        S.log[2 * step + 1] = se[0] / sn[0];
        if (K == 1) S.step = step + 1;
        else S.k = 1;
    }
}

}  // namespace

cudaError_t launch_cheb_iteration(ChebState *st, const long long *prefix, int nitems, int64_t total,
                                  const double *X, const double *Y, double *P, double *A, cudaStream_t s)
{
    if (nitems <= 0 || total <= 0) return cudaSuccess;
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, 152 * 8));
    k_cheb_update<<<blocks, 256, 0, s>>>(st, prefix, nitems, X, Y, P, A);
    return launch_early(k_cheb_log_advance, dim3((unsigned)nitems), kLogThreads, 0, s, st, prefix, X, Y);
}

cudaError_t launch_cheb_log_advance(ChebState *st, const long long *prefix, int nitems, const double *X,
                                    const double *Y, cudaStream_t s)
{
    if (nitems <= 0) return cudaSuccess;
    return launch_early(k_cheb_log_advance, dim3((unsigned)nitems), kLogThreads, 0, s, st, prefix, X, Y);
}

}  // namespace sg
