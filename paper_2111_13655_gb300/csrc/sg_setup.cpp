// Host setup of libsmolyak: 1D tables, terms, compact ranking, capacities.
//
// Everything here runs once per sg_create.  The formulas follow the paper
// (arXiv 2111.13655):
//   - terms l in R(l): L-n+1 <= |l| <= L, coefficient D_l = (-1)^{L-|l|} C(n-1, L-|l|)
//     (Sec. 2, Eq. (8)), numbered in Table-2 order (l_0 varies fastest);
//   - level -> size rules nb(l) = A + B l, nq(l) = A' + B' l (Sec. 2);
//   - compact basis = union of the term boxes, lexicographic with mode 0
//     slowest (Table 2), ranked combinatorially instead of through a stored
//     mapping table M^B (Sec. 3);
//   - 1D transfer matrices of Eqs. (14)/(15) on Gauss-Hermite grids.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <numeric>

#include "sg_internal.h"

namespace sg {

namespace {

// Orthonormal Hermite functions h_0..h_{n-1} at x (stable normalised recurrence).
void hermite_fns(int n, double x, double *h)
{
    const double pi_m14 = 0.75112554446494248286;  // pi^(-1/4)
    h[0] = pi_m14 * std::exp(-0.5 * x * x);
    if (n > 1) h[1] = std::sqrt(2.0) * x * h[0];
    for (int k = 2; k < n; k++)
        h[k] = std::sqrt(2.0 / k) * x * h[k - 1] - std::sqrt((k - 1.0) / k) * h[k - 2];
}

int64_t binom(int n, int k)
{
    if (k < 0 || n < 0 || k > n) return 0;
    int64_t r = 1;
    for (int i = 1; i <= k; i++) r = r * (n - k + i) / i;
    return r;
}

int nsz(int A, int B, int l) { return A + B * l; }

}  // namespace

// Gauss-Hermite rule: nodes are the n zeros of h_n, bracketed by a sign scan of
// h_n over (-sqrt(2n+1)-1/2, sqrt(2n+1)+1/2), bisected and Newton-polished with
// h_n' = sqrt(2n) h_{n-1} - x h_n; weights in the Hermite-function
// normalisation from the Christoffel function, wf_u = 1 / sum_{k<n} h_k(x_u)^2
// (so that sum_u wf_u h_k(x_u) h_k'(x_u) = delta_kk' for k, k' < n).
std::string gauss_hermite(int n, std::vector<double> *x, std::vector<double> *wf)
{
    x->assign(n, 0.0);
    wf->assign(n, 0.0);
    if (n < 1 || n > 64) return "gauss_hermite: n out of range";
    std::vector<double> h(n + 1);
    auto hn = [&](double t) { hermite_fns(n + 1, t, h.data()); return h[n]; };
    const double a = std::sqrt(2.0 * n + 1.0) + 0.5;
    const int scan = 400 * n;
    auto polish = [&](double r) {
        for (int it = 0; it < 3; it++) {
            hermite_fns(n + 1, r, h.data());
            double d = std::sqrt(2.0 * n) * h[n - 1] - r * h[n];
            if (d != 0.0 && h[n] != 0.0) r -= h[n] / d;
        }
        return r;
    };
    int found = 0;
    double t0 = -a, f0 = hn(t0);
    for (int i = 1; i <= scan && found < n; i++) {
        double t1 = -a + 2.0 * a * i / scan, f1 = hn(t1);
        if (f1 == 0.0) {                 // the scan landed on a zero
            (*x)[found++] = polish(t1);
        } else if (f0 != 0.0 && (f0 < 0) != (f1 < 0)) {
            double lo = t0, hi = t1, flo = f0;
            for (int it = 0; it < 200 && hi - lo > 1e-15 * (1 + std::fabs(lo)); it++) {
                double mid = 0.5 * (lo + hi), fm = hn(mid);
                if (fm == 0.0) { lo = hi = mid; break; }
                if ((fm < 0) == (flo < 0)) { lo = mid; flo = fm; } else { hi = mid; }
            }
            (*x)[found++] = polish(0.5 * (lo + hi));
        }
        t0 = t1; f0 = f1;
    }
    if (found != n) return "gauss_hermite: root bracketing failed";
    if (n % 2 == 1) (*x)[n / 2] = 0.0;
    for (int u = 0; u < n; u++) {  // enforce the exact symmetry of the rule
        double s = 0.5 * ((*x)[n - 1 - u] - (*x)[u]);
        if (u < n / 2) { (*x)[u] = -s; (*x)[n - 1 - u] = s; }
    }
    for (int u = 0; u < n; u++) {
        hermite_fns(n, (*x)[u], h.data());
        double s = 0.0;
        for (int k = 0; k < n; k++) s += h[k] * h[k];
        (*wf)[u] = 1.0 / s;
    }
    return "";
}

// Whether every monomial touches at most two modes, in at most kMaxPairs mode
// pairs: the potentials that SG_DF64 and sg_tune take.
static bool pair_potential(const Problem &p)
{
    std::vector<std::pair<int, int>> pairs;
    for (int m = 0; m < (int)p.mcoef.size(); m++) {
        int a = -1, b = -1;
        for (int f = p.mfoff[m]; f < p.mfoff[m + 1]; f++) {
            const int i = p.mfmode[f];
            if (i == a || i == b) continue;
            if (a < 0) a = i;
            else if (b < 0) b = i;
            else return false;
        }
        if (b < 0) continue;
        const std::pair<int, int> ab(std::min(a, b), std::max(a, b));
        if (std::find(pairs.begin(), pairs.end(), ab) == pairs.end()) pairs.push_back(ab);
    }
    return pairs.size() <= (size_t)kMaxPairs;
}

std::string build_tables(const Problem &p, int smem_budget, int rb, HostTables *out)
{
    HostTables &T = *out;
    const int D = p.D, L = p.L;
    char buf[256];

    // ---------------- per (mode, level) 1D tables ----------------
    T.pmax = 0;
    for (int m = 0; m < (int)p.mnfac.size(); m++) {
        // largest total power of one mode inside one monomial
        int pw[kMaxD] = {0};
        for (int f = p.mfoff[m]; f < p.mfoff[m + 1]; f++) pw[p.mfmode[f]] += p.mfpow[f];
        for (int i = 0; i < D; i++) T.pmax = std::max(T.pmax, pw[i]);
    }
    T.lvl.assign((size_t)D * (L + 1), LevelInfo{});
    T.tabd.clear();
    std::vector<std::vector<double>> rule_x(kMaxLevelSize + 1), rule_w(kMaxLevelSize + 1);  // by number of nodes
    for (int i = 0; i < D; i++) {
        const double q0 = p.basis[i].q0, s = p.basis[i].scale;
        // an earlier mode with the same basis, grid and kinetic prefactor has the same tables
        int same = 0;
        while (same < i && !(p.basis[same].q0 == q0 && p.basis[same].scale == s && p.omega[same] == p.omega[i] &&
                             p.basis[same].nb_A == p.basis[i].nb_A && p.basis[same].nb_B == p.basis[i].nb_B &&
                             p.grids[same].nq_A == p.grids[i].nq_A && p.grids[same].nq_B == p.grids[i].nq_B))
            same++;
        for (int l = 0; l <= L; l++) {
            LevelInfo &li = T.lvl[(size_t)i * (L + 1) + l];
            if (same < i) {
                li = T.lvl[(size_t)same * (L + 1) + l];
                continue;
            }
            li.nb = nsz(p.basis[i].nb_A, p.basis[i].nb_B, l);
            li.nq = nsz(p.grids[i].nq_A, p.grids[i].nq_B, l);
            const int nb = li.nb, nq = li.nq;
            if (rule_x[nq].empty()) {
                const std::string e = gauss_hermite(nq, &rule_x[nq], &rule_w[nq]);
                if (!e.empty()) return e;
            }
            const std::vector<double> &xg = rule_x[nq], &wf = rule_w[nq];
            std::vector<double> h(nb + 2), B(nq * nb), BW(nb * nq), D2(nq * nb), Q(nq), W(nq);
            for (int u = 0; u < nq; u++) {
                hermite_fns(nb + 2, xg[u], h.data());
                W[u] = wf[u] / s;
                Q[u] = q0 + xg[u] / s;
                for (int k = 0; k < nb; k++) {
                    B[u * nb + k] = std::sqrt(s) * h[k];
                    // b_k'' from the ladder form of d/dx applied twice:
                    //   h_k'' = 1/2 sqrt(k(k-1)) h_{k-2} - (k+1/2) h_k + 1/2 sqrt((k+1)(k+2)) h_{k+2}
                    double d2 = -(k + 0.5) * h[k] + 0.5 * std::sqrt((k + 1.0) * (k + 2.0)) * h[k + 2];
                    if (k >= 2) d2 += 0.5 * std::sqrt(k * (k - 1.0)) * h[k - 2];
                    D2[u * nb + k] = std::sqrt(s) * s * s * d2;
                }
            }
            for (int k = 0; k < nb; k++)
                for (int u = 0; u < nq; u++) BW[k * nq + u] = W[u] * B[u * nb + k];
            li.offB = (int)T.tabd.size();
            T.tabd.insert(T.tabd.end(), B.begin(), B.end());
            li.offBW = (int)T.tabd.size();
            T.tabd.insert(T.tabd.end(), BW.begin(), BW.end());
            li.offK = (int)T.tabd.size();
            for (int k = 0; k < nb; k++)
                for (int kp = 0; kp < nb; kp++) {
                    double acc = 0.0;
                    for (int u = 0; u < nq; u++) acc += BW[k * nq + u] * D2[u * nb + kp];
                    T.tabd.push_back(-0.5 * p.omega[i] * acc);
                }
            li.offQ = (int)T.tabd.size();
            T.tabd.insert(T.tabd.end(), Q.begin(), Q.end());
            li.offMu = (int)T.tabd.size();
            for (int pw = 0; pw <= T.pmax; pw++) {
                double acc = 0.0;
                for (int u = 0; u < nq; u++) acc += W[u] * B[u * nb] * B[u * nb] * std::pow(Q[u], pw);
                T.tabd.push_back(acc);
            }
            // single-mode potential factors in the basis: M_p = B^T W diag(Q^p) B
            li.offM = (int)T.tabd.size();
            for (int pw = 1; pw <= std::max(T.pmax, 1); pw++) {
                std::vector<double> Qp(nq);
                for (int u = 0; u < nq; u++) Qp[u] = std::pow(Q[u], pw);
                for (int k = 0; k < nb; k++)
                    for (int kp = 0; kp < nb; kp++) {
                        double acc = 0.0;
                        for (int u = 0; u < nq; u++) acc += BW[k * nq + u] * Qp[u] * B[u * nb + kp];
                        T.tabd.push_back(acc);
                    }
            }
        }
    }
    // Harmonic split.  For a mode centred at q0 = 0 with scale s, the basis
    // functions are eigenfunctions of -omega/2 d^2/dQ^2 + omega s^4/2 Q^2 with
    // eigenvalue omega s^2 (k+1/2), at every level and on every grid with
    // nq >= nb.  When the potential holds exactly that quadratic monomial, the
    // pair is diagonal in every term, and the combination identity
    // sum_{l in R(l), l >= k} D_l = 1 adds it once: it is taken out of the
    // term actions and applied in the compact basis.
    T.harm_mono.assign(D, -1);
    for (int i = 0; i < D; i++) {
        if (p.basis[i].q0 != 0.0 || !(p.omega[i] > 0.0)) continue;
        const double s = p.basis[i].scale;
        const double want = 0.5 * p.omega[i] * s * s * s * s;
        for (int m = 0; m < (int)p.mnfac.size(); m++)
            if (p.mnfac[m] == 1 && p.mfmode[p.mfoff[m]] == i && p.mfpow[p.mfoff[m]] == 2 &&
                std::fabs(p.mcoef[m] - want) <= 4e-16 * std::fabs(want)) {
                T.harm_mono[i] = m;
                break;
            }
    }
    if (T.tabd.size() >= (size_t)1 << 30) return "tables too large";

    // ---------------- compact ranking ----------------
    // lmin_i(k) = smallest level whose basis holds function k of mode i.
    T.kw = 0;
    for (int i = 0; i < D; i++) T.kw = std::max(T.kw, nsz(p.basis[i].nb_A, p.basis[i].nb_B, L));
    const int kw = T.kw;
    T.lmin_tab.assign((size_t)D * kw, 255);
    for (int i = 0; i < D; i++)
        for (int k = 0; k < kw; k++) {
            int l = 0;
            while (l <= L && nsz(p.basis[i].nb_A, p.basis[i].nb_B, l) <= k) l++;
            if (l <= L) T.lmin_tab[(size_t)i * kw + k] = (uint8_t)l;
        }
    // cnt[i][R] = number of tails (k_i..k_{D-1}) with sum of lmin <= R (R = 0..L)
    std::vector<int64_t> cnt((size_t)(D + 1) * (L + 1), 0);
    for (int R = 0; R <= L; R++) cnt[(size_t)D * (L + 1) + R] = 1;
    for (int i = D - 1; i >= 0; i--)
        for (int R = 0; R <= L; R++) {
            int64_t c = 0;
            for (int k = 0; k < kw; k++) {
                int lm = T.lmin_tab[(size_t)i * kw + k];
                if (lm <= R) c += cnt[(size_t)(i + 1) * (L + 1) + (R - lm)];
            }
            cnt[(size_t)i * (L + 1) + R] = c;
        }
    T.n_cs = cnt[L];
    if (T.n_cs >= ((int64_t)1 << 31) - 1) return "N_cs >= 2^31 is outside this build's limits";
    // rank(k) = sum_i T_i[s_i][k_i], s_i = sum_{j<i} lmin_j(k_j),
    // T_i[s][k] = sum_{v<k} cnt[i+1][L - s - lmin_i(v)]  (tails that precede k_i = k)
    T.rank_tab.assign((size_t)D * (L + 1) * kw, 0);
    for (int i = 0; i < D; i++)
        for (int s = 0; s <= L; s++) {
            int64_t acc = 0;
            for (int k = 0; k < kw; k++) {
                T.rank_tab[((size_t)i * (L + 1) + s) * kw + k] = (int)acc;
                int lm = T.lmin_tab[(size_t)i * kw + k];
                int R = L - s - lm;
                if (lm <= L && R >= 0) acc += cnt[(size_t)(i + 1) * (L + 1) + R];
            }
        }

    // harmonic energies of the split modes over the compact basis, enumerated
    // in compact order (lexicographic, mode 0 slowest) under sum lmin <= L
    {
        T.esplit.assign(T.n_cs, 0.0);
        std::vector<int> k(D, 0), c(D, 0);
        int sum = 0;
        int64_t r = 0;
        for (;;) {
            double e = 0.0;
            for (int i = 0; i < D; i++)
                if (T.harm_mono[i] >= 0)
                    e += p.omega[i] * p.basis[i].scale * p.basis[i].scale * (k[i] + 0.5);
            if (r >= T.n_cs) return "compact enumeration overran N_cs";
            T.esplit[r++] = e;
            int i = D - 1;
            while (i >= 0) {
                k[i]++;
                int lm = k[i] < kw ? T.lmin_tab[(size_t)i * kw + k[i]] : 255;
                if (lm <= L && sum - c[i] + lm <= L) { sum += lm - c[i]; c[i] = lm; break; }
                sum -= c[i]; c[i] = 0; k[i] = 0; i--;
            }
            if (i < 0) break;
        }
        if (r != T.n_cs) return "compact enumeration does not match N_cs";
    }

    // ---------------- terms in Table-2 order (l_0 fastest) ----------------
    T.Dpad = (D + 3) / 4 * 4;
    T.levels.clear();
    T.coefs.clear();
    std::vector<int> l(D, 0);
    // depth-first over modes D-1 (slowest) .. 0 (fastest), remaining budget `rem`
    struct Rec {
        static void run(int i, int rem, int sum, int D, int L, std::vector<int> &l, HostTables &T)
        {
            if (i < 0) {
                if (sum >= L - D + 1) {
                    for (int j = 0; j < T.Dpad; j++) T.levels.push_back(j < D ? (uint8_t)l[j] : 0);
                    int r = L - sum;
                    int64_t c = binom(D - 1, r);
                    T.coefs.push_back((int)((r % 2) ? -c : c));
                }
                return;
            }
            for (int v = 0; v <= rem; v++) {
                l[i] = v;
                run(i - 1, rem - v, sum + v, D, L, l, T);
            }
            l[i] = 0;
        }
    };
    Rec::run(D - 1, L, 0, D, L, l, T);
    T.n_terms = (int64_t)T.coefs.size();
    if (T.n_terms >= ((int64_t)1 << 31)) return "too many terms";

    // ---------------- per-term sizes, capacities, work ----------------
    // Pair-table bound: distinct mode pairs that share a monomial.
    std::vector<char> pair_seen((size_t)D * D, 0);
    int64_t pair_entries = 0;
    for (int m = 0; m < (int)p.mnfac.size(); m++)
        for (int f = p.mfoff[m]; f < p.mfoff[m + 1]; f++)
            for (int g = f + 1; g < p.mfoff[m + 1]; g++) {
                int a = std::min(p.mfmode[f], p.mfmode[g]), b = std::max(p.mfmode[f], p.mfmode[g]);
                if (a == b || pair_seen[(size_t)a * D + b]) continue;
                pair_seen[(size_t)a * D + b] = 1;
                int nqa = 0, nqb = 0;
                for (int lv = 0; lv <= L; lv++) {
                    nqa = std::max(nqa, T.lvl[(size_t)a * (L + 1) + lv].nq);
                    nqb = std::max(nqb, T.lvl[(size_t)b * (L + 1) + lv].nq);
                }
                pair_entries += (int64_t)nqa * nqb;
            }

    std::vector<int64_t> cost(T.n_terms);
    T.maxnb = 1;
    T.matcap = 1;
    int fsum_max = 1, stage_min_max = 1;
    T.n_s = 0;
    T.n_grid = 0;
    for (int64_t t = 0; t < T.n_terms; t++) {
        const uint8_t *lt = &T.levels[(size_t)t * T.Dpad];
        int nb[kMaxD], nq[kMaxD], m = 0;
        int64_t NB = 1, NG = 1, NGfull = 1;
        int mats = 0, fsum = 0;
        for (int i = 0; i < D; i++) {
            const LevelInfo &li = T.lvl[(size_t)i * (L + 1) + lt[i]];
            NGfull *= li.nq;
            if (li.nb > 1) {
                nb[m] = li.nb; nq[m] = li.nq; m++;
                NB *= li.nb; NG *= li.nq;
                mats += 2 * li.nb * li.nq + li.nb * li.nb;
                fsum += li.nq;
            }
        }
        T.n_s += NB;
        T.n_grid += NGfull;
        T.maxnb = (int)std::max<int64_t>(T.maxnb, NB);
        T.matcap = std::max(T.matcap, mats);
        fsum_max = std::max(fsum_max, fsum);
        if (m > 0) stage_min_max = std::max(stage_min_max, nb[m - 1]);
        // cost of the term: multiply-adds of the forward and backward chains and the kinetic matrices
        int64_t fma = 0;
        for (int tt = 0; tt < m; tt++) {
            int64_t sz = (int64_t)nb[tt] * nq[tt];
            for (int j = 0; j < tt; j++) sz *= nq[j];
            for (int j = tt + 1; j < m; j++) sz *= nb[j];
            fma += 2 * sz;
        }
        for (int j = 0; j < m; j++) fma += NB * nb[j];
        cost[t] = 2 * fma + 8 * NG + 16 * NB + 256;
    }
    T.vtabcap = fsum_max + (int)std::min<int64_t>(pair_entries, 1 << 24);

    // Shared memory: fixed part + two grid buffers of `cap` elements.
    const int nm = std::max(1, (int)p.mnfac.size());
    size_t fixed = (size_t)rb * (T.matcap + T.vtabcap + 4 * (size_t)T.maxnb) + 4 * (size_t)T.maxnb +
                   (size_t)nm * (16 + 24 + 16 + 16) + 1024;
    if (fixed + 2 * (size_t)rb * stage_min_max > (size_t)smem_budget) {
        snprintf(buf, sizeof buf, "a term needs %zu bytes of shared memory (budget %d)",
                 fixed + 2 * (size_t)rb * stage_min_max, smem_budget);
        return buf;
    }
    T.cap = (int)(((size_t)smem_budget - fixed) / (2 * (size_t)rb));
    T.cap = std::max(T.cap, stage_min_max);

    // processing order: most expensive terms first (longest-processing-time first)
    T.order.resize(T.n_terms);
    std::iota(T.order.begin(), T.order.end(), 0);
    std::stable_sort(T.order.begin(), T.order.end(),
                     [&](int a, int b) { return cost[a] > cost[b]; });
    T.pcost.resize(T.n_terms);
    for (int64_t q = 0; q < T.n_terms; q++) T.pcost[q] = cost[T.order[q]];

    T.pairs = pair_potential(p);
    build_row_shifts(p, &T);
    return "";
}

}  // namespace sg
