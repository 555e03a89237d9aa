// Host half of the row form of H_S (described in sg_internal.h): the index
// shifts that its products of one-mode matrices couple, the size of the row
// operator, and the windows its rows are cut into.
#include <algorithm>
#include <map>

#include "sg_internal.h"

namespace sg {

namespace {

struct Factor { int mode, op; };  // op: power of Q, 0 = the kinetic matrix

// Shifts k' - k at which the one-mode matrix of `op` can be non-zero at any
// level: the Jacobi matrix of the grid is tridiagonal, with a zero diagonal
// for a grid symmetric about Q = 0; the kinetic matrix couples k to k, k +- 2
// wherever the basis is centred.
void op_shifts(const Problem &p, const Factor &f, std::vector<int> *out)
{
    out->clear();
    const int reach = f.op == 0 ? 2 : f.op;
    const int step = f.op == 0 || p.basis[f.mode].q0 == 0.0 ? 2 : 1;
    for (int d = -reach; d <= reach; d += step) out->push_back(d);
}

}  // namespace

// Products, shifts and the entry count.  rows = false when the levels or the
// shifts exceed what the row form is built for (RowShifts stays empty).
void build_row_shifts(const Problem &p, HostTables *Tp)
{
    HostTables &T = *Tp;
    const int D = p.D, L = p.L, kw = T.kw;
    T.rows = false;
    if (L > kRowMaxL) return;
    T.pr_off.assign(1, 0);
    T.pr_mode.clear(); T.pr_op.clear(); T.pr_coef.clear();
    auto add_product = [&](double c, const std::vector<Factor> &f) {
        for (const Factor &q : f) { T.pr_mode.push_back(q.mode); T.pr_op.push_back(q.op); }
        T.pr_off.push_back((int)T.pr_mode.size());
        T.pr_coef.push_back(c);
    };
    for (int m = 0; m < (int)p.mcoef.size(); m++) {
        bool split = false;
        for (int i = 0; i < D; i++) split |= T.harm_mono[i] == m;
        if (split) continue;  // harmonic part: the FP64 diagonal esplit
        std::vector<Factor> f;
        for (int q = p.mfoff[m]; q < p.mfoff[m + 1]; q++) {
            bool found = false;
            for (Factor &g : f)
                if (g.mode == p.mfmode[q]) { g.op += p.mfpow[q]; found = true; }
            if (!found) f.push_back({p.mfmode[q], p.mfpow[q]});
        }
        add_product(p.mcoef[m], f);
    }
    for (int i = 0; i < D; i++)
        if (T.harm_mono[i] < 0) add_product(1.0, {{i, 0}});

    // distinct shifts (sorted (mode, d) pairs) and the products behind each.
    // A shift that needs more levels than L between its two ends never occurs.
    std::map<std::vector<std::pair<int, int>>, std::vector<int>> shifts;
    const int np = (int)T.pr_coef.size();
    for (int q = 0; q < np; q++) {
        const int nf = T.pr_off[q + 1] - T.pr_off[q];
        std::vector<std::vector<int>> sh(nf);
        for (int a = 0; a < nf; a++) op_shifts(p, {T.pr_mode[T.pr_off[q] + a], T.pr_op[T.pr_off[q] + a]}, &sh[a]);
        std::vector<std::pair<int, int>> cur;
        bool ok = true;
        // depth first over the factors, pruned by the levels the shifts need
        auto walk = [&](auto &self, int a, int used) -> void {
            if (!ok) return;
            if (a == nf) {
                std::vector<std::pair<int, int>> key(cur);
                std::sort(key.begin(), key.end());
                shifts[key].push_back(q);
                if ((int)shifts.size() > kRowMaxShifts) ok = false;
                return;
            }
            const int mode = T.pr_mode[T.pr_off[q] + a];
            for (int d : sh[a]) {
                const int ad = d < 0 ? -d : d;
                if (ad >= kw) continue;
                const int lm = T.lmin_tab[(size_t)mode * kw + ad];
                if (lm > L || used + lm > L) continue;
                if (d) cur.push_back({mode, d});
                self(self, a + 1, used + lm);
                if (d) cur.pop_back();
            }
        };
        walk(walk, 0, 0);
        if (!ok) return;
    }
    // in the order of the column index: lexicographic in the dense shift
    std::vector<const std::pair<const std::vector<std::pair<int, int>>, std::vector<int>> *> ord;
    for (const auto &s : shifts) ord.push_back(&s);
    auto dense_less = [D](const std::vector<std::pair<int, int>> &a, const std::vector<std::pair<int, int>> &b) {
        size_t i = 0, j = 0;
        for (int m = 0; m < D; m++) {
            int x = 0, y = 0;
            if (i < a.size() && a[i].first == m) x = a[i++].second;
            if (j < b.size() && b[j].first == m) y = b[j++].second;
            if (x != y) return x < y;
        }
        return false;
    };
    std::sort(ord.begin(), ord.end(), [&](const auto *a, const auto *b) { return dense_less(a->first, b->first); });
    T.sh_off.assign(1, 0);
    T.sh_src_off.assign(1, 0);
    T.sh_mode.clear(); T.sh_d.clear(); T.sh_src.clear();
    for (const auto *s : ord) {
        for (const auto &md : s->first) { T.sh_mode.push_back(md.first); T.sh_d.push_back(md.second); }
        T.sh_off.push_back((int)T.sh_mode.size());
        T.sh_src.insert(T.sh_src.end(), s->second.begin(), s->second.end());
        T.sh_src_off.push_back((int)T.sh_src.size());
    }

    // Entries: per shift, the k with sum_i lmin_i(max(k_i, k_i + d_i)) <= L,
    // counted by level with one polynomial per mode.
    T.row_nnz = 0;
    std::vector<double> acc, nxt, g;
    double total = 0.0;
    for (size_t s = 0; s + 1 < T.sh_off.size(); s++) {
        acc.assign(L + 1, 0.0);
        acc[0] = 1.0;
        int q = T.sh_off[s];
        for (int i = 0; i < D; i++) {
            int d = 0;
            if (q < T.sh_off[s + 1] && T.sh_mode[q] == i) d = T.sh_d[q++];
            g.assign(L + 1, 0.0);
            for (int k = std::max(0, -d); k < kw && k + d < kw; k++) {
                const int lm = T.lmin_tab[(size_t)i * kw + std::max(k, k + d)];
                if (lm <= L) g[lm] += 1.0;
            }
            nxt.assign(L + 1, 0.0);
            for (int a = 0; a <= L; a++)
                if (acc[a] != 0.0)
                    for (int b = 0; a + b <= L; b++) nxt[a + b] += acc[a] * g[b];
            acc.swap(nxt);
        }
        for (double v : acc) total += v;
    }
    if (total * 12.0 > (double)kRowMaxBytes) return;
    T.row_nnz = (int64_t)total;
    T.rows = true;
}

int row_value_bytes(sg_precision prec) { return prec == SG_MIXED ? 4 : 8; }
int row_vt(const HostTables &T, sg_precision prec)
{
    return T.slice_vt > 0 ? T.slice_vt : prec == SG_MIXED ? SG_F32_VT : prec == SG_DF64 ? SG_DF_VT : SG_F64_VT;
}
int row_window_units(const HostTables &T) { return T.warp_vt > 0 ? T.warp_vt : SG_ROW_WINDOW; }
int row_budget(const HostTables &T, sg_precision prec)
{
    return T.fbudget > 0 ? T.fbudget : 1024 * (prec == SG_MIXED ? SG_F32_SMEM_KB : SG_F64_SMEM_KB);
}

// Rows per window: 16 * units, fewer on small problems so that the windows
// cover the SMs about twice (at least 16).
int row_window_rows(int64_t n, int units)
{
    int w = std::min(16 * units, kRowWindowMax);
    while (w > 16 && (n + w - 1) / w < 304) w >>= 1;
    return w;
}

// (every row filled up by up to three entries)
static int64_t most_entries(const HostTables &T) { return T.row_nnz + 3 * T.n_cs; }

int64_t row_form_windows(const HostTables &T, sg_precision prec)
{
    if (!T.rows) return 0;
    // a window for every 16 rows, and one more for every 4 KB of entries that may end one early
    return T.n_cs / 16 + 1 + most_entries(T) * (4 + row_value_bytes(prec)) / 4096;
}

int64_t row_form_bytes(const HostTables &T, sg_precision prec)
{
    if (!T.rows) return 0;
    return most_entries(T) * (4 + row_value_bytes(prec)) + 8 * T.n_cs +
           row_form_windows(T, prec) * (8 + (int64_t)sizeof(RowWin));
}

// entries of a row with its last group of four filled
static int padded(int n) { return (n + 3) & ~3; }

RowWindows cut_rows(const std::vector<int> &cnt, int wrows, int budget, int value_bytes)
{
    RowWindows W;
    const int n = (int)cnt.size();
    // a block's shared memory: a record (rows' entries behind 8 bytes per row) and a tile of 8 vectors
    const int room = budget / SG_ROW_SHARE - 64 * wrows - 8 * wrows - 32;
    const int cap = std::max(64, room / (4 + value_bytes));
    W.meta.resize(n);
    W.win.resize(n);
    W.start.resize(n);
    std::vector<int> head;
    for (int r0 = 0; r0 < n;) {
        int r1 = r0, ne = 0, longest = 0;
        while (r1 < n && r1 - r0 < wrows && (r1 == r0 || ne + padded(cnt[r1]) <= cap)) {
            W.win[r1] = (int)W.wins.size();
            W.start[r1] = ne;
            longest = std::max(longest, cnt[r1]);
            ne += padded(cnt[r1++]);
        }
        // rows by decreasing length (counting sort, equal lengths in row order)
        head.assign(longest + 2, 0);
        for (int r = r0; r < r1; r++) head[longest - cnt[r] + 1]++;
        for (int l = 0; l <= longest; l++) head[l + 1] += head[l];
        for (int r = r0; r < r1; r++)
            W.meta[r0 + head[longest - cnt[r]]++] =
                make_uint2((unsigned)W.start[r] | ((unsigned)(r - r0) << 24), (unsigned)cnt[r]);
        const RowWin w{(long long)W.bytes, r0, r1 - r0, ne, 0};
        const int bytes = row_win_bytes(w, value_bytes);
        if (ne <= cap) W.cap = std::max(W.cap, bytes);
        W.bytes += bytes;
        W.wins.push_back(w);
        r0 = r1;
    }
    W.wrows = wrows;
    return W;
}

}  // namespace sg
