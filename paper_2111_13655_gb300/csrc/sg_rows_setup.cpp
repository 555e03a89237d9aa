// Host half of the row form of H_S (described in sg_internal.h): the index
// shifts that its products of one-mode matrices couple, the size of the row
// operator, and the windows its rows are cut into.
#include <algorithm>
#include <array>
#include <cstdlib>
#include <cstring>
#include <unordered_set>

#include "sg_internal.h"

namespace sg {

namespace {

struct Factor { int mode, op; };  // op: power of Q, 0 = the kinetic matrix

// Shifts k' - k at which the one-mode matrix of a factor can be non-zero at any
// level: -reach, -reach + step, ..., reach.  The Jacobi matrix of the grid is
// tridiagonal, with a zero diagonal for a grid symmetric about Q = 0; the
// kinetic matrix couples k to k, k +- 2 wherever the basis is centred.
struct Reach {
    int mode, reach, step;
    Reach(const Problem &p, int m, int op)
        : mode(m), reach(op == 0 ? 2 : op), step(op == 0 || p.basis[m].q0 == 0.0 ? 2 : 1)
    {
    }
    bool holds(int d) const
    {
        const int a = d < 0 ? -d : d;
        return a <= reach && (step == 1 || (reach - a) % 2 == 0);
    }
    bool within(const Reach &o) const { return mode == o.mode && (o.step == 1 || step == 2) && o.holds(reach); }
};
// Whether every shift of product a is one of product b.
bool within(const std::vector<Reach> &a, const std::vector<Reach> &b)
{
    for (const Reach &f : a)
        if (std::none_of(b.begin(), b.end(), [&](const Reach &g) { return f.within(g); })) return false;
    // b's other modes stay where they are
    for (const Reach &g : b)
        if (!g.holds(0) && std::none_of(a.begin(), a.end(), [&](const Reach &f) { return f.mode == g.mode; })) return false;
    return true;
}

// A shift k' - k over all modes, as bytes whose order is that of the shifts.
constexpr int kNoShift = 128;
struct Shift {
    std::array<unsigned char, kMaxD> d;
    bool operator==(const Shift &o) const { return d == o.d; }
};
static_assert(kMaxLevelSize <= 127 && kMaxD % 8 == 0, "a shift per byte, eight to a word");
struct ShiftHash {
    size_t operator()(const Shift &s) const
    {
        uint64_t h = 0, w;
        for (int i = 0; i < kMaxD; i += 8) {
            std::memcpy(&w, s.d.data() + i, 8);
            h = (h ^ w) * 0x9E3779B97F4A7C15ull;
            h ^= h >> 29;
        }
        return (size_t)h;
    }
};

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

    // Distinct shifts and the products behind each.  A shift that needs more
    // levels than L between its two ends never occurs.
    // They are collected from the products whose shifts are not all another's
    // (a force field's products differ mostly in the powers: 64 six-mode
    // products over 3,003 functions have one such, and collecting from each made
    // a plan of 93 ms instead of 12).
    const int np = (int)T.pr_coef.size();
    std::vector<std::vector<Reach>> prod(np);
    for (int q = 0; q < np; q++)
        for (int f = T.pr_off[q]; f < T.pr_off[q + 1]; f++) prod[q].emplace_back(p, T.pr_mode[f], T.pr_op[f]);
    std::unordered_set<Shift, ShiftHash> found;
    Shift cur;
    cur.d.fill(kNoShift);
    for (int q = 0; q < np; q++) {
        bool inside = false;
        for (int o = 0; o < np && !inside; o++)
            inside = o != q && within(prod[q], prod[o]) && (o < q || !within(prod[o], prod[q]));
        if (inside) continue;
        bool ok = true;
        // depth first over the factors, pruned by the levels the shifts need
        auto walk = [&](auto &self, size_t a, int used) -> void {
            if (!ok) return;
            if (a == prod[q].size()) {
                found.insert(cur);
                if ((int)found.size() > kRowMaxShifts) ok = false;
                return;
            }
            const Reach &f = prod[q][a];
            for (int d = -f.reach; d <= f.reach; d += f.step) {
                const int ad = d < 0 ? -d : d;
                if (ad >= kw) continue;
                const int lm = T.lmin_tab[(size_t)f.mode * kw + ad];
                if (lm > L || used + lm > L) continue;
                cur.d[f.mode] = (unsigned char)(kNoShift + d);
                self(self, a + 1, used + lm);
            }
            cur.d[f.mode] = kNoShift;
        };
        walk(walk, 0, 0);
        if (!ok) return;
    }
    // in the order of the column index: lexicographic in the shift
    std::vector<Shift> shifts(found.begin(), found.end());
    std::sort(shifts.begin(), shifts.end(), [](const Shift &a, const Shift &b) { return a.d < b.d; });
    // per mode and |d| the products that a move by d belongs to, a bit each
    const int words = (np + 63) / 64;
    std::vector<uint64_t> takes((size_t)D * kw * words, 0), all(words);
    for (int q = 0; q < np; q++) {
        const uint64_t bit = 1ull << (q % 64);
        auto at = [&](int mode, int ad) -> uint64_t & { return takes[((size_t)mode * kw + ad) * words + q / 64]; };
        for (int i = 0; i < D; i++) at(i, 0) |= bit;
        for (const Reach &f : prod[q])
            for (int ad = 0; ad < kw; ad++) at(f.mode, ad) = f.holds(ad) ? at(f.mode, ad) | bit : at(f.mode, ad) & ~bit;
    }
    T.sh_off.assign(1, 0);
    T.sh_src_off.assign(1, 0);
    T.sh_mode.clear(); T.sh_d.clear(); T.sh_src.clear();
    for (const Shift &s : shifts) {
        all.assign(words, ~0ull);
        for (int i = 0; i < D; i++) {
            const int d = (int)s.d[i] - kNoShift;
            if (d) { T.sh_mode.push_back(i); T.sh_d.push_back(d); }
            const uint64_t *t = &takes[((size_t)i * kw + std::abs(d)) * words];
            for (int w = 0; w < words; w++) all[w] &= t[w];
        }
        T.sh_off.push_back((int)T.sh_mode.size());
        for (int w = 0; w < words; w++)
            for (uint64_t m = all[w]; m; m &= m - 1) {
                const int q = 64 * w + __builtin_ctzll(m);
                if (q < np) T.sh_src.push_back(q);
            }
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
