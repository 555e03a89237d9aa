"""The index shifts of the row form and the products behind each (host half,
csrc/sg_rows_setup.cpp) against their plain enumeration, product by product and
factor by factor, over random rules, centres, powers and monomials; and how long
they take where many products share their shifts, as a force field's do."""
import os
import subprocess

from paper_2111_13655_gb300 import build

import fake_device

DRIVER = r"""
#include <chrono>
#include <cstdio>
#include <map>
#include <random>
#include "sg_internal.h"
using namespace sg;
using Key = std::vector<int>;

// shift (one entry per mode) -> products, by visiting every combination of factor shifts
static std::map<Key, std::vector<int>> plain(const Problem &p, const HostTables &T)
{
    std::map<Key, std::vector<int>> out;
    for (int q = 0; q + 1 < (int)T.pr_off.size(); q++) {
        Key cur(p.D, 0);
        auto walk = [&](auto &self, int f, int used) -> void {
            if (f == T.pr_off[q + 1]) { out[cur].push_back(q); return; }
            const int m = T.pr_mode[f], op = T.pr_op[f], reach = op ? op : 2;
            for (int d = -reach; d <= reach; d += op == 0 || p.basis[m].q0 == 0.0 ? 2 : 1) {
                const int lm = std::abs(d) < T.kw ? T.lmin_tab[(size_t)m * T.kw + std::abs(d)] : 255;
                if (used + lm > p.L) continue;
                cur[m] = d;
                self(self, f + 1, used + lm);
            }
            cur[m] = 0;
        };
        walk(walk, T.pr_off[q], 0);
    }
    return out;
}
static bool same(const Problem &p, const HostTables &T, const std::map<Key, std::vector<int>> &ref)
{
    if (T.sh_off.size() != ref.size() + 1 || T.sh_src_off.size() != ref.size() + 1) return false;
    size_t s = 0;
    for (const auto &r : ref) {  // (the map's order is the column order)
        Key d(p.D, 0);
        for (int e = T.sh_off[s]; e < T.sh_off[s + 1]; e++) d[T.sh_mode[e]] = T.sh_d[e];
        const std::vector<int> src(T.sh_src.begin() + T.sh_src_off[s], T.sh_src.begin() + T.sh_src_off[s + 1]);
        if (d != r.first || src != r.second) return false;
        s++;
    }
    return true;
}
static double seconds() { return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count(); }

int main()
{
    std::mt19937 r(5);
    auto U = [&](int a, int b) { return (int)(r() % (unsigned)(b - a + 1)) + a; };
    int rows = 0;
    for (int t = 0; t < 300; t++) {
        Problem p;
        p.D = U(1, 7);
        p.L = U(0, 9);
        p.mfoff.push_back(0);
        for (int i = 0; i < p.D; i++) {
            const int a = U(1, 3), b = U(0, 2);
            p.basis.push_back({a, b, U(0, 2) ? 0.0 : 0.1 * U(1, 3), U(0, 1) ? 1.0 : 1.1});
            p.grids.push_back({a + U(0, 2), b});
            p.omega.push_back(U(0, 1) ? 1.0 : -0.5);
        }
        for (int m = U(0, 20); m > 0; m--) {
            const int nf = U(0, 3) ? U(0, 4) : 1;
            for (int f = 0; f < nf; f++) { p.mfmode.push_back(U(0, p.D - 1)); p.mfpow.push_back(U(1, 4)); }
            p.mcoef.push_back(nf == 1 && p.mfpow.back() == 2 && U(0, 1) ? 0.5 * p.omega[p.mfmode.back()] : 0.1 * U(-3, 3));
            p.mnfac.push_back(nf);
            p.mfoff.push_back(p.mfoff.back() + nf);
        }
        HostTables T;
        if (!build_tables(p, 110000, 8, &T).empty()) continue;
        if (!T.rows) { std::printf("problem %d is outside the row form\n", t); return 1; }
        rows++;
        if (!same(p, T, plain(p, T))) { std::printf("problem %d differs\n", t); return 1; }
    }
    // 243 six-mode products that differ in their powers
    Problem p;
    p.D = 6;
    p.L = 10;
    p.mfoff.push_back(0);
    for (int i = 0; i < 6; i++) { p.basis.push_back({1, 1, 0.1 * (i + 1), 1.0}); p.grids.push_back({2, 1}); p.omega.push_back(1.0); }
    for (int e = 0; e < 243; e++) {
        for (int i = 0, x = e; i < 6; i++, x /= 3) { p.mfmode.push_back(i); p.mfpow.push_back(i < 5 ? x % 3 + 1 : 1); }
        p.mcoef.push_back(0.01);
        p.mnfac.push_back(6);
        p.mfoff.push_back(p.mfoff.back() + 6);
    }
    HostTables T;
    if (!build_tables(p, 110000, 8, &T).empty() || !T.rows) return 1;
    double a = 1e9, b = 1e9;
    for (int k = 0; k < 3; k++) {
        const double t0 = seconds();
        build_row_shifts(p, &T);
        const double t1 = seconds();
        const auto ref = plain(p, T);
        const double t2 = seconds();
        if (!same(p, T, ref)) { std::printf("the force field differs\n"); return 1; }
        a = std::min(a, t1 - t0);
        b = std::min(b, t2 - t1);
    }
    std::printf("%d %.6f %.6f\n", rows, a, b);
    return 0;
}
"""


def test_shifts_and_their_products_equal_the_plain_enumeration(tmp_path):
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(DRIVER)
    units = [os.path.join(build.CSRC, f) for f in ("sg_setup.cpp", "sg_rows_setup.cpp")]
    subprocess.run([*fake_device.compiler(), "-O2", str(src), *units, "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    rows, took, plain = out.stdout.split()
    assert int(rows) > 250
    # visiting every product's combinations takes about ten times as long (2.1 million of them over 35,143 shifts)
    assert float(took) < 0.4 * float(plain), out.stdout
