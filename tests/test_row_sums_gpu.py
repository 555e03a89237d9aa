"""How a row is summed, entry by entry against bounds derived from the arithmetic.

Mixed precision (u = 2^-24): the element and the value are rounded to FP32, a
group of four products is one product and three multiply-adds, each rounded, and
the groups are added by two-sum into a pair whose low part collects the errors.
A product passes through at most 2 + 4 roundings; the low part's own roundings
add (m/4)^2 u^2 of the terms' sum for m entries (below 0.02 u here):
    |y_i - (H x)_i| <= 6.1 u sum_j |H_ij x_j|.
An FP32 sum of the groups alone would add up to (m/4) u of the partial sums.
Double-float: each step is within 8 u^2 (|product| + |sum so far|)
(test_df_arith.py), element and value are split to 2^-48 each:
    |y_i - (H x)_i| <= (8 (m + 1) + 2) u^2 sum_j |H_ij x_j|.
The harmonic diagonal is added in FP64 and left out of the sums above.
"""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2111_13655_gb300 as sg
from paper_2111_13655_gb300 import synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
PROBLEMS = {
    # rows of up to 2,026 entries
    "dense, three modes": synth.polynomial_problem(
        3, 28, [1.0, 0.9, 1.1],
        [(0.01 / (1 + a + b + c), [(0, a), (1, b), (2, c)]) for a, b, c in itertools.product((5, 6), repeat=3)],
        nq_rule=(2, 1), q0=[0.1, -0.1, 0.2]),
    "dense, two modes": synth.polynomial_problem(
        2, 30, [1.0, 0.9], [(0.01 / (1 + a + b), [(0, a), (1, b)]) for a, b in itertools.product((5, 6), repeat=2)],
        q0=[0.1, -0.1]),
    "chain": synth.workload_C2(),
}


def apply(ctx, x):
    y = torch.full_like(x, float("nan"))
    sg.sg_apply_H(ctx, x, y, x.shape[0])
    return y


def dense(p):
    """H_S from FP64 applies to unit vectors (one product per entry: exact to its rounding)."""
    with sg.sg_create(p, "fp64") as ctx:
        eye = torch.eye(ctx.n_cs, dtype=torch.float64, device="cuda")
        H = torch.cat([apply(ctx, eye[i:i + 500]) for i in range(0, ctx.n_cs, 500)]).T.contiguous()
    return H


@pytest.mark.parametrize("name,prec", [(n, q) for n in PROBLEMS for q in ("mixed", "df64")
                                       if (n, q) != ("dense, three modes", "df64")])
def test_row_sums_stay_within_the_bound_of_their_arithmetic(name, prec):
    p = PROBLEMS[name]
    H = dense(p)
    n = H.shape[0]
    rows = H.clone()
    if name == "chain":                    # centred cubic couplings: the diagonal is the harmonic part
        rows.fill_diagonal_(0.0)
    count = (rows != 0.0).sum(1)
    x = torch.from_numpy(synth.random_vectors(n, 6, 3)).cuda()
    # the longest row: a large product first, its negative last, and between them
    # products that one FP32 accumulator at that height would lose one by one
    r = int(count.argmax())
    cols = torch.nonzero(rows[r]).reshape(-1)
    for v, (first, small, last) in enumerate([(1.0, 2.0 ** -27, -1.0), (1.0, 2.0 ** -27, 1.0), (2.0 ** 20, 2.0 ** -8, -2.0 ** 20)]):
        t = torch.full((len(cols),), small, dtype=torch.float64, device="cuda")
        t[0], t[-1] = first, last
        x[v] = 0.0
        x[v, cols] = t / rows[r, cols]
    with sg.sg_create(p, prec) as ctx:
        err = (apply(ctx, x) - x @ H.T).abs()
        assert sg.sg_device_error(ctx) == 0
    scale = x.abs() @ rows.abs().T
    bound = 6.1 * U * scale if prec == "mixed" else (8.0 * (count + 1) + 2.0) * U * U * scale
    exact = 2.0 ** -52 * (x.abs() @ H.abs().T) * 64       # rounding of the reference's products and sums
    assert (err <= bound + exact).all(), float(((err - exact) / scale.clamp_min(1e-300)).max() / U)
    if prec == "mixed" and name == "dense, three modes":
        # one FP32 accumulator would lose the small products of this row, which is far outside the bound
        assert len(cols) > 2000 and len(cols) * 2.0 ** -27 > 10.0 * float(bound[0, r])
