"""The row form of H_S against the literal oracle, on the CPU.

The apply does not visit the terms of Eq. (16): the combination telescopes
mode by mode, so that a product of one-mode operators over the modes S couples
k and k' by
    c * sum over levels (l_i, i in S), |l_S| <= L - sum_{i not in S} lmin_i(k_i)
          of prod_{i in S} (M_i(l_i) - M_i(l_i - 1))[k_i, k'_i],
M_i(l) the operator's matrix on the level's basis and grid (zero outside it),
and only where k_i = k'_i outside S.  Both the sum and the shifts k' - k it is
restricted to are restated here from the library's 1D tables, and compared
with the term-by-term oracle over level rules, centres, scales and monomials.
"""
import itertools

import numpy as np
import pytest

import paper_2111_13655_gb300 as sg
from oracle import oracle as orc
from paper_2111_13655_gb300 import synth

from helpers import dense_oracle, literal_elem_tol

MONOS = [(0.3, [(0, 1)]), (0.2, [(0, 2), (1, 2)]), (-0.1, [(1, 3)]), (0.05, [(0, 1), (1, 1), (2, 1)]), (0.7, []),
         (0.02, [(2, 4)]), (0.01, [(0, 1), (0, 1), (2, 2)])]
RULES = [((1, 1), (1, 1)), ((1, 1), (2, 1)), ((1, 2), (1, 2)), ((2, 1), (3, 1)), ((1, 1), (1, 2)), ((3, 0), (4, 0))]


def shifts_of(op, centred):
    """Index shifts at which the matrix of Q^op (0: the kinetic matrix) can be non-zero."""
    reach = op or 2
    return range(-reach, reach + 1, 2 if op == 0 or centred else 1)


@pytest.mark.parametrize("q0,scale", [([0.0] * 3, [1.0] * 3), ([0.3, 0.0, -0.2], [1.3, 0.8, 1.0])])
@pytest.mark.parametrize("nb_rule,nq_rule", RULES)
def test_telescoped_products_equal_the_literal_sum_over_terms(nb_rule, nq_rule, q0, scale):
    D, L = 3, 4
    p = synth.polynomial_problem(D, L, [0.9, 1.1, 1.0], MONOS, nb_rule=nb_rule, nq_rule=nq_rule, q0=q0, scale=scale,
                                 name=f"row form {nb_rule} {nq_rule} {q0}")
    with sg.sg_plan(p) as ctx:
        T = [[sg.sg_mode_tables(ctx, i, l) for l in range(L + 1)] for i in range(D)]
    if nb_rule[1]:
        ks = np.asarray(orc.enumerate_compact(D, L, *nb_rule))
    else:
        ks = np.array(list(itertools.product(range(nb_rule[0]), repeat=D)))
    n, kw = len(ks), int(ks.max()) + 1
    lmin = np.array([next(l for l in range(L + 1) if nb_rule[0] + nb_rule[1] * l > k) for k in range(kw)])

    def deltas(i, op):  # M_i(l) - M_i(l - 1) on kw x kw, all levels; zero outside the stated shifts
        out, last = [], np.zeros((kw, kw))
        for l in range(L + 1):
            t = T[i][l]
            m = t["K"] if op == 0 else t["BW"] @ np.diag(t["Q"] ** op) @ t["B"]
            cur = np.zeros((kw, kw))
            cur[:m.shape[0], :m.shape[1]] = m[:kw, :kw]
            out.append(cur - last)
            last = cur
        allowed = np.zeros((kw, kw), bool)
        for d in shifts_of(op, q0[i] == 0.0):
            allowed |= np.eye(kw, k=d, dtype=bool)
        for m in out:
            # the level's Jacobi matrix is banded: outside the shifts only rounding of B and B^T W
            assert np.abs(m[~allowed]).max(initial=0.0) <= 1e-12 * max(1.0, np.abs(m).max())
            m[~allowed] = 0.0
        return out

    H = np.zeros((n, n))
    products = [(1.0, {i: 0}) for i in range(D)]
    for c, f in MONOS:
        d = {}
        for m, q in f:
            d[m] = d.get(m, 0) + q
        products.append((c, d))
    for c, f in products:
        S = sorted(f)
        D1 = [deltas(i, f[i]) for i in S]
        rest = np.delete(np.arange(D), S)
        room = L - lmin[ks[:, rest]].sum(axis=1)
        same = (ks[:, None, rest] == ks[None, :, rest]).all(axis=2)
        for ls in itertools.product(range(L + 1), repeat=len(S)):
            if sum(ls) > L:
                continue
            v = np.full((n, n), c)
            for a, i in enumerate(S):
                v *= D1[a][ls[a]][ks[:, None, i], ks[None, :, i]]
            H += np.where(same & (sum(ls) <= room)[:, None], v, 0.0)
    if nb_rule[1]:
        R = dense_oracle(p)
    else:  # constant sizes: every term is the same full product, and the D_l sum to 1
        R = np.zeros((n, n))
        for c, f in products:
            t = [T[i][0] for i in range(D)]
            one = [np.eye(kw) if i not in f else t[i]["K"] if f[i] == 0 else
                   t[i]["BW"] @ np.diag(t[i]["Q"] ** f[i]) @ t[i]["B"] for i in range(D)]
            R += c * np.kron(one[0], np.kron(one[1], one[2]))
    tol = literal_elem_tol(p) if nb_rule[1] else 1e-12
    assert np.abs(H - R).max() <= tol * np.abs(R).max()
