"""Forming the row operator: elements of wide products against the oracle (rows
of no, one and many chunks of entries), and set-up time in proportion to the
host's planning for potentials whose products touch many modes."""
import itertools
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2111_13655_gb300 as sg
from oracle import oracle as orc
from paper_2111_13655_gb300 import synth

from helpers import elem_rel, literal_elem_tol, norm_rel

pytestmark = pytest.mark.gpu


def field(D, L, powers, nq=2):
    monos = [(0.01 / (1 + sum(e)), [(i, q) for i, q in zip(m, e)]) for m, e in powers]
    return synth.polynomial_problem(D, L, np.linspace(0.9, 1.1, D), monos, nb_rule=(1, 1), nq_rule=(nq, 1),
                                    q0=[0.1 * (1 + i) for i in range(D)])


SIX = [(tuple(range(6)), e) for e in itertools.product((1, 2), repeat=6)]
CASES = {
    "six modes": field(6, 5, SIX),
    "six modes, inexact quadrature": field(6, 4, SIX, nq=1),
    "five of seven modes": field(7, 5, [(m, (1,) * 5) for m in itertools.combinations(range(7), 5)]),
    "one mode, rows of 1 to 21": field(1, 25, [((0,), (10,))]),
    "a constant": synth.polynomial_problem(3, 4, [1.0] * 3, [(0.5 * 1.0, [(i, 2)]) for i in range(3)] + [(0.7, [])]),
    "nothing but the harmonic diagonal": synth.chained_henon_heiles(4, 5, [1.0] * 4, 0.0),
}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", list(CASES))
def test_elements_match_the_oracle(name, prec):
    p = CASES[name]
    with sg.sg_create(p, prec) as ctx:
        xh = synth.random_vectors(ctx.n_cs, 3, 5)
        x = torch.from_numpy(xh).cuda()
        y = torch.empty_like(x)
        sg.sg_apply_H(ctx, x, y, 3)
        torch.cuda.synchronize()
        assert sg.sg_device_error(ctx) == 0
    r = orc.apply_H(p, xh)
    n, e = norm_rel(y.cpu().numpy(), r), elem_rel(y.cpu().numpy(), r)
    tol = literal_elem_tol(p) if prec == "fp64" else 5e-6
    assert n <= tol and e <= tol, (n, e)


def test_set_up_of_many_mode_products_takes_about_as_long_as_their_plan():
    """64 six-mode products over 3,003 functions: 11 ms of which the plan is 6 (a warp per row that summed over all
    levels took 64)."""
    p = field(6, 8, SIX)

    def best(make):
        t = []
        for _ in range(3):
            t0 = time.perf_counter()
            sg.sg_destroy(make(p, "fp64"))
            t.append(time.perf_counter() - t0)
        return min(t)

    sg.sg_destroy(sg.sg_create(p, "fp64"))
    plan, create = best(sg.sg_plan), best(sg.sg_create)
    assert create <= 5.0 * plan, (create, plan)
