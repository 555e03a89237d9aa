"""What sg_size reports for a planned context is what sg_create keeps, from above
and closely (host code on a stand-in device that counts the allocations), tuned
or not; and a plan depends on the potential alone, not on the sizes of terms."""
import itertools

import pytest

import paper_2111_13655_gb300 as sg
from paper_2111_13655_gb300 import synth

import fake_device

FIELD = [(0.02 / (1 + a + b), [(a, 2), (b, 1), (c, 1)]) for a, b, c in itertools.combinations(range(5), 3)]
PROBLEMS = {
    "C1": synth.workload_C1(),
    "C2": synth.workload_C2(),
    "D=12 L=5": synth.workload_C3(L=5),
    "D=12 L=7": synth.workload_C3(L=7),
    "no coupling": synth.chained_henon_heiles(5, 6, [1.0] * 5, 0.0),
    "three-mode field": synth.polynomial_problem(5, 6, [1.0] * 5, FIELD, q0=[0.1, 0.0, -0.1, 0.2, 0.0]),
    "steep levels": synth.chained_henon_heiles(3, 4, synth.draw_omega(3, 2), 0.2, nb_rule=(1, 2), nq_rule=(1, 2)),
    "constant sizes": synth.polynomial_problem(3, 8, [1.0] * 3, [(0.2, [(0, 2), (1, 1)])], nb_rule=(3, 0), nq_rule=(4, 0)),
    "L=64": synth.polynomial_problem(2, 64, [1.0] * 2, [(0.2, [(0, 2), (1, 1)])], nb_rule=(3, 0), nq_rule=(4, 0)),
}


@pytest.fixture()
def fake(tmp_path_factory):
    with fake_device.use(tmp_path_factory.mktemp("fake")) as lib:
        yield lib


@pytest.mark.parametrize("prec", ["fp64", "mixed", "df64"])
@pytest.mark.parametrize("name", list(PROBLEMS))
def test_plan_bounds_what_the_context_holds(fake, name, prec):
    p = PROBLEMS[name]
    if prec == "df64" and name in ("three-mode field", "L=64"):
        pytest.skip("not a double-float problem")
    with sg.sg_plan(p, prec) as ctx:
        plan = sg.sg_size(ctx)["bytes_device"]
    with sg.sg_create(p, prec) as ctx:
        held = sg.sg_size(ctx)["bytes_device"]
        assert fake.fake_live() <= plan
        assert held <= plan <= 1.25 * held + 16384, (held, plan)
        assert fake.sg_tune(ctx.ptr, 2, None, None, None) == sg.SG_OK
        assert sg.sg_size(ctx)["bytes_device"] <= plan
        # the apply workspace apart, tuning leaves nothing behind
        assert fake.fake_live() <= plan + 2 * ctx.n_cs * 64 + 4096


def test_a_pair_potential_has_a_plan_whatever_its_terms_hold(fake):
    """The largest terms of this problem have 2,744 functions or 88,434 grid points, which no kernel keeps in shared memory."""
    p = synth.chained_henon_heiles(4, 5, [1.0] * 4, 0.1, nb_rule=(6, 1), nq_rule=(16, 1))
    with sg.sg_plan(p, "mixed") as ctx:
        plan = sg.sg_tune_plan(ctx)
        assert plan == {"slice_vt": 4, "warp_vt": 4, "smem_kb": 52}
    with sg.sg_create(p, "mixed") as ctx:
        assert sg.sg_tune_plan(ctx) == plan
        assert fake.sg_tune(ctx.ptr, 2, None, None, None) == sg.SG_OK
