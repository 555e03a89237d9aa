"""Problems applied term by term beside problems in the row form: in one batch,
and as requests of one server.  nb(l) = 3, nq(l) = 4 at every level with L = 64,
which the row form is not built for; 27 functions, 6,241 equal terms."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2111_13655_gb300 as sg
from paper_2111_13655_gb300 import synth

pytestmark = pytest.mark.gpu

TERMS = synth.polynomial_problem(3, 64, [0.9, 1.1, 1.0], [(0.2, [(0, 2), (1, 1)]), (0.05, [(0, 1), (1, 1), (2, 1)])],
                                 nb_rule=(3, 0), nq_rule=(4, 0), q0=[0.3, 0.0, -0.2])
ROWS = [synth.workload_C1(), synth.chained_henon_heiles(6, 6, synth.draw_omega(6, 21), synth.HH_LAMBDA)]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_a_batch_of_both_forms_equals_each_context_bitwise(prec):
    ctxs = [sg.sg_create(p, prec) for p in (ROWS[0], TERMS, ROWS[1], TERMS)]
    b = sg.sg_batch_create(ctxs)
    try:
        for call, nvec in enumerate((3, 5, 2)):
            xs = [torch.from_numpy(synth.random_vectors(c.n_cs, nvec, 10 * call + j)).cuda().contiguous().view(-1)
                  for j, c in enumerate(ctxs)]
            want = []
            for c, x in zip(ctxs, xs):
                want.append(torch.empty_like(x))
                sg.sg_apply_H(c, x, want[-1], nvec)
            y = torch.full((sum(x.numel() for x in xs),), float("nan"), dtype=torch.float64, device="cuda")
            x = torch.cat(xs)
            for _ in range(2):
                sg.sg_apply_H_batch(b, x, y, nvec)
                torch.cuda.synchronize()
                assert torch.equal(y, torch.cat(want)), (call, nvec)
        assert all(sg.sg_device_error(c) == 0 for c in ctxs)
    finally:
        sg.sg_batch_destroy(b)
        for c in ctxs:
            sg.sg_destroy(c)


def state(p):
    with sg.sg_plan(p) as c:
        psi = synth.random_vectors(c.n_cs, 1, 5)[0].astype(complex)
    return psi / np.linalg.norm(psi)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_server_requests_of_both_forms_equal_themselves_alone(prec):
    """Alone, the row form's requests take a launch per Chebyshev term; beside one applied term by term, an apply and
    an update."""
    problems = {"terms": (TERMS, 2), "small": (ROWS[0], 6), "rows": (ROWS[1], 4)}
    psi0 = {k: state(p) for k, (p, _) in problems.items()}
    alone = {}
    for k, (p, steps) in problems.items():
        with sg.Server(prec) as srv:
            rid = srv.submit(p, 0.05, steps, order=32, psi0=psi0[k])
            srv.run()
            alone[k] = srv.result(rid)[:3]
    with sg.Server(prec) as srv:
        ids = {"rows": srv.submit(problems["rows"][0], 0.05, problems["rows"][1], order=32, psi0=psi0["rows"])}
        srv.progress(5)
        for k in ("terms", "small"):
            ids[k] = srv.submit(problems[k][0], 0.05, problems[k][1], order=32, psi0=psi0[k])
        srv.run()
        for k, rid in ids.items():
            for got, want in zip(srv.result(rid)[:3], alone[k]):
                assert np.array_equal(got, want), k
        assert srv.stats()["bytes_in_use"] == 0
    # and the one applied term by term is a unitary propagation
    assert np.abs(alone["terms"][1] - 1.0).max() <= (1e-11 if prec == "fp64" else 1e-4)
