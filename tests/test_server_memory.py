"""The server's admission counts what a request holds on the device (host code on
a stand-in device that counts the allocations): the planned bytes of the active
requests, which stay within the budget, cover the live allocations."""
import itertools
import re

import numpy as np
import pytest

import paper_2111_13655_gb300 as sg
from paper_2111_13655_gb300 import synth

import fake_device

# three-mode terms; a pair potential; L > 63 (applied term by term)
FIELD = synth.polynomial_problem(8, 7, [1.0] * 8, [(0.01, [(a, 1), (b, 1), (c, 1)])
                                                   for a, b, c in itertools.combinations(range(8), 3)])
PAIRS = synth.workload_C3(L=6)
TERMS = synth.polynomial_problem(3, 64, [1.0] * 3, [(0.2, [(0, 2), (1, 1)])], nb_rule=(10, 0), nq_rule=(10, 0))
PROBLEMS = {"field": FIELD, "pairs": PAIRS}


@pytest.fixture()
def fake(tmp_path_factory):
    with fake_device.use(tmp_path_factory.mktemp("fake")) as lib:
        yield lib


def needed(prec, submit):
    """Planned bytes of a request, from the refusal of a server that has one byte."""
    with sg.Server(prec, hbm_budget_bytes=1) as srv, pytest.raises(sg.SgError) as ei:
        submit(srv)
    assert ei.value.status == sg.SG_EBUDGET
    return int(re.search(r"needs (\d+) bytes", str(ei.value)).group(1))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("nev,block,vectors", [(1, 1, False), (10, 4, True), (100, 8, False)])
@pytest.mark.parametrize("name", list(PROBLEMS))
def test_an_eigen_request_is_counted_whole(fake, name, nev, block, vectors, prec):
    submit = lambda srv: srv.submit_eigs(PROBLEMS[name], nev, block=block, tol=1e-6, max_it=5, vectors=vectors)
    need = needed(prec, submit)
    assert fake.fake_live() == 0
    fake.fake_clear_peak()
    with sg.Server(prec, hbm_budget_bytes=need) as srv:
        submit(srv)
        while srv.progress(1) != (0, 0):    # (no arithmetic on this device: the request ends at its first step)
            pass
    peak = fake.fake_peak()
    assert peak <= need <= 1.5 * peak + (1 << 20), (peak, need)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("order", [8, 200000])
@pytest.mark.parametrize("mix", [["field"], ["pairs"], ["pairs", "field"], ["terms"], ["terms", "pairs"]])
def test_propagation_requests_are_counted_whole(fake, mix, order, prec):
    problems = [dict(PROBLEMS, terms=TERMS)[m] for m in mix]
    psi0 = []
    for p in problems:
        with sg.sg_plan(p, prec) as ctx:
            psi0.append(np.ones(ctx.n_cs, complex))
    submit = [lambda srv, p=p, v=v: srv.submit(p, 0.1, 3, order=order, psi0=v) for p, v in zip(problems, psi0)]
    need = sum(needed(prec, f) for f in submit)
    with sg.Server(prec, hbm_budget_bytes=need) as srv:
        for f in submit:
            f(srv)
        srv.progress(1)
        srv.progress(1)
        assert srv.stats()["bytes_in_use"] == need
        live = fake.fake_live()
    assert live <= need <= 2 * live + len(mix) * (1 << 20), (live, need)
    assert fake.fake_live() == 0
