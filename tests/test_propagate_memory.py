"""sg_propagate's device memory (host code on a stand-in device): inner products
are kept for the steps that are logged, and without a log nothing grows with
the number of steps."""
import numpy as np
import pytest

import paper_2111_13655_gb300 as sg
from paper_2111_13655_gb300 import synth

import fake_device


@pytest.fixture()
def fake(tmp_path_factory):
    with fake_device.use(tmp_path_factory.mktemp("fake")) as lib:
        yield lib


@pytest.mark.parametrize("logged", [(False, False), (True, False), (False, True), (True, True)])
def test_memory_of_a_long_propagation(fake, logged):
    with sg.sg_create(synth.workload_C1(), "fp64") as ctx:
        psi = np.zeros(2 * ctx.n_cs)
        assert fake.sg_propagate(ctx.ptr, psi.ctypes.data, 0.1, 1, 2, None, None, None) == sg.SG_OK  # the context's workspace
        peak = {}
        for steps in (1, 20000):
            logs = [np.zeros(steps) for _ in logged]
            at = [v.ctypes.data if on else None for v, on in zip(logs, logged)]
            fake.fake_clear_peak()
            before = fake.fake_live()
            assert fake.sg_propagate(ctx.ptr, psi.ctypes.data, 0.1, steps, 2, *at, None) == sg.SG_OK
            peak[steps] = fake.fake_peak() - before
            assert fake.fake_live() == before
    assert peak[20000] - peak[1] <= (8 * 8 * 20000 if any(logged) else 0)
