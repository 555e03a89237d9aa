"""sg_create when the row operator does not fit the device's free memory (host
code on a stand-in device): FP64 and mixed contexts are applied term by term,
which needs a small part of it; double-float has no such kernel and reports
SG_ENOMEM.  Nothing stays allocated either way."""
import ctypes
import itertools

import numpy as np
import pytest

import paper_2111_13655_gb300 as sg
from paper_2111_13655_gb300 import synth

import fake_device

# three-mode terms (wide rows), and a pair potential
FIELD = synth.polynomial_problem(4, 6, [1.0, 0.9, 1.1, 1.0],
                                 [(0.01, [(a, 2), (b, 2), (c, 1)]) for a, b, c in itertools.permutations(range(4), 3)],
                                 q0=[0.1, -0.1, 0.2, 0.0])
PAIRS = synth.workload_C3(L=5)


@pytest.fixture()
def fake(tmp_path_factory):
    with fake_device.use(tmp_path_factory.mktemp("fake")) as lib:
        yield lib


def operator_bytes(lib, p, prec):
    """The row operator's allocation, the largest that a context makes."""
    lib.fake_clear_peak()
    with sg.sg_create(p, prec):
        return lib.fake_largest()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("p", [FIELD, PAIRS], ids=["field", "pairs"])
def test_without_memory_for_the_rows_the_terms_are_applied(fake, p, prec):
    fake.fake_fail_after(0, operator_bytes(fake, p, prec))
    before = fake.fake_live()
    with sg.sg_create(p, prec) as ctx:
        assert sg.sg_size(ctx)["bytes_device"] == fake.fake_live() - before
        x = synth.random_vectors(ctx.n_cs, 2, 1)
        y = np.empty_like(x)
        fake.fake_fail_after(-1, 0)
        rows = fake.fake_launches(b"rows")
        assert fake.sg_apply_H(ctx.ptr, x.ctypes.data, y.ctypes.data, 2, None) == sg.SG_OK
        b = ctypes.c_void_p()
        ptrs = (ctypes.c_void_p * 1)(ctx.ptr)
        assert fake.sg_batch_create(ctypes.addressof(ptrs), 1, ctypes.byref(b)) == sg.SG_OK
        assert fake.sg_apply_H_batch(b, x.ctypes.data, y.ctypes.data, 2, None) == sg.SG_OK
        fake.sg_batch_destroy(b)
        assert fake.fake_launches(b"terms") == 2 and fake.fake_launches(b"rows") == rows
        assert fake.sg_tune(ctx.ptr, 2, None, None, None) == sg.SG_OK and sg.sg_tune_plan(ctx)["slice_vt"] == 0
    assert fake.fake_live() == before


def test_double_float_without_memory_is_refused(fake):
    fake.fake_fail_after(0, operator_bytes(fake, PAIRS, "df64"))
    with pytest.raises(sg.SgError) as ei:
        sg.sg_create(PAIRS, "df64")
    assert ei.value.status == sg.SG_ENOMEM and fake.fake_live() == 0


@pytest.mark.parametrize("prec", ["fp64", "mixed", "df64"])
def test_without_any_memory_the_context_is_refused(fake, prec):
    fake.fake_fail_after(0, 0)
    with pytest.raises(sg.SgError) as ei:
        sg.sg_create(PAIRS, prec)
    assert ei.value.status == sg.SG_ENOMEM and fake.fake_live() == 0
