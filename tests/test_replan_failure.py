"""sg_tune when device memory runs out (host code on a stand-in device): a plan
whose row operator cannot be allocated is not taken, the context keeps the
operator it has and goes on applying it, and no batch reads a released one."""
import ctypes

import numpy as np
import pytest

import paper_2111_13655_gb300 as sg
from paper_2111_13655_gb300 import synth

import fake_device


@pytest.fixture()
def fake(tmp_path_factory):
    with fake_device.use(tmp_path_factory.mktemp("fake")) as lib:
        yield lib


def apply(lib, ctx, x):
    y = np.full_like(x, np.nan)
    st = lib.sg_apply_H(ctx.ptr, x.ctypes.data, y.ctypes.data, x.shape[0], None)
    return st, y


def tune(lib, ctx):
    return lib.sg_tune(ctx.ptr, 2, None, None, None)


@pytest.mark.parametrize("prec", ["fp64", "mixed", "df64"])
def test_a_plan_that_does_not_fit_leaves_the_context_as_it_was(fake, prec):
    p = synth.workload_C3(L=5)
    with sg.sg_create(p, prec) as ctx:
        x = synth.random_vectors(ctx.n_cs, 2, 1)
        st, want = apply(fake, ctx, x)
        assert st == sg.SG_OK and np.isfinite(want).all()
        op = sg.sg_size(ctx)["bytes_device"] // 2        # the row operator is most of what a context holds
        fake.fake_fail_after(-1, op)
        assert tune(fake, ctx) == sg.SG_OK
        builds = fake.fake_matching()
        assert builds >= 3
        plan = sg.sg_tune_plan(ctx)
        # no new operator, one and then the rest not, all but the last (back to the fastest plan)
        for n in (0, 1, builds - 1):
            fake.fake_fail_after(n, op)
            st = tune(fake, ctx)
            fake.fake_fail_after(-1, op)
            assert st == sg.SG_OK if n == 0 else st in (sg.SG_OK, sg.SG_ENOMEM)
            st, y = apply(fake, ctx, x)
            assert st == sg.SG_OK and np.array_equal(y, want), n
            kept = sg.sg_tune_plan(ctx)
            if n == 0:
                # the plan in force is that of the operator in force: nothing could replace it
                assert (kept["warp_vt"], kept["smem_kb"]) == (plan["warp_vt"], plan["smem_kb"])
        assert tune(fake, ctx) == sg.SG_OK and np.array_equal(apply(fake, ctx, x)[1], want)


@pytest.mark.parametrize("done", [0, 1])
def test_a_batch_refuses_after_a_re_plan_that_failed_half_way(fake, done):
    p = synth.workload_C3(L=5)
    with sg.sg_create(p, "fp64") as ctx:
        x = synth.random_vectors(ctx.n_cs, 2, 1)
        y = np.empty_like(x)
        op = sg.sg_size(ctx)["bytes_device"] // 2
        b = ctypes.c_void_p()
        ptrs = (ctypes.c_void_p * 1)(ctx.ptr)
        assert fake.sg_batch_create(ctypes.addressof(ptrs), 1, ctypes.byref(b)) == sg.SG_OK
        assert fake.sg_apply_H_batch(b, x.ctypes.data, y.ctypes.data, 2, None) == sg.SG_OK
        fake.fake_fail_after(done, op)                    # the operators formed before memory runs out
        tune(fake, ctx)
        fake.fake_fail_after(-1, op)
        n = fake.fake_launches(b"rows_batch")
        assert fake.sg_apply_H_batch(b, x.ctypes.data, y.ctypes.data, 2, None) == sg.SG_EINVAL
        assert b"recreate" in fake.sg_batch_last_error(b) and fake.fake_launches(b"rows_batch") == n
        fake.sg_batch_destroy(b)
