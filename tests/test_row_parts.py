"""The parts of a sharded apply in the row form (host code on a stand-in device):
every row belongs to one part, whatever the number of parts, the parts hold
about the same number of entries, and sg_part_size says how many."""
import numpy as np
import pytest

import paper_2111_13655_gb300 as sg
from paper_2111_13655_gb300 import synth

import fake_device


@pytest.fixture()
def fake(tmp_path_factory):
    with fake_device.use(tmp_path_factory.mktemp("fake")) as lib:
        yield lib


# 2, 188, 403 and about 2,000 windows: the largest part is within a few windows of the mean
@pytest.mark.parametrize("p,spread", [(synth.workload_C1(), None), (synth.workload_C2(), 1.1),
                                      (synth.workload_C3(L=8, D=8), 1.1), (synth.workload_C3(L=8), 1.02)],
                         ids=["D=2 L=6", "D=6 L=8", "D=8 L=8", "D=12 L=8"])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_parts_cover_every_row_once_and_balance_the_entries(fake, p, spread, prec):
    nvec = 2
    with sg.sg_create(p, prec) as ctx:
        x = np.ones((nvec, ctx.n_cs))
        words = sg.acc_words(ctx, nvec) // (ctx.n_cs * nvec)
        for nparts in (1, 2, 3, 8):
            acc, entries, counted = np.zeros((ctx.n_cs, nvec, words), np.int64), [], []
            for part in range(nparts):
                before = fake.fake_entries()
                assert fake.sg_apply_H_part(ctx.ptr, x.ctypes.data, nvec, part, nparts, acc.ctypes.data, None) == sg.SG_OK
                entries.append(fake.fake_entries() - before)
                rows = int((acc[:, 0, 0] == 1).sum()) - sum(counted)
                assert sg.sg_part_size(ctx, part, nparts) == (rows, entries[-1])
                counted.append(rows)
            assert (acc[:, :, 0] == 1).all() and not acc[:, :, 1:].any(), nparts
            if spread:
                assert max(entries) <= spread * np.mean(entries), (nparts, entries)
