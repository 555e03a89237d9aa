"""The row kernels where their dispatch changes: lanes and passes over the
vectors, input gathered directly or from the entry-major copy, vectors settled
by the last block or by a launch of their own, rows too long for shared memory,
non-finite input on every entry point, problems outside the row form, and the
solver kernels on both sides of their size rule.

A row's sum is made in one order whatever the block size and entry point, so
these are compared bitwise; parity is with the closed form or a dense matrix,
within the tolerances of helpers.py.
"""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2111_13655_gb300 as sg
from oracle import galerkin
from oracle import oracle as orc
from paper_2111_13655_gb300 import synth

from helpers import FP64_TOL, assert_parity, elem_rel, literal_elem_tol, norm_rel

pytestmark = pytest.mark.gpu

# N_cs 924: 17 vectors gathered directly, few windows.  12,870: 5 vectors
# gathered directly, 7 from the copy, the last block settles.  125,970: the copy
# and about 2,000 windows, settled by a launch.
SIZES = {"D=6 L=6": synth.workload_C3(L=6, D=6), "D=8 L=8": synth.workload_C3(L=8, D=8),
         "D=12 L=8": synth.workload_C3(L=8)}


def apply(ctx, x):
    y = torch.full_like(x, float("nan"))
    sg.sg_apply_H(ctx, x, y, x.shape[0])
    return y


@pytest.mark.parametrize("prec", ["fp64", "mixed", "df64"])
@pytest.mark.parametrize("name", list(SIZES))
def test_every_block_size_equals_single_vectors_bitwise(name, prec):
    p = SIZES[name]
    with sg.sg_create(p, prec) as ctx:
        xh = synth.random_vectors(ctx.n_cs, 17, 41)
        x = torch.from_numpy(xh).cuda()
        one = torch.cat([apply(ctx, x[v:v + 1]) for v in range(17)])
        for nvec in (2, 3, 4, 5, 6, 7, 8, 9, 12, 16, 17):
            assert torch.equal(apply(ctx, x[:nvec]), one[:nvec]), nvec
        assert sg.sg_device_error(ctx) == 0
    assert_parity(one[:2].cpu().numpy(), galerkin.apply_H(p, xh[:2]), prec, name)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_rows_longer_than_the_staged_record(prec):
    """Dense coupling in off-centre modes: rows of up to 2,026 entries, some of them beyond a block's share of
    shared memory (read in place)."""
    monos = [(0.01 / (1 + a + b + c), [(0, a), (1, b), (2, c)]) for a, b, c in itertools.product((5, 6), repeat=3)]
    p = synth.polynomial_problem(3, 28, [1.0, 0.9, 1.1], monos, nb_rule=(1, 1), nq_rule=(2, 1), q0=[0.1, -0.1, 0.2])
    with sg.sg_create(p, prec) as ctx:
        xh = synth.random_vectors(ctx.n_cs, 3, 5)
        x = torch.from_numpy(xh).cuda()
        y = apply(ctx, x)
        assert torch.equal(apply(ctx, x[1:2]), y[1:2])
        assert sg.sg_device_error(ctx) == 0
    r = orc.apply_H(p, xh)
    n, e = norm_rel(y.cpu().numpy(), r), elem_rel(y.cpu().numpy(), r)
    tol = literal_elem_tol(p) if prec == "fp64" else 5e-6
    assert n <= tol and e <= tol, (n, e)


@pytest.mark.parametrize("name", ["D=6 L=6", "D=8 L=8", "D=12 L=8"])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_one_non_finite_entry_makes_its_vector_nan_on_every_entry_point(name, prec, bad):
    p, nvec = SIZES[name], 7
    with sg.sg_create(p, prec) as ctx:
        n = ctx.n_cs
        x = torch.from_numpy(synth.random_vectors(n, nvec, 8)).cuda()
        clean = apply(ctx, x)
        z = x.clone()
        z[2, n - 1] = bad
        z[5, 0] = bad

        def part_sum():
            y = torch.empty_like(z)
            total = torch.zeros(sg.acc_words(ctx, nvec), dtype=torch.int64, device="cuda")
            for part in range(2):
                acc = torch.zeros_like(total)
                sg.sg_apply_H_part(ctx, z, acc, nvec, part, 2)
                total += acc
            sg.sg_apply_H_finish(ctx, z, total, y, nvec)
            return y

        def batched():
            y = torch.empty_like(z)
            b = sg.sg_batch_create([ctx])
            try:
                sg.sg_apply_H_batch(b, z.view(-1), y.view(-1), nvec)
                torch.cuda.synchronize()
            finally:
                sg.sg_batch_destroy(b)
            return y

        def noalloc():
            y = torch.empty_like(z)
            sg.sg_apply_H_noalloc(ctx, z, y, nvec)
            return y

        routes = [lambda: apply(ctx, z), part_sum, batched]
        if n * nvec <= 524272:
            routes.append(noalloc)
        keep = [v for v in range(nvec) if v not in (2, 5)]
        for route in routes:
            y = route()
            torch.cuda.synchronize()
            assert sg.sg_device_error(ctx) == 201
            assert torch.isnan(y[[2, 5]]).all() and torch.equal(y[keep], clean[keep])
            assert torch.equal(apply(ctx, x), clean)      # nothing is left behind
            assert sg.sg_device_error(ctx) == 0


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_subnormal_and_extreme_scales(prec):
    """Powers of two scale the result exactly as long as nothing leaves the value type's normal range; below it the
    sum is still that of the rounded values."""
    p = SIZES["D=6 L=6"]
    with sg.sg_create(p, prec) as ctx:
        x = torch.from_numpy(synth.random_vectors(ctx.n_cs, 3, 9)).cuda()
        y = apply(ctx, x)
        for k in (60, -60):
            assert torch.equal(apply(ctx, x * 2.0 ** k), y * 2.0 ** k)
        tiny = apply(ctx, x * 2.0 ** -135)                # FP32: subnormal inputs, spacing 2^-149
        # each of a row's m entries is off by half a spacing times |H_kk'|; ||H|| bounds them together
        h = float((y.norm(dim=1) / x.norm(dim=1)).max())
        tol = (2.0 ** -150 * 64 * max(1.0, h) * 40 if prec == "mixed" else 0.0) + 1e-6 * 2.0 ** -135 * float(y.abs().max())
        assert float((tiny - y * 2.0 ** -135).abs().max()) <= tol
        assert sg.sg_device_error(ctx) == 0


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("D,L", [(2, 70), (3, 64), (2, 63), (3, 5)])
def test_constant_basis_sizes_inside_and_outside_the_row_form(D, L, prec):
    """nb(l) = 3, nq(l) = 4 at every level: all terms are the same full product and the D_l sum to 1, so H_S is that
    product's matrix whatever L.  L > 63 goes term by term; every entry point agrees bitwise."""
    monos = [(0.2, [(0, 2), (1, 1)]), (0.1, [(D - 1, 3)]), (0.3, []), (0.05, [(i, 1) for i in range(D)])]
    p = synth.polynomial_problem(D, L, [0.9, 1.1, 1.0][:D], monos, nb_rule=(3, 0), nq_rule=(4, 0),
                                 q0=[0.3, 0.0, -0.2][:D], scale=[1.3, 0.8, 1.0][:D])
    nvec = 3
    with sg.sg_create(p, prec) as ctx:
        t = [sg.sg_mode_tables(ctx, i, 0) for i in range(D)]
        H = np.zeros((3 ** D, 3 ** D))
        for c, f in [(1.0, [(i, 0)]) for i in range(D)] + monos:
            m = np.eye(1)
            for i in range(D):
                o = np.eye(3)
                for j, q in f:
                    if j == i:
                        o = t[i]["K"] if q == 0 else t[i]["BW"] @ np.diag(t[i]["Q"] ** q) @ t[i]["B"]
                m = np.kron(m, o)
            H += c * m
        assert ctx.n_cs == 3 ** D
        xh = synth.random_vectors(ctx.n_cs, nvec, 3)
        x = torch.from_numpy(xh).cuda()
        y = apply(ctx, x)
        z = torch.empty_like(x)
        sg.sg_apply_H_noalloc(ctx, x, z, nvec)
        assert torch.equal(z, y)
        b = sg.sg_batch_create([ctx, ctx])
        x2, z2 = x.repeat(2, 1), torch.empty((2 * nvec, ctx.n_cs), dtype=torch.float64, device="cuda")
        sg.sg_apply_H_batch(b, x2.view(-1), z2.view(-1), nvec)
        torch.cuda.synchronize()
        sg.sg_batch_destroy(b)
        assert torch.equal(z2[:nvec], y) and torch.equal(z2[nvec:], y)
        acc = torch.zeros(sg.acc_words(ctx, nvec), dtype=torch.int64, device="cuda")
        for part in range(2):
            sg.sg_apply_H_part(ctx, x, acc, nvec, part, 2)
        sg.sg_apply_H_finish(ctx, x, acc, z, nvec)
        torch.cuda.synchronize()
        assert torch.equal(z, y) and sg.sg_device_error(ctx) == 0
        r = xh @ H.T
        # (equal terms: their rounding is the same, and the D_l sum it to that of one)
        assert elem_rel(y.cpu().numpy(), r) <= (FP64_TOL if prec == "fp64" else 5e-6)


# N_cs 8,008, 27,132 and 74,613: one, two and five chunks per inner product; grouped and plain column sums
@pytest.mark.parametrize("D,L", [(6, 10), (6, 13), (6, 16)])
def test_solvers_with_products_in_one_and_in_several_chunks(D, L):
    p = synth.chained_henon_heiles(D, L, synth.draw_omega(D, 6), 0.1)
    nev, tol = 5, 1e-9
    with sg.sg_create(p, "fp64") as ctx:
        assert (ctx.n_cs <= 16384) == (L == 10)
        ev, rn, vec, _ = sg.sg_eigs(ctx, nev, "davidson", block=4, tol=tol, max_it=300, vectors=True)
        v = vec.view(nev, ctx.n_cs)
        r = apply(ctx, v) - torch.from_numpy(np.asarray(ev)).cuda()[:, None] * v
        # the returned residuals are those of the returned pairs, up to the rounding of H v
        assert float(r.norm(dim=1).max()) <= tol * max(1.0, float(np.max(np.abs(ev)))) + 1e-11
        assert float((v @ v.T - torch.eye(nev, dtype=torch.float64, device="cuda")).abs().max()) <= 1e-12
        psi = torch.zeros(2 * ctx.n_cs, dtype=torch.float64, device="cuda")
        psi[:ctx.n_cs] = v[0]
        norm, energy = sg.sg_propagate(ctx, psi, 0.1, 5)
        # an eigenstate: norm and energy stay, the vector turns by e^{-i E t}
        assert np.abs(np.asarray(norm) - 1.0).max() <= 1e-11 and np.abs(np.asarray(energy) - ev[0]).max() <= 1e-10
        c, s = np.cos(0.5 * ev[0]), np.sin(0.5 * ev[0])
        want = torch.cat([c * v[0], -s * v[0]])
        assert float((psi - want).abs().max()) <= 1e-8    # residual 1e-9 times the time, and rounding


@pytest.mark.parametrize("prec", ["fp64", "mixed", "df64"])
@pytest.mark.parametrize("name", list(SIZES))
def test_captured_applies_replay_bitwise(name, prec):
    """The launches wait for one another on the device; in a caller's graph, with a kernel of the caller's before and
    after each apply, they keep that order (x is overwritten in between)."""
    p, nvec = SIZES[name], 5
    with sg.sg_create(p, prec) as ctx:
        x0 = torch.from_numpy(synth.random_vectors(ctx.n_cs, nvec, 12)).cuda()
        want1 = apply(ctx, x0)
        want2 = apply(ctx, want1 * 0.125)
        x, y = torch.zeros_like(x0), torch.zeros_like(x0)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            s = torch.cuda.current_stream()
            sg.sg_apply_H(ctx, x, y, nvec, stream=s)
            first = y.clone()
            x.copy_(y * 0.125)
            sg.sg_apply_H(ctx, x, y, nvec, stream=s)
        for _ in range(3):
            x.copy_(x0)
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(first, want1) and torch.equal(y, want2)
        assert sg.sg_device_error(ctx) == 0
