"""Error measures and tolerances of the GPU parity tests, and a cached dense
oracle matrix for the propagation checks.

Two measures, both per vector, the worst vector reported:
  norm_rel(y, r) = ||y - r||_2 / ||r||_2
  elem_rel(y, r) = max_i |y_i - r_i| / max_i |r_i|
The element-wise form catches a single wrong entry (a mis-ranked compact
index, a dropped or doubled term) that the 2-norm would dilute by up to
sqrt(N_cs).

FP64 mode: both <= 1e-12 against an exact reference (the masked-Galerkin
closed form where it applies).  The literal oracle sums the terms' D_l y_l in
floating point; at the compact function k = 0, which every term touches, its
own rounding reaches u * sum_l |D_l| * max|y_l| (u = 2^-53): 3.3e-12 of
max|y| at D=12 L=5 against the closed form, measured.  Element-wise
comparisons with the literal oracle therefore allow max(1e-12, u sum_l |D_l|)
(literal_elem_tol); norm-wise stays 1e-12.
Mixed mode: a row's sum is within 6.1 * 2^-24 of the sum of its terms' sizes
(test_row_sums_gpu.py holds every entry to that); the harmonic diagonal, which
is most of H_S, is FP64.  Measured on GB300 over the cases of these tests:
norm-wise and element-wise at most 5.5e-9 for the chained potentials (D=12 L=10:
1.5e-9 and 4.2e-9) and 4.9e-8 for the general polynomial, whose shifted modes
have no FP64 part.  MIXED_TOL = MIXED_ELEM_TOL = 4e-7 is eight times that.
(Problems applied term by term, where the D_l sum the terms' rounding, state
their own tolerances.)
Double-float mode: each step of a row's sum is within a few 2^-48 of its
operands (test_df_arith.py).  Measured against the exact closed form: norm-wise
4.4e-16 and element-wise 1.7e-15 at most; against the literal oracle, whose own
rounding dominates (FP64 shows the same), 5.5e-15 and 2.4e-14.  DF64_TOL = 5e-14
and DF64_ELEM_TOL = 2e-13 are eight times the latter.
"""
import numpy as np

FP64_TOL = 1e-12
MIXED_TOL = 4e-7
MIXED_ELEM_TOL = 4e-7
DF64_TOL = 5e-14
DF64_ELEM_TOL = 2e-13


def literal_elem_tol(p):
    """Element-wise FP64 tolerance against the literal oracle: its own
    floating-point compress-add bound u * sum_l |D_l| (Eq. (8)), at least 1e-12."""
    from oracle import oracle as orc
    _, c = orc.enumerate_terms(p.D, p.L)
    return max(FP64_TOL, 2.0 ** -53 * float(np.abs(np.asarray(c, float)).sum()))


def norm_rel(y, r):
    y = np.atleast_2d(y); r = np.atleast_2d(r)
    return float(np.max(np.linalg.norm(y - r, axis=1) / np.linalg.norm(r, axis=1)))


def elem_rel(y, r):
    y = np.atleast_2d(y); r = np.atleast_2d(r)
    return float(np.max(np.max(np.abs(y - r), axis=1) / np.max(np.abs(r), axis=1)))


def assert_parity(y, r, precision, what=""):
    """Both measures within the tolerances of `precision` ("fp64", "df64" or "mixed")."""
    n, e = norm_rel(y, r), elem_rel(y, r)
    if precision == "fp64":
        assert n <= FP64_TOL and e <= FP64_TOL, f"{what}: norm-wise {n:.3e}, element-wise {e:.3e}"
    elif precision == "df64":
        assert n <= DF64_TOL and e <= DF64_ELEM_TOL, f"{what}: norm-wise {n:.3e}, element-wise {e:.3e}"
    else:
        assert n <= MIXED_TOL and e <= MIXED_ELEM_TOL, f"{what}: norm-wise {n:.3e}, element-wise {e:.3e}"
    return n, e


_DENSE = {}


def dense_oracle(p):
    """H_S of problem p as a dense symmetric matrix, column j = H_S e_j, from
    the literal CPU oracle (symmetrised: H_S is symmetric, Sec. 2); cached per
    problem name within a test process."""
    from oracle import oracle as orc
    key = (p.name, p.D, p.L, tuple(np.asarray(p.omega).round(15)), tuple(np.asarray(p.coef).round(15)))
    if key not in _DENSE:
        n = orc.n_compact(p)
        H = orc.apply_H(p, np.eye(n)).T
        _DENSE[key] = 0.5 * (H + H.T)
    return _DENSE[key]


def exact_propagator(H):
    """(w, U) with H = U diag(w) U^T, for psi(t) = U exp(-i w t) U^T psi(0)."""
    return np.linalg.eigh(H)
