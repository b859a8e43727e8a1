"""Products with matrices shared by classes of cells, macro elements and vertex
patches, against the general forms (every block its own) on the GPU.

DPGMG_FLAG_RECOMPUTE_PATCHES keeps every block separate, so a system set up
with it runs the general kernels on the same matrices: the smoother's FP32
factors are the same and the products differ by FP32 rounding order only.
Tolerances: complex64 sums of up to 8 x 302 terms, 2^-24 each in a random walk
over cancelling terms, 1e-5; the V-cycle as elsewhere against the oracle.  The
CG operator takes x as two FP32 parts (2^-48) and sums at most 8 x 302 products
of at least 2^-46, with cancellation up to 100: 1e-12 of complex128.
"""
import numpy as np
import pytest

from paper_2304_01728_gb300 import dpgmg as D
from tests.oracle_adapter import MIXED_THETA_TOL, MIXED_VCYCLE_TOL, rand_vec, rel

pytestmark = pytest.mark.gpu


def layers(n, seed):
    c = np.random.default_rng(seed).choice([0.4, 0.7, 1.0], n[2])
    return np.repeat(c, n[0] * n[1])


CASES = [   # n, p, wavespeed layers, levels, p_min, flags
    ((9, 7, 6), 1, False, 1, 1, 0),               # one level below the finest only; 14 local functions
    ((8, 8, 8), 2, False, 3, 1, 0),
    ((16, 8, 4), 2, True, 3, 2, 0),               # h levels, classes of few cells
    ((8, 8, 8), 3, False, 3, 2, 0),
    ((8, 8, 4), 3, True, 3, 2, D.FLAG_COMPLEX_STORAGE),
    ((12, 6, 5), 3, True, 2, 2, 0),               # odd extents
    ((6, 6, 6), 4, False, 2, 3, 0),               # two column chunks in the CG operator
    ((5, 4, 6), 5, False, 2, 4, 0),               # three
]


def solver(case, flags=0, precision="mixed"):
    n, p, lay, nl, p_min, fl = case
    pk = dict(n=n, p=p, omega=4.0, src_center=(0.4, 0.55, 0.5), src_width=0.2)
    if lay:
        pk["wavespeed"] = layers(n, sum(n))
    return D.Solver(pk, n_levels=nl, p_min=p_min, precision=precision, tol=1e-8, flags=fl | flags)


@pytest.mark.parametrize("case", [c for c in CASES if c[3] > 1])
def test_class_products_against_separate_blocks(case):
    with solver(case) as s0, solver(case, D.FLAG_RECOMPUTE_PATCHES) as s1:
        for l in range(1, case[3]):
            g0, g1 = s0.level(l), s1.level(l)
            n, nc = g0.n_dof, s0.level(l - 1).n_dof
            x, xc = rand_vec(n, 7 + l), rand_vec(nc, 9 + l)
            a0 = D.dpgmg_apply(s0.h, s0.s, D.OP_A, l, x, n)
            assert rel(a0, D.dpgmg_apply(s1.h, s1.s, D.OP_A, l, x, n)) < 1e-5
            D.dpgmg_spmv_group(s0.h, s0.s, l, 1)     # rows of the assembled operator
            assert rel(a0, D.dpgmg_apply(s0.h, s0.s, D.OP_A, l, x, n)) < 1e-5
            assert abs(g0.theta - g1.theta) < MIXED_THETA_TOL * g1.theta
            ops = [(D.OP_SMOOTH, x, n, 1e-5), (D.OP_VCYCLE, x, n, MIXED_VCYCLE_TOL), (D.OP_RESTRICT, x, nc, 1e-5),
                   (D.OP_PROLONG, xc, n, 1e-5)]
            if g0.kind == 2:
                ops.append((D.OP_CONDENSE, x, n, 1e-5))
            for op, v, m, tol in ops:
                y0, y1 = (D.dpgmg_apply(s.h, s.s, op, l, v, m) for s in (s0, s1))
                assert rel(y0, y1) < tol, (op, l)


@pytest.mark.parametrize("case", CASES)
def test_cg_operator_against_complex128(case):
    """Random values, ten decades of magnitudes, zero, and values that are not finite."""
    with solver(case) as s0, solver(case, D.FLAG_CG_C128) as s1:
        L = case[3] - 1
        n = s0.level(L).n_dof

        def both(v):
            return [D.dpgmg_apply(s.h, s.s, D.OP_AFULL, L, v, n) for s in (s0, s1)]
        x = rand_vec(n, 3)
        for v in (x, x * 10.0 ** np.random.default_rng(4).uniform(-10, 0, n), 1e-25 * x, 1e25 * x):
            y0, y1 = both(v)
            assert rel(y0, y1) < 1e-12
        assert np.all(both(np.zeros(n, dtype=complex))[0] == 0)
        for bad in (np.nan, np.inf):
            v = x.copy()
            v[n // 2] = bad
            y0 = D.dpgmg_apply(s0.h, s0.s, D.OP_AFULL, L, v, n)
            D.dpgmg_spmv_group(s0.h, s0.s, -1, 1)
            assert np.array_equal(np.isfinite(y0), np.isfinite(D.dpgmg_apply(s0.h, s0.s, D.OP_AFULL, L, v, n)))


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("mixed", 1e-3)])
@pytest.mark.parametrize("n,p", [((1, 1, 1), 1), ((1, 2, 2), 1), ((2, 2, 2), 1), ((2, 2, 2), 2), ((3, 3, 3), 2),
                                 ((5, 4, 3), 3)])
def test_coarse_factor_sizes(n, p, precision, tol):
    """A_0^-1 on a one-level hierarchy, sizes around the 64- and 16-wide blocks
    of the factorisation: A_0 (A_0^-1 x) = x with the assembled operator."""
    pk = dict(n=n, p=p, omega=3.0, src_center=(0.5, 0.5, 0.5), src_width=0.2)
    with D.Solver(pk, n_levels=1, p_min=p, precision=precision, tol=1e-8) as s:
        m = s.level(0).n_dof
        x = rand_vec(m, 2)
        y = D.dpgmg_apply(s.h, s.s, D.OP_COARSE, 0, x, m)
        assert rel(D.dpgmg_apply(s.h, s.s, D.OP_AFULL, 0, y, m), x) < tol
