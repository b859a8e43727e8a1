"""Every product with class matrices, selected explicitly, against its general
form on the same system; and the selection itself.

The two forms of an operator differ in summation order: complex64 sums of up to
8 x 302 products, 2^-24 each in a random walk over cancelling terms, 1e-5; the
CG operator sums products good to 2^-46, 1e-12.
"""
import numpy as np
import pytest

from oracle.assembly import FineSystem
from oracle.mesh import Mesh
from paper_2304_01728_gb300 import dpgmg as D
from tests.oracle_adapter import MIXED_VCYCLE_TOL, rand_vec, rel

pytestmark = pytest.mark.gpu


def layers(n, seed):
    c = np.random.default_rng(seed).choice([0.4, 0.7, 1.0], n[2])
    return np.repeat(c, n[0] * n[1])


CASES = [   # n, p, wavespeed layers, levels, p_min, flags
    ((4, 4, 4), 2, False, 3, 1, 0),               # few cells per class
    ((8, 8, 8), 2, False, 3, 1, 0),               # p and h levels
    ((16, 16, 8), 2, False, 3, 1, 0),             # every form on every level
    ((16, 8, 4), 2, True, 3, 2, 0),
    ((8, 8, 4), 3, True, 3, 2, D.FLAG_COMPLEX_STORAGE),
    ((12, 6, 5), 3, True, 2, 2, 0),               # odd extents
    ((6, 6, 6), 4, False, 2, 3, 0),               # two column chunks in the CG operator
    ((5, 4, 6), 5, False, 2, 4, 0),               # three
]


def solver(case):
    n, p, lay, nl, p_min, fl = case
    # a frequency and a box at which the CG operator's digits are kept
    pk = dict(n=n, p=p, omega=20.0 if p == 5 else 24.0, x1=(1, 0.8, 1.2) if p == 5 else (1, 1, 1),
              src_center=(0.4, 0.55, 0.5), src_width=0.2)
    if lay:
        pk["wavespeed"] = layers(n, sum(n))
    return D.Solver(pk, n_levels=nl, p_min=p_min, precision="mixed", tol=1e-8, flags=fl)


def forms(s, L):
    """(read or set, name) of every product that may have a class form."""
    out = []
    for l in range(1, L + 1):
        out.append((lambda on=None, l=l: D.dpgmg_spmv_group(s.h, s.s, l, {None: 0, 1: D.SPMV_CELLS, 0: 1}[on]) ==
                    D.SPMV_CELLS, ("A", l)))
        for f, name in ((D.FORM_SMOOTH, "S"), (D.FORM_CONDENSE, "C"), (D.FORM_BACKSUB, "B")):
            out.append((lambda on=None, l=l, f=f: D.dpgmg_class_form(s.h, s.s, l, f, -1 if on is None else on) == 1,
                        (name, l)))
    out.append((lambda on=None: D.dpgmg_spmv_group(s.h, s.s, -1, {None: 0, 1: D.SPMV_CELLS, 0: 1}[on]) == D.SPMV_CELLS,
                ("CG", L)))
    return out


def select(s, L, on):
    """Class forms wherever they are kept (on) or nowhere; returns the kept ones."""
    kept = set()
    for form, name in forms(s, L):
        try:
            assert form(1) and form()
            kept.add(name)
        except D.DpgmgError:
            assert not form()
        if not on:
            assert not form(0) and not form()
    return kept


@pytest.mark.parametrize("case", CASES)
def test_class_forms_against_general_forms(case):
    with solver(case) as s:
        L = case[3] - 1
        for l in range(1, L + 1):
            g = s.level(l)
            n, nc = g.n_dof, s.level(l - 1).n_dof
            x, xc = rand_vec(n, 7 + l), rand_vec(nc, 9 + l)
            ops = [(D.OP_A, x, n, 1e-5), (D.OP_SMOOTH, x, n, 1e-5), (D.OP_RESTRICT, x, nc, 1e-5),
                   (D.OP_PROLONG, xc, n, 1e-5), (D.OP_VCYCLE, x, n, MIXED_VCYCLE_TOL)]
            if g.kind == 2:
                ops.append((D.OP_CONDENSE, x, n, 1e-5))
            if l == L:
                ops.append((D.OP_AFULL, x, n, 1e-12))
            out = []
            for on in (1, 0):
                kept = select(s, L, on)
                out.append([D.dpgmg_apply(s.h, s.s, op, l, v, m) for op, v, m, _ in ops])
            for (op, _, _, tol), a, b in zip(ops, *out):
                assert rel(a, b) < tol, (op, l, rel(a, b))
        # the finest cells are shared in every case (the CG operator keeps them on a p level), and every form
        # at 16 x 16 x 8
        assert ("A", L) in kept and (("CG", L) in kept) == (s.level(L).kind == 1)
        if case[0] == (16, 16, 8):
            assert kept == {name for _, name in forms(s, L) if name[0] not in "CB" or s.level(name[1]).kind == 2}


@pytest.mark.parametrize("case", [CASES[6], CASES[7], CASES[1]])
def test_digits_with_values_that_are_not_finite(case):
    with solver(case) as s:
        L = case[3] - 1
        n = s.level(L).n_dof
        for bad in (np.nan, np.inf):
            v = rand_vec(n, 3)
            v[n // 2] = bad
            fin = []
            for g in (D.SPMV_CELLS, 1):
                assert D.dpgmg_spmv_group(s.h, s.s, -1, g) == g
                fin.append(np.isfinite(D.dpgmg_apply(s.h, s.s, D.OP_AFULL, L, v, n)))
            assert np.array_equal(*fin)


@pytest.mark.parametrize("case", CASES[:3])
def test_reading_and_writing_back_a_form_restores_it(case):
    """The value read is the form in force: set(get()) changes nothing, and an
    override followed by set(get()) gives the first form's results, bit for bit."""
    with solver(case) as s:
        L, kept = case[3] - 1, set()
        for start in (None, 0, 1):      # None: as setup chose them
            if start is not None:
                kept = select(s, L, start)
            for l in list(range(1, L + 1)) + [-1]:
                op, lv = (D.OP_AFULL, L) if l == -1 else (D.OP_A, l)
                n = s.level(lv).n_dof
                x = rand_vec(n, 5)
                g = D.dpgmg_spmv_group(s.h, s.s, l)
                y = D.dpgmg_apply(s.h, s.s, op, lv, x, n)
                assert D.dpgmg_spmv_group(s.h, s.s, l, g) == g
                assert np.array_equal(y, D.dpgmg_apply(s.h, s.s, op, lv, x, n))
                D.dpgmg_spmv_group(s.h, s.s, l, 4)
                D.dpgmg_spmv_group(s.h, s.s, l, g)
                assert np.array_equal(y, D.dpgmg_apply(s.h, s.s, op, lv, x, n))
            for l in range(1, L + 1):
                n = s.level(l).n_dof
                x = rand_vec(n, 6)
                if ("S", l) not in kept:
                    continue
                f = D.dpgmg_class_form(s.h, s.s, l, D.FORM_SMOOTH)
                y = D.dpgmg_apply(s.h, s.s, D.OP_SMOOTH, l, x, n)
                D.dpgmg_class_form(s.h, s.s, l, D.FORM_SMOOTH, 1 - f)
                D.dpgmg_class_form(s.h, s.s, l, D.FORM_SMOOTH, f)
                assert np.array_equal(y, D.dpgmg_apply(s.h, s.s, D.OP_SMOOTH, l, x, n))


def test_forms_that_a_system_does_not_have_are_refused():
    pk = dict(n=(4, 4, 4), p=2, omega=4.0, src_center=(0.4, 0.55, 0.5), src_width=0.2)
    rnd = dict(pk, wavespeed=np.random.default_rng(1).uniform(0.5, 1.0, 64))
    for prob, kw in ((pk, dict(precision="fp64")), (rnd, dict(precision="mixed")),
                     (pk, dict(precision="mixed", flags=D.FLAG_RECOMPUTE_PATCHES))):
        with D.Solver(prob, n_levels=3, p_min=1, **kw) as s:
            for l in (1, 2, -1):
                g = D.dpgmg_spmv_group(s.h, s.s, l)
                assert g != D.SPMV_CELLS
                with pytest.raises(D.DpgmgError):
                    D.dpgmg_spmv_group(s.h, s.s, l, D.SPMV_CELLS)
                assert D.dpgmg_spmv_group(s.h, s.s, l) == g
            for f in (D.FORM_SMOOTH, D.FORM_CONDENSE, D.FORM_BACKSUB):
                assert D.dpgmg_class_form(s.h, s.s, 1, f) == 0
                with pytest.raises(D.DpgmgError):
                    D.dpgmg_class_form(s.h, s.s, 1, f, 1)
            for level, which, v in ((0, 0, 0), (3, 0, 0), (1, 3, 0), (1, -1, 0), (1, 0, 2)):
                with pytest.raises(D.DpgmgError):
                    D.dpgmg_class_form(s.h, s.s, level, which, v)


@pytest.mark.parametrize("n,p,omega,box,digits", [
    ((4, 4, 4), 2, 6.0, (1, 1, 1), True), ((6, 3, 1), 3, 12.0, (1.6, 1, 0.3), True),
    ((6, 3, 1), 4, 8.0, (1, 0.5, 1 / 6), True), ((5, 4, 6), 5, 20.0, (1, 0.8, 1.2), True),
    ((6, 3, 1), 3, 0.02, (2e3, 1e3, 300), True), ((6, 3, 1), 3, 12.0, (2e-3, 1e-3, 3e-4), False),
    ((6, 3, 1), 3, 8.0, (2, 1, 0.003), False), ((6, 3, 1), 2, 8.0, (2, 0.1, 0.003), False)])
def test_cg_operator_entry_by_entry(n, p, omega, box, digits):
    """Error of every entry against complex128, relative to sum |A_ak| |x_k|.

    The double-float form's operands and products are good to 2^-48; sums of up
    to 8 x 302 products stay below 2^-43 of that sum.  The digits of a matrix row
    and of a cell's values are relative to the largest of each, so they are kept
    only where the class matrices' diagonals do not spread (cells.cuh), and are
    there as good as the assembled rows (1.25: scatter of the two samples)."""
    pk = dict(n=n, p=p, omega=omega, x1=box, src_center=tuple(0.4 * b for b in box), src_width=0.2 * max(box))
    kw = dict(n_levels=2, p_min=p - 1, precision="mixed", tol=1e-8, max_iter=300)
    g = np.asarray(FineSystem(Mesh(n, p, (0, 0, 0), box), omega, elements=[]).dofs)
    nloc = g.shape[1]
    with D.Solver(pk, **kw) as s, D.Solver(pk, flags=D.FLAG_CG_C128, **kw) as s1:
        m = s.n_trace
        if digits:
            assert D.dpgmg_spmv_group(s.h, s.s, -1, D.SPMV_CELLS) == D.SPMV_CELLS
        else:
            assert D.dpgmg_spmv_group(s.h, s.s, -1) != D.SPMV_CELLS
            with pytest.raises(D.DpgmgError):
                D.dpgmg_spmv_group(s.h, s.s, -1, D.SPMV_CELLS)
        sol = s1.solve(fields=False)[0]
        K = np.array([np.abs(D.dpgmg_element_matrix(s.h, s.s, 1, e, nloc)) for e in range(len(g))])
        for x in (sol, rand_vec(m, 3), D.dpgmg_rhs(s.h, s.s, m)):
            xl = np.where(g >= 0, np.abs(x)[np.maximum(g, 0)], 0)
            bound = np.zeros(m)
            np.add.at(bound, g[g >= 0], np.einsum("eij,ej->ei", K, xl)[g >= 0])
            want, q = D.dpgmg_apply(s1.h, s1.s, D.OP_AFULL, 1, x, m), []
            for form in (D.SPMV_CELLS, 1) if digits else (1,):
                assert D.dpgmg_spmv_group(s.h, s.s, -1, form) == form
                err = np.abs(D.dpgmg_apply(s.h, s.s, D.OP_AFULL, 1, x, m) - want) / np.maximum(bound, 1e-300)
                assert np.max(err) <= 2.0 ** -43
                q.append(np.sqrt(np.mean(err ** 2)))
            assert q[0] <= 1.25 * q[-1], q


def test_bytes_of_the_form_that_ran():
    """Bytes per launch follow the form in force; bytes per iteration count what
    is distinct, whichever form runs."""
    case = CASES[2]
    n, p, nel = case[0], case[1], 16 * 16 * 8
    loc = (p + 1) ** 3 - (p - 1) ** 3 + 6 * p * p
    tiles = (loc + 15) // 16
    ldr, ld = (loc + 3) // 4 * 4, (loc + 1) // 2 * 2
    with solver(case) as s:
        L, g = case[3] - 1, s.level(case[3] - 1)
        # 27 classes by boundary faces, the interior one real; digits: 7 of 2 bytes per entry and part
        mat = 26 * loc * ld * 8 + loc * ldr * 4
        dig = (2 * 27 - 1) * (16 * tiles) ** 2 * 14 + 27 * tiles * 16 * 4
        want = {(D.PROF_SPMV_FINE, 1): mat + nel * loc * (8 + 3 * 8) + g.n_dof * 8,
                (D.PROF_SPMV_CG, 1): dig + nel * loc * (8 + 3 * 16) + g.n_dof * 16,
                (D.PROF_SPMV_FINE, 0): (g.op_nnz - g.op_real_nnz) * 8 + g.op_real_nnz * 4,
                (D.PROF_SPMV_CG, 0): (g.op_nnz - g.op_real_nnz) * 16 + g.op_real_nnz * 8}
        per_iter = set()
        for on in (1, 0):
            select(s, L, on)
            for which in (D.PROF_SPMV_FINE, D.PROF_SPMV_CG):
                D.dpgmg_profile(s.h, s.s, which)
                per_iter.add(s.solve(fields=False)[2].bytes_per_iter)
                ms, launches, b = D.dpgmg_profile_read(s.h, s.s)
                assert launches > 0 and ms > 0 and b == want[which, on], (which, on, b, want[which, on])
        assert len(per_iter) == 1 and per_iter.pop() > 2 * mat + dig


@pytest.mark.parametrize("scale", [1e-30, 1e-32, 1e-34, 1e-36])
def test_digits_of_small_values(scale):
    """Values whose low FP32 parts are denormal keep what those parts hold: 2^-149
    of resolution in the operands and in the parts of the cells' products, up to 8
    cells of 54 terms, beside the double-float form's 1e-12."""
    with solver(CASES[1]) as s:
        L = CASES[1][3] - 1
        n = s.level(L).n_dof
        x = rand_vec(n, 3)
        assert D.dpgmg_spmv_group(s.h, s.s, -1, D.SPMV_CELLS) == D.SPMV_CELLS
        want = scale * D.dpgmg_apply(s.h, s.s, D.OP_AFULL, L, x, n)
        err = rel(D.dpgmg_apply(s.h, s.s, D.OP_AFULL, L, scale * x, n), want)
        assert err < 1e-12 + 8 * 54 * 2.0 ** -149 / scale, err
