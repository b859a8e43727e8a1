"""Cases for timing the solver through its public binding (``paper_2304_01728_gb300.dpgmg``).

What a user has the framework do, in four forms:

``solve``        MG-PCG and field recovery on a system that is already set up (``dpgmg_solve``
                 with device outputs): the inner call of a program that keeps its system.
``setup_solve``  the whole request, problem in, solution in host memory out (``dpgmg_setup``,
                 ``dpgmg_solve``, ``dpgmg_release``): what a serving slot or a one-off run does.
``block``        several loads on one system at once (``dpgmg_solve_block``).
``smooth``       the additive Schwarz smoother on caller-owned device vectors
                 (``dpgmg_smooth_noalloc``), for programs with their own Krylov loop.

Sizes, hierarchies and media are those of ``workloads.py``, ``bench.py`` and the tests: meshes
from 4^3 to 32x32x16, orders 2 to 5, complex128 and mixed V-cycles, wavespeeds that are
constant, layered, or different in every element.

A mixed solve's outputs are handed on as complex64: its V-cycle runs in complex64 and CG stops
at a relative residual of 1e-8, where two equally valid runs of the layered medium differ by
1e-6 in the solution.  complex128 solves are handed on as they are.
"""
import ctypes
import math
import random
import weakref

import numpy as np
import torch

from paper_2304_01728_gb300 import dpgmg, workloads

_STREAM = None
_HANDLE = None


def _handle():
    """One solver handle per process, on a torch stream, as a program that mixes both keeps it."""
    global _STREAM, _HANDLE
    if _HANDLE is None:
        _STREAM = torch.cuda.Stream()
        _HANDLE = dpgmg.dpgmg_create(0, 0, ctypes.c_void_p(_STREAM.cuda_stream))
    return _HANDLE


class _System:
    """A system that is released when its last user drops it."""

    def __init__(self, pk, opts):
        h = _handle()
        pb, keep = dpgmg.make_problem(**pk)
        op = dpgmg.make_opts(**opts)
        self.n_trace, self.n_field, _ = dpgmg.dpgmg_query_sizes(pb, op)
        self.s = dpgmg.dpgmg_setup(h, pb, op)
        weakref.finalize(self, dpgmg.dpgmg_release, h, self.s)


# ------------------------------------------------------------------ cases
def _case(name, what, n, p, omega, precision, medium="constant", source="gaussian", levels=4, p_min=2,
          coarsest="cholesky", loads=1, sigma=0.1, medium_seed=0, iters=30):
    c = dict(what=what, nx=n[0], ny=n[1], nz=n[2], p=p, omega=omega, precision=precision, medium=medium,
             source=source, levels=levels, p_min=p_min, coarsest=coarsest, loads=loads, sigma=sigma,
             medium_seed=medium_seed, iters=iters)
    if name:
        c["name"] = name
    return c


def listed():
    pi = math.pi
    c16 = dict(n=(16, 16, 16), p=3, omega=16 * pi, precision="mixed", levels=3, iters=42)
    lay = dict(n=(32, 32, 16), p=3, omega=20 * pi, precision="mixed", medium="layers6", levels=4, sigma=0.02, iters=205)
    return [
        # the smallest solve: the 4^3 p = 2 verification run with a known polynomial solution,
        # complex128 throughout; launches and latency
        _case("solve_cube4_p2_fp64", "solve", (4, 4, 4), 2, 4.0, "fp64", source="manufactured", levels=2, p_min=1, iters=14),
        # an odd, flat box at high order, where h-coarsening does not apply, with a complex load
        _case("solve_ragged_9x7x6_p4_mixed", "solve", (9, 7, 6), 4, 4 * pi, "mixed", source="manufactured", p_min=1,
              coarsest="auto", iters=40),
        # the unit-cube workload of the convergence studies, system kept between solves
        _case("solve_cube16_p3_mixed", "solve", **c16),
        # the layered high-contrast medium: the headline workload
        _case("solve_layered_p3_mixed", "solve", **lay),
        # a velocity model with its own wavespeed in every element
        _case("solve_random_12cubed_p3_mixed", "solve", (12, 12, 12), 3, 8 * pi, "mixed", medium="random", levels=4,
              medium_seed=7, iters=45),
        # four sources of one model at once
        _case("block4_cube16_p3_mixed", "block", loads=4, **c16),
        # the smoother inside a caller's own iteration
        _case("smooth_cube16_p3_mixed", "smooth", **dict(c16, iters=1)),
        # a small request of the serving stream: odd mesh, four layers
        _case("setup_solve_layers4_11cubed_p2_mixed", "setup_solve", (11, 11, 11), 2, 6 * pi, "mixed", medium="layers4",
              p_min=1, coarsest="auto", medium_seed=5, iters=60),
        # the default options (complex128), whole request
        _case("setup_solve_cube8_p3_fp64", "setup_solve", (8, 8, 8), 3, 8 * pi, "fp64", levels=3, iters=28),
        # one-off runs of the two workloads above and of a per-element velocity model
        _case("setup_solve_random_10x10x8_p3_mixed", "setup_solve", (10, 10, 8), 3, 6 * pi, "mixed", medium="random",
              levels=3, medium_seed=9, iters=45),
        _case("setup_solve_cube16_p3_mixed", "setup_solve", **c16),
        _case("setup_solve_layered_p3_mixed", "setup_solve", **lay),
    ]


def _dofs_per_element(p):
    return 1 + 3 * (p - 1) + 3 * (p - 1) ** 2 + 3 * p * p


def _patch_dofs(p):
    """DOFs of an interior vertex patch: those of the entities that meet in the vertex."""
    return 1 + 6 * (p - 1) + 12 * (p - 1) ** 2 + 12 * p * p


def draw(rng):
    what = rng.choice(["solve", "solve", "setup_solve", "setup_solve", "block", "smooth"])
    precision = "fp64" if rng.random() < 0.25 else "mixed"
    while True:
        p = rng.choice([2, 2, 3, 3, 3, 4, 4, 5])
        cap = (0.02 if precision == "fp64" else 0.12) * 17 ** 3 * 155.0 ** 2 * 4
        top = min(24.0, (cap / _patch_dofs(p) ** 2) ** (1.0 / 3.0))
        m = math.exp(rng.uniform(math.log(4.0), math.log(max(top, 5.0))))
        n = [max(3, int(round(m * rng.uniform(0.75, 1.25)))) for _ in range(3)]
        if rng.random() < 0.5:
            n = [2 * ((k + 1) // 2) for k in n]
        if n[0] * n[1] * n[2] * _patch_dofs(p) ** 2 <= cap:
            break
    even = all(k % 2 == 0 for k in n)
    medium = rng.choice(["constant", "constant", "layers4", "layers4", "random"])
    if p == 5:   # hundreds of distinct p = 5 element matrices cost more than the largest listed case
        medium = "constant"
    omega = rng.uniform(4.0, max(5.0, 0.8 * math.pi * min(n)))
    return _case(None, what, tuple(n), p, round(omega, 6), precision, medium=medium, levels=4, p_min=2 if even else 1,
                 coarsest="auto", loads=rng.choice([2, 3, 4, 5]) if what == "block" else 1,
                 medium_seed=rng.randrange(1 << 20), iters=40)


# ----------------------------------------------------------------- inputs
def _problem(case, rng):
    """The problem: mesh, order and medium are the case's, the source is the seed's."""
    n = (case["nx"], case["ny"], case["nz"])
    pk = dict(n=n, p=case["p"], omega=case["omega"])
    nel = n[0] * n[1] * n[2]
    mrng = random.Random(case["medium_seed"])
    if case["medium"] == "layers6":
        w = workloads.config3()["problem"]
        pk.update(x0=w["x0"], x1=w["x1"], wavespeed=w["wavespeed"],
                  src_center=(rng.uniform(0.5, 1.5), rng.uniform(0.5, 1.5), rng.uniform(0.25, 0.75)))
    else:
        if case["medium"] == "layers4":   # four layers along z
            c = [mrng.uniform(0.4, 1.0) for _ in range(4)]
            pk["wavespeed"] = [c[min(3, (4 * kz) // n[2])] for kz in range(n[2]) for _ in range(n[0] * n[1])]
        elif case["medium"] == "random":
            pk["wavespeed"] = [mrng.uniform(0.6, 1.4) for _ in range(nel)]
        pk["src_center"] = tuple(rng.uniform(0.3, 0.7) for _ in range(3))
    pk["src_width"] = case["sigma"]
    if case["source"] == "manufactured":
        pk.update(source="manufactured", mf_coeffs=_polynomial(case, rng))
    return pk


def _polynomial(case, rng):
    """Coefficients of a polynomial solution (p and u, tensor Legendre in box coordinates) that
    the trial space holds exactly."""
    m = case["p"]
    return np.array([rng.gauss(0, 1) + 1j * rng.gauss(0, 1) for _ in range(4 * m ** 3)]).reshape(4, m, m, m)


def _opts(case):
    return dict(n_levels=case["levels"], p_min=case["p_min"], precision=case["precision"],
                coarsest=case["coarsest"], tol=1e-8)


def prepare(case, seed):
    rng = random.Random(seed)
    h = _handle()
    st = dict(case=case, h=h, out=torch.complex64 if case["precision"] == "mixed" else torch.complex128)
    pk = _problem(case, rng)
    if case["what"] == "setup_solve":
        st["pb"], st["keep"] = dpgmg.make_problem(**pk)
        st["op"] = dpgmg.make_opts(**_opts(case))
        nt, nf, _ = dpgmg.dpgmg_query_sizes(st["pb"], st["op"])
        st["trace"], st["field"] = np.zeros(nt, dtype=np.complex128), np.zeros(nf, dtype=np.complex128)
        return st
    sys_ = st["sys"] = _System(pk, _opts(case))
    with torch.cuda.stream(_STREAM):
        if case["what"] == "solve":
            st["trace"] = torch.zeros(sys_.n_trace, dtype=torch.complex128, device="cuda")
            st["field"] = torch.zeros(sys_.n_field, dtype=torch.complex128, device="cuda")
        elif case["what"] == "block":
            rhs = [dpgmg.dpgmg_rhs(h, sys_.s, sys_.n_trace)]
            for _ in range(case["loads"] - 1):   # the loads of other sources, each from its own system
                o = _System(_problem(case, rng), _opts(case))
                rhs.append(dpgmg.dpgmg_rhs(h, o.s, o.n_trace))
                del o
            st["rhs"] = torch.from_numpy(np.stack(rhs)).cuda()
            st["trace"] = torch.zeros_like(st["rhs"])
        else:
            g = torch.Generator(device="cuda")
            g.manual_seed(seed)
            r = torch.randn(2 * sys_.n_trace, dtype=torch.float64, device="cuda", generator=g)
            st["r"] = torch.view_as_complex(r.view(-1, 2))
            st["trace"] = torch.zeros_like(st["r"])
            st["level"] = len(_levels(case)) - 1
    _STREAM.synchronize()
    return st


def _check(code, where):
    if code != dpgmg.DPGMG_OK:
        raise RuntimeError("%s: %s" % (where, dpgmg.strerror(code)))


def run(state):
    case, h = state["case"], state["h"]
    if case["what"] == "setup_solve":
        s = dpgmg.dpgmg_setup(h, state["pb"], state["op"])
        try:
            code, _ = dpgmg.dpgmg_solve(h, s, state["trace"], state["field"])
        finally:
            dpgmg.dpgmg_release(h, s)
        _check(code, "dpgmg_solve")
        return {k: torch.from_numpy(state[k]).to(state["out"], copy=True) for k in ("trace", "field")}
    s = state["sys"].s
    with torch.cuda.stream(_STREAM):
        if case["what"] == "solve":
            code, _ = dpgmg.dpgmg_solve(h, s, state["trace"].data_ptr(), state["field"].data_ptr(), True)
            _check(code, "dpgmg_solve")
            return {"trace": state["trace"].to(state["out"]), "field": state["field"].to(state["out"])}
        if case["what"] == "block":
            code, _, _ = dpgmg.dpgmg_solve_block(h, s, state["rhs"].data_ptr(), state["trace"].data_ptr(), True,
                                                 case["loads"])
            _check(code, "dpgmg_solve_block")
        else:
            dpgmg.dpgmg_smooth_noalloc(h, s, state["level"], state["r"].data_ptr(), state["trace"].data_ptr())
        return {"trace": state["trace"].to(state["out"])}


# ------------------------------------------------------------------- work
def _levels(case):
    """(nx, ny, nz, p, transition below) of each level, finest first: lower p to p_min, then halve."""
    n, p, out = [case["nx"], case["ny"], case["nz"]], case["p"], []
    while True:
        out.append([*n, p, ""])
        if len(out) == case["levels"]:
            return out
        if p > case["p_min"]:
            out[-1][4], p = "p", p - 1
        elif all(k % 2 == 0 for k in n):
            out[-1][4], n = "h", [k // 2 for k in n]
        else:
            return out


def work(case):
    """Bytes: the loads read and the solutions written, once.  Flops: the real multiply-adds
    (counted twice, two per real coefficient and complex unknown) of the smoothing blocks, level operators
    and CG operator applications of `iters` iterations; and, for a whole request, of the distinct
    element matrices' Gram factorisation and test-space solve."""
    nel, p = case["nx"] * case["ny"] * case["nz"], case["p"]
    nt, nf = nel * _dofs_per_element(p), nel * 4 * p ** 3
    k = case["loads"]
    if case["what"] == "smooth":
        return {"bytes": 2.0 * 16 * nt, "flops": 4.0 * nel * _patch_dofs(p) ** 2}
    loc = (p + 1) ** 3 - (p - 1) ** 3 + 6 * p * p
    per = 8.0 * nel * loc * loc                             # CG operator, two products kept per entry
    for nx, ny, nz, q, below in _levels(case):
        if below:
            m = nx * ny * nz
            lq = (q + 1) ** 3 - (q - 1) ** 3 + 6 * q * q
            cells, size = (m, _patch_dofs(q)) if below == "p" else (m // 8, 4 * _patch_dofs(q) // 2)
            per += 2 * 4.0 * cells * size ** 2 + 2 * 4.0 * m * lq * lq
    flops = k * case["iters"] * per
    bytes_ = 16.0 * k * (2 * nt) + (16.0 * nf if case["what"] != "block" else 0.0)
    if case["what"] == "setup_solve":
        t = (p + 2) ** 3 + 3 * (p + 2) * (p + 1) ** 2       # enriched test space
        distinct = {"constant": 27, "layers4": 108, "layers6": 162, "random": nel}[case["medium"]]
        flops += min(distinct, nel) * (t ** 3 / 3.0 + t * t * (4 * p ** 3 + loc))
        bytes_ += 8.0 * nel
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------ exact
def exact(case, seed):
    """The fields of a manufactured solution: the given polynomial's coefficients on every element.
    Other sources have no closed form (and a smoother's blocks are the framework's own): None."""
    if case["source"] != "manufactured" or case["what"] not in ("solve", "setup_solve"):
        return None
    rng = random.Random(seed)
    rng.uniform(0, 1), rng.uniform(0, 1), rng.uniform(0, 1)   # the source centre, drawn before the polynomial
    C = _polynomial(case, rng)                                # [component, c, b, a]
    p, n = case["p"], (case["nx"], case["ny"], case["nz"])
    x, w = np.polynomial.legendre.leggauss(p + 2)             # on [-1, 1]
    V = np.polynomial.legendre.legvander(x, p - 1)            # L_a at the points of one element
    T = []                                                    # per axis: [element, element mode, box mode]
    for d in range(3):
        t = np.empty((n[d], p, p))
        for i in range(n[d]):
            X = 2.0 * (i + 0.5 * (x + 1.0)) / n[d] - 1.0
            t[i] = np.einsum("q,qa,qb->ab", 0.5 * w, V, np.polynomial.legendre.legvander(X, p - 1))
            t[i] *= (2.0 * np.arange(p) + 1.0)[:, None]
        T.append(t)
    F = np.einsum("zcC,ybB,xaA,mCBA->zyxmcba", T[2], T[1], T[0], C, optimize=True)
    return {"trace": None, "field": F.reshape(-1)}
