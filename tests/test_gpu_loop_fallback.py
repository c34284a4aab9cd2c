"""Small solves where the one-kernel CG loop cannot run: the same solve with the
separate kernels, and nothing left behind for the thread's next solves.  The
failures are made on the host (dw_test_refuse)."""
import ctypes

import numpy as np
import pytest

from oracle import oracle as O
from paper_2001_05218_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LOOP_CAPTURE, LOOP_START, LOOP_WAIT = 0, 1, 2  # kinds of failure, as in csrc/dw_internal.h
DIMS, KAPPA = (8, 8, 8, 16), 0.12


@pytest.fixture(scope="module")
def dw():
    import torch
    assert torch.cuda.is_available()
    from paper_2001_05218_gb300 import dw as m
    return m


def _refuse(dw, what, count):
    assert ctypes.CDLL(dw.LIB_PATH).dw_test_refuse(what, count) == dw.DW_OK


def _solve(dw, keep, U, b, **kw):
    """A solve on fields of its own (kept, so that no plan of another solve fits):
    status, solution, iterations, kernels launched."""
    Ug, bg, xg = dw.gauge(DIMS, KAPPA, U), dw.spinor(DIMS, b), dw.spinor(DIMS)
    keep.append((Ug, bg, xg))
    dw.profile_start(time_stencils=False)
    try:
        s, st = dw.cg_solve(Ug, bg, xg, dw.params(tol=1e-10, **kw))
    finally:
        _, launches = dw.profile_stop()
    assert s == dw.DW_OK and st[0]["true_rel_resid"] <= 1e-10
    return xg.download(), st[0]["iters"], launches


@pytest.mark.parametrize("what", [LOOP_CAPTURE, LOOP_START])
@pytest.mark.parametrize("kw", [dict(inner="f16", compress12=1, outer="df64"), dict(inner="f32")])
def test_refused_cooperative_launch_falls_back(dw, what, kw):
    U, b = I.gauge_field(DIMS, "exp", 71, 1, 0.4), I.gaussian_spinor(DIMS, 71, 2)
    keep = []
    x0, n0, l0 = _solve(dw, keep, U, b, **kw)
    _refuse(dw, what, 1)
    try:
        x1, n1, l1 = _solve(dw, keep, U, b, **kw)
    finally:
        _refuse(dw, what, 0)
    # the separate kernels give the one kernel's results bit by bit; nine or more
    # launches per iteration show that they ran
    assert n1 == n0 and np.array_equal(x1, x0)
    assert l0 < 4 * n0 < l1
    # the thread's next plan: captured anew, in one kernel again
    x2, n2, l2 = _solve(dw, keep, U, b, **kw)
    assert n2 == n0 and np.array_equal(x2, x0) and l2 == l0


@pytest.mark.parametrize("kw", [dict(inner="f16", compress12=1, outer="df64"), dict(inner="f32"),
                                dict(inner="f32", timeout_s=60.0)])
def test_barrier_that_gives_up_is_followed_by_the_separate_kernels(dw, kw):
    """32 blocks whose barriers never open: the count of arrivals starts one short, so
    every block waits its bound (about a second) and leaves."""
    U, b = I.gauge_field(DIMS, "exp", 72, 1, 0.4), I.gaussian_spinor(DIMS, 72, 2)
    keep = []
    x0, n0, l0 = _solve(dw, keep, U, b, **kw)
    _refuse(dw, LOOP_WAIT, 1)
    try:
        x1, n1, l1 = _solve(dw, keep, U, b, **kw)
    finally:
        _refuse(dw, LOOP_WAIT, 0)
    r = O.dirac(DIMS, KAPPA, U, x1) - b
    assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b)
    assert l0 < 4 * n0 < l1
    # the plan goes on without the one kernel
    Ug, bg, xg = keep[1]
    xg.storage.zero_()
    s, st = dw.cg_solve(Ug, bg, xg, dw.params(tol=1e-10, **kw))
    assert s == dw.DW_OK and st[0]["iters"] == n0 and np.array_equal(xg.download(), x0)
    x2, n2, l2 = _solve(dw, keep, U, b, **kw)
    assert n2 == n0 and np.array_equal(x2, x0) and l2 == l0


@pytest.mark.parametrize("op,dims,n,nrhs,one", [
    ("wilson", (8, 8, 16, 16), 1, 8, True),      # 65536 sites x right-hand sides in all
    ("wilson", (8, 8, 16, 16), 1, 12, False),    # 98304
    ("wilson", (16, 16, 16, 16), 4, 1, True),    # four lattices, 131072
    ("wilson", (16, 16, 16, 16), 5, 1, False),
    ("normal", (16, 16, 16, 16), 1, 2, True),    # 131072 with both parities
    ("normal", (16, 16, 16, 16), 1, 3, False),
    ("laplace", (8, 8, 16, 16), 1, 12, False),
])
def test_one_kernel_rule_counts_all_sites(dw, op, dims, n, nrhs, one):
    """With 32-site blocks, which a caller may ask for (tile) and the tuner may
    find fastest, the line lies at 65536 sites x right-hand sides x parities, and
    at 131072 with at most four columns."""
    Us, bs, xs = [], [], []
    for i in range(n):
        U = I.gauge_field(dims, "exp", 73 + i, 1, 0.4)
        b = np.stack([I.gaussian_spinor(dims, 73 + i, 2 + r) for r in range(nrhs)])
        Us.append(dw.gauge(dims, 0.11, U))
        bs.append(dw.spinor(dims, b if nrhs > 1 else b[0], nrhs=nrhs))
        xs.append(dw.spinor(dims, nrhs=nrhs))
    p = dw.params(tol=1e-10, inner="f32", outer="df64", tile=32)
    dw.profile_start(time_stencils=False)
    try:
        if n > 1:
            s, st = dw.cg_solve_batched(Us, bs, xs, p)
        else:
            solve = {"wilson": dw.cg_solve, "normal": dw.cg_solve_normal, "laplace": dw.cg_solve_laplace}[op]
            s, st = solve(Us[0], bs[0], xs[0], p)
    finally:
        _, launches = dw.profile_stop()
    iters = max(v["iters"] for v in st)
    assert s == dw.DW_OK and max(v["true_rel_resid"] for v in st) <= 1e-10
    # the separate kernels are six or more launches per iteration
    assert (launches < 3 * iters + 20) == one, (launches, iters)
