"""The sizes at which the solver and the FP64-class stencils change their way of
running: four threads per site up to 16384 sites, one kernel for all CG
iterations up to 65536 sites (sites x right-hand sides x parities), four
iterations per pass of the loop graph beyond, block shapes of the two-thread
stencils, partial tiles and warps.  The graph-run solve must equal the
host-stepped one, which launches every kernel by itself, bit by bit."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from helpers import ROOT, parity_of_sites, site_err
from oracle import oracle as O
from paper_2001_05218_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dw():
    import torch
    assert torch.cuda.is_available()
    from paper_2001_05218_gb300 import dw as m
    return m


def _solve(dw, op, Ug, bg, xg, p):
    solve = {"wilson": dw.cg_solve, "normal": dw.cg_solve_normal, "laplace": dw.cg_solve_laplace}[op]
    return solve(Ug, bg, xg, p)


F16, F32 = dict(inner="f16", compress12=1, outer="df64"), dict(inner="f32", outer="df64")
SIZES = [
    ("wilson", (4, 4, 4, 4), 1, dict(inner="f32")),          # one block, no grid barrier
    ("wilson", (2, 2, 2, 4), 1, F16),                         # half a tile
    ("wilson", (6, 10, 6, 6), 3, F16),                        # a tile cut short, several columns
    ("wilson", (8, 8, 16, 32), 1, F16),                       # 16384 sites of a parity: the last with four threads per site
    ("wilson", (8, 8, 18, 32), 1, dict(inner="bf16", outer="df64")),
    ("wilson", (16, 16, 16, 32), 1, F32),                     # 65536: the last in one kernel
    ("wilson", (8, 8, 16, 16), 12, F16),                      # 98304 with the right-hand sides
    ("wilson", (16, 16, 18, 32), 1, F16),                     # 73728: four iterations per pass
    ("wilson", (6, 4, 4, 6), 17, F32),                        # more columns than the one kernel holds
    ("wilson", (8, 8, 8, 8), 1, dict(inner="i16", compress12=1, outer="df64", defect_correction=1)),
    ("normal", (6, 10, 6, 6), 1, F32),
    ("normal", (16, 16, 16, 16), 1, F16),                     # 65536 with both parities
    ("normal", (16, 16, 16, 18), 1, F32),
    ("laplace", (6, 10, 6, 6), 2, F32),
    ("laplace", (16, 16, 18, 32), 1, F16),
]


@pytest.mark.parametrize("op,dims,nrhs,kw", SIZES)
def test_graph_and_stepped_solves_agree_across_the_size_rules(dw, op, dims, nrhs, kw):
    kappa = 0.11
    U = I.gauge_field(dims, "exp", 41, 1, 0.4)
    bs = [I.gaussian_spinor(dims, 42, 2 + r) for r in range(nrhs)]
    Ug = dw.gauge(dims, kappa, U)
    bg = dw.spinor(dims, np.stack(bs) if nrhs > 1 else bs[0], nrhs=nrhs)
    p = dw.params(tol=1e-10, maxiter=5000, **kw)
    out = []
    for stepped in (False, True):
        xg = dw.spinor(dims, nrhs=nrhs)
        if stepped:
            dw.profile_start(time_stencils=True)
        s, st = _solve(dw, op, Ug, bg, xg, p)
        if stepped:
            dw.profile_stop()
        assert s == dw.DW_OK and max(v["true_rel_resid"] for v in st) <= 1e-10
        out.append((xg.download().reshape(nrhs, -1, 4, 3), [v["iters"] for v in st], [v["reliable_updates"] for v in st]))
    assert out[0][1] == out[1][1] and out[0][2] == out[1][2]
    assert np.array_equal(out[0][0], out[1][0])
    if I.volume(dims) <= 10000:  # the oracle's residual, from the caller's fields
        for r in range(nrhs):
            x = out[0][0][r]
            if op == "wilson":
                y = O.dirac(dims, kappa, U, x)
            elif op == "normal":
                y = O.dirac(dims, kappa, U, O.dirac(dims, kappa, U, x), dag=True)
            else:
                y = O.laplace(dims, kappa, U, x)
            assert np.linalg.norm(y - bs[r]) <= 1e-10 * np.linalg.norm(bs[r])


def test_one_kernel_loop_stops_at_maxiter_and_deadline(dw):
    dims, kappa = (8, 8, 8, 8), 0.12
    U = I.gauge_field(dims, "exp", 43, 1, 0.4)
    Ug, bg = dw.gauge(dims, kappa, U), dw.spinor(dims, I.gaussian_spinor(dims, 43, 2))
    x = dw.spinor(dims)
    s, st = dw.cg_solve(Ug, bg, x, dw.params(tol=1e-10, maxiter=3), raise_on_fail=False)
    assert s == dw.DW_ERR_NOT_CONVERGED and st[0]["iters"] == 3
    x = dw.spinor(dims)
    s, st = dw.cg_solve(Ug, bg, x, dw.params(tol=1e-14, timeout_s=1e-9, maxiter=100000), raise_on_fail=False)
    assert s in (dw.DW_ERR_TIMEOUT, dw.DW_ERR_NOT_CONVERGED) and st[0]["iters"] <= 2


def test_ragged_batch_in_one_kernel(dw):
    systems = [((4, 4, 4, 4), 0.12), ((6, 10, 6, 6), 0.115), ((8, 8, 8, 8), 0.118)]
    Us, bs, xs, host = [], [], [], []
    for i, (dims, kappa) in enumerate(systems):
        U, b = I.gauge_field(dims, "exp", 50 + i, 1, 0.4), I.gaussian_spinor(dims, 50 + i, 2)
        if i == 1:
            b[:] = 0.0  # a zero source beside the others
        host.append((dims, kappa, U, b))
        Us.append(dw.gauge(dims, kappa, U))
        bs.append(dw.spinor(dims, b))
        xs.append(dw.spinor(dims))
    s, st = dw.cg_solve_batched(Us, bs, xs, dw.params(tol=1e-10, **F16))
    assert s == dw.DW_OK
    for (dims, kappa, U, b), x in zip(host, xs):
        r = O.dirac(dims, kappa, U, x.download()) - b
        assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b)


CHILD = r'''
import json, os, sys
import numpy as np
sys.path.insert(0, os.environ["REPO"])
import torch
from paper_2001_05218_gb300 import dw, inputs as I
dims, n = (6, 10, 6, 6), 4
U = I.gauge_field(dims, "exp", 61, 1, 0.4)
psi = np.stack([I.gaussian_spinor(dims, 61, 2 + r) for r in range(n)])
for prec, c12 in (("df64", 0), ("df64", 1), ("f64", 0)):
    P = dw.PREC[prec]
    Ug = dw.gauge(dims, 0.12, U, prec=P, compress12=c12)
    x, y = dw.spinor(dims, psi, prec=P, nrhs=n), dw.spinor(dims, prec=P, nrhs=n)
    for op in (dw.apply, dw.laplace_apply):
        op(Ug, x, y)
        np.save(os.path.join(os.environ["OUT"], "%s_%d_%s.npy" % (prec, c12, op.__name__)), y.download())
'''


@pytest.mark.parametrize("shape", ["32 1 0", "128 2 0", "256 1 0", "64 4 0"])
def test_two_thread_stencils_in_every_block_shape(tmp_path, shape):
    """FP64 and double-float results do not depend on the block shape (which also
    sets the shared memory of the double-float copies, up to 168 KB)."""
    import torch
    name = torch.cuda.get_device_name(0).replace(" ", "_")
    got = []
    for k, lines in enumerate(([], ["%s/v5/%s/r4/6x10x6x6 %s\n" % (name, key, shape)
                                    for key in ("df64c18", "df64c12", "f64c18")])):
        d = tmp_path / str(k)
        d.mkdir()
        (d / "tune.txt").write_text("".join(lines))
        env = dict(os.environ, DW_TUNE_CACHE=str(d / "tune.txt"), REPO=ROOT, OUT=str(d))
        r = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-3000:]
        got.append({f: np.load(d / f) for f in sorted(os.listdir(d)) if f.endswith(".npy")})
    assert list(got[0]) == list(got[1]) and len(got[0]) == 6
    for f in got[0]:
        assert np.array_equal(got[0][f], got[1][f]), f


@pytest.mark.parametrize("prec,c12", [("f64", 0), ("f64", 1), ("df64", 0), ("df64", 1)])
@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (4, 2, 2, 6), (6, 10, 6, 6)])
def test_fp64_class_stencils_on_partial_warps(dw, prec, c12, dims):
    """Sites that fill no warp or tile, every parity and both operators, to the
    FP64 bar of the operator tests (1e-13 per site)."""
    kappa = 0.12
    U = I.gauge_field(dims, "haar", 62, 1)
    psi = I.gaussian_spinor(dims, 62, 2)
    P = dw.PREC[prec]
    Ug = dw.gauge(dims, kappa, U, prec=P, compress12=c12)
    par = parity_of_sites(dims)
    for kind, keep in ((dw.DW_SPINOR_FULL, par >= 0), (dw.DW_SPINOR_EVEN, par == 0), (dw.DW_SPINOR_ODD, par == 1)):
        src = np.where(keep[:, None, None], psi, 0)
        x, y = dw.spinor(dims, src[keep], kind=kind, prec=P), dw.spinor(dims, kind=kind, prec=P)
        for dag in (False, True):
            dw.apply(Ug, x, y, dag=dag)
            ref = O.dirac(dims, kappa, U, src, dag=dag) if kind == dw.DW_SPINOR_FULL else \
                O.schur(dims, kappa, U, src, parity=0 if kind == dw.DW_SPINOR_EVEN else 1, dag=dag)[keep]
            assert site_err(y.download(), ref) <= 1e-13
        dw.laplace_apply(Ug, x, y)
        if kind == dw.DW_SPINOR_FULL:
            assert site_err(y.download(), O.laplace(dims, kappa, U, src)) <= 1e-13


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("kind,nrhs", [("EVEN", 3), ("ODD", 1), ("FULL", 2)])
def test_export_writes_every_site(dw, prec, kind, nrhs):
    """Sites that fill no warp of the export kernel; values that both storages hold exactly."""
    dims = (2, 2, 2, 6)
    f = dw.spinor(dims, kind=getattr(dw, "DW_SPINOR_" + kind), prec=dw.PREC[prec], nrhs=nrhs)
    shape = f.canonical_shape()
    a = (np.arange(np.prod(shape)) + 1j * (np.arange(np.prod(shape)) + 0.5)).reshape(shape)
    f.upload(a)
    assert np.array_equal(f.download(), a)
    assert np.array_equal(f.export().cpu().numpy(), a)
