"""Forms of the two-threads-per-site stencils that only the solvers run: one warp
per mu on small lattices (up to 4096 sites of a parity), and the Laplacian in the
block shapes of an FP64-inner solve."""
import numpy as np
import pytest

from helpers import parity_of_sites, site_err
from oracle import oracle as O
from paper_2001_05218_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dw():
    import torch
    assert torch.cuda.is_available()
    from paper_2001_05218_gb300 import dw as m
    return m


@pytest.mark.parametrize("op", ["wilson", "laplace"])
@pytest.mark.parametrize("outer", ["f64", "df64"])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (6, 10, 6, 6), (8, 8, 8, 16)])
def test_one_warp_per_mu_to_the_operators_bar(dw, op, outer, dims):
    """A solve stopped early shows its stencils: x_o = b_o + kappa H_oe x_e takes the
    outer precision's, the reported residual IEEE FP64's, each to the 1e-13 per site
    of the operator tests (the residual's error is that of D x: 1e-13 |x| / |b|)."""
    kappa = 0.11
    U, b = I.gauge_field(dims, "exp", 91, 1, 0.4), I.gaussian_spinor(dims, 91, 2)
    x = dw.spinor(dims)
    solve = dw.cg_solve if op == "wilson" else dw.cg_solve_laplace
    apply = O.dirac if op == "wilson" else O.laplace
    # (converged to 1e-2 or not: the residual is of that size either way)
    s, st = solve(dw.gauge(dims, kappa, U), dw.spinor(dims, b), x, dw.params(tol=1e-2, inner="f32", outer=outer),
                  raise_on_fail=False)
    assert s in (dw.DW_OK, dw.DW_ERR_NOT_CONVERGED)
    got = x.download()
    r = b - apply(dims, kappa, U, got)
    odd = parity_of_sites(dims) == 1
    assert site_err(got[odd], (got + r)[odd]) <= 1e-13  # (x + r)_o = b_o + kappa H_oe x_e
    nb = np.linalg.norm(b)
    assert st[0]["true_rel_resid"] > 1e-5
    assert abs(st[0]["true_rel_resid"] - np.linalg.norm(r) / nb) <= 1e-13 * (1 + np.linalg.norm(got) / nb)


@pytest.mark.parametrize("tile", [32, 96, 128, 256])
def test_laplacian_fp64_solve_in_every_block_shape(dw, tile):
    dims, kappa = (6, 10, 6, 6), 0.12
    U, b = I.gauge_field(dims, "exp", 92, 1, 0.4), I.gaussian_spinor(dims, 92, 2)
    Ug, bg = dw.gauge(dims, kappa, U), dw.spinor(dims, b)
    x, y = dw.spinor(dims), dw.spinor(dims)
    _, ref = dw.cg_solve_laplace(Ug, bg, x, dw.params(tol=1e-10, inner="f64"))
    _, st = dw.cg_solve_laplace(Ug, bg, y, dw.params(tol=1e-10, inner="f64", tile=tile))
    assert st[0]["iters"] == ref[0]["iters"]
    r = O.laplace(dims, kappa, U, y.download()) - b
    assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b)
