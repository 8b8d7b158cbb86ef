"""GPU tests of what a new configuration builds and a solve repeats, at the sizes
where the kernels change: the proxy fit by a cluster of CTAs (at most 512 rows) and
by one, the contact block's inversion by clusters of sixteen and eight CTAs and by
launches, and the orthogonalisation with chunks of one and of several tiles.

Tolerances.  Fit: 1e-10 of the parity tests times ten, the fits here being up to
twice as large.  Contact block: two solutions of relative residual 1e-10 of an
operator whose condition number is below 1e3 there.  Residual: the solver's own
criterion, with as much again for the application that checks it.
"""
import numpy as np
import pytest

from paper_1912_04501_gb300 import workloads
from tests.conftest import oracle_operator

pytestmark = pytest.mark.gpu

bie = pytest.importorskip("paper_1912_04501_gb300.bie")


def _rel(a, b):
    return np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(b).max()


@pytest.mark.parametrize("n_proxy,n_coll", [(30, 17), (48, 24), (64, 48), (70, 50)])
def test_proxy_fit_sizes(n_proxy, n_coll):
    """196 x 60, 288 x 96, 512 x 128 and 540 x 140."""
    cell = workloads.small_cell(n_bodies=3, nodes=64, seed=4)
    cell["solver"].update(n_proxy=n_proxy, n_coll=n_coll)
    ctx = bie.Context(cell, precision=bie.BIE_FP64)
    sigma = np.random.default_rng(8).standard_normal(2 * ctx.N)
    ref = oracle_operator(cell).apply(sigma.reshape(-1, 2)).ravel()
    assert _rel(ctx.apply(sigma, precision=bie.BIE_FP64), ref) < 1e-9
    ctx.close()


@pytest.mark.parametrize("n", [48, 320, 512, 768, 1536])
def test_contact_block_sizes(n):
    cell = workloads.two_ellipses(2e-3, n)
    sols, its = [], []
    for precond in (1, 0):
        ctx = bie.Context(cell, precision=bie.BIE_DF64, precond=precond, gmres_tol=1e-10)
        sig, info = ctx.solve()
        sols.append(sig)
        its.append(info["iterations"])
        ctx.close()
    assert its[0] < its[1]
    assert _rel(sols[0], sols[1]) < 2e-7


@pytest.mark.parametrize("bodies,nodes", [(1, 8), (3, 64), (24, 256), (60, 256)])
def test_solution_residual(bodies, nodes):
    """Vectors of 16, 384, 12288 and 30720 entries: chunks of 128 and of 256."""
    cell = workloads.small_cell(n_bodies=bodies, nodes=nodes, seed=6, gap=0.05 if bodies < 10 else 0.01)
    tol = 1e-9
    ctx = bie.Context(cell, precision=bie.BIE_FP64, gmres_tol=tol)
    sig, info = ctx.solve()
    b = ctx.rhs()
    r = np.asarray(ctx.apply(sig, precision=bie.BIE_FP64)) - np.asarray(b)
    assert np.linalg.norm(r) / np.linalg.norm(b) < 2 * tol
    ctx.close()
