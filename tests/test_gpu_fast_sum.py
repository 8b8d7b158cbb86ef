"""GPU tests of the near image sum by expansions (csrc/fmm.cu) against the
oracle's direct sum at sampled targets, over what decides its boxes: lattice
(skewed, turned), node counts that leave leaves ragged, one crowded
body beside many sparse ones, stars, bodies reaching out of the cell or placed
outside it, both image sets, and a configuration set later.

Tolerances, relative to the largest entry: FP64 and double-float 1e-10 (the
parity tolerance of the operator; the proxy fit's gain sets it, the series are
truncated far below).  Single precision 5e-6: a row adds about 1e3 near pairs
and a few hundred translated terms, each rounded to 6e-8, independently enough
that their sum is off by about sqrt(1e3) 6e-8 = 2e-6 of the terms' scale.
"""
import math

import numpy as np
import pytest

from paper_1912_04501_gb300 import workloads
from tests.conftest import oracle_operator

pytestmark = pytest.mark.gpu

bie = pytest.importorskip("paper_1912_04501_gb300.bie")


def _cell(n_bodies, nodes, phi, e1=(1.0, 0.0), e2=(0.0, 1.0), seed=1, gap=5e-3):
    c = workloads.random_cell(n_bodies, phi, (1.0, 2.5), gap, nodes, seed, e1=e1, e2=e2, centre=(0.3, -0.2),
                              equal_area=False)
    c.update(solver=dict(n_proxy=48, proxy_radius=1.5 * max(math.hypot(*e1), math.hypot(*e2)), n_coll=24,
                         gmres_tol=1e-10), dt=1e-3, steps=1)
    return c


def _crowded():
    c = _cell(24, 128, 0.15, e2=(0.2, 1.0), seed=4, gap=2e-2)
    c["bodies"][3]["n"] = 4096
    return c


CELLS = {
    "skewed": lambda: _cell(40, lambda a, b: 2 * int(300 * (a + b)) + 90, 0.25, e2=(0.45, 1.0)),
    "turned": lambda: _cell(30, 130, 0.2, e1=(0.8, 0.6), e2=(-0.5, 0.9), seed=2),
    "crowded": _crowded,
    "stars": lambda: dict(workloads.stars(4, n=1500), centre=[0.5, 0.5]),
}


def _check(ctx, cell, seed=0, n=40, **kw):
    rng = np.random.default_rng(seed)
    idx = np.sort(rng.choice(ctx.N, n, replace=False))
    sigma = rng.standard_normal(2 * ctx.N)
    ref = oracle_operator(cell, close_targets=np.unique(np.concatenate([[0], idx])), **kw).apply(
        sigma.reshape(-1, 2), targets=idx)
    for prec, tol in ((bie.BIE_FP64, 1e-10), (bie.BIE_DF64, 1e-10), (bie.BIE_MIXED, 5e-6)):
        y = ctx.apply(sigma, precision=prec).reshape(-1, 2)[idx]
        err = np.abs(y - ref).max() / np.abs(ref).max()
        assert err < tol, (prec, err)


@pytest.mark.parametrize("which", list(CELLS))
def test_matches_oracle(which):
    cell = CELLS[which]()
    ctx = bie.Context(cell, precision=bie.BIE_FP64)
    _check(ctx, cell)
    ctx.close()


def test_bodies_placed_outside_the_cell():
    """Centres a lattice vector away from the cell (nothing wraps them before
    the first time step), first at creation, then by set_state."""
    cell = _cell(30, 140, 0.2, e2=(0.3, 1.0), seed=6)
    moved = dict(cell, bodies=[dict(b, xc=[b["xc"][0] + (1.0 if k % 3 == 0 else 0.0), b["xc"][1]])
                               for k, b in enumerate(cell["bodies"])])
    a = bie.Context(moved, precision=bie.BIE_FP64)
    b = bie.Context(cell, precision=bie.BIE_FP64)
    b.set_state(0.0, cell["e2"], [bd["xc"] for bd in moved["bodies"]], [bd["theta"] for bd in moved["bodies"]])
    sigma = np.random.default_rng(5).standard_normal(2 * a.N)
    for prec, tol in ((bie.BIE_FP64, 1e-11), (bie.BIE_MIXED, 5e-6)):
        ya, yb = a.apply(sigma, precision=prec), b.apply(sigma, precision=prec)
        assert np.abs(ya - yb).max() < tol * np.abs(ya).max()
    # and back inside: the boxes of before still hold every body
    b.set_state(0.0, cell["e2"], [bd["xc"] for bd in cell["bodies"]], [bd["theta"] for bd in cell["bodies"]])
    _check(b, cell, seed=4)
    a.close()
    b.close()


def test_steps_follow_the_shearing_lattice():
    """After steps that take the lattice past half a cell of skew (where it
    jumps back) the sorted boxes follow: applications match the oracle at the
    configuration reached."""
    cell = _cell(26, 128, 0.12, e2=(0.48, 1.0), seed=8, gap=2e-2)
    ctx = bie.Context(cell, precision=bie.BIE_MIXED)
    ctx.step(1e-2, 4)
    st = ctx.get_state()
    assert abs(st["e2"][0]) < 0.5 and st["e2"][0] < 0  # it did jump
    now = dict(cell, e2=list(st["e2"]), bodies=[dict(b, xc=x.tolist(), theta=float(t))
                                               for b, x, t in zip(cell["bodies"], st["xc"], st["theta"])])
    _check(ctx, now)
    ctx.close()


def test_doubled_cell_crosses_walls():
    from oracle import bie as obie
    from tests.conftest import oracle_suspension
    cell = _cell(40, 130, 0.25, e2=(-0.3, 1.0), seed=9)
    ctx = bie.Context(cell, precision=bie.BIE_FP64, n_images=4, n_proxy=128, n_coll=32)
    rng = np.random.default_rng(2)
    idx = np.sort(rng.choice(ctx.N, 40, replace=False))
    sigma = rng.standard_normal(2 * ctx.N)
    op = obie.OperatorUtilde(oracle_suspension(cell), close_targets=np.unique(np.concatenate([[0], idx])))
    ref = op.apply(sigma.reshape(-1, 2), targets=idx)
    for prec, tol in ((bie.BIE_FP64, 1e-10), (bie.BIE_DF64, 1e-10), (bie.BIE_MIXED, 5e-6)):
        y = ctx.apply(sigma, precision=prec).reshape(-1, 2)[idx]
        assert np.abs(y - ref).max() < tol * np.abs(ref).max(), prec
    ctx.close()


def test_batch_of_uneven_cells():
    """Cells of very different size share the boxes' launches; a cell switched
    off by the solver keeps its neighbours' sums right (the solve converges)."""
    cells = [_cell(30, 150, 0.2, seed=11), workloads.config1(), _cell(12, 96, 0.1, e2=(0.2, 1.0), seed=12, gap=2e-2),
             dict(workloads.two_ellipses(1e-2, 256), centre=[0.5, 0.5])]
    for c in cells:
        c["solver"] = dict(n_proxy=48, proxy_radius=1.5, n_coll=24, gmres_tol=1e-10)
    ctx = bie.Context(cells, precision=bie.BIE_MIXED)
    sigma = np.random.default_rng(3).standard_normal(2 * ctx.N)
    for prec, tol in ((bie.BIE_FP64, 1e-10), (bie.BIE_DF64, 1e-10), (bie.BIE_MIXED, 5e-6)):
        y = ctx.apply(sigma, precision=prec)
        for k, c in enumerate(cells):
            sl = slice(2 * ctx.node_offsets[k], 2 * ctx.node_offsets[k + 1])
            ref = oracle_operator(c).apply(sigma[sl].reshape(-1, 2)).ravel()
            assert np.abs(y[sl] - ref).max() < tol * np.abs(ref).max(), (prec, k)
    _, info = ctx.solve()
    assert info["rel_residual"] <= 1e-10
    ctx.close()
