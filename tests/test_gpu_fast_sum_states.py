"""GPU tests of the near image sum by expansions in a context whose configuration is
set after the boxes were laid out: centres past a skewed cell (inside and outside the
rectangle of before), a flatter lattice, and back; on a stream of its own; and in a batch.

A context made in the configuration itself sums the walls with boxes chosen for it, on the
same proxy fit bit for bit; the two agree to the rounding of the sums times the fit's gain:
FP64 1e-11, double-float 1e-10, single precision 5e-6 of the largest entry, as in
test_gpu_fast_sum.py.  The oracle's fit is another one; its rounding moves the result by
1.2e-8 for sources a lattice vector outside the cell, so 1e-7 there and 1e-10 inside.
(The fit's gain takes single precision's rounding of the walls to 4e-5 there, in the
direct sums as in these: past the cell it is compared between contexts alone.)"""
import numpy as np
import pytest

from paper_1912_04501_gb300 import workloads
from tests.conftest import oracle_operator
from tests.test_fast_sum_plan_cpu import relisted

pytestmark = pytest.mark.gpu

bie = pytest.importorskip("paper_1912_04501_gb300.bie")

PRECS = ((bie.BIE_FP64, 1e-11), (bie.BIE_DF64, 1e-10), (bie.BIE_MIXED, 5e-6))


def _cell(bodies, nodes, e2, seed=1001, phi=0.3):
    c = workloads.random_cell(bodies, phi, (1.0, 3.0), 5e-3, nodes, seed, e2=e2)
    c.update(solver=dict(n_proxy=48, proxy_radius=1.5, n_coll=24, gmres_tol=1e-10), dt=1e-3, steps=1)
    return c


def _fast(ctx):
    return all(ctx.near_work(p)[1] > 0 for p, _ in PRECS)


def _compare(ctx, cell, oracle_tol, seed=0):
    """ctx, set to cell's configuration, against a new context and the oracle."""
    new = bie.Context(cell, precision=bie.BIE_FP64)
    rng = np.random.default_rng(seed)
    idx = np.sort(rng.choice(ctx.N, 30, replace=False))
    sigma = rng.standard_normal(2 * ctx.N)
    ref = oracle_operator(cell, close_targets=np.unique(np.concatenate([[0], idx]))).apply(
        sigma.reshape(-1, 2), targets=idx)
    for prec, tol in PRECS:
        y, z = ctx.apply(sigma, precision=prec), new.apply(sigma, precision=prec)
        assert np.abs(y - z).max() < tol * np.abs(z).max(), prec
        if prec != bie.BIE_MIXED or oracle_tol < 1e-9:
            err = np.abs(y.reshape(-1, 2)[idx] - ref).max() / np.abs(ref).max()
            assert err < max(tol, oracle_tol), (prec, err)
    new.close()


def _set(ctx, cell):
    ctx.set_state(0.0, cell["e2"], [b["xc"] for b in cell["bodies"]], [b["theta"] for b in cell["bodies"]])


@pytest.mark.parametrize("skew", [-0.3, -0.45, 0.45])
def test_centres_past_a_skewed_cell(skew):
    cell = _cell(25, 256, (skew, 1.0))
    ctx = bie.Context(cell, precision=bie.BIE_FP64)
    assert _fast(ctx)
    for past in (0.3, 0.45):
        xc, n = relisted(cell, past)
        assert n > 0
        now = dict(cell, bodies=[dict(b, xc=x.tolist()) for b, x in zip(cell["bodies"], xc)])
        _set(ctx, now)
        _compare(ctx, now, 1e-7)
    _set(ctx, cell)
    _compare(ctx, cell, 1e-10)
    ctx.close()


@pytest.mark.parametrize("bodies", [24, 40])
def test_centres_outside_and_a_flatter_lattice(bodies):
    """Bodies a whole lattice vector away (the walls' images are then among them: no box is
    well away), and a lattice of 0.6 of the height; 6144 nodes keep their boxes, 10240
    get others."""
    flat = _cell(bodies, 256, (0.3, 0.6), seed=7)
    tall = dict(flat, e2=[0.3, 1.0])
    ctx = bie.Context(tall, precision=bie.BIE_FP64)
    assert _fast(ctx)
    _set(ctx, flat)
    _compare(ctx, flat, 1e-10)
    away = dict(tall, bodies=[dict(b, xc=[b["xc"][0] + (k % 3 == 0) * 1.0, b["xc"][1]])
                              for k, b in enumerate(tall["bodies"])])
    _set(ctx, away)
    _compare(ctx, away, 1e-7)
    _set(ctx, tall)
    _compare(ctx, tall, 1e-10)
    ctx.close()


def test_stream_of_its_own():
    """On a stream of its own a context's launches begin before the ones ahead have ended;
    the results are those of the default stream, bit for bit, and so they are with the
    profiler on."""
    torch = pytest.importorskip("torch")
    cell = _cell(25, 200, (0.2, 1.0), seed=5)
    stream = torch.cuda.Stream()
    got = []
    for own, prof in ((False, False), (True, False), (True, True)):
        ctx = bie.Context(cell, precision=bie.BIE_MIXED)
        assert _fast(ctx)
        if own:
            ctx.set_stream(stream.cuda_stream)
        ctx.profile(prof)
        sigma = np.random.default_rng(1).standard_normal(2 * ctx.N)
        out = [ctx.apply(sigma, precision=p) for p, _ in PRECS for _ in range(3)]
        s, _ = ctx.solve()
        v, om, mu = ctx.velocities(s)
        mus, _ = ctx.step(1e-3, 2)
        st = ctx.get_state()
        got.append([*out, s, v, om, mu, mus, st["xc"], st["theta"], st["sigma"]])
        ctx.close()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)


def test_batch_by_expansions_with_cells_switched_off():
    """A batch whose sums all run by expansions: every cell's application against the
    oracle, and a lockstep solve in which cells drop out at different iterations, against
    each cell's own solve (two solutions of a 1e-10 residual: 1e-8)."""
    cells = [_cell(30, 150, (0.0, 1.0), seed=11), _cell(12, 230, (0.2, 1.0), seed=12, phi=0.1), _cell(25, 160, (-0.4, 1.0), seed=13)]
    ctx = bie.Context(cells, precision=bie.BIE_MIXED)
    assert _fast(ctx)
    sigma = np.random.default_rng(3).standard_normal(2 * ctx.N)
    cut = [slice(2 * a, 2 * b) for a, b in zip(ctx.node_offsets[:-1], ctx.node_offsets[1:])]
    ref = [oracle_operator(c).apply(sigma[sl].reshape(-1, 2)).ravel() for c, sl in zip(cells, cut)]
    for prec, tol in ((bie.BIE_FP64, 1e-10), (bie.BIE_DF64, 1e-10), (bie.BIE_MIXED, 5e-6)):
        y = ctx.apply(sigma, precision=prec)
        for r, sl in zip(ref, cut):
            assert np.abs(y[sl] - r).max() < tol * np.abs(r).max(), prec
    s, info = ctx.solve()
    assert info["rel_residual"] <= 1e-10
    assert len({c["iterations"] for c in ctx.cell_info()}) > 1  # some ended before others
    for c, sl in zip(cells, cut):
        one = bie.Context(c, precision=bie.BIE_MIXED)
        t, _ = one.solve()
        one.close()
        assert np.abs(s[sl] - t).max() < 1e-8 * np.abs(t).max()
    ctx.close()
