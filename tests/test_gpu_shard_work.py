"""GPU test of the target partition's work: with the near sum by expansions a process
evaluates the boxes that hold its own targets (and the cell's first node) and passes over
the others, and its rows stay those of the whole application, bit for bit."""
import numpy as np
import pytest

from paper_1912_04501_gb300 import workloads

pytestmark = pytest.mark.gpu

bie = pytest.importorskip("paper_1912_04501_gb300.bie")
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("images", [9, 4])
def test_partition_leaves_out_other_boxes(images):
    from paper_1912_04501_gb300 import shard
    cell = workloads.random_cell(40, 0.25, (1.0, 2.0), 1e-2, 256, 2, e2=(0.2, 1.0))
    cell["bodies"].sort(key=lambda b: b["xc"][1])  # a process owns a band of the cell
    cell.update(solver=dict(n_proxy=48, proxy_radius=1.5, n_coll=24, gmres_tol=1e-10))
    kw = dict(n_images=images) if images == 9 else dict(n_images=4, n_proxy=128, n_coll=32)
    ctx = bie.Context(cell, precision=bie.BIE_FP64, **kw)
    sigma = torch.tensor(np.random.default_rng(4).standard_normal(2 * ctx.N), dtype=torch.float64, device="cuda")
    precs = (bie.BIE_FP64, bie.BIE_DF64, bie.BIE_MIXED)
    whole, y = {}, {}
    for p in precs:
        whole[p] = ctx.near_work(p)
        assert whole[p][1] > 0
        y[p] = ctx.apply(sigma, torch.empty_like(sigma), precision=p)
    nothing = shard.EXCHANGE(lambda ptr, n2, user: 0)
    for first, last in ((0, 10), (10, 20), (30, 40)):
        ctx.set_partition(first, last, nothing)
        rows = slice(2 * 256 * first, 2 * 256 * last)
        for p in precs:
            # a quarter of the cell and the boxes around it: below half the pairs and two
            # thirds of the translations (the coarse boxes are few)
            pairs, translations, _ = ctx.near_work(p)
            assert 0 < pairs < 0.5 * whole[p][0] and 0 < translations < 0.67 * whole[p][1], (p, pairs, translations)
            got = ctx.apply(sigma, torch.full_like(sigma, float("nan")), precision=p)
            assert torch.equal(got[rows], y[p][rows]), p
    ctx.set_partition(0, 40, None)
    for p in precs:
        assert ctx.near_work(p) == whole[p]
        assert torch.equal(ctx.apply(sigma, torch.empty_like(sigma), precision=p), y[p])
    ctx.close()
