"""GPU tests of bie_apply_static on a stream of the caller's own, captured into a CUDA graph
between configurations: an application before the first replay, replays after later
configurations (inside and outside the boxes as laid out, with more close pairs and with
fewer) and plain calls all equal a context that never saw a capture, bit for bit (the same
kernels on the same numbers)."""
import numpy as np
import pytest

from paper_1912_04501_gb300 import workloads

pytestmark = pytest.mark.gpu

bie = pytest.importorskip("paper_1912_04501_gb300.bie")
torch = pytest.importorskip("torch")


def _placed(cell, dx=0.0, dy=0.0, tall=1.0):
    c = cell["centre"]
    return [[b["xc"][0] + dx, c[1] + tall * (b["xc"][1] - c[1]) + dy] for b in cell["bodies"]]


@pytest.mark.parametrize("which", ["fast", "direct", "doubled"])
def test_capture_between_configurations(which):
    cell = workloads.random_cell(*((4, 0.2, (1.0, 2.0), 1e-2, 64, 3) if which == "direct" else
                                   (40, 0.25, (1.0, 2.0), 1.2e-2, 160, 5)))
    cell.update(solver=dict(n_proxy=48, proxy_radius=1.5, n_coll=24, gmres_tol=1e-10))
    kw = dict(n_images=4, n_proxy=128, n_coll=32) if which == "doubled" else {}
    ctx = bie.Context(cell, precision=bie.BIE_MIXED, **kw)
    ref = bie.Context(cell, precision=bie.BIE_MIXED, **kw)
    assert (ctx.near_work(bie.BIE_MIXED)[1] > 0) == (which != "direct")
    # the close pairs' storage holds this many: no later configuration may have more (it
    # would be moved, and a captured application with it left behind)
    most, room = ctx.close_info()[0], min(ctx.N, 1024)
    assert most + 8 < room or most > room
    theta = [b["theta"] for b in cell["bodies"]]
    sigma = torch.tensor(np.random.default_rng(3).standard_normal(2 * ctx.N), device="cuda")
    out, eager, want = torch.empty_like(sigma), torch.empty_like(sigma), torch.empty_like(sigma)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx.set_stream(stream.cuda_stream)
    ctx.apply_static(sigma, out)  # looks up the array's address, before any capture
    stream.synchronize()

    def at(e2, xc):
        ctx.set_state(0.0, e2, xc, theta)
        ref.set_state(0.0, e2, xc, theta)
        ref.apply(sigma, want, precision=bie.BIE_MIXED)
        torch.cuda.synchronize()
        n = ctx.close_info()[0]
        assert n <= most + 8
        return n

    # a taller cell: the bodies farther apart, fewer close pairs
    few = at((0.0, 1.06), _placed(cell, tall=1.06))
    assert 0 < few < most
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ctx.apply_static(sigma, out)
    # the capture ran nothing: an application before its first replay
    ctx.apply(sigma, eager, precision=bie.BIE_MIXED)
    assert torch.equal(eager, want)

    def replay():
        out.fill_(float("nan"))
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            graph.replay()
        stream.synchronize()
        assert torch.equal(out, want)

    replay()
    states = [((0.0, 1.0), _placed(cell)), ((0.0, 1.06), _placed(cell, 0.03, 0.04, 1.06))]
    if which != "doubled":  # past the cell, and the same lattice by another second vector
        states += [((0.0, 1.0), _placed(cell, 1.1)), ((1.0, 1.0), _placed(cell)), ((0.0, 1.0), _placed(cell))]
    for e2, xc in states:
        at(e2, xc)
        replay()
        ctx.apply_static(sigma, eager)
        stream.synchronize()
        assert torch.equal(eager, want)
    ctx.close()
    ref.close()


def test_beside_the_context_s_other_calls():
    """The allocation-free application on one stream while the context's own application
    runs on another: neither writes what the other reads."""
    cell = workloads.random_cell(40, 0.25, (1.0, 2.0), 1.2e-2, 160, 5)
    cell.update(solver=dict(n_proxy=48, proxy_radius=1.5, n_coll=24, gmres_tol=1e-10))
    ctx = bie.Context(cell, precision=bie.BIE_MIXED)
    assert ctx.near_work(bie.BIE_MIXED)[1] > 0 and ctx.close_info()[0] > 0
    rng = np.random.default_rng(4)
    a, b = (torch.tensor(rng.standard_normal(2 * ctx.N), device="cuda") for _ in range(2))
    want_a, want_b, got_a, got_b = (torch.empty_like(a) for _ in range(4))
    ctx.apply(a, want_a, precision=bie.BIE_MIXED)
    ctx.apply(b, want_b, precision=bie.BIE_MIXED)
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(100):
        ctx.set_stream(one.cuda_stream)
        for _ in range(3):
            ctx.apply_static(a, got_a)
        ctx.set_stream(two.cuda_stream)
        ctx.apply(b, got_b, precision=bie.BIE_MIXED)  # waits for the second stream only
        one.synchronize()
        assert torch.equal(got_a, want_a) and torch.equal(got_b, want_b)
    ctx.close()


def test_takes_and_refuses_what_it_did():
    """The array's limit goes by the splits it was sized for (partials of at least 64
    sources): 40 cells of 204 nodes and 128 collocation points per wall take 3.82 of its
    4.19 MB, 52 of 156 would take 4.66."""
    def batch(cells, nodes):
        return [dict(e1=[1.0, 0.0], e2=[0.0, 1.0], centre=[0.5, 0.5], mu=1.0, gamma=1.0,
                     bodies=[dict(a=0.2, b=0.1, xc=[0.5, 0.5], theta=0.01 * k, n=nodes)],
                     solver=dict(n_proxy=48, proxy_radius=1.5, n_coll=128, gmres_tol=1e-10)) for k in range(cells)]
    ctx = bie.Context(batch(40, 204), precision=bie.BIE_MIXED)
    sigma = torch.tensor(np.random.default_rng(6).standard_normal(2 * ctx.N), device="cuda")
    want, got = torch.empty_like(sigma), torch.full_like(sigma, float("nan"))
    ctx.apply(sigma, want, precision=bie.BIE_MIXED)
    ctx.apply_static(sigma, got)
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    ctx.close()
    ctx = bie.Context(batch(52, 156), precision=bie.BIE_MIXED)
    with pytest.raises(bie.BieError) as e:
        ctx.apply_static(sigma[:2 * ctx.N], got[:2 * ctx.N])
    assert e.value.code == bie.BIE_EINVAL and "bytes of scratch" in str(e.value)
    ctx.close()
