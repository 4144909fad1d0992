"""Solves captured into a CUDA graph: replays give the solve's own bits, whatever the plan
did in between."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cs():
    from paper_2511_03093_gb300 import build as b

    b.build()
    import paper_2511_03093_gb300 as m

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return m


def _problem(cs, seed, Z, H, W):
    g = torch.Generator().manual_seed(seed)
    masks = (torch.rand(Z, H, W, generator=g) < 0.5).to(torch.uint8).cuda()
    return cs.Plan(H, W, 1, Z, masks), (torch.rand(1, H, W, generator=g) * Z / 2).cuda()


def _capture(plan, b, prm, v):
    """A graph of one solve into v (the plan has run the same solve before)."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        plan.solve(b, prm, v_out=v)
    return graph


def _replay(graph, v):
    v.zero_()
    graph.replay()
    torch.cuda.synchronize()
    return v.cpu()


@pytest.mark.parametrize("denoiser,tv_inner", [("tv", 20), ("tv", 30), ("bm3d", 1), ("wnnm", 1)])
def test_replay_after_a_solve_that_needs_more_memory(cs, denoiser, tv_inner):
    """gamma > 0, slice by slice, is captured with the plan's small buffers; gamma = 0 needs
    larger ones.  The replay still finds its own."""
    plan, b = _problem(cs, 3, 6, 64, 72)
    small, large = (cs.Params(rho=1.0, lam=0.05, gamma=g, iters=3, denoiser=denoiser,
                              tv_inner=tv_inner) for g in (0.3, 0.0))
    cs.zsweep_config(False)
    try:
        v = torch.empty(plan.vol_shape, device="cuda")
        want = plan.solve(b, small, v_out=v).cpu()
        graph = _capture(plan, b, small, v)
        other = plan.solve(b, large).cpu()
        junk = torch.full((1 << 20,), 3.0, device="cuda")  # takes memory that was given back
        for _ in range(2):
            assert torch.equal(_replay(graph, v), want)
        assert torch.equal(plan.solve(b, large).cpu(), other)
        del junk
    finally:
        cs.zsweep_config(True)
        torch.cuda.synchronize()
        plan.close()


def test_capture_where_the_batch_route_applies(cs):
    """BF16 state and many tiles: the solve runs as a persistent batch, its capture as launches
    of the same bits; a forced batch refuses the capture."""
    plan, b = _problem(cs, 5, 16, 512, 512)
    prm = cs.Params(rho=1.0, lam=0.05, iters=2, denoiser="tv", tv_inner=20, storage="bf16")
    v = torch.empty(plan.vol_shape, device="cuda")
    want = plan.solve(b, prm, v_out=v).cpu()
    graph = _capture(plan, b, prm, v)
    for _ in range(2):
        assert torch.equal(_replay(graph, v), want)
    cs.set_tv_route(2)
    try:
        assert torch.equal(plan.solve(b, prm).cpu(), want)
        with pytest.raises(cs.CslsmError) as e:
            _capture(plan, b, prm, v)
        assert e.value.status == 4
    finally:
        cs.set_tv_route(0)
    torch.cuda.synchronize()
    assert torch.equal(plan.solve(b, prm).cpu(), want)
    plan.close()


@pytest.mark.parametrize("Z,H,W", [(2, 40, 36), (6, 200, 200), (5, 255, 257)])
@pytest.mark.parametrize("storage", ["fp32", "bf16"])
def test_replays_of_the_z_sweep(cs, Z, H, W, storage):
    """The sweep's tiles wait for one another by epoch ids: a replay must not be satisfied by
    the ids of the one before, nor a later solve by a replay's."""
    plan, b = _problem(cs, Z + H, Z, H, W)
    prm, other = (cs.Params(rho=1.0, lam=0.05, gamma=0.3, iters=4, denoiser="tv", tv_inner=t,
                            storage=storage) for t in (20, 7))
    v = torch.empty(plan.vol_shape, device="cuda")
    want = plan.solve(b, prm, v_out=v).cpu()
    want_other = plan.solve(b, other).cpu()
    graph = _capture(plan, b, prm, v)
    for _ in range(5):
        assert torch.equal(_replay(graph, v), want)
        assert torch.equal(plan.solve(b, other).cpu(), want_other)
        assert torch.equal(_replay(graph, v), want)
    assert torch.equal(plan.solve(b, prm).cpu(), want)
    plan.close()
