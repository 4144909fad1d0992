"""TV denoiser: the phases' exchange is the caller's scratch, so that a call between two
synchronisations maps no memory; with it, without it and under a capture the same bits."""
import ctypes

import pytest
import torch

from tests.test_zz_no_alloc import _RESERVED_MEM_HIGH, _USED_MEM_CURRENT, _USED_MEM_HIGH, _Pool

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cs():
    from paper_2511_03093_gb300 import build as b

    b.build()
    import paper_2511_03093_gb300 as m

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return m


def _x(Z, H, W):
    return torch.rand(Z, H, W, generator=torch.Generator().manual_seed(Z + H + W)).cuda()


def _raw(cs, x, prm, nbytes):
    """cslsm_denoise_ws with nbytes of scratch (None: cslsm_denoise)."""
    cp, (Z, H, W) = prm.to_c(), x.shape
    out = torch.empty_like(x)
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    xp, op = (ctypes.c_void_p(t.data_ptr()) for t in (x, out))
    if nbytes is None:
        st = cs.lib().cslsm_denoise(cp.denoiser, xp, op, Z, H, W, ctypes.byref(cp), s)
    else:
        ws = torch.empty(max(nbytes, 1), dtype=torch.uint8, device="cuda")
        st = cs.lib().cslsm_denoise_ws(cp.denoiser, xp, op, Z, H, W, ctypes.byref(cp),
                                       ctypes.c_void_p(ws.data_ptr()), nbytes, s)
    assert st == 0, cs.lib().cslsm_last_error()
    return out.cpu()


@pytest.mark.parametrize("Z,H,W", [(1, 64, 64), (2, 97, 131), (4, 300, 260)])
@pytest.mark.parametrize("T", [2, 20, 24, 30])
def test_scratch_does_not_change_the_bits(cs, Z, H, W, T):
    x, prm = _x(Z, H, W), cs.Params(rho=1.0, lam=0.1, tv_inner=T, denoiser="tv")
    cp = prm.to_c()
    need = cs.lib().cslsm_denoise_workspace_bytes(cp.denoiser, Z, H, W, ctypes.byref(cp))
    assert need in (0, 16 * Z * H * W) and (T < 20 or need)
    want = _raw(cs, x, prm, None)
    for nbytes in (0, max(need - 4, 0), need, need + 64):
        assert torch.equal(_raw(cs, x, prm, nbytes), want), nbytes
    assert torch.equal(cs.denoise(x, prm).cpu(), want)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    out = cs.denoise(x, prm, out=torch.empty_like(x), stream=side)
    side.synchronize()
    assert torch.equal(out.cpu(), want)


def test_calls_leave_the_memory_pool_alone(cs):
    """As before the phases: nothing from the stream-ordered pool, which gives its memory back
    at every synchronisation."""
    x, prm = _x(16, 128, 160), cs.Params(rho=1.0, lam=0.1, tv_inner=20, denoiser="tv")
    cs.denoise(x, prm)
    torch.cuda.synchronize()
    pool = _Pool(torch.cuda.current_device())
    used = pool.get(_USED_MEM_CURRENT)
    pool.reset_high_marks()
    high = pool.get(_RESERVED_MEM_HIGH)
    for _ in range(3):
        cs.denoise(x, prm)
        _raw(cs, x, prm, None)
        torch.cuda.synchronize()
    assert pool.get(_USED_MEM_HIGH) == used
    assert pool.get(_RESERVED_MEM_HIGH) == high


def test_misaligned_scratch_is_refused(cs):
    cp = cs.Params(lam=0.1, denoiser="tv").to_c()
    fake = [ctypes.c_void_p(a) for a in (0x1000, 0x100000, 0x200008)]
    assert cs.lib().cslsm_denoise_ws(cp.denoiser, fake[0], fake[1], 1, 8, 8, ctypes.byref(cp),
                                     fake[2], 4096, None) == 1


def test_captured_call(cs):
    x, prm = _x(8, 200, 150), cs.Params(rho=1.0, lam=0.1, tv_inner=20, denoiser="tv")
    want = cs.denoise(x, prm).cpu()
    out = torch.empty_like(x)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        cs.denoise(x, prm, out=out)
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out.cpu(), want)


@pytest.mark.parametrize("Z,H,W", [(1, 131, 97), (3, 70, 45), (2, 256, 200)])
@pytest.mark.parametrize("T", [7, 24, 25, 53])
def test_tile_kernel_without_scratch(cs, Z, H, W, T):
    """cslsm_denoise runs the whole-prox tiles for up to 24 steps: the model's shape, every
    forced variant (several launches beyond 24 steps) and the timed choice, first measured
    and then kept, all give the phases' bits."""
    x, prm = _x(Z, H, W), cs.Params(rho=1.0, lam=0.1, tv_inner=T, denoiser="tv")
    want = _raw(cs, x, prm, 16 * Z * H * W)
    try:
        for mode in (0, 2, 3, 4, 5):
            cs.set_autotune(mode)
            assert torch.equal(_raw(cs, x, prm, None), want), mode
        cs.set_autotune(1)
        launches = []
        for _ in range(2):
            n = cs.launch_count()
            assert torch.equal(_raw(cs, x, prm, None), want)
            launches.append(cs.launch_count() - n)
        cp = prm.to_c()  # phases that need no exchange (few steps) run instead
        need = cs.lib().cslsm_denoise_workspace_bytes(cp.denoiser, Z, H, W, ctypes.byref(cp))
        if T <= 24 and need:  # three runs of each variant, then the launch itself
            assert launches[0] > launches[1] == 1
        assert need or T < 24
    finally:
        cs.set_autotune(0)


def test_solve_captured_on_a_fresh_plan(cs):
    """The exchange is not there yet and is not allocated under capture: whole-prox tiles."""
    g = torch.Generator().manual_seed(2)
    masks = (torch.rand(4, 90, 70, generator=g) < 0.5).to(torch.uint8).cuda()
    b = torch.rand(1, 90, 70, generator=g).cuda()
    prm = cs.Params(rho=1.0, lam=0.05, iters=3, denoiser="tv", tv_inner=20)
    fresh, other = (cs.Plan(90, 70, 1, 4, masks) for _ in range(2))
    v = torch.empty(fresh.vol_shape, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fresh.solve(b, prm, v_out=v)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(v.cpu(), other.solve(b, prm).cpu())
    fresh.close()
    other.close()
