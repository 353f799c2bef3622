"""Reading back a frame's denoised map and flags into device buffers: whole
and partial runs of the copy kernel, either map alone, and buffers that it
does not take (unaligned device memory, host memory)."""
import pytest
import torch

from scenes import Scene, SceneConfig

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(1, 1), (5, 3), (4, 4), (17, 1), (64, 65)])
def test_denoised_into_any_buffer(W, H):
    import paper_2303_02608_gb300 as m
    sim = m.Simulator(m.SimConfig(width=W, height=H, radius=2, frames=2, contrast=0.1, rgb=True))
    frames = Scene(SceneConfig(kind="rects", width=W, height=H, frames=2, spp=2, seed=2, rgb=True, n_rects=3)).sequence()
    for f in frames:
        sim.push({k: f[k].cuda() for k in ("radiance", "normal", "albedo", "depth")})
    n = W * H
    host_a, host_f = torch.empty(n), torch.empty(n, dtype=torch.uint8)
    m.esim_ad_denoised(sim.ctx, host_a.data_ptr(), host_f.data_ptr(), False)
    a, f = sim.denoised()
    assert torch.equal(a.cpu().view(-1), host_a) and torch.equal(f.cpu().view(-1), host_f)
    for off in (0, 1):   # off 1: neither buffer on a 16-byte boundary
        buf_a = torch.full((n + 8,), -7.0, device="cuda")
        buf_f = torch.full((n + 8,), 77, dtype=torch.uint8, device="cuda")
        for want_a, want_f in ((True, True), (True, False), (False, True)):
            buf_a.fill_(-7.0)
            buf_f.fill_(77)
            m.esim_ad_denoised(sim.ctx, buf_a.data_ptr() + 4 * off if want_a else 0,
                               buf_f.data_ptr() + off if want_f else 0, True)
            exp_a, exp_f = torch.full((n + 8,), -7.0), torch.full((n + 8,), 77, dtype=torch.uint8)
            if want_a:
                exp_a[off:off + n] = host_a
            if want_f:
                exp_f[off:off + n] = host_f
            assert torch.equal(buf_a.cpu(), exp_a) and torch.equal(buf_f.cpu(), exp_f)
    sim.close()


@pytest.mark.parametrize("alpha_bytes,flag_bytes", [(256, 1 << 20), (1 << 20, 256)])
def test_denoised_into_a_buffer_that_is_too_small(alpha_bytes, flag_bytes):
    """An allocation smaller than its map is refused, as a copy call refuses it."""
    import ctypes
    import paper_2303_02608_gb300 as m
    W, H = 64, 65
    sim = m.Simulator(m.SimConfig(width=W, height=H, radius=2, frames=2, contrast=0.1, rgb=True))
    f = Scene(SceneConfig(kind="rects", width=W, height=H, frames=1, spp=2, seed=2, rgb=True, n_rects=3)).sequence()[0]
    sim.push({k: f[k].cuda() for k in ("radiance", "normal", "albedo", "depth")})
    cu = ctypes.CDLL("libcuda.so.1")
    ptrs = []
    for size in (alpha_bytes, 1 << 18, flag_bytes, 1 << 18):   # with room of our own behind each
        p = ctypes.c_uint64()
        assert cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(size)) == 0
        ptrs.append(p.value)
    try:
        with pytest.raises(m.EsimError) as e:
            m.esim_ad_denoised(sim.ctx, ptrs[0], ptrs[2], True)
        assert e.value.status == m.ESIM_AD_ECUDA
    finally:
        sim.close()
        torch.cuda.synchronize()
        for p in ptrs:
            cu.cuMemFree_v2(ctypes.c_uint64(p))
