"""Window boxes of few flagged pixels: items in one row, in two, over as many rows
as a tile has (the height of a small box), at the image's borders and spread
over a tile, against the same frame read through L1.  Flags are chosen by
a brightness step under the variance guard.  Either form is within 1e-4 of the
FP64 oracle, so the two lie within 2e-4 of one another."""
import os

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

W, H = 150, 61


def _mask():
    m = np.zeros((H, W), bool)
    m[10, 5:30] = True                 # one row
    m[20:22, 34:60] = True             # two rows
    m[26:34, 70] = True                # a column over two tiles
    m[32, 75:77] = m[39, 75:77] = True   # the first and last row of a tile
    m[40:43, 70:73] = True             # three rows
    m[48, 100] = m[48, 103] = m[50, 101] = m[55, 98] = True
    m[0, 0] = m[0, W - 1] = m[H - 1, 0] = m[H - 1, W - 1] = True
    m[H - 2:, 60:64] = True
    return torch.from_numpy(m)


def _alpha(frames, r, mixed, stage):
    import paper_2303_02608_gb300 as m
    env = {"ESIM_AD_SPARSE_MAX": "4294967295", "ESIM_AD_SPARSE_STAGE": stage}
    old = {k: os.environ.get(k) for k in env}
    os.environ.update(env)
    try:
        sim = m.Simulator(m.SimConfig(width=W, height=H, radius=r, frames=2, contrast=0.5, guard_kappa=1.0,
                                      radiance_fmt=m.ESIM_AD_LOGLUMA_F16, feature_fmt=m.ESIM_AD_FEAT_F32,
                                      precision=m.ESIM_AD_MIXED if mixed else m.ESIM_AD_FP32))
    finally:
        for k, v in old.items():
            os.environ.pop(k, None)
            if v is not None:
                os.environ[k] = v
    for f in frames:
        sim.push(f)
    alpha, flags = sim.denoised()
    sim.close()
    return alpha, flags


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("r", [1, 2, 3, 7, 8, 9, 10, 13])
def test_boxes_match_windows_read_through_l1(r, mixed):
    mask = _mask()
    g = torch.Generator(device="cuda").manual_seed(r)
    feat = 2.0 * torch.rand(7, H, W, generator=g, device="cuda") - 1.0
    frames = []
    for t in range(3):
        y = 0.01 * torch.randn(H, W, generator=g, device="cuda") + 2.0 * (t == 2) * mask.cuda()
        frames.append({"radiance": y.half(), "variance": torch.zeros(H, W, device="cuda"),
                       "normal": feat[:3].contiguous(), "depth": feat[3].contiguous(), "albedo": feat[4:].contiguous()})
    a, flags = _alpha(frames, r, mixed, "1")
    b, flags_b = _alpha(frames, r, mixed, "0")
    assert torch.equal(flags.cpu() != 0, mask) and torch.equal(flags, flags_b)
    assert (a - b).abs().max().item() <= 2e-4
