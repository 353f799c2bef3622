"""The row boxes of densely flagged adaptive frames: chosen flag patterns (runs of
pixels that need one box, runs over more rows than a box holds, every number of
lanes per pixel, clipped tiles), by a brightness step under the variance guard,
against the window-box form of the same frame.  Each form is within 1e-4 of the
FP64 oracle, so the two lie within 2e-4 of one another."""
import os

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

W, H = 101, 21


def _mask(kind, rng):
    m = np.zeros((H, W), bool)
    if kind == "all":
        m[:] = True
    elif kind == "edges":      # 1, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 256 flagged pixels of a tile
        for i, n in enumerate([1, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 256][rng.integers(0, 12):][:6]):
            y, x = np.unravel_index(rng.permutation(256)[:n], (8, 32))
            m[8 * (i // 3) + y, 32 * (i % 3) + x] = True
    else:                      # "spread": a unit's pixels lie on all rows after a dense start
        for ty in (0, 8):
            m[ty:ty + 3, 0:32] = True
            m[ty + 3:ty + 8, 3:10] = True          # 131 pixels: 32 lanes over five rows
            m[ty, 32:58] = True
            m[ty + 1:ty + 8, 40] = True            # 33 pixels: eight of them over seven rows
            m[ty:ty + 8, 64] = True                # a column
            m[ty:ty + 8, W - 1] = True             # at the image's border
    return m


def _alpha(frames, r, T, precision, path):
    import paper_2303_02608_gb300 as m
    keys = {"ESIM_AD_SPARSE_MAX": path, "ESIM_AD_ROWS_MIN": "0"}
    old = {k: os.environ.pop(k, None) for k in keys}
    os.environ.update(keys)
    try:
        sim = m.Simulator(m.SimConfig(width=W, height=H, radius=r, frames=T, contrast=0.5, mode=m.ESIM_AD_ADAPTIVE,
                                      radiance_fmt=m.ESIM_AD_LOGLUMA_F16, feature_fmt=m.ESIM_AD_FEAT_F32,
                                      precision=precision, guard_kappa=1.0))
    finally:
        for k in keys:
            os.environ.pop(k, None)
            if old[k] is not None:
                os.environ[k] = old[k]
    for f in frames:
        sim.push({k: v.cuda() for k, v in f.items()})
    a, flags = sim.denoised()
    a, flags, stats = a.cpu().numpy(), flags.cpu().numpy(), sim.stats()
    sim.close()
    return a, flags, stats


@pytest.mark.parametrize("kind,seed", [("all", 0), ("edges", 1), ("edges", 2), ("spread", 3)])
@pytest.mark.parametrize("precision,r,T", [("mixed", 7, 3), ("mixed", 1, 2), ("mixed", 8, 2),
                                           ("fp32", 3, 3), ("fp32", 4, 2)])
def test_queue_form_matches_window_boxes(precision, r, T, kind, seed):
    import paper_2303_02608_gb300 as m
    rng = np.random.default_rng(seed)
    mask = torch.from_numpy(_mask(kind, rng))
    feat = torch.from_numpy(rng.uniform(-1, 1, (7, H, W)).astype(np.float32))
    frames = []
    for t in range(3):
        y = torch.from_numpy(rng.normal(0.0, 0.01, (H, W)).astype(np.float32)) + 2.0 * (t == 2) * mask
        frames.append({"radiance": y.half(), "variance": torch.zeros(H, W), "normal": feat[:3].contiguous(),
                       "depth": feat[3].contiguous(), "albedo": feat[4:].contiguous()})
    prec = m.ESIM_AD_MIXED if precision == "mixed" else m.ESIM_AD_FP32
    a, flags, sa = _alpha(frames, r, T, prec, "0")
    b, flags_b, sb = _alpha(frames, r, T, prec, "4294967295")
    assert np.array_equal(flags != 0, mask.numpy()) and np.array_equal(flags, flags_b)
    assert np.abs(a - b)[mask.numpy()].max() <= 2e-4
    assert sa["regressions"] == sb["regressions"]
