"""The exhaustive regression's two forms (tiles of 16 x 4 pixels, four lanes each,
for large windows; tile-staged otherwise) against the FP64 oracle: whole and
partial tiles, windows larger than the image.
Tolerance: alpha within 1e-4."""
import numpy as np
import pytest
import torch

from oracle import EXHAUSTIVE, Oracle, OracleConfig
from scenes import Scene, SceneConfig

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,r,T,n", [
    (1, 1, 1, 1, 2),      # one pixel
    (1, 1, 7, 5, 2),
    (16, 4, 7, 5, 6),     # large windows: exactly one tile
    (17, 5, 8, 5, 6),     # one pixel past it
    (16, 4, 3, 2, 3),     # exactly one tile
    (17, 5, 3, 2, 3),     # one pixel past it
    (40, 21, 7, 5, 7),    # interior and clipped tiles, a full temporal window
])
def test_exhaustive_alpha_matches_oracle(W, H, r, T, n):
    import paper_2303_02608_gb300 as m
    cfg = SceneConfig(kind="rects", width=W, height=H, frames=n, spp=2, seed=W + r, rgb=True,
                      n_rects=max(3, W * H // 150), bg_depth=10.0)
    sim = m.Simulator(m.SimConfig(width=W, height=H, radius=r, frames=T, contrast=0.2, mode=m.ESIM_AD_EXHAUSTIVE))
    orc = Oracle(OracleConfig(W, H, radius=r, frames=T, channels=3, mode=EXHAUSTIVE, contrast=0.2))
    for f in Scene(cfg).sequence():
        sim.push({k: f[k].cuda() for k in ("radiance", "normal", "albedo", "depth")})
        orc.push({k: f[k].numpy() for k in ("radiance", "normal", "albedo", "depth")})
        a, flags = sim.denoised()
        assert np.abs(a.cpu().numpy() - orc.outputs()["alpha"].reshape(H, W)).max() <= 1e-4
        assert bool(torch.all(flags == 1))
    stats = sim.stats()
    assert stats["regressions"] == W * H * n
    sim.close()


@pytest.mark.parametrize("W,H,r,T,n", [
    (5, 40, 7, 5, 6),     # narrower than the window
    (40, 5, 7, 5, 6),     # lower
    (3, 17, 8, 5, 6),     # both
    (8, 8, 7, 6, 7),      # every offset of the window reaches some pixel
    (7, 9, 7, 5, 6),      # all but the outermost columns
])
def test_exhaustive_images_smaller_than_the_window(W, H, r, T, n):
    test_exhaustive_alpha_matches_oracle(W, H, r, T, n)
