"""Row boxes against the tile-staged form on the same densely flagged frames.
Both give a pixel the same lanes and add its sums in the same order, so the
results are the same bit for bit, whichever form a frame's flagged total picks.
Flags are chosen by a brightness step under the variance guard; the totals give
work items of 16, 32, 64, 128 and 256 pixels (the whole tile, where row boxes
are taken by default), and the patterns every number of lanes per pixel, units
over more rows than a box holds, and clipped tiles."""
import os

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

W, H = 1017, 637    # the last tiles of a row and of a column are partial


def _mask(total, seed):
    """About `total` flagged pixels: whole tiles up to three quarters of them, the rest in
    tiles of one pattern each."""
    rng = np.random.default_rng(seed)
    m = np.zeros((H + 8, W + 32), bool)
    tiles = [(y, x) for y in range(0, H, 8) for x in range(0, W, 32)]
    left = total
    for i, k in enumerate(rng.permutation(len(tiles))):
        y, x = tiles[k]
        t = np.zeros((8, 32), bool)
        if left > total // 4:
            t[:] = True
        elif i % 4 == 0:       # 131 pixels: one lane each, the last whole warp over five rows
            t[:3] = True
            t[3:, 4:11] = True
        elif i % 4 == 1:       # a column: 32 lanes per pixel
            t[:, 17] = True
        elif i % 4 == 2:       # 33 pixels: four lanes each
            t[0] = True
            t[7, 31] = True
        else:
            t.flat[rng.permutation(256)[:rng.integers(1, 257)]] = True
        m[y:y + 8, x:x + 32] = t
        left -= int(m[y:min(y + 8, H), x:min(x + 32, W)].sum())
        if left <= 0:
            break
    return torch.from_numpy(m[:H, :W].copy())


def _simulator(m, r, T, mixed, env):
    env = {"ESIM_AD_SPARSE_MAX": "0", **env}
    old = {k: os.environ.get(k) for k in env}
    os.environ.update(env)
    try:
        return m.Simulator(m.SimConfig(width=W, height=H, radius=r, frames=T, contrast=0.5,
                                       radiance_fmt=m.ESIM_AD_LOGLUMA_F16, feature_fmt=m.ESIM_AD_FEAT_F32,
                                       precision=m.ESIM_AD_MIXED if mixed else m.ESIM_AD_FP32, guard_kappa=1.0,
                                       event_capacity=16 * W * H))
    finally:
        for k, v in old.items():
            os.environ.pop(k, None)
            if v is not None:
                os.environ[k] = v


def _frames(mask):
    g = torch.Generator(device="cuda").manual_seed(2)
    feat = 2.0 * torch.rand(7, H, W, generator=g, device="cuda") - 1.0
    out = []
    for t in range(3):
        y = 0.01 * torch.randn(H, W, generator=g, device="cuda") + 2.0 * (t == 2) * mask.cuda()
        out.append({"radiance": y.half(), "variance": torch.zeros(H, W, device="cuda"),
                    "normal": feat[:3].contiguous(), "depth": feat[3].contiguous(), "albedo": feat[4:].contiguous()})
    return out


@pytest.mark.parametrize("total", [20_000, 65_000, 118_000, 229_000, 393_000])
@pytest.mark.parametrize("r,T,mixed", [(7, 2, True), (3, 3, True), (1, 2, True), (3, 3, False), (1, 2, False)])
def test_row_boxes_give_the_bits_of_the_tile_staged_form(r, T, mixed, total):
    import paper_2303_02608_gb300 as m
    mask = _mask(total, total + r)
    frames = _frames(mask)
    runs = []
    for env in ({"ESIM_AD_ROWS_MIN": "4294967295"}, {"ESIM_AD_ROWS_MIN": "0"}, {}):
        sim = _simulator(m, r, T, mixed, env)
        for f in frames:
            sim.push(f)
        alpha, flags = sim.denoised()
        runs.append((alpha, flags, sim.events(), sim.stats()["regressions"], sim.profile()["neighbours"]))
        sim.close()
    tiles, *others = runs
    assert torch.equal(tiles[1].cpu() != 0, mask)
    assert len(tiles[2]) > 0
    for o in others:
        assert torch.equal(tiles[0], o[0]) and torch.equal(tiles[1], o[1])
        assert np.array_equal(tiles[2], o[2]) and tiles[3:] == o[3:]


def _form(total, r, mixed):
    """Which form takes a frame of `total` flagged pixels by default: a run whose
    row boxes are never copied reports a timeout, the tile-staged form does not."""
    import paper_2303_02608_gb300 as m
    mask = torch.zeros(H * W, dtype=torch.bool)
    mask[torch.randperm(H * W, generator=torch.Generator().manual_seed(1))[:total]] = True
    sim = _simulator(m, r, 2, mixed, {"ESIM_AD_TEST_WITHHOLD_COPY": "1"})
    try:
        for f in _frames(mask.view(H, W)):
            sim.push(f)
        assert torch.equal(sim.denoised()[1].cpu() != 0, mask.view(H, W))
        return "tiles"
    except m.EsimError as e:
        assert e.status == m.ESIM_AD_ETIMEOUT
        return "rows"
    finally:
        sim.close()


def _whole_tiles():
    """The total from which a work item is a whole tile: it holds a power of two of pixels,
    at least the flagged total over 8 items per CTA, two CTAs per SM."""
    return 2 * torch.cuda.get_device_properties(0).multi_processor_count * 8 * 129


def test_row_boxes_start_where_work_items_are_whole_tiles():
    assert _form(_whole_tiles(), 7, True) == "rows" and _form(_whole_tiles() - 1, 7, True) == "tiles"


@pytest.mark.parametrize("r,mixed,form", [(1, True, "rows"), (7, True, "rows"), (8, True, "tiles"), (1, False, "tiles"),
                                          (2, False, "tiles"), (3, False, "rows"), (4, False, "tiles")])
def test_windows_that_row_boxes_take(r, mixed, form):
    assert _form(_whole_tiles() + 5000, r, mixed) == form
