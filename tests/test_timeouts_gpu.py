"""Waits that run out: with ESIM_AD_TEST_WITHHOLD_COPY=1 a regression kernel never
issues its first copies from the second frame on and bounds each wait to 64
polls.  Nothing is in flight for that wait; it gives up, the kernel records the
timeout and returns.  The host reports ETIMEOUT at the next synchronising call,
every later call ESTATE, and after a reset the context works again."""
import os

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _run(config, env):
    import paper_2303_02608_gb300 as m
    env = {"ESIM_AD_TEST_WITHHOLD_COPY": "1", **env}
    old = {k: os.environ.get(k) for k in env}
    os.environ.update(env)
    try:
        sim = m.Simulator(config(m))
    finally:
        for k, v in old.items():
            os.environ.pop(k, None)
            if v is not None:
                os.environ[k] = v
    w, h = sim.cfg.width, sim.cfg.height
    rng = np.random.default_rng(1)
    feat = torch.from_numpy(rng.uniform(0, 1, (7, h, w)).astype(np.float32)).cuda()
    rad = torch.from_numpy(rng.uniform(0.1, 1, (3, h, w)).astype(np.float32)).cuda()
    f0 = {"radiance": rad, "normal": feat[:3].contiguous(), "depth": feat[3].contiguous(),
          "albedo": feat[4:].contiguous()}
    f1 = {k: v.flip(-1).contiguous() for k, v in f0.items()}   # features move: pixels flag
    sim.push(f0)
    first = sim.denoised()[0]
    sim.push(f1)
    for call, status in ((sim.denoised, m.ESIM_AD_ETIMEOUT), (lambda: sim.push(f0), m.ESIM_AD_ESTATE),
                         (sim.events, m.ESIM_AD_ESTATE)):
        with pytest.raises(m.EsimError) as e:
            call()
        assert e.value.status == status
    sim.reset()
    sim.push(f0)
    assert torch.equal(sim.denoised()[0], first)
    sim.close()
    torch.cuda.synchronize()


@pytest.mark.parametrize("w,h", [(16, 4), (64, 48), (333, 251)])   # one tile, fewer tiles than CTAs, more
def test_exhaustive_large_windows(w, h):
    _run(lambda m: m.SimConfig(width=w, height=h, radius=7, frames=5, contrast=0.05, mode=m.ESIM_AD_EXHAUSTIVE), {})


@pytest.mark.parametrize("mixed,r", [(False, 3), (True, 7)])
def test_row_boxes(mixed, r):
    _run(lambda m: m.SimConfig(width=101, height=45, radius=r, frames=3, contrast=0.05,
                               precision=m.ESIM_AD_MIXED if mixed else m.ESIM_AD_FP32),
         {"ESIM_AD_SPARSE_MAX": "0", "ESIM_AD_ROWS_MIN": "0"})
