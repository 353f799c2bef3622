"""Contexts whose kernels need different amounts of shared memory, alive together:
each goes on working after another one was made."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

W, H = 70, 44


def _frames(n, mixed):
    rng = np.random.default_rng(3)
    out = []
    for _ in range(n):
        feat = torch.from_numpy(np.kron(rng.uniform(0, 1, (7, 11, 14)), np.ones((4, 5))).astype(np.float32)).cuda()
        rad = torch.from_numpy(rng.uniform(0.1, 1.0, (1, H, W)).astype(np.float32)).cuda()
        out.append({"radiance": rad[0].log().half(), "features": feat.bfloat16()} if mixed else
                   {"radiance": rad, "normal": feat[:3].contiguous(), "depth": feat[3].contiguous(),
                    "albedo": feat[4:].contiguous()})
    return out


def _config(m, radius, mixed):
    extra = dict(radiance_fmt=m.ESIM_AD_LOGLUMA_F16, feature_fmt=m.ESIM_AD_FEAT_BF16,
                 precision=m.ESIM_AD_MIXED) if mixed else {}
    return m.SimConfig(width=W, height=H, radius=radius, frames=3, contrast=0.2, rgb=False, **extra)


def _agree(a, b):
    """Two runs [(alpha, flags) per frame] of one sequence.  A pixel's alpha is
    the regression of the frame that flagged it last, within 1e-4 of the oracle
    in either run.  Sums of few flagged pixels are taken in an order that varies,
    so a pixel at the threshold of the flag test may be flagged in one run only."""
    same = torch.stack([fa == fb for (_, fa), (_, fb) in zip(a, b)]).all(0)
    assert same.float().mean().item() > 0.99
    assert (a[-1][0] - b[-1][0])[same].abs().max().item() <= 2e-4


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("radii", [(7, 3), (3, 7, 1), (15, 2)])
def test_simulators_of_different_radii_in_turn(radii, mixed):
    import paper_2303_02608_gb300 as m
    frames = _frames(4, mixed)

    def step(sim, f):
        sim.push(f)
        return sim.denoised()

    alone = []
    for r in radii:
        sim = m.Simulator(_config(m, r, mixed))
        alone.append([step(sim, f) for f in frames])
        sim.close()
    sims = [m.Simulator(_config(m, r, mixed)) for r in radii]
    for _ in range(2):   # frame 0 and adaptive frames, before and after a reset
        runs = list(zip(*[[step(sim, f) for sim in sims] for f in frames]))
        for sim, run, ref in zip(sims, runs, alone):
            _agree(run, ref)
            sim.reset()
    for sim in sims:
        sim.close()


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("radii", [(7, 3), (3, 15, 1)])
def test_batches_of_different_radii_in_turn(radii, mixed):
    import paper_2303_02608_gb300 as m
    frames = _frames(4, mixed)

    def step(batch, f):
        batch.step([f, f])
        return batch.denoised(1)

    alone = []
    for r in radii:
        batch = m.Batch([_config(m, r, mixed)] * 2)
        alone.append([step(batch, f) for f in frames])
        batch.close()
    batches = [m.Batch([_config(m, r, mixed)] * 2) for r in radii]
    runs = list(zip(*[[step(batch, f) for batch in batches] for f in frames]))
    for batch, run, ref in zip(batches, runs, alone):
        _agree(run, ref)
        batch.close()
