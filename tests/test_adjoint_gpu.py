"""Differentiation form on the GPU: forward alpha against the FP64 oracle, and
the hand-written adjoint's gradients against (a) FP64 central finite
differences of the oracle's loss (h = 1e-4) and (b) autograd through the FP64
dense reference (least squares on the augmented system, and the normal
equations), on a 32x32 crop (radiance and the seven bandwidths)."""
import numpy as np
import pytest
import torch

from oracle import EXHAUSTIVE, Oracle, OracleConfig
from scenes import Scene, SceneConfig, preset
from wlr_reference import log_luminance, mse_loss, wlr_alpha

pytestmark = pytest.mark.gpu

R, T, EPS, RIDGE = 3, 3, 1e-3, 1e-4
B = [0.7, 1.3, 1.0, 2.0, 0.5, 1.0, 1.5]


def _crop(cfg, x0, y0, w, h, n):
    fr = Scene(cfg).sequence(n)
    sl = (slice(y0, y0 + h), slice(x0, x0 + w))
    rad = torch.stack([f["radiance"][(slice(None),) + sl] for f in fr]).contiguous()
    feat = torch.stack([torch.cat([f["normal"], f["depth"][None], f["albedo"]])[(slice(None),) + sl]
                        for f in fr]).contiguous()
    clean = torch.stack([f["clean"][(slice(None),) + sl] for f in fr]).contiguous()
    return rad, feat, clean


def _oracle_alpha(rad, feat, b, rows=None):
    F, C, H, W = rad.shape
    o = Oracle(OracleConfig(W, H, radius=R, frames=T, channels=C, mode=EXHAUSTIVE, bandwidth=list(b),
                            ridge=RIDGE, log_eps=EPS))
    out = []
    for t in range(F):
        o.push({"radiance": rad[t].numpy(), "normal": feat[t, 0:3].numpy(), "depth": feat[t, 3].numpy(),
                "albedo": feat[t, 4:7].numpy()}, rows)
        out.append(o.outputs()["alpha"])
    return np.stack(out)


def _gpu(rad, feat, clean, b):
    from paper_2303_02608_gb300 import wlr
    rd = rad.cuda().requires_grad_(True)
    bd = torch.tensor(b, dtype=torch.float32, device="cuda", requires_grad=True)
    alpha = wlr(rd, feat.cuda(), bd, radius=R, frames=T, log_eps=EPS, ridge=RIDGE)
    loss = ((alpha - log_luminance(clean.cuda(), EPS)) ** 2).mean()
    loss.backward()
    return alpha.detach().cpu(), rd.grad.cpu(), bd.grad.cpu(), float(loss.detach())


RECTS = SceneConfig(kind="rects", width=160, height=120, frames=6, spp=2, seed=4, rgb=True, n_rects=12,
                    bg_depth=10.0)


def test_forward_alpha_matches_oracle():
    rad, feat, clean = _crop(RECTS, 20, 30, 48, 40, 5)
    alpha, _, _, _ = _gpu(rad, feat, clean, B)
    ref = _oracle_alpha(rad, feat, B)
    err = np.abs(alpha.numpy() - ref).max()
    assert err <= 1e-4, err


@pytest.mark.parametrize("solver", ["lstsq", "solve"])
def test_gradients_match_dense_autograd_reference(solver):
    """Against autograd through the FP64 dense regression: least squares on the
    sqrt(w)-weighted augmented system, and the weighted normal equations."""
    rad, feat, clean = _crop(RECTS, 40, 40, 32, 32, 4)
    _, g_rad, g_b, _ = _gpu(rad, feat, clean, B)
    b64 = torch.tensor(B, dtype=torch.float64, requires_grad=True)
    r64 = rad.double().requires_grad_(True)
    mse_loss(wlr_alpha(r64, feat.double(), b64, R, T, eps=EPS, ridge=RIDGE, solver=solver),
             clean.double(), EPS).backward()
    gb_ref = b64.grad.numpy()
    np.testing.assert_allclose(g_b.numpy(), gb_ref, rtol=2e-3, atol=2e-3 * np.abs(gb_ref).max())
    gr_ref = r64.grad.numpy()
    scale = np.abs(gr_ref).max()
    err = np.abs(g_rad.numpy() - gr_ref)
    print(f"radiance gradient vs FP64 {solver}: max abs {err.max():.3e} (scale {scale:.3e}), "
          f"max rel where |g| > 1e-2 scale {np.max(err[np.abs(gr_ref) > 1e-2 * scale] / np.abs(gr_ref[np.abs(gr_ref) > 1e-2 * scale])):.3e}")
    np.testing.assert_allclose(g_rad.numpy(), gr_ref, rtol=1e-4, atol=1e-5 * scale)


def test_gradients_match_oracle_finite_differences():
    rad, feat, clean = _crop(RECTS, 40, 40, 32, 32, 4)
    _, g_rad, g_b, _ = _gpu(rad, feat, clean, B)
    y_clean = log_luminance(clean.double(), EPS).numpy()

    def loss(r, b):
        return float(np.mean((_oracle_alpha(r, feat, b) - y_clean) ** 2))

    hb = 1e-4
    for j in range(7):
        bp, bm = list(B), list(B)
        bp[j] += hb
        bm[j] -= hb
        fd = (loss(rad, bp) - loss(rad, bm)) / (2 * hb)
        assert g_b[j].item() == pytest.approx(fd, rel=2e-3, abs=1e-6)
    # radiance: h = 1e-4; the oracle reads float32, so the step actually taken
    # is the float32 difference of the perturbed and original values (FP64 sums)
    he = 1e-4
    for (t, c, yy, xx) in [(0, 0, 10, 12), (2, 1, 0, 31), (3, 2, 16, 16), (1, 0, 31, 0)]:
        rp, rm = rad.clone(), rad.clone()
        rp[t, c, yy, xx] += he
        rm[t, c, yy, xx] -= he
        step = float(rp[t, c, yy, xx]) - float(rm[t, c, yy, xx])
        fd = (loss(rp, B) - loss(rm, B)) / step
        assert g_rad[t, c, yy, xx].item() == pytest.approx(fd, rel=2e-3, abs=1e-7)


@pytest.mark.parametrize("w,h,n,r,frames", [
    (32, 8, 2, 3, 2),     # exactly one centre tile
    (33, 9, 3, 2, 3),     # one pixel past it
    (7, 5, 3, 3, 2),      # an image smaller than the window
    (70, 20, 2, 4, 2),    # three tiles across and down
    (36, 20, 3, 9, 3),    # tile sums larger than the workspace: the gather over the centres
])
def test_radiance_gradient_paths(w, h, n, r, frames):
    from paper_2303_02608_gb300 import wlr
    rad, feat, clean = _crop(RECTS, 20, 30, w, h, n)
    rd = rad.cuda().requires_grad_(True)
    bd = torch.tensor(B, dtype=torch.float32, device="cuda", requires_grad=True)
    alpha = wlr(rd, feat.cuda(), bd, radius=r, frames=frames, log_eps=EPS, ridge=RIDGE)
    ((alpha - log_luminance(clean.cuda(), EPS)) ** 2).mean().backward()
    r64, b64 = rad.double().requires_grad_(True), torch.tensor(B, dtype=torch.float64, requires_grad=True)
    mse_loss(wlr_alpha(r64, feat.double(), b64, r, frames, eps=EPS, ridge=RIDGE), clean.double(), EPS).backward()
    gb, gr = b64.grad.numpy(), r64.grad.numpy()
    np.testing.assert_allclose(bd.grad.cpu().numpy(), gb, rtol=2e-3, atol=2e-3 * np.abs(gb).max())
    np.testing.assert_allclose(rd.grad.cpu().numpy(), gr, rtol=1e-4, atol=1e-5 * np.abs(gr).max())


def test_masked_centres_add_nothing():
    """Centres whose alpha the loss leaves out contribute nothing, even where
    their inputs are not numbers."""
    from paper_2303_02608_gb300 import wlr
    rad, feat, _ = _crop(RECTS, 20, 30, 40, 16, 1)
    rad[0, :, 0, 0] = float("nan")
    rd = rad.cuda().requires_grad_(True)
    bd = torch.tensor(B, dtype=torch.float32, device="cuda", requires_grad=True)
    wlr(rd, feat.cuda(), bd, radius=R, frames=1)[0, :, 20:].sum().backward()
    assert torch.isfinite(bd.grad).all()
    assert torch.isfinite(rd.grad[:, :, :, 17:]).all() and not rd.grad[0, :, :, 4:10].any()


def test_masked_centres_add_nothing_in_wide_windows():
    """The same where the tile sums do not fit the workspace."""
    from paper_2303_02608_gb300 import wlr
    rad, feat, _ = _crop(RECTS, 20, 30, 60, 16, 3)
    rad[0, :, 0, 0] = float("nan")
    rd = rad.cuda().requires_grad_(True)
    bd = torch.tensor(B, dtype=torch.float32, device="cuda", requires_grad=True)
    wlr(rd, feat.cuda(), bd, radius=9, frames=3)[0, :, 40:].sum().backward()
    assert torch.isfinite(bd.grad).all()
    assert torch.isfinite(rd.grad[0, :, :, 31:]).all() and not rd.grad[0, :, :, 10:31].any()


def test_backward_is_deterministic():
    rad, feat, clean = _crop(RECTS, 0, 0, 64, 48, 4)
    a = _gpu(rad, feat, clean, B)
    b = _gpu(rad, feat, clean, B)
    assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])


def test_full_size_sequence_sampled():
    """The differentiation workload at full size: 512x512, 16 frames, 2 spp;
    alpha sampled on a band of rows against the oracle, gradients finite."""
    sc = Scene(preset("rects512"))
    fr = sc.sequence()
    rad = torch.stack([f["radiance"] for f in fr])
    feat = torch.stack([torch.cat([f["normal"], f["depth"][None], f["albedo"]]) for f in fr])
    clean = torch.stack([f["clean"] for f in fr])
    b = [1.0] * 7
    alpha, g_rad, g_b, loss = _gpu(rad, feat, clean, b)
    ref = _oracle_alpha(rad, feat, b, rows=(250, 254))
    err = np.abs(alpha.numpy()[:, 250:254] - ref[:, 250:254]).max()
    assert err <= 1e-4, err
    assert np.isfinite(loss) and torch.isfinite(g_rad).all() and torch.isfinite(g_b).all()


def test_infinite_share_of_the_bandwidth_gradient():
    """A centre tile's share of the gradient that exceeds FP32's range leaves the
    gradient infinite with its sign.  Rows of equal pixels make the 32 centres of
    one row of the middle tile contribute the same, so that scaling the loss by
    a power of two takes their sum past the range and no summand near it (each
    at most 2^124).  Scaling is exact but for underflows at the smaller scale."""
    from paper_2303_02608_gb300 import wlr
    rng = np.random.default_rng(6)
    rows = torch.from_numpy(rng.uniform(0.0, 1.0, (8, 24)).astype(np.float32)).cuda()
    rad = torch.exp(20.0 * (rows[0] - 0.5)).view(1, 1, 24, 1).expand(1, 1, 24, 96).contiguous()
    feat = (2.0 * rows[1:]).view(1, 7, 24, 1).expand(1, 7, 24, 96).contiguous()
    g = torch.zeros(1, 24, 96, device="cuda")
    g[0, 12, 32:64] = 1.0

    def grad(scale):
        bd = torch.ones(7, device="cuda", requires_grad=True)
        alpha = wlr(rad, feat, bd, radius=7, frames=1)
        return torch.autograd.grad(alpha, bd, g * scale)[0].cpu().numpy().astype(np.float64)

    one = grad(1.0)
    shares = np.abs(one) * 0.5 * np.log2(np.e)          # dL/db = sum of shares / (k^2 b), k^2 = log2(e) / 2
    scale = 2.0 ** np.floor(124 - np.log2(shares.max() / 32))
    got, want = grad(scale), one * scale
    over = shares * scale >= 2.0 ** 128
    assert over.any() and not np.isnan(got).any()
    np.testing.assert_array_equal(got[over], np.sign(want[over]) * np.inf)
    fits = np.abs(want) < 0.99 * float(np.finfo(np.float32).max)
    np.testing.assert_allclose(got[fits], want[fits], rtol=1e-4)
