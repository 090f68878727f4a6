"""The adjoint where a loss gradient or a frame colour is infinite or NaN: it
reaches the records and pixels whose disc holds it, and no others, although
both passes read the pixels (records) of neighbouring discs together. Bit for
bit against the same call with a finite value in its place."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2510_15876_gb300 import _lib as L  # noqa: E402

T_NOW = 1.0


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_15876_gb300.build import build
    build()
    return torch.device("cuda:0")


def _filled(dev, W, H, b, R):
    from paper_2510_15876_gb300.api import Reconstructor
    g = torch.Generator(dev).manual_seed(W + R)
    n = 2 * W * H * b
    pos = torch.rand(n, 4, generator=g, device=dev) * torch.tensor([W - 0.01, H - 0.01, 1.0, 1.0], device=dev)
    rec = Reconstructor(W, H, b, radius=R, device=dev)
    rec.insert(pos, torch.rand(n, 4, generator=g, device=dev), torch.randn(n, 2, generator=g, device=dev))
    rec.estimate_gradients(T_NOW)
    rec.reproject(T_NOW)
    return rec


def _bins(rec):
    _, frec, _ = rec.export_frame()
    return np.floor(frec[:, 0]).astype(int), np.floor(frec[:, 1]).astype(int)


@pytest.mark.parametrize("R", [0, 1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_a_loss_gradient_reaches_the_records_of_its_disc_only(dev, R, value):
    W, H = 41, 33
    rec = _filled(dev, W, H, 3, R)
    rec.reconstruct(T_NOW)
    g = torch.randn(H, W, 4, generator=torch.Generator().manual_seed(1)).to(dev)
    at = ((20, 16), (0, 0), (40, 20), (7, 32))
    bad = g.clone()
    for x, y in at:
        g[y, x] = 0.0
        bad[y, x] = value
    want, _ = rec.backward(g, want_params=False)
    got, _ = rec.backward(bad, want_params=False)
    bx, by = _bins(rec)
    near = np.zeros(len(bx), bool)
    for x, y in at:
        near |= (bx - x) ** 2 + (by - y) ** 2 <= R * R
    got, want = got.cpu().numpy(), want.cpu().numpy()
    assert near.any() and not np.isfinite(got[near]).any()
    np.testing.assert_array_equal(got[~near], want[~near])
    rec.close()


@pytest.mark.parametrize("W,H,R", [(41, 33, 3), (41, 33, 5), (700, 640, 4)])   # a pixel a thread, and three rows
def test_a_colour_reaches_the_pixels_whose_disc_holds_it_only(dev, W, H, R):
    """The pixels around the bad record have widths held at their minimum, which
    have no gradient; every other pixel's share of the parameter gradients is
    as without it."""
    rec = _filled(dev, W, H, 3, R)
    bx, by = _bins(rec)
    e = int(np.flatnonzero((bx == W // 2) & (by == H // 2))[0])
    ys, xs = np.mgrid[0:H, 0:W]
    near = ((xs - W // 2) ** 2 + (ys - H // 2) ** 2 <= R * R).reshape(-1)
    rng = np.random.default_rng(0)
    gt = rng.uniform(0.5, 1.5, W * H).astype(np.float32)
    rec.import_map(L.AFR_MAP_GT, np.where(near, 1e4, gt))
    for m in (L.AFR_MAP_GX, L.AFR_MAP_GY):
        rec.import_map(m, np.where(near, 1e-3, 1.0))
    theta = (-1.0, 2.0, 3.0, 1.0, 0.0, 4.0)   # wide where the ratio G_t / G_s is small, at the minimum where it is large
    colors = torch.rand(rec.query()["frame"], 3, generator=torch.Generator().manual_seed(2)).to(dev)
    gout = torch.randn(H, W, 4, generator=torch.Generator().manual_seed(3)).to(dev)
    got = []
    for value in (0.5, float("nan"), float("inf")):
        colors[e] = value
        rec.set_frame_colors(colors)
        rec.reconstruct(T_NOW, theta)
        got.append(rec.backward(gout, want_colors=False)[1].cpu())
    sigma_s, sigma_t = rec.export_map(L.AFR_MAP_SIGMA_S), rec.export_map(L.AFR_MAP_SIGMA_T)
    assert (sigma_s[near] == 0.5).all() and (sigma_t[near] == np.float32(0.05)).all()
    assert (sigma_s[~near] > 0.5).all() and (sigma_t[~near] > 0.05).all()
    assert got[0].abs().max() > 0 and torch.isfinite(got[0]).all()
    assert torch.equal(got[1], got[0]) and torch.equal(got[2], got[0])
    rec.close()
