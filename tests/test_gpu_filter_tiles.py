"""The filter at the edges of its tiles and row ranges: images that end inside
a CTA tile or a 2x2 block, every tile shape, the smallest and largest discs,
rows with none, fewer than 32 and many records (the gather's two row steps),
16-bit colours; against the FP64 oracle given its widths. The bound is the
parity tests' 1e-5 relative: every term is nonnegative, so the FP32 sums and
the 2^-22 of each weight leave a few 1e-6."""
import numpy as np
import pytest
import torch

import oracle

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


def _batch(seed, W, H, n, crowd, gap):
    """n samples; a share `crowd` of them on the first two pixels, none in a band of rows."""
    rng = np.random.default_rng(seed)
    x, y = rng.uniform(0, W, n), rng.uniform(0, H, n)
    few = rng.random(n) < crowd
    x[few], y[few] = rng.uniform(0, min(W, 2), few.sum()), rng.uniform(0, 1, few.sum())
    if gap:
        y = np.where((y > H * 0.4) & (y < H * 0.4 + gap), 0.25, y)
    x, y = (np.minimum(v.astype(np.float32), np.nextafter(np.float32(m), np.float32(0))) for v, m in ((x, W), (y, H)))
    pos = np.stack([x, y, np.sort(rng.uniform(0, 1, n)).astype(np.float32), np.ones(n, np.float32)], 1)
    col = np.zeros((n, 4), np.float32)
    col[:, :3] = rng.uniform(0, 1, (n, 3))
    return {"pos": np.ascontiguousarray(pos), "color": col,
            "motion": rng.uniform(-3, 3, (n, 2)).astype(np.float32)}


@pytest.mark.parametrize("W,H,b,R,tbx,ct,per_pixel,crowd,gap", [
    (1, 1, 4, 4, 4, "f32", 3, 0.0, 0), (2, 70, 8, 8, 2, "f32", 8, 0.1, 9), (67, 5, 3, 1, 16, "f32", 0.2, 0.0, 0),
    (41, 35, 32, 8, 16, "f32", 32, 0.0, 0), (33, 17, 24, 3, 8, "f16", 24, 0.2, 4), (31, 66, 16, 5, 2, "bf16", 12, 0.0, 7),
    (63, 49, 1, 8, 4, "f32", 0.3, 0.3, 12), (130, 18, 32, 2, 8, "f32", 40, 0.0, 0), (19, 23, 12, 0, 4, "f16", 12, 0.5, 0),
    (16, 32, 32, 6, 4, "bf16", 30, 0.0, 0)])
def test_filter_edges_match_oracle(dev, W, H, b, R, tbx, ct, per_pixel, crowd, gap):
    from paper_2510_15876_gb300.api import Reconstructor, set_tuning, to_device_batch
    batch = _batch(W * 100 + H, W, H, max(1, int(W * H * per_pixel)), crowd, gap)
    rec = Reconstructor(W, H, b, radius=R, color_type=ct, device=dev)
    set_tuning(rec, R, tbx)
    tensors = to_device_batch(batch, dev, rec.color_dtype)
    rec.insert(*tensors)
    batch["color"] = tensors[1].float().cpu().numpy()      # as stored
    ring = oracle.Ring(W, H, b)
    ring.insert(batch["pos"], batch["color"], batch["motion"])
    rec.estimate_gradients(T_NOW)
    rec.reproject(T_NOW)
    ss, st = (v.astype(np.float32) for v in oracle.sigma(ring.count, W, H, oracle.gradients(ring, T_NOW),
                                                         oracle.DEFAULT_THETA))
    rec.import_map(L.AFR_MAP_SIGMA_S, ss)
    rec.import_map(L.AFR_MAP_SIGMA_T, st)
    img = rec.reconstruct(T_NOW, flags=L.AFR_RECON_KEEP_SIGMA).cpu().numpy().reshape(-1, 4).astype(np.float64)
    rec.close()
    off, frec, _, _ = oracle.reproject(ring, T_NOW)
    ref = oracle.filter_image(W, H, off, frec, ss.astype(np.float64), st.astype(np.float64), R=R)
    hole = ref[:, 3] == 0
    np.testing.assert_array_equal(img[hole], 0.0)
    err = np.abs(img[~hole, :3] - ref[~hole, :3]) / np.maximum(np.abs(ref[~hole, :3]), 1e-3)
    assert err.size == 0 or err.max() <= 1e-5


@pytest.mark.parametrize("W,H,b,R,ct,per_pixel,crowd,gap", [
    (1, 1, 2, 4, "f32", 1, 0.0, 0), (9, 70, 8, 4, "f32", 8, 0.1, 9), (67, 21, 3, 5, "f32", 0.4, 0.0, 0),
    (30, 35, 24, 3, "f16", 24, 0.0, 0), (33, 17, 8, 8, "f32", 8, 0.2, 4), (40, 26, 16, 0, "bf16", 12, 0.0, 7),
    (64, 40, 4, 2, "f32", 3, 0.0, 0)])
def test_adjoint_edges_match_oracle(dev, W, H, b, R, ct, per_pixel, crowd, gap):
    """Both passes of the adjoint where they can go wrong: borders, discs known
    at compile time and not, neighbouring records in one bin, in adjacent bins,
    across gaps and row ends, an odd number of records; either output alone.
    Bounds as in the parity test of the adjoint."""
    from paper_2510_15876_gb300.api import Reconstructor, to_device_batch
    batch = _batch(W * 10 + H, W, H, max(1, int(W * H * per_pixel)), crowd, gap)
    rec = Reconstructor(W, H, b, radius=R, color_type=ct, device=dev)
    tensors = to_device_batch(batch, dev, rec.color_dtype)
    rec.insert(*tensors)
    ring = oracle.Ring(W, H, b)
    ring.insert(batch["pos"], tensors[1].float().cpu().numpy(), batch["motion"])
    rec.estimate_gradients(T_NOW)
    rec.reproject(T_NOW)
    maps = [np.asarray(v).astype(np.float32) for v in oracle.gradients(ring, T_NOW)[1:]]
    for m, v in zip((L.AFR_MAP_GX, L.AFR_MAP_GY, L.AFR_MAP_GT), maps):
        rec.import_map(m, v)
    theta = np.array([0.9, 0.15, 2.4, 1.1, 0.02, 0.7])
    rec.reconstruct(T_NOW, theta)
    g = np.random.default_rng(W).normal(size=(W * H, 4)).astype(np.float32)
    gt = torch.from_numpy(g).to(dev).reshape(H, W, 4)
    gcol, gprm = rec.backward(gt)
    only_colors, _ = rec.backward(gt, want_params=False)
    _, only_params = rec.backward(gt, want_colors=False)
    off, frec, _, _ = oracle.reproject(ring, T_NOW)
    wcol, wprm = oracle.backward(ring.count, W, H, (None, *(v.astype(np.float64) for v in maps)), off, frec,
                                 g[:, :3].astype(np.float64), theta, R=R)
    for got in (gprm, only_params):
        np.testing.assert_allclose(got.cpu().numpy(), wprm, rtol=2e-4, atol=1e-4 * max(np.abs(wprm).max(), 1e-30))
    for got in (gcol, only_colors):
        np.testing.assert_allclose(got.cpu().numpy()[:len(wcol)], wcol, rtol=1e-3,
                                   atol=1e-5 * max(np.abs(wcol).max(initial=0.0), 1e-30))
    rec.close()
