"""The gradient passes over queue depths with a kernel of their own and without,
warps with a partial last group of pixels, queues that wrap and whose heads
differ, times out of order and tied, 16-bit colours, and statistics tiles of
one pixel, ragged ones, up to and above 32x32; against the FP64 oracle on the
stored colours. Bounds: 1e-5 of the value plus 5e-7 for the means and their
differences (luminances here spread over 1 within a pixel; FP32 weights good to
2^-23 and FP32 sums of up to 32 of them leave a few 2^-24 of that spread, twice
in a difference), the tile tests' bounds for the tiles."""
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


@pytest.mark.parametrize("W,H,b,S,ct,order", [
    (1, 1, 1, 1, "f32", "sorted"), (37, 5, 1, 32, "f16", "any"), (19, 13, 2, 7, "f32", "any"), (33, 31, 3, 33, "bf16", "ties"),
    (70, 41, 4, 64, "f32", "any"), (45, 23, 5, 32, "f16", "sorted"), (40, 17, 6, 1, "f32", "any"), (131, 9, 8, 16, "f16", "ties"),
    (50, 34, 12, 256, "f32", "any"), (61, 35, 16, 32, "bf16", "any"), (29, 33, 24, 20, "f16", "any"), (35, 18, 32, 32, "f32", "ties"),
    (33, 9, 31, 9, "f32", "any")])
def test_gradients_and_tiles_match_oracle(dev, W, H, b, S, ct, order):
    from paper_2510_15876_gb300.api import Reconstructor, decode_tiles
    rng = np.random.default_rng(W * 1000 + b)
    rec = Reconstructor(W, H, b, tile=S, color_type=ct, device=dev)
    ring = oracle.Ring(W, H, b)
    for part in range(3):   # full, partly filled and empty queues, heads anywhere
        n = max(1, int(W * H * b * (0.7, 0.3, 0.4)[part]))
        t = rng.uniform(0, 1, n) if order != "ties" else rng.integers(0, 5, n) / 8.0
        if order == "sorted":
            t = (part + np.sort(t)) / 3
        pos = np.stack([rng.uniform(0, W, n), rng.uniform(0, H, n), t, np.ones(n)], 1).astype(np.float32)
        pos[:, 0] = np.minimum(pos[:, 0], np.nextafter(np.float32(W), np.float32(0)))
        pos[:, 1] = np.minimum(pos[:, 1], np.nextafter(np.float32(H), np.float32(0)))
        pos[pos[:, 0] < W * 0.1, 0] = W * 0.5     # empty columns
        col = torch.zeros((n, 4), dtype=rec.color_dtype)
        col[:, :3] = torch.from_numpy(rng.uniform(0, 1, (n, 3))).to(rec.color_dtype)
        mo = np.zeros((n, 2), np.float32)
        rec.insert(torch.from_numpy(pos).to(dev), col.to(dev), torch.from_numpy(mo).to(dev))
        ring.insert(pos, col.float().numpy(), mo)
    rec.estimate_gradients(T_NOW)
    want = oracle.gradients(ring, T_NOW)
    for m, ref in zip((L.AFR_MAP_LBAR, L.AFR_MAP_GX, L.AFR_MAP_GY, L.AFR_MAP_GT), want):
        got = rec.export_map(m).astype(np.float64)
        np.testing.assert_array_equal(np.isnan(got), np.isnan(ref))
        ok = ~np.isnan(ref)
        assert (np.abs(got[ok] - ref[ok]) <= 1e-5 * np.abs(ref[ok]) + 5e-7).all()
    tiles = oracle.tile_feedback(ring, want, S=S, t_now=T_NOW, m=2.0)
    got = decode_tiles(rec.tile_feedback())
    np.testing.assert_array_equal(got["n"], tiles[:, 0].astype(np.uint32))
    np.testing.assert_array_equal(got["empty_slots"], tiles[:, 1].astype(np.uint32))
    np.testing.assert_allclose(got["mean_L"], tiles[:, 2], rtol=1e-5, atol=1e-6)
    np.testing.assert_allclose(got["var_L"], tiles[:, 3], rtol=1e-4, atol=1e-6)
    for k, f in ((4, "mean_Gx"), (5, "mean_Gy"), (6, "mean_Gt")):
        np.testing.assert_allclose(got[f], tiles[:, k], rtol=1e-4, atol=2e-6)
    np.testing.assert_allclose(got["u"], tiles[:, 7], rtol=1e-6, atol=1e-6)
    E, gain = rec.tile_error(0.35, 0.4, 1.25)
    tiles[tiles[:, 0] <= 1, 3] = 0.0   # one sample has no variance; the oracle's sums leave a rounding error there
    E_ref, g_ref = oracle.tile_error(ring, tiles, S, T_NOW, None, 0.35, 0.4, 1.25)
    if tiles[:, 7].sum() > 1e-6 or not got["u"].any():   # else shares of a sum that is rounding alone
        np.testing.assert_allclose(E.cpu().numpy(), E_ref, rtol=1e-4, atol=1e-5 * max(np.abs(E_ref).max(), 1e-30))
    np.testing.assert_allclose([gain[k] for k in rec.GAIN_KEYS], g_ref, rtol=1e-4)
    rec.close()
