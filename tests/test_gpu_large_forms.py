"""The forms that only larger images take, at their edges: the adjoint's three
rows a thread (ragged last bands, borders, empty rows), the filter's whole tiles
at every tile shape (images that end inside a tile and a 2x2 block), and scans of
more than 2048 blocks (8.4M counts), whose block sums are scanned by a launch of
their own. Bounds as in the tests of the small forms."""
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


def _batch(seed, W, H, n, gap):
    """n samples at rest or moving a little, none in a band of rows near the bottom."""
    rng = np.random.default_rng(seed)
    x, y = rng.uniform(0, W, n), rng.uniform(0, H, n)
    y = np.where((y > H - 40) & (y < H - 40 + gap), 0.25, y)
    x, y = (np.minimum(v.astype(np.float32), np.nextafter(np.float32(m), np.float32(0))) for v, m in ((x, W), (y, H)))
    pos = np.stack([x, y, np.sort(rng.uniform(0, 1, n)).astype(np.float32), np.ones(n, np.float32)], 1)
    col = np.zeros((n, 4), np.float32)
    col[:, :3] = rng.uniform(0, 1, (n, 3))
    return {"pos": np.ascontiguousarray(pos), "color": col, "motion": rng.uniform(-2, 2, (n, 2)).astype(np.float32)}


@pytest.mark.parametrize("W,H,R,ct", [(515, 517, 3, "f32"), (515, 518, 5, "f16"), (513, 519, 8, "f32"), (515, 528, 2, "f32")])
def test_adjoint_of_large_images_matches_oracle(dev, W, H, R, ct):
    from paper_2510_15876_gb300.api import Reconstructor, to_device_batch
    b = 2
    batch = _batch(W + R, W, H, W * H * b, 20)
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
    off, frec, _, _ = oracle.reproject(ring, T_NOW)
    rng = np.random.default_rng(W)
    everywhere = rng.normal(size=(H, W, 4)).astype(np.float32)
    border = everywhere.copy()
    border[R:H - 12, R:W - R] = 0    # the bottom bands and the borders alone
    for g in (everywhere, border):
        gcol, gprm = rec.backward(torch.from_numpy(g).to(dev))
        only_colors, _ = rec.backward(torch.from_numpy(g).to(dev), want_params=False)
        wcol, wprm = oracle.backward(ring.count, W, H, (None, *(v.astype(np.float64) for v in maps)), off, frec,
                                     g.reshape(-1, 4)[:, :3].astype(np.float64), theta, R=R)
        np.testing.assert_allclose(gprm.cpu().numpy(), wprm, rtol=2e-4, atol=1e-4 * np.abs(wprm).max())
        for got in (gcol, only_colors):
            np.testing.assert_allclose(got.cpu().numpy(), wcol, rtol=1e-3, atol=1e-5 * np.abs(wcol).max())
    rec.close()


@pytest.mark.parametrize("W,H,b,R,tbx,ct", [(401, 403, 2, 8, 2, "f32"), (401, 403, 2, 4, 4, "f16"), (403, 405, 3, 5, 8, "f32"),
                                            (417, 399, 2, 8, 16, "bf16"), (399, 401, 1, 1, 4, "f32")])
def test_filter_of_whole_tiles_matches_oracle(dev, W, H, b, R, tbx, ct):
    from paper_2510_15876_gb300.api import Reconstructor, set_tuning, to_device_batch
    batch = _batch(W * R, W, H, W * H * b, 24)
    rec = Reconstructor(W, H, b, radius=R, color_type=ct, device=dev)
    set_tuning(rec, R, tbx)
    tensors = to_device_batch(batch, dev, rec.color_dtype)
    rec.insert(*tensors)
    ring = oracle.Ring(W, H, b)
    ring.insert(batch["pos"], tensors[1].float().cpu().numpy(), batch["motion"])
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
    assert err.max() <= 1e-5


def test_scan_of_more_than_2048_blocks(dev):
    """4099 x 2053 pixels, depth 1: samples at pixel centres with whole-number
    motion over one time unit, so every position is exact; offsets, sequence
    numbers and positions bit for bit, over two batches."""
    from paper_2510_15876_gb300.api import Reconstructor
    W, H = 4099, 2053
    P = W * H
    assert (P + 4095) // 4096 > 2048
    rng = np.random.default_rng(0)
    rec = Reconstructor(W, H, 1, device=dev)
    pixel, move, seq, base = np.full(P, -1), np.zeros((P, 2)), np.zeros(P, np.int64), 0
    for n in (1 << 21, 1 << 20):
        p = rng.integers(0, P, n)
        p[: n // 8] = P - 1 - rng.integers(0, 5000, n // 8)    # the last blocks hold many
        mo = rng.integers(-3, 4, (n, 2)).astype(np.float32)
        pos = np.stack([p % W + 0.5, p // W + 0.5, np.zeros(n), np.ones(n)], 1).astype(np.float32)
        rec.insert(*(torch.from_numpy(a).to(dev) for a in (pos, np.zeros((n, 4), np.float32), mo)))
        newest = np.zeros(P, np.int64)
        np.maximum.at(newest, p, np.arange(1, n + 1))         # the newest sample of each pixel stays
        hit = np.flatnonzero(newest)
        pixel[hit], move[hit], seq[hit] = hit, mo[newest[hit] - 1], base + newest[hit] - 1
        base += n
        rec.reproject(T_NOW)
        off, frec, fseq = rec.export_frame()
        q = np.flatnonzero(pixel >= 0)
        x, y = q % W + move[q, 0], q // W + move[q, 1]
        ok = (x >= 0) & (x < W) & (y >= 0) & (y < H)
        to, sq = (y * W + x).astype(np.int64)[ok], seq[q][ok]
        np.testing.assert_array_equal(off, np.concatenate([[0], np.cumsum(np.bincount(to, minlength=P))]))
        order = np.lexsort((sq, to))
        np.testing.assert_array_equal(fseq, sq[order])
        np.testing.assert_array_equal(frec[:, 0], (to % W + 0.5)[order])
        np.testing.assert_array_equal(frec[:, 1], (to // W + 0.5)[order])
        assert rec.query()["dropped"] == (~ok).sum()
    rec.close()
