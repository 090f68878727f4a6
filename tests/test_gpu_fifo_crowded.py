"""The reconstructor's queue with crowded bins: bins at the edges of the length
that a thread places (64), that a warp sorts (512) and of the sorted range
(4096), around powers of two, queues that have wrapped and not, a camera, 16-bit
colours; the frame view bit for bit against the oracle, crowded and uncrowded
reprojections in turn. Bins above 4096 records hold the same records in any
order."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

T_NOW = 1.0


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_15876_gb300.build import build
    build()
    return torch.device("cuda:0")


def _batch(rng, W, H, lengths, spread):
    """Samples at rest: lengths[k] of them in bin 7 k (mod the image), `spread` anywhere, in random order."""
    bins = np.concatenate([np.full(m, 7 * k % (W * H)) for k, m in enumerate(lengths)] + [rng.integers(0, W * H, spread)])
    rng.shuffle(bins)
    n = len(bins)
    pos = np.stack([bins % W + 0.5, bins // W + 0.5, np.sort(rng.uniform(0, 1, n)), np.ones(n)], 1).astype(np.float32)
    col = np.zeros((n, 4), np.float32)
    col[:, :3] = rng.integers(0, 256, (n, 3)) / 256
    col[rng.random(n) < 0.02, 1] = np.inf     # rejected: gaps in the sequence numbers
    return {"pos": pos, "color": col, "motion": np.zeros((n, 2), np.float32)}


def _check(rec, fifo, sorted_up_to=4096):
    rec.reproject(T_NOW)
    off, frec, fseq = rec.export_frame()
    woff, wrec, wseq, _ = oracle.reproject_fifo(fifo, T_NOW)
    np.testing.assert_array_equal(off, woff)
    length = np.diff(off.astype(np.int64))
    for p in np.flatnonzero(length > sorted_up_to):
        a, b = off[p], off[p + 1]
        k = np.argsort(fseq[a:b], kind="stable")
        fseq[a:b], frec[a:b] = fseq[a:b][k], frec[a:b][k]
    np.testing.assert_array_equal(fseq, wseq)
    np.testing.assert_array_equal(frec[:, :2], wrec[:, :2])
    np.testing.assert_array_equal(frec[:, 3:6], wrec[:, 3:6])
    age = (np.float32(T_NOW) - wrec[:, 2]).astype(np.float32)
    np.testing.assert_array_equal(frec[:, 2], age * age)
    return length


@pytest.mark.parametrize("W,H,N,ct", [(64, 48, 40000, "f32"), (91, 37, 17003, "f16"), (1, 1, 3000, "f32"), (300, 200, 60001, "bf16")])
def test_crowded_bins_match_oracle(dev, W, H, N, ct):
    from paper_2510_15876_gb300.api import Reconstructor, to_device_batch
    rng = np.random.default_rng(N)
    rec, fifo = Reconstructor(W, H, 2, color_type=ct, fifo_capacity=N, device=dev), oracle.Fifo(W, H, N)
    lengths = [64, 65, 66, 63, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 1100, 130, 3, 4300]
    seen = set()
    for crowd, spread in ((lengths, 500), ([], W * H // 2), (lengths[::-1], 100), ([70] * 200, 0), ([4090, 5000], 2000)):
        batch = _batch(rng, W, H, crowd, spread) if crowd or spread else None
        if batch is None:
            continue
        rec.insert(*to_device_batch(batch, dev, rec.color_dtype))
        fifo.insert(batch["pos"], batch["color"], batch["motion"])
        seen |= set(_check(rec, fifo).tolist())
        rec.estimate_gradients(T_NOW)
        img = rec.reconstruct(T_NOW)
        assert torch.isfinite(img).all() and (img[..., 3] > 0).any()
    assert max(seen) > 64
    # emptied: the crowded flag of the last reprojection does not outlive it
    rec.reset()
    fifo = oracle.Fifo(W, H, N)
    batch = _batch(rng, W, H, [], 60)
    rec.insert(*to_device_batch(batch, dev, rec.color_dtype))
    fifo.insert(batch["pos"], batch["color"], batch["motion"])
    _check(rec, fifo)
    rec.close()


def test_crowded_bins_seen_by_a_camera(dev):
    """A camera that looks down on a line: every sample of a column in one bin. The same records as the queues' form."""
    from paper_2510_15876_gb300.api import Reconstructor
    W, H, n = 40, 30, 30000
    g = torch.Generator(dev).manual_seed(0)
    pos = torch.rand(n, 4, generator=g, device=dev) * torch.tensor([W - 0.01, H - 0.01, 1.0, 1.0], device=dev)
    col, mo = torch.rand(n, 4, generator=g, device=dev), torch.zeros(n, 2, device=dev)
    world = torch.rand(n, 4, generator=g, device=dev) * 2 - 1
    vp = np.array([[0.9, 0, 0, 0], [0, 0, 0, 0.05], [0, 0, 1, 0], [0, 0, 0, 1]], np.float32)
    queue, deep = (Reconstructor(W, H, 32, fifo_capacity=f, world_points=True, device=dev) for f in (n, 0))
    for rec in (queue, deep):
        rec.insert(pos, col, mo, world)
        rec.reproject_camera(T_NOW, vp)
    (o1, r1, s1), (o2, r2, s2) = queue.export_frame(), deep.export_frame()
    length = np.diff(o1.astype(np.int64))
    assert length.max() > 500
    keep = np.isin(s1, s2)        # the queues hold the newest 32 of each pixel, the reconstructor's queue all
    np.testing.assert_array_equal(s1[keep], s2)
    np.testing.assert_array_equal(r1[keep], r2)
    for p in range(W * H):
        assert (np.diff(s1[o1[p]:o1[p + 1]].astype(np.int64)) > 0).all()
    queue.close()
    deep.close()
