"""The scans of ingest and reprojection at the ends of their blocks (one pixel,
a block less and more one, a partial 256-bit access), counts and cursors that
must be clean for the next call, batches after a reset beside queues that get
none, and an output array that is only 4-byte aligned; queues and frame views
bit for bit against the oracle."""
import ctypes

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


def _batch(rng, W, H, n, cols):
    x = rng.uniform(0, max(1, W * cols), n).astype(np.float32)
    pos = np.stack([np.minimum(x, np.nextafter(np.float32(W), np.float32(0))),
                    np.minimum(rng.uniform(0, H, n).astype(np.float32), np.nextafter(np.float32(H), np.float32(0))),
                    np.sort(rng.uniform(0, 1, n)), np.ones(n)], 1).astype(np.float32)
    col = np.zeros((n, 4), np.float32)
    col[:, :3] = rng.uniform(0, 1, (n, 3))
    col[rng.random(n) < 0.02, 0] = np.nan     # rejected after the position was counted
    return {"pos": pos, "color": col, "motion": rng.uniform(-9, 9, (n, 2)).astype(np.float32)}


@pytest.mark.parametrize("W,H", [(1, 1), (7, 1), (64, 64), (4097, 1), (4095, 1), (129, 64), (91, 91)])
def test_steps_leave_the_next_one_clean(dev, W, H):
    from paper_2510_15876_gb300.api import Reconstructor, to_device_batch
    rng = np.random.default_rng(W + H)
    b = 3
    rec, ring = Reconstructor(W, H, b, device=dev), oracle.Ring(W, H, b)
    for reset, share, cols in ((False, 2.0, 1.0), (False, 0.5, 0.4), (True, 1.5, 0.5), (False, 0.01, 1.0)):
        batch = _batch(rng, W, H, max(1, int(W * H * share)), cols)
        if W * H < 9:
            batch = {k: np.repeat(v, 300, 0) for k, v in batch.items()}   # past the commit's largest pixel
        if reset:
            ring = oracle.Ring(W, H, b)
        rec.insert(*to_device_batch(batch, dev), reset=reset)
        ring.insert(batch["pos"], batch["color"], batch["motion"])
        count, slot, seq = rec.export_ring()
        np.testing.assert_array_equal(count, ring.count)
        np.testing.assert_array_equal(seq, ring.seq)
        np.testing.assert_array_equal(slot, ring.slot)
        for t_now in (1.0, 1.25):
            rec.reproject(t_now)
            off, frec, fseq = rec.export_frame()
            woff, wrec, wseq, dropped = oracle.reproject(ring, t_now)
            np.testing.assert_array_equal(off, woff)
            np.testing.assert_array_equal(fseq, wseq)
            np.testing.assert_array_equal(frec[:, :2], wrec[:, :2])
            assert rec.query()["dropped"] == dropped
    rec.close()


def test_static_binning_with_a_4_byte_aligned_offset_array(dev):
    lib = L.load()
    W, H, n = 91, 91, 20000
    rng = np.random.default_rng(5)
    batch = _batch(rng, W, H, n, 1.0)
    pos, col, mo = (torch.from_numpy(np.ascontiguousarray(batch[k])).to(dev) for k in ("pos", "color", "motion"))
    got = []
    for shift in (0, 1, 3):
        off = torch.zeros(W * H + 9, dtype=torch.int32, device=dev)
        rec, out = torch.zeros((n, 4), device=dev), torch.zeros((n, 4), device=dev)
        seq = torch.zeros(n, dtype=torch.int32, device=dev)
        b = L.AfrSampleBatch(pos.data_ptr(), col.data_ptr(), mo.data_ptr())
        st = lib.afr_reproject_batch_static(ctypes.byref(b), n, W, H, 0, T_NOW, off.data_ptr() + 4 * shift, rec.data_ptr(),
                                            out.data_ptr(), seq.data_ptr(), None,
                                            torch.cuda.current_stream().cuda_stream)
        assert st == L.AFR_OK
        torch.cuda.synchronize()
        assert not off[:shift].any() and not off[shift + W * H + 1:].any()
        got.append((off[shift:shift + W * H + 1].cpu(), rec.cpu(), seq.cpu()))
    for g in got[1:]:
        for a, c in zip(got[0], g):
            assert torch.equal(a, c)
