"""Samples too old for their weights in single precision (exp(-3.47 a) is below
the least normal number from a = 25 and 0 from a = 30): the gain control's mean
age counts the ages of all buffered samples, those of pixels left without a
weight included, over the samples of the tile records; a tile's mean luminance
is good to single precision while any of its weights is left."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_15876_gb300.build import build
    build()
    return torch.device("cuda:0")


def _rec(dev, W, H, S, x, y, t, rgb):
    from paper_2510_15876_gb300.api import Reconstructor
    n = len(x)
    rec = Reconstructor(W, H, 2, tile=S, device=dev)
    pos = np.stack([x + 0.5, y + 0.5, t, np.ones(n)], 1).astype(np.float32)
    col = np.zeros((n, 4), np.float32)
    col[:, :3] = rgb[:, None]
    rec.insert(*(torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(dev) for a in (pos, col, np.zeros((n, 2)))))
    return rec


@pytest.mark.parametrize("S", [4, 8, 16, 32, 40])
def test_mean_age_counts_every_buffered_sample(dev, S):
    W, H, t_now = 4 * S, 3 * S, 64.0
    y, x = (v.reshape(-1) for v in np.mgrid[0:H, 0:W])
    old = (x + y) % 3 == 0
    t = np.where(old, 0.0, 63.0)
    rec = _rec(dev, W, H, S, x, y, t, np.full(W * H, 0.5))
    from paper_2510_15876_gb300.api import decode_tiles
    rec.estimate_gradients(t_now)
    n = decode_tiles(rec.tile_feedback())["n"].reshape(3, 4)
    tiles = old.reshape(3, S, 4, S).transpose(0, 2, 1, 3).reshape(3, 4, S * S)
    np.testing.assert_array_equal(n, S * S - tiles.sum(2))
    _, gain = rec.tile_error()
    want = ((64.0 * tiles.sum(2) + 1.0 * n) / n).mean()
    np.testing.assert_allclose(gain["mean_age"], want, rtol=1e-5)
    rec.close()


@pytest.mark.parametrize("S,age", [(2, 29.0), (2, 27.0), (8, 29.0), (32, 28.0), (34, 29.0), (2, 1.0)])
def test_tile_mean_of_samples_with_tiny_weights(dev, S, age):
    """One sample a pixel and all of one age: the weights are equal, so the mean
    is the plain mean. Bound: the FP32 luminances and the result, 2^-24 each, and
    the reference's own rounding of the colours, within 4 of those."""
    from paper_2510_15876_gb300.api import decode_tiles
    W, H = 6 * S, 5 * S
    y, x = (v.reshape(-1) for v in np.mgrid[0:H, 0:W])
    L = np.random.default_rng(S).uniform(0.1, 1.0, W * H).astype(np.float32)
    rec = _rec(dev, W, H, S, x, y, np.zeros(W * H), L)
    rec.estimate_gradients(age)
    got = decode_tiles(rec.tile_feedback())
    assert (got["n"] == S * S).all()
    want = L.astype(np.float64).reshape(5, S, 6, S).mean((1, 3)).reshape(-1)
    np.testing.assert_allclose(got["mean_L"], want, rtol=4 * 2.0 ** -24)
    rec.close()
