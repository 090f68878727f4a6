"""refresh() as one native call: every option it passes on (parameters, flags,
a camera, the caller's streams and event) against the calls it stands for, bit
for bit, plainly and replayed from a graph; what those calls refuse, it refuses."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2510_15876_gb300 import _lib as L  # noqa: E402

W, H, b = 61, 43, 5
VP = np.array([[1.1, 0.1, 0, 0], [0, 0.9, 0.1, 0], [0, 0, 1, 0], [0, 0, 0.2, 2]], np.float32)


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_15876_gb300.build import build
    build()
    return torch.device("cuda:0")


def _filled(dev):
    from paper_2510_15876_gb300.api import Reconstructor
    rng = np.random.default_rng(5)
    n = 4 * W * H
    pos = np.stack([rng.uniform(0, W - 1, n), rng.uniform(0, H - 1, n), np.sort(rng.uniform(0, 1, n)), np.ones(n)], 1)
    arrays = (pos, rng.uniform(0, 1, (n, 4)), rng.uniform(-2, 2, (n, 2)), rng.uniform(-1, 1, (n, 4)))
    rec = Reconstructor(W, H, b, world_points=True, device=dev)
    rec.insert(*(torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(dev) for a in arrays))
    return rec


@pytest.mark.parametrize("theta,flags,camera,streams", [
    (None, 0, False, "default"), ((0.8, 0.1, 2.5, 1.2, 0.02, 0.9), 0, True, "own"),
    (None, L.AFR_RECON_ADAPTIVE_SUPPORT, False, "captured"), ((1.1, 0.0, 3.0, 0.9, 0.01, 0.7), 0, True, "captured")])
def test_refresh_equals_its_calls(dev, theta, flags, camera, streams):
    a, s = _filled(dev), _filled(dev)
    out, tiles = torch.empty((H, W, 4), device=dev), torch.empty((a.n_tiles, 8), device=dev)
    kw = dict(out=out, tiles=tiles, params=theta, flags=flags, view_proj=VP if camera else None)
    if streams == "default":
        done = torch.cuda.Event()   # never recorded before
        a.refresh(1.0, reads_done=done, **kw)
        torch.cuda.synchronize()
        assert done.query()
    elif streams == "own":
        main, side = torch.cuda.Stream(dev), torch.cuda.Stream(dev)
        main.wait_stream(torch.cuda.current_stream())
        a.refresh(1.0, stream=main, side_stream=side, **kw)
    else:
        a._side = torch.cuda.Stream(dev)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            a.refresh(1.0, **kw)
        graph.replay()
    torch.cuda.synchronize()
    s.estimate_gradients(1.0)
    want_tiles = s.tile_feedback()
    s.reproject_camera(1.0, VP) if camera else s.reproject(1.0)
    want = s.reconstruct(1.0, theta, flags=flags)
    torch.cuda.synchronize()
    assert torch.equal(out, want) and torch.equal(tiles.view(torch.int32), want_tiles.view(torch.int32))


def test_refresh_refuses_what_its_calls_refuse(dev):
    from paper_2510_15876_gb300.api import Reconstructor
    a = _filled(dev)
    for kw in (dict(t_now=float("nan")), dict(params=(1, 0, -3, 1, 0, 1)), dict(flags=64),
               dict(view_proj=np.full((4, 4), np.inf))):
        with pytest.raises(L.AfrError) as err:
            a.refresh(**kw)
        assert err.value.status == L.AFR_ERR_INVALID_ARG
    with pytest.raises(L.AfrError) as err:
        Reconstructor(W, H, b, device=dev).refresh(1.0, view_proj=VP)   # stores no hit points
    assert err.value.status == L.AFR_ERR_BAD_STATE
    img, _ = a.refresh(1.0)
    assert torch.isfinite(img).all()
