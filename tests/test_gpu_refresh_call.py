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


@pytest.mark.parametrize("camera", [False, True])
def test_captured_refresh_records_an_external_event_at_every_replay(dev, camera):
    """reads_done made with external=True is recorded by a node of the graph, as
    by torch's own record between the calls: after a replay it has a time, between
    that of an event before the refresh and that of one after it. One without the
    flag orders streams inside the capture."""
    a, s = _filled(dev), _filled(dev)
    out, tiles = torch.empty((H, W, 4), device=dev), torch.empty((a.n_tiles, 8), device=dev)
    kw = dict(out=out, tiles=tiles, view_proj=VP if camera else None)
    a._side = torch.cuda.Stream(dev)
    before, done, after = (torch.cuda.Event(enable_timing=True, external=True) for _ in range(3))
    inside, other = torch.cuda.Event(), torch.cuda.Stream(dev)
    flag = torch.zeros(1, device=dev)
    done.record()   # as a pipeline does before its first image: the event exists
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        main = torch.cuda.current_stream(dev)
        before.record(main)
        a.refresh(1.0, reads_done=done, **kw)
        after.record(main)
        a.refresh(1.0, reads_done=inside, **kw)
        other.wait_event(inside)
        with torch.cuda.stream(other):
            flag.add_(1)
        main.wait_stream(other)
    for k in range(2):
        graph.replay()
        torch.cuda.synchronize()
        assert done.query() and 0 < before.elapsed_time(done) <= before.elapsed_time(after)
        assert flag.item() == k + 1
    want, want_tiles = s.refresh(1.0, view_proj=VP if camera else None)
    torch.cuda.synchronize()
    assert torch.equal(out, want) and torch.equal(tiles.view(torch.int32), want_tiles.view(torch.int32))


def test_a_refused_refresh_launches_nothing(dev):
    """After a refusal both streams are idle, so nothing still reads the queues
    or writes the tile records when the caller's next batch arrives, and a
    capture that a refusal happened in goes on."""
    import ctypes
    from paper_2510_15876_gb300.api import Reconstructor
    w, h, depth, n = 1024, 768, 8, 1 << 21
    batches = []
    for seed in range(2):
        g = torch.Generator(dev).manual_seed(seed)
        pos = torch.rand(n, 4, generator=g, device=dev) * torch.tensor([w - 0.5, h - 0.5, 1.0, 1.0], device=dev)
        batches.append((pos, torch.rand(n, 4, generator=g, device=dev), torch.randn(n, 2, generator=g, device=dev)))
    rec, fresh = Reconstructor(w, h, depth, device=dev), Reconstructor(w, h, depth, device=dev)
    rec.reserve(n)
    rec._side = torch.cuda.Stream(dev, priority=-1)
    main = torch.cuda.current_stream(dev)
    out, tiles = torch.empty((h, w, 4), device=dev), torch.empty((rec.n_tiles, 8), device=dev)
    default = L.AfrParams(1.0, 0.0, 3.0, 1.0, 0.0, 1.0)

    def native(params=default, flags=0, image=out, stats=tiles):
        st = rec.lib.afr_refresh(rec.h, 1.0, None, ctypes.byref(params), flags, image.data_ptr() if image is not None else None,
                                 stats.data_ptr() if stats is not None else None, rec._side.cuda_stream, None, main.cuda_stream)
        if st != L.AFR_OK:
            raise L.AfrError(st, "refused")

    calls = [lambda: rec.refresh(float("nan")), lambda: rec.refresh(1.0, params=(1, 0, -3, 1, 0, 1)),
             lambda: rec.refresh(1.0, flags=64), lambda: rec.refresh(1.0, view_proj=np.full((4, 4), np.inf)),
             lambda: rec.refresh(1.0, view_proj=VP), lambda: native(image=None), lambda: native(stats=None),
             lambda: native(image=out.view(-1)[1:])]
    fresh.insert(*batches[1])
    want, want_tiles = fresh.refresh(1.0)
    for call in calls:
        rec.insert(*batches[0], reset=True)
        torch.cuda.synchronize()
        with pytest.raises(L.AfrError):
            call()
        assert rec._side.query() and main.query()
        rec.insert(*batches[1], reset=True)
        rec.refresh(1.0, out=out, tiles=tiles)
        torch.cuda.synchronize()
        assert torch.equal(out, want) and torch.equal(tiles.view(torch.int32), want_tiles.view(torch.int32))
    graph = torch.cuda.CUDAGraph()
    out.zero_(), tiles.zero_()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        for kw in (dict(view_proj=VP), dict(flags=64)):
            with pytest.raises(L.AfrError):
                rec.refresh(1.0, out=out, tiles=tiles, **kw)
        rec.refresh(1.0, out=out, tiles=tiles)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want) and torch.equal(tiles.view(torch.int32), want_tiles.view(torch.int32))


@pytest.mark.parametrize("w,h,depth,color,fifo", [
    (1, 1, 2, "f32", 0), (61, 43, 5, "bf16", 0), (640, 360, 8, "f16", 0), (300, 200, 4, "f32", 3 * 300 * 200)])
def test_overlapped_launches_keep_their_order(dev, w, h, depth, color, fifo):
    """A step's kernels are launched before the ones they read from have ended
    (waiting inside), at one block and at many waves: steps issued without a
    pause, and replayed from a graph, equal steps with a synchronisation after
    every call, bit for bit, whole state included."""
    from paper_2510_15876_gb300.api import Reconstructor
    dtype = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[color]
    n = 2 * w * h * depth
    batches = []
    for seed in range(3):
        g = torch.Generator().manual_seed(seed)
        pos = torch.rand(n, 4, generator=g) * torch.tensor([w, h, 1.0, 1.0])
        pos[:, 2] = pos[:, 2].sort().values
        pos[::13, 0] = float("nan")
        batches.append((pos.to(dev), torch.rand(n, 4, generator=g).to(dev, dtype), torch.randn(n, 2, generator=g).to(dev)))

    def context():
        rec = Reconstructor(w, h, depth, color_type=color, fifo_capacity=fifo, device=dev)
        rec.reserve(n)
        return rec

    plain, graphed, slow = context(), context(), context()
    outs = []
    for rec in (plain, graphed):
        out, tiles = torch.empty((h, w, 4), device=dev), torch.empty((rec.n_tiles, 8), device=dev)
        outs.append((out, tiles))
    static = [t.clone() for t in batches[0]]
    graphed._side = torch.cuda.Stream(dev)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        graphed.insert(*static, reset=True)
        graphed.refresh(1.0, out=outs[1][0], tiles=outs[1][1])
    for batch in batches:
        plain.insert(*batch, reset=True)
        plain.refresh(1.0, out=outs[0][0], tiles=outs[0][1])
        for s, t in zip(static, batch):
            s.copy_(t)
        graph.replay()
        slow.reset()
        for call in (lambda: slow.insert(*batch), lambda: slow.estimate_gradients(1.0), lambda: slow.reproject(1.0)):
            call()
            torch.cuda.synchronize()
        want, want_tiles = slow.reconstruct(1.0), slow.tile_feedback()
        torch.cuda.synchronize()
        for out, tiles in outs:
            assert torch.equal(out, want) and torch.equal(tiles.view(torch.int32), want_tiles.view(torch.int32))
        for a, b in zip(plain.export_ring(), slow.export_ring()):
            assert np.array_equal(a, b)


def test_batch_of_large_and_small_contexts(dev):
    """Contexts above and below the size that takes its turn on one worker
    stream: every image equals the calls in series, bit for bit."""
    from paper_2510_15876_gb300.api import BatchReconstructor, Reconstructor
    recs = []
    for seed, (w, h, depth) in enumerate(((1280, 720, 16), (64, 48, 4), (1100, 800, 16), (320, 200, 8))):
        g = torch.Generator(dev).manual_seed(seed)
        n = w * h * depth
        pos = torch.rand(n, 4, generator=g, device=dev) * torch.tensor([w - 0.5, h - 0.5, 1.0, 1.0], device=dev)
        rec = Reconstructor(w, h, depth, color_type="f16", device=dev)
        rec.insert(pos, torch.rand(n, 4, generator=g, device=dev).half(), torch.randn(n, 2, generator=g, device=dev))
        recs.append(rec)
    got = [img.clone() for img in BatchReconstructor(recs).refresh(1.0)]
    for rec, img in zip(recs, got):
        rec.estimate_gradients(1.0)
        rec.reproject(1.0)
        want = rec.reconstruct(1.0)
        torch.cuda.synchronize()
        assert torch.equal(img, want)
