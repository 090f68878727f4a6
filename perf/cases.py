"""What a user of the reconstruction library has it do, as measurable cases.

Every case goes through the public Python entry points (Reconstructor,
BatchReconstructor, autograd.reconstruct), which pass straight to the C ABI.
The kinds of pass ("do"):

  step       a display loop that replaces its samples: insert a whole batch
             (reset), then refresh: gradients, tile statistics, reprojection,
             filter.
  increment  the frameless loop of the paper: the queues are full, a pass
             inserts the samples traced since the last image and refreshes.
             With "fifo" the frame comes from the queue of the newest samples,
             with "world" it is rendered from stored hit points by a camera.
  redisplay  the same samples shown at another time: reproject, reconstruct
             (with "adaptive", per-pixel footprints from the coverage map).
  sampler    what the adaptive sampler asks between images: gradients, tile
             statistics, tile errors and gain control.
  filter     the image again with other width parameters: reconstruct alone.
  fit        one optimisation step of the width mapping and the sample
             colours: forward, and the adjoint to both.
  streams    many viewers' images in one call: BatchReconstructor.refresh.

Inputs are drawn on the GPU from the seed: opaque discs moving over a
checkerboard, sample positions uniform or clustered in 32x32 tiles, times
sorted ascending, exact colours and screen motions at the samples.
"""
import math

import torch

T_NOW = 1.0
TILE, WINDOW, EPS, UNDER_M = 32, 1.0, 1e-4, 2.0
THETA = (1.0, 0.0, 3.0, 1.0, 0.0, 1.0)
DEVICE = "cuda:0"
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


def _case(do, width, height, depth, color="f32", radius=4, rate=1.0, clustered=False, fifo=0, world=False,
          adaptive=False, t_now=T_NOW, mix=""):
    """rate: samples a pass inserts, per queue slot of the image. fifo: capacity in samples per pixel.
    mix: the viewers of a "streams" case, width x height x depth of each."""
    return dict(do=do, width=width, height=height, depth=depth, color=color, radius=radius, rate=rate,
                clustered=clustered, fifo=fifo, world=world, adaptive=adaptive, t_now=t_now, mix=mix)


def listed():
    out = []

    def add(name, *a, **k):
        out.append(dict(_case(*a, **k), name=name))

    # a thumbnail or a test loop: every call is shorter than its launch
    add("step_128x128x4", "step", 128, 128, 4)
    # interactive frameless rendering: a sixteenth of the buffer is new each image
    add("increment_640x480x8_f16", "increment", 640, 480, 8, "f16", rate=1 / 16)
    # adaptive sampling: samples crowd into the tiles that need them
    add("step_1024x1024x8_clustered", "step", 1024, 1024, 8, clustered=True)
    # the library's headline: a full-HD image from a 16-deep buffer
    add("step_1920x1080x16", "step", 1920, 1080, 16)
    # the same loop in half precision at 720p
    add("step_1280x720x16_f16", "step", 1280, 720, 16, "f16")
    # an odd window size and queue depth, bfloat16 colours, a later display time
    add("redisplay_1366x767x5_bf16", "redisplay", 1366, 767, 5, "bf16", radius=3, t_now=1.0625)
    # the sampler's questions about a full-HD buffer
    add("sampler_1920x1080x16", "sampler", 1920, 1080, 16)
    # a wider footprint, widths recomputed for new parameters
    add("filter_1280x720x8_r5", "filter", 1280, 720, 8, radius=5)
    # footprints from the coverage map, settled after a few images
    add("adaptive_1920x1080x16", "redisplay", 1920, 1080, 16, adaptive=True)
    # fitting the filter to ground truth, 512x512
    add("fit_512x512x8", "fit", 512, 512, 8)
    # a server with six viewers of different sizes
    add("streams_mixed_f16", "streams", 0, 0, 0, "f16", radius=3, 
        mix="256x256x4 256x256x16 640x480x8 640x480x16 1280x720x4 1280x720x8")
    # the paper's own reconstructor: newest samples of the whole image, rendered by the current camera
    add("camera_fifo_1024x1024x8", "increment", 1024, 1024, 8, rate=1 / 32, fifo=4, world=True)
    return out


def _disc(r):
    """Bin offsets (dx, dy) of the integer disc of radius r."""
    return [(dx, dy) for dy in range(-r, r + 1) for dx in range(-r, r + 1) if dx * dx + dy * dy <= r * r]


def _cost(c):
    """Rough microseconds of a pass: samples moved, pairs filtered, bytes of the buffer walked."""
    slots = c["width"] * c["height"] * c["depth"]
    pairs = slots * len(_disc(c["radius"]))
    moved = slots * c["rate"] if c["do"] in ("step", "increment") else 0
    return moved * 6e-5 + slots * 5e-5 + pairs * (5e-6 if c["do"] == "fit" else 1.1e-6)


def draw(rng):
    do = rng.choice(("step", "step", "increment", "increment", "redisplay", "sampler", "filter", "fit", "streams"))
    color = rng.choice(("f32", "f32", "f16", "bf16"))
    if do == "streams":
        sizes = ("256x256", "320x200", "640x480", "1000x563", "1280x720")
        mix = " ".join("%sx%d" % (rng.choice(sizes), rng.choice((4, 8, 16))) for _ in range(rng.randrange(2, 9)))
        return _case(do, 0, 0, 0, color, radius=rng.choice((3, 4, 5)), mix=mix)
    most = _cost(_case("step", 1920, 1080, 16))
    while True:
        pixels = math.exp(rng.uniform(math.log(128 * 128), math.log(1920 * 1080 if do != "fit" else 640 * 640)))
        aspect = math.exp(rng.uniform(math.log(0.75), math.log(2.4)))
        w, h = int(round(math.sqrt(pixels * aspect))), int(round(math.sqrt(pixels / aspect)))
        if rng.random() < 0.5:
            w, h = (w + 7) // 8 * 8, (h + 7) // 8 * 8
        c = _case(do, w, h, rng.choice((2, 3, 4, 5, 8, 8, 12, 16, 24)), color, radius=rng.choice((2, 3, 4, 4, 5)),
                  clustered=rng.random() < 0.25)
        if do == "increment":
            c["rate"] = math.exp(rng.uniform(math.log(1 / 64), math.log(1 / 2)))
            if rng.random() < 0.3:
                c["fifo"] = rng.choice((2, 4, 8))
            if rng.random() < 0.3:
                c["world"] = True
        if do == "redisplay":
            c["t_now"] = 1.0 + rng.randrange(0, 9) / 64
            c["adaptive"] = rng.random() < 0.4
        if _cost(c) <= most:
            return c


# ---- inputs -------------------------------------------------------------------------

_CELL, _PER_CELL, _CHECK = 128.0, 2, 16.0


class _Scene:
    """Two discs for each 128-pixel cell, each moving by less than a cell."""

    def __init__(self, c, seed, dev):
        g = torch.Generator(device=dev)
        g.manual_seed(seed)
        self.g, self.dev, self.W, self.H = g, dev, c["width"], c["height"]
        self.nx, self.ny = max(1, math.ceil(self.W / _CELL)), max(1, math.ceil(self.H / _CELL))
        k = self.nx * self.ny * _PER_CELL
        cell = torch.arange(k, device=dev) // _PER_CELL
        u = torch.rand((k, 8), generator=g, device=dev)
        small = min(1.0, min(self.W, self.H) / 256.0)
        self.cx, self.cy = ((cell % self.nx) + u[:, 0]) * _CELL, ((cell // self.nx) + u[:, 1]) * _CELL
        self.vx, self.vy = (u[:, 2] * 128 - 64) * small, (u[:, 3] * 128 - 64) * small
        self.r, self.rgb, self.z = (12 + 32 * u[:, 4]) * small, u[:, 5:8], torch.rand(k, generator=g, device=dev)
        self.clustered = c["clustered"]
        if self.clustered:
            self.ntx, self.nty = -(-self.W // TILE), -(-self.H // TILE)
            p = torch.rand(self.ntx * self.nty, generator=g, device=dev).double() ** 4
            self.tiles = torch.cumsum(0.95 * p / p.sum() + 0.05 / p.numel(), 0)

    def rand(self, n):
        return torch.rand(n, generator=self.g, device=self.dev)

    def samples(self, n, t0, t1):
        """(x, y, t, depth), (r, g, b, 0), (m_x, m_y) of n samples with times in [t0, t1) ascending."""
        W, H = self.W, self.H
        x, y = self.rand(n), self.rand(n)
        if self.clustered:
            t = torch.rand(n, generator=self.g, device=self.dev, dtype=torch.float64)
            i = torch.searchsorted(self.tiles, t * self.tiles[-1]).clamp_(max=self.ntx * self.nty - 1)
            tx, ty = (i % self.ntx) * TILE, (i // self.ntx) * TILE
            x, y = tx + x * (W - tx).clamp(max=TILE), ty + y * (H - ty).clamp(max=TILE)
        else:
            x, y = x * W, y * H
        x.clamp_(max=math.nextafter(W, 0) if W < 2 else W - W * 2.0 ** -23)
        y.clamp_(max=math.nextafter(H, 0) if H < 2 else H - H * 2.0 ** -23)
        t = torch.sort(t0 + (t1 - t0) * self.rand(n)).values
        pan = 8.0 if self.clustered else 0.0
        white = ((torch.floor((x - pan * t) / _CHECK) + torch.floor(y / _CHECK)).long() & 1) == 0
        col = torch.zeros((n, 4), device=self.dev)
        col[:, :3] = white.float()[:, None]
        mo = torch.zeros((n, 2), device=self.dev)
        mo[:, 0] = pan
        best = torch.full((n,), float("inf"), device=self.dev)
        gx, gy = (x / _CELL).long().clamp_(0, self.nx - 1), (y / _CELL).long().clamp_(0, self.ny - 1)
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                qx, qy = gx + dx, gy + dy
                inside = (qx >= 0) & (qx < self.nx) & (qy >= 0) & (qy < self.ny)
                for k in range(_PER_CELL):
                    i = torch.where(inside, (qy * self.nx + qx) * _PER_CELL + k, 0)
                    d2 = (x - self.cx[i] - self.vx[i] * t) ** 2 + (y - self.cy[i] - self.vy[i] * t) ** 2
                    hit = torch.nonzero(inside & (d2 <= self.r[i] ** 2) & (self.z[i] < best)).squeeze(1)
                    j = i[hit]
                    best[hit] = self.z[j]
                    rgb = self.rgb[j]
                    if self.clustered:   # a highlight on each disc
                        rgb = rgb + torch.exp(-d2[hit] / (0.1 * self.r[j]) ** 2)[:, None]
                    col[hit, :3] = rgb
                    mo[hit, 0], mo[hit, 1] = self.vx[j], self.vy[j]
        pos = torch.stack([x, y, t, best], 1).contiguous()
        return pos, col, mo


def _camera(t):
    """Row-major view-projection of a camera that pans, rolls a little and moves forward over the window."""
    a, dx, dy, dz = 0.01 * (1 - t), 0.06 * (1 - t), -0.03 * (1 - t), 0.05 * (1 - t)
    return [[math.cos(a), -math.sin(a), 0.0, dx], [math.sin(a), math.cos(a), 0.0, dy], [0.0, 0.0, 1.0, 0.0],
            [0.0, 0.0, 1.0, dz]]


def _hit_points(pos, W, H):
    """Hit points (X, Y, Z, 0) whose image is the sample's position for the camera of the sample's time (roll left out)."""
    x, y, t, z = pos.unbind(1)
    Z = torch.where(torch.isfinite(z), 2 + 6 * z, torch.full_like(z, 10.0))
    w = Z + 0.05 * (1 - t)
    out = torch.zeros((pos.shape[0], 4), device=pos.device)
    out[:, 0] = (2 * x / W - 1) * w - 0.06 * (1 - t)
    out[:, 1] = (2 * y / H - 1) * w + 0.03 * (1 - t)
    out[:, 2] = Z
    return out


def _batches(c, seed, dev=DEVICE):
    """The sample batches of a case in insertion order: what fills the buffer, then what a pass inserts (None: nothing)."""
    scene, slots = _Scene(c, seed, dev), c["width"] * c["height"] * c["depth"]
    inc = max(1, int(round(slots * c["rate"]))) if c["do"] == "increment" else 0
    parts = {"step": (0, slots), "increment": (slots, inc)}.get(c["do"], (slots, 0))
    out = []
    for n, span in zip(parts, ((0.0, 1.0 if not inc else 0.9), (0.0 if not inc else 0.9, 1.0))):
        if n == 0:
            out.append(None)
            continue
        pos, col, mo = scene.samples(n, *span)
        world = None
        if c["world"]:
            world = _hit_points(pos, c["width"], c["height"])
            mo = torch.zeros_like(mo)   # static geometry: the camera moves
        out.append((pos, col.to(DTYPES[c["color"]]), mo, world))
    return out


def _stream_cases(c):
    return [_case("redisplay", w, h, b, c["color"], c["radius"]) 
            for w, h, b in (map(int, v.split("x")) for v in c["mix"].split())]


def _new_theta(seed):
    """Width parameters near the defaults."""
    u = torch.rand(6, generator=torch.Generator().manual_seed(seed + 7)).tolist()
    v = (0.8 + 0.4 * u[0], 0.2 * u[1], 2 + u[2], 0.8 + 0.4 * u[3], 0.1 * u[4], 0.6 + 0.4 * u[5])
    return tuple(torch.tensor(v, dtype=torch.float32).tolist())


def prepare(case, seed):
    from paper_2510_15876_gb300.api import BatchReconstructor, Reconstructor

    c = case
    if c["do"] == "streams":
        recs = []
        for k, q in enumerate(_stream_cases(c)):
            rec = Reconstructor(q["width"], q["height"], q["depth"], radius=q["radius"], color_type=q["color"],
                                device=DEVICE)
            rec.insert(*_batches(q, seed * 16 + k)[0][:3])
            recs.append(rec)
        return dict(case=c, recs=recs, batch=BatchReconstructor(recs))
    W, H = c["width"], c["height"]
    rec = Reconstructor(W, H, c["depth"], radius=c["radius"], color_type=c["color"], fifo_capacity=c["fifo"] * W * H,
                        world_points=c["world"], device=DEVICE)
    dev = rec.device
    fill, inc = _batches(c, seed)
    s = dict(case=c, rec=rec, inc=inc, camera=_camera(T_NOW) if c["world"] else None,
             out=torch.empty((H, W, 4), device=dev), tiles=torch.empty((rec.n_tiles, 8), device=dev))
    if inc is not None:
        rec.reserve(max(inc[0].shape[0], fill[0].shape[0] if fill else 0))
    if fill is not None:
        rec.insert(*fill)
    if c["do"] == "sampler":
        s["error"] = (torch.empty(rec.n_tiles, device=dev), torch.empty(5, device=dev))
    if c["do"] in ("redisplay", "filter", "fit"):
        t = c["t_now"] if c["do"] == "redisplay" else T_NOW
        rec.estimate_gradients(t)
        rec.reproject(t)
    if c["adaptive"]:
        for _ in range(SETTLE):
            rec.reconstruct(c["t_now"], out=s["out"], flags=ADAPTIVE)
    if c["do"] in ("filter", "fit"):
        s["theta"] = _new_theta(seed)
    if c["do"] == "fit":
        n = rec.query()["frame"]
        g = torch.Generator(device=dev)
        g.manual_seed(seed + 3)
        s["theta"] = torch.tensor(s["theta"], device=dev, requires_grad=True)
        s["colors"] = torch.rand((n, 3), generator=g, device=dev).requires_grad_()
        s["gout"] = torch.randn((H, W, 4), generator=g, device=dev)
        s["grads"] = torch.zeros((W * H * c["depth"], 3), device=dev)   # the optimiser's buffer, a row per slot
    return s


ADAPTIVE, SETTLE = 2, 5   # AFR_RECON_ADAPTIVE_SUPPORT; images after which most footprints have settled


def _tiles(raw):
    return {"counts": raw.view(torch.int32)[:, :2], "values": raw[:, 2:]}


def run(state):
    c, rec = state["case"], state.get("rec")
    do = c["do"]
    if do in ("step", "increment"):
        pos, col, mo, world = state["inc"]
        rec.insert(pos, col, mo, world, reset=do == "step")
        img, tiles = rec.refresh(T_NOW, out=state["out"], tiles=state["tiles"], view_proj=state["camera"])
        return {"image": img, "tiles": _tiles(tiles)}
    if do == "redisplay":
        rec.reproject(c["t_now"])
        return {"image": rec.reconstruct(c["t_now"], out=state["out"], flags=ADAPTIVE if c["adaptive"] else 0)}
    if do == "sampler":
        rec.estimate_gradients(T_NOW)
        tiles = rec.tile_feedback(out=state["tiles"])
        err, gain = rec.tile_error(out=state["error"], gain_on_device=True)
        return {"tiles": _tiles(tiles), "error": err, "gain": gain}
    if do == "filter":
        return {"image": rec.reconstruct(T_NOW, state["theta"], out=state["out"])}
    if do == "fit":
        from paper_2510_15876_gb300.autograd import reconstruct
        img = reconstruct(rec, state["theta"], T_NOW, state["colors"])
        g_theta, g_colors = torch.autograd.grad(img, (state["theta"], state["colors"]), state["gout"])
        state["grads"][:g_colors.shape[0]].copy_(g_colors)
        return {"image": img.detach(), "theta": g_theta, "colors": state["grads"]}
    return {"images": state["batch"].refresh(T_NOW)}


# ---- work ---------------------------------------------------------------------------


def _kept(per_pixel, depth):
    """Expected samples a queue keeps when its pixel gets Poisson(per_pixel) of them."""
    p, kept, left = math.exp(-per_pixel), 0.0, 1.0
    for k in range(depth):
        kept, left = kept + k * p, left - p
        p *= per_pixel / (k + 1)
    return kept + depth * left


def work(case):
    c = case
    if c["do"] == "streams":
        parts = [work(q) for q in _stream_cases(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    P, b = c["width"] * c["height"], c["depth"]
    color = 16 if c["color"] == "f32" else 8
    sample = 16 + color + 8 + (16 if c["world"] else 0)   # of a batch: position, colour, motion, hit point
    slot = sample + 4                                     # of a queue: the same and a sequence number
    resident = P * _kept(b, b)
    frame = c["fifo"] * P if c["fifo"] else resident
    pairs = 16.0 * frame * len(_disc(3 if c["adaptive"] else c["radius"])) * (0.2 if c["adaptive"] else 1)
    image, tiles = 16 * P, 32 * -(-c["width"] // TILE) * -(-c["height"] // TILE)
    if c["do"] == "step":
        return {"bytes": P * b * sample + resident * slot + image + tiles, "flops": pairs}
    if c["do"] == "increment":
        n = P * b * c["rate"]
        walk = resident * (4 + 4 + color) + frame * (slot - 4) if c["fifo"] else resident * (slot - 4)
        return {"bytes": n * (sample + slot) + walk + image + tiles, "flops": pairs}
    if c["do"] == "redisplay":   # buffer read, image written; the maps of the widths are read
        return {"bytes": resident * (slot - 4) + 16 * P + image, "flops": pairs}
    if c["do"] == "sampler":
        return {"bytes": resident * (8 + color) + 4 * P + 2 * tiles, "flops": 30.0 * resident}
    if c["do"] == "filter":
        return {"bytes": resident * (16 + color) + 20 * P + image, "flops": pairs}
    # fit: frame read and colour gradients written, image and its gradient
    return {"bytes": resident * (16 + color + 12 + 12) + 20 * P + 2 * image, "flops": 3 * pairs}


# ---- the same in 64 bits --------------------------------------------------------------


def _luminance(c):
    return 0.2126 * c[:, 0] + 0.7152 * c[:, 1] + 0.0722 * c[:, 2]


def _sum_at(i, v, n):
    return torch.zeros(n, dtype=torch.float64, device=v.device).index_add_(0, i, v)


def _newest(pixel, P, b):
    """Indices of the b newest samples of each pixel, by pixel, oldest first."""
    order = torch.sort(pixel, stable=True).indices
    p = pixel[order]
    end = torch.cumsum(torch.bincount(p, minlength=P), 0)
    return order[end[p] - torch.arange(p.numel(), device=p.device) <= b]


class _Exact:
    def __init__(self, c, seed):
        self.c, self.W, self.H, self.b = c, c["width"], c["height"], c["depth"]
        self.P = self.W * self.H
        got = [p for p in _batches(c, seed) if p is not None]
        pos, col, mo, world = (None if p[0] is None else torch.cat(p) for p in zip(*got))
        dev = pos.device
        px = pos[:, 1].floor().long() * self.W + pos[:, 0].floor().long()
        keep = _newest(px, self.P, self.b)
        self.px, self.t, self.col, self.seq = px[keep], pos[keep, 2], col[keep, :3].double(), keep
        n = pos.shape[0]
        src = torch.arange(max(0, n - c["fifo"] * self.P), n, device=dev) if c["fifo"] else torch.sort(keep).values
        self.src = tuple(None if v is None else v[src] for v in (pos, col, mo, world))
        ty, tx = torch.arange(self.P, device=dev) // self.W // TILE, torch.arange(self.P, device=dev) % self.W // TILE
        self.ntx, self.nty = -(-self.W // TILE), -(-self.H // TILE)
        self.tile = ty * self.ntx + tx
        self.nt = self.ntx * self.nty

    def gradients(self, t_now):
        P, W, H, px = self.P, self.W, self.H, self.px
        age = (t_now - self.t.double()).clamp_(min=0)
        w, lum = torch.exp(-3.47 * age), _luminance(self.col)
        self.cnt = torch.bincount(px, minlength=P)
        sw = _sum_at(px, w, P)
        some = self.cnt > 0
        mean = torch.where(some, _sum_at(px, w * lum, P) / sw, float("nan"))
        m2 = _sum_at(px, w * (lum - mean[px]) ** 2, P)
        by_t = torch.sort(self.t, stable=True).indices            # keeps older sequence numbers first within a pixel
        o = by_t[torch.sort(px[by_t], stable=True).indices]       # by pixel, then time, oldest first
        same = px[o][1:] == px[o][:-1]
        new, old = o[1:][same], o[:-1][same]
        num = _sum_at(px[new], w[new] * (lum[new] - lum[old]).abs(), P)
        den = _sum_at(px[new], w[new] * (self.t[new].double() - self.t[old].double()), P)
        self.gt = torch.where(den > 0, num / den.clamp(min=1e-300), 0.0)
        m = mean.view(H, W)
        side = []
        for dim in (1, 0):
            d = torch.diff(m, dim=dim).abs()
            ok = ~torch.isnan(d)
            d = torch.nan_to_num(d)
            size = list(m.shape)
            size[dim] = 1
            z = torch.zeros(size, dtype=torch.float64, device=m.device)
            s = torch.cat([z, d], dim) + torch.cat([d, z], dim)
            k = torch.cat([z, ok.double()], dim) + torch.cat([ok.double(), z], dim)
            side.append(torch.where(k > 0, s / k.clamp(min=1), 0.0).reshape(-1))
        self.gx, self.gy = side
        # tile statistics: moments merged over pixels
        T, nt = self.tile, self.nt
        self.area = torch.bincount(T, minlength=nt).double()
        self.n = _sum_at(T, self.cnt.double(), nt)
        ne = _sum_at(T, some.double(), nt)
        tw, ml = _sum_at(T, sw, nt), torch.nan_to_num(mean)
        tmean = torch.where(tw > 0, _sum_at(T, sw * ml, nt) / tw.clamp(min=1e-300), 0.0)
        var = _sum_at(T, m2 + sw * torch.where(some, ml - tmean[T], 0.0) ** 2, nt)
        self.var = torch.where(tw > 0, var / tw.clamp(min=1e-300), 0.0)
        self.empty = self.area * self.b - self.n
        self.u = torch.where(self.empty > 0, 1 - (UNDER_M * self.empty.mean() / self.empty.clamp(min=1)).clamp(max=1), 0.0)
        self.ne, self.sums = ne, [_sum_at(T, g, nt) for g in (self.gx, self.gy, self.gt)]
        self.age = _sum_at(T[px], age, nt)
        means = [torch.where(ne > 0, g / ne.clamp(min=1), 0.0) for g in self.sums]
        values = torch.stack([tmean, self.var, *means, self.u], 1)
        counts = torch.stack([self.n, self.empty], 1).to(torch.int32)
        return {"counts": counts, "values": values}

    def tile_error(self):
        kappa = lam = 0.5
        e = self.area * sum(k * v / v.sum() if float(v.sum()) > 0 else 0 * v for k, v in ((kappa, self.var), (lam, self.u)))
        ne, held = self.ne.sum(), self.n > 0
        ds, dt = 0.5 * (self.sums[0].sum() + self.sums[1].sum()) / ne, self.sums[2].sum() / ne
        age = (self.age[held] / self.n[held]).mean()
        width = dt * age / ds.clamp(min=EPS)
        count = torch.where(width > 0, (self.P / width ** 2).clamp(1.0, float(self.P)), float(self.P))
        return e, torch.stack([ds, dt, age, width, count])

    def reproject(self, t_now, camera=None):
        pos, col, mo, world = self.src
        W, H = self.W, self.H
        a = torch.tensor(t_now, dtype=torch.float32, device=pos.device) - pos[:, 2]   # single precision, as the entry point states
        x, y, ok = pos[:, 0], pos[:, 1], torch.ones_like(a, dtype=torch.bool)
        if camera is not None:
            m = torch.tensor(camera, dtype=torch.float32)
            r = []
            for k in (0, 1, 3):
                v = world[:, 0] * m[k, 0].item()
                for i in (1, 2):
                    v = v + world[:, i] * m[k, i].item()
                r.append(v + m[k, 3].item())
            x, y, ok = (r[0] / r[2] * 0.5 + 0.5) * W, (r[1] / r[2] * 0.5 + 0.5) * H, r[2] > 0
        sx, sy = mo[:, 0] * a, mo[:, 1] * a
        x, y = x + sx, y + sy
        ok = ok & (x >= 0) & (x < W) & (y >= 0) & (y < H)
        q = torch.nonzero(ok).squeeze(1)
        x, y, a = x[q], y[q], a[q]
        fbin = y.floor().long() * W + x.floor().long()
        o = torch.sort(fbin, stable=True).indices                # the sources are in sequence order
        self.fbin, self.fx, self.fy = fbin[o], x[o].double(), y[o].double()
        self.fa2, self.fc = (a[o].double()) ** 2, col[q][o, :3].double()
        return self.fbin.numel()

    def widths(self, theta):
        V = (self.area * WINDOW / self.n.clamp(min=1))[self.tile]
        gs, gt = (0.5 * (self.gx + self.gy)).clamp(min=EPS), self.gt.clamp(min=EPS)
        self.es, self.et = (V * gt / gs) ** (1 / 3), (V * gs * gs / (gt * gt)) ** (1 / 3)
        self.raw_s, self.raw_t = theta[0] * self.es + theta[1], theta[3] * self.et + theta[4]
        self.ss, self.st = self.raw_s.clamp(min=0.5).clamp(max=theta[2]), self.raw_t.clamp(min=0.05).clamp(max=theta[5])

    def pairs(self, radius):
        """(records, pixels, d^2, weight) of every record and the pixel at each offset of the disc, in parts.
        radius: the footprint of every pixel, or a map of them."""
        W, H, part = self.W, self.H, 1 << 23
        one = isinstance(radius, int)
        for dx, dy in _disc(radius if one else int(radius.max())):
            for k in range(0, self.fbin.numel(), part):
                e = torch.arange(k, min(k + part, self.fbin.numel()), device=self.fbin.device)
                px, py = self.fbin[e] % W - dx, self.fbin[e] // W - dy
                ok = (px >= 0) & (px < W) & (py >= 0) & (py < H)
                if not one:
                    ok &= radius[(py.clamp(0, H - 1) * W + px.clamp(0, W - 1))] ** 2 >= dx * dx + dy * dy
                e, px, py = e[ok], px[ok], py[ok]
                p = py * W + px
                d2 = (self.fx[e] - (px + 0.5)) ** 2 + (self.fy[e] - (py + 0.5)) ** 2
                w = torch.exp(-d2 / (2 * self.ss[p] ** 2) - self.fa2[e] / (2 * self.st[p] ** 2))
                yield e, p, d2, w

    def image(self, radius, more=False):
        S = torch.zeros((self.P, 12 if more else 4), dtype=torch.float64, device=self.fx.device)
        for e, p, d2, w in self.pairs(radius):
            v = torch.cat([self.fc[e] * w[:, None], w[:, None]], 1)
            if more:
                v = torch.cat([v, v * d2[:, None], v * self.fa2[e][:, None]], 1)
            S.index_add_(0, p, v)
        some = S[:, 3] > 0
        self.S = S
        out = torch.where(some[:, None], torch.cat([S[:, :3] / S[:, 3:4].clamp(min=1e-300), S[:, 3:4]], 1), 0.0)
        return out.view(self.H, self.W, 4)

    def adjoint(self, radius, gout, theta):
        S, g = self.S, gout.view(-1, 4)[:, :3].double()
        some = S[:, 3] > 0
        inv = torch.where(some, 1 / S[:, 3].clamp(min=1e-300), 0.0)
        C = S[:, :3] * inv[:, None]
        gs = (g * (S[:, 4:7] - C * S[:, 7:8])).sum(1) * inv / self.ss ** 3
        gt = (g * (S[:, 8:11] - C * S[:, 11:12])).sum(1) * inv / self.st ** 3
        out = []
        for gv, raw, e, lo, hi in ((gs, self.raw_s, self.es, 0.5, theta[2]), (gt, self.raw_t, self.et, 0.05, theta[5])):
            top = raw.clamp(min=lo) >= hi
            mid = ~top & (raw > lo)
            out += [(gv * e)[mid].sum(), gv[mid].sum(), gv[top].sum()]
        gc, gn = torch.zeros_like(self.fc), g * inv[:, None]
        for e, p, d2, w in self.pairs(radius):
            gc.index_add_(0, e, gn[p] * w[:, None])
        return torch.stack(out), gc

    def footprints(self, images):
        """Footprint radii of an adaptive reconstruction after as many images: single precision, in the stated order."""
        W, H, dev = self.W, self.H, self.fx.device
        cnt = torch.bincount(self.fbin, minlength=self.P).view(H, W)
        r, n = torch.full((H, W), float(self.c["radius"]), device=dev), torch.full((H, W), -1, device=dev)
        for _ in range(images):
            s, k = torch.zeros((H, W), device=dev), torch.zeros((H, W), device=dev)
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    to = (slice(max(0, -dy), H - max(0, dy)), slice(max(0, -dx), W - max(0, dx)))
                    at = (slice(max(0, dy), H - max(0, -dy)), slice(max(0, dx), W - max(0, -dx)))
                    s[to] += r[at]
                    k[to] += 1
            f = torch.where((n >= 0) & (n < 4), 4.0, torch.where(n > 32, 0.7, 1.0)).float()
            r = ((s / k) * f).clamp(0.5, 8.0)
            R = torch.floor(r + 0.5).long()
            n = torch.zeros((H, W), dtype=torch.long, device=dev)
            for dx, dy in _disc(int(R.max())):
                if abs(dx) >= W or abs(dy) >= H:
                    continue
                to = (slice(max(0, -dy), H - max(0, dy)), slice(max(0, -dx), W - max(0, dx)))
                at = (slice(max(0, dy), H - max(0, -dy)), slice(max(0, dx), W - max(0, -dx)))
                n[to] += torch.where(R[to] ** 2 >= dx * dx + dy * dy, cnt[at], 0)
        return R.reshape(-1)


def exact(case, seed):
    c = case
    if c["do"] == "streams":
        out = []
        for k, q in enumerate(_stream_cases(c)):
            x = _Exact(q, seed * 16 + k)
            x.gradients(T_NOW)
            x.reproject(T_NOW)
            x.widths(THETA)
            out.append(x.image(q["radius"]))
        return {"images": out}
    x, R = _Exact(c, seed), c["radius"]
    t = c["t_now"] if c["do"] == "redisplay" else T_NOW
    tiles = x.gradients(t)
    if c["do"] == "sampler":
        err, gain = x.tile_error()
        return {"tiles": tiles, "error": err, "gain": gain}
    n = x.reproject(t, _camera(T_NOW) if c["world"] else None)
    theta = _new_theta(seed) if c["do"] in ("filter", "fit") else THETA
    x.widths(theta)
    if c["do"] in ("step", "increment"):
        return {"image": x.image(R), "tiles": tiles}
    if c["do"] == "fit":
        g = torch.Generator(device=x.fx.device)
        g.manual_seed(seed + 3)
        x.fc = torch.rand((n, 3), generator=g, device=x.fx.device).to(DTYPES[c["color"]]).double()
        gout = torch.randn((x.H, x.W, 4), generator=g, device=x.fx.device)
        img = x.image(R, more=True)
        g_theta, g_colors = x.adjoint(R, gout, theta)
        pad = torch.zeros((x.P * x.b - n, 3), dtype=torch.float64, device=x.fx.device)
        return {"image": img, "theta": g_theta, "colors": torch.cat([g_colors, pad])}
    return {"image": x.image(x.footprints(SETTLE + 1) if c["adaptive"] else R)}
