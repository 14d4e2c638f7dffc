"""The calls this library is used for, as timed cases.

listed() names them, draw() gives others of the same ranges, prepare() makes
what a program has in hand before the call, run() is one pass through the
package's public entry points, work() the bytes and operations a pass cannot
do without, and exact() the floating outputs in 64 bits, from plain torch.

Kinds of case:
  frame      one image at a time: Segmenter.segment (or, with noalloc, the
             allocation-free entry point), the camera or service call
  stages     the same stages called one by one: convert, init, assign,
             update, two connectivity passes
  batch      many frames per call: BatchSegmenter.segment
  host       the batch from and to page-locked host buffers
  video      a batch bound to new frames and started from given centres
  warm       a batch started from the network's labels
  logits     the warm-start network's forward pass
  gradients  the network's forward and backward pass, with the gradients read
"""
import math

import numpy as np
import torch

import paper_1509_04232_gb300 as slic
from paper_1509_04232_gb300.warmstart import WarmStartNet

REGIONS = 400
MIXED = ((640, 480), (1280, 720), (1920, 1080), (3840, 2160))


def listed():
    return [
        # a small image at full iterations: launches and latency decide
        dict(name="frame_320x240", kind="frame", width=320, height=240, K=300, S=0, m=10.0, iterations=10),
        # one HD frame, the live-camera call
        dict(name="frame_1080p", kind="frame", width=1920, height=1080, K=0, S=16, m=10.0, iterations=5),
        # a ragged RGBA frame with the original algorithm's options on
        dict(name="frame_ragged", kind="frame", width=1283, height=721, K=0, S=13, m=10.0, iterations=10, channels=4,
             perturb=True, convergence=0.2),
        # the stage-by-stage interface, as a program with its own driver calls it
        dict(name="stages_720p", kind="stages", width=1280, height=720, S=16, m=10.0, connectivity=1),
        # the throughput batch at full iterations, in the launch shape the autotuner's cache gives it
        dict(name="batch_1080p", kind="batch", frames=32, width=1920, height=1080, S=16, m=10.0, iterations=10,
             connectivity=1, tuned=True),
        # a service's mixed queue: four sizes, three grid intervals, three compactness values, library defaults
        dict(name="batch_mixed", kind="batch", frames=16, width=0, height=0, S=0, m=0.0, iterations=5, connectivity=1,
             tuned=False),
        # the batch with component connectivity (segments without stray islands)
        dict(name="components_1080p", kind="batch", frames=8, width=1920, height=1080, S=16, m=10.0, iterations=5,
             connectivity=2, tuned=True),
        # end to end: frames in page-locked host memory, labels and centres back
        dict(name="host_1080p", kind="host", frames=16, width=1920, height=1080, S=16, m=10.0, iterations=5,
             connectivity=1, tuned=True),
        # 4K video, eight frames a call, two iterations from the previous centres
        dict(name="video_4k", kind="video", frames=8, width=3840, height=2160, S=16, m=10.0, iterations=2,
             connectivity=1, tuned=False),
        # a batch started from the network's labels
        dict(name="warm_1080p", kind="warm", frames=4, width=1920, height=1080, S=16, m=10.0, iterations=3,
             connectivity=1, tuned=False),
        # the network's scores for four HD frames
        dict(name="logits_1080p", kind="logits", frames=4, width=1920, height=1080, S=16, m=10.0),
        # one training batch of the network: forward and backward, gradients read
        dict(name="gradients_256", kind="gradients", frames=32, width=256, height=256, S=16, m=10.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "stages", "batch", "batch", "host", "video", "warm", "logits",
                       "gradients"])
    while True:
        w, h = _log(rng, 32, 3840), _log(rng, 32, 2160)
        if rng.random() < 0.5:  # half of the widths as cameras give them
            w = max(16, w // 16 * 16)
        if 1 / 8 <= w / h <= 8:
            break
    S = rng.choice([8, 16, 16, 16, 32, rng.randint(5, 40)])
    c = dict(kind=kind, width=w, height=h, S=S, m=rng.choice([5.0, 10.0, 20.0]))
    if kind == "frame":
        c.update(K=0, iterations=rng.randint(1, 10), channels=rng.choice([3, 3, 4]),
                 color_space=rng.choice([slic.SLIC_CIELAB, slic.SLIC_CIELAB, slic.SLIC_RGB, slic.SLIC_XYZ]),
                 perturb=rng.random() < 0.2, convergence=rng.choice([0.0, 0.0, 0.2]),
                 connectivity=rng.choice([0, 1, 1, 2]), noalloc=rng.random() < 0.2 and w * h <= 900_000)
        return c
    if kind == "stages":
        return dict(c, connectivity=rng.choice([1, 2]))
    if kind in ("logits", "gradients", "warm"):
        c["S"] = rng.choice([8, 16, 16, 32])
        most = {"logits": 8_000_000, "gradients": 2_000_000, "warm": 8_000_000}[kind]
        if kind == "gradients":
            c.update(width=_log(rng, 48, 640), height=_log(rng, 48, 480))
        c["frames"] = max(1, min(32, _log(rng, 1, 32), most // (c["width"] * c["height"])))
        if kind == "warm":
            c.update(iterations=rng.randint(0, 5), connectivity=rng.choice([0, 1]), tuned=False)
        return c
    c["iterations"] = rng.randint(1, 3) if kind == "video" else rng.randint(1, 10)
    c["connectivity"] = rng.choice([0, 1, 1, 2]) if kind == "batch" else 1
    c["frames"] = max(2, min(32, _log(rng, 2, 32), 60_000_000 // (w * h)))
    c["tuned"] = S % 8 == 0 and rng.random() < 0.5
    if kind == "batch" and rng.random() < 0.25:
        c.update(width=0, height=0, S=0, m=0.0, frames=rng.randint(4, 16), iterations=rng.randint(1, 6), tuned=False)
    return c


def _geometry(case):
    """(width, height, S, m) of every frame of a case."""
    n = case.get("frames", 1)
    if case["width"]:
        S = case["S"] or max(1, round(math.sqrt(case["width"] * case["height"] / case["K"])))
        return [(case["width"], case["height"], S, case["m"])] * n
    rng = np.random.Generator(np.random.PCG64(2))  # the mixed queue: equal shares of the sizes, S and m drawn
    return [MIXED[f * 4 // n] + (int(rng.choice([8, 16, 32])), float(rng.choice([5.0, 10.0, 20.0]))) for f in range(n)]


# --- inputs -----------------------------------------------------------------

def _image(W, H, gen, channels=3, scene=None, t=0):
    """uint8 [H, W, channels]: nearest-site regions of uniform colour, a global gradient, Gaussian noise."""
    dev = gen.device
    R = 40 if W * H <= 100_000 else REGIONS
    rand = lambda *s: torch.rand(*s, generator=gen, device=dev)  # noqa: E731
    if scene is None:
        scene = _scene(W, H, R, gen)
    sites = scene["sites"] + t * scene["velocity"]
    colours = (scene["colours"] + t * scene["drift"]).clamp(0, 255)
    y, x = torch.meshgrid(torch.arange(H, device=dev, dtype=torch.float32),
                          torch.arange(W, device=dev, dtype=torch.float32), indexing="ij")
    out = torch.empty((H, W, channels), dtype=torch.uint8, device=dev)
    rows = max(1, 2_000_000 // W)
    half = 0.5 * (sites * sites).sum(1)
    for r in range(0, H, rows):
        xs, ys = x[r:r + rows].reshape(-1, 1), y[r:r + rows].reshape(-1, 1)
        region = (half - xs * sites[:, 0] - ys * sites[:, 1]).argmin(1)
        v = colours[region]
        v = v + scene["amplitude"] * (scene["direction"][0] * (xs / W - 0.5) + scene["direction"][1] * (ys / H - 0.5))
        v = v + scene["sigma"] * torch.randn(v.shape, generator=gen, device=dev)
        v = v.round().clamp(0, 255).to(torch.uint8)
        out[r:r + rows, :, :3] = v.view(-1, W, 3)
    if channels == 4:
        out[..., 3] = (rand(H, W) * 256).to(torch.uint8)
    return out


def _scene(W, H, R, gen):
    rand = lambda *s: torch.rand(*s, generator=gen, device=gen.device)  # noqa: E731
    angle, turn = 2 * math.pi * rand(1), 2 * math.pi * rand(R)
    speed = 4.0 * rand(R)
    return dict(sites=rand(R, 2) * torch.tensor([W, H], device=gen.device), colours=255 * rand(R, 3),
                amplitude=30 * rand(3), direction=torch.cat([angle.cos(), angle.sin()]), sigma=6.0 if R > 40 else 8.0,
                velocity=torch.stack([speed * turn.cos(), speed * turn.sin()], 1),
                drift=2.0 * torch.randn(R, 3, generator=gen, device=gen.device))


def _images(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(1_000_003 * seed + 17)
    geo = _geometry(case)
    if case["kind"] == "video":  # frames 1 .. n of one moving scene; the start is frame 0
        W, H = geo[0][:2]
        scene = _scene(W, H, REGIONS, gen)
        return [_image(W, H, gen, scene=scene, t=t) for t in range(len(geo) + 1)]
    return [_image(W, H, gen, case.get("channels", 3)) for W, H, _, _ in geo]


def _weights(seed):
    """A checkpoint of the network: it passes the nine distances through (a trained network's main path), with
    He-normal weights of a twentieth beside them."""
    rng = np.random.Generator(np.random.PCG64(seed + 99))
    parts = []
    for l, (ci, co) in enumerate(((14, 32), (32, 32), (32, 32), (32, 9))):
        w = 0.05 * rng.standard_normal((3, 3, ci, co)) * math.sqrt(2.0 / (9 * ci))
        b = 0.01 * rng.standard_normal(co)
        for t in range(9):
            w[1, 1, 5 + t if l == 0 else t, t] += -2.0 if l == 0 else 1.0
        if l == 0:
            b[:9] += 1.0
        parts += [w.reshape(-1), b]
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    kind, geo = case["kind"], _geometry(case)
    W, H, S, m = geo[0]
    images = _images(case, seed)
    st = dict(kind=kind, images=images)
    if kind in ("frame", "stages"):
        kw = dict(S=S, m=m, iterations=case.get("iterations", 0), color_space=case.get("color_space", 0),
                  enforce_connectivity=case.get("connectivity", 1), in_channels=case.get("channels", 3),
                  perturb_seeds=case.get("perturb", False), convergence=case.get("convergence", 0.0))
        if case.get("K"):
            kw.update(K=case["K"], S=0)
        st["seg"] = slic.Segmenter(W, H, **kw)
        st["noalloc"] = case.get("noalloc", False)
        st["components"] = case.get("connectivity", 1) == 2
        return st
    if kind in ("logits", "gradients", "warm"):
        net = st["net"] = WarmStartNet(W, H, S, max_batch=len(geo), seed=0, m=m)
        net.set_params(_weights(seed))
        if kind != "warm":
            st["stack"] = torch.stack(images)
            st["images"] = None
            if kind == "logits":
                st["logits"] = torch.empty((len(geo), H, W, 16), dtype=torch.float32, device="cuda")
            else:
                st["targets"] = _targets(st["stack"], S, m)
                st["stats"] = torch.zeros(2, dtype=torch.float32, device="cuda")
            return st
    bs = st["bs"] = slic.BatchSegmenter([dict(width=w, height=h, S=s, m=mm) for w, h, s, mm in geo],
                                        iterations=case["iterations"], enforce_connectivity=case["connectivity"])
    if case["tuned"]:  # what the autotuner's cache holds for batches whose S is a multiple of 8
        bs.set_tuning(1, 3, 2, 64, fused=False, groups=min(4, len(geo)))
    if kind == "video":
        st["start"] = _slic64(images[0], S, m, 2)[0].float()
        st["images"] = images = images[1:]
    bs.bind(images)
    if kind == "warm":
        bs.set_warmstart(st["net"])
    if kind == "host":
        st["host"] = torch.stack(images).cpu().pin_memory()
        st["labels"] = torch.empty((len(geo), H, W), dtype=torch.int32).pin_memory()
        st["centres"] = torch.empty((len(geo), bs.K_eff[0], 6), dtype=torch.float32).pin_memory()
    return st


def run(st):
    kind = st["kind"]
    if kind == "frame":
        seg, img = st["seg"], st["images"][0]
        if not st["noalloc"]:
            return seg.segment(img)
        p = seg.params
        labels = torch.empty((p.height, p.width), dtype=torch.int32, device=img.device)
        centres = torch.empty((seg.K_eff, 6), dtype=torch.float32, device=img.device)
        slic.slic_segment_noalloc(p, img.data_ptr(), labels.data_ptr(), centres.data_ptr(),
                                  torch.cuda.current_stream().cuda_stream)
        return labels, centres
    if kind == "stages":
        seg = st["seg"]
        feat = seg.convert(st["images"][0])
        start = seg.init_centres(feat)
        labels = seg.assign(feat, start)
        centres = seg.update(feat, labels, start)
        if st["components"]:
            final = seg.connectivity_components(labels)
        else:
            final = seg.connectivity_pass(seg.connectivity_pass(labels))
        return feat, start, labels, centres, final
    if kind == "logits":
        st["net"].forward(st["stack"], logits=st["logits"])
        return st["logits"]
    if kind == "gradients":
        st["net"].gradients(st["stack"], st["targets"], st["stats"])
        return st["stats"], st["net"].grads()
    bs = st["bs"]
    if kind == "host":
        bs.segment_host(st["host"], st["labels"], st["centres"])
        torch.cuda.current_stream().synchronize()  # the caller reads the results on the host
        return st["labels"], st["centres"]
    if kind == "video":
        bs.bind(st["images"], init_centres=[st["start"]] * len(st["images"]))
    labels, centres = bs.segment()
    return labels, centres


def work(case):
    """Image bytes in, labels and centres (logits, gradients) out; Eq. (1)'s 16 operations for each of 9 candidates of
    every pixel and pass, about 40 for the conversion, 2 x 25,056 for a pixel's way through the network."""
    geo, kind = _geometry(case), case["kind"]
    n_bytes = flops = 0.0
    for W, H, S, _ in geo:
        px, K = W * H, -(-W // S) * -(-H // S)
        if kind in ("logits", "gradients"):
            n_bytes += px * (3 + 64 if kind == "logits" else 4)
            flops += px * 50112.0 * (1 if kind == "logits" else 3)
            continue
        n_bytes += px * (case.get("channels", 3) + 4) + 24 * K
        if kind == "stages":  # five calls: features written once and read twice, labels written three times, read three
            n_bytes += px * (12 * 3 + 4 * 5) + 24 * 4 * K
        flops += px * (40 + 144.0 * (case.get("iterations", 0) + 1))
        if kind == "warm":
            flops += px * 50112.0
    if kind == "gradients":
        n_bytes += 2 * 4 * 25600
    return {"bytes": n_bytes, "flops": flops}


# --- the same results in 64 bits --------------------------------------------

def _features(img, color_space=slic.SLIC_CIELAB, dtype=torch.float64):
    """[3, H, W] features of a uint8 [H, W, C] image: sRGB (IEC 61966-2-1), D65, CIE 1976 L*a*b*."""
    v = img[..., :3].to(dtype)
    if color_space == slic.SLIC_RGB:
        return v.permute(2, 0, 1).contiguous()
    v = v / 255
    lin = torch.where(v <= 0.04045, v / 12.92, ((v + 0.055) / 1.055) ** 2.4)
    M = torch.tensor([[0.4124564, 0.3575761, 0.1804375], [0.2126729, 0.7151522, 0.0721750],
                      [0.0193339, 0.1191920, 0.9503041]], dtype=torch.float64, device=img.device).to(dtype)
    xyz = [sum(M[r, k] * lin[..., k] for k in range(3)) for r in range(3)]
    if color_space == slic.SLIC_XYZ:
        return torch.stack([100 * c for c in xyz])
    f = []
    for r in range(3):
        t = xyz[r] / M[r].sum()
        f.append(torch.where(t > 216 / 24389, t ** (1 / 3), (24389 / 27 * t + 16) / 116))
    return torch.stack([116 * f[1] - 16, 500 * (f[0] - f[1]), 200 * (f[1] - f[2])])


def _grid(f, S, perturb=False):
    """Grid centres [K, 6] of features [3, H, W]: cell midpoints and the colour under them; perturb moves a seed to
    the lowest-gradient pixel of its 3x3 surroundings."""
    _, H, W = f.shape
    dev = f.device
    mid = lambda n: [(i * S + min(i * S + S, n) - 1) / 2 for i in range(-(-n // S))]  # noqa: E731
    ys, xs = (torch.tensor(mid(n), dtype=f.dtype, device=dev) for n in (H, W))
    y, x = (v.reshape(-1) for v in torch.meshgrid(ys, xs, indexing="ij"))
    py, px = y.floor().long(), x.floor().long()
    if perturb:
        at = lambda dy, dx: f[:, (py + dy).clamp(0, H - 1), (px + dx).clamp(0, W - 1)]  # noqa: E731
        grad = lambda dy, dx: (((at(dy, dx + 1) - at(dy, dx - 1)) ** 2).sum(0)  # noqa: E731
                               + ((at(dy + 1, dx) - at(dy - 1, dx)) ** 2).sum(0))
        best, by, bx = grad(0, 0), torch.zeros_like(py), torch.zeros_like(px)
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                if dy or dx:
                    g = grad(dy, dx)
                    ok = (g < best) & (py + dy >= 0) & (py + dy < H) & (px + dx >= 0) & (px + dx < W)
                    best, by, bx = torch.where(ok, g, best), torch.where(ok, dy, by), torch.where(ok, dx, bx)
        moved = (by != 0) | (bx != 0)
        py, px = py + by, px + bx
        x, y = torch.where(moved, px.to(x.dtype), x), torch.where(moved, py.to(y.dtype), y)
    c = f[:, py, px]
    return torch.stack([c[0], c[1], c[2], x, y, torch.zeros_like(x)], 1)


def _window(f, S, centres, w):
    """Yields (slot, cell index, in-grid mask, D) of the 9 cells around each pixel's own."""
    _, H, W = f.shape
    nr, nc = -(-H // S), -(-W // S)
    y = torch.arange(H, device=f.device)[:, None]
    x = torch.arange(W, device=f.device)[None, :]
    for t in range(9):
        r, c = y // S + t // 3 - 1, x // S + t % 3 - 1
        ok = (r >= 0) & (r < nr) & (c >= 0) & (c < nc)
        k = r.clamp(0, nr - 1) * nc + c.clamp(0, nc - 1)
        g = centres[k]
        d = sum((g[..., i] - f[i]) ** 2 for i in range(3)).sqrt()
        yield t, k, ok, d + w * ((g[..., 3] - x) ** 2 + (g[..., 4] - y) ** 2).sqrt()


def _assign(f, S, centres, w):
    best = torch.full(f.shape[1:], float("inf"), dtype=f.dtype, device=f.device)
    lab = torch.zeros(f.shape[1:], dtype=torch.int64, device=f.device)
    for _, k, ok, d in _window(f, S, centres, w):
        take = ok & (d < best)
        best, lab = torch.where(take, d, best), torch.where(take, k, lab)
    return lab


def _update(f, lab, centres):
    _, H, W = f.shape
    y = torch.arange(H, device=f.device, dtype=f.dtype)[:, None].expand(H, W)
    x = torch.arange(W, device=f.device, dtype=f.dtype)[None, :].expand(H, W)
    rows = torch.stack([f[0], f[1], f[2], x, y, torch.ones_like(f[0])], -1).reshape(-1, 6)
    s = torch.zeros_like(centres).index_add_(0, lab.reshape(-1), rows)
    n = s[:, 5:]
    return torch.where(n > 0, torch.cat([s[:, :5] / n.clamp(min=1), n], 1), torch.cat([centres[:, :5], n], 1))


def _slic64(img, S, m, iterations, color_space=0, perturb=False, convergence=0.0, start=None, labels=None):
    """(centres, labels before connectivity) of the whole method."""
    f = _features(img, color_space)
    c = _grid(f, S, perturb) if start is None else start.to(f.dtype)
    if labels is not None:
        c = _update(f, labels, c)
    lab = _assign(f, S, c, m / S)
    move = math.inf
    for _ in range(iterations):
        if convergence > 0 and move < convergence:
            break
        new = _update(f, lab, c)
        move = float((new[:, 3:5] - c[:, 3:5]).abs().sum() / c.shape[0])
        c = new
        lab = _assign(f, S, c, m / S)
    return c, lab


def _channels(img, S, m):
    """The network's 14 input channels [14, H, W] of one image, in 64 bits."""
    f = _features(img)
    _, H, W = f.shape
    y = torch.arange(H, device=f.device, dtype=f.dtype)[:, None].expand(H, W)
    x = torch.arange(W, device=f.device, dtype=f.dtype)[None, :].expand(H, W)
    out = [f[0] / 100, f[1] / 128, f[2] / 128, (x % S) / S, (y % S) / S]
    for _, _, ok, d in _window(f, S, _grid(f, S), m / S):
        out.append(torch.where(ok, d / 100, torch.full_like(d, 2.0)))
    return torch.stack(out)


def _network(x, layers):
    """Logits [H, W, 9] of channels [14, H, W]: four 3x3 layers, zero padding, ReLU between."""
    H, W = x.shape[1:]
    a = x.permute(1, 2, 0)
    for i, (w, b) in enumerate(layers):
        p = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1))
        a = b + sum(p[dy:dy + H, dx:dx + W] @ w[dy, dx] for dy in range(3) for dx in range(3))
        if i < 3:
            a = a.relu()
    return a


def _layers(seed):
    flat, out = torch.from_numpy(_weights(seed)).cuda().double(), []
    for ci, co in ((14, 32), (32, 32), (32, 32), (32, 9)):
        w, flat = flat[:9 * ci * co].view(3, 3, ci, co), flat[9 * ci * co:]
        out.append((w, flat[:co]))
        flat = flat[co:]
    return out


def _slots_ok(H, W, S):
    y, x = torch.arange(H, device="cuda")[:, None] // S, torch.arange(W, device="cuda")[None, :] // S
    nr, nc = -(-H // S), -(-W // S)
    return torch.stack([(y + t // 3 - 1 >= 0) & (y + t // 3 - 1 < nr) & (x + t % 3 - 1 >= 0) & (x + t % 3 - 1 < nc)
                        for t in range(9)], -1)


def _targets(stack, S, m):
    """Slots of the nearest grid centres, uint8 [n, H, W]: what labels of a first assignment give."""
    return torch.stack([_channels(i, S, m)[5:].argmin(0) for i in stack]).to(torch.uint8)


def exact(case, seed):
    kind, geo = case["kind"], _geometry(case)
    images = _images(case, seed)
    if kind == "stages":
        W, H, S, m = geo[0]
        f = _features(images[0])
        start = _grid(f, S)
        return f, start, None, _update(f, _assign(f, S, start, m / S), start), None
    if kind in ("logits", "gradients"):
        W, H, S, m = geo[0]
        layers = _layers(seed)
        ok = _slots_ok(H, W, S)
        if kind == "logits":
            return torch.stack([torch.nn.functional.pad(_network(_channels(i, S, m), layers), (0, 7)) for i in images])
        targets = _targets(torch.stack(images), S, m).long()
        flat = [p.clone().requires_grad_() for l in layers for p in l]
        loss = right = 0.0
        for i, t in zip(images, targets):
            z = _network(_channels(i, S, m), list(zip(flat[::2], flat[1::2]))).masked_fill(~ok, float("-inf"))
            one = -z.log_softmax(-1).gather(-1, t[..., None]).sum()
            (one / (W * H * len(images))).backward()
            loss += float(one)
            right += float((z.argmax(-1) == t).sum())
        grads = torch.cat([p.grad.reshape(-1) for p in flat])
        return torch.tensor([loss, right], dtype=torch.float64), grads.cpu().numpy()
    opts = dict(color_space=case.get("color_space", 0), perturb=case.get("perturb", False),
                convergence=case.get("convergence", 0.0))
    if kind == "video":
        W, H, S, m = geo[0]
        opts["start"] = _slic64(images[0], S, m, 2)[0].float()
        images = images[1:]
    centres = []
    for img, (W, H, S, m) in zip(images, geo):
        if kind == "warm":
            z = _network(_channels(img, S, m), _layers(seed)).masked_fill(~_slots_ok(H, W, S), float("-inf"))
            t, nc = z.argmax(-1), -(-W // S)
            y, x = torch.arange(H, device="cuda")[:, None], torch.arange(W, device="cuda")[None, :]
            opts["labels"] = (y // S + t // 3 - 1) * nc + x // S + t % 3 - 1
        centres.append(_slic64(img, S, m, case["iterations"], **opts)[0])
    if kind == "frame":
        return None, centres[0]
    if kind == "host":
        return None, torch.stack(centres)
    return [None] * len(centres), centres
