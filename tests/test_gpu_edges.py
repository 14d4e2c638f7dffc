"""Edges of the batched block pass, of the label sums and of the network's
weight gradients: remainders, the smallest sizes, and the sizes where a launch
splits its work differently."""
import numpy as np
import pytest

import oracle
from oracle import net_oracle as NO
from paper_1509_04232_gb300 import synth

pytestmark = pytest.mark.gpu


def _img(W, H, seed, channels=3):
    import torch
    return torch.from_numpy(synth.voronoi_frame(W, H, 60, 8.0, seed, channels=channels)).cuda()


# (frames as (W, H, S, options), iterations, launch shape, groups). S = 8 and
# multiples of 16 run over blocks, other S over tiles, all in one batch.
BLOCKS = [
    ([(16, 16, 16, {}), (17, 15, 16, {}), (1, 1, 16, {}), (31, 33, 16, {})], 3, None, 1),
    ([(640, 360, 16, {}), (333, 257, 32, {}), (500, 90, 48, {}), (97, 400, 64, {})], 4, (0, 3, 2, 64), 2),
    ([(320, 240, 16, {}), (320, 240, 8, {}), (200, 100, 32, {}), (211, 130, 13, {}), (64, 64, 16, {})], 3, None, 3),
    ([(320, 240, 32, dict(in_channels=4)), (322, 243, 8, {}), (401, 300, 16, dict(color_space=1))], 2, (1, 3, 2, 64), 1),
    ([(300, 200, 16, dict(convergence=0.5)), (300, 200, 16, {}), (170, 200, 32, dict(convergence=1.0))], 6, None, 1),
    ([(8, 8, 8, {}), (9, 17, 8, {}), (1, 1, 8, {}), (23, 41, 8, {}), (16, 16, 8, {}), (7, 100, 8, {})], 3, None, 1),
    ([(642, 203, 8, dict(convergence=0.5)), (120, 88, 8, dict(perturb_seeds=True)), (48, 48, 24, {}),
      (333, 64, 8, dict(in_channels=4))], 5, None, 2),
    ([(40, 600, 16, dict(perturb_seeds=True)), (2000, 20, 16, dict(color_space=2))], 2, (2, 4, 2, 32), 2),
]


@pytest.mark.parametrize("frames,iterations,shape,groups", BLOCKS)
def test_blocks_equal_launch_per_stage(slic_gpu, frames, iterations, shape, groups):
    """Every frame of the batch is bit-identical to the single frame run stage
    by stage (a handle whose per-launch timers are on)."""
    import torch
    bs = slic_gpu.BatchSegmenter([dict(width=W, height=H, S=S, **kw) for W, H, S, kw in frames], iterations=iterations)
    if shape:
        bs.set_tuning(*shape)
    bs.set_groups(groups)
    imgs = [_img(W, H, 300 + k, kw.get("in_channels", 3)) for k, (W, H, S, kw) in enumerate(frames)]
    bs.bind(imgs)
    for _ in range(2):
        labels, centres = bs.segment()
        bs.status()
    ran = bs.iterations_run
    for k, (W, H, S, kw) in enumerate(frames):
        seg = slic_gpu.Segmenter(W, H, S=S, iterations=iterations, **kw)
        slic_gpu.slic_profile_enable(seg.handle, True)
        want = seg.segment(imgs[k])
        assert torch.equal(labels[k], want[0]) and torch.equal(centres[k], want[1]), k
        assert ran[k] == seg.iterations_run


def test_blocks_of_many_frames_per_warp(slic_gpu):
    """Hundreds of small frames: a warp's run of blocks crosses from frame to
    frame, where its totals go out and its state changes. Every copy of a frame
    is bit-identical to the single frame, on every repetition."""
    import torch
    kinds = [(48, 48, 16), (70, 33, 16), (40, 24, 8), (17, 90, 8), (96, 40, 32), (16, 16, 16)]
    n = 600
    imgs = [_img(W, H, 900 + k) for k, (W, H, _) in enumerate(kinds)]
    want = [slic_gpu.Segmenter(W, H, S=S, iterations=3).segment(imgs[k]) for k, (W, H, S) in enumerate(kinds)]
    of = [f % len(kinds) for f in range(n)]
    bs = slic_gpu.BatchSegmenter([dict(width=kinds[k][0], height=kinds[k][1], S=kinds[k][2]) for k in of], iterations=3)
    bs.bind([imgs[k] for k in of])
    for _ in range(5):
        labels, centres = bs.segment()
        bs.status()
        for f, k in enumerate(of):
            assert torch.equal(labels[f], want[k][0]) and torch.equal(centres[f], want[k][1]), f


SHAPES = [(0, 3, 1, 32), (2, 4, 1, 32), (0, 3, 2, 32), (1, 4, 2, 32), (0, 3, 2, 64), (1, 3, 2, 64)]
TILES = [  # (W, H, S, options): S = 24, 40 and 56 run over tiles, the others over blocks
    [(333, 211, 24, {}), (200, 130, 40, dict(m=20.0))],
    [(1, 1, 24, {}), (33, 65, 40, {}), (64, 32, 24, {}), (31, 100, 56, {})],
    [(320, 240, 16, {}), (333, 257, 24, {}), (100, 90, 8, {}), (130, 211, 40, dict(in_channels=4)), (97, 64, 32, {})],
    [(200, 150, 40, dict(convergence=0.5)), (96, 96, 16, {}), (210, 64, 24, dict(perturb_seeds=True)),
     (70, 130, 24, dict(color_space=1)), (48, 48, 8, {})],
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("frames", TILES)
def test_tiles_of_every_shape_equal_launch_per_stage(slic_gpu, frames, shape):
    """One launch per pass over tiles, in every tile shape and group count,
    alone and among frames that run over blocks: bit-identical to single frames
    run stage by stage."""
    import torch
    bs = slic_gpu.BatchSegmenter([dict(width=W, height=H, S=S, **kw) for W, H, S, kw in frames], iterations=3)
    imgs = [_img(W, H, 500 + k, kw.get("in_channels", 3)) for k, (W, H, S, kw) in enumerate(frames)]
    bs.bind(imgs)
    bs.set_tuning(*shape)
    assert bs.info[3:6] == shape[1:]
    want = []
    for k, (W, H, S, kw) in enumerate(frames):
        seg = slic_gpu.Segmenter(W, H, S=S, iterations=3, **kw)
        slic_gpu.slic_profile_enable(seg.handle, True)
        want.append(seg.segment(imgs[k]))
    for groups in (1, 2, min(4, len(frames))):
        bs.set_groups(groups)
        labels, centres = bs.segment()
        bs.status()
        for k in range(len(frames)):
            assert torch.equal(labels[k], want[k][0]) and torch.equal(centres[k], want[k][1]), (groups, k)


@pytest.mark.parametrize("S", [24, 40])
def test_large_clusters_over_tiles_sum_exactly(slic_gpu, S):
    """One centre wins the 3x3 cells around it (a white square on black, the
    other eight centres on black dots, m small): more pixels of a 32x32 and of a
    32x64 tile than a 32-bit sum of their colours holds (1000 x 100 x 2^15 >
    2^31), in every tile shape of the plain passes."""
    import torch
    W, H = 8 * S, 8 * S
    ns_c = W // S
    img = np.zeros((H, W, 3), np.uint8)
    img[2 * S:5 * S, 3 * S:6 * S] = 255
    white = 3 * ns_c + 4
    cen = oracle.init_centres(oracle.convert(img), S)
    for r in (2, 3, 4):
        for c in (3, 4, 5):
            if r * ns_c + c != white:
                x, y = (int(np.floor(v)) for v in cen[r * ns_c + c, 3:5])
                img[y - 1:y + 2, x - 1:x + 2] = 0
    d_img = torch.from_numpy(img).cuda()
    seg = slic_gpu.Segmenter(W, H, S=S, m=1.0, iterations=3, enforce_connectivity=0)
    slic_gpu.slic_profile_enable(seg.handle, True)
    l1, c1 = seg.segment(d_img)
    lab = l1.cpu().numpy() == white
    tiles = lab[:H // 32 * 32, :W // 32 * 32].reshape(H // 32, 32, W // 32, 32).sum((1, 3))
    assert tiles.max() >= 990 and (tiles[::2][:len(tiles[1::2])] + tiles[1::2]).max() >= 1100
    assert float(c1[white, 0]) > 99.0
    bs = slic_gpu.BatchSegmenter([dict(width=W, height=H, S=S, m=1.0)], iterations=3, enforce_connectivity=0)
    bs.bind([d_img])
    for shape in SHAPES:
        bs.set_tuning(*shape)
        labels, centres = bs.segment()
        bs.status()
        assert torch.equal(labels[0], l1) and torch.equal(centres[0], c1), shape


def _start_centres(seg, kind):
    """Initial centres that the grid's sentinel centres (1e18) can beat: all of
    them, or those around the first and the last cell."""
    import torch
    value = dict(nan=float("nan"), inf=float("inf"), far=3e18, overflow=1e30, corner=float("nan"))[kind]
    c = torch.rand(seg.K_eff, 6, device="cuda") * 20
    if kind != "corner":
        c[:] = value
    else:
        g = c.view(seg.ns_r, seg.ns_c, 6)
        g[:2, :2] = value
        g[-2:, -2:] = value
    return c


@pytest.mark.parametrize("kind", ["nan", "inf", "far", "overflow", "corner", "m"])
def test_labels_and_sums_stay_in_the_grid(slic_gpu, kind):
    """Centres from the caller that are not finite or further off than the
    sentinels around the grid, and an m whose distances would overflow: every
    path gives every pixel a label of the grid, counts every pixel once, leaves
    a neighbouring frame of the batch alone, and agrees with the others."""
    import torch
    geo = [(100, 61, 16), (75, 50, 8), (90, 70, 13), (121, 96, 24), (64, 48, 32), (50, 33, 3), (130, 40, 40)]
    m = 3e38 if kind == "m" else 10.0
    imgs = [_img(W, H, 40 + k) for k, (W, H, _) in enumerate(geo)]
    for iterations in (0, 1):
        kw = dict(m=m, iterations=iterations, enforce_connectivity=0)
        want, start = [], []
        for (W, H, S), img in zip(geo, imgs):
            one = slic_gpu.Segmenter(W, H, S=S, **kw)
            per = slic_gpu.Segmenter(W, H, S=S, **kw)
            slic_gpu.slic_profile_enable(per.handle, True)  # (a launch per stage)
            init = None if kind == "m" else _start_centres(per, kind)
            l, c = per.segment(img, init_centres=init)
            assert int(l.min()) >= 0 and int(l.max()) < per.K_eff
            if iterations:
                assert int(c[:, 5].sum()) == W * H
            l1, c1 = one.segment(img, init_centres=init)
            assert torch.equal(l1, l) and torch.equal(c1.view(torch.int32), c.view(torch.int32))
            want.append((l, c))
            start.append(init)
        ordinary = slic_gpu.Segmenter(80, 48, S=16, iterations=iterations, enforce_connectivity=0)
        good = _img(80, 48, 7)
        want_good = ordinary.segment(good)
        for shape in ([0], [1, 2, 0], [3, 4], [3], [6], [5, 2]):  # blocks, tiles, two row groups, small S
            frames, ims, inits, refs = [], [], [], []
            for k in shape:
                frames += [dict(width=80, height=48, S=16), dict(width=geo[k][0], height=geo[k][1], S=geo[k][2], m=m)]
                ims += [good, imgs[k]]
                inits += [None, start[k]]
                refs += [want_good, want[k]]
            bs = slic_gpu.BatchSegmenter(frames, iterations=iterations, enforce_connectivity=0)
            bs.bind(ims, init_centres=inits)
            same8 = all(f["S"] % 8 == 0 for f in frames)
            for tune, fused in ([((0, 3, 1, 32), False), ((0, 3, 1, 32), True)] +
                                ([((0, 3, 2, 32), False), ((0, 3, 2, 64), False), ((0, 3, 2, 64), True)] if same8 else [])):
                bs.set_tuning(*tune, fused=fused)
                labels, centres = bs.segment()
                bs.status()
                for f, (l, c) in enumerate(refs):
                    assert torch.equal(labels[f], l), (shape, tune, fused, f)
                    assert torch.equal(centres[f].view(torch.int32), c.view(torch.int32)), (shape, tune, fused, f)


@pytest.mark.parametrize("W,H,S,kind", [(64, 8, 8, "noise"), (65, 9, 4, "noise"), (130, 70, 16, "blocks"),
                                        (333, 57, 13, "slots"), (3, 2, 2, "noise"), (256, 128, 2, "noise")])
def test_label_sums(slic_gpu, W, H, S, kind):
    """slic_update from label maps with few and with very many labels per tile
    (more than its table holds), runs, and labels outside [0, K): counts exact,
    means within the centre tolerance 1e-4 max(1, |ref|)."""
    import torch
    seg = slic_gpu.Segmenter(W, H, S=S)
    K = seg.K_eff
    rng = np.random.default_rng(W * H)
    y, x = np.mgrid[0:H, 0:W]
    if kind == "blocks":
        lab = (y // S) * seg.ns_c + x // S
    elif kind == "slots":
        lab = np.clip(y // S + rng.integers(-1, 2, (H, W)), 0, seg.ns_r - 1) * seg.ns_c
        lab += np.clip(x // S + rng.integers(-1, 2, (H, W)), 0, seg.ns_c - 1)
    else:
        lab = rng.integers(-1, K + 1, (H, W))
    feat = rng.uniform(-128, 128, (3, H, W)).astype(np.float32)
    start = rng.uniform(0, 50, (K, 6)).astype(np.float32)
    got = seg.update(torch.from_numpy(feat).cuda(), torch.from_numpy(lab.astype(np.int32)).cuda(),
                     torch.from_numpy(start).cuda()).cpu().numpy()
    ok = (lab >= 0) & (lab < K)
    n = np.bincount(lab[ok], minlength=K)
    np.testing.assert_array_equal(got[:, 5], n)
    for c, v in enumerate([*feat.astype(np.float64), x.astype(np.float64), y.astype(np.float64)]):
        ref = np.where(n > 0, np.bincount(lab[ok], weights=v[ok], minlength=K) / np.maximum(n, 1), start[:, c])
        assert np.all(np.abs(got[:, c] - ref) <= 1e-4 * np.maximum(1.0, np.abs(ref)))


def _away_from_zero(seed):
    """Parameters that keep every hidden pre-activation away from zero: the odd
    channels' biases at +2, the even ones' at -2 (dead channels). At so few
    pixels one ReLU derivative that differs between two roundings of a value
    near zero would be a large part of an element."""
    params = NO.init_params(seed)
    for w, b in params[:3]:
        b += np.where(np.arange(len(b)) % 2, 2.0, -2.0).astype(np.float32)
        w *= 0.1
    return params


@pytest.mark.parametrize("n,W,H", [(1, 64, 2), (3, 65, 3), (2, 30, 1), (2, 31, 5), (1, 129, 7), (2, 72, 4)])
def test_gradients_at_the_edges(slic_gpu, n, W, H):
    """Weight and bias gradients where rows leave half a row pair, columns a
    part of a 64-pixel stage or of a 30-pixel segment, and the batch is below
    the network's largest: the element-wise bound of the gradient test,
    2^-6 |g| + 2^-8 T + 2^-14 T1 (test_gpu_net.py derives it), at parameters
    that meet its premise (no ReLU derivative in doubt). Dead channels'
    gradients are zero exactly."""
    import torch
    import test_gpu_net as N
    from paper_1509_04232_gb300.warmstart import WarmStartNet
    S = 8
    net = WarmStartNet(W, H, S, max_batch=n + 1, seed=11)
    net.set_params(np.concatenate([np.concatenate([w.ravel(), b]) for w, b in _away_from_zero(11)]).astype(np.float32))
    host = np.stack([synth.voronoi_frame(W, H, 12, 8.0, 700 + i) for i in range(n)])
    valid = NO.slot_mask(H, W, S)
    rng = np.random.default_rng(5)
    target = np.array([[[rng.choice(np.flatnonzero(valid[y, x])) for x in range(W)] for y in range(H)]
                       for _ in range(n)], np.uint8)
    net.gradients(torch.from_numpy(host).cuda(), torch.from_numpy(target).cuda())
    torch.cuda.synchronize()
    net.status()
    got, params = N._split(net.grads()), N._split(net.params())
    ref = [[np.zeros_like(v) for v in p] for p in params]
    t0 = [[np.zeros_like(v) for v in p] for p in params]
    t1 = [[np.zeros_like(v) for v in p] for p in params]
    for i in range(n):
        x0 = NO.input_channels(oracle.convert(host[i]), S, 10.0)
        assert min(np.abs(z).min() for _, _, z in NO.forward(x0, params)[1][:3]) > 0.5
        _, g, dzs = NO.backward(x0, params, target[i].astype(np.int64), valid, bf16=True, bf16_grad=True,
                                return_dz=True)
        for l, m in enumerate(N._term_magnitudes(dzs, params)):
            for k in range(2):
                ref[l][k] += g[l][k] / n
                t0[l][k] += m[k] / n
                t1[l][k] += m[2 + k] / n
    for l in range(4):
        for k in range(2):
            bound = 2.0 ** -6 * np.abs(ref[l][k]) + 2.0 ** -8 * t0[l][k] + 2.0 ** -14 * t1[l][k]
            assert np.all(np.abs(got[l][k] - ref[l][k]) <= bound), (l, k)
