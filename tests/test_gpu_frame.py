"""The one-launch path of a single frame (features resident in shared
memory) against the launch-per-stage path, which a handle takes while its
per-launch timers are on: labels, centres and the updates performed are equal
bit for bit. Geometries cover every split of a cell into units (1 to 4 pixel
pairs per lane, 16-column and narrower units, cells wider than a unit), ragged
last cells, fewer units than CTAs, and the largest resident frames."""
import pytest

from paper_1509_04232_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [  # (W, H, S, iterations, options)
    (320, 240, 16, 10, {}),
    (321, 243, 16, 3, dict(in_channels=4)),
    (1920, 1080, 16, 5, {}),
    (1283, 721, 13, 4, dict(in_channels=4, perturb_seeds=True, convergence=0.2)),
    (640, 480, 8, 2, dict(color_space=1)),
    (333, 257, 7, 3, dict(color_space=2)),
    (500, 400, 21, 3, {}),
    (1000, 700, 32, 2, dict(convergence=0.5)),
    (257, 129, 100, 2, {}),
    (17, 5, 9, 4, {}),
    (64, 1, 16, 2, {}),
    (1, 64, 16, 2, {}),
    (40, 30, 64, 3, {}),
    (1, 2000, 12, 3, {}),
    (2000, 1300, 16, 1, dict(enforce_connectivity=0)),
    (700, 500, 15, 0, {}),
    (900, 650, 10, 2, dict(enforce_connectivity=2)),
]


def _frame(W, H, channels, seed):
    import torch
    return torch.from_numpy(synth.voronoi_frame(W, H, 60, 8.0, seed, channels=channels)).cuda()


@pytest.mark.parametrize("W,H,S,iterations,kw", CASES)
def test_one_launch_equals_launch_per_stage(slic_gpu, W, H, S, iterations, kw):
    import torch
    img = _frame(W, H, kw.get("in_channels", 3), 5000 + W)
    one = slic_gpu.Segmenter(W, H, S=S, iterations=iterations, **kw)
    per = slic_gpu.Segmenter(W, H, S=S, iterations=iterations, **kw)
    slic_gpu.slic_profile_enable(per.handle, True)
    for start in (None, torch.rand(one.K_eff, 6, device="cuda") * 20):  # grid start, then given centres
        if start is not None:
            start[:, 3] = start[:, 3] * W / 20
            start[:, 4] = start[:, 4] * H / 20
        want = per.segment(img, init_centres=start)
        for _ in range(2):  # the second run finds the barrier counters and sums of the first
            got = one.segment(img, init_centres=start)
            one.status()
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
            assert one.iterations_run == per.iterations_run


def test_one_launch_replays_in_a_graph_and_in_place(slic_gpu):
    import torch
    img = _frame(640, 480, 3, 77)
    seg = slic_gpu.Segmenter(640, 480, S=16, iterations=4)
    labels, centres = seg.segment(img)
    out_l, out_c = torch.empty_like(labels), torch.empty_like(centres)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        seg.segment(img, out_l, out_c)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            seg.segment(img, out_l, out_c)
        for _ in range(3):
            out_l.zero_()
            g.replay()
    torch.cuda.synchronize()
    seg.status()
    assert torch.equal(out_l, labels) and torch.equal(out_c, centres)
    # initial centres in the output buffer itself
    start = centres.clone()
    want = seg.segment(img, init_centres=start)
    got = seg.segment(img, centres=centres, init_centres=centres)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def _captured_nodes(call, stream):
    """Node types of the graph that `call` is captured into on `stream`, and the graph's launch."""
    import ctypes
    cu = ctypes.CDLL("libcuda.so.1")
    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    ok = lambda r: r == 0 or pytest.fail(f"driver call failed: {r}")  # noqa: E731
    s = ctypes.c_void_p(stream.cuda_stream)
    ok(cu.cuStreamBeginCapture_v2(s, 1))  # (thread-local mode)
    call()
    ok(cu.cuStreamEndCapture(s, ctypes.byref(graph)))
    ok(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    ok(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
    kinds = []
    for node in nodes:
        kind = ctypes.c_int()
        ok(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        kinds.append(kind.value)
    ok(cu.cuGraphDestroy(graph))
    return kinds


@pytest.mark.parametrize("noalloc", [False, True])
def test_the_barrier_counter_is_cleared_for_every_launch(slic_gpu, noalloc):
    """A call of either entry point is the clear of the barrier counter and the
    one kernel: no launch relies on what the one before it has left."""
    import torch
    kernel, memset = 0, 2  # CU_GRAPH_NODE_TYPE_KERNEL, CU_GRAPH_NODE_TYPE_MEMSET
    img = _frame(320, 240, 3, 5)
    seg = slic_gpu.Segmenter(320, 240, S=16, iterations=3)
    want = seg.segment(img)
    labels, centres = torch.empty_like(want[0]), torch.empty_like(want[1])
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    if noalloc:
        run = lambda: slic_gpu.slic_segment_noalloc(seg.params, img.data_ptr(), labels.data_ptr(),  # noqa: E731
                                                    centres.data_ptr(), stream.cuda_stream)
    else:
        run = lambda: seg.segment(img, labels, centres, stream=stream)  # noqa: E731
    run()
    torch.cuda.synchronize()
    assert torch.equal(labels, want[0]) and torch.equal(centres, want[1])
    assert sorted(_captured_nodes(run, stream)) == [kernel, memset]
