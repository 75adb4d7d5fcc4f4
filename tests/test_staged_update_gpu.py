"""The staged update of the pipelined kernel against the plain kernel, bit for
bit, where its rare branches meet: states whose bias product is about to be
rescaled, with empty, equal, zero and largest keys, under flushed pixels, every
rule, bias and colour precision, with and without the fused resolve."""
import numpy as np
import pytest
import torch

import paper_2510_03964_gb300 as wrs

pytestmark = pytest.mark.gpu


def _seeded_state(st, K, hw, rng):
    raw = st.export_raw()
    pl, lay = st.layout.plane_px, st.layout

    def plane(off, n):
        return raw[off: off + 4 * n * pl].view(np.float32).reshape(n, pl)[:, :hw]

    plane(lay.W_off, 1)[:] = rng.choice(np.float32([0.0, 0.5, 3.0, 40.0]), (1, hw))
    plane(lay.P_off, 1)[:] = rng.choice(np.float32([2.0 ** -64, 1.5 * 2.0 ** -64, 1e-3, 1.0]), (1, hw))
    plane(lay.key_off, K)[:] = rng.choice(
        np.float32([np.inf, 0.0, 1e-22, 1e-22, 3e-2, 3e-2, 5e30, 3.4028235e38]), (K, hw))
    return raw


@pytest.mark.parametrize("out", [True, False])
@pytest.mark.parametrize("bias", [0, 1, 2])
@pytest.mark.parametrize("K,rule,fp16", [(1, 0, False), (1, 1, False), (1, 1, True), (2, 0, True), (3, 0, False),
                                         (4, 0, True), (8, 0, False), (8, 0, True), (16, 0, True)])
def test_rare_branches_equal_the_plain_kernel(K, rule, fp16, bias, out):
    w, h = 132, 31
    rng = np.random.default_rng(K + 10 * bias)
    a, b = (wrs.Stream(w, h, K, 20.0, seed=5, color_fp16=fp16, temporal_bias=bias, update_rule=rule)
            for _ in range(2))
    b.set_pipeline(False)
    raw = _seeded_state(a, K, w * h, rng)
    outs = [torch.zeros((h, w, 3), device="cuda") for _ in range(2)]
    for st in (a, b):
        st.import_raw(raw, 7)
    for t in range(20):
        frame = torch.from_numpy(rng.random((h, w, 3), dtype=np.float32)).cuda()
        fm = torch.from_numpy(rng.choice(np.uint8([0, 3, 255]), (h, w), p=[0.6, 0.35, 0.05])).cuda() if t % 3 else None
        for st, o in zip((a, b), outs):
            st.push_frame(frame, (40.0 + t, 11.0), fov_map=fm, out=o if out else None)
    assert a.check_status() == 0 and b.check_status() == 0
    assert np.array_equal(a.export_raw()[256:], b.export_raw()[256:])
    assert a.replacements() == b.replacements()
    assert torch.equal(outs[0].view(torch.int32), outs[1].view(torch.int32))


@pytest.mark.parametrize("K,rule,fp16", [(1, 1, False), (2, 0, True), (4, 0, False), (5, 0, True), (8, 0, False)])
@pytest.mark.parametrize("wh", [(1, 1), (3, 1), (1, 7), (255, 1), (257, 1), (259, 3), (85, 6), (1365, 96), (134, 33)])
def test_any_width_equals_the_plain_kernel(wh, K, rule, fp16):
    """Widths not divisible by 4 (every remainder of the last tile and of the
    frame's last 16 bytes) through the pipelined kernel."""
    w, h = wh
    rng = np.random.default_rng(w + h)
    a, b = (wrs.Stream(w, h, K, 20.0, seed=6, color_fp16=fp16, update_rule=rule) for _ in range(2))
    b.set_pipeline(False)
    outs = [torch.full((h, w, 3), -1.0, device="cuda") for _ in range(2)]
    for t in range(18):
        frame = torch.from_numpy(rng.random((h, w, 3), dtype=np.float32)).cuda()
        fm = torch.from_numpy(rng.choice(np.uint8([0, 255]), (h, w), p=[0.9, 0.1])).cuda() if t % 4 == 3 else None
        for st, o in zip((a, b), outs):
            st.push_frame(frame, (0.4 * w, 0.6 * h), fov_map=fm, out=o)
    assert a.check_status() == 0
    x, y = a.export_state(), b.export_state()
    for plane in x:
        assert np.array_equal(x[plane].view(np.uint8), y[plane].view(np.uint8)), plane
    assert a.replacements() == b.replacements()
    assert torch.equal(outs[0].view(torch.int32), outs[1].view(torch.int32))


def test_captured_calls_equal_eager_calls():
    """Early launches and the tile queue inside a captured CUDA graph: foveate,
    push, push_foveated and a reprojected push, replayed once."""
    w, h, K = 1280, 720, 4
    rng = np.random.default_rng(3)
    img = torch.from_numpy(rng.random((h, w, 3), dtype=np.float32)).cuda()
    motion = torch.full((h, w, 2), 1.25, device="cuda")
    outs = []
    for captured in (False, True):
        st = wrs.Stream(w, h, K, 60.0, seed=9)
        st.set_reprojection_buffer()
        fov = wrs.Foveation(img, (60.0, 150.0, 300.0), filter="bilinear")
        frame, ring = torch.empty_like(img), torch.empty((h, w), dtype=torch.uint8, device="cuda")
        out = [torch.empty_like(img) for _ in range(3)]

        def calls():
            fov.rebuild()
            fov.frame((600.0, 300.0), out=frame, ring_map=ring)
            st.push_frame(frame, (600.0, 300.0), out=out[0])
            st.push_foveated(fov, (620.0, 310.0), out=out[1])
            st.push_frame_reproject(frame, (600.0, 300.0), motion, out=out[2])

        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                calls()
            g.replay()
        else:
            calls()
        torch.cuda.synchronize()
        assert st.check_status() == 0
        state = st.export_state()
        outs.append([frame, ring, *out, *(torch.from_numpy(np.ascontiguousarray(state[k]).view(np.uint8)) for k in state)])
    for a, b in zip(*outs):
        assert torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))


@pytest.mark.parametrize("foveated", [False, True])
@pytest.mark.parametrize("w,h,K,rule,fp16", [(1024, 516, 1, 1, True), (1024, 512, 1, 0, False), (1280, 772, 6, 0, True),
                                             (1600, 1028, 3, 0, False)])
def test_large_general_batches_equal_the_batched_kernel(w, h, K, rule, fp16, foveated):
    """Batches outside the K = 4 / 8 families whose streams are large enough for
    their own kernels (default launch shape) against the batched kernel (an
    explicit shape): mixed biases, a flush map and a missing output."""
    rng = np.random.default_rng(w + K)
    runs = []
    for shape in (None, (1, 1, 0, True)):
        streams = [wrs.Stream(w, h, K, 80.0, seed=4, stream_id=i, color_fp16=fp16, update_rule=rule,
                              temporal_bias=i % 3) for i in range(3)]
        b = wrs.Batch(3)
        if shape:
            b.set_launch(*shape)
        runs.append((streams, b, [torch.zeros((h, w, 3), device="cuda") for _ in range(3)]))
    for t in range(4):
        frames = [torch.from_numpy(rng.random((h, w, 3), dtype=np.float32)).cuda() for _ in range(3)]
        fov = torch.from_numpy(rng.choice(np.uint8([0, 255]), (h, w), p=[0.95, 0.05])).cuda()
        gazes = [(100.0 * i + t, 50.0 * i) for i in range(3)]
        sources = [wrs.Foveation(f, (80.0, 200.0, 400.0), filter="bilinear") for f in frames] if foveated else frames
        for streams, b, outs in runs:
            push = b.push_foveated if foveated else b.push
            push(streams, sources, gazes, fov_maps=[None, fov, None], outs=[outs[0], outs[1], None])
    for i in range(3):
        a, c = runs[0][0][i], runs[1][0][i]
        assert a.check_status() == 0 and c.check_status() == 0
        assert a.frame_index == c.frame_index == 4
        x, y = a.export_state(), c.export_state()
        for plane in x:
            assert np.array_equal(x[plane].view(np.uint8), y[plane].view(np.uint8)), (i, plane)
        assert a.replacements() == c.replacements()
        assert torch.equal(runs[0][2][i].view(torch.int32), runs[1][2][i].view(torch.int32))


def test_large_general_batches_take_streams_with_a_disabled_pipeline():
    """A shape set with the pipelined kernel disabled is not checked against shared memory; the
    batch, which always pipelines, takes the stream all the same."""
    w, h = 1024, 516
    shapes = [(True, 0, 0, 0), (False, 4, 8, 1), (False, 0, 0, 0)]
    streams = [wrs.Stream(w, h, 1, 80.0, seed=4, stream_id=i, update_rule=1) for i in range(3)]
    solo = [wrs.Stream(w, h, 1, 80.0, seed=4, stream_id=i, update_rule=1) for i in range(3)]
    for st, shape in zip(streams, shapes):
        st.set_pipeline(*shape)
    b = wrs.Batch(3)
    frames = [torch.rand((h, w, 3), device="cuda") for _ in range(3)]
    outs = [torch.empty_like(f) for f in frames]
    for t in range(2):
        b.push(streams, frames, [(100.0, 50.0 * t)] * 3, outs=outs)
        for st, f in zip(solo, frames):
            st.push_frame(f, (100.0, 50.0 * t))
    for a, c in zip(streams, solo):
        assert a.check_status() == 0 and a.frame_index == 2
        assert np.array_equal(a.export_raw()[256:], c.export_raw()[256:])


@pytest.mark.parametrize("captured", [False, True])
def test_large_general_batches_of_changing_streams(captured):
    """Rounds of changing number, order and kind of streams through one launcher (the graph of own
    kernels is updated or built anew), eagerly and inside a captured graph, against single pushes."""
    kinds = [(1280, 772, 1, 1, False), (1280, 772, 6, 0, True), (1600, 1028, 3, 0, True), (1024, 512, 16, 0, False)]
    mixed, solo = ([wrs.Stream(w, h, K, 60.0, seed=8, stream_id=i, color_fp16=f, update_rule=r)
                    for i, (w, h, K, r, f) in enumerate(kinds)] for _ in range(2))
    frames = [torch.rand((h, w, 3), device="cuda") for w, h, *_ in kinds]
    outs, single = ([torch.zeros_like(f) for f in frames] for _ in range(2))
    b = wrs.Batch(4)
    for t, members in enumerate(([0, 1, 2], [0, 1, 2], [2, 0, 1], [1, 2], [3, 2, 1, 0], [2], [0, 1, 2])):
        def push():
            b.push([mixed[i] for i in members], [frames[i] for i in members],
                   [(30.0 * t, 40.0 * i) for i in members], outs=[outs[i] for i in members])

        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                push()
            g.replay()
            torch.cuda.synchronize()
        else:
            push()
        for i in members:
            solo[i].push_frame(frames[i], (30.0 * t, 40.0 * i), out=single[i])
    for i, (a, c) in enumerate(zip(mixed, solo)):
        assert a.check_status() == 0 and c.check_status() == 0 and a.frame_index == c.frame_index
        assert a.replacements() == c.replacements()
        assert np.array_equal(a.export_raw()[256:], c.export_raw()[256:]), i
        assert torch.equal(outs[i].view(torch.int32), single[i].view(torch.int32)), i


@pytest.mark.parametrize("wh,K,rule,fp16,bias,shape", [
    ((1365, 767), 1, 1, False, 1, None), ((1365, 767), 4, 0, False, 2, None), ((1365, 767), 6, 0, True, 1, None),
    ((2064, 1104), 1, 0, True, 2, None), ((2064, 1104), 2, 0, False, 1, None), ((2064, 1104), 4, 0, True, 1, None),
    ((2064, 1104), 8, 0, True, 2, None), ((2064, 1104), 8, 0, False, 1, None), ((2064, 1104), 3, 0, False, 2, None),
    ((2064, 1104), 1, 1, True, 2, None), ((1364, 768), 5, 0, False, 1, (1, 1, 1)), ((1364, 768), 8, 0, True, 1, (1, 2, 1)),
    ((1364, 768), 4, 0, False, 2, (1, 8, 1)), ((2064, 1104), 2, 0, True, 1, (4, 2, 1)), ((2064, 1104), 16, 0, True, 1, None),
])
def test_refilled_stages_equal_the_plain_kernel(wh, K, rule, fp16, bias, shape):
    """Seven to 29 tiles per CTA (152 to 456 CTAs, 256 to 1,024 pixels per tile): the stages are
    refilled after their columns were written (flushes, rescales, replaced slots), and the queue's
    answers wrap around. Some colours are infinite, NaN or beyond FP16."""
    w, h = wh
    rng = np.random.default_rng(K + 10 * bias)
    gen = torch.Generator(device="cuda").manual_seed(K)
    a, b = (wrs.Stream(w, h, K, 60.0, seed=5, color_fp16=fp16, temporal_bias=bias, update_rule=rule) for _ in range(2))
    b.set_pipeline(False)
    if shape:
        a.set_pipeline(True, *shape)
    raw = _seeded_state(a, K, w * h, rng)
    outs = [torch.zeros((h, w, 3), device="cuda") for _ in range(2)]
    for st in (a, b):
        st.import_raw(raw, 7)
    odd = torch.tensor([float("inf"), -float("inf"), float("nan"), 1e6, -0.0, 3e38], device="cuda")
    for t in range(18):
        frame = torch.rand((h, w, 3), device="cuda", generator=gen)
        at = torch.randint(0, frame.numel(), (200,), device="cuda", generator=gen)
        frame.view(-1)[at] = odd[torch.randint(0, len(odd), (200,), device="cuda", generator=gen)]
        fm = torch.where(torch.rand((h, w), device="cuda", generator=gen) < 0.2, 255, 3).to(torch.uint8) if t % 3 else None
        for st, o in zip((a, b), outs):
            st.push_frame(frame, (400.0 + 9 * t, 311.0), fov_map=fm, out=o)
        assert torch.equal(outs[0].view(torch.int32), outs[1].view(torch.int32)), t
    assert a.check_status() == 0 and b.check_status() == 0
    assert np.array_equal(a.export_raw()[256:], b.export_raw()[256:])
    assert a.replacements() == b.replacements()
