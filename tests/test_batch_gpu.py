"""pc_compute_batch: uneven frames in one persistent launch over a flattened
tile queue equal pc_compute frame by frame, bit for bit, with and without
the CUDA graph, across repeated calls and capacity growth."""
import json

import numpy as np
import pytest

import synth

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_00385_gb300 import build
    build.build()
    import paper_1707_00385_gb300 as pc
    pc.load()
    return pc


SIZES = [(240, 320), (424, 512), (480, 640), (720, 1280), (37, 45), (8, 32), (1, 1)]


@pytest.fixture(scope="module")
def frames():
    out = []
    for i, (H, W) in enumerate(SIZES * 2):
        s = synth.kinect_scene(100 + i, H=H, W=W, noise="tof" if (H, W) == (424, 512) else "kinect",
                               nprims=6) if H >= 100 else \
            synth.crop(synth.kinect_scene(100 + i), 200, 300, H, W)
        out.append(s)
    return out


def per_frame(pc, scenes, r, T, **kw):
    import torch
    res = []
    for s in scenes:
        c = pc.Curvature(*s.intrinsics, window_radius=r, iterations=T, **kw)
        k1, k2, n = c(torch.from_numpy(s.depth).cuda())
        torch.cuda.synchronize()
        res.append((k1.cpu().numpy(), k2.cpu().numpy(), n.cpu().numpy()))
        c.close()
    return res


def batched(pc, c, scenes, with_normal=True):
    import torch
    args, outs = [], []
    for s in scenes:
        d = torch.from_numpy(s.depth).cuda()
        k1, k2 = torch.full(d.shape, 5.0, device="cuda"), torch.full(d.shape, 5.0, device="cuda")
        n = torch.full(d.shape + (3,), 5.0, device="cuda") if with_normal else None
        args.append((d, s.intrinsics, k1, k2, n))
        outs.append((k1, k2, n))
    c.batch(args)
    torch.cuda.synchronize()
    return [(a.cpu().numpy(), b.cpu().numpy(), n.cpu().numpy() if n is not None else None)
            for a, b, n in outs]


def same(a, b):
    return np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("graph", [1, 0])
def test_batch_equals_per_frame(gpu, frames, graph):
    ref = per_frame(gpu, frames, 7, 5)
    c = gpu.Curvature(525.0, 525.0, 0.0, 0.0, window_radius=7, iterations=5, batch_graph=graph)
    got = batched(gpu, c, frames)
    c.close()
    for (a1, a2, an), (b1, b2, bn) in zip(ref, got):
        assert same(a1, b1) and same(a2, b2) and same(an, bn)


def test_repeated_calls_growth_and_alternation(gpu, frames):
    """Several calls in a row on one context: small, large (capacity grows,
    graphs are recaptured), small again; both staging copies get reused."""
    import torch
    ref = per_frame(gpu, frames, 5, 3)
    c = gpu.Curvature(525.0, 525.0, 0.0, 0.0, window_radius=5, iterations=3)
    plan = [frames[:3], frames, frames[3:6], frames[:1], frames[2:14], frames[:3]]
    idx = [list(range(3)), list(range(len(frames))), [3, 4, 5], [0], list(range(2, 14)), [0, 1, 2]]
    for sel, ids in zip(plan, idx):
        got = batched(gpu, c, sel)
        for i, (b1, b2, bn) in zip(ids, got):
            a1, a2, an = ref[i]
            assert same(a1, b1) and same(a2, b2) and same(an, bn)
    c.close()
    torch.cuda.synchronize()


def test_batch_skips_empty_frames_and_normals_optional(gpu, frames):
    import torch
    c = gpu.Curvature(525.0, 525.0, 0.0, 0.0, window_radius=3, iterations=2)
    ref = per_frame(gpu, frames[:3], 3, 2)
    empty = torch.zeros((0, 7), device="cuda")
    e1, e2 = torch.zeros((0, 7), device="cuda"), torch.zeros((0, 7), device="cuda")
    args = []
    outs = []
    for s in frames[:3]:
        d = torch.from_numpy(s.depth).cuda()
        k1, k2 = torch.empty(d.shape, device="cuda"), torch.empty(d.shape, device="cuda")
        args.append((d, s.intrinsics, k1, k2, None))
        outs.append((k1, k2))
        args.append((empty, (1.0, 1.0, 0.0, 0.0), e1, e2, None))
    c.batch(args)
    torch.cuda.synchronize()
    for (k1, k2), (a1, a2, _) in zip(outs, ref):
        assert same(k1.cpu().numpy(), a1) and same(k2.cpu().numpy(), a2)
    c.batch([])   # nothing to do
    c.close()


def test_batch_runtime_radius_and_stride(gpu, frames):
    sel = [frames[0], frames[4], frames[1]]
    for kw in ({"window_radius": 15}, {"window_radius": 9, "stride": 3}):
        r = kw.pop("window_radius")
        ref = per_frame(gpu, sel, r, 3, **kw)
        c = gpu.Curvature(525.0, 525.0, 0.0, 0.0, window_radius=r, iterations=3, **kw)
        got = batched(gpu, c, sel)
        c.close()
        for (a1, a2, an), (b1, b2, bn) in zip(ref, got):
            assert same(a1, b1) and same(a2, b2) and same(an, bn)


def test_batched_frame_against_oracle(gpu, orc, frames):
    """One frame of a batch checked directly against the oracle."""
    from oracle import parity
    s = synth.crop(frames[2], 150, 250, 60, 90)
    c = gpu.Curvature(*s.intrinsics, window_radius=7, iterations=5)
    (k1, k2, n), = batched(gpu, c, [s])
    c.close()
    ref = parity.reference(s.depth, orc.params(*s.intrinsics, r=7, T=5, pivot_tol=1e-5))
    rep = parity.compare(k1, k2, n, ref, pivot_tol=1e-5)
    assert rep.ok() and rep.n_well_posed > 0.3 * rep.n_valid_oracle, rep.summary()
    assert rep.frac_within_tol_all > 0.9, rep.summary()


def test_benchmark_launch_sampled_against_oracle(gpu, orc):
    """The benchmark's own launch: 128 distinct 640 x 480 frame buffers (8
    seeded scenes) in one persistent launch at r = 7, T = 5; pixels sampled
    from four frames (random ones plus a whole corner tile) against the oracle."""
    import torch
    import bench
    from oracle import parity
    sc = bench.scenes(8)
    F = 128
    dev = [torch.from_numpy(sc[i % 8].depth).cuda() for i in range(F)]
    outs = [(torch.empty(480, 640, device="cuda"), torch.empty(480, 640, device="cuda"),
             torch.empty(480, 640, 3, device="cuda")) for _ in range(F)]
    c = gpu.Curvature(*sc[0].intrinsics, window_radius=bench.RADIUS, iterations=bench.ITERS)
    c.batch([(dev[i], sc[i % 8].intrinsics) + outs[i] for i in range(F)])
    torch.cuda.synchronize()
    c.close()
    rng = np.random.default_rng(17)
    corner = np.stack(np.meshgrid(np.arange(608, 640), np.arange(472, 480)), -1).reshape(-1, 2)
    for f in (0, 37, 90, 127):
        s = sc[f % 8]
        uv = np.concatenate([np.stack([rng.integers(0, 640, 400), rng.integers(0, 480, 400)], 1), corner])
        uv = uv.astype(np.int32)
        k1, k2, n = (t.cpu().numpy() for t in outs[f])
        ref = parity.reference(s.depth, orc.params(*s.intrinsics, r=bench.RADIUS, T=bench.ITERS,
                                                   pivot_tol=1e-5), uv=uv)
        rep = parity.compare(k1[uv[:, 1], uv[:, 0]], k2[uv[:, 1], uv[:, 0]], n[uv[:, 1], uv[:, 0]], ref,
                             pivot_tol=1e-5)
        print(f, rep.summary())
        print("PARITY_ROW " + json.dumps({"case": f"benchmark launch frame {f}", **rep.row()}))
        # sampled frames gate 0.49-0.75 of their pixels and have 0.917-0.959 of
        # them within tolerance (GB300)
        assert rep.ok() and rep.n_well_posed > 0.45 * rep.n_valid_oracle, rep.summary()
        assert rep.frac_within_tol_all > 0.90, rep.summary()
        # at least as many as the oracle with single-precision sums (GB300: 0.007-0.010 more)
        assert rep.frac_within_tol_all >= rep.frac_within_tol_f32_sums - 0.005, rep.summary()


def test_largest_batch(gpu):
    """PC_MAX_BATCH frames in one call: four small crops of different sizes
    and principal points, repeated; every frame equals its crop computed
    alone, for the FP32 batch and the 16-bit storage batch."""
    import torch
    k = synth.kinect_scene(7)
    crops = [synth.crop(k, 200, 300, H, W) for H, W in [(1, 1), (9, 33), (8, 32), (13, 17)]]
    n = gpu.pcurv.PC_MAX_BATCH
    c = gpu.Curvature(*crops[0].intrinsics, window_radius=7, iterations=5)
    ref = per_frame(gpu, crops, 7, 5)
    sizes = [crops[i % 4].depth.size for i in range(n)]
    offs = np.concatenate([[0], np.cumsum(sizes)])
    k1, k2 = torch.full((int(offs[-1]),), 5.0, device="cuda"), torch.full((int(offs[-1]),), 5.0, device="cuda")
    nrm = torch.full((3 * int(offs[-1]),), 5.0, device="cuda")
    depth = [torch.from_numpy(s.depth).cuda() for s in crops]

    def views(i):
        H, W = crops[i % 4].depth.shape
        a, b = int(offs[i]), int(offs[i + 1])
        return k1[a:b].view(H, W), k2[a:b].view(H, W), nrm[3 * a:3 * b].view(H, W, 3)

    def check(ref):
        torch.cuda.synchronize()
        h1, h2, hn = k1.cpu().numpy(), k2.cpu().numpy(), nrm.cpu().numpy()
        for i in range(n):
            a1, a2, an = ref[i % 4]
            a, b = int(offs[i]), int(offs[i + 1])
            assert same(a1.ravel(), h1[a:b]) and same(a2.ravel(), h2[a:b]) and same(an.ravel(), hn[3 * a:3 * b]), i

    c.batch([(depth[i % 4], crops[i % 4].intrinsics, *views(i)) for i in range(n)])
    check(ref)
    for fmt in (1, 2):
        packed = [c.pack(d, fmt) for d in depth]
        ref = []
        for s, (q, b) in zip(crops, packed):
            cs = gpu.Curvature(*s.intrinsics, window_radius=7, iterations=5)
            ref.append(tuple(x.cpu().numpy() for x in cs.compute_packed(q, b, fmt)))
            cs.close()
        k1.fill_(5.0), k2.fill_(5.0), nrm.fill_(5.0)
        c.batch_packed([(*packed[i % 4], crops[i % 4].intrinsics, *views(i)) for i in range(n)], fmt)
        check(ref)
    c.close()


# queues of one tile, of about one and eight tiles per CTA of the persistent grid and more, without strips and with
@pytest.mark.parametrize("n,H,W", [(1, 4, 32), (1, 48, 64), (2, 480, 640), (3, 480, 640), (2, 241, 323)])
@pytest.mark.parametrize("r,kw", [(6, {}), (9, {}), (12, {"reject": 1}), (18, {"stride": 3}), (18, {"stride": 3, "reject": 1}),
                                  (14, {}), (9, {"tile_height": 4})])
def test_short_and_long_queues_equal_per_frame(gpu, n, H, W, r, kw):
    s = synth.kinect_scene(31)
    scenes = [synth.kinect_scene(31 + i, H=H, W=W) if H >= 200 else synth.crop(s, 100 + i, 120, H, W) for i in range(n)]
    c = gpu.Curvature(525.0, 525.0, 0.0, 0.0, window_radius=r, iterations=2, **kw)
    for want, got in zip(per_frame(gpu, scenes, r, 2, **kw), batched(gpu, c, scenes)):
        for a, b in zip(want, got):
            assert same(a, b)
    c.close()


def test_alternating_tile_heights_do_not_capture_anew(gpu):
    """Two batches that take different tile heights, in turn: the results of
    each alone, and a call takes no more than twice the host time it takes when
    one batch is repeated (12 us; a capture on every change makes it 33)."""
    import time
    import torch
    c = gpu.Curvature(525.0, 525.0, 320.0, 240.0, window_radius=5, iterations=5)
    scenes = [synth.kinect_scene(7, H=480, W=640), synth.kinect_scene(8, H=330, W=640)]
    if c.tile_height(480, 640) == c.tile_height(330, 640):
        pytest.skip("one tile height serves both on this device")
    batches, want = [], []
    for s in scenes:
        d = torch.from_numpy(s.depth).cuda()
        batches.append([(d, s.intrinsics, torch.full_like(d, 5.0), torch.full_like(d, 5.0),
                         torch.full(d.shape + (3,), 5.0, device="cuda"))])
        one = gpu.Curvature(*s.intrinsics, window_radius=5, iterations=5)
        want.append([t.cpu().numpy() for t in one(d)])
        one.close()

    def host_us(order):
        ts = []
        for k in range(80):
            for i in order:
                t0 = time.perf_counter()
                c.batch(batches[i])
                t1 = time.perf_counter()
                torch.cuda.synchronize()
                if k >= 20:
                    ts.append(t1 - t0)
        return 1e6 * float(np.median(ts))

    # the median of 60 rounds; a busy host may still disturb one try
    tries = [(max(host_us([0]), host_us([1])), host_us([0, 0, 1, 1])) for _ in range(3)]
    print("host us a call, repeated and in turn:", tries)
    for b, w in zip(batches, want):
        for t, x in zip(b[0][2:], w):
            assert same(t.cpu().numpy(), x)
    c.close()
    assert any(turn <= 2 * alone for alone, turn in tries), tries
