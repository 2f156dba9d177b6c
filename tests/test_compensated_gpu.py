"""Compensated sums (kahan = 1, every term of all 26 window sums compensated):
parity over small and large windows, a strided window, the rejection filter, a
batch; the same bits at every radius for the same points; and a gain over plain
sums that plain sums would not pass."""
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


@pytest.fixture(scope="module")
def crop():
    return synth.crop(synth.kinect_scene(21), 200, 260, 43, 77)


def run(gpu, s, r, T, **kw):
    import torch
    c = gpu.Curvature(*s.intrinsics, window_radius=r, iterations=T, **kw)
    out = [t.cpu().numpy() for t in c(torch.from_numpy(s.depth).cuda())]
    c.close()
    return out


@pytest.mark.parametrize("r,kw", [(4, {}), (5, {}), (8, {}), (18, {"stride": 3}), (24, {}), (6, {"reject": 1}),
                                  (7, {"fp64_solve_cond": 1e6})])
def test_against_oracle(gpu, orc, crop, r, kw):
    from oracle import parity
    p = orc.params(*crop.intrinsics, r=r, T=5, pivot_tol=1e-5, **{k: v for k, v in kw.items() if k != "fp64_solve_cond"})
    ref = parity.reference(crop.depth, p, nthreads=0)
    plain = parity.compare(*run(gpu, crop, r, 5, **kw), ref, pivot_tol=1e-5)
    comp = parity.compare(*run(gpu, crop, r, 5, kahan=1, **kw), ref, pivot_tol=1e-5)
    print(r, kw, "plain:", plain.summary(), "compensated:", comp.summary())
    assert comp.n_well_posed_bad == 0 and comp.nan_pattern_ok, comp.summary()
    assert comp.frac_within_tol_all >= plain.frac_within_tol_all - 0.005


@pytest.mark.parametrize("r", [4, 5, 11])
@pytest.mark.parametrize("fmt", [0, 1, 2])
def test_batch_equals_frame(gpu, crop, r, fmt):
    import torch
    views = [crop, synth.crop(crop, 3, 5, 9, 41), synth.crop(crop, 0, 0, 33, 32)]
    c = gpu.Curvature(*crop.intrinsics, window_radius=r, iterations=3, kahan=1)
    frames, want = [], []
    for v in views:
        d = torch.from_numpy(v.depth).cuda()
        one = gpu.Curvature(*v.intrinsics, window_radius=r, iterations=3, kahan=1)
        src = c.pack(d, fmt) if fmt else (d,)
        want.append([t.cpu().numpy() for t in (one.compute_packed(*src, fmt) if fmt else one(d))])
        one.close()
        frames.append((*src, v.intrinsics, torch.full_like(d, 7.0), torch.full_like(d, 7.0),
                       torch.full(d.shape + (3,), 7.0, device="cuda")))
    c.batch_packed(frames, fmt) if fmt else c.batch(frames)
    torch.cuda.synchronize()
    c.close()
    for f, w in zip(frames, want):
        for a, b in zip(f[-3:], w):
            assert np.array_equal(a.cpu().numpy(), b, equal_nan=True)


@pytest.mark.parametrize("fmt", [0, 1, 2])
def test_same_points_give_the_same_bits_at_every_radius(gpu, fmt):
    """9 x 9 patches with a range, seen from their centres: every window of
    radius 4 and more holds the same points in the same order, with terms of
    weight 0 between them.  A compensated sum stays as it is when 0 is added,
    unless its lost part is above half a unit in the last place (a sum just at a
    power of two, or one smaller than a term before it), so the radii agree in
    nearly every bit; a sum that is compensated once for several terms depends on
    where the window's columns are cut."""
    import torch
    rng = np.random.default_rng(5)
    H, W, step = 255, 340, 17
    v, u = np.mgrid[0:H, 0:W]
    z = (1.0 + 4e-4 * u - 3e-4 * v + 2e-5 * (u % step - 8.0) ** 2 + rng.normal(0, 3e-4, (H, W))).astype(np.float32)
    z[(abs(u % step - 8) > 4) | (abs(v % step - 8) > 4)] = 0.0
    centres = []
    for r in (4, 5, 6, 7, 9, 11, 12):
        c = gpu.Curvature(525.0, 525.0, W / 2.0, H / 2.0, window_radius=r, iterations=4, kahan=1)
        d = torch.from_numpy(z).cuda()
        out = c.compute_packed(*c.pack(d, fmt), fmt) if fmt else c(d)
        centres.append([t.cpu().numpy()[8::step, 8::step] for t in out])
        c.close()
    assert np.isfinite(centres[0][0]).all()
    for r, got in zip((5, 6, 7, 9, 11, 12), centres[1:]):
        same = [float((a == b).mean()) for a, b in zip(got, centres[0])]
        print("radius", r, "same bits as radius 4:", same)
        assert min(same) >= 0.9, r


@pytest.mark.parametrize("r,gap", [(7, 0.0127), (11, 0.0198)])
def test_more_accurate_than_plain_sums(gpu, orc, r, gap):
    """A whole 640 x 480 frame against the oracle (GB300): plain sums reach 0.9399
    (r = 7) and 0.9110 (r = 11) within tolerance and differ from it in the
    validity of 331 and 389 pixels, compensated sums 0.9526 and 0.9308 with 121
    and 143.  Asked for: half of the gap in the first, two thirds of plain sums'
    number in the second, so that plain sums fail both."""
    import bench
    s = bench.scenes(1)[0]
    ref = orc.curvature_image(s.depth, orc.params(*s.intrinsics, r=r, T=5, pivot_tol=1e-5))
    ok = ref.status == orc.OK
    share, lost = {}, {}
    for kahan in (0, 1):
        k1, k2, _ = run(gpu, s, r, 5, kahan=kahan)
        both = ok & np.isfinite(k1)
        within = (np.abs(k1 - ref.k1) <= 1e-4 + 1e-4 * np.abs(ref.k1)) & (np.abs(k2 - ref.k2) <= 1e-4 + 1e-4 * np.abs(ref.k2))
        share[kahan], lost[kahan] = within[both].mean(), int(np.sum(ok != np.isfinite(k1)))
    print(r, "within tolerance plain %.5f compensated %.5f, validity %d %d" % (share[0], share[1], lost[0], lost[1]))
    assert share[1] >= share[0] + gap / 2
    assert lost[1] <= lost[0] * 2 / 3
