"""Block-wise compensated sums (kahan = 1 from 5 samples to each side) at the
edges of their range: the smallest window that takes them and the largest that
does not, columns in one, two and seven blocks, a strided window, the rejection
filter, 16-bit storage, ragged widths and rows, batches.  The parity rule is
that of every other kernel; the pixels within tolerance are at least those of
plain sums, up to the 0.005 that reordered single-precision sums differ by."""
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
