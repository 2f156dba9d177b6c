"""16-bit range storage at every unrolled window radius and beyond, both
formats through the one kernel that reads them: the bits of the float32 path on
the decoded ranges."""
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


@pytest.mark.parametrize("fmt", [1, 2])
@pytest.mark.parametrize("r,kw", [(1, {}), (2, {}), (4, {}), (6, {}), (8, {}), (9, {}), (10, {}), (12, {}), (13, {}),
                                  (18, {"stride": 3}), (8, {"reject": 1}), (4, {"kahan": 1}), (6, {"kahan": 1})])
def test_bits_of_the_float32_path(gpu, fmt, r, kw):
    import torch
    s = synth.crop(synth.kinect_scene(31), 90, 110, 45, 83)
    c = gpu.Curvature(*s.intrinsics, window_radius=r, iterations=3, **kw)
    d = torch.from_numpy(s.depth).cuda()
    q, base = c.pack(d, fmt)
    got = [t.cpu().numpy() for t in c.compute_packed(q, base, fmt)]
    off = q.view(torch.float16 if fmt == 1 else torch.bfloat16).float()
    H, W = d.shape
    dec = off + base.repeat_interleave(8, 0).repeat_interleave(32, 1)[:H, :W]
    dec = torch.where(torch.isfinite(dec), dec, torch.zeros_like(dec)).contiguous()
    want = [t.cpu().numpy() for t in c(dec)]
    c.close()
    for a, b in zip(got, want):
        assert np.array_equal(a, b, equal_nan=True)
