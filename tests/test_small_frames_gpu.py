"""Frames of at most one 32 x 4 tile per SM, which run the per-frame kernel with
room for more registers: the bits of the batch kernel, at one tile, around one
tile per SM and beyond it, with and without strips, autotuned and forced."""
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
def scene():
    return synth.kinect_scene(31)


@pytest.mark.parametrize("H,W", [(1, 1), (48, 64), (82, 109), (120, 160), (121, 161), (150, 165)])
@pytest.mark.parametrize("r,kw", [(3, {}), (4, {}), (5, {}), (7, {}), (12, {}), (18, {"stride": 3}), (7, {"reject": 1}),
                                  (6, {"tile_height": 4})])
def test_bits_of_the_batch_kernel(gpu, scene, H, W, r, kw):
    import torch
    s = synth.crop(scene, 100, 120, H, W)
    d = torch.from_numpy(s.depth).cuda()
    c = gpu.Curvature(*s.intrinsics, window_radius=r, iterations=4, **kw)
    got = [t.cpu().numpy() for t in c(d)]
    outs = [torch.full_like(d, 7.0), torch.full_like(d, 7.0), torch.full(d.shape + (3,), 7.0, device="cuda")]
    c.batch([(d, s.intrinsics, *outs)])
    torch.cuda.synchronize()
    c.close()
    for a, b in zip(got, outs):
        assert np.array_equal(a, b.cpu().numpy(), equal_nan=True)
