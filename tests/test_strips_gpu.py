"""Ragged widths: the 16- and 8-pixel strips at the right edge against lane
groups' 32-pixel columns are another order of sums, so the check is on the
bits of what has no strips: the same pixels inside a wider image whose width
fills its columns.  A pixel whose window ends before the cut sees the same
points in both; frames alone, in a batch and from host memory agree."""
import numpy as np
import pytest

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


def surface(H, W):
    rng = np.random.default_rng(H * 4099 + W)
    v, u = np.mgrid[0:H, 0:W]
    z = (1.0 + 3e-4 * u - 2e-4 * v + 0.01 * np.sin(u / 11.0) * np.cos(v / 7.0) + rng.normal(0, 4e-4, (H, W)))
    z[rng.random((H, W)) < 0.02] = 0.0
    return z.astype(np.float32)


# remainders of the width: one strip of 8, of 16, both, and the column kept; rows below, at and above the strips' tiles
@pytest.mark.parametrize("rem", [1, 8, 9, 16, 17, 24, 25, 31])
@pytest.mark.parametrize("H,th", [(5, 0), (31, 8), (33, 4), (72, 0)])
@pytest.mark.parametrize("r,kw", [(3, {}), (7, {}), (12, {"stride": 2}), (14, {})])
def test_same_bits_as_a_width_without_strips(gpu, rem, H, th, r, kw):
    import torch
    W = 64 + rem
    z = surface(H, W)
    wide = np.zeros((H, 96), np.float32)      # no range beyond the cut: what lies outside the narrow image
    wide[:, :W] = z
    c = gpu.Curvature(525.0, 525.0, 40.0, H / 2.0, window_radius=r, iterations=3, tile_height=th, **kw)
    d = torch.from_numpy(z).cuda()
    got = [t.cpu().numpy() for t in c(d)]
    want = [t.cpu().numpy()[:, :W] for t in c(torch.from_numpy(wide).cuda())]
    outs = [torch.full_like(d, 7.0), torch.full_like(d, 7.0), torch.full(d.shape + (3,), 7.0, device="cuda")]
    c.batch([(d, (525.0, 525.0, 40.0, H / 2.0), *outs)])
    host = [torch.full((H, W), 7.0).pin_memory(), torch.full((H, W), 7.0).pin_memory(), torch.full((H, W, 3), 7.0).pin_memory()]
    c.compute_host(torch.from_numpy(z).pin_memory(), *host)
    torch.cuda.synchronize()
    c.close()
    for a, b, o, h in zip(got, want, outs, host):
        assert np.array_equal(a, b, equal_nan=True)
        assert np.array_equal(a, o.cpu().numpy(), equal_nan=True)
        assert np.array_equal(a, h.numpy(), equal_nan=True)


# the windows that leave strips out where those save no step of an SM (33 rows), and take them where they do (2000)
@pytest.mark.parametrize("H", [33, 2000])
@pytest.mark.parametrize("rem", [3, 20])
@pytest.mark.parametrize("r,kw", [(1, {}), (1, {"reject": 1}), (6, {}), (18, {"stride": 3}), (5, {"kahan": 1}),
                                  (5, {"kahan": 1, "reject": 1})])
def test_strips_left_out_or_taken(gpu, rem, H, r, kw):
    import torch
    W = 32 + rem
    z = surface(H, W)
    c = gpu.Curvature(525.0, 525.0, 20.0, H / 2.0, window_radius=r, iterations=3, **kw)
    d = torch.from_numpy(z).cuda()
    wide = np.zeros((H, 64), np.float32)
    wide[:, :W] = z
    got = [t.cpu().numpy() for t in c(d)]
    want = [t.cpu().numpy()[:, :W] for t in c(torch.from_numpy(wide).cuda())]
    c.close()
    for a, b in zip(got, want):
        assert np.array_equal(a, b, equal_nan=True)
