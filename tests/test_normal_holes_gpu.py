"""The normal field's unmasked sums (warps whose patch rows hold no invalid
range) against the normals pc_compute starts from: the same bits with single
holes on every edge of a tile, spread over the image, none at all, and images
smaller than a patch; every patch radius beside the unrolled one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("H,W", [(1, 1), (6, 40), (7, 7), (38, 70), (33, 97), (480, 640), (1201, 1603)])
@pytest.mark.parametrize("holes", ["none", "edges", "row", "spread"])
@pytest.mark.parametrize("rn", [3, 1, 5])
def test_bits_of_the_full_method(gpu, H, W, holes, rn):
    import torch
    rng = np.random.default_rng(H * 10007 + W)
    v, u = np.mgrid[0:H, 0:W]
    z = (1.0 + 2e-4 * u - 1e-4 * v + 0.01 * np.sin(u / 9.0) + rng.normal(0, 5e-4, (H, W))).astype(np.float32)
    if holes == "edges":  # one hole at and beside each edge of the 32-column tiles and of every eighth row
        for k, (dv, du) in enumerate([(-1, -1), (0, 0), (-1, 31), (3, 34), (4, -4)]):
            z[(16 * k + 8 + dv)::80, (32 + du)::96] = [0.0, np.nan, -1.0, np.inf, 0.0][k]
    elif holes == "row":
        z[H // 2] = 0.0
    elif holes == "spread":
        z[rng.random((H, W)) < 0.02] = 0.0
    f = 525.0 * max(W, 64) / 640.0
    c = gpu.Curvature(f, f, (W - 1) / 2.0, (H - 1) / 2.0, window_radius=7, iterations=0, min_window=6, normal_radius=rn)
    d = torch.from_numpy(z).cuda()
    got = c.initial_normals(d).cpu().numpy()
    want = c(d)[2].cpu().numpy()
    c.close()
    # a normal wherever the centre has a range and its patch points to fit a plane
    # to, none without a range at the centre or with fewer than three points
    valid = np.isfinite(z) & (z > 0)
    padded = np.pad(valid, rn)
    points = sum(padded[j:j + H, i:i + W].astype(int) for j in range(2 * rn + 1) for i in range(2 * rn + 1))
    n = ~np.isnan(got)
    assert (n.all(-1) == n.any(-1)).all()
    assert not n[~valid | (points < 3)].any()
    assert n[valid & (points >= 8)].all()
    m = ~np.isnan(want)
    assert np.array_equal(got[m], want[m])
    if H >= 16 and W >= 16 and holes != "row":
        assert m.mean() > 0.9
