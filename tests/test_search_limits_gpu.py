"""Searches that may not fall back on the exact scan (exhaustive = 0): what
max_box_cells lets through does not depend on the widths chosen for speed."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F = np.float32


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def lattice(nx, ny, nz):
    g = np.stack(np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"), -1)
    return g.reshape(-1, 3).astype(F)


# ---------------------------------------------------------------- GICP
def pairs(t, mp, src, max_dist):
    eye = np.tile(np.array([1, 0, 0, 1, 0, 1], F), (max(len(mp), len(src)), 1))
    corr = torch.full((len(src),), -2, dtype=torch.int32, device="cuda")
    pose = dev(np.concatenate([np.eye(3).ravel(), np.zeros(3)]).astype(F))
    t.gicp_linearize(dev(eye[:len(mp)]), dev(src), dev(eye[:len(src)]), pose, max_dist, corr=corr)
    return corr.cpu().numpy()


@pytest.mark.parametrize("appended", [False, True])
def test_gicp_boxes_over_the_limit_start_again(gpu_lib, appended):
    """Lattice of spacing 1 in cells of 0.25: a box of the 2nd neighbour's radius (0.9) has at most 9^3 cells, one of
    the 8th's (1.27) at least 11^3.  With a limit between the two, no point needs the scan of the whole map."""
    mp = lattice(16, 16, 16)
    half = len(mp) // 2 if appended else len(mp)
    t = gpu_lib.Target(dev(mp[:half]), cell_size=0.25, max_box_cells=1000)
    if appended:
        t.append(dev(mp[half:]))
    np.testing.assert_array_equal(pairs(t, mp, mp + F(0.05), 0.5), np.arange(len(mp)))
    assert t.sync_status() == gpu_lib.PC_OK
    assert t.stats()["exhaustive"] == 0
    t.close()


def clusters(seed, n):
    """40 tight clusters, and n queries from 1 cm to 10 m off them."""
    g = np.random.default_rng(seed)
    c = g.random((40, 3)) * [60, 60, 6]
    mp = (c[g.integers(0, 40, 8000)] + 0.05 * g.standard_normal((8000, 3))).astype(F)
    s = 10.0 ** g.uniform(-2, 1.0, (n, 1))
    return mp, (mp[g.integers(0, 8000, n)] + s * g.standard_normal((n, 3))).astype(F)


def boxes(info, q, r):
    """Cells and rows of the box of half-width r around each query, clamped to the grid."""
    o, h, dim = np.array(info["origin"]), info["cell_size"], np.array(info["dims"])
    lo = np.maximum(np.floor((q - r - o) / h), 0)
    hi = np.minimum(np.floor((q + r - o) / h), dim - 1)
    e = np.maximum(hi - lo + 1, 0)
    return e.prod(1), e[:, 1] * e[:, 2]


@pytest.mark.parametrize("cells", [27, 64, 512])
def test_gicp_reach(gpu_lib, cells):
    """A source point is paired when some radius r 2^j, r the calibrated 2nd-neighbour radius, holds its nearest point
    in a box within the limit."""
    mp, src = clusters(cells, 3000)
    t = gpu_lib.Target(dev(mp), cell_size=1.0, max_box_cells=cells, exhaustive=False)
    info = t.info()
    d = np.sqrt(oracle.knn_brute(src, mp, 1)[1][:, 0])
    r = 0.9 * info["rho_hint"][1] if info["rho_hint"][1] > 0 else 0.9 * info["cell_size"]
    must = np.zeros(len(src), bool)
    for j in range(16):
        must |= (boxes(info, src.astype(np.float64), r * 2 ** j)[0] <= cells) & (d < 0.999 * r * 2 ** j)
    corr = pairs(t, mp, src, float("inf"))
    t.sync_status()
    t.close()
    assert must.sum() > 300
    assert (corr[must] >= 0).all()
    np.testing.assert_array_equal(corr[corr >= 0], oracle.knn_brute(src, mp, 1)[0][corr >= 0, 0])
