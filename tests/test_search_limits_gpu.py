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


@pytest.mark.parametrize("max_dist", [0.0, 1e-30, 1e-3, 1.0])
@pytest.mark.parametrize("exhaustive", [False, True])
def test_gicp_max_dist_of_nothing(gpu_lib, exhaustive, max_dist):
    """A map and a source of one place, the origin: no scale to take margins from."""
    mp, src = np.zeros((5, 3), F), np.zeros((40, 3), F)
    src[1::2, 0] = 2.0
    t = gpu_lib.Target(dev(mp), exhaustive=exhaustive)
    want = np.where(np.arange(40) % 2 == 0, 0, -1)
    np.testing.assert_array_equal(pairs(t, mp, src, max_dist), want)
    assert t.sync_status() == gpu_lib.PC_OK
    assert t.stats()["exhaustive"] == 0
    t.close()


# ---------------------------------------------------------------- kNN
@pytest.mark.parametrize("n", [3000, 24_600])
@pytest.mark.parametrize("k", [1, 10, 20, 32])
@pytest.mark.parametrize("cells", [8, 64, 512])
def test_knn_reach(gpu_lib, cells, k, n):
    """A query is answered when one of the three fixed radii (1.46, 2.63, 4.73 times the calibrated one) holds its k
    neighbours in a box of at most 4096 cells and 256 rows, the smaller ones having held fewer."""
    mp, q = clusters(cells, n)
    t = gpu_lib.Target(dev(mp), cell_size=1.0, max_box_cells=cells, exhaustive=False)
    info = t.info()
    head = q[:3000]
    ri, rd = oracle.knn_brute(head, mp, k)
    d = np.sqrt(rd[:, -1])
    hint = info["rho_hint"][k - 1]
    r = 1.46 * 0.9 * (hint if hint > 0 else info["cell_size"])
    must = np.zeros(len(head), bool)
    for j in range(3):
        ncl, rows = boxes(info, head.astype(np.float64), r * 1.8 ** j)
        must |= (ncl <= 4096) & (rows <= 256) & (d < 0.999 * r * 1.8 ** j)
    t.set_tune(probe=1)  # every query from the calibrated radius
    idx, d2 = t.knn(dev(q), k)
    t.sync_status()
    idx, d2 = idx.cpu().numpy()[:3000], d2.cpu().numpy()[:3000]
    t.close()
    got = idx[:, 0] >= 0
    assert must.sum() > 300
    assert got[must].all()
    np.testing.assert_array_equal(idx[got], ri[got])
    np.testing.assert_array_equal(d2[got], rd[got])


def test_far_query_stays_refused(gpu_lib):
    mp = lattice(24, 24, 20)
    t = gpu_lib.Target(dev(mp), cell_size=0.5, max_box_cells=8, exhaustive=False)
    idx, d2 = t.knn(dev(np.array([[5e3, 0, 0]], F)), 8)
    assert t.sync_status() == gpu_lib.PC_ERR_SEARCH_LIMIT
    assert (idx == -1).all()
    t.close()


@pytest.mark.parametrize("k", [40, 64])
def test_wide_k_does_not_depend_on_the_call(gpu_lib, k):
    """Of 64 queries the same ones are answered alone and at the head of a call of 20,000."""
    mp, q = clusters(k, 20_000)
    differ = 0
    for cells in (64, 512):
        t = gpu_lib.Target(dev(mp), max_box_cells=cells, exhaustive=False)
        whole = t.knn(dev(q), k)[0].cpu().numpy()
        for at in range(0, 640, 64):
            part = t.knn(dev(q[at:at + 64]), k)[0].cpu().numpy()
            differ += int((part != whole[at:at + 64]).any(1).sum())
        t.sync_status()
        t.close()
    assert differ == 0
