"""The target build's device steps against numpy: the cell-size bisection
(trial counts of occupied cells, binary32 cell rule) and the calibration's
percentiles, at the edges of the sample and the sort."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F = np.float32


def cells(p, o, h):
    c = np.floor((p - o) * (F(1.0) / F(h))).astype(np.int64)
    return np.clip(c, 0, (1 << 21) - 1)


def cell_size(p, target=12.0):
    o, mx = p.min(0), p.max(0)
    ext = F((mx - o).max())
    if ext == 0:
        return F(1.0)
    lo, hi = float(ext / F(1048576.0) * F(1.001)), float(ext) * 1.001
    if len(p) >= target:
        for _ in range(14):
            mid = np.sqrt(lo * hi)
            u = len(np.unique(cells(p, o, F(mid)), axis=0))
            if len(p) / u < target:
                lo = mid
            else:
                hi = mid
    return max(F(hi), ext / F(1048576.0) * F(1.001))


@pytest.mark.parametrize("m", [1, 2, 11, 12, 63, 64, 1023, 1024, 1025, 2049, 20000])
def test_cell_size_and_hints(gpu_lib, m):
    g = np.random.default_rng(m)
    p = (g.random((m, 3)) * [30, 20, 3] - [5, 5, 1]).astype(F)
    p[m // 2:m // 2 + 5] = p[m // 2]  # equal points
    t = gpu_lib.Target(torch.from_numpy(p).cuda())
    i = t.info()
    t.close()
    assert F(i["cell_size"]) == cell_size(p)
    kc, s = min(64, m), min(m, 1024)
    d2 = oracle.knn_brute(np.ascontiguousarray(p[::m // s][:s]), p, kc)[1]
    want = np.zeros(64, F)
    want[:kc] = np.sqrt(np.sort(d2, axis=0)[s * 3 // 4])
    np.testing.assert_array_equal(np.array(i["rho_hint"], F), want)


@pytest.mark.parametrize("m", [1024, 1025, 524288, 524289])
def test_sort_tile_edges(gpu_lib, m):
    """Both sort tiles and their remainders: every point is found where it is."""
    p = (np.random.default_rng(m).random((m, 3)) * [300, 200, 3]).astype(F)
    t = gpu_lib.Target(torch.from_numpy(p).cuda())
    at = np.unique(np.concatenate([np.arange(0, m, max(1, m // 4000)), [m - 1]]))
    idx, d2 = t.knn(torch.from_numpy(p[at]).cuda(), 1)
    t.close()
    assert (d2 == 0).all()
    np.testing.assert_array_equal(p[idx.cpu().numpy()[:, 0]], p[at])


@pytest.mark.parametrize("n", [1, 300, 5000, 70000])
def test_wall_of_a_small_scan_in_a_large_detector(gpu_lib, n):
    """A detector made for 600k points (its tables and sort follow the scan)."""
    from paper_2308_07173_gb300 import workloads as W

    pts = torch.from_numpy(np.ascontiguousarray(W.body_frame_scan(seed=3)[:n])).cuda()
    got = []
    for cap in (n, 600_000):
        det = gpu_lib.WallDetector(cap)
        det.detect(pts)
        got.append(det.result(arrays=True))
        det.close()
    a, b = got
    assert a.keys() == b.keys()
    for k in a:
        np.testing.assert_array_equal(np.asarray(a[k]), np.asarray(b[k]))
