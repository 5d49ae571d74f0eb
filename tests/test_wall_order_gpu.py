"""Voxel centroids are binary64 sums in index order, also where the order shows:
voxels whose sum is not exact, so that adding the same points in another order
(or in strands) rounds to another binary32 centroid."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

OPTS = dict(voxel=0.2, cell2d=0.2, min_votes=2, tol=0.45, min_cluster=10)
F = np.float32


def centroids(pc, pts):
    det = pc.WallDetector(len(pts), **OPTS)
    det.detect(torch.from_numpy(np.ascontiguousarray(pts)).cuda())
    r = det.result(arrays=True)
    det.close()
    return r["centroids"]


def tie(axis):
    """Two neighbouring binary32 values whose mean over 16 points is a tie, and 14 values that index order loses one
    by one while pairs of them move the sum past the tie."""
    b = F(0.1)
    if b.view(np.uint32) & 1:
        b = np.nextafter(b, F(1))
    p = np.full((16, 3), 0.05, F)
    p[:, axis] = 2.0 ** -57
    p[0, axis], p[1, axis] = b, np.nextafter(b, F(1))
    col = p[:, axis].astype(np.float64)
    in_order = F(np.add.accumulate(col)[-1] / 16)
    strands = F(np.add.reduce(np.add.reduce(col.reshape(2, 8), axis=0).reshape(4, 2)[[1, 2, 3, 0]].sum(1)) / 16)
    assert in_order != strands
    return p


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_order_decides_a_tie(gpu_lib, axis):
    p = tie(axis)
    want = oracle.wall_detect(p, **OPTS)["centroids"]
    np.testing.assert_array_equal(centroids(gpu_lib, p).view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("n", [1, 7, 8, 9, 600, 40_000])
def test_wide_exponents_match_index_order(gpu_lib, n):
    """Coordinates from 1e-44 (not normal) to 100 m, zeros among them, both signs."""
    g = np.random.default_rng(n)
    e = g.uniform(-146.0, -2.4, (n, 3))
    p = (np.exp2(e) * g.choice([-1.0, 1.0], (n, 3))).astype(F)
    p[g.random((n, 3)) < 0.1] = 0
    p[n // 2:] = (g.random((n - n // 2, 3)) * [100.0, 20.0, 2.0]).astype(F)
    want = oracle.wall_detect(p, **OPTS)["centroids"]
    np.testing.assert_array_equal(centroids(gpu_lib, p).view(np.uint32), want.view(np.uint32))
