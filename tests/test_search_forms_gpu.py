"""The search's forms at both group widths (eight lanes a query up to 24,576
queries, four beyond) and on maps without a row index: windows, weights,
appended points and batches, with far, equal and non-finite queries among them."""
import numpy as np
import pytest

import oracle
from tests import helpers as H

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F = np.float32
INF = float("inf")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def bits(t):
    return t.contiguous().view(torch.int32)


def scene():
    """3000 points, 40 of them equal; 2500 queries: near, on the equal points, clusters of far ones, non-finite."""
    g = np.random.default_rng(31)
    m = (g.random((3000, 3)) * [20, 20, 2]).astype(F)
    m[1100:1140] = m[1100]
    q = (g.random((2500, 3)) * [22, 22, 3] - [1, 1, 0.5]).astype(F)
    q[200:260] += F(90.0)
    q[700] = m[1100]
    q[701] = [3000.0, -50.0, 4.0]
    q[1300:1310] = m[1100] + F(1e-3)
    q[1999, 2] = np.inf
    return m, q


WINDOW = ([3.0, -1.0, -1.0], [INF, 14.5, 3.0])


def oracle_rows(m, q, k, window):
    ok = np.isfinite(q).all(1)
    idx, d2 = np.full((len(q), k), -1, np.int32), np.full((len(q), k), np.inf, F)
    idx[ok], d2[ok] = oracle.knn_window(q[ok], m, k, *WINDOW) if window else oracle.knn_brute(q[ok], m, k)
    return idx, d2


@pytest.mark.parametrize("window", [False, True], ids=["whole", "window"])
@pytest.mark.parametrize("weighted", [False, True], ids=["plain", "weighted"])
@pytest.mark.parametrize("grown", [False, True], ids=["built", "grown"])
@pytest.mark.parametrize("k", [20, 32])
def test_forms_at_both_widths(gpu_lib, k, grown, weighted, window):
    m, q = scene()
    t = gpu_lib.Target(dev(m[:1000] if grown else m))
    if grown:
        t.append(dev(m[1000:]))
    if weighted:
        t.set_cov_kernel("laplacian", sigma=0.5)
    if window:
        t.set_window(*WINDOW)
    ri, rd = oracle_rows(m, q, k, window)
    fin = np.isfinite(q).all(1)
    many = np.concatenate([q] * 10 + [q[:37]])  # 25,037 queries
    for eps in (1e-3, -1.0):
        small = t.knn_cov(dev(q), k, eps)
        assert t.sync_status() == gpu_lib.PC_ERR_NONFINITE
        np.testing.assert_array_equal(small[0].cpu().numpy(), ri)
        np.testing.assert_array_equal(small[1].cpu().numpy().view(np.uint32), rd.view(np.uint32))
        large = t.knn_cov(dev(many), k, eps)
        assert t.sync_status() == gpu_lib.PC_ERR_NONFINITE
        for s, b in zip(small, large):
            assert torch.equal(bits(torch.cat([s] * 10 + [s[:37]])), bits(b))
        if not grown:  # planned, the sizes of one wide call
            out = [torch.empty_like(x) for x in large]
            dq = dev(many)
            plan = gpu_lib.Batch(t, [(dq[:9001], *(o[:9001] for o in out)), (dq[9001:], *(o[9001:] for o in out))], k, eps)
            plan.run()
            for a, b in zip(out, large):
                assert torch.equal(bits(a), bits(b))
            t.sync_status()
            plan.close()
        if eps < 0:
            cov = small[2].cpu().numpy()[fin]
            p = m[ri[fin]]
            same = (p == p[:, :1]).all((1, 2))  # k copies of one point: exactly zero
            assert (cov[same] == 0).all()
            far = np.abs(q[fin]).max(1) > 60  # every weight underflows: no covariance
            rows = ~(same | far) if weighted else ~same
            want = (oracle.cov_weighted(m, q[fin], ri[fin], eps, "laplacian", sigma=0.5, origin=m.min(0)) if weighted
                    else oracle.cov(m, ri[fin], eps))
            H.check_raw_cov(cov[rows], want[rows])
    t.close()


def sparse():
    """Tight clusters over 120 m: cells of 0.1 are far too many for the row index, and few hold all of a query's
    neighbours."""
    g = np.random.default_rng(8)
    c = g.random((12, 3)) * [120, 120, 40]
    m = (c[g.integers(0, 12, 9000)] + 0.15 * g.standard_normal((9000, 3))).astype(F)
    q = (m[g.integers(0, 9000, 2000)] + 0.02 * g.standard_normal((2000, 3))).astype(F)
    q[50:60] += F(3.0)
    q[90] = m[4]
    return m, q, c


@pytest.mark.parametrize("window", [False, True], ids=["whole", "window"])
@pytest.mark.parametrize("probe", [1, 2])
@pytest.mark.parametrize("k", [4, 10])
def test_maps_without_a_row_index(gpu_lib, k, probe, window):
    m, q, c = sparse()
    t = gpu_lib.Target(dev(m), cell_size=0.1)
    t.set_tune(probe=probe)
    info = t.info()
    assert (np.prod(np.array(info["dims"], np.int64)) + 1) * 4 > 8 * 16 * len(m)  # no index this large is built
    if window:
        mid = [float(v) for v in c[0]]  # through the middle of a cluster
        w = ([mid[0], -INF, -INF], [INF, INF, mid[2] + 0.05])
        t.set_window(*w)
        ri, rd = oracle.knn_window(q, m, k, *w)
    else:
        ri, rd = oracle.knn_brute(q, m, k)
    many = np.concatenate([q] * 13)
    t.stats(reset=True)
    small = t.knn_cov(dev(q), k, 1e-3)
    st = t.stats(reset=True)
    if probe == 1:  # per-query radii have no counts to go by here: three cells, a box too large for a group
        assert st["warp_search"] < 0.75 * st["queries"]  # the groups' cell walk answered the others
    np.testing.assert_array_equal(small[0].cpu().numpy(), ri)
    np.testing.assert_array_equal(small[1].cpu().numpy().view(np.uint32), rd.view(np.uint32))
    large = t.knn_cov(dev(many), k, 1e-3)
    out = [torch.empty_like(x) for x in large]
    dq = dev(many)
    plan = gpu_lib.Batch(t, [(dq[:20_001], *(o[:20_001] for o in out)), (dq[20_001:], *(o[20_001:] for o in out))], k, 1e-3)
    plan.run()
    pinned = tuple(torch.empty(x.shape, dtype=x.dtype, pin_memory=True) for x in small)
    t.knn_cov_host(torch.from_numpy(q).pin_memory(), k, 1e-3, out=pinned)
    for s, b, o, p in zip(small, large, out, pinned):
        assert torch.equal(bits(torch.cat([s] * 13)), bits(b))
        assert torch.equal(bits(o), bits(b))
        assert torch.equal(bits(p.cuda()), bits(s))
    plan.close()
    t.close()
