"""The group search (k <= 32) and the kernel that finishes it: units with
remainders, both group widths, both sort capacities, more equal distances than
are sorted, clusters of far queries, and the same through the batched,
host-buffer and grown-map forms.  Indices and distances equal the brute-force
oracle bit for bit; covariances equal pc_cov of those rows bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2308_07173_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def scene(n, seed):
    """A small cloud with 40 copies of one point, and n queries: near ones, a
    cluster far off, one on the copies, one not finite in the last place."""
    g = np.random.default_rng(seed)
    m = (g.random((3000, 3)) * [20, 20, 2]).astype(np.float32)
    m[100:140] = m[100]
    q = (g.random((n, 3)) * [22, 22, 3] - [1, 1, 0.5]).astype(np.float32)
    if n >= 9:
        q[2:7] += np.float32(90.0)
        q[7] = m[100]
        q[8] = [3000.0, -50.0, 4.0]
    return m, q


def check(m, q, k, idx, d2):
    ri, rd = oracle.knn_brute(q, m, k)
    np.testing.assert_array_equal(idx.cpu().numpy(), ri)
    np.testing.assert_array_equal(d2.cpu().numpy().view(np.uint32), rd.view(np.uint32))


@pytest.mark.parametrize("k", [1, 3, 20, 24, 25, 32])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 9, 33, 1000, 24577])
def test_units_and_leftovers(gpu_lib, n, k):
    m, q = scene(n, 10 * n + k)
    t = gpu_lib.Target(dev(m))
    idx, d2, cov = t.knn_cov(dev(q), k, 1e-3)
    assert t.sync_status() == gpu_lib.PC_OK
    check(m, q, k, idx, d2)
    assert torch.equal(cov.view(torch.int32), t.cov(idx, 1e-3).view(torch.int32))
    ki, kd = t.knn(dev(q), k)
    assert torch.equal(ki, idx) and torch.equal(kd, d2)
    t.close()


@pytest.mark.parametrize("eps", [1e-3, -1.0])
def test_forms_agree_on_leftovers(gpu_lib, eps):
    k, n = 20, 300
    m, q = scene(n, 5)
    t = gpu_lib.Target(dev(m))
    ref = t.knn_cov(dev(q), k, eps)
    check(m, q, k, ref[0], ref[1])
    # batched, two scans of odd sizes
    out = [torch.empty_like(x) for x in ref]
    dq = dev(q)
    plan = gpu_lib.Batch(t, [(dq[:101], *(o[:101] for o in out)), (dq[101:], *(o[101:] for o in out))], k, eps)
    plan.run()
    for a, b in zip(out, ref):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    plan.close()
    # page-locked host outputs
    host = tuple(torch.empty(x.shape, dtype=x.dtype, pin_memory=True) for x in ref)
    t.knn_cov_host(torch.from_numpy(q).pin_memory(), k, eps, out=host)
    for a, b in zip(host, ref):
        assert torch.equal(a.view(torch.int32), b.cpu().view(torch.int32))
    t.close()
    # the same map, a third of it appended
    t = gpu_lib.Target(dev(m[:2000]))
    t.append(dev(m[2000:]))
    got = t.knn_cov(dev(q), k, eps)
    for a, b in zip(got, ref):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    t.close()


def test_nonfinite_beside_far_queries(gpu_lib):
    k = 10
    m, q = scene(50, 7)
    q[0, 1] = np.nan  # first row of a unit whose next rows are far
    t = gpu_lib.Target(dev(m))
    idx, d2, cov = t.knn_cov(dev(q), k, 1e-3)
    assert t.sync_status() == gpu_lib.PC_ERR_NONFINITE
    assert (idx[0] == -1).all() and torch.isinf(d2[0]).all() and (d2[0] > 0).all() and torch.isnan(cov[0]).all()
    check(m, q[1:], k, idx[1:], d2[1:])
    t.close()
