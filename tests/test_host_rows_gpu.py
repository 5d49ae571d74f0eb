"""Searches that write page-locked host memory (k <= 32): rows on 128-byte lines
(one-warp units) and off them (blocks of four units with remainders), far, equal
and non-finite queries in every place of a block, windows and weights.  Every
row equals the device-memory search's bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from tests.test_group_search_gpu import dev, scene  # noqa: E402

SETTINGS = {
    "plain": lambda t: None,
    "window": lambda t: t.set_window([-1.0, 4.0, -1.0], [15.5, 30.0, 3.0]),
    "weighted": lambda t: t.set_cov_kernel("laplacian", sigma=0.3),
    "window, weighted": lambda t: (t.set_window([2.0, -1.0, -1.0], [30.0, 12.5, 3.0]), t.set_cov_kernel("rbf", sigma=1.0)),
}


def queries(n, seed):
    m, q = scene(max(n, 9), seed)
    q = q[:n]
    q[::37] += np.float32(70.0)  # left over by the group search, in every place of a block
    if n > 3:
        q[n // 2, 1] = np.nan
    return m, np.ascontiguousarray(q)


def bits(t):
    return t.cpu().contiguous().view(torch.int32)


@pytest.mark.parametrize("setting", list(SETTINGS))
@pytest.mark.parametrize("k", [1, 3, 20, 24, 25, 32])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 33, 300, 24_590])
def test_rows_in_host_memory(gpu_lib, n, k, setting):
    m, q = queries(n, n + k)
    t = gpu_lib.Target(dev(m))
    SETTINGS[setting](t)
    for eps in (1e-3, -1.0):
        want = t.knn_cov(dev(q), k, eps)
        t.sync_status()
        for off in (0, 1, 32):  # rows from a line, from off one, and from a later line
            out = tuple(torch.full((n + 33, w), -7, dtype=d, pin_memory=True)
                        for w, d in ((k, torch.int32), (k, torch.float32), (6, torch.float32)))
            part = tuple(o[off:off + n] for o in out)
            qp = torch.from_numpy(q).pin_memory()
            rc = gpu_lib.pc_knn_cov_host(t.handle, qp.data_ptr(), n, k, eps, *(p.data_ptr() for p in part), 0)
            assert rc in (gpu_lib.PC_OK, gpu_lib.PC_ERR_NONFINITE, gpu_lib.PC_ERR_K_GT_M)
            for a, b in zip(part, want):
                assert torch.equal(bits(a), bits(b))
            for o in out:
                assert (o[:off] == -7).all() and (o[off + n:] == -7).all()  # nothing beside the rows
    t.close()


@pytest.mark.parametrize("with_cov", [True, False])
@pytest.mark.parametrize("k", [5, 20, 32])
@pytest.mark.parametrize("sizes", [(1, 40, 0, 17), (31, 33, 9000, 5), (20_001, 8_000, 3), (32, 640, 24_000, 7)])
def test_batches_in_host_memory(gpu_lib, sizes, k, with_cov):
    n = sum(sizes)
    m, q = queries(n, n + k)
    t = gpu_lib.Target(dev(m))
    want = t.knn_cov(dev(q), k, 1e-3)
    t.sync_status()
    qp = torch.from_numpy(q).pin_memory()
    out = tuple(torch.full((n, w), -7, dtype=d, pin_memory=True)
                for w, d in ((k, torch.int32), (k, torch.float32), (6, torch.float32)))
    at = np.concatenate([[0], np.cumsum(sizes)])
    scans = [gpu_lib.pc_scan(qp[a:].data_ptr() if b > a else 0, b - a, *(o[a:].data_ptr() if b > a else 0 for o in out[:2]),
                             out[2][a:].data_ptr() if with_cov and b > a else None) for a, b in zip(at, at[1:])]
    rc = gpu_lib.pc_batch_run_noalloc(t.handle, scans, k, 1e-3, 0)
    assert rc == gpu_lib.PC_OK
    torch.cuda.synchronize()
    for a, b in list(zip(out, want))[:3 if with_cov else 2]:
        assert torch.equal(bits(a), bits(b))
    if not with_cov:
        assert (out[2] == -7).all()
    t.sync_status()
    t.close()
