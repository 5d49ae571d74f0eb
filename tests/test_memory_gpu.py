"""Device memory of targets: what builds and closed handles give back, closing
beside captures in progress, and entries that take no memory."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MB = 1 << 20
KEPT = 256 * MB + 32 * MB  # the pool's unused bytes, and the granularity of allocations


def free():
    return torch.cuda.mem_get_info()[0]


def cloud(n, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand((n, 3), device="cuda", generator=g) * torch.tensor([300.0, 200.0, 3.0], device="cuda")


def test_builds_and_closed_targets_keep_little(gpu_lib):
    p = cloud(20_000_000)
    gpu_lib.Target(p[:1000]).close()
    torch.cuda.synchronize()
    before = free()
    t = gpu_lib.Target(p)
    assert before - free() <= t.info()["device_bytes"] + KEPT
    t.append(p[:5_000_000])
    assert before - free() <= t.info()["device_bytes"] + KEPT
    t.close()
    assert before - free() <= KEPT


def test_other_allocations_take_what_the_pool_keeps(gpu_lib):
    gpu_lib.Target(cloud(20_000_000)).close()
    torch.cuda.empty_cache()
    hold = torch.empty(free() - 80 * MB, dtype=torch.uint8, device="cuda")
    try:
        gpu_lib.WallDetector(1_000_000).close()  # 135 MB
    finally:
        del hold
        torch.cuda.empty_cache()


SETUP = """
import sys, threading, torch
from paper_2308_07173_gb300 import pc
cloud = lambda n: torch.rand((n, 3), device="cuda") * torch.tensor([300.0, 200.0, 3.0], device="cuda")
free = lambda: torch.cuda.mem_get_info()[0]
big, q = cloud(20_000_000), cloud(1000)
t = pc.Target(q)
want, _ = t.knn(q, 5)
idx, d2 = torch.empty_like(want), torch.empty((1000, 5), device="cuda")
torch.cuda.synchronize()
before = free()
other = pc.Target(big)
"""

CLOSE = {
    "another thread": """
def close():
    th = threading.Thread(target=other.close)
    th.start()
    th.join()
""",
    "this thread": """
def close():
    other.close()
""",
}

CAPTURE = """
graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
with torch.cuda.graph(graph, stream=s, capture_error_mode=sys.argv[1]):
    close()
    t.knn(q, 5, idx, d2, stream=s)
graph.replay()
torch.cuda.synchronize()
assert torch.equal(idx, want)
assert before - free() <= (256 + 64) << 20, (before - free()) >> 20
"""


def child(code, *args):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code, *args], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-1500:]


@pytest.mark.parametrize("mode", ["thread_local", "global", "relaxed"])
@pytest.mark.parametrize("who", list(CLOSE))
def test_close_beside_a_capture(gpu_lib, who, mode):
    """The capture stays valid and the memory comes back."""
    child(SETUP + CLOSE[who] + CAPTURE, mode)


def test_close_waits_for_searches_on_other_streams(gpu_lib):
    t = gpu_lib.Target(cloud(200_000))
    q = cloud(300_000, 1)
    want = t.knn(q, 20)[0]
    idx, d2 = torch.empty_like(want), torch.empty((len(q), 20), device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(40_000_000)
    t.knn(q, 20, idx, d2, stream=s)
    done = torch.cuda.Event()
    done.record(s)
    t.close()
    assert done.query()
    assert torch.equal(idx, want)


def test_first_noalloc_call_takes_no_memory(gpu_lib):
    child("""
import torch
from paper_2308_07173_gb300 import pc
p, q = torch.rand((200_000, 3), device="cuda") * 50, torch.rand((50_000, 3), device="cuda") * 50
t = pc.Target(p)
o = (torch.empty((50_000, 20), dtype=torch.int32, device="cuda"), torch.empty((50_000, 20), device="cuda"),
     torch.empty((50_000, 6), device="cuda"))
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
scan = pc.pc_scan(q.data_ptr(), 50_000, *(x.data_ptr() for x in o))
assert pc.pc_batch_run_noalloc(t.handle, [scan], 20, 1e-3, 0) == pc.PC_OK
torch.cuda.synchronize()
assert torch.cuda.mem_get_info()[0] == before
""")


@pytest.mark.parametrize("mode", ["thread_local", "global", "relaxed"])
def test_append_and_compact_refuse_a_capture_and_leave_nothing_in_it(gpu_lib, mode):
    p = cloud(1014, 2)
    t = gpu_lib.Target(p[:1000])
    t.append(p[1000:1010])
    t.append(p[1010:1011])  # room for 20: the next ones do not allocate
    graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    x = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s, capture_error_mode=mode):
        x.add_(1)
        for refused in (lambda: t.append(p[1013:1014], stream=s), lambda: t.compact(stream=s)):
            with pytest.raises(gpu_lib.PcError) as e:
                refused()
            assert e.value.code == gpu_lib.PC_ERR_CUDA
    t.append(p[1011:1012])
    graph.replay()
    torch.cuda.synchronize()
    t.append(p[1012:1013])  # the grid of appended points is built again
    idx, d2 = t.knn(p[1011:1013].contiguous(), 1)
    assert idx.flatten().tolist() == [1011, 1012] and (d2 == 0).all()
    assert (x == 1).all()
    t.close()
