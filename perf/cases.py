"""The work that a user of this library has it do, as measurable cases.

Each case is one call (or the short run of calls that belong together) of the
public Python entry points: neighbour searches with fused covariances over a
resident map, the batched form, the host-buffer form, searches over a map
grown by appended points, the covariances of a whole cloud (a target built
from it and queried with it), GICP registration and wall detection.  Inputs
are the repository's own seeded generators (race-track LiDAR scans and maps).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2308_07173_gb300 import gicp, pc
from paper_2308_07173_gb300 import workloads as W

EPS = 1e-3


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call in earnest: a small cloud against itself, k = 10; launches and latency count
        {"name": "box8k", "call": "search", "scene": "box", "map": 8192, "queries": 8192, "k": 10, "eps": EPS},
        # the ordinary call: one 128-channel scan against the resident map of the track
        {"name": "scan131k", "call": "search", "scene": "track", "map": 2_000_000, "queries": 131_000, "k": 20,
         "eps": EPS},
        # a thinned scan in the sliding window of its place on the race line, Laplacian-weighted raw covariances, odd k
        {"name": "window_weighted", "call": "search", "scene": "track", "map": 2_000_000, "queries": 60_001, "k": 15,
         "eps": -1.0, "kernel": "laplacian", "window": 130.0},
        # wide neighbourhoods of a thinned scan (k above 32)
        {"name": "wide_k48", "call": "search", "scene": "track", "map": 300_000, "queries": 20_011, "k": 48,
         "eps": EPS},
        # the ordinary scan while the map grows: 200k points appended and not yet compacted
        {"name": "grown_map", "call": "search", "scene": "track", "map": 1_800_000, "queries": 131_000, "k": 20,
         "eps": EPS, "appended": 200_000},
        # the ordinary scan from page-locked host memory, results back in host memory
        {"name": "host_scan", "call": "host", "scene": "track", "map": 2_000_000, "queries": 131_000, "k": 20,
         "eps": EPS},
        # many scans in one call: 64 scans of 20k-130k points, a planned batch
        {"name": "batch64", "call": "batch", "scene": "track", "map": 2_000_000, "scans": 64, "lo": 20_000,
         "hi": 130_000, "k": 20, "eps": EPS},
        # the largest search: eight scans against a large map of uneven density, k = 32
        {"name": "large_pit", "call": "search", "scene": "pit", "map": 5_000_000, "queries": 1_048_000, "k": 32,
         "eps": EPS},
        # per scan in registration: the scan's own covariances (a target built from it, queried with it)
        {"name": "self_scan", "call": "self", "scene": "track", "points": 131_000, "k": 20, "eps": EPS},
        # once per map: the map's target and the covariances of all its points
        {"name": "self_map", "call": "self", "scene": "map", "points": 2_000_000, "k": 20, "eps": EPS},
        # one scan registered against the map: ten linearise-and-update iterations
        {"name": "register", "call": "gicp", "map": 2_000_000, "queries": 100_000, "iters": 10},
        # wall detection on one body-frame scan, read back
        {"name": "wall", "call": "wall", "points": 131_000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["search", "search", "search", "search", "host", "batch", "self", "self", "gicp", "wall"])
    eps = rng.choice([EPS, EPS, EPS, 0.01, -1.0])
    k = rng.choice([10, 20, 20, 32, rng.randint(4, 32), rng.randint(5, 24)])
    if call == "wall":
        return {"call": "wall", "points": _log_int(rng, 5_000, 131_000)}
    if call == "gicp":
        return {"call": "gicp", "map": _log_int(rng, 300_000, 3_000_000), "queries": _log_int(rng, 3_000, 100_000),
                "iters": rng.choice([5, 10])}
    if call == "self":
        scene = rng.choice(["track", "map", "box"])
        hi = {"track": 131_000, "map": 2_000_000, "box": 100_000}[scene]
        return {"call": "self", "scene": scene, "points": _log_int(rng, 3_000, hi), "k": k, "eps": eps}
    if call == "batch":
        lo = _log_int(rng, 2_000, 60_000)
        return {"call": "batch", "scene": "track", "map": _log_int(rng, 100_000, 3_000_000),
                "scans": rng.randint(2, 64), "lo": lo, "hi": min(130_000, 4 * lo), "k": k, "eps": eps}
    if call == "host":
        return {"call": "host", "scene": "track", "map": _log_int(rng, 100_000, 3_000_000),
                "queries": _log_int(rng, 1_000, 131_000), "k": k, "eps": eps}
    case = {"call": "search", "scene": rng.choice(["track", "track", "pit", "box"]), "k": k, "eps": eps}
    if case["scene"] == "box":
        case["map"] = _log_int(rng, 2_000, 200_000)
        case["queries"] = _log_int(rng, 500, 65_536)
        return case
    case["map"] = _log_int(rng, 100_000, 5_000_000)
    case["queries"] = _log_int(rng, 500, 600_000)
    option = rng.choice(["plain", "plain", "wide", "window", "kernel", "appended"])
    if option == "wide":
        case["k"] = rng.randint(33, 64)
        case["queries"] = min(case["queries"], 40_000)
    elif option == "window" and case["scene"] == "track":
        case["window"] = rng.choice([130.0, 150.0])
        case["queries"] = min(case["queries"], 131_000)
    elif option == "kernel":
        case["kernel"] = rng.choice(["laplacian", "gaussian", "rbf"])
        case["queries"] = min(case["queries"], 200_000)
    elif option == "appended":
        case["appended"] = max(1_000, case["map"] // rng.choice([7, 10, 30]))
        case["queries"] = min(case["queries"], 200_000)
    return case


# ---------------------------------------------------------------- inputs
def _scan(tr, n, g):
    """n points of ray-cast scans at random poses (as many full scans as it takes, the last a random subset kept in
    scan order), and the first pose's position."""
    parts, left, at = [], n, None
    while left > 0:
        pose = tr.random_pose(g)
        full = tr.raycast(*pose, g)
        if at is None:
            p, _, nr = tr.pose(np.array([pose[0]]))
            at = np.array([*(p[0] + nr[0] * pose[1]), 0.8])
        if left < len(full):
            full = full[np.sort(g.choice(len(full), left, replace=False))]
        parts.append(full)
        left -= len(full)
    return np.concatenate(parts), at


def _search_inputs(case, seed):
    """map (appended points last), queries, sensor position; float32 arrays."""
    g = W.rng_for(7919 * seed + 11)
    m_all = case["map"] + case.get("appended", 0)
    if case["scene"] == "box":
        m = W.uniform_box(m_all, seed=seed + 1)
        q = m if case["queries"] == m_all else W.uniform_box(case["queries"], seed=seed + 2)
        return m, q, np.zeros(3)
    pit = case["scene"] == "pit"
    tr = W.oval_4000_pit() if pit else W.oval_1500()
    m = tr.sample_map(m_all, seed + 1, noise=0.01 if pit else 0.0)
    if case.get("appended"):  # the track generator puts wall points last: appended points are of every kind
        m = m[g.permutation(m_all)]
    q, at = _scan(tr, case["queries"], g)
    return m, q, at


def _cloud(case, seed):
    if case["scene"] == "box":
        return W.uniform_box(case["points"], seed=seed + 1)
    tr = W.oval_1500()
    if case["scene"] == "map":
        return tr.sample_map(case["points"], seed + 1)
    return _scan(tr, case["points"], W.rng_for(7919 * seed + 11))[0]


def _batch_inputs(case, seed):
    """The map and scans of log-uniform sizes between lo and hi (subsets, in scan order, of ray casts at up to 16
    poses)."""
    tr = W.oval_1500()
    m = tr.sample_map(case["map"], seed + 1)
    sizes = np.exp(W.rng_for(case["scans"]).uniform(math.log(case["lo"]), math.log(case["hi"]), case["scans"]))
    g = W.rng_for(7919 * seed + 11)
    casts = [_scan(tr, 131_000, g)[0] for _ in range(min(16, case["scans"]))]
    scans = []
    for i, n in enumerate(sizes.astype(np.int64)):
        full = casts[i % len(casts)]
        scans.append(full[np.sort(g.choice(len(full), int(n), replace=False))])
    return m, scans


def _gicp_inputs(case, seed):
    """A map of the track with its pit lane, and an independent sample of it around a sensor in the pit lane (whose
    walls constrain all six degrees of freedom), ring by ring in the sensor's frame; the pose starts a little off."""
    tr = W.oval_4000_pit()
    m = tr.sample_map(case["map"], seed + 1, noise=0.01)
    g = W.rng_for(7919 * seed + 11)
    o = np.array([g.uniform(-200.0, 200.0), tr.r + tr.half_width + tr.pit_width / 2, 0.8])
    near = tr.sample_map(25 * case["queries"], seed + 2, noise=0.01).astype(np.float64) - o
    near = near[np.argsort(np.hypot(near[:, 0], near[:, 1]))[:case["queries"]]]
    ring = np.floor(np.rad2deg(np.arctan2(near[:, 2], np.hypot(near[:, 0], near[:, 1]))) / 0.2)
    near = near[np.lexsort((np.arctan2(near[:, 1], near[:, 0]), ring))]
    yaw = float(g.uniform(-0.4, 0.4))
    rot = _exp_so3(np.array([0.0, 0.0, yaw]))
    src = (near @ rot).astype(np.float32)
    off = _exp_so3(np.array([0.003, -0.004, 0.02]) * g.uniform(0.5, 1.0))
    pose = np.concatenate([(off @ rot).ravel(), o + np.array([0.2, -0.15, 0.05]) * g.uniform(0.5, 1.0)])
    return m, src, pose.astype(np.float32)


def _exp_so3(w):
    th = float(np.linalg.norm(w))
    k = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
    if th < 1e-9:
        return np.eye(3) + k
    return np.eye(3) + math.sin(th) / th * k + (1 - math.cos(th)) / th ** 2 * (k @ k)


def _wall_inputs(case, seed):
    g = W.rng_for(7919 * seed + 11)
    pts = W.body_frame_scan(s0=float(g.uniform(0.0, 1500.0)), w0=float(g.uniform(-2.0, 2.0)), seed=seed + 1)
    while len(pts) < case["points"]:
        pts = np.concatenate([pts, pts[:case["points"] - len(pts)]])
    return pts[np.sort(g.choice(len(pts), case["points"], replace=False))]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    call = case["call"]
    if call == "self":
        return {"call": call, "k": case["k"], "eps": case["eps"], "xyz": _dev(_cloud(case, seed))}
    if call == "wall":
        pts = _dev(_wall_inputs(case, seed))
        n = pts.shape[0]
        return {"call": call, "det": pc.WallDetector(n), "pts": pts,
                "voxels": {"centroids": np.zeros((n, 3), np.float32), "vertical": np.zeros(n, bool),
                           "labels": np.zeros(n, np.int32)}}
    if call == "gicp":
        m, src, pose = _gicp_inputs(case, seed)
        reg = gicp.Registration(_dev(m), k=20, eps=EPS)
        src = _dev(src)
        return {"call": call, "reg": reg, "src": src, "src_cov": reg.source_covariances(src), "pose": _dev(pose),
                "iters": case["iters"]}
    if call == "batch":
        m, scans = _batch_inputs(case, seed)
        n, k = sum(len(s) for s in scans), case["k"]
        t = pc.Target(_dev(m))
        q = _dev(np.concatenate(scans))
        idx = torch.empty((n, k), dtype=torch.int32, device="cuda")
        d2 = torch.empty((n, k), dtype=torch.float32, device="cuda")
        cov = torch.empty((n, 6), dtype=torch.float32, device="cuda")
        at = np.cumsum([0] + [len(s) for s in scans])
        rows = [slice(int(a), int(b)) for a, b in zip(at[:-1], at[1:])]
        plan = pc.Batch(t, [(q[r], idx[r], d2[r], cov[r]) for r in rows], k, case["eps"])
        return {"call": call, "target": t, "plan": plan, "out": (idx, d2, cov)}
    m, q, at = _search_inputs(case, seed)
    t = pc.Target(_dev(m[:case["map"]]))
    if case.get("appended"):
        t.append(_dev(m[case["map"]:]))
    if case.get("kernel"):
        t.set_cov_kernel(case["kernel"], sigma=0.1 if case["kernel"] != "rbf" else 20.0)
    if case.get("window"):
        w = case["window"]
        t.set_window(at - [w, w, math.inf], at + [w, w, math.inf])
    n, k = len(q), case["k"]
    if call == "host":
        out = (torch.empty((n, k), dtype=torch.int32, pin_memory=True),
               torch.empty((n, k), dtype=torch.float32, pin_memory=True),
               torch.empty((n, 6), dtype=torch.float32, pin_memory=True))
        return {"call": call, "target": t, "q": torch.from_numpy(q).pin_memory(), "k": k, "eps": case["eps"],
                "out": out}
    out = (torch.empty((n, k), dtype=torch.int32, device="cuda"),
           torch.empty((n, k), dtype=torch.float32, device="cuda"),
           torch.empty((n, 6), dtype=torch.float32, device="cuda"))
    return {"call": call, "target": t, "q": _dev(q), "k": k, "eps": case["eps"], "out": out}


def run(state):
    call = state["call"]
    if call == "search":
        return state["target"].knn_cov(state["q"], state["k"], state["eps"], *state["out"])
    if call == "host":
        return state["target"].knn_cov_host(state["q"], state["k"], state["eps"], out=state["out"])
    if call == "batch":
        state["plan"].run()
        return state["out"]
    if call == "self":
        t = pc.Target(state["xyz"])
        out = t.knn_cov(state["xyz"], state["k"], state["eps"])
        t.close()
        return out
    if call == "gicp":
        pose = state["pose"].clone()
        lin, xi = state["reg"].align(state["src"], state["src_cov"], pose, iters=state["iters"], max_dist=1.0)
        return pose, lin, xi
    state["det"].detect(state["pts"])
    got = state["det"].result(arrays=True)
    for name, rows in state["voxels"].items():  # the program's own buffers, as many rows as points
        rows[:got["n_voxels"]] = got.pop(name)
    return {**got, **state["voxels"]}


# ---------------------------------------------------------------- work
def work(case):
    """Bytes: the queries, the outputs, and about as many map points as there are queries (a scan's neighbourhoods
    overlap), or the whole cloud where a target is built.  Operations: k distances, the moments and the normal."""
    call = case["call"]
    if call == "wall":  # the points in; about one voxel for every eight points out: centroid, flag, label
        n = case["points"]
        return {"bytes": 12 * n + 20 * n / 8, "flops": 12 * n}
    if call == "gicp":  # per iteration: the points, their covariances, the pairs' points and covariances
        n = case["queries"]
        return {"bytes": case["iters"] * n * (12 + 24 + 16 + 24), "flops": case["iters"] * n * 350}
    k = case["k"]
    if call == "self":
        n = read = case["points"]
    elif call == "batch":
        lo, hi = case["lo"], case["hi"]
        n = case["scans"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo)
        read = min(case["map"], n)
    else:
        n = case["queries"]
        read = min(case["map"] + case.get("appended", 0), n)
    return {"bytes": n * (12 + 8 * k + 24) + 12 * read, "flops": n * (8 * k + 24 * k + 200)}


# ---------------------------------------------------------------- 64-bit values
def _near64(q, m, k, cand=None):
    """The k nearest rows of m (of its rows `cand`, if given) of each row of q, in chunks that fit."""
    near = m if cand is None else m[cand]
    vals, idxs = [], []
    for r in torch.split(q, max(1, int(3e8 // near.shape[0]))):
        d = torch.cdist(r, near, compute_mode="donot_use_mm_for_euclid_dist")
        v, i = torch.topk(d, k, largest=False, sorted=True) if k > 1 else d.min(1, keepdim=True)
        vals.append(v)
        idxs.append(i if cand is None else cand[i])
    return torch.cat(vals), torch.cat(idxs)


def _knn64(q, m, k, columns_most=6000):
    """Distances and indices of the k nearest rows of m for each row of q (binary64, on the GPU).  Queries are taken
    by square columns of edge s in x and y: the k nearest of the 3 x 3 columns around are the answer where the k-th
    lies within s; the queries left over are taken again with columns four times as wide."""
    n, M = q.shape[0], m.shape[0]
    val = torch.full((n, k), math.inf, dtype=torch.float64, device=q.device)
    idx = torch.zeros((n, k), dtype=torch.int64, device=q.device)
    lo = torch.minimum(q.amin(0), m.amin(0))[:2]
    ext = float((torch.maximum(q.amax(0), m.amax(0))[:2] - lo).max())

    def columns(s):
        cm, cq = torch.floor((m[:, :2] - lo) / s).long() + 1, torch.floor((q[:, :2] - lo) / s).long() + 1
        ny = int(max(cm[:, 1].max(), cq[:, 1].max())) + 2
        return cm[:, 0] * ny + cm[:, 1], cq[:, 0] * ny + cq[:, 1], ny

    s = 0.5
    while s < ext:
        km, kq, ny = columns(s)
        if torch.unique(kq).numel() <= columns_most:
            break
        s *= 2.0
    left = torch.arange(n, device=q.device)
    while left.numel() and s < ext:
        km, kq, ny = columns(s)
        km, order = torch.sort(km)
        kq, perm = torch.sort(kq[left])
        left = left[perm]
        cells, counts = torch.unique_consecutive(kq, return_counts=True)
        offs = torch.tensor([-ny, 0, ny], device=q.device)
        first = torch.searchsorted(km, cells[:, None] + offs - 1).tolist()
        last = torch.searchsorted(km, cells[:, None] + offs + 1, right=True).tolist()
        for rows, f, e in zip(torch.split(left, counts.tolist()), first, last):
            cand = torch.cat([order[a:b] for a, b in zip(f, e)])
            if cand.numel() >= k:
                val[rows], idx[rows] = _near64(q[rows], m, k, cand)
        left = left[val[left, -1] > s]
        s *= 4.0
    if left.numel():
        val[left], idx[left] = _near64(q[left], m, k)
    return val, idx


def _cov64(q, m, idx, eps, weights=None):
    out = torch.empty((idx.shape[0], 6), dtype=torch.float64, device=m.device)
    for a in range(0, idx.shape[0], 1 << 14):
        i = idx[a:a + (1 << 14)]
        p = m[i]
        w = torch.ones(i.shape, dtype=torch.float64, device=m.device)
        if weights is not None:
            w = weights(torch.linalg.norm(p - q[a:a + (1 << 14), None, :], dim=-1))
        w = w / w.sum(1, keepdim=True)
        d = p - (w[..., None] * p).sum(1, keepdim=True)
        C = torch.einsum("nk,nki,nkj->nij", w, d, d)
        if eps >= 0:
            nrm = torch.linalg.eigh(C)[1][:, :, 0]
            C = torch.eye(3, dtype=torch.float64, device=m.device) - (1.0 - eps) * nrm[:, :, None] * nrm[:, None, :]
        out[a:a + (1 << 14)] = C[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]]
    return out


def _rows64(q, m, k, eps, weights=None):
    if q.shape[0] > 2_200_000:  # takes too long
        return None
    r = _knn64(q, m, k)
    return None, r[0] ** 2, _cov64(q, m, r[1], float(np.float32(eps)), weights)


def _gicp64(case, seed):
    m, src, pose = _gicp_inputs(case, seed)
    m, src = _dev(m).double(), _dev(src).double()
    cp = _unpack(_cov64(src, src, _knn64(src, src, 20)[1], EPS))
    R, t = torch.tensor(pose[:9].astype(np.float64).reshape(3, 3)).cuda(), torch.tensor(pose[9:].astype(np.float64)).cuda()
    near = torch.linalg.norm(m[:, :2] - t[:2], dim=1) < float(torch.linalg.norm(src, dim=1).max()) + 5.0
    m = m[near]
    cm = _unpack(_cov64(m, m, _knn64(m, m, 20)[1], EPS))
    lins, xis = [], []
    for _ in range(case["iters"]):
        p = src @ R.T + t
        r = _knn64(p, m, 1, 1500)
        ok = r[0][:, 0] <= 1.0
        j = r[1][ok, 0]
        p = p[ok]
        d = m[j] - p
        om = torch.linalg.inv(cm[j] + R @ cp[ok] @ R.T)
        z = torch.zeros_like(p[:, 0])
        px = torch.stack([z, -p[:, 2], p[:, 1], p[:, 2], z, -p[:, 0], -p[:, 1], p[:, 0], z], 1).reshape(-1, 3, 3)
        J = torch.cat([px, -torch.eye(3, dtype=torch.float64, device=p.device).expand(len(p), 3, 3)], 2)
        H = torch.einsum("nai,nab,nbj->ij", J, om, J)
        b = torch.einsum("nai,nab,nb->i", J, om, d)
        e = torch.einsum("na,nab,nb->", d, om, d)
        u = torch.triu_indices(6, 6)
        lins.append(torch.cat([H[u[0], u[1]], b, e[None], torch.tensor([float(len(p))], device=p.device).double()]))
        xi = -torch.linalg.solve(H, b)
        xis.append(xi)
        E = torch.tensor(_exp_so3(xi[:3].cpu().numpy())).cuda()
        R, t = E @ R, E @ t + xi[3:]
    return torch.cat([R.reshape(-1), t]), torch.stack(lins), torch.stack(xis)


def _unpack(c):
    return c[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(-1, 3, 3)


def _wall64(case, seed):
    """The voxel centroids; flags, labels and the wall follow from comparisons of them."""
    p = _wall_inputs(case, seed)
    inv = np.float32(1.0) / np.float32(0.2)
    c = np.floor(p * inv).astype(np.int64)
    key = (c[:, 0] + (1 << 20)) | (c[:, 1] + (1 << 20)) << 21 | (c[:, 2] + (1 << 20)) << 42
    _, inverse, count = np.unique(key, return_inverse=True, return_counts=True)
    cent = np.zeros((len(p), 3))
    for a in range(3):
        cent[:len(count), a] = np.bincount(inverse, p[:, a].astype(np.float64)) / count
    return {"centroids": cent}


def exact(case, seed):
    call = case["call"]
    if call == "wall":
        return _wall64(case, seed)
    if call == "gicp":
        return _gicp64(case, seed)
    if call == "self":
        x = _dev(_cloud(case, seed)).double()
        return _rows64(x, x, case["k"], case["eps"])
    if call == "batch":
        m, scans = _batch_inputs(case, seed)
        return _rows64(_dev(np.concatenate(scans)).double(), _dev(m).double(), case["k"], case["eps"])
    m, q, at = _search_inputs(case, seed)
    weights = None
    if case.get("kernel"):
        s = float(np.float32(20.0 if case["kernel"] == "rbf" else 0.1))
        weights = {"laplacian": lambda r: torch.exp(-r / s), "rbf": lambda r: torch.exp(-r * r * s),
                   "gaussian": lambda r: torch.exp(-r * r / (2.0 * s * s))}[case["kernel"]]
    if case.get("window"):
        w = case["window"]
        lo, hi = (at - [w, w, math.inf]).astype(np.float32), (at + [w, w, math.inf]).astype(np.float32)
        m = m[np.all((m >= lo) & (m <= hi), axis=1)]
    return _rows64(_dev(q).double(), _dev(m).double(), case["k"], case["eps"], weights)
