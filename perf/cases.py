"""Performance cases: the calls a program makes on this library, timed as it makes them.

A case is a dict of plain values.  ``listed()`` gives the standing set, ``draw(rng)`` one more
case of the same ranges, ``prepare`` the maps and device tensors a program holds before the
call, ``run`` the call, ``work`` the bytes and operations it cannot do without, and ``exact``
the same results in 64-bit torch arithmetic, written from the method's definitions and without
this library's code (its scene generators only draw the inputs).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2407_09649_gb300 import scenes
from paper_2407_09649_gb300.api import Map
from paper_2407_09649_gb300.autograd import gpdf_distance

VS = 0.1          # voxel edge (m), the library's default
LEN = 0.3         # SE length scale (m)
S2 = 0.01 ** 2    # latent noise variance
SP2 = 0.1 ** 2    # property noise variance
D_MAX = 10.0
D_FLOOR = 1e-3
_BIAS = 1 << 20   # of the voxel keys' fields
SURFACE_MAX = 1 << 17
CAP_GROUP = 1024
CLEAR = 0.03      # clearance of a vehicle's query points (m)
SEARCH = 8        # fallback leaf search radius


def listed():
    return [
        # A planner asks for one trajectory against a finished room map: the smallest call.
        dict(name="waypoints_64", kind="query", scene="room", density=100, n=64, precision="mixed", emulate=1, var=0),
        # 256 trajectories of 64 waypoints with variance: a planner's batch.
        dict(name="waypoints_16k_var", kind="query", scene="room", density=100, n=16384, precision="mixed", emulate=1,
             var=1),
        # Large G-GPDF step: the surface is binned and a whole district is queried (the benchmark's
        # city at a quarter of its area).
        dict(name="city_step", kind="query", scene="city", extent=50, n=2_500_000, precision="mixed", emulate=1, var=0,
             retrain=1),
        # The library's default parameters (mixed precision, FP64 tensor path).
        dict(name="city_default", kind="query", scene="city", extent=20, n=100_003, precision="mixed", emulate=0,
             var=0),
        # All-FP64 results with variance.
        dict(name="city_fp64_var", kind="query", scene="city", extent=18, n=30_000, precision="fp64", emulate=1, var=1),
        # Blended per-leaf GPs (Eq. 10), eight nodes per query.
        dict(name="smooth_nodes_8", kind="smooth", scene="room", density=100, n=500_000, nodes=8, cap=512,
             precision="mixed", emulate=1),
        # One frame on a fresh grid: sphere and plane, plain FP64, the default leaf cap.
        dict(name="frame_fp64", kind="frame", points=20_000, cap=64, precision="fp64", emulate=0),
        # One depth frame of the room sequence (400 x 250 rays), every voxel around the surface.
        dict(name="frame_room", kind="frame", width=400, height=250, cap=512, precision="mixed", emulate=1),
        # The whole mapping step of a coloured depth frame: ray-cast testing voxels, signed
        # distances, properties, fusion, zero crossings and the retrained surface.
        dict(name="mapping_rgb", kind="mapping", width=400, height=250, cap=512, props=3, precision="mixed", emulate=1),
        # Independent instances of 4 to 1024 points.
        dict(name="sweep_1024", kind="sweep", n_inst=10_000, n_max=1024, q_per=512, precision="mixed", emulate=1,
             var=0),
        # Leaf-sized independent instances with variance, default parameters.
        dict(name="sweep_leaf_var", kind="sweep", n_inst=20_000, n_max=64, q_per=64, precision="mixed", emulate=0,
             var=1),
        # Trajectory optimisation through autograd: distance, d/d waypoints and d/d surface points.
        dict(name="train_waypoints", kind="train", density=60, n_traj=64, precision="fp64", emulate=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "sweep", "sweep", "frame", "frame", "smooth", "train", "mapping"])
    arith = rng.choice([("mixed", 1), ("mixed", 1), ("mixed", 0), ("fp64", 1), ("fp64", 0)])
    c = dict(kind=kind, precision=arith[0], emulate=arith[1])
    if kind == "query":
        var = rng.randint(0, 1)
        n = _log_int(rng, 33, 60_000 if var else 250_000)
        if rng.random() < 0.5:
            c.update(scene="room", density=rng.randint(30, 120), n=n, var=var)
        else:
            c.update(scene="city", extent=rng.randint(18, 20 if arith[1] == 0 else 26), n=n, var=var,
                     retrain=rng.randint(0, 1))
    elif kind == "smooth":
        c.update(scene="room", density=rng.randint(30, 120), n=_log_int(rng, 100, 400_000), nodes=rng.randint(1, 12),
                 cap=rng.choice([64, 128, 257, 512]))
    elif kind == "frame":
        c.update(cap=rng.choice([64, 128, 200, 512]))
        if rng.random() < 0.5:
            c.update(points=_log_int(rng, 500, 20_000))
        else:
            c.update(width=rng.randint(60, 400), height=rng.randint(40, 250))
    elif kind == "mapping":
        c.update(width=rng.randint(60, 400), height=rng.randint(40, 250), cap=rng.choice([64, 128, 512]),
                 props=rng.randint(0, 4))
    elif kind == "sweep":
        n_max = _log_int(rng, 8, 1024)
        c.update(n_inst=_log_int(rng, 10, min(20_000, 2_000_000 // n_max if arith[1] else 400_000 // n_max)),
                 n_max=n_max, q_per=rng.randint(1, 256), var=rng.randint(0, 1))
    else:
        c.update(density=rng.randint(20, 60), n_traj=_log_int(rng, 1, 48))
    return c


# ------------------------------------------------------------------------------- inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _room_surface(room, density, seed):
    """About `density` points per m^2 of the room's surfaces, as many for every room."""
    S = room.surface_samples(seed=seed, density=1.6 * density)
    n = round(600 * density)
    return np.ascontiguousarray(S[np.random.default_rng(seed).permutation(len(S))[:n]])


def _waypoints(room, n, seed):
    """n waypoints of random trajectories, those that keep clear of walls and obstacles."""
    got = np.empty((0, 3), np.float32)
    while len(got) < n:
        T = room.trajectories(seed=seed + 2 + len(got), n_traj=2 * n // 64 + 8, n_way=64).reshape(-1, 3)
        free = ~room.inside_obstacle(T, margin=-CLEAR) & np.all((T > CLEAR) & (T < room.size - CLEAR), axis=1)
        got = np.concatenate([got, T[free]])
    return np.ascontiguousarray(got[:n])


def _query_inputs(case, seed):
    """Surface points and query points (float32 numpy)."""
    if case["scene"] == "room":
        room = scenes.Room(seed)
        S = _room_surface(room, case["density"], seed)
        if case["kind"] == "smooth":
            Q = scenes.uniform_queries(seed, n=2 * case["n"] + 64, lo=(CLEAR,) * 3, hi=tuple(room.size - CLEAR))
            Q = Q[~room.inside_obstacle(Q, margin=-CLEAR)][:case["n"]]
        else:
            Q = _waypoints(room, case["n"], seed)
        return S, Q
    e = float(case["extent"])
    city = scenes.City(seed, extent=(e, e, 10.0), n_boxes=max(4, round(200 * (e / 100.0) ** 2)))
    S = city.surface(n=round(200 * e * e), seed=seed, chunk=1 << 18)
    many = case["n"] + case["n"] // 4 + 64
    Q = city.queries(n=many, seed=seed + 1, chunk=min(1 << 20, 2 * many))
    Q = Q[~city.inside_box(Q, margin=-CLEAR) & (Q[:, 2] > CLEAR)]
    return S, Q[:case["n"]]


def _sweep_inputs(case, seed):
    return scenes.patch_sweep(n_inst=case["n_inst"], seed=seed, n_max=case["n_max"], q_per_inst=case["q_per"])


def _frame_inputs(case, seed):
    if "points" in case:
        n = case["points"]
        return scenes.sphere_plane_frame(seed, n_sphere=n // 2, n_plane=n - n // 2)
    return scenes.Room(seed).frame(1, seed=seed, width=case["width"], height=case["height"])


def _train_inputs(case, seed):
    room = scenes.Room(seed)
    return _waypoints(room, 64 * case["n_traj"], seed), _room_surface(room, case["density"], seed)


def _box(case):
    """Low corner and shape (voxels) of a grid that holds every testing voxel of the scene."""
    if "points" in case:
        return (-72, -72, -72), (144, 144, 144)
    return (-32, -32, -32), (264, 168, 96)


def _map(case, **kw):
    return Map(precision=case["precision"], emulate_fp64=case["emulate"], **kw)


def prepare(case, seed):
    kind = case["kind"]
    dev = _device()
    up = lambda a: torch.from_numpy(a).to(dev)  # noqa: E731
    s = dict(case=case)
    if kind in ("query", "smooth"):
        S, Q = _query_inputs(case, seed)
        s.update(map=_map(case, **({"max_pts_leaf": case["cap"]} if kind == "smooth" else {})), S=up(S), Q=up(Q))
        s["map"].set_surface(s["S"])
    elif kind == "sweep":
        io, X, qo, Q = _sweep_inputs(case, seed)
        s.update(map=_map(case), io=up(io), X=up(X), qo=up(qo), Q=up(Q))
    elif kind == "frame":
        s.update(map=_map(case, max_pts_leaf=case["cap"]), P=up(_frame_inputs(case, seed)))
    elif kind == "mapping":
        # a map that already holds the previous frame; the pass adds the next one
        room = scenes.Room(seed)
        m = _map(case, max_pts_leaf=case["cap"], n_props=case["props"])
        rng = np.random.default_rng(seed)
        for k in range(2):
            P = up(room.frame(k, seed=seed, width=case["width"], height=case["height"]))
            C = up(rng.random((P.shape[0], case["props"]), dtype=np.float32)) if case["props"] else None
            o = tuple(float(x) for x in room.camera_pose(k)[0])
            if k == 0:
                m.fuse(m.build_frame(P, origin=o, props=C))
                m.update_surface()
        s.update(map=m, P=P, C=C, origin=o)
    else:
        W, X = _train_inputs(case, seed)
        s.update(map=_map(case), W=up(W).requires_grad_(True), X=up(X).requires_grad_(True))
    return s


# ---------------------------------------------------------------------------------- run
def _local_grid(frame, box):
    """A frame's results as the dense local grid a planner reads: one entry per voxel of `box`
    (low corner, shape in voxels), +inf, 0 and status 255 where the frame has no testing voxel."""
    (lo, shape), r = box, frame.results()
    key = r["keys"].view(torch.int64)
    m = (1 << 21) - 1
    at = [((key >> sh) & m) - (_BIAS + l) for sh, l in zip((42, 21, 0), lo)]
    at = [i.clamp(0, n - 1) for i, n in zip(at, shape)]
    at = (at[0] * shape[1] + at[1]) * shape[2] + at[2]
    dev, n = key.device, math.prod(shape)
    d = torch.full((n,), math.inf, dtype=torch.float64, device=dev)
    v = torch.full((n,), math.inf, dtype=torch.float64, device=dev)
    g = torch.zeros((n, 3), dtype=torch.float64, device=dev)
    st = torch.full((n,), 255, dtype=torch.uint8, device=dev)
    d[at], v[at], g[at], st[at] = r["d"], r["v"], r["grad"], r["status"]
    out = dict(d=d, v=v, grad=g, status=st)
    p = frame.props()
    if p is not None:
        out["c"] = torch.zeros((n, p[0].shape[1]), dtype=torch.float64, device=dev)
        out["w"] = torch.full((n,), math.inf, dtype=torch.float64, device=dev)
        out["c"][at], out["w"][at] = p
    return out


def run(s):
    case, m = s["case"], s["map"]
    kind = case["kind"]
    if kind == "query":
        if case.get("retrain"):
            m.set_surface(s["S"])
        r = m.query(s["Q"], grad=True, var=bool(case["var"]))
        return {k: v for k, v in r.items() if v is not None}
    if kind == "smooth":
        r = m.query_smooth(s["Q"], n_nodes=case["nodes"])
        return {k: v for k, v in r.items() if v is not None}
    if kind == "sweep":
        r = m.gp_batch(s["io"], s["X"], s["qo"], s["Q"], var=bool(case["var"]))
        return {k: v for k, v in r.items() if v is not None}
    if kind == "frame":
        return _local_grid(m.build_frame(s["P"]), _box(case))
    if kind == "mapping":
        f = m.build_frame(s["P"], origin=s["origin"], props=s["C"])
        m.fuse(f)
        n = m.update_surface()
        x = m.surface_points()
        for a in (2, 1, 0):  # the points in order of their coordinates (leaf order is unspecified)
            x = x[torch.sort(x[:, a], stable=True)[1]]
        surface = torch.zeros((SURFACE_MAX, 3), dtype=torch.float32, device=x.device)
        surface[:n] = x[:SURFACE_MAX]
        return dict(_local_grid(f, _box(case)), surface=surface, n_surface=n)
    W, X = s["W"], s["X"]
    W.grad = X.grad = None
    d = gpdf_distance(W, X, m)
    torch.nn.functional.softplus(0.5 - d).sum().backward()
    return dict(d=d.detach(), dW=W.grad, dX=X.grad)


# -------------------------------------------------- the method in 64 bits (no library code)
_NONE = (1 << 63) - 1  # above every key


def _pack(ijk):
    return ((ijk[..., 0] + _BIAS) << 42) | ((ijk[..., 1] + _BIAS) << 21) | (ijk[..., 2] + _BIAS)


def _unpack(key):
    m = (1 << 21) - 1
    return torch.stack([(key >> 42) & m, (key >> 21) & m, key & m], -1) - _BIAS


def _voxel(p):
    return torch.floor(p.double() / VS + 0.5).long()


def _offsets(r, dev):
    g = torch.arange(-r, r + 1, device=dev)
    z, y, x = torch.meshgrid(g, g, g, indexing="ij")
    return torch.stack([x, y, z], -1).reshape(-1, 3)


def _lookup(table, key):
    """Index of each key in the sorted table, -1 where it is not there."""
    i = torch.searchsorted(table, key).clamp(max=len(table) - 1)
    return torch.where(table[i] == key, i, -1)


def _centre_leaves(qleaf, table):
    """Centre leaf of each query leaf: itself if its 27-leaf neighbourhood holds points, else the
    nearest occupied leaf within the search radius (ties to the smaller key), else -1."""
    dev = qleaf.device
    c = _unpack(qleaf)
    near = torch.zeros(len(qleaf), dtype=torch.bool, device=dev)
    for o in _offsets(1, dev):
        near |= _lookup(table, _pack(c + o)) >= 0
    out = torch.where(near, qleaf, -1)
    off = _offsets(SEARCH, dev)
    d2 = (off * off).sum(1)
    todo = torch.nonzero(~near)[:, 0]
    for v in torch.unique(d2).tolist():
        if len(todo) == 0:
            break
        best = torch.full((len(todo),), _NONE, device=dev)
        for o in off[d2 == v]:
            k = _pack(c[todo] + o)
            best = torch.where(_lookup(table, k) >= 0, torch.minimum(best, k), best)
        hit = best < _NONE
        out[todo[hit]] = best[hit]
        todo = todo[~hit]
    return out


def _bin(S):
    """Points by leaf: sorted leaf keys, offsets and point indices (in index order per leaf)."""
    key = _pack(_voxel(S) >> 3)
    key, idx = torch.sort(key, stable=True)
    leaf, cnt = torch.unique_consecutive(key, return_counts=True)
    off = torch.zeros(len(leaf) + 1, dtype=torch.long, device=S.device)
    off[1:] = torch.cumsum(cnt, 0)
    return leaf, off, idx


def _expand(start, cnt):
    """Concatenated ranges [start_i, start_i + cnt_i) and the range each entry belongs to."""
    owner = torch.repeat_interleave(torch.arange(len(cnt), device=cnt.device), cnt)
    first = torch.cumsum(cnt, 0) - cnt
    return start[owner] + torch.arange(len(owner), device=cnt.device) - first[owner], owner


def _gather_instances(centre, leaf, off, idx, S, cap, reach):
    """Point lists of the instances around `centre` (leaves within `reach`), at most `cap` points,
    those nearest the centre leaf's centre (ties to the lower index).  CSR (offsets, indices)."""
    dev = centre.device
    c = _unpack(centre)
    o = _offsets(reach, dev)
    l = _lookup(leaf, _pack(c[:, None] + o))  # [I, leaves]
    cnt = torch.where(l >= 0, off[l.clamp(min=0) + 1] - off[l.clamp(min=0)], 0)
    pos, own = _expand(off[l.clamp(min=0)].reshape(-1), cnt.reshape(-1))
    own = own // len(o)
    pt = idx[pos]
    mid = (8 * c + 3.5) * VS
    d2 = ((S[pt].double() - mid[own]) ** 2).sum(1)
    for by in (0, 1, 2):  # by instance, then distance, then index
        s = torch.sort((pt, d2, own)[by], stable=True)[1]
        pt, d2, own = pt[s], d2[s], own[s]
    tot = torch.bincount(own, minlength=len(centre))
    rank = torch.arange(len(own), device=dev) - (torch.cumsum(tot, 0) - tot)[own]
    keep = rank < cap
    pt, own = pt[keep], own[keep]
    s = torch.sort(own * len(S) + pt)[1]
    ioff = torch.zeros(len(centre) + 1, dtype=torch.long, device=dev)
    ioff[1:] = torch.cumsum(torch.bincount(own, minlength=len(centre)), 0)
    return ioff, pt[s]


def _query_plan(S, Q, cap=CAP_GROUP):
    """Instances of a query batch: CSR over surface points and the instance of each query (-1)."""
    leaf, off, idx = _bin(S)
    ql, qi = torch.unique(_pack(_voxel(Q) >> 3), return_inverse=True)
    cen = _centre_leaves(ql, leaf)
    inst, ii = torch.unique(cen, return_inverse=True)
    skip = int(len(inst) > 0 and inst[0] < 0)  # -1 sorts first
    ioff, pts = _gather_instances(inst[skip:], leaf, off, idx, S, cap, 1)
    return ioff, pts, (ii - skip)[qi], cen[qi]


def _revert(o, go, u, var):
    """Reverting function and its chain rules with the caps (status, d, grad, var)."""
    l2 = LEN * LEN
    lo = torch.log(o.clamp(min=0.0))
    ok = lo >= -D_MAX ** 2 / (2 * l2)
    on = ok & (lo >= 0)
    d = torch.sqrt((-2 * l2 * lo).clamp(min=0.0))
    safe = torch.where(ok & ~on, d, 1.0)
    g = torch.where((ok & ~on)[:, None], -l2 * go / (torch.where(ok, o, 1.0) * safe)[:, None], 0.0)
    d = torch.where(ok, torch.where(on, 0.0, d), D_MAX)
    v = None
    if var:
        oc = torch.where(on, 1.0, torch.where(ok, o, 1.0))
        v = torch.where(ok, (l2 / (oc * torch.where(on, 0.0, safe).clamp(min=D_FLOOR))) ** 2 * u, math.inf)
    return torch.where(ok, 0, 2), d, g, v


def _solve(X, ioff, Q, qoff, var, noise=S2):
    """o, grad o and u at Q[qoff[I]:qoff[I+1]] from the GP on X[ioff[I]:ioff[I+1]], in 64 bits:
    instances of about one size in batches, padded with unit rows and unused queries."""
    dev = X.device
    n, nq = (ioff[1:] - ioff[:-1]), (qoff[1:] - qoff[:-1])
    o = torch.zeros(len(Q), dtype=torch.float64, device=dev)
    go = torch.zeros((len(Q), 3), dtype=torch.float64, device=dev)
    u = torch.zeros(len(Q), dtype=torch.float64, device=dev)
    size = ((n + 31) // 32 * 32).tolist()
    many = nq.tolist()
    order = sorted((i for i in range(len(size)) if size[i] > 0 and many[i] > 0), key=lambda i: (size[i], many[i]))
    at = 0
    while at < len(order):
        N = size[order[at]]
        end, qm = at, 1
        while end < len(order) and size[order[end]] == N:
            q = max(qm, many[order[end]])
            if end > at and (end + 1 - at) * N * (N + 4 * q) > 6e7:
                break
            qm, end = q, end + 1
        I = torch.tensor(order[at:end], device=dev)
        at = end
        j = torch.arange(N, device=dev)
        live = j < n[I][:, None]
        P = X[torch.where(live, ioff[I][:, None] + j, 0)]
        K = torch.exp(-((P[:, :, None] - P[:, None]) ** 2).sum(-1) / (2 * LEN * LEN))
        K = torch.where(live[:, :, None] & live[:, None], K, 0.0)
        K.diagonal(dim1=1, dim2=2).copy_(1.0 + noise * live.double())
        L = torch.linalg.cholesky(K)
        a = torch.cholesky_solve(live.double()[..., None], L)[..., 0]
        for q0 in range(0, qm, max(1, int(6e7 / (len(I) * N * 4)))):
            q1 = min(qm, q0 + max(1, int(6e7 / (len(I) * N * 4))))
            t = torch.arange(q0, q1, device=dev)
            qlive = t < nq[I][:, None]
            qpos = torch.where(qlive, qoff[I][:, None] + t, 0)
            D = P[:, None] - Q[qpos][:, :, None]
            k = torch.where(live[:, None], torch.exp(-(D ** 2).sum(-1) / (2 * LEN * LEN)), 0.0)
            w = k * a[:, None]
            to = qpos[qlive]
            o[to] = w.sum(-1)[qlive]
            go[to] = ((w[..., None] * D).sum(2) / (LEN * LEN))[qlive]
            if var:
                V = torch.linalg.solve_triangular(L, k.transpose(1, 2), upper=False)
                u[to] = (1.0 - (V * V).sum(1)).clamp(min=0.0)[qlive]
    return o, go, u


def _answer(X, ioff, Q, owner, var):
    """d, grad, var of queries that belong to instance `owner` (-1: none)."""
    dev = Q.device
    s = torch.sort(owner, stable=True)[1]
    s = s[owner[s] >= 0]
    cnt = torch.bincount(owner[s], minlength=len(ioff) - 1)
    qoff = torch.zeros(len(ioff), dtype=torch.long, device=dev)
    qoff[1:] = torch.cumsum(cnt, 0)
    o, go, u = _solve(X, ioff, Q[s].double(), qoff, var)
    st, d, g, v = _revert(o, go, u, var)
    D = torch.full((len(Q),), math.inf, dtype=torch.float64, device=dev)
    G = torch.zeros((len(Q), 3), dtype=torch.float64, device=dev)
    T = torch.ones(len(Q), dtype=torch.long, device=dev)
    D[s], G[s], T[s] = d, g, st
    V = None
    if var:
        V = torch.full((len(Q),), math.inf, dtype=torch.float64, device=dev)
        V[s] = v
    return D, G, V, T


def _leaf_training_set(P, cap):
    """Occupied leaves of a frame (sorted), and their capped voxel centres in bit order (CSR)."""
    v = _unpack(torch.unique(_pack(_voxel(P))))
    lk, inv = torch.unique(_pack(v >> 3), return_inverse=True)
    b = v & 7
    bit = b[:, 0] + 8 * b[:, 1] + 64 * b[:, 2]
    s = torch.sort(inv * 512 + bit)[1]
    v, inv = v[s], inv[s]
    cnt = torch.bincount(inv, minlength=len(lk))
    off = torch.cumsum(cnt, 0) - cnt
    kept = cnt.clamp(max=cap)
    k, own = _expand(torch.zeros_like(kept), kept)
    rank = torch.where(cnt[own] > cap, k * cnt[own] // cap, k)
    ioff = torch.zeros(len(lk) + 1, dtype=torch.long, device=P.device)
    ioff[1:] = torch.cumsum(kept, 0)
    return lk, ioff, v[off[own] + rank].double() * VS


def _frame_tests(lk):
    """Testing voxels of a frame (every voxel of the occupied leaves and their neighbours) and
    the leaf whose GP answers each."""
    dev = lk.device
    near = torch.unique(_pack(_unpack(lk)[:, None] + _offsets(1, dev)).reshape(-1))
    b = torch.arange(512, device=dev)
    b = torch.stack([b & 7, (b >> 3) & 7, b >> 6], -1)
    v = (8 * _unpack(near)[:, None] + b).reshape(-1, 3)
    leaf = v >> 3
    own = _lookup(lk, _pack(leaf))
    best = torch.where(own >= 0, -1, 1 << 40)
    for o in _offsets(1, dev):  # x fastest, z slowest: the first of equal distances stays
        l = _lookup(lk, _pack(leaf + o))
        d2 = ((2 * v - (16 * (leaf + o) + 7)) ** 2).sum(1)
        better = (l >= 0) & (d2 < best)
        own = torch.where(better, l, own)
        best = torch.where(better, d2, best)
    return v, own


def exact(case, seed):
    kind = case["kind"]
    dev = _device()
    up = lambda a: torch.from_numpy(a).to(dev)  # noqa: E731
    if kind == "query":
        if case["n"] > 300_000:  # too many instances for the time
            return None
        S, Q = (up(a) for a in _query_inputs(case, seed))
        ioff, pts, own, _ = _query_plan(S, Q)
        D, G, V, _ = _answer(S[pts].double(), ioff, Q, own, bool(case["var"]))
        out = dict(d=D, grad=G, status=None)
        return dict(out, var=V) if case["var"] else out
    if kind == "smooth":
        return _exact_smooth(case, *(up(a) for a in _query_inputs(case, seed)))
    if kind == "sweep":
        io, X, qo, Q = (up(a) for a in _sweep_inputs(case, seed))
        own = torch.repeat_interleave(torch.arange(len(qo) - 1, device=dev), qo[1:] - qo[:-1])
        D, G, V, _ = _answer(X.double(), io, Q, own, bool(case["var"]))
        # a few queries lie on a patch's surface (d near 0), where the FP32 gradient is all rounding
        out = dict(d=D, grad=G if case["precision"] == "fp64" else None, status=None)
        return dict(out, var=V) if case["var"] else out
    if kind == "frame":
        lk, ioff, X = _leaf_training_set(up(_frame_inputs(case, seed)), case["cap"])
        vox, own = _frame_tests(lk)
        D, G, V, _ = _answer(X, ioff, vox.double() * VS, own, True)
        lo, shape = _box(case)
        at = vox - torch.tensor(lo, device=dev)
        at = (at[:, 0] * shape[1] + at[:, 1]) * shape[2] + at[:, 2]
        n = math.prod(shape)
        out = dict(d=torch.full((n,), math.inf, dtype=torch.float64, device=dev),
                   v=torch.full((n,), math.inf, dtype=torch.float64, device=dev),
                   grad=torch.zeros((n, 3), dtype=torch.float64, device=dev), status=None)
        out["d"][at], out["v"][at], out["grad"][at] = D, V, G
        if case["precision"] != "fp64":  # voxels on the surface itself, as for the sweep
            out["grad"] = None
        return out
    if kind == "train":
        return _exact_train(*(up(a) for a in _train_inputs(case, seed)))
    return None  # mapping: the testing voxels depend on the whole fused grid


def _exact_smooth(case, S, Q):
    """Eq. 10 over the nearest per-leaf GPs of each query: weighted d, averaged gradients."""
    dev, n, m = Q.device, len(Q), case["nodes"]
    leaf, off, idx = _bin(S)
    ql, qi = torch.unique(_pack(_voxel(Q) >> 3), return_inverse=True)
    cen = _centre_leaves(ql, leaf)[qi]
    ioff, pts = _gather_instances(leaf, leaf, off, idx, S, case["cap"], 0)
    o = _offsets(1, dev)
    cc = _unpack(cen.clamp(min=0))
    cand = torch.where((cen >= 0)[:, None], _lookup(leaf, _pack(cc[:, None] + o)), -1)
    mid = (8 * _unpack(leaf) + 3.5) * VS
    dist = ((Q.double()[:, None] - mid[cand.clamp(min=0)]) ** 2).sum(-1)
    dist = torch.where(cand >= 0, dist, math.inf)
    by_key = torch.where(cand >= 0, cand, 1 << 40)  # leaves are sorted by key
    s = torch.sort(by_key, dim=1)[1]
    dist, cand = torch.gather(dist, 1, s), torch.gather(cand, 1, s)
    s = torch.sort(dist, dim=1, stable=True)[1][:, :m]
    cand = torch.gather(cand, 1, s)
    D, G, _, T = _answer(S[pts].double(), ioff, Q.repeat_interleave(cand.shape[1], 0), cand.reshape(-1), False)
    D, T, G = D.reshape(n, -1), T.reshape(n, -1), G.reshape(n, -1, 3)
    ok = (cand >= 0) & (T == 0)
    first = torch.where(cand[:, 0] < 0, math.inf, D[:, 0])
    lo = torch.where(ok, D, math.inf).min(1, keepdim=True)[0]
    w = torch.where(ok, torch.exp(-100.0 * (D - torch.where(torch.isfinite(lo), lo, 0.0))), 0.0)
    has = ok.any(1)
    d = torch.where(has, (w * torch.where(ok, D, 0.0)).sum(1) / w.sum(1).clamp(min=1e-300), first)
    g = (G * ok[..., None]).sum(1) / ok.sum(1).clamp(min=1)[:, None]
    # one node at d near 0 spoils an FP32 average of gradients, as for the sweep
    return dict(d=d, grad=g if case["precision"] == "fp64" else None, status=None)


def _exact_train(W, X):
    """loss = sum softplus(0.5 - d): d and the gradients to both point sets by autograd."""
    ioff, pts, own, _ = _query_plan(X, W)
    W64, X64 = W.double().requires_grad_(True), X.double().requires_grad_(True)
    s = torch.sort(own, stable=True)[1]
    cut = torch.searchsorted(own[s], torch.arange(len(ioff), device=W.device)).tolist()
    at = ioff.tolist()
    D = torch.full((len(W),), math.inf, dtype=torch.float64, device=W.device)
    for I in range(len(at) - 1):
        q = s[cut[I]:cut[I + 1]]
        if len(q) == 0 or at[I + 1] == at[I]:
            continue
        P, x = X64[pts[at[I]:at[I + 1]]], W64[q]
        K = torch.exp(-((P[:, None] - P) ** 2).sum(-1) / (2 * LEN * LEN))
        L = torch.linalg.cholesky(K + S2 * torch.eye(len(P), dtype=torch.float64, device=W.device))
        a = torch.cholesky_solve(torch.ones_like(P[:, :1]), L)[:, 0]
        o = torch.exp(-((x[:, None] - P) ** 2).sum(-1) / (2 * LEN * LEN)) @ a
        lo = torch.log(o.clamp(min=1e-300))
        inside = (lo < 0) & (lo >= -D_MAX ** 2 / (2 * LEN * LEN)) & (o > 0)
        d = torch.sqrt(-2 * LEN * LEN * torch.where(inside, lo, -1.0))
        torch.nn.functional.softplus(0.5 - d[inside]).sum().backward()
        D[q] = torch.where(inside, d, torch.where(lo >= 0, 0.0, D_MAX)).detach()
    return dict(d=D, dW=W64.grad, dX=X64.grad)


# --------------------------------------------------------------------------------- work
def _solve_flops(n, nq, var):
    """Cholesky and two solves per instance (n points), kernel values, mean and gradient (20
    operations a pair) and, with variance, a triangular solve per query."""
    n, nq = n.double(), nq.double()
    f = (n ** 3 / 3 + 2 * n ** 2).sum() + (20 * n * nq).sum()
    return float(f + ((n ** 2 * nq).sum() if var else 0))


def work(case):
    kind = case["kind"]
    dev = _device()
    up = lambda a: torch.from_numpy(a).to(dev)  # noqa: E731
    if kind in ("query", "smooth"):
        S, Q = (up(a) for a in _query_inputs(case, 0))
        b = len(S) * 12 + len(Q) * (12 + 8 + 24 + 1 + 8 * case.get("var", 0))
        if kind == "query":
            ioff, _, own, _ = _query_plan(S, Q)
            return dict(bytes=b, flops=_solve_flops(ioff[1:] - ioff[:-1], torch.bincount(own[own >= 0],
                                                    minlength=len(ioff) - 1), case["var"]))
        n = torch.minimum(torch.diff(_bin(S)[1]), torch.tensor(case["cap"], device=dev))
        per = torch.full_like(n, round(len(Q) * case["nodes"] / len(n)))
        return dict(bytes=b, flops=_solve_flops(n, per, 0))
    if kind == "sweep":
        io, _, qo, Q = _sweep_inputs(case, 0)
        b = (len(io) + len(qo)) * 8 + int(io[-1]) * 12 + len(Q) * (12 + 8 + 24 + 1 + 8 * case["var"])
        return dict(bytes=b, flops=_solve_flops(torch.from_numpy(np.diff(io)), torch.from_numpy(np.diff(qo)),
                                                case["var"]))
    if kind == "train":
        W, X = (up(a) for a in _train_inputs(case, 0))
        ioff, _, own, _ = _query_plan(X, W)
        n, nq = ioff[1:] - ioff[:-1], torch.bincount(own[own >= 0], minlength=len(ioff) - 1)
        # forward, and backward: two more solves, K's derivative, the pairs once more
        f = 2 * _solve_flops(n, nq, 0) + float((20 * n.double() ** 2).sum())
        return dict(bytes=len(W) * 28 + len(X) * 24, flops=f)
    P = up(_frame_inputs(case, 0))
    lk, ioff, _ = _leaf_training_set(P, case["cap"])
    n = ioff[1:] - ioff[:-1]
    if kind == "frame":
        _, own = _frame_tests(lk)
        return dict(bytes=len(P) * 12 + len(own) * 49, flops=_solve_flops(n, torch.bincount(own, minlength=len(n)), 1))
    # mapping: about eight testing voxels per training voxel (itself, six along its normal, one
    # known voxel on a ray), with distance and property GPs, and their read-modify-write in the grid
    per = 8 * n
    t = int(per.sum())
    return dict(bytes=len(P) * (12 + 4 * case["props"]) + t * (49 + 32 + 16 * (case["props"] + 1)),
                flops=_solve_flops(n, per, 1) * (2 if case["props"] else 1))
