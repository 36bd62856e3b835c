"""The solve's routes: clusters of CTAs on one instance, chunked queries, launch shapes chosen by the
number of instances and queries, and the smallest instances on a stream of their own.

Which of them answers a query depends on what else is in the batch and must not show in the
result, so the routes are compared bit for bit; the plain FP64 kernels at the edges of their tiles
and buckets are compared with the oracle at the FP64 contract (|dd| <= 1e-4 m, gradient
angle <= 0.1 deg, variance 1e-5 relative).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

KEYS = ("d", "grad", "var", "status")


@pytest.fixture(scope="module")
def vg():
    import paper_2407_09649_gb300 as P
    P.build()
    from paper_2407_09649_gb300 import api
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return api


def _instances(sizes, nq, seed):
    """Points at a density that keeps |K| well conditioned, nq queries around each instance."""
    rng = np.random.default_rng(seed)
    X, Q = [], []
    for N in sizes:
        c = rng.uniform(-20, 20, 3)
        X.append((c + rng.uniform(-0.05, 0.05, (N, 3)) * np.sqrt(N)).astype(np.float32))
        Q.append((c + rng.uniform(-1, 1, (nq, 3))).astype(np.float32))
    return X, Q


def _solve(m, X, Q, var):
    io = np.concatenate([[0], np.cumsum([len(x) for x in X])])
    qo = np.concatenate([[0], np.cumsum([len(q) for q in Q])])
    out = m.gp_batch(io, np.vstack(X), qo, np.vstack(Q), var=var)
    out = {k: out[k].cpu().numpy() for k in KEYS if out[k] is not None}
    return [{k: v[a:b] for k, v in out.items()} for a, b in zip(qo, qo[1:])]


def _same(a, b):
    for k in a:
        x, y = (np.ascontiguousarray(t[k]).view(np.uint8) for t in (a, b))
        assert np.array_equal(x, y), k


@pytest.mark.parametrize("var", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_clusters_do_not_show(vg, precision, var):
    """Eight, four, two CTAs per instance and one: 1, 40, 100 and 400 instances at the edges of the
    32-column blocks and 128-row bands, among them the largest size and one bad query."""
    sizes = [129, 160, 161, 225, 256, 257, 1000, 1024]
    X, Q = _instances(sizes, 5, 51)
    Q[3][2] = np.nan
    m = vg.Map(precision=precision, emulate_fp64=1)
    small, qs = _instances([130] * 392, 1, 52)
    ref = _solve(m, X + small, Q + qs, var)[:len(sizes)]
    assert (ref[3]["status"] == 3).tolist() == [False, False, True, False, False]
    for n in (0, 32, 92):
        for a, b in zip(_solve(m, X + small[:n], Q + qs[:n], var), ref):
            _same(a, b)
    for x, q, r in zip(X, Q, ref):
        _same(_solve(m, [x], [q], var)[0], r)


@pytest.mark.parametrize("emulate,sizes,n_fill", [(1, [33, 40, 300], 0), (0, [20, 33, 64, 65], 0), (0, [225, 231, 260], 1300)])
@pytest.mark.parametrize("var", [False, True])
def test_chunks_and_shapes_do_not_show(vg, emulate, sizes, n_fill, var):
    """Instances with 3000 queries, which are split over work items, against 24 of the same
    queries on their own; and few large instances against the same ones in a batch of more than
    eight per SM (three smaller CTAs per SM)."""
    X, Q = _instances(sizes, 3000, 53)
    fill, qf = _instances([226] * n_fill, 1, 54)
    for precision in ("fp64", "mixed"):
        m = vg.Map(precision=precision, emulate_fp64=emulate)
        full = _solve(m, X + fill, Q + qf, var)
        part = _solve(m, X, [q[::125] for q in Q], var)
        for f, p in zip(full, part):
            _same({k: v[::125] for k, v in f.items()}, p)


def test_smallest_instances_follow_their_stream(vg):
    """Instances of at most 32 points run beside the others on a stream of the map's own: inputs that
    the caller's stream writes late are seen, and what it does next sees the results."""
    X, Q = _instances([8] * 50 + [150] * 50, 40, 55)
    m = vg.Map(precision="fp64")
    ref = _solve(m, X, Q, True)
    io = torch.from_numpy(np.concatenate([[0], np.cumsum([len(x) for x in X])])).cuda()
    qo = torch.arange(len(Q) + 1, dtype=torch.int64, device="cuda") * 40
    xs, qs = (torch.from_numpy(np.vstack(a)).cuda() for a in (X, Q))
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        busy = torch.zeros((8192, 8192), device="cuda")
        x, q = torch.zeros_like(xs), torch.zeros_like(qs)
        for _ in range(4):
            busy = busy @ busy
        x.copy_(xs)
        q.copy_(qs)
        out = m.gp_batch(io, x, qo, q, var=True)
        got = {k: out[k].clone() for k in KEYS}
        for t in [x, q] + [out[k] for k in KEYS]:
            t.zero_()
    s.synchronize()
    want = {k: np.concatenate([r[k] for r in ref]) for k in KEYS}
    _same({k: v.cpu().numpy() for k, v in got.items()}, want)


def test_plain_kernels_at_tile_edges(vg, orc):
    sizes = [1, 7, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 224, 225, 232, 233]
    X, Q = _instances(sizes, 30, 56)
    io = np.concatenate([[0], np.cumsum(sizes)])
    qo = np.arange(len(sizes) + 1) * 30
    ref = orc.gp_batch(io, np.vstack(X).astype(np.float64), qo, np.vstack(Q).astype(np.float64), orc.params())
    out = _solve(vg.Map(precision="fp64", emulate_fp64=0), X, Q, True)
    d, g, v, s = (np.concatenate([o[k] for o in out]) for k in KEYS)
    assert np.array_equal(s, ref.status)
    ok = ref.status == 0
    assert np.abs(d[ok] - ref.d[ok]).max() <= 1e-4
    na, nb = np.linalg.norm(g, axis=1), np.linalg.norm(ref.grad, axis=1)
    big = ok & (nb > 0.1)
    cos = np.sum(g * ref.grad, 1)[big] / (na * nb)[big]
    assert np.degrees(np.arccos(np.clip(cos, -1, 1))).max() <= 0.1
    fin = ok & np.isfinite(ref.var)
    np.testing.assert_allclose(v[fin], ref.var[fin], rtol=1e-5, atol=1e-12)


@pytest.mark.parametrize("n_nodes,lam", [(1, 100.0), (27, 2000.0), (27, 1e-3)])
def test_blend_weights_at_their_range(vg, orc, n_nodes, lam):
    """Blend weights exp(-lambda (d - d_min)) from underflow to all but equal, one node and every
    node of the neighbourhood, queries at leaf corners (ties between nodes) among them."""
    from paper_2407_09649_gb300 import scenes
    rng = np.random.default_rng(57)
    surf = scenes.sphere_plane_frame(4, n_sphere=2000, n_plane=2000).astype(np.float32)
    q = (surf[rng.integers(0, len(surf), 600)] + rng.normal(0, 0.1, (600, 3))).astype(np.float32)
    P = orc.params()
    q[:100] = np.round(q[:100] / 0.8) * 0.8
    ref = orc.Surface(surf, P).query_smooth(q, n_nodes=n_nodes, lam=lam, want_var=False)
    m = vg.Map(precision="fp64")
    m.set_surface(torch.from_numpy(surf).cuda())
    out = {k: v.cpu().numpy() for k, v in m.query_smooth(torch.from_numpy(q).cuda(), n_nodes=n_nodes, lam=lam).items()
           if v is not None}
    assert np.array_equal(out["status"], ref["status"])
    ok = ref["status"] == 0
    assert ok.sum() > 100
    assert np.abs(out["d"][ok] - ref["d"][ok]).max() <= 1e-4


@pytest.mark.parametrize("sizes,nq", [([240] + [100] * 200 + [20] * 40, [4000] + [40] * 240),
                                      ([1000] * 2 + [200] * 2000 + [8] * 100, [300] * 2 + [24] * 2000 + [300] * 100)])
def test_workspaces_grow_beside_the_smallest(vg, sizes, nq):
    """The first call of a map whose few large instances need less workspace than the many of the next
    size, with instances of at most 32 points on the map's stream beside them: no launch may be
    given memory that another one still uses."""
    X, Q = _instances(sizes, max(nq), 58)
    Q = [q[:k] for q, k in zip(Q, nq)]
    ref = vg.Map(precision="fp64", emulate_fp64=0)
    want = []
    for n in sorted(set(sizes), reverse=True):  # one size at a time: one launch, nothing beside it
        pick = [i for i, s in enumerate(sizes) if s == n]
        want += _solve(ref, [X[i] for i in pick], [Q[i] for i in pick], True)
    for _ in range(3):
        for a, b in zip(_solve(vg.Map(precision="fp64", emulate_fp64=0), X, Q, True), want):
            _same(a, b)


def test_caller_waits_for_the_smallest(vg):
    """The smallest instances take far longer than the one beside them, on a map that has run nothing
    before: what the caller's stream does next sees their results."""
    sizes = [40] + [32] * 6000
    X, Q = _instances(sizes, 200, 59)
    io = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)])).cuda()
    qo = torch.arange(len(Q) + 1, dtype=torch.int64, device="cuda") * 200
    x, q = (torch.from_numpy(np.vstack(a)).cuda() for a in (X, Q))
    ref = vg.Map(precision="fp64", emulate_fp64=0)
    want = [_solve(ref, X[a:b], Q[a:b], True) for a, b in ((0, 1), (1, len(sizes)))]
    want = {k: np.concatenate([r[k] for part in want for r in part]) for k in KEYS}
    for m in (vg.Map(precision="fp64", emulate_fp64=0), ref):
        out = m.gp_batch(io, x, qo, q, var=True)
        got = {k: out[k].clone() for k in KEYS}
        for k in KEYS:
            out[k].zero_()
        torch.cuda.synchronize()
        _same({k: v.cpu().numpy() for k, v in got.items()}, want)


def test_work_items_of_many_instances(vg):
    """More instances than the planning CTA has threads, with none to 3000 queries each: every query is
    answered, call after call, as in batches that are planned in one pass."""
    rng = np.random.default_rng(60)
    sizes = rng.integers(33, 65, 2500)
    X, Q = _instances(sizes, 0, 60)
    nq = np.where(rng.random(2500) < 0.02, 3000, rng.integers(0, 60, 2500))
    Q = [(x[0] + rng.uniform(-1, 1, (k, 3))).astype(np.float32) for x, k in zip(X, nq)]
    for emulate in (0, 1):
        m = vg.Map(precision="mixed", emulate_fp64=emulate)
        want = [r for a in range(0, 2500, 500) for r in _solve(m, X[a:a + 500], Q[a:a + 500], True)]
        for _ in range(3):
            for a, b in zip(_solve(m, X, Q, True), want):
                _same(a, b)


@pytest.mark.parametrize("precision,nc,raycast", [("fp64", 4, False), ("mixed", 3, True), ("mixed", 1, False)])
def test_voxel_frames_with_properties_in_clusters(vg, orc, precision, nc, raycast):
    """Frames of one to five leaves of 129 to 512 points, whose distance and property GPs clusters of CTAs
    work on: the oracle's values, and the same bits as in a frame of so many other leaves that each
    instance has one CTA."""
    rng = np.random.default_rng(61)
    leaves = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [6, 0, 0], [0, -6, 2]])
    keep = [512, 129, 256, 300, 161]
    origin = np.array([0.4, 0.4, 3.0]) if raycast else None
    vox = [8 * L + np.stack(np.unravel_index(rng.permutation(512)[:k], (8, 8, 8)), 1) for L, k in zip(leaves, keep)]
    far = np.array([[8 * (20 + 4 * i), 8 * 4 * j, 0] for i in range(12) for j in range(12)])
    far = (far[:, None] + np.stack(np.meshgrid(np.arange(8), np.arange(8), [3, 4]), -1).reshape(1, -1, 3)).reshape(-1, 3)
    pr = lambda v: (0.5 + 0.4 * np.sin(0.13 * v @ np.array([[1.0, 2, 3, 1], [2, 1, 0, 3], [0, 3, 1, 2]]))[:, :nc]).astype(np.float32)

    def frame(v):
        m = vg.Map(precision=precision, max_pts_leaf=512, n_props=nc, emulate_fp64=1)
        pts = torch.from_numpy((v * 0.1).astype(np.float32)).cuda()
        f = m.build_frame(pts, origin=origin, props=torch.from_numpy(pr(v)).cuda())
        r = {k: t.cpu().numpy() for k, t in f.results().items()}
        c, w = (t.cpu().numpy() for t in f.props())
        return {int(k): i for i, k in enumerate(r["keys"])}, (r["d"], r["v"], r["grad"], c, w)

    for n in (1, 2, 5):
        v = np.concatenate(vox[:n])
        at, val = frame(v)
        if n < 5 and not raycast:  # eight and two CTAs each (rays to the far leaves would add voxels here)
            many, ref = frame(np.concatenate([v, far]))
            pick = [many[k] for k in at]
            for a, b in zip(val, ref):
                assert np.array_equal(np.ascontiguousarray(a).view(np.uint8), np.ascontiguousarray(b[pick]).view(np.uint8))
        want = orc.frame((v * 0.1).astype(np.float32), orc.params(max_pts_leaf=512, n_props=nc), origin=origin, props=pr(v))
        assert len(at) == len(want.test_key)
        pick = [at[int(k)] for k in want.test_key]
        fin = np.isfinite(want.w)
        assert fin.any() and np.array_equal(np.isfinite(val[4][pick]), fin)
        # (property values as in the property tests: linear in the data, solved in FP64 on both sides)
        assert np.abs(val[3][pick][fin] - want.c[fin]).max() <= 1e-8
        assert np.abs(val[4][pick][fin] - want.w[fin]).max() <= 1e-8
        if precision == "fp64":
            ok = want.status == 0
            assert np.abs(val[0][pick][ok] - want.d[ok]).max() <= 1e-4


@pytest.mark.parametrize("threads", [640, 672, 768, 1024])
def test_largest_launch_shapes(vg, threads):
    """Every shape that vgp_set_launch takes runs, in each kernel and launch mode that uses it."""
    rng = np.random.default_rng(62)
    surf = rng.uniform(-1, 1, (9000, 3)).astype(np.float32) * [1, 1, 0.4]
    q = torch.from_numpy(rng.uniform(-1, 1, (600, 3)).astype(np.float32)).cuda()
    surf = torch.from_numpy(surf.astype(np.float32)).cuda()
    gd = torch.from_numpy(rng.uniform(-1, 1, 600)).cuda()
    X, Q = _instances([9, 40, 100, 200, 300], 30, 62)
    ref = None
    for launch, chosen in (("batched", None), ("batched", threads), ("graph", threads)):
        m = vg.Map(precision="fp64", launch=launch, max_pts_leaf=256, n_props=1)
        if chosen:
            m.set_launch([threads] * 5, [0] * 5, 1)
        m.set_surface(surf)
        out = [v.cpu().numpy() for v in m.query(q, grad=True, var=True).values()]
        dq, dX = m.query_backward(q, gd)
        out += [dq.cpu().numpy()] + [v for r in _solve(m, X, Q, True) for v in r.values()]
        f = m.build_frame(surf, props=surf[:, :1].contiguous())
        out += [v.cpu().numpy() for v in f.results().values()] + [v.cpu().numpy() for v in f.props()]
        if ref is None:
            ref, ref_x = out, dX
            continue
        for a, b in zip(out[:-7], ref[:-7]):
            assert np.array_equal(np.ascontiguousarray(a).view(np.uint8), np.ascontiguousarray(b).view(np.uint8))
        # testing voxels come in an order of their own
        oa, ob = (np.argsort(o[-7], kind="stable") for o in (out, ref))
        for a, b in zip(out[-7:], ref[-7:]):
            assert np.array_equal(np.ascontiguousarray(a[oa]).view(np.uint8), np.ascontiguousarray(b[ob]).view(np.uint8))
        # (each point's sum of two parts per instance, by atomics in any order: 54 terms at most, which
        # may exceed their sum by 1e4)
        assert (dX - ref_x).abs().max().item() <= 1e-9 * ref_x.abs().max().item()


@pytest.mark.parametrize("launch", ["batched", "graph", "per_instance"])
def test_stats_tell_the_shapes_launched(vg, launch):
    """Defaults, shapes that follow from the batch, pinned shapes, the emulated kernel's own."""
    def shapes(m, sizes, nq, var):
        _solve(m, *_instances(sizes, nq, 63), var)
        st = m.stats()
        return st["cfg_threads"], st["cfg_per_sm"], st["cfg_stage_panel"]

    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    dflt = [512, 512, 256, 128, 64]
    follow = launch == "batched"  # (only these launches know their counts)
    m = vg.Map(precision="fp64", launch=launch)
    assert shapes(m, [300, 40, 8], 4, True) == (dflt, [1, 0, 0, 0, 0], 1)
    many = [226] * (8 * n_sm + 1)
    want = ([256] + dflt[1:], [3, 0, 0, 0, 0], 0)
    assert shapes(m, many, 1, False) == (want if follow else (dflt, [1, 0, 0, 0, 0], 1))
    want = (dflt[:3] + [256, 64], [1, 0, 0, 0, 0], 1)
    assert shapes(m, [40], 600, True) == (want if follow else (dflt, [1, 0, 0, 0, 0], 1))
    if launch == "per_instance":
        return
    m.set_launch([384, 1024, 96, 32, 128], [2, 0, 1, 0, 3], 0)
    assert shapes(m, [300, 200, 100, 40, 8], 4, True) == ([384, 640, 96, 32, 128], [2, 0, 1, 0, 3], 0)
    e = vg.Map(precision="fp64", launch=launch, emulate_fp64=1)
    got = shapes(e, [300], 4, True)
    assert got[0][0] == 256 and got[1][0] == 0 and got[2] == 0


def _best_ms(m, sizes):
    X, Q = _instances(sizes, 5, 64)
    io = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)])).cuda()
    qo = torch.arange(len(sizes) + 1, dtype=torch.int64, device="cuda") * 5
    x, q = (torch.from_numpy(np.vstack(a)).cuda() for a in (X, Q))
    ms = []
    for _ in range(40):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        m.gp_batch(io, x, qo, q, var=False)
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    return min(ms)


@pytest.mark.parametrize("per_sm", [4, 2])
def test_clusters_all_run_at_once(vg, per_sm):
    """As many instances as clusters of eight (four) would fill the GPU's CTAs with: not all of those
    clusters run at once, and a second round must not make the call slower than one more instance does,
    with smaller clusters (1.5 times as slow, had it one)."""
    n = torch.cuda.get_device_properties(0).multi_processor_count // per_sm
    m = vg.Map(precision="mixed", emulate_fp64=1)
    assert _best_ms(m, [130] * n) <= 1.2 * _best_ms(m, [130] * (n + 1))


def test_small_instances_follow_in_a_second_round(vg):
    """The same number with a few large ones: the small ones beyond the clusters of eight that run at once
    end before the large ones do, which smaller clusters would make 1.4 times as long."""
    n = torch.cuda.get_device_properties(0).multi_processor_count // 4
    m = vg.Map(precision="mixed", emulate_fp64=1)
    assert _best_ms(m, [1024] * 4 + [300] * (n - 4)) <= 1.15 * _best_ms(m, [1024] * 4 + [300] * (n - 8))


def test_autotuner_chooses_for_the_buckets_it_timed(vg):
    """Neighbourhoods above 224 points only: that bucket is timed and chosen, the others keep the rules
    that follow the batch, and an emulated map, whose kernel has one shape there, keeps the defaults."""
    rng = np.random.default_rng(65)
    surf = torch.from_numpy((rng.uniform(-1, 1, (40000, 3)) * [2, 2, 0.2]).astype(np.float32)).cuda()
    q = (torch.from_numpy((rng.uniform(-1, 1, (2000, 3)) * [1.5, 1.5, 0.2]).astype(np.float32))).cuda()
    dflt = [512, 512, 256, 128, 64]
    for emulate in (0, 1):
        m = vg.Map(precision="mixed", emulate_fp64=emulate)
        m.set_surface(surf)
        m.query(q)
        assert m.stats()["bucket_count"][:3] == [0, 0, 0]
        cfg = m.autotune(q)
        assert cfg["bucket_ms"][0] > 0 and cfg["bucket_ms"][1:] == [0, 0, 0, 0]
        assert cfg["threads"][1:] == dflt[1:] and (not emulate or cfg["threads"][0] == dflt[0])
        if not emulate:
            _solve(m, *_instances([40], 600, 65), True)
            assert m.stats()["cfg_threads"][3] == 256
            assert (m.stats()["cfg_threads"][0], m.stats()["cfg_stage_panel"]) == (cfg["threads"][0], cfg["stage_panel"])
            _solve(m, *_instances([226] * 1300, 1, 65), False)
            assert m.stats()["cfg_threads"][0] == cfg["threads"][0]


def test_graph_workspaces_follow_the_batch(vg):
    """Graph launches size their CTAs and workspaces before the counts are known, but not beyond the
    batch: three instances with variance took 5 GB; later calls of more give the direct launches' bits."""
    m = vg.Map(precision="mixed", emulate_fp64=1, launch="graph")
    direct = vg.Map(precision="mixed", emulate_fp64=1)
    sizes, nq = [300, 40, 8], 5
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        X, Q = _instances(sizes, nq, 66)
        out = _solve(m, X, Q, True)
        torch.cuda.synchronize()
        if nq == 5:  # a CTA's rows are 1024 and the variance's 1024: 17 MB, and 8 of them at most
            assert free - torch.cuda.mem_get_info()[0] < 1 << 29
        for a, b in zip(out, _solve(direct, X, Q, True)):
            _same(a, b)
        sizes, nq = [33, 65, 129, 225, 300, 1024] * 20, 700


@pytest.mark.parametrize("emulate,sizes", [(0, [8]), (1, [8]), (0, [300, 40, 8])])
def test_kernels_of_a_small_call(vg, emulate, sizes):
    """A mean-only call of a few small instances plans no work items, so it is four kernels (points and
    centres, sizes, two for the order) and a launch for each bucket."""
    from paper_2407_09649_gb300 import _lib
    lib = _lib.load()
    m = vg.Map(precision="mixed", emulate_fp64=emulate)
    X, Q = _instances(sizes, 8, 67)
    _solve(m, X, Q, False)
    n0 = lib.vgp_launch_count()
    _solve(m, X, Q, False)
    assert lib.vgp_launch_count() - n0 == 4 + len(sizes)


def test_work_items_are_counted_by_instance(vg):
    """Queries that no instance has enough of for two work items are not planned as such, however many they
    are together: no planning kernel."""
    from paper_2407_09649_gb300 import _lib
    lib = _lib.load()
    m = vg.Map(precision="mixed", emulate_fp64=1)
    X, Q = _instances([130] * 75, 100, 68)
    _solve(m, X, Q, True)
    n0 = lib.vgp_launch_count()
    _solve(m, X, Q, True)
    assert lib.vgp_launch_count() - n0 == 5
    n0 = lib.vgp_launch_count()
    _solve(m, X, Q[:74] + [np.concatenate([Q[74]] * 2)], True)  # 200 queries: two items of 130 at most
    assert lib.vgp_launch_count() - n0 == 6


@pytest.mark.parametrize("launch", ["batched", "graph"])
@pytest.mark.parametrize("sizes,nq", [([1000] + [40] * 300, 5), ([1000] * 8, 20000)])
def test_short_memory_takes_fewer_workspaces(vg, launch, sizes, nq):
    """A workspace for every CTA of the GPU would take 5 GB; with 1.5 GB left fewer CTAs share the work, as
    they did when each size had its own launch, and the bits are the same."""
    import gc
    X, Q = _instances(sizes, nq, 69)
    want = _solve(vg.Map(precision="mixed", emulate_fp64=1, launch=launch), X, Q, True)
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    m = vg.Map(precision="mixed", emulate_fp64=1, launch=launch)
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (3 << 29), dtype=torch.uint8, device="cuda")
    got = _solve(m, X, Q, True)
    del fill
    torch.cuda.empty_cache()
    for a, b in zip(got, want):
        _same(a, b)
