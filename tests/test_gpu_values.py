"""Device arithmetic at the edges of its range: the paired exponential, both halves of the packed
float-pair kernel values, the sign test of zero crossings."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vg():
    import paper_2407_09649_gb300 as P
    P.build()
    return P


def _ptr(t):
    return C.c_void_p(t.data_ptr())


def _stream():
    return C.c_void_p(torch.cuda.current_stream().cuda_stream)


def test_paired_exp_below_its_bound(vg):
    """The exponential of Eq. 10's weights and of the backward pass: below 0.85 ulp (half an ulp of the
    last sum, r^5 / 120 <= 0.342 ulp for |r| <= ln2 / 512, the reduction's 0.006), the library's
    values below -700."""
    from paper_2407_09649_gb300 import _lib
    m = vg.Map()
    rng = np.random.default_rng(70)
    mid = -(np.arange(1, 5000) + 0.5) * np.log(2) / 256  # |r| at its largest
    y = np.concatenate([-rng.uniform(0, 40, 1000000), -rng.uniform(0, 700, 300000), mid, np.nextafter(mid, 0),
                        [-0.0, 0.0, -5e-324, -1e-300, -1e-17, -699.999, -700.0]])
    yt = torch.from_numpy(y).cuda()
    out = torch.empty_like(yt)
    _lib.check(_lib.load().vgp_debug_exp_near(m._h, _ptr(yt), _ptr(out), len(y), _stream()))
    got = out.cpu().numpy()
    ref = np.exp(y.astype(np.longdouble))
    err = np.abs(got.astype(np.longdouble) - ref) / np.spacing(ref.astype(np.float64))
    assert float(err.max()) <= 0.85
    assert np.all(got[y == 0.0] == 1.0)
    far = torch.tensor([-np.nextafter(700.0, 800.0), -740.0, -800.0, -np.inf, np.nan], device="cuda", dtype=torch.float64)
    out = torch.empty_like(far)
    _lib.check(_lib.load().vgp_debug_exp_near(m._h, _ptr(far), _ptr(out), len(far), _stream()))
    assert torch.equal(out[:4], torch.exp(far[:4])) and torch.isnan(out[4])


def test_both_halves_of_packed_kernel_values(vg):
    """An entry's bits do not depend on the half it is computed in nor on the other half's entry, from
    coincident points to values beyond the fixed point's range."""
    from paper_2407_09649_gb300 import _lib
    m = vg.Map(precision="mixed", emulate_fp64=1)
    rng = np.random.default_rng(71)
    n = 100001
    xa = (np.array([103.7, -45.3, 12.9]) + rng.uniform(-1.5, 1.5, (n, 3))).astype(np.float32)
    xb = (xa + rng.normal(size=(n, 3)) * 10.0 ** rng.uniform(-6, 1.5, (n, 1))).astype(np.float32)
    xb[::7] = xa[::7]

    def run(a, b):
        ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        out = torch.empty(len(a), dtype=torch.int64, device="cuda")
        _lib.check(_lib.load().vgp_debug_kernel_fix(m._h, _ptr(ta), _ptr(tb), len(a), _ptr(out), _stream()))
        return out.cpu().numpy()

    got = run(xa, xb)
    assert np.all(got[::7] == 2**61) and np.any(got == 0)
    assert np.array_equal(run(xa[1:].copy(), xb[1:].copy()), got[1:])  # every entry in the other half
    L = np.longdouble
    y = np.sum((xa.astype(L) - xb.astype(L)) ** 2, axis=1) / (2 * L(0.3) * L(0.3))
    exact = np.exp(-y) * L(2.0) ** 61
    assert np.all(np.abs(got.astype(L) - exact) <= exact * (1 + y) * L(2.0) ** -45 + 2)


def test_crossings_of_special_values(vg, orc):
    """Zero crossings (inside is D < 0) between voxels that hold zeros of both signs, subnormals, the
    largest finite values, infinities and NaN, against the rule written out."""
    rng = np.random.default_rng(72)
    vs = 0.1
    vals = np.array([0.0, -0.0, 5e-324, -5e-324, 1e-310, -1e-310, 0.3, -0.3, 0.02, -0.07, 1.7e308, -1.7e308, np.inf,
                     -np.inf, np.nan, np.copysign(np.nan, -1.0)])
    ijk = np.stack(np.meshgrid(np.arange(-8, 16), np.arange(-8, 8), np.arange(0, 8), indexing="ij"), -1).reshape(-1, 3)
    D = vals[rng.integers(0, len(vals), len(ijk))]
    m = vg.Map(precision="fp64", voxel_size=vs)
    m.import_grid(orc.pack_key(ijk), D, np.ones(len(D)), np.ones(len(D), np.uint8))
    x, o, s = (t.cpu().numpy() for t in m.extract_mesh(triangles=False)["crossings"])
    at = {tuple(v): d for v, d in zip(ijk.tolist(), D)}
    want = {}
    with np.errstate(all="ignore"):
        for v, da in at.items():
            for axis in range(3):
                w = tuple(c + (k == axis) for k, c in enumerate(v))
                if w not in at or (da < 0) == (at[w] < 0):
                    continue
                t = np.float64(da) / (np.float64(da) - np.float64(at[w]))
                p = np.array([np.float32((c + (t if k == axis else 0.0)) * vs) for k, c in enumerate(v)])
                if not np.all(np.isfinite(p)):
                    continue
                own = tuple(np.floor(p.astype(np.float64) / vs + 0.5).astype(int))
                for u, slot in ((v, 2 * axis + 1), (w, 2 * axis)):
                    if own == u:
                        want[(int(orc.pack_key(np.array([u]))[0]), slot)] = p
    got = {(int(k), int(c)): p for k, c, p in zip(o, s, x)}
    assert len(got) == len(x) and got.keys() == want.keys() and len(got) > 1000
    for k, p in got.items():
        assert np.array_equal(p.view(np.uint32), want[k].view(np.uint32))
