"""The rounding order of the leapfrog update, bit for bit: every form of the
step forms g (2 a + m L a - g a') as u = fma(2, a, RN(m L a)), fma(-g, a', u)
and one product with g.  The order decides how the rounding of a few early
steps near the source grows into the records and the gradient, so it is pinned
here rather than bounded."""
import numpy as np
import pytest

import paper_2507_11067_gb300 as mms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mms.build()
    mms.load()


def fma32(a, b, c):
    """RN32(a b + c) of FP32 arrays, and where that is certain: the product is
    exact in FP64 and the sum rounds there first, which decides the FP32 value
    except where an inexact sum lands on a midpoint."""
    x, y = a.astype(np.float64) * b.astype(np.float64), c.astype(np.float64)
    s = x + y
    d = s - x
    inexact = (x - (s - d)) + (y - d) != 0
    return s.astype(np.float32), ~(inexact & ((s.view(np.int64) & 0x1fffffff) == 0x10000000))


def update(c, p, m, lap, g):
    u, ok1 = fma32(np.float32(2) * np.ones_like(c), c, m * lap)
    v, ok2 = fma32(-g, p, u)
    return g * v, ok1 & ok2


@pytest.mark.parametrize("r,nx", [(1, 45), (2, 70), (3, 33), (4, 45), (4, 132)])
def test_update_rounding_order(r, nx):
    ny, nz, ns = 19, 7, 2
    rng = np.random.default_rng(10 * r + nx)
    field = lambda: mms.padded_empty(nx, ny, nz, r, nshots=ns)
    inner = np.s_[..., r:-r, r:-r, r:-r]
    c, p, nxt, nxt2, lap = (field() for _ in range(5))
    m = mms.padded_empty(nx, ny, nz, r)
    host = {}
    for name, f, lo, hi in (("c", c, -1, 1), ("p", p, -1, 1), ("m", m, 0.05, 0.4)):
        host[name] = rng.uniform(lo, hi, tuple(f[inner].shape)).astype(np.float32)
        f[inner] = torch.from_numpy(host[name]).cuda()
    w = rng.normal(size=3 * (2 * r + 1)).astype(np.float32)
    py, pz, ss = mms.field_geometry(c)
    geo = (nx, ny, nz, r, ns, py, pz, ss, 2, 0.2)
    desc, _keep = mms.wave_desc(*geo)
    amp = torch.zeros(ns, device="cuda")
    # g on every plane: a step from zero fields with a residual of one and m = 1
    g = np.empty((nz, ny, nx), np.float32)
    one = mms.padded_empty(nx, ny, nz, r)
    one[inner] = 1.0
    for z in range(nz):
        dz, _kz = mms.wave_desc(*geo, rec_z=z)
        z1, z2 = field(), field()
        mms.wave_adjoint_scaled(dz, w, one, z1, z2, torch.ones(ns, ny, nx, device="cuda"))
        g[z] = z2[inner][0, z].cpu().numpy()
    assert g.max() == 1.0 and g.min() < 0.9
    mms.wave_step_lap(desc, w, m, c, p, nxt, lap, amp)
    want, ok = update(host["c"], host["p"], host["m"], lap[inner].cpu().numpy(), g)
    assert ok.mean() > 0.999
    mms.wave_step_to(desc, w, m, c, p, nxt2, amp)
    got = {"recompute": nxt, "forward": nxt2}
    # the scaled adjoint's forms: no gradient, one shared slice, a slice per shot
    n = nx * ny * nz
    for form, gss in (("adjoint", None), ("shared", 0), ("slices", n)):
        q = field()
        q.copy_(p)
        d = desc if not gss else mms.wave_desc(*geo, grad_shot_stride=gss)[0]
        grad = None if gss is None else torch.zeros(n * (ns if gss else 1), device="cuda", dtype=torch.float64)
        mms.wave_adjoint_scaled(d, w, m, c, q, None, None if gss is None else lap, grad)
        got[form] = q
    torch.cuda.synchronize()
    mms.check_device()
    for form, f in got.items():
        res = f[inner].cpu().numpy()
        assert np.array_equal(res[ok], want[ok]), (form, np.abs(res - want).max())
