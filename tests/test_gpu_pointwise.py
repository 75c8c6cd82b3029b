"""The pointwise kernels around the wave steps on ragged rows: the model, the
division of the gradient by m (an FP64 quotient without an FP64 division)
against numpy's, and the chain rule."""
import numpy as np
import pytest

import paper_2507_11067_gb300 as mms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mms.build()
    mms.load()


def geometry(nx, ny, nz, r=4):
    m = mms.padded_empty(nx, ny, nz, r)
    desc, keep = mms.wave_desc(nx, ny, nz, r, 1, m.stride(1), m.stride(0))
    return m, desc, keep


@pytest.mark.parametrize("n", [(1, 1, 1), (67, 5, 3), (130, 33, 9), (64, 4, 257)])
def test_model_rows(n):
    nx, ny, nz = n
    m, desc, _ = geometry(nx, ny, nz)
    m.fill_(-1.0)
    v = np.random.default_rng(nx).uniform(1500, 4500, (nz, ny, nx)).astype(np.float32)
    dt, h = np.float32(1e-3), np.float32(10.0)
    mms.model_from_velocity(desc, torch.from_numpy(v).cuda(), m, float(dt), float(h))
    want = np.zeros((nz + 8, ny + 8, nx + 8), np.float32)
    want[4:-4, 4:-4, 4:-4] = v * v * (dt * dt / (h * h))
    assert np.allclose(m.cpu().numpy(), want, rtol=3e-7, atol=0)   # three FP32 roundings


@pytest.mark.parametrize("n", [(67, 5, 3), (256, 16, 40)])
def test_divide_by_m(n):
    nx, ny, nz = n
    m, desc, _ = geometry(nx, ny, nz)
    g = np.random.default_rng(nx)
    shape = (nz, ny, nx)
    mv = np.exp2(g.uniform(-12, 4, shape)).astype(np.float32)
    gv = g.standard_normal(shape) * np.exp2(g.uniform(-200, 200, shape))
    flat_m, flat_g = mv.reshape(-1), gv.reshape(-1)
    flat_m[:9] = [0.0, 1e-40, np.inf, np.nan, 1e-30, 1e30, -0.5, 2.0, 3.0]
    flat_g[9:17] = [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e308, 1e-308]
    m[4:-4, 4:-4, 4:-4] = torch.from_numpy(mv).cuda()
    grad = torch.from_numpy(gv).cuda()
    mms.grad_divide_m(desc, m, grad)
    with np.errstate(all="ignore"):
        want = gv / mv.astype(np.float64)
    got = grad.cpu().numpy()
    special = ~np.isfinite(want) | (want == 0)
    assert np.array_equal(got[special], want[special], equal_nan=True)
    assert np.array_equal(np.signbit(got[want == 0]), np.signbit(want[want == 0]))
    ok = ~special
    assert np.all(np.abs(got[ok] - want[ok]) <= np.spacing(np.abs(want[ok])))   # one ulp


def test_chain_rule():
    g = np.random.default_rng(3)
    gm, v = g.standard_normal(1001), g.uniform(1500, 4500, 1001).astype(np.float32)
    out = torch.empty(1001, device="cuda", dtype=torch.float64)
    dt, h = float(np.float32(1e-3)), 10.0
    mms.grad_to_velocity(torch.from_numpy(gm).cuda(), torch.from_numpy(v).cuda(), out, dt, h)
    assert np.allclose(out.cpu().numpy(), gm * 2.0 * v.astype(np.float64) * (dt * dt / (h * h)), rtol=1e-15, atol=0)
