"""The model and the division by m on narrow grids, whose rows take 8 to 64
threads, with more rows than the blocks of a launch cover at once."""
import numpy as np
import pytest

import paper_2507_11067_gb300 as mms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 4])
@pytest.mark.parametrize("nx", [1, 5, 8, 9, 16, 17, 33, 64, 65])
def test_narrow_rows(nx, r):
    mms.build()
    mms.load()
    ny, nz = 331, 307
    m = mms.padded_empty(nx, ny, nz, r)
    desc, _keep = mms.wave_desc(nx, ny, nz, r, 1, m.stride(1), m.stride(0))
    m.fill_(-1.0)
    v = np.random.default_rng(nx).uniform(1500, 4500, (nz, ny, nx)).astype(np.float32)
    dt, h = np.float32(1e-3), np.float32(10.0)
    mms.model_from_velocity(desc, torch.from_numpy(v).cuda(), m, float(dt), float(h))
    got = m.cpu().numpy()
    want = np.zeros_like(got)
    want[r:-r, r:-r, r:-r] = v * v * (dt * dt / (h * h))
    assert np.allclose(got, want, rtol=3e-7, atol=0)   # three FP32 roundings
    g = np.random.default_rng(1).standard_normal(v.shape)
    grad = torch.from_numpy(g).cuda()
    mms.grad_divide_m(desc, m, grad)
    assert np.array_equal(grad.cpu().numpy(), g / got[r:-r, r:-r, r:-r].astype(np.float64))
