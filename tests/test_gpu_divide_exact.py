"""The gradient's division by m gives the IEEE quotient, every bit of it: on
random values and on dividends whose quotient lies as near as it can to the
midpoint of two FP64 numbers."""
import numpy as np
import pytest

import paper_2507_11067_gb300 as mms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_quotient_is_correctly_rounded():
    mms.build()
    mms.load()
    nx, ny, nz, r = 512, 64, 64, 4
    m = mms.padded_empty(nx, ny, nz, r)
    desc, _keep = mms.wave_desc(nx, ny, nz, r, 1, m.stride(1), m.stride(0))
    rng = np.random.default_rng(7)
    n = nx * ny * nz
    mv = np.ldexp(rng.integers(1 << 23, 1 << 24, n).astype(np.float64), rng.integers(-80, 30, n) - 23).astype(np.float32)
    g = np.ldexp(rng.integers(1 << 52, 1 << 53, n).astype(np.float64), rng.integers(-500, 500, n)) * rng.choice([-1.0, 1.0], n)
    # every other dividend: an odd 54-bit number times m, cut to 53 bits (and the next)
    mant, _ = np.frexp(mv.astype(np.float64))
    for i in range(0, 400000, 2):
        p = (int(rng.integers(1 << 53, 1 << 54)) | 1) * int(mant[i] * (1 << 24))
        g[i] = float((p >> (p.bit_length() - 53)) + (i >> 1) % 2)
    m[r:-r, r:-r, r:-r] = torch.from_numpy(mv.reshape(nz, ny, nx)).cuda()
    grad = torch.from_numpy(g.reshape(nz, ny, nx)).cuda()
    mms.grad_divide_m(desc, m, grad)
    assert np.array_equal(grad.cpu().numpy().reshape(-1), g / mv.astype(np.float64))
