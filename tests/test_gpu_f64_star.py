"""The FP64 star on small and ragged grids against the oracle's FP64 sums
(27 products in another order: 27 roundings of 2^-53 of the sum of magnitudes
on each side), on grids larger than a launch's y and z extents included."""
import numpy as np
import pytest

import oracle
import paper_2507_11067_gb300 as mms
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [(1, 1, 1), (33, 3, 2), (31, 33, 35), (65, 7, 66), (2, 131073, 1), (3, 1, 65537)])
def test_small_and_ragged(r, n):
    mms.build()
    mms.load()
    nx, ny, nz = n
    grid = workloads.uniform_grid(nx, ny, nz, r, workload=2, salt=r).astype(np.float64)
    c = workloads.normal_coeffs("star", r, workload=2, salt=r).astype(np.float64)
    out = mms.apply_f64("star", r, c, torch.from_numpy(grid).cuda())
    torch.cuda.synchronize()
    got, ref = out.cpu().numpy(), oracle.stencil("star", r, c, grid)
    assert np.abs(got - ref).max() <= 2 * 27 * 2.0 ** -53 * np.abs(c).sum()
