"""AUTO on grids TMA cannot read (odd pitches, odd bases, dense rows): the
staged copies of 4 and of 8 bytes against the FP64 oracle and, bit for bit for
the boxes (the same order of FMAs), the point-by-point kernel; and the z
chunks of small grids, whose last one is short."""
import numpy as np
import pytest

import oracle
import paper_2507_11067_gb300 as mms
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5  # max|gpu - oracle| / max|oracle|, the bar of the FP32 paths


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mms.build()
    mms.load()


def rel(g, o):
    return float(np.abs(np.asarray(g, np.float64) - o).max() / max(np.abs(o).max(), 1e-300))


# one tile and less, tile edges of 64 x 16 (x 32 planar), ragged tails, one-plane chunks
SIZES = [(1, 1, 1), (5, 3, 2), (63, 17, 3), (64, 32, 19), (131, 33, 40)]


@pytest.mark.parametrize("shape", ["star", "box", "star2d", "box2d"])
@pytest.mark.parametrize("r", [1, 2, 3, 4])
def test_unaligned_auto(shape, r):
    planar = shape.endswith("2d")
    rz = 0 if planar else r
    for i, (nx, ny, nz) in enumerate(SIZES):
        make = workloads.uniform_grid2d if planar else workloads.uniform_grid
        grid = make(nx, ny, nz, r, workload=2, salt=40 + i)
        c = workloads.normal_coeffs(shape, r, workload=2, salt=40 + i)
        ref = oracle.stencil2d(shape, r, c, grid) if planar else oracle.stencil(shape, r, c, grid)
        X, Y, Z = nx + 2 * r, ny + 2 * r, nz + 2 * rz
        # (floats before the grid, floats added to each row): 4-byte copies for
        # an odd base or pitch, 8-byte ones where both are even
        for base, extra in ((0, 0), (1, 0), (2, X % 2), (0, 1 + X % 2), (2, (6 - X) % 4)):
            py = X + extra
            size = base + (Z - 1) * Y * py + (Y - 1) * py + X   # the buffer ends with the grid's last element
            flat = torch.full((size,), float("nan"), device="cuda")
            inp = torch.as_strided(flat, (Z, Y, X), (Y * py, py, 1), base)
            inp.copy_(torch.from_numpy(grid))
            outs = {}
            for path in ("auto", "naive"):
                buf = torch.full((nz, ny, nx + 3), -7.0, device="cuda")
                mms.apply(shape, r, c, inp, out=buf[..., :nx], path=path)
                torch.cuda.synchronize()
                mms.check_device()
                outs[path] = buf[..., :nx].cpu().numpy()
                assert bool((buf[..., nx:] == -7.0).all()), (path, nx, ny, nz)
            assert rel(outs["auto"], ref) <= TOL, (nx, ny, nz, base, extra)
            if shape.startswith("box") and (base % 4 or py % 4):   # (an aligned one may take the tensor cores)
                assert np.array_equal(outs["auto"], outs["naive"]), (nx, ny, nz, base, extra)


@pytest.mark.parametrize("shape,r,path", [("star", 1, "cuda_core"), ("star", 4, "cuda_core"), ("box", 2, "cuda_core"),
                                          ("box", 2, "bf16x3"), ("box", 4, "bf16x3")])
def test_short_z_chunks(shape, r, path):
    # depths around what one SM, all SMs and the tuned chunk take
    for nx, ny, nz in ((64, 16, 1), (64, 16, 151), (64, 16, 305), (300, 40, 29), (65, 130, 64)):
        grid = workloads.uniform_grid(nx, ny, nz, r, workload=2, salt=nz)
        c = workloads.normal_coeffs(shape, r, workload=2, salt=nz)
        out = mms.apply(shape, r, c, mms.to_padded_device(grid, r), path=path)
        torch.cuda.synchronize()
        mms.check_device()
        assert rel(out.cpu().numpy(), oracle.stencil(shape, r, c, grid)) <= TOL, (nx, ny, nz)
