"""Planar sweeps under AUTO on planes TMA cannot read, against the
point-by-point kernel bit for bit: both add the taps in the same order, the
star tap by tap over its two lines."""
import numpy as np
import pytest

import paper_2507_11067_gb300 as mms
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    mms.build()
    mms.load()


def unaligned(grid, base, py):
    """The planes at element `base` of a buffer of row pitch py that ends with the grid's last element."""
    Z, Y, X = grid.shape
    flat = torch.full((base + (Z - 1) * Y * py + (Y - 1) * py + X,), float("nan"), device="cuda")
    inp = torch.as_strided(flat, (Z, Y, X), (Y * py, py, 1), base)
    inp.copy_(grid)
    return inp


def same_as_naive(shape, r, c, inp):
    got = {}
    for path in ("auto", "naive"):
        got[path] = mms.apply(shape, r, c, inp, path=path)
    torch.cuda.synchronize()
    mms.check_device()
    return torch.equal(got["auto"], got["naive"])


@pytest.mark.parametrize("r", [1, 2, 3, 4])
def test_planar_star_adds_tap_by_tap(r):
    c = workloads.normal_coeffs("star2d", r, workload=2, salt=r)
    for nx, ny, nz in ((1, 1, 1), (63, 33, 2), (130, 70, 3)):
        grid = torch.from_numpy(workloads.uniform_grid2d(nx, ny, nz, r, workload=2, salt=nx)).cuda()
        X = nx + 2 * r
        for base, py in ((1, X), (0, X | 1), (2, X + X % 2)):
            assert same_as_naive("star2d", r, c, unaligned(grid, base, py)), (nx, ny, nz, base, py)


@pytest.mark.parametrize("shape", ["star2d", "box2d"])
@pytest.mark.parametrize("r", [1, 2, 3, 4])
def test_planes_of_many_row_blocks(shape, r):
    # 35 row blocks in groups of eight, the last group of three and its last
    # block of 23 rows: ring stages are refilled and the copy re-aimed in mid-march
    nx, ny, nz = 4090 - r, 1111, 10
    X = nx + 2 * r
    c = workloads.normal_coeffs(shape, r, workload=2, salt=50 + r)
    grid = torch.empty(nz, ny + 2 * r, X, device="cuda").uniform_(
        -1, 1, generator=torch.Generator(device="cuda").manual_seed(r))
    even = X + (2 - X) % 4
    for base, py in ((1, X), (0, X | 1), (2, even), (0, even)):
        inp = unaligned(grid, base, py)
        mms.apply(shape, r, c, inp)
        assert mms.last_planes() == 8
        assert same_as_naive(shape, r, c, inp), (base, py)
