"""The staged 3D sweeps of grids TMA cannot read, on grids large enough that
AUTO takes them (smaller ones run point by point, bit for bit): thin and ragged
grids of short marches, and one whose march is long, with 4- and 8-byte copies,
against the point-by-point kernel -- the boxes bit for bit, the stars within
the roundings of both."""
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


def unaligned(nx, ny, nz, r, base, py, seed):
    """A grid at element `base` of a buffer of row pitch py that ends with the grid's last element."""
    X, Y, Z = nx + 2 * r, ny + 2 * r, nz + 2 * r
    flat = torch.full((base + (Z - 1) * Y * py + (Y - 1) * py + X,), float("nan"), device="cuda")
    inp = torch.as_strided(flat, (Z, Y, X), (Y * py, py, 1), base)
    return inp.uniform_(-1, 1, generator=torch.Generator(device="cuda").manual_seed(seed))


def both(shape, r, c, inp):
    got = mms.apply(shape, r, c, inp)
    planes = mms.last_planes()
    ref = mms.apply(shape, r, c, inp, path="naive")
    torch.cuda.synchronize()
    mms.check_device()
    return got, ref, planes


def agree(shape, c, got, ref):
    if shape == "box":
        return torch.equal(got, ref)
    n = c.size + 1   # FMAs of |w| |x| <= |w| in either order, each sum within n 2^-24
    return float((got - ref).abs().max()) <= 2 * n * 2.0 ** -24 * float(np.abs(c).sum())


@pytest.mark.parametrize("shape", ["star", "box"])
@pytest.mark.parametrize("r", [1, 2, 3, 4])
@pytest.mark.parametrize("n,depth", [((131, 67, 40), 1), ((63, 17, 301), 1), ((601, 171, 3), 1), ((1021, 771, 70), 60)])
def test_staged_grids(shape, r, n, depth):
    nx, ny, nz = n
    c = workloads.normal_coeffs(shape, r, workload=2, salt=r)
    X = nx + 2 * r
    for base, py in ((0, X | 1), (1, X + (4 - X) % 4), (2, X + X % 2)):
        got, ref, planes = both(shape, r, c, unaligned(nx, ny, nz, r, base, py, nx))
        assert planes >= depth
        assert agree(shape, c, got, ref), (base, py)


@pytest.mark.parametrize("shape,r,below,above", [("star", 2, (63, 17, 279), (63, 17, 281)), ("box", 4, (63, 17, 92), (63, 17, 94))])
def test_small_grids_run_point_by_point(shape, r, below, above):
    # 298809 and 300951 points; 98532 and 100674
    c = workloads.normal_coeffs(shape, r, workload=2, salt=r)
    mms.apply("box", 1, np.ones(27, np.float32), mms.padded_empty(33, 8, 700, 1))
    before = mms.last_planes()   # the point-by-point kernel leaves it as it is
    for n, staged in ((below, False), (above, True)):
        got, ref, planes = both(shape, r, c, unaligned(*n, r, 1, (n[0] + 2 * r) | 1, 3))
        assert (planes != before) == staged
        assert agree(shape, c, got, ref) if staged else torch.equal(got, ref)
