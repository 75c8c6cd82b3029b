"""The steady state of every marching kernel: thread blocks that take many
planes (ring stages refilled, barrier phases flipped, queues shifted or rotated
all the way round) and a short last chunk, at every point.  Small grids are
divided into marches of a plane or two, so the grids here keep every SM busy,
and each test asserts the depth it needs.

Sweeps are compared with the point-by-point kernel: the boxes bit for bit (the
same order of FMAs), the stars within the roundings of both.  The wave steps
are compared bit for bit with the same step on crops of the grid, whose short
marches the oracle tests cover."""
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


def sweep(shape, r, c, inp, **kw):
    out = mms.apply(shape, r, c, inp, **kw)
    planes = mms.last_planes()
    torch.cuda.synchronize()
    mms.check_device()
    return out, planes


def agree(shape, r, c, got, ref):
    if shape.startswith("box"):
        return torch.equal(got, ref)
    # n FMAs of |w| |x| <= |w| in either order, each within n 2^-24 of the sum
    n = c.size + 1
    return float((got - ref).abs().max()) <= 2 * n * 2.0 ** -24 * float(np.abs(c).sum())


def uniform(inp, seed):
    return inp.uniform_(-1, 1, generator=torch.Generator(device="cuda").manual_seed(seed))


# enough columns for the least threads per block (64: eight blocks per SM), and
# chunks of 32 to 70 planes with a last one of 6 at 32 and 64
@pytest.mark.parametrize("shape", ["star", "box"])
@pytest.mark.parametrize("r", [1, 2, 3, 4])
def test_cuda_core_variants_march(shape, r):
    nx, ny, nz = 1530, 1019, 70
    inp = uniform(mms.padded_empty(nx, ny, nz, r, zero=False), r)
    c = workloads.normal_coeffs(shape, r, workload=2, salt=r)
    ref, _ = sweep(shape, r, c, inp, path="naive")
    for v in range(mms.num_variants(shape, r, "cuda_core")):
        got, planes = sweep(shape, r, c, inp, path="cuda_core", variant=v)
        assert planes >= 32, (v, planes)
        assert agree(shape, r, c, got, ref), v
        del got


@pytest.mark.parametrize("shape", ["star2d", "box2d"])
@pytest.mark.parametrize("r", [1, 2, 3, 4])
def test_planar_variants_march(shape, r):
    nx, ny, nz = 4093, 1111, 20          # 35 to 139 row blocks in groups of 8 to 32
    inp = uniform(mms.padded_empty2d(nx, ny, nz, r, zero=False), r)
    c = workloads.normal_coeffs(shape, r, workload=2, salt=r)
    ref, _ = sweep(shape, r, c, inp, path="naive")
    for v in range(mms.num_variants(shape, r, "cuda_core")):
        got, blocks = sweep(shape, r, c, inp, path="cuda_core", variant=v)
        assert blocks >= 8, (v, blocks)
        assert agree(shape, r, c, got, ref), v


# ------------------------------------------------------------- wave steps

NX, NY, NZ, CX, CY = 1024, 512, 131, 256, 128     # chunks of 128 and 3 planes; crops of the whole depth
R = 4


def crops():
    for y in range(0, NY, CY):
        for x in range(0, NX, CX):
            yield x, y


def geometry(nx, ny, f, **kw):
    py, pz, ss = mms.field_geometry(f)
    return mms.wave_desc(nx, ny, NZ, R, 1, py, pz, ss, **kw)[0]


def field(nx, ny, value=None):
    f = mms.padded_empty(nx, ny, NZ, R, nshots=1)
    if value is not None:
        f.copy_(value)
    return f


def random_fields(n, seed):
    return [uniform(field(NX, NY), seed + i) for i in range(n)]


def cut(f, x, y):
    return field(CX, CY, f[..., y:y + CY + 2 * R, x:x + CX + 2 * R])


def inner(f):
    return f[..., R:-R, R:-R, R:-R]


def check_crops(step, nout, depth):
    """step(nx, ny, cut) runs on the fields cut(f) and returns its outputs, all (.., z, y, x) without halo."""
    whole = step(NX, NY, lambda f: f)
    planes = mms.last_planes()
    torch.cuda.synchronize()
    mms.check_device()
    assert planes >= depth, planes
    for x, y in crops():
        part = step(CX, CY, lambda f: cut(f, x, y))
        assert mms.last_planes() < planes
        torch.cuda.synchronize()
        assert len(part) == nout
        for k in range(nout):
            assert torch.equal(whole[k][..., y:y + CY, x:x + CX], part[k]), (k, x, y)
    mms.check_device()


@pytest.mark.parametrize("form", ["forward", "recompute", "adjoint", "bulk", "slices", "lam"])
def test_acoustic_steps_march(form):
    w = workloads.fd8_star_coeffs()
    c, p, lap = random_fields(3, 1)
    m = uniform(field(NX, NY), 9).add_(2.0).mul_(0.1)
    amp = torch.zeros(1, device="cuda")

    def step(nx, ny, cut):
        fc, fp, fm, fl, nxt = cut(c), cut(p), cut(m)[0], cut(lap), field(nx, ny)
        d = geometry(nx, ny, fc)
        if form == "forward":
            mms.wave_step_to(d, w, fm, fc, fp, nxt, amp)
            return [inner(nxt)]
        if form == "recompute":
            out = field(nx, ny)
            mms.wave_step_lap(d, w, fm, fc, fp, nxt, out, amp)
            return [inner(nxt), inner(out)]
        nxt.copy_(fp)
        if form == "adjoint":
            mms.wave_adjoint_scaled(d, w, fm, fc, nxt)
            return [inner(nxt)]
        if form == "slices":
            d = geometry(nx, ny, fc, grad_shot_stride=nx * ny * NZ)
        grad = torch.zeros((NZ, ny, nx), device="cuda", dtype=torch.float64)
        fn = mms.wave_adjoint_lap if form == "lam" else mms.wave_adjoint_scaled
        fn(d, w, fm, fc, nxt, None, fl, grad)
        return [inner(nxt), grad]

    # (the forward forms' plan may prefer shorter marches; twelve planes past the ring's three still)
    check_crops(step, 1 if form in ("forward", "adjoint") else 2, 15 if form in ("forward", "recompute") else 100)


@pytest.mark.parametrize("variant", range(9))
def test_vti_step_marches(variant):
    assert mms.aniso_num_variants("vti") == 9
    w = workloads.fd8_star_coeffs()
    h, v, hp, vp = random_fields(4, 21)
    mv, rho = (uniform(field(NX, NY), s).add_(2.0).mul_(0.4) for s in (31, 32))
    amp = torch.zeros(1, device="cuda")

    def step(nx, ny, cut):
        f = [cut(x) for x in (h, v, hp, vp)]
        hn, vn = field(nx, ny), field(nx, ny)
        mms.vti_step(geometry(nx, ny, f[0]), w, cut(mv)[0], cut(rho)[0], *f, hn, vn, amp)
        return [inner(hn), inner(vn)]

    try:
        mms.aniso_set_variant("vti", variant)
        check_crops(step, 2, 100)
    finally:
        mms.aniso_set_variant("vti", 0)


def test_tti_step_marches():
    w2, w1 = workloads.fd8_rows()
    p, q, pp, qp = random_fields(4, 41)
    med = torch.empty((8, NZ, NY, NX), device="cuda").uniform_(
        0.2, 0.5, generator=torch.Generator(device="cuda").manual_seed(5))
    amp = torch.zeros(1, device="cuda")
    places = iter([None] + list(crops()))

    def step(nx, ny, cut):
        f = [cut(x) for x in (p, q, pp, qp)]
        at = next(places)
        dense = med if at is None else med[..., at[1]:at[1] + CY, at[0]:at[0] + CX].contiguous()
        pn, qn = field(nx, ny), field(nx, ny)
        mms.tti_step(geometry(nx, ny, f[0]), w2, w1, dense, *f, pn, qn,
                     torch.empty((4, 1, NZ, ny, nx), device="cuda"), amp)
        return [inner(pn), inner(qn)]

    check_crops(step, 2, 100)
