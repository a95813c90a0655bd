"""Volumes whose second and third planes begin beyond the 2^31st element: a vector field of more
than 2^30 voxels, and a lattice of more than 2^31 points. Every kernel here is local, so the last
rows of the whole volume equal, bit for bit, what the rows alone give away from their first ones."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1806_09907_gb300 import airgb  # noqa: E402

DEV = "cuda"
SHAPE = (32808, 32768)  # 2^30 voxels and a few rows more; 32808 = 24 * 1367
ROWS = 96               # the last rows: four bricks of spacing 8
EDGE = 16               # rows of the crop whose neighbours differ


@pytest.fixture(autouse=True)
def room():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 130 << 30:
        pytest.skip("needs 130 GB of free device memory")
    yield
    torch.cuda.empty_cache()


def field(shape, size, seed=1):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return torch.rand((len(shape),) + shape, generator=g, device=DEV).sub_(0.5).mul_(2 * size)


def image(shape, seed):
    return torch.rand(shape, generator=torch.Generator(device=DEV).manual_seed(seed), device=DEV)


def crop(t, axis):
    return t.narrow(axis, t.shape[axis] - ROWS, ROWS).contiguous()


def same_rows(whole, rows, axis):
    a = whole.narrow(axis, whole.shape[axis] - ROWS + EDGE, ROWS - EDGE)
    b = rows.narrow(axis, EDGE, ROWS - EDGE)
    return torch.equal(a, b)


@pytest.mark.parametrize("accumulate", [False, True])
def test_warp_adjoint_beyond_2_30_voxels(accumulate):
    M, gW, u = image(SHAPE, 2), image(SHAPE, 3), field(SHAPE, 3.0)
    mask = torch.ones(SHAPE, dtype=torch.uint8, device=DEV)
    start = torch.full_like(u, 0.25) if accumulate else None
    first = torch.full((2, ROWS, SHAPE[1]), 0.25, device=DEV) if accumulate else None
    out = airgb.al_warp_adjoint(M, u, mask, gW, start, accumulate)
    ref = airgb.al_warp_adjoint(crop(M, 0), crop(u, 1), crop(mask, 0), crop(gW, 0), first,
                                accumulate)
    assert same_rows(out, ref, 1)


@pytest.mark.parametrize("shape", [SHAPE, (724, 2050, 725)])
def test_exponential_beyond_2_30_voxels(shape):
    axis = len(shape) - 1  # of the field: the rows
    v = field(shape, 3.0)
    u, traj = airgb.al_exp_field(v, 1, True)
    uc, tc = airgb.al_exp_field(crop(v, axis), 1, True)
    assert same_rows(u, uc, axis) and same_rows(traj[0], tc[0], axis)
    del u, v
    if len(shape) == 3:
        return
    g = field(shape, 1.0, 4)
    g[0, -1, -1] = 1.5  # the scale of the fixed point, in both
    gv = airgb.al_exp_field_adjoint(traj, g, 1)
    gc = airgb.al_exp_field_adjoint(tc, crop(g, axis), 1)
    assert same_rows(gv, gc, axis)


def test_fused_local_correlation_beyond_2_30_voxels():
    """The gradient times the number of masked voxels is a sum of local terms. Both evaluations
    are fp32 within rel-L2 1e-4 of it (the bar of the objectives against the oracle)."""
    spacing = 8
    F, M = image(SHAPE, 5), image(SHAPE, 6)
    c = field(airgb.lattice_shape(SHAPE, spacing), 2.0, 7)
    cc = c[:, (SHAPE[0] - ROWS) // spacing:].contiguous()
    got = []
    for f, m, k in ((F, M, c), (crop(F, 0), crop(M, 0), cc)):
        value, grad = airgb.Objective(f.shape, spacing, "lcc", 0.0)(f, m, k)
        got.append(grad[:, -cc.shape[1] + 5:].double() * value[3])
    assert float((got[0] - got[1]).norm() / got[1].norm()) <= 2e-4


def test_expansion_of_a_lattice_beyond_2_31_points():
    shape = (2, 32760, 32760)
    lat = airgb.lattice_shape(shape, 1)
    assert lat[0] * lat[1] * lat[2] > 2 ** 31
    c = torch.empty((3,) + lat, device=DEV)
    for k in range(3):
        c[k].normal_(generator=torch.Generator(device=DEV).manual_seed(k))
    u = airgb.al_displacement(shape, 1, c)
    cc = c[:, :, shape[1] - ROWS:].contiguous()
    ref = airgb.al_displacement((2, ROWS, shape[2]), 1, cc)
    assert torch.equal(u[:, :, -ROWS:], ref)
