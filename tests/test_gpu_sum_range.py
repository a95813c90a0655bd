"""Sums of the step kernels near fp32's range: a sum of terms that fp32 holds is finite, as an FP64
sum of them is."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1806_09907_gb300 import airgb  # noqa: E402

DEV = "cuda"
SHAPES = [(64, 64, 64), (101, 163, 165), (300, 301)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("size", [3e-18, 1.0, 1e15, 2.5e18])
def test_mse_of_large_differences(shape, size):
    """fp32 squares and sums of a few, the rest exact: 2^-20 is ample."""
    g = torch.Generator(device=DEV).manual_seed(1)
    F = size * torch.rand(shape, generator=g, device=DEV)
    W = -size * torch.rand(shape, generator=g, device=DEV)
    m = (torch.rand(shape, generator=g, device=DEV) < 0.9).to(torch.uint8)
    value, _ = airgb.al_similarity("mse", F, W, m)
    ref = (W.double() - F.double())[m.bool()].square().mean()
    assert float(value[1]) == float(m.sum())
    assert abs(float(value[0]) - float(ref)) <= 2.0 ** -20 * float(ref)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("size", [3e-17, 1.0, 2e17, 3e18])
def test_regulariser_of_large_displacements(shape, size):
    d = len(shape)
    g = torch.Generator(device=DEV).manual_seed(2)
    u = size * (torch.rand((d,) + shape, generator=g, device=DEV) - 0.5)
    u[0, 0] = 0.9 * size  # rows of terms near the others' size, up to 3e38
    value, _ = airgb.al_regulariser(u, 1.0, False)
    v = u.double()
    ref = sum(v.diff(dim=a).square().sum() for a in range(1, d + 1)) / u[0].numel()
    assert torch.isfinite(value).all()
    assert abs(float(value[0]) - float(ref)) <= 2.0 ** -20 * float(ref)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("level", [0.0, -1e30, 2.0 ** 120])
def test_ncc_of_a_constant_image(shape, level):
    """A constant image has no variance: the similarity is 1 whatever its level."""
    g = torch.Generator(device=DEV).manual_seed(3)
    F = torch.full(shape, level, device=DEV)
    W = torch.rand(shape, generator=g, device=DEV)
    m = torch.ones(shape, dtype=torch.uint8, device=DEV)
    value, gw = airgb.al_similarity("ncc", F, W, m)
    assert float(value[0]) == 1.0 and float(value[1]) == F.numel()
    assert torch.isfinite(gw).all()


def test_terms_that_are_not_finite():
    F = torch.rand((40, 40, 40), device=DEV)
    m = torch.ones(F.shape, dtype=torch.uint8, device=DEV)
    W = F + 1.0
    for bad, seen in ((float("nan"), torch.isnan), (float("inf"), torch.isinf)):
        X = W.clone()
        X[7, 9, 11] = bad
        assert bool(seen(airgb.al_similarity("mse", F, X, m)[0][0]))
        u = torch.rand((3,) + tuple(F.shape), device=DEV)
        u[1, 20, 20, 20] = bad
        assert bool(seen(airgb.al_regulariser(u, 1.0, False)[0][0]))
    X = W.clone()
    X[7, 9, 11] = float("nan")
    m[7, 9, 11] = 0
    assert abs(float(airgb.al_similarity("mse", F, X, m)[0][0]) - 1.0) < 1e-6
