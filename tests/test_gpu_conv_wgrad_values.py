"""The weight adjoint of the strided layers: values that are not finite stay in the sums that read
them, and the error against 64 bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1806_09907_gb300 import airgb  # noqa: E402

DEV = "cuda"


def wgrad64(x, gy, stride):
    """gw, gb in 64 bits: only voxels inside the grid take part."""
    o, cin, cout = gy.shape[1:4], x.shape[-1], gy.shape[-1]
    p = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1, 1, 1))
    g2 = gy.double().reshape(-1, cout)
    gw = torch.empty((cout, 27, cin), dtype=torch.float64, device=DEV)
    for t in range(27):
        a = (t // 9, t // 3 % 3, t % 3)
        at = tuple(slice(a[k], a[k] + (o[k] - 1) * stride + 1, stride) for k in range(3))
        gw[:, t] = g2.T @ p[(slice(None),) + at].reshape(-1, cin)
    return gw, g2.sum(0)


def layer(nb, dims, cin, cout, seed=1):
    g = torch.Generator(device=DEV).manual_seed(seed)
    cv = airgb.make_conv(nb, dims, cin, cout, 2)
    x = torch.randn((nb,) + dims + (cin,), generator=g, device=DEV).relu().to(torch.bfloat16)
    gy = (1e-3 * torch.randn((nb,) + airgb.conv_output_size(cv) + (cout,), generator=g,
                             device=DEV)).to(torch.bfloat16)
    return cv, x, gy


SHAPES = [(2, (6, 10, 12), 16, 32),     # even sizes: the last column and row are read once
          (1, (5, 24, 26), 32, 48),     # several bands
          (3, (7, 9, 11), 16, 16),      # odd sizes
          (2, (4, 8, 32), 16, 32),      # rows of 16 outputs
          (1, (4, 40, 64), 32, 32),     # rows of 32 outputs, several bands
          (2, (3, 2, 2), 16, 32),
          (1, (2, 13, 4), 32, 16)]


@pytest.mark.parametrize("nb,dims,cin,cout", SHAPES)
@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
def test_input_that_is_not_finite(nb, dims, cin, cout, bad):
    """A bad input makes the weights it meets not finite and leaves the others at their sums
    (bound: n 2^-24 of the sum of magnitudes)."""
    cv, x, gy = layer(nb, dims, cin, cout)
    D, H, W = dims
    places = [(0, 0, 0), (D - 1, H - 1, W - 1), (D // 2, H - 1, 0), (0, H // 2, W - 1),
              (D - 1, min(1, H - 1), W // 2), (D // 2, H // 2, min(1, W - 1))]
    S, _ = wgrad64(x.abs(), gy.abs(), 2)
    n = gy[..., 0].numel()
    for k, at in enumerate(places):
        y = x.clone()
        y[(nb - 1,) + at + ((5 * k + 3) % cin,)] = bad
        gw, gb = airgb.al_conv3d_backward_weight(cv, y, gy)
        ref, refb = wgrad64(y, gy, 2)
        ok = torch.isfinite(ref)
        assert not bool(ok.all())
        assert torch.equal(torch.isfinite(gw), ok), at
        assert bool(((gw.double() - ref).abs()[ok] <= (n + 1) * 2.0 ** -24 * S[ok]).all()), at
        assert torch.isfinite(gb).all()


@pytest.mark.parametrize("nb,dims,cin,cout", SHAPES)
def test_output_gradient_that_is_not_finite(nb, dims, cin, cout):
    cv, x, gy = layer(nb, dims, cin, cout)
    gy[(0, -1, -1, -1, cout - 1)] = float("inf")
    gw, gb = airgb.al_conv3d_backward_weight(cv, x, gy)
    ref, refb = wgrad64(x, gy, 2)  # padding zeros meet the infinity here as well
    assert torch.equal(torch.isfinite(gw), torch.isfinite(ref))
    assert torch.equal(torch.isfinite(gb), torch.isfinite(refb))


@pytest.mark.parametrize("nb,dims,cin,cout,most", [
    (16, (64, 64, 64), 16, 32, 1.15e-6), (8, (41, 37, 29), 16, 32, 1.15e-7),
    (12, (30, 21, 47), 16, 32, 1.16e-7), (16, (22, 30, 26), 32, 48, 1.5e-7),
    (9, (26, 31, 20), 32, 48, 8.9e-8)])
def test_error_against_64_bits(nb, dims, cin, cout, most):
    """No larger than what gathered operands and chains of one split's voxels give (`most`,
    measured for these sizes on other inputs), and a tenth for the inputs' spread."""
    cv, x, gy = layer(nb, dims, cin, cout, seed=7)
    gw, gb = airgb.al_conv3d_backward_weight(cv, x, gy)
    ref, refb = wgrad64(x, gy, 2)
    assert float((gw.double() - ref).norm() / ref.norm()) <= 1.1 * most
    assert float((gb.double() - refb).norm() / refb.norm()) <= 1e-7
