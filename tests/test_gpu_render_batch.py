"""Blob volumes: a volume's bits do not depend on how many volumes share its call."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1806_09907_gb300 import airgb  # noqa: E402

DEV = "cuda"


@pytest.mark.parametrize("shape", [(40, 100, 101), (33, 64, 68), (20, 30, 17)])
@pytest.mark.parametrize("blobs", [3, 64, 130])
def test_volume_alone_equals_volume_in_batch(shape, blobs):
    """Few narrow blobs leave most voxels to terms around 6 sigma, where a box decides."""
    count = 48
    g = torch.Generator(device=DEV).manual_seed(5)
    scale = torch.tensor([s - 1.0 for s in reversed(shape)] + [1.5, 1.0], device=DEV)
    table = torch.rand((count, blobs, 5), generator=g, device=DEV) * scale
    table[..., 3] += 0.8
    both = airgb.al_render_blobs(shape, table)
    for v in (0, 17, count - 1):
        alone = airgb.al_render_blobs(shape, table[v:v + 1].clone())
        assert torch.equal(alone[0], both[v])
