"""Batches either side of the number of bricks at which the kernel changes: the same coefficients
as the single-problem path, bit for bit, in every order of the items."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import test_gpu_batch as batch  # noqa: E402
from paper_1806_09907_gb300 import airgb, registration  # noqa: E402


def bricks(shapes, spacing):
    bx, by = ((8, 4) if spacing == 4 else (4, 3))
    n = 0
    for s in shapes:
        cells = [-(-k // spacing) for k in reversed(s)]
        n += -(-cells[0] // bx) * -(-cells[1] // by) * (-(-cells[2] // 4) if len(s) == 3 else 1)
    return n


@pytest.mark.parametrize("spacing,many", [(8, 5), (8, 6), (6, 3), (6, 4), (4, 2), (4, 3)])
def test_lines_between_kernels(spacing, many):
    shapes = [(129, 120), (33, 40, 45)] * many
    shapes += [(70, 130)]
    assert (bricks(shapes, spacing) <= (160 if spacing == 4 else 200)) == \
        ((spacing, many) in ((8, 5), (6, 3), (4, 2)))
    pairs, K = batch.pairs_for(shapes, seed=31), 2
    cs, hs, _ = registration.register_sequential(pairs, spacing, 0.1, K)
    for policy in range(4):
        b = airgb.Batch(pairs, spacing, 0.1, history=K)
        b.set_policy(policy)
        for k in range(K):
            b.step(k + 1, k)
        assert b.status() == 0
        for i in range(len(pairs)):
            assert torch.equal(b.ctrl[i], cs[i]), (policy, i)
            assert torch.equal(b.values[i][:, 3], hs[i][:K, 3])
            assert torch.allclose(b.values[i][:, 0], hs[i][:K, 0], rtol=1e-6, atol=0)
