"""The staged convolution passes in the form they were written for, against the oracle: unsplit
forward passes, and more bands per block than the ring has stages, so that stages, barrier phases
and accumulator sets are used again."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import test_gpu_initnet as layers  # noqa: E402
from oracle import initnet as onet  # noqa: E402
from paper_1806_09907_gb300 import airgb  # noqa: E402

DEV = "cuda"


def off16(t):
    """A copy 16 bytes off a 32-byte boundary."""
    flat = torch.empty(t.numel() + 16, dtype=t.dtype, device=DEV)
    n = 16 // t.element_size()
    v = flat[n:n + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 32 == 16
    return v


def check_forward(nb, dims, cin, cout, stride, relu=True):
    """The unsplit forward pass: fp32 output within the accumulation bound n 2^-24 S of the
    oracle, the bf16 one its rounding, also in a buffer on 16 bytes only."""
    x, w, b = layers._layer(21, nb, dims, cin, cout)
    cv = airgb.make_conv(nb, dims, cin, cout, stride)
    pf, _ = airgb.al_conv3d_pack(cv, torch.from_numpy(w).to(DEV), True, False)
    xd, bd = layers._to_dev_bf16(x), torch.from_numpy(b).to(DEV)
    y = airgb.al_conv3d_forward(cv, xd, pf, bd, relu=relu, out_f32=True, split=False)
    wq = layers._bf16(w)
    ref = onet.conv3d(x, wq, b.astype(np.float64), stride, relu)
    S = onet.conv3d(np.abs(x), np.abs(wq), np.abs(b.astype(np.float64)), stride, False)
    assert np.all(np.abs(layers._np(y) - ref) <= 27 * cin * layers.U * S)
    yb = airgb.al_conv3d_forward(cv, xd, pf, bd, relu=relu, split=False)
    assert torch.equal(yb, y.to(torch.bfloat16))
    out = off16(torch.zeros_like(yb))
    assert torch.equal(airgb.al_conv3d_forward(cv, off16(xd), pf, bd, relu=relu, out=out,
                                               split=False), yb)
    assert airgb.al_get_device_error() == 0


@pytest.mark.parametrize("cin", [16, 32, 48, 64])
@pytest.mark.parametrize("stride", [1, 2])
def test_forward_unsplit(cin, stride):
    for nb, dims, cout in ((2, (5, 9, 11), 16), (1, (4, 7, 13), 48), (1, (3, 6, 8), 128),
                           (1, (1, 1, 1), 32)):
        check_forward(nb, dims, cin, cout, stride, relu=cin != 32)


@pytest.mark.parametrize("dims,stride", [
    ((2, 3, 126), 1),   # staged rows of 128 positions
    ((2, 3, 254), 1),   # the longest staged row
    ((2, 2, 256), 1),   # one beyond it
    ((3, 4, 510), 2),   # the longest with stride 2
    ((3, 2, 512), 2),
    ((2, 100, 3), 1),   # bands of many short rows
    ((2, 131, 5), 2),
])
def test_forward_row_lengths(dims, stride):
    check_forward(1, dims, 16, 32, stride)


# items per block of a 152-SM device (forward and input adjoint; ring of 2 to 4 stages):
# 14 and 7, 7, 7, 3.5, 4.6 and 3.3, 7 and 5
@pytest.mark.parametrize("nb,dims,cin,cout,stride", [
    (16, (65, 39, 37), 16, 32, 2),
    (16, (33, 31, 14), 16, 16, 1),
    (16, (33, 31, 14), 32, 32, 1),
    (4, (33, 31, 14), 48, 48, 1),
    (3, (21, 31, 14), 64, 48, 1),
    (16, (45, 33, 18), 32, 48, 2),
])
def test_staged_passes_reuse_their_ring(nb, dims, cin, cout, stride):
    check_forward(nb, dims, cin, cout, stride)
    layers.test_conv_dgrad_parity(nb, dims, cin, cout, stride)
    layers.test_conv_wgrad_parity(nb, dims, cin, cout, stride)
    assert airgb.al_get_device_error() == 0


# either side of the lines at which a pass takes the gathering kernel: short rows in many bands,
# large weights for few bands, two stages with one-row bands
@pytest.mark.parametrize("nb,dims,cin,cout,stride", [
    (8, (40, 40, 3), 16, 16, 1), (8, (40, 40, 4), 16, 16, 1),
    (8, (40, 40, 6), 48, 16, 1), (8, (40, 40, 7), 48, 16, 1),
    (8, (40, 40, 12), 16, 32, 2), (8, (40, 40, 14), 16, 32, 2), (8, (40, 40, 18), 16, 32, 2),
    (4, (16, 16, 14), 32, 48, 2), (8, (16, 16, 14), 32, 48, 2), (8, (32, 32, 32), 32, 48, 2),
    (8, (40, 40, 12), 48, 64, 2), (2, (12, 12, 12), 48, 64, 2),
])
def test_lines_between_kernels(nb, dims, cin, cout, stride):
    check_forward(nb, dims, cin, cout, stride)
    layers.test_conv_dgrad_parity(nb, dims, cin, cout, stride)
    layers.test_conv_wgrad_parity(nb, dims, cin, cout, stride)
    assert airgb.al_get_device_error() == 0
