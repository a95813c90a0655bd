"""Edges of the tiled kernels, against the oracle: tile and band remainders, the shortest and
longest rows a tiling takes, the shapes at which a pass changes its kernel, buffers that lie on
16 bytes only, and overlapping buffers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import test_gpu_initnet as layers  # noqa: E402
import test_gpu_parity as parity  # noqa: E402
from paper_1806_09907_gb300 import airgb  # noqa: E402

DEV = "cuda"


@pytest.mark.parametrize("nb,dims,cin,cout,stride", [
    (2, (5, 6, 7), 2, 16, 1),        # two channels, stride 1
    (1, (4, 5, 66), 2, 32, 2),       # two channels, even rows over several warps
    (1, (3, 2, 33), 2, 32, 2),       # two channels, odd rows
    (1, (2, 3, 126), 16, 16, 1),     # staged rows of 128 positions
    (1, (2, 3, 254), 16, 16, 1),     # the longest staged row (256)
    (1, (2, 2, 256), 16, 16, 1),     # one beyond it
    (1, (3, 4, 510), 16, 32, 2),     # the longest with stride 2
    (1, (3, 1, 512), 16, 32, 2),
    (2, (1, 1, 1), 32, 16, 2),       # one voxel
    (1, (2, 2, 2), 16, 32, 2),
    (3, (22, 21, 23), 32, 48, 2),    # several bands and parities, odd sizes
    (2, (33, 18, 20), 16, 32, 2),    # bands that end inside the grid
    (1, (13, 15, 14), 64, 48, 1),
    (1, (5, 9, 8), 48, 128, 1),      # the widest output
    (3, (8, 6, 10), 80, 32, 2),      # channels without a staged kernel
    (1, (3, 5, 11), 24, 16, 1),
])
def test_conv_tile_edges(nb, dims, cin, cout, stride):
    layers.test_conv_forward_parity(nb, dims, cin, cout, stride, relu=True)
    layers.test_conv_wgrad_parity(nb, dims, cin, cout, stride)
    if cin % 16 == 0 and cin <= 128:
        layers.test_conv_dgrad_parity(nb, dims, cin, cout, stride)
    assert airgb.al_get_device_error() == 0


@pytest.mark.parametrize("stride", [1, 2])
def test_conv_buffers_on_16_bytes(stride):
    """Outputs and ReLU factors 16 bytes off a 32-byte boundary give the bits of aligned ones."""
    nb, dims, cin, cout = 2, (9, 10, 12), 16, 32
    x, w, b = layers._layer(3, nb, dims, cin, cout)
    cv = airgb.make_conv(nb, dims, cin, cout, stride)
    osz = airgb.conv_output_size(cv)
    pf, pd = airgb.al_conv3d_pack(cv, torch.from_numpy(w).to(DEV))
    xd, bd = layers._to_dev_bf16(x), torch.from_numpy(b).to(DEV)
    g = torch.randn((nb,) + osz + (cout,), device=DEV).to(torch.bfloat16)

    def off(t):
        flat = torch.empty(t.numel() + 8, dtype=t.dtype, device=DEV)
        v = flat[8:].view(t.shape)
        v.copy_(t)
        assert v.data_ptr() % 32 == 16
        return v

    y = airgb.al_conv3d_forward(cv, xd, pf, bd)
    y2 = airgb.al_conv3d_forward(cv, off(xd), pf, bd, out=off(y.zero_() + 0))
    y = airgb.al_conv3d_forward(cv, xd, pf, bd)
    assert torch.equal(y, y2)
    gx = airgb.al_conv3d_backward_data(cv, g, pd, relu_input=xd)
    gx2 = airgb.al_conv3d_backward_data(cv, off(g), pd, relu_input=off(xd), grad_in=off(gx))
    assert torch.equal(gx, gx2)


@pytest.mark.parametrize("shape", [(3, 300), (70, 131), (9, 17, 66), (26, 25, 130), (40, 16, 9)])
@pytest.mark.parametrize("factor", [2, 3, 4, 5, 7, 8])
def test_pyramid_tile_edges(shape, factor):
    """A sum of n = 2 r + 1 taps of unit sum per axis: |err| <= (d n + d) 2^-24 max|image|."""
    shape = tuple(max(s, factor + 1) for s in shape)
    im = np.random.default_rng(5).uniform(-1000, 1500, shape).astype(np.float32)
    out = airgb.al_pyramid_level(torch.from_numpy(im).to(DEV), factor).cpu().numpy()
    ref = oracle.pyramid_level(im, factor)
    n = 2 * int(1.5 * factor) + 1
    assert out.shape == ref.shape
    assert np.abs(out - ref).max() <= len(shape) * (n + 1) * 2.0 ** -24 * np.abs(im).max()


@pytest.mark.parametrize("shape", [(64, 96), (20, 24, 32)])
def test_pyramid_level_inside_its_image(shape):
    im = torch.rand(shape, device=DEV)
    ref = airgb.al_pyramid_level(im, 2)
    out = airgb.al_pyramid_level(im, 2, level=im.view(-1)[:ref.numel()].view(ref.shape))
    assert torch.equal(out, ref)


@pytest.mark.parametrize("shape,delta", [((5, 260), 1), ((140, 9), 32), ((3, 4, 257), 2),
                                         ((33, 70, 129), 7), ((20, 35, 400), 13), ((9, 600), 3)])
def test_expansion_tile_edges(shape, delta):
    parity.test_displacement(shape, delta)
    parity.test_displacement_adjoint(shape, delta)


@pytest.mark.parametrize("shape", [(9, 33), (5, 17, 65)])
def test_exponential_adjoint_of_non_finite_gradients(shape):
    """An infinity or a NaN in the incoming gradient stays where the transposed interpolation
    takes it: every value away from it keeps the bits it has without it."""
    d = len(shape)
    v = 0.3 * torch.randn((d,) + shape, device=DEV)
    _, traj = airgb.al_exp_field(v, 1, True)
    g = torch.randn((d,) + shape, device=DEV).clamp(-3, 3)
    g.view(-1)[0] = 3.9  # sets the fixed point's scale in both calls
    ref = airgb.al_exp_field_adjoint(traj, g, 1)
    bad = g.clone()
    at = (1,) + tuple(s // 2 for s in shape)
    bad[at] = float("nan")
    out = airgb.al_exp_field_adjoint(traj, bad, 1)
    near = torch.zeros(shape, dtype=torch.bool, device=DEV)
    near[tuple(slice(max(s // 2 - 4, 0), s // 2 + 5) for s in shape)] = True
    assert torch.equal(out[:, ~near], ref[:, ~near])
    assert torch.isnan(out[at])


@pytest.mark.parametrize("shape,count,blobs", [
    ((40, 100, 101), 4, 70),   # 16 x 16 boxes, rows that end inside four columns, two chunks
    ((33, 65, 64), 16, 64),    # whole 16-byte rows, a full chunk
    ((9, 20, 24), 1, 129),     # 8 x 8 boxes, a chunk of one blob
])
def test_render_blobs_boxes(shape, count, blobs):
    """Against the sum over every blob. Per voxel the fp32 sum of at most 129 terms, each of
    three roundings and exponentials of a few ulp, is within (129 + 12) 2^-24 of the sum of
    magnitudes, and 129 dropped terms add 129 * 1.6e-8: below 1.1e-5 of the largest value
    when amplitudes are below 1 and the largest value is above 1."""
    table = layers.synth.blob_table(count, shape, blobs, seed=11)
    out = airgb.al_render_blobs(shape, torch.from_numpy(table).to(DEV)).double().cpu().numpy()
    for v in (0, count - 1):
        ref = layers.synth.render_blob_table(shape, table[v])
        assert np.max(np.abs(out[v] - ref)) <= 1.1e-5 * max(1.0, np.max(np.abs(ref)))


@pytest.mark.parametrize("shape,delta", [((21, 35, 45), 8), ((9, 13, 50), 6), ((11, 17, 33), 4),
                                         ((33, 66), 4)])
def test_warp_ctrl_bricks(shape, delta):
    """Bricks of one and two control cells in y, with remainders in every axis."""
    parity.test_warp_ctrl_batch(shape, delta)


@pytest.mark.parametrize("shape,delta", [((9, 21, 35), 4), ((14, 20, 26), 6), ((18, 17, 33), 8),
                                         ((40, 37), 8)])
def test_brick_cells_at_faces_and_beyond(shape, delta):
    """A zero displacement puts every sample on its voxel, the last faces included: the warp is
    the image bit for bit and the mask full. Displacements far outside, at the limits of the
    cell's integer arithmetic and not finite leave the mask empty and the warp zero."""
    d, lat = len(shape), airgb.lattice_shape(shape, delta)
    M = torch.rand((1,) + shape, device=DEV) + 1.0
    mask = torch.empty((1,) + shape, dtype=torch.uint8, device=DEV)
    c = torch.zeros((1, d) + lat, device=DEV)
    W = airgb.al_warp_ctrl(shape, delta, M, c, mask=mask)
    assert torch.equal(W, M) and bool(mask.all())
    ob = airgb.Objective(shape, delta, "mse")
    assert float(ob(M[0], M[0], c[0])[0][3]) == M[0].numel()
    inf = float("inf")
    for axis in range(d):
        for v in (inf, -inf, float("nan"), 1e3, -1e3, 2.0 ** 22, -2.0 ** 22, 2.0 ** 23,
                  -2.0 ** 24, 1e9, -3e9, 3e38, -3e38):
            c.zero_()
            c[0, axis] = v
            W = airgb.al_warp_ctrl(shape, delta, M, c, mask=mask)
            assert not bool(mask.any()) and not bool(W.any()), (axis, v)
            assert float(ob(M[0], M[0], c[0])[0][3]) == 0.0, (axis, v)
