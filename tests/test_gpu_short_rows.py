"""Rows much shorter than a warp, either side of the widths at which a kernel changes its tiles or
a pass its kernel, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import test_gpu_parity as parity  # noqa: E402
from paper_1806_09907_gb300 import airgb, synth  # noqa: E402

DEV = "cuda"


@pytest.mark.parametrize("x", [2, 3, 4, 5, 8, 9, 12, 16, 17, 20, 33, 40, 48, 63])
def test_point_kernels(x):
    for shape in ((5, 11, x), (37, x)):
        parity.test_warp_and_adjoint(shape)
        parity.test_regulariser(shape)
        v = synth.smooth_field(shape, 1.5, 3, min_wavelength=12.0).astype(np.float32)
        u, traj = airgb.al_exp_field(torch.from_numpy(v).to(DEV), 3, True)
        assert np.abs(u.cpu().numpy() - oracle.exp_field(v, 3)).max() <= 1e-5 * np.abs(v).max()
        g = np.random.default_rng(x).normal(size=v.shape).astype(np.float32)
        gv = airgb.al_exp_field_adjoint(traj, torch.from_numpy(g).to(DEV), 3)
        ref = oracle.exp_field_adjoint(traj.cpu().numpy(), g, 3)
        assert parity.rel_l2(gv.cpu().numpy().astype(np.float64), ref) <= 1e-4


@pytest.mark.parametrize("shape,delta", [
    ((110, 100, 3), 5), ((110, 100, 23), 2), ((110, 100, 24), 2),    # 32,768 rows and more
    ((110, 100, 79), 16), ((110, 100, 80), 16), ((180, 190, 5), 32),
    ((20, 30, 3), 5), ((16400, 7), 3), ((16400, 23), 1), ((5, 16390), 6),
    ((4, 9, 256), 3), ((4, 9, 263), 3), ((3, 40, 320), 32), ((3, 40, 321), 32),  # one and two tiles
    ((3, 40, 316), 16), ((2, 25, 404), 1), ((2, 70, 31), 1), ((2, 70, 33), 1),
])
def test_expansion_and_transpose(shape, delta):
    parity.test_displacement(shape, delta)
    parity.test_displacement_adjoint(shape, delta)
