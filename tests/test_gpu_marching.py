"""The marching kernels on a volume large enough for columns of eight slices, with remainders in
every axis, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import test_gpu_parity as parity  # noqa: E402
from paper_1806_09907_gb300 import airgb, synth  # noqa: E402

DEV = "cuda"
MARCH = (101, 163, 165)  # 6 x 21 tiles of 32 x 8 columns, 13 chunks of 8 slices


def fields():
    rough = np.random.default_rng(8).normal(0.0, 2.0, (3,) + MARCH).astype(np.float32)
    return {"smooth": synth.smooth_field(MARCH, 3.0, 9, min_wavelength=24.0).astype(np.float32),
            "rough": rough}


@pytest.mark.parametrize("kind", ["smooth", "rough"])
def test_marching_exponential(kind):
    """Smooth: a sample's far z corners join the next sample's near ones; rough: hardly ever.
    The oracle takes the GPU's trajectory, so both see the same cells. Bars of the
    exponential's tests: 1e-5 max|v|, and rel-L2 1e-4 for the adjoint."""
    v, K = fields()[kind], 2
    u, traj = airgb.al_exp_field(torch.from_numpy(v).to(DEV), K, True)
    ref = oracle.exp_field(v, K)
    assert np.abs(u.cpu().numpy() - ref).max() <= 1e-5 * np.abs(v).max()
    g = np.random.default_rng(10).normal(size=v.shape).astype(np.float32)
    gd = torch.from_numpy(g).to(DEV)
    gv = airgb.al_exp_field_adjoint(traj, gd, K)
    assert torch.equal(gv, airgb.al_exp_field_adjoint(traj, gd, K))
    gref = oracle.exp_field_adjoint(traj.cpu().numpy(), g, K)
    assert parity.rel_l2(gv.cpu().numpy().astype(np.float64), gref) <= 1e-4


@pytest.mark.parametrize("kind", ["smooth", "rough"])
def test_marching_regulariser(kind):
    u = fields()[kind]
    val, gu = airgb.al_regulariser(torch.from_numpy(u).to(DEV), weight=0.1)
    R, gr = oracle.diffusion(u)
    assert abs(float(val[0]) - R) <= parity.J_TOL * abs(R)
    assert parity.rel_l2(gu.cpu().numpy(), 0.1 * gr) <= 1e-5


@pytest.mark.parametrize("sim", ["mse", "ncc", "lcc"])
def test_marching_objective(sim):
    F, M = synth.ct_pair(MARCH, n_inner=10)
    c = synth.random_ctrl(oracle.lattice_shape(MARCH, 5), 3, 1.5, 9907)
    parity.check_objective(F, M, c, 5, sim, fused=False)
