"""The field's contraction with the densities: one wave takes the FP64 product, several
the tensor-core product (csrc/tc_product64.cuh), both with the points of the upper medium
gathered in front.  Several waves against one at a time, points of both media interleaved,
random densities.  Bar: each side's sums of 4 N products err by at most 4 N u of their
absolute sum, which for random densities is about sqrt(4 N) of the result: 2 (4 N)^1.5 u,
N = 65: 1e-12 of a mode's 2-norm.  A NaN in one wave's densities stays in that wave and medium."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npts,waves", [(1, 2), (5, 3), (130, 9), (257, 2), (64, 16)])
def test_waves_together_and_apart(npts, waves):
    import torch
    from paper_2412_11162_gb300 import Problem
    N, M = 65, 32
    P = Problem(2 * np.pi, 3 * np.pi, N, M)
    rng = np.random.default_rng(npts)
    rho, reg = rng.uniform(0, 2, npts), rng.integers(0, 2, npts)
    z = np.where(reg == 0, 1.0, -1.0) * rng.uniform(0.8, 1.5, npts)
    dens = {k: torch.from_numpy(rng.standard_normal((M // 2, N, waves)) + 1j * rng.standard_normal((M // 2, N, waves))).cuda()
            for k in ("u1", "phi1", "u2", "phi2")}
    got = P.field(rho, z, reg, dens).cpu().numpy()
    for r in range(waves):
        one = P.field(rho, z, reg, {k: v[:, :, r:r + 1].contiguous() for k, v in dens.items()})[:, :, 0].cpu().numpy()
        err = np.linalg.norm(got[:, :, r] - one, axis=1) / np.linalg.norm(one, axis=1)
        assert np.max(err) <= 2 * (4 * N) ** 1.5 * 2.0 ** -53, (r, err)
    dens["u1"][2, 40, 1] = float("nan")
    bad = P.field(rho, z, reg, dens).cpu().numpy()
    hit = np.zeros(got.shape, bool)
    hit[2, reg == 0, 1] = True
    assert np.isnan(bad[hit]).all() and np.array_equal(np.isnan(bad), hit)
