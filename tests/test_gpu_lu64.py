"""Complex128 LU with tensor-core updates (csrc/tc_update64.cuh) and integer panel
updates at sizes around the 64 x 32 tiles and the 32-column panels: the FP64 densities'
backward error in the oracle's systems, every mode (the bar of the FP64 parity tests)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# n = 2 N: trailing blocks of 2, 34, 66 rows; 130 = 4 x 32 + 2; whole tiles; one panel more than a tile
@pytest.mark.parametrize("N", [49, 65, 80, 97])
def test_backward_error(N):
    from oracle.assemble import Solution
    from oracle.problem import Params
    from paper_2412_11162_gb300 import Problem
    from paper_2412_11162_gb300.binding import PMLBIE_FP64
    M, k1, k2 = 32, 2 * np.pi, 3 * np.pi
    ref = Solution(Params(k1=k1, k2=k2, N=N, M=M), keep_matrices=True)
    P = Problem(k1, k2, N, M)
    for _ in range(3):          # direct, captured, replayed
        out, _ = P.solve([np.pi / 6], precision=PMLBIE_FP64)
    u, phi = (out[k].cpu().numpy()[:, :, 0] for k in ("u1", "phi1"))
    for n in range(M // 2):
        A, B = ref.A[n]
        x = np.concatenate([u[n], phi[n]])
        eta = np.linalg.norm(A @ x - B) / (np.linalg.norm(A) * np.linalg.norm(x) + np.linalg.norm(B))
        assert eta <= 1e-11, (n, eta)
