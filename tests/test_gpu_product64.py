"""Complex128 products with several right-hand sides on the tensor cores
(csrc/tc_product64.cuh), which form the right-hand sides and the residuals of the
solves: row blocks of 128 and column chunks of 32 with remainders, groups of 8
right-hand sides with remainders; and the streamed complex64 solves
(csrc/lu_solve32.cuh) with 1 to 8 right-hand sides and more than one segment of 512 rows.  A solution of the wrong system shows as a backward
error in the systems that the library's own kernels, corrections and diagonal give.
Bars: mixed 1e-13 (the documented stop), FP64 4 n u (elimination with a growth of at
most 4), plus the rounding n u of this test's own products, n = 2 N, u = 2^-53."""
import numpy as np
import pytest

from test_gpu_lu64 import systems

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,waves", [(47, 2), (48, 5), (64, 8), (65, 9), (80, 17), (130, 2), (290, 8)])
def test_backward_error(N, waves):
    from paper_2412_11162_gb300 import Problem
    from paper_2412_11162_gb300.binding import PMLBIE_FP64, PMLBIE_MIXED
    P = Problem(2 * np.pi, 3 * np.pi, N, 32)
    S, u = systems(P), 2.0 ** -53
    for precision, bar in ((PMLBIE_MIXED, 1e-13 + 2 * N * u), (PMLBIE_FP64, 5 * 2 * N * u)):
        out, _ = P.solve(np.linspace(0.1, 1.3, waves), precision=precision)
        u1, phi1, u2, phi2 = (out[k].cpu().numpy() for k in ("u1", "phi1", "u2", "phi2"))
        for n, A in enumerate(S):
            x, b = np.concatenate([u1[n], phi1[n]]), np.concatenate([u1[n] - u2[n], phi1[n] - phi2[n]])
            B = np.concatenate([np.zeros((N, waves)), A[N:] @ b])
            norm = lambda v: np.linalg.norm(v, axis=0)
            eta = norm(A @ x - B) / (np.linalg.norm(A) * norm(x) + norm(B))
            assert np.max(eta) <= bar, (precision, n, eta)
