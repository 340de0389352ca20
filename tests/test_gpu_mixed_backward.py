"""Mixed solves at orders 2 N around multiples of 32 (the complex64 factors are padded
to whole 32-row blocks) with one and several right-hand sides: the backward error of
the densities in the systems that the library's own kernels, corrections and diagonal
give.  Bar: the documented stop |B - A x| <= 1e-13 |B|, plus the rounding 2 N 2^-53 of
this test's own products."""
import numpy as np
import pytest

from test_gpu_lu64 import systems

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("waves", [1, 3])
@pytest.mark.parametrize("N", [48, 49, 63, 65, 97])
def test_backward_error(N, waves):
    from paper_2412_11162_gb300 import Problem
    from paper_2412_11162_gb300.binding import PMLBIE_MIXED
    P = Problem(2 * np.pi, 3 * np.pi, N, 32)
    for _ in range(3):          # direct, captured, replayed
        out, _ = P.solve(np.linspace(0.1, 1.2, waves), precision=PMLBIE_MIXED)
    u1, phi1, u2, phi2 = (out[k].cpu().numpy() for k in ("u1", "phi1", "u2", "phi2"))
    for n, A in enumerate(systems(P)):
        x, b = np.concatenate([u1[n], phi1[n]]), np.concatenate([u1[n] - u2[n], phi1[n] - phi2[n]])
        B = np.concatenate([np.zeros((N, waves)), A[N:] @ b])
        norm = lambda v: np.linalg.norm(v, axis=0)
        eta = norm(A @ x - B) / (np.linalg.norm(A) * norm(x) + norm(B))
        assert np.max(eta) <= 1e-13 + 2 * N * 2.0 ** -53, (n, eta)
