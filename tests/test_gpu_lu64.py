"""Complex128 LU with tensor-core updates (csrc/tc_update64.cuh) and integer panel
updates at sizes around the 64 x 32 tiles and the 32-column panels: the backward error
of the FP64 densities in the systems that the library's own kernels, corrections and
diagonal give, every mode.  Bar: 4 n u (u = 2^-53), n = 2 N, the usual bound n g u of
Gaussian elimination with a growth g of at most 4 on these systems."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def systems(P):
    """[mode] -> the block matrix, from the C ABI's kernels and tables."""
    import torch
    from paper_2412_11162_gb300 import binding as B
    N, nm, h = P.N, P.n_modes, 1.0 / (P.N + 2)
    T = P.node_tables()
    grid = P.modal_kernels(precision=B.PMLBIE_FP64).cpu().numpy() * h
    g, c = P.near_count()
    close = torch.empty((g + c, 4, nm), dtype=torch.complex128, device="cuda")
    close = B.pmlbie_close_pair_kernels(P.handle, B.PMLBIE_FP64, 0, nm, close).cpu().numpy()[g:]
    tgt, _, col, coef = P.corrections()
    Da, Db = P.diagonal()
    for s in range(col.shape[1]):
        ok = col[:, s] >= 0
        for k in range(4):
            for n in range(nm):
                np.add.at(grid[n, k], (tgt[ok], col[ok, s]), coef[ok, s] * close[ok, k, n])
    S, K = grid[:, 0::2] * T["Wphi"], grid[:, 1::2] * T["Wu"]
    return [np.block([[K[n, 0] - np.diag(Da), -S[n, 0]], [K[n, 1] - np.diag(Db), S[n, 1]]]) for n in range(nm)]


# n = 2 N: trailing blocks of 2, 34, 66 rows; 130 = 4 x 32 + 2; whole tiles; one panel more than a tile
@pytest.mark.parametrize("N", [49, 65, 80, 97])
def test_backward_error(N):
    from paper_2412_11162_gb300 import Problem
    from paper_2412_11162_gb300.binding import PMLBIE_FP64
    P = Problem(2 * np.pi, 3 * np.pi, N, 32)
    for _ in range(3):          # direct, captured, replayed
        out, _ = P.solve([np.pi / 6], precision=PMLBIE_FP64)
    u1, phi1, u2, phi2 = (out[k].cpu().numpy()[:, :, 0] for k in ("u1", "phi1", "u2", "phi2"))
    for n, A in enumerate(systems(P)):
        x, b = np.concatenate([u1[n], phi1[n]]), np.concatenate([u1[n] - u2[n], phi1[n] - phi2[n]])
        B = np.concatenate([np.zeros(N), A[N:] @ b])
        eta = np.linalg.norm(A @ x - B) / (np.linalg.norm(A) * np.linalg.norm(x) + np.linalg.norm(B))
        assert eta <= 4 * 2 * N * 2.0 ** -53, (n, eta)
