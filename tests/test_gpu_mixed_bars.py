"""The mixed path at the FP64 path's bars.

* Its modal kernels are the FP64 path's: far and physical close pairs against the oracle
  within 1e-12 of a block's largest entry, PML close pairs within 1e-12 of the split's
  term scale (the bars of test_gpu_parity.test_modal_kernels_config1), all pairs and
  correction pairs at N = 128, M = 64.
* Its solves meet the documented stop mode by mode and right-hand side by right-hand side:
  |B - A x| <= max(1e-13 |B|, f (|A|_F |x| + |B|)), f = 4e-16, or 1e-14 where a mode went to
  GMRES; the residual in extended precision, plus 4 u |A|_F |x| (u = 2^-53) for the rounding
  of the entries of A, which this test forms in another order than the library.
"""
import numpy as np
import pytest

from test_gpu_lu64 import systems
from test_gpu_parity import CFG1, _split_term_scale, oracle_solution, split_scale

pytestmark = pytest.mark.gpu
KERNELS = (("a", "S"), ("a", "K"), ("b", "S"), ("b", "K"))


def test_modal_kernels():
    from paper_2412_11162_gb300 import Problem
    from paper_2412_11162_gb300.binding import PMLBIE_MIXED
    K = Problem(CFG1["k1"], CFG1["k2"], CFG1["N"], CFG1["M"]).modal_kernels(precision=PMLBIE_MIXED).cpu().numpy()
    S = oracle_solution(**CFG1).sys
    li, mi = S.grid_pairs
    rt = S.G.nodes["rho_t"].imag
    loose = S.near[: S.ngrid] & ((rt[li] > 0) | (rt[mi] > 0))
    for n in range(CFG1["M"] // 2):
        for kern, (reg, which) in enumerate(KERNELS):
            ref = S.grid_kernel(reg, which, n)
            d = np.abs(K[n, kern] - ref)[li, mi]
            assert d[~loose].max() <= 1e-12 * np.abs(ref).max(), (n, kern)
            if which == "S":
                assert (d[loose] / (_split_term_scale(S, reg, n)[loose] + 1e-300)).max() <= 1e-12, (n, kern)


def test_correction_pairs():
    import torch
    from paper_2412_11162_gb300 import Problem
    from paper_2412_11162_gb300 import binding as B
    P = Problem(CFG1["k1"], CFG1["k2"], CFG1["N"], CFG1["M"])
    g, c = P.near_count()
    vals = torch.empty((g + c, 4, P.n_modes), dtype=torch.complex128, device="cuda")
    B.pmlbie_close_pair_kernels(P.handle, B.PMLBIE_MIXED, 0, P.n_modes, vals)
    vals = vals[g:].cpu().numpy()
    S = oracle_solution(**CFG1).sys
    rows = S.ngrid + np.arange(c)
    pg = {k: v[rows] for k, v in S.pg.items()}
    loose = S.near[rows] & ((pg["rho_t"].imag > 0) | (pg["rho_t_s"].imag > 0))
    lap = np.searchsorted(np.nonzero(S.near)[0], rows[loose])
    for kern, (reg, which) in enumerate(KERNELS):
        ref = S.kern[reg][which == "K"][rows]
        for n in range(P.n_modes):
            d = np.abs(vals[:, kern, n] - ref[:, n])
            assert d[~loose].max() <= 1e-12 * np.abs(ref[:, n]).max(), (kern, n)
            if which == "S" and loose.any():
                sc = split_scale({k: v[loose] for k, v in pg.items()}, S.lap_near[0][lap],
                                 CFG1["k1"] if reg == "a" else CFG1["k2"], CFG1["M"], 5, n)
                assert (d[loose] / sc).max() <= 1e-12, (kern, n)


@pytest.mark.parametrize("N,waves", [(48, 1), (65, 3), (97, 8)])
def test_documented_stop(N, waves):
    from paper_2412_11162_gb300 import Problem
    from paper_2412_11162_gb300.binding import PMLBIE_MIXED
    P, L = Problem(2 * np.pi, 3 * np.pi, N, 32), np.clongdouble
    out, rep = P.solve(np.linspace(0.1, 1.2, waves), precision=PMLBIE_MIXED)
    u1, phi1, u2, phi2 = (out[k].cpu().numpy() for k in ("u1", "phi1", "u2", "phi2"))
    norm = lambda v: np.linalg.norm(v.astype(complex), axis=0)
    f = 1e-14 if rep.gmres_modes else 4e-16
    for n, A in enumerate(systems(P)):
        x, b = np.concatenate([u1[n], phi1[n]]), np.concatenate([u1[n] - u2[n], phi1[n] - phi2[n]])
        A, F = A.astype(L), np.linalg.norm(A)
        B = np.concatenate([np.zeros((N, waves), L), A[N:] @ b.astype(L)])
        r, nb, ax = norm(A @ x.astype(L) - B), norm(B), F * norm(x)
        assert np.all(r <= np.maximum(1e-13 * nb, f * (ax + nb)) + 4 * 2.0 ** -53 * ax), (n, r / nb, r / (ax + nb))
