"""Phases, exponentials and 1/sqrt of the sampling loops on the integer pipe
(csrc/fxtrig.cuh) over the wavenumbers from a fraction of a turn to hundreds of
turns across the domain, real and complex distances, against plain numpy sums of
the same samples; and the two precisions' modal kernels, which share every kernel.

Tolerance, relative to the sum of |samples| times 2 pi / M: a sample of either
side is good to about 8 ulp plus the rounding of the phase (|q| ulp), the
transform adds a few units of 2^-57; (16 + 2 max|q|) 2^-53 bounds the sum.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

M, N = 96, 64


@pytest.mark.parametrize("k", [0.02, 0.5, 2.0, 24.0, 150.0, 600.0])
def test_point_modes_over_wavenumbers(k):
    import torch
    from paper_2412_11162_gb300 import Problem
    w = k * np.pi
    P = Problem(w, 1.25 * w, N, M)
    node, T = P.nodes(), P.node_tables()
    h = 1.0 / (N + 2)                      # two segments: Nt = N + 2
    pts = [(0.0, 1.0), (0.7, 0.9), (1.9, 2.0), (2.4, 30.0)]
    rho, z = (np.array(v) for v in zip(*pts))
    psi = 2 * np.pi * np.arange(M) / M
    s2 = np.sin(psi / 2) ** 2
    th = 2 * np.arange(M, dtype=np.longdouble) * np.arccos(np.longdouble(-1)) / M
    idx = np.outer(np.arange(M // 2), np.arange(M)) % M
    E = (np.cos(th) - 1j * np.sin(th))[idx] * (2 * np.arccos(np.longdouble(-1)) / M)
    for m in (0, 31, 63):                  # next to the axis, physical, PML end
        unit = torch.zeros((M // 2, N, 1), dtype=torch.complex128, device="cuda")
        unit[:, m] = 1.0
        zero = torch.zeros_like(unit)
        got = P.field(rho, z, np.zeros(len(pts), int), dict(u1=zero, phi1=unit, u2=zero, phi2=unit))[:, :, 0].cpu().numpy()
        rt = node["rho"][m] + 1j * T["I"][m]
        for p, (r, zz) in enumerate(pts):
            R = np.sqrt((r - rt) ** 2 + (zz - node["z"][m]) ** 2 + 4.0 * r * rt * s2)
            q = w * R
            S = 0.5 * h * T["Wphi"][m] * np.exp(1j * q) / (4 * np.pi * R)
            bar = (16 + 2 * np.max(np.abs(q))) * 2.0 ** -53 * np.sum(np.abs(S)) * 2 * np.pi / M
            err = np.max(np.abs(got[:, p] - E @ S.astype(np.clongdouble)))
            assert err <= bar, (k, m, p, err, bar)


@pytest.mark.parametrize("k", [0.5, 20.0])
@pytest.mark.parametrize("M", [16, 96, 144])
def test_modal_kernels_same_in_both_precisions(k, M):
    import torch
    from paper_2412_11162_gb300 import Problem, binding as B
    P = Problem(k * np.pi, 1.25 * k * np.pi, N, M)
    a, b = (P.modal_kernels(0, M // 2, precision=q) for q in (B.PMLBIE_FP64, B.PMLBIE_MIXED))
    off = ~torch.eye(N, dtype=torch.bool, device="cuda")      # l = m is not defined
    assert torch.equal(torch.view_as_real(a[:, :, off]), torch.view_as_real(b[:, :, off]))
