"""Block fixed-point even DFTs (csrc/fxdft.cuh) at every transform size the
library takes: the modal kernels of (point, node) pairs, read out of the field
entry point with unit densities, against plain numpy sums of the same samples.

Tolerance, relative to the sum of |samples| times 2 pi / M: a sample of either
side is good to about 8 ulp plus the rounding of the phase (|q| ulp), the
transform adds a few units of 2^-57; (16 + 2 max|q|) 2^-53 bounds the sum.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [16, 24, 32, 36, 48, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 324, 384, 432, 512, 576, 648, 768]


@pytest.mark.parametrize("M", SIZES)
def test_point_modes_against_plain_sums(M):
    import torch
    from paper_2412_11162_gb300 import Problem
    k1, k2, N = 2 * np.pi, 3 * np.pi, 64
    P = Problem(k1, k2, N, M)
    node, T = P.nodes(), P.node_tables()
    h = 1.0 / (N + 2)                      # two segments: Nt = N + 2
    pts = [(0.0, 1.0, 0), (0.7, 0.9, 0), (1.9, 2.0, 0), (0.4, -1.1, 1), (2.2, -0.8, 1)]
    rho, z, reg = (np.array(v) for v in zip(*pts))
    psi = 2 * np.pi * np.arange(M) / M
    # the transform's own sums in extended precision
    th = 2 * np.arange(M, dtype=np.longdouble) * np.arccos(np.longdouble(-1)) / M
    idx = np.outer(np.arange(M // 2), np.arange(M)) % M
    E = (np.cos(th) - 1j * np.sin(th))[idx] * (2 * np.arccos(np.longdouble(-1)) / M)
    for m in (0, 31, 40, 63):              # next to the axis, on the bump, physical, PML end
        unit = torch.zeros((M // 2, N, 1), dtype=torch.complex128, device="cuda")
        unit[:, m] = 1.0
        zero = torch.zeros_like(unit)
        got = {}
        for name, u, phi in (("S", zero, unit), ("K", unit, zero)):
            got[name] = P.field(rho, z, reg, dict(u1=u, phi1=phi, u2=u, phi2=phi))[:, :, 0].cpu().numpy()
        rt = node["rho"][m] + 1j * T["I"][m]
        for p, (r, zz, g) in enumerate(pts):
            w, sg = (k1, 1.0) if g == 0 else (k2, -1.0)
            dz, s2 = zz - node["z"][m], np.sin(psi / 2) ** 2
            R = np.sqrt((r - rt) ** 2 + dz * dz + 4.0 * r * rt * s2)
            q = w * R
            S = np.exp(1j * q) / (4 * np.pi * R)
            nd = sg * (T["nuc_r"][m] * (rt - r + 2 * r * s2) - T["nuc_z"][m] * dz)
            K = -nd / R ** 2 * S * (1 - 1j * q)
            fs, fk = 0.5 * sg * h * T["Wphi"][m], -0.5 * h * T["Wu"][m]
            tol = (16 + 2 * np.max(np.abs(q))) * 2.0 ** -53
            for name, x, f in (("S", S, fs), ("K", K, fk)):
                bar = tol * abs(f) * np.sum(np.abs(x)) * 2 * np.pi / M
                if name == "K":            # the normal factor's own cancellation
                    bar *= 1 + np.max(np.abs(T["nuc_r"][m] * (rt + r)) + np.abs(T["nuc_z"][m] * (abs(zz) + 1))) \
                        / max(np.max(np.abs(nd)), 1e-300)
                err = np.max(np.abs(got[name][:, p] - f * (E @ x.astype(np.clongdouble))))
                assert err <= bar, (M, m, p, name, err, bar)
