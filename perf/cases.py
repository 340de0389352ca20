"""Performance cases of the PML-BIE modal solver: what a user's program has it do, over the sizes it is
used at, through `Problem`, `solve_batch` and the binding's calls.

Four kinds of call:
  * "solve": a scattering run -- Problem.solve for the incident waves (or point sources) and Problem.field at
    the receivers; the pass returns the scattered-field modes at the receivers, which is what a study of a
    scatterer reads.  (The surface densities go from one call to the other on the device.  Next to the axis and
    the PML they are determined by the discrete equations only up to their condition number, 1e7 .. 1e9, times
    the rounding; the field is not.)  Mixed precision as in the sweeps, FP64 (the default of Problem.solve) as in
    a reference run.
  * "batch": several independent instances in one solve_batch call, then their fields.
  * "kernels" / "close": the modal kernels of every grid pair, and the split kernels of the close pairs alone --
    the layers under a solve, which a program that builds its own systems calls directly.
  * "field": a field map from densities already on the device.

Geometries: "dent" is the rectangular dent of depth and radius 1 with a1 = T = S = 2 (omega = 2 pi above,
2.4 pi below, plane wave pi/3, source (0.3, 0.5)); "bump" the Gaussian bump of height 0.2 with a1 = 2.5, T = 1,
S = 3 (omega_2 = 1.5 omega_1).  The seed moves the wavenumbers, the geometry, the incidence and the receivers.

`exact` restates the whole discrete scheme in plain torch, in 64 bits.
"""
import math

import numpy as np
import torch

PI = math.pi
FP64, MIXED = 0, 1
# azimuthal sample counts the library takes (2^a 3^b, multiples of 4)
M_SIZES = [32, 36, 48, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 324, 384, 432, 512]


def listed():
    return [
        # one step of a parameter sweep on a coarse mesh: the smallest call, latency and launches
        dict(name="sweep_step_n96", kind="solve", geom="dent", N=96, M=48, prec=MIXED, k=2.0, waves=1, azimuths=1,
             source=False, points=32),
        # FP64 reference run at the parity size of the dent
        dict(name="reference_fp64_n160", kind="solve", geom="dent", N=160, M=64, prec=FP64, k=2.0, waves=1, azimuths=1,
             source=False, points=32),
        # FP64 run of a refined mesh
        dict(name="fp64_n256", kind="solve", geom="dent", N=256, M=128, prec=FP64, k=2.0, waves=1, azimuths=1,
             source=False, points=64),
        # a point source above the dent, an odd number of nodes
        dict(name="source_n241", kind="solve", geom="dent", N=241, M=144, prec=MIXED, k=2.0, waves=1, azimuths=1,
             source=True, points=64),
        # eight polar angles times eight azimuths, the angle grid of a scattering pattern
        dict(name="angles_n384", kind="solve", geom="dent", N=384, M=192, prec=MIXED, k=2.0, waves=8, azimuths=8,
             source=False, points=64),
        # the finest mesh of a convergence study
        dict(name="study_n800", kind="solve", geom="dent", N=800, M=256, prec=MIXED, k=2.0, waves=1, azimuths=1,
             source=False, points=64),
        # independent instances (a wavenumber scan) in one call on two worker streams
        dict(name="batch4_n256", kind="batch", geom="dent", N=256, M=128, prec=MIXED, k=2.0, waves=4, count=4,
             points=32),
        # modal kernels of the benchmark's instance, the mixed path's arithmetic
        dict(name="kernels_mixed_n512", kind="kernels", geom="bump", N=512, M=256, prec=MIXED, k=4.0, lo=0, hi=128),
        # the same layer in FP64 with a radix-3 azimuthal size
        dict(name="kernels_fp64_n384", kind="kernels", geom="bump", N=384, M=192, prec=FP64, k=3.0, lo=0, hi=96),
        # a few low modes of a coarse mesh: the small call of that layer
        dict(name="kernels_fp64_n128", kind="kernels", geom="bump", N=128, M=64, prec=FP64, k=2.0, lo=0, hi=8),
        # close pairs of the large high-frequency instance
        dict(name="close_mixed_n1024", kind="close", geom="bump", N=1024, M=512, prec=MIXED, k=10.0, lo=0, hi=256),
        # a field map: many receivers, one wave
        dict(name="field_map_n512", kind="field", geom="bump", N=512, M=256, k=4.0, points=512, waves=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _azimuthal(rng, N, most=512):
    """An azimuthal size near N / 2, as the meshes are used."""
    near = [m for m in M_SIZES if 0.3 * N <= m <= 0.62 * N and m <= most]
    return rng.choice(near or [M_SIZES[0]])


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "kernels", "close", "field"])
    if kind == "solve":
        prec = rng.choice([MIXED, MIXED, FP64])
        N = _log_int(rng, 96, 288 if prec == FP64 else 640)
        waves = 1 if prec == FP64 else rng.choice([1, 1, 2, 3, 5, 8])
        M = _azimuthal(rng, N, 288)
        # a source half a unit above the interface needs M >= 96 to be resolved by the M-point rule
        return dict(kind=kind, geom="dent", N=N, M=M, prec=prec, k=2.0, waves=waves,
                    azimuths=rng.choice([1, 1, 4]) if waves > 1 else 1,
                    source=96 <= M and N <= 320 and rng.random() < 0.4, points=rng.choice([16, 33, 64]))
    if kind == "batch":
        N = _log_int(rng, 96, 320)
        return dict(kind=kind, geom="dent", N=N, M=_azimuthal(rng, N, 192), prec=MIXED, k=2.0,
                    waves=rng.choice([1, 3, 4]), count=rng.randint(2, 5), points=32)
    N = _log_int(rng, 96, 512 if kind == "kernels" else 900)
    M = _azimuthal(rng, N)
    lo = rng.choice([0, 0, 1, M // 8])
    hi = rng.choice([M // 2, M // 2, lo + 1 + M // 16])
    k = rng.choice([2.0, 3.0, 4.0])
    if kind == "field":
        return dict(kind=kind, geom="bump", N=N, M=M, k=k, points=_log_int(rng, 16, 512), waves=rng.choice([1, 1, 3, 8]))
    return dict(kind=kind, geom="bump", N=N, M=M, prec=rng.choice([FP64, MIXED]), k=k, lo=lo, hi=hi)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _instance(case, rng):
    """Keyword arguments of one Problem: the geometry, PML and wavenumbers of the case, moved by the seed."""
    k1 = case["k"] * PI * (1.0 + 0.03 * (rng.random() - 0.5))
    kw = dict(N=case["N"], M=case["M"], k1=k1)
    if case["geom"] == "dent":
        d = 1.0 + 0.05 * (rng.random() - 0.5)
        kw.update(k2=1.2 * k1, a1=2.0, T=2.0, S=2.0, curve="polyline", vertices=[(0.0, -d), (1.0, -d), (1.0, 0.0)])
    else:
        kw.update(k2=1.5 * k1, a1=2.5, T=1.0, S=3.0, bump_h=0.2 * (1.0 + 0.1 * (rng.random() - 0.5)))
    return kw


def _receivers(case, rng, n):
    """(rho, z, region) of n receivers well off the curve, upper and lower medium in turn."""
    region = np.arange(n) % 2
    rho = 1.8 * rng.random(n)
    depth = 0.8 if case["geom"] == "bump" else 1.6
    z = np.where(region == 0, 0.8 + rng.random(n), -depth - rng.random(n))
    return rho, z, region.astype(np.int32)


def _incidence(case, rng):
    """Keyword arguments of Problem.solve: distinct polar angles times azimuths, or point sources."""
    n, na = case["waves"], case.get("azimuths", 1)
    azimuth = np.tile(2.0 * PI * np.arange(na) / na, n) if na > 1 else None
    if case.get("source"):
        src = np.stack([0.2 + 0.2 * rng.random(n), 0.5 + 0.1 * rng.random(n)], axis=1)
        return dict(sources=np.repeat(src, na, axis=0), azimuth=azimuth)
    polar = PI / 3 * (np.arange(n) + 0.5 + 0.4 * rng.random(n)) / n
    return dict(polar=np.repeat(polar, na), azimuth=azimuth)


def _densities(case, rng, device):
    """Densities u1, phi1, u2, phi2 [mode][node][wave] whose modes decay as a scattered field's do."""
    shape = (case["M"] // 2, case["N"], case["waves"])
    g = torch.Generator(device=device)
    g.manual_seed(int(rng.integers(1 << 30)))
    decay = torch.exp(-torch.arange(shape[0], device=device, dtype=torch.float64) / (0.08 * case["M"]))[:, None, None]
    return {key: torch.complex(torch.randn(shape, generator=g, device=device, dtype=torch.float64),
                               torch.randn(shape, generator=g, device=device, dtype=torch.float64)) * decay
            for key in ("u1", "phi1", "u2", "phi2")}


def _inputs(case, seed, device):
    """Everything the seed makes, without the library."""
    rng = np.random.default_rng(seed)
    out = {"kw": [_instance(case, rng) for _ in range(case.get("count", 1))]}
    if "points" in case:
        out["receivers"] = _receivers(case, rng, case["points"])
    if case["kind"] in ("solve", "batch"):
        out["incidence"] = _incidence(case, rng)
    if case["kind"] == "field":
        out["densities"] = _densities(case, rng, device)
    return out


def prepare(case, seed):
    from paper_2412_11162_gb300 import Problem
    state = dict(case=case, **_inputs(case, seed, "cuda"))
    state["problems"] = [Problem(**kw) for kw in state["kw"]]
    if case["kind"] == "close":
        P = state["problems"][0]
        state["out"] = torch.empty((sum(P.near_count()), 4, case["hi"] - case["lo"]), dtype=torch.complex128,
                                   device="cuda")
    return state


def run(state):
    from paper_2412_11162_gb300 import binding as B
    from paper_2412_11162_gb300 import solve_batch
    case, P = state["case"], state["problems"][0]
    if case["kind"] == "solve":
        densities, _ = P.solve(precision=case["prec"], **state["incidence"])
        return P.field(*state["receivers"], densities)
    if case["kind"] == "batch":
        densities, _ = solve_batch(state["problems"], state["incidence"]["polar"], precision=case["prec"])
        return [Q.field(*state["receivers"], d) for Q, d in zip(state["problems"], densities)]
    if case["kind"] == "kernels":
        return P.modal_kernels(case["lo"], case["hi"], precision=case["prec"])
    if case["kind"] == "close":
        return B.pmlbie_close_pair_kernels(P.handle, case["prec"], case["lo"], case["hi"], state["out"])
    return P.field(*state["receivers"], state["densities"])


def work(case):
    """Bytes: the call's arrays once each.  Flops: the method's own steps -- samples of both media at M/2 + 1 angles
    of each unordered pair (about 250 operations with the exponentials), their transforms, and per mode the LU and
    the solves of the block system."""
    N, M = case["N"], case["M"]
    modes = case.get("hi", M // 2) - case.get("lo", 0)
    transform = 5.0 * (M // 2) * math.log2(M // 2) + 15.0 * (M // 2)
    pair = 250.0 * (M // 2 + 1) + 4.0 * transform
    waves = case.get("waves", 1)
    field = case.get("points", 0) * (N * (0.5 * pair + 16.0 * modes * waves * case.get("azimuths", 1)))
    out = 16.0 * case.get("points", 0) * modes * waves * case.get("azimuths", 1)
    if case["kind"] in ("solve", "batch"):
        n = 2.0 * N
        flops = 0.5 * N * N * pair + modes * (8.0 / 3.0 * n ** 3 + 8.0 * n * n * waves)
        return dict(bytes=case.get("count", 1) * out, flops=case.get("count", 1) * (flops + field))
    if case["kind"] == "kernels":
        return dict(bytes=16.0 * 4 * N * N * modes, flops=0.5 * N * N * pair)
    if case["kind"] == "close":
        # about 20 corrections per node and 16 pi N^2 / M grid pairs within the split distance
        pairs = 20.0 * N + 0.28 * 8.0 * 2.0 * PI * N * N / M
        return dict(bytes=16.0 * 4 * pairs * modes, flops=pairs * (2.0 * pair + 12.0 * transform))
    return dict(bytes=out + 16.0 * 4 * N * modes * waves, flops=field)


# ----------------------------------------------------------------------------
# the same results in plain torch, 64 bits: the scheme of the paper as the header states it
# ----------------------------------------------------------------------------
# Alpert's hybrid rule for a logarithmic singularity, order 10 (10 nodes, 10 grid points skipped)
ALPERT_X = [0.0043165781478727050961, 0.062462243891320907225, 0.29146925421248575821, 0.82963840779149708395,
            1.77255591469832904711, 3.11814318303491891616, 4.74121441516633602128, 6.41006450395182652724,
            7.86005278732722340490, 8.99273223152158502904]
ALPERT_W = [0.0163864137528612664170, 0.120239663177631007894, 0.361947963293578402058, 0.731288522266955256195,
            1.15465327444656328787, 1.51539238394578760384, 1.69105158191145748227, 1.59950687764490668255,
            1.27833398679945484979, 1.03119933276081047176]
SKIP, STENCIL = 10, 10


class _Curve:
    """Graded nodes, PML tables and pair geometry of one instance."""

    def __init__(self, kw, dev):
        self.kw, self.dev, self.p = kw, dev, 6
        self.L = kw["a1"] + kw["T"]
        if kw.get("curve") == "polyline":
            v = list(kw["vertices"]) + [(self.L, 0.0)]
            self.segs = [("line", a, b) for a, b in zip(v[:-1], v[1:])]
        else:
            self.segs = [("bump", kw["bump_h"]), ("line", (1.0, 0.0), (self.L, 0.0))]
        x, w = np.polynomial.legendre.leggauss(64)
        lens = []
        for s in self.segs:
            _, _, dr, dz = self._seg(s, torch.tensor(0.5 * (x + 1.0)))
            lens.append(float(0.5 * (torch.tensor(w) * torch.hypot(dr, dz)).sum()))
        Nt = self.Nt = kw["N"] + len(lens)
        steps = [max(2 * SKIP + 4, int(round(Nt * l / sum(lens)))) for l in lens]
        steps[int(np.argmax(lens))] += Nt - sum(steps)
        self.h = 1.0 / Nt
        self.brk = [0] + [int(b) for b in np.cumsum(steps)]
        self.grid = torch.tensor([i for i in range(Nt + 1) if i not in set(self.brk)], device=dev)
        self.unknown = torch.full((Nt + 1,), -1, dtype=torch.long, device=dev)
        self.unknown[self.grid] = torch.arange(kw["N"], device=dev)
        self.nodes = self.at(self.grid.double() * self.h)

    @staticmethod
    def _seg(seg, s):
        one = torch.ones_like(s)
        if seg[0] == "bump":
            w, e0 = 0.5, math.exp(-1.0 / 0.5)
            g = torch.exp(-s * s / w)
            return s, seg[1] * (g - e0) / (1 - e0), one, seg[1] * (-2.0 * s / w) * g / (1 - e0)
        (r0, z0), (r1, z1) = seg[1:]
        return r0 + s * (r1 - r0), z0 + s * (z1 - z0), (r1 - r0) * one, (z1 - z0) * one

    @staticmethod
    def _offset(seg, s, sc, end):
        """r(s) minus the segment's start (end 0) or end (end 1), without cancellation; sc = 1 - s."""
        if seg[0] == "bump":
            w, c = 0.5, seg[1] / (1 - math.exp(-1.0 / 0.5))
            if end == 0:
                return s, c * torch.expm1(-s * s / w)
            return -sc, c * math.exp(-1.0 / w) * torch.expm1(sc * (1.0 + s) / w)
        (r0, z0), (r1, z1) = seg[1:]
        t = s if end == 0 else -sc
        return t * (r1 - r0), t * (z1 - z0)

    def sigma(self, rho):
        kw, p = self.kw, self.p
        rb = (rho - self.L) / kw["T"]
        f1 = (0.5 - 1.0 / p) * rb ** 3 + rb / p + 0.5
        val = 2.0 * kw["S"] * f1 ** p / (f1 ** p + (1.0 - f1) ** p)
        val = torch.where(rho >= self.L, torch.full_like(val, kw["S"]), val)
        return torch.where(rho > kw["a1"], val, torch.zeros_like(val))

    def delta_I(self, rho, step, panels=8):
        """Integral of sigma over [rho, rho + step], clipped where sigma starts."""
        a1 = self.kw["a1"]
        lo, hi = torch.minimum(rho, rho + step), torch.maximum(rho, rho + step)
        inside = lo >= a1
        start = torch.where(inside, rho, torch.full_like(rho, a1))
        length = torch.where(inside, step, (hi - a1).clamp(min=0.0) * torch.sign(step))
        span = torch.where(inside, length, length.abs())
        x, w = np.polynomial.legendre.leggauss(16)
        tot = torch.zeros_like(rho)
        for k in range(panels):
            for xi, wi in zip(x, w):
                tot = tot + (0.5 / panels * wi) * self.sigma(start + span * ((k + 0.5 * (xi + 1.0)) / panels))
        return length * tot

    def at(self, t):
        n, dev = t.numel(), self.dev
        rho, z, dr, dz, ox, oz = (torch.zeros(n, dtype=torch.float64, device=dev) for _ in range(6))
        bk = torch.zeros(n, dtype=torch.long, device=dev)
        seg_of = torch.bucketize(t, torch.tensor([b * self.h for b in self.brk], device=dev, dtype=torch.float64),
                                 right=True).sub(1).clamp(0, len(self.segs) - 1)
        for k, seg in enumerate(self.segs):
            m = seg_of == k
            t0, t1 = self.brk[k] * self.h, self.brk[k + 1] * self.h
            u = (t[m] - t0) / (t1 - t0)
            p, A = self.p, 0.5 - 1.0 / self.p
            xi = 2.0 * u - 1.0
            x1 = 2.0 * u * (A * xi * xi - A * xi + 0.5)
            x2 = 2.0 * (1.0 - u) * (A * xi * xi + A * xi + 0.5)
            den = x1 ** p + x2 ** p
            s, sc = x1 ** p / den, x2 ** p / den
            ds = p * x1 ** (p - 1) * x2 ** (p - 1) / den ** 2 * (3.0 * A * xi * xi + 1.0 / p) * 2.0
            r_, z_, dr_, dz_ = self._seg(seg, s)
            rho[m], z[m], dr[m], dz[m] = r_, z_, dr_ * ds / (t1 - t0), dz_ * ds / (t1 - t0)
            end = u > 0.5
            a, b = self._offset(seg, s, sc, 0), self._offset(seg, s, sc, 1)
            ox[m], oz[m] = torch.where(end, b[0], a[0]), torch.where(end, b[1], a[1])
            bk[m] = k + end.long()
        speed = torch.hypot(dr, dz)
        nr, nz = dz / speed, -dr / speed
        I = self.delta_I(torch.full_like(rho, self.kw["a1"]), (rho - self.kw["a1"]).clamp(min=0.0), 64)
        alpha = torch.complex(torch.ones_like(rho), self.sigma(rho))
        rt = torch.complex(rho, I)
        return dict(rho=rho, z=z, speed=speed, nr=nr, nz=nz, I=I, rt=rt, ncr=nr * (rt / rho) / alpha,
                    ncz=nz * (rt / rho) * alpha, bk=bk, ox=ox, oz=oz)

    def pair(self, tgt, src):
        """Pair quantities of two tables of equal length."""
        same = tgt["bk"] == src["bk"]
        dr = torch.where(same, tgt["ox"] - src["ox"], tgt["rho"] - src["rho"])
        dz = torch.where(same, tgt["oz"] - src["oz"], tgt["z"] - src["z"])
        drt = torch.complex(dr, self.delta_I(src["rho"], dr))
        return dict(d2=drt * drt + dz * dz, rr=tgt["rt"] * src["rt"], nd0=-src["ncr"] * drt - src["ncz"] * dz,
                    nds=2.0 * src["ncr"] * tgt["rt"], subst=(tgt["I"] > 0) | (src["I"] > 0), dr=dr, dz=dz,
                    rho=tgt["rho"], srho=src["rho"], nr=src["nr"], nz=src["nz"])


def _take(d, i):
    return {k: v[i] for k, v in d.items()}


def _taylor(L=5):
    e = [(-2j) ** k / math.factorial(k) for k in range(L + 1)]
    a = [((1.0 if k == 0 else 0.0) + e[k]) / 2.0 for k in range(L + 1)]
    b = [a[k] + (-1j * ((1.0 if k == 1 else 0.0) - e[k - 1]) / 2.0 if k else 0.0) for k in range(L + 1)]
    return a, b


def _poly(c, q):
    out = torch.zeros_like(q)
    for ck in reversed(c):
        out = out * q + ck
    return out


def _sin2(M, dev):
    return torch.sin(PI * torch.arange(M, device=dev, dtype=torch.float64) / M) ** 2


def _modes(x, n):
    return torch.fft.fft(x, dim=-1)[:, :n] * (2.0 * PI / x.shape[-1])


def _far(g, w, sign, M):
    s2 = _sin2(M, g["d2"].device)
    R = torch.sqrt(g["d2"][:, None] + 4.0 * g["rr"][:, None] * s2)
    q = w * R
    S = torch.exp(1j * q) / (4.0 * PI * R)
    K = -sign * (g["nd0"][:, None] + g["nds"][:, None] * s2) / (R * R) * S * (1.0 - 1j * q)
    return _modes(S, M // 2), _modes(K, M // 2)


def _psi_rule(mmax, dev):
    """Gauss-Legendre panels on [0, pi], graded toward 0, for integrands with a near-singularity at 0."""
    cap, edges = min(0.25, 16.0 / (mmax + 1)), [0.0, 2.0 ** -52]
    while edges[-1] * 2 < 1.0:
        edges.append(edges[-1] * 2)
    edges.append(PI)
    fine = [0.0]
    for a, b in zip(edges[:-1], edges[1:]):
        n = max(1, math.ceil((b - a) / cap))
        fine += [a + (b - a) * i / n for i in range(1, n + 1)]
    x, w = np.polynomial.legendre.leggauss(32)
    e = np.array(fine)
    pts = (0.5 * (e[:-1] + e[1:])[:, None] + 0.5 * (e[1:] - e[:-1])[:, None] * x).ravel()
    wts = (0.5 * (e[1:] - e[:-1])[:, None] * w).ravel()
    return torch.tensor(pts, device=dev), torch.tensor(wts, device=dev)


def _matmul(z, c):
    return torch.complex(z.real @ c, z.imag @ c)


def _near(g, ws, M):
    """Split kernels of both media: [(S, K), (S, K)]."""
    dev, nh = g["d2"].device, M // 2
    pts, wts = _psi_rule(M - 2, dev)
    C = 2.0 * wts[:, None] * torch.cos(pts[:, None] * torch.arange(M - 1, device=dev))
    s2 = torch.sin(0.5 * pts) ** 2
    R2 = g["d2"][:, None] + 4.0 * g["rr"][:, None] * s2
    iR = 1.0 / torch.sqrt(R2)
    Z = _matmul(iR / (4.0 * PI), C)
    D = _matmul(-(g["nd0"][:, None] + g["nds"][:, None] * s2) * iR / R2 / (4.0 * PI), C)
    del R2, iR
    a, b = _taylor()
    u1, v3 = [-x for x in a[1:]], [-x for x in b[3:]]
    s2 = _sin2(M, dev)
    R = torch.sqrt(g["d2"][:, None] + 4.0 * g["rr"][:, None] * s2)
    ND = g["nd0"][:, None] + g["nds"][:, None] * s2
    sub = g["subst"][:, None]
    k = torch.arange(-(nh - 1), nh, device=dev)
    out = []
    for w, sign in zip(ws, (1.0, -1.0)):
        q = w * R
        q2, e, sn, cs = q * q, torch.exp(1j * q), torch.sin(q), torch.cos(q)
        sinc = torch.where(q.abs() < 1e-3, 1.0 - q2 / 6.0 + q2 * q2 / 120.0, sn / q)
        h4 = torch.where(q.abs() < 1e-2, 1.0 / 3.0 - q2 / 30.0 + q2 * q2 / 840.0 - q2 ** 3 / 45360.0,
                         (sn - q * cs) / (q * q2))
        f1 = torch.where(sub, e * _poly(a, q), cs)
        r1 = w / (4.0 * PI) * torch.where(sub, e * _poly(u1, q), 1j * sinc)
        f3 = torch.where(sub, e * _poly(b, q), cs + q * sn)
        r3 = -sign * w ** 3 / (4.0 * PI) * ND * torch.where(sub, e * _poly(v3, q), 1j * h4)
        F1, F3 = torch.fft.fft(f1, dim=1) * (1.0 / M), torch.fft.fft(f3, dim=1) * (sign / M)
        F1, F3 = F1[:, k % M], F3[:, k % M]          # coefficients |k| < M/2, over 2 pi
        S, K = _modes(r1, nh), _modes(r3, nh)
        for n in range(nh):
            idx = (n - k).abs()
            S[:, n] += (Z[:, idx] * F1).sum(1)
            K[:, n] += (D[:, idx] * F3).sum(1)
        out.append((S, K))
    return out


def _all_kernels(c, tgt, src, chunk):
    """[S^a, K^a, S^b, K^b] as (pairs, modes) of every pair of two tables, and the mask of the close ones."""
    M, ws = c.kw["M"], (c.kw["k1"], c.kw["k2"])
    n = tgt["rho"].numel()
    out = [torch.empty((n, M // 2), dtype=torch.complex128, device=c.dev) for _ in range(4)]
    close = torch.zeros(n, dtype=torch.bool, device=c.dev)
    for i in range(0, n, 1 << 20):
        g = c.pair(_take(tgt, slice(i, i + (1 << 20))), _take(src, slice(i, i + (1 << 20))))
        x = g["d2"] / g["rr"]
        near = torch.sqrt(((x.abs() + x.real) * 0.5).clamp(min=0.0)) < 8.0 * 2.0 * PI / M
        close[i:i + near.numel()] = near
        at = torch.nonzero(~near).flatten()
        for j in at.split(chunk):
            h = _take(g, j)
            for r in range(2):
                out[2 * r][i + j], out[2 * r + 1][i + j] = _far(h, ws[r], 1.0 - 2.0 * r, M)
        at = torch.nonzero(near).flatten()
        for j in at.split(max(1, chunk // 16)):
            for r, (S, K) in enumerate(_near(_take(g, j), ws, M)):
                out[2 * r][i + j], out[2 * r + 1][i + j] = S, K
    return out, close


def _grid_pairs(c):
    l, m = torch.nonzero((c.grid[:, None] - c.grid[None, :]).abs() >= SKIP, as_tuple=True)
    return l, m


def _corrections(c):
    """(target, source table, stencil unknowns, coefficients) of every Alpert correction point."""
    dev, h, Nt = c.dev, c.h, c.Nt
    x = torch.tensor(ALPERT_X, dtype=torch.float64, device=dev)
    w = torch.tensor(ALPERT_W, dtype=torch.float64, device=dev)
    t = c.grid.double()[:, None, None] * h + torch.tensor([-h, h], device=dev, dtype=torch.float64)[None, :, None] * x
    l = torch.arange(c.kw["N"], device=dev)[:, None, None].expand(t.shape)
    wk = (w * h).expand(t.shape)
    ok = (t > 0.0) & (t < 1.0)
    t, l, wk = t[ok], l[ok], wk[ok]
    i0 = (torch.floor(t / h).long() - (STENCIL // 2 - 1)).clamp(0, Nt + 1 - STENCIL)
    idx = i0[:, None] + torch.arange(STENCIL, device=dev)
    tj = idx.double() * h
    lag = torch.ones_like(tj)
    for a in range(STENCIL):
        for b in range(STENCIL):
            if a != b:
                lag[:, a] *= (t - tj[:, b]) / (tj[:, a] - tj[:, b])
    m = c.unknown[idx]
    return l, c.at(t), m.clamp(min=0), torch.where(m >= 0, wk[:, None] * lag, torch.zeros_like(lag))


def _matrix(c, values, grid, corr, weight):
    """Per-mode matrices [mode][l][m] from grid values and correction values (pairs, modes)."""
    (l, m), (lc, _, mc, coef), ng = grid, corr, grid[0].numel()
    N, nm = c.kw["N"], values.shape[1]
    A = torch.zeros((N, N, nm), dtype=values.dtype, device=c.dev)
    A[l, m] = values[:ng] * c.h
    for s in range(STENCIL):
        A.index_put_((lc, mc[:, s]), coef[:, s, None].to(values.dtype) * values[ng:], accumulate=True)
    return (A * weight[None, :, None]).permute(2, 0, 1).contiguous()


def _diagonal(c, grid, corr):
    n, (l, m) = c.nodes, grid
    pts, wts = _psi_rule(8, c.dev)
    s2 = torch.sin(0.5 * pts) ** 2

    def mode0(g):
        out = []
        for i in range(0, g["dr"].numel(), 1 << 15):
            h = _take(g, slice(i, i + (1 << 15)))
            R2 = (h["dr"] ** 2 + h["dz"] ** 2)[:, None] + 4.0 * (h["rho"] * h["srho"])[:, None] * s2
            num = h["nr"][:, None] * (2.0 * h["rho"][:, None] * s2 - h["dr"][:, None]) - (h["nz"] * h["dz"])[:, None]
            out.append((-num / (4.0 * PI * R2 ** 1.5)) @ (2.0 * wts))
        return torch.cat(out)

    values = torch.cat([mode0(c.pair(_take(n, l), _take(n, m))), mode0(c.pair(_take(n, corr[0]), corr[1]))])[:, None]
    K0 = _matrix(c, values, grid, corr, 2.0 * n["rho"] * n["speed"])[0].sum(1)
    th = 2.0 * PI * torch.arange(4096, device=c.dev, dtype=torch.float64) / 4096
    s = -n["rho"][:, None] * torch.cos(th) + torch.sqrt(c.L ** 2 - (n["rho"][:, None] * torch.sin(th)) ** 2)
    az = n["z"].abs()[:, None]
    disc = 2.0 * PI - (2.0 * PI / 4096) * (az / torch.sqrt(az * az + s * s)).sum(1)
    full = torch.where(n["z"] > 0, 4.0 * PI - disc, torch.where(n["z"] < 0, disc, torch.full_like(disc, 2.0 * PI)))
    return K0 - full / (2.0 * PI), -K0 - (4.0 * PI - full) / (2.0 * PI)


def _jumps(c, inc):
    """b1, b2 as [mode][node][wave] of the plane waves or the point sources."""
    kw, n, dev = c.kw, c.nodes, c.dev
    M, w1, w2 = kw["M"], kw["k1"], kw["k2"]
    order = torch.arange(M // 2, device=dev, dtype=torch.float64)
    b1, b2 = [], []
    count = len(inc["sources"] if "sources" in inc else inc["polar"])
    for r in range(count):
        if "sources" in inc:
            rs, zs = (float(v) for v in inc["sources"][r])
            drt = torch.complex(rs - n["rho"], -n["I"])
            dz = zs - n["z"]
            g = dict(d2=drt * drt + dz * dz, rr=rs * n["rt"], nd0=-n["ncr"] * drt - n["ncz"] * dz, nds=2.0 * n["ncr"] * rs)
            S, K = _far(g, w1, 1.0, M)
            v1, v2 = -S, -K * n["speed"][:, None]
        else:
            ph = float(inc["polar"][r])
            kx, kz = w1 * math.sin(ph), w1 * math.cos(ph)
            ks = complex(math.sqrt(w2 * w2 - kx * kx)) if w2 > kx else 1j * math.sqrt(kx * kx - w2 * w2)
            R = 2.0 / (1.0 + ks / kz) - 1.0
            th = 2.0 * PI * torch.arange(M, device=dev, dtype=torch.float64) / M
            z = n["z"][:, None]
            lat = torch.exp(-1j * kx * n["rho"][:, None] * torch.cos(th))
            ui, ur = lat * torch.exp(-1j * kz * z), R * lat * torch.exp(1j * kz * z)
            u1, u2 = ui + ur, (R + 1.0) * lat * torch.exp(-1j * ks * z)
            across = -1j * kx * torch.cos(th) * n["nr"][:, None]
            d1 = across * u1 + n["nz"][:, None] * 1j * kz * (ur - ui)
            d2 = across * u2 - n["nz"][:, None] * 1j * ks * u2
            v1, v2 = _modes(u2 - u1, M // 2), _modes(d2 - d1, M // 2) * n["speed"][:, None]
        az = 0.0 if inc.get("azimuth") is None else float(inc["azimuth"][r])
        rot = torch.exp(-1j * order * az)
        b1.append((v1 * rot).T)
        b2.append((v2 * rot).T)
    return torch.stack(b1, 2), torch.stack(b2, 2)


def _solve(c, inc):
    n, N = c.nodes, c.kw["N"]
    grid, corr = _grid_pairs(c), _corrections(c)
    l, m = grid
    tgt = {k: torch.cat([n[k][l], n[k][corr[0]]]) for k in n}
    src = {k: torch.cat([n[k][m], corr[1][k]]) for k in n}
    val, _ = _all_kernels(c, tgt, src, 1 << 15)
    wu, wp = 2.0 * n["rho"] * n["speed"], 2.0 * n["rho"]
    Da, Db = _diagonal(c, grid, corr)
    nm = c.kw["M"] // 2
    A = torch.empty((nm, 2 * N, 2 * N), dtype=torch.complex128, device=c.dev)
    for r, (D, sign) in enumerate(((Da, -1.0), (Db, 1.0))):
        rows = slice(r * N, (r + 1) * N)
        A[:, rows, N:] = sign * _matrix(c, val[2 * r], grid, corr, wp)
        A[:, rows, :N] = _matrix(c, val[2 * r + 1], grid, corr, wu) - torch.diag(D)
    del val
    b1, b2 = _jumps(c, inc)
    B = torch.cat([torch.zeros_like(b1), A[:, N:] @ torch.cat([b1, b2], 1)], 1)
    x = torch.cat([torch.linalg.solve(A[i:i + 8], B[i:i + 8]) for i in range(0, nm, 8)])
    u, phi = x[:, :N], x[:, N:]
    return dict(u1=u, phi1=phi, u2=u - b1, phi2=phi - b2)


def _field(c, receivers, dens):
    n, M = c.nodes, c.kw["M"]
    rho, z, region = receivers
    out = []
    for p in range(len(rho)):
        up = region[p] == 0
        drt = torch.complex(float(rho[p]) - n["rho"], -n["I"])
        dz = float(z[p]) - n["z"]
        g = dict(d2=drt * drt + dz * dz, rr=float(rho[p]) * n["rt"], nd0=-n["ncr"] * drt - n["ncz"] * dz,
                 nds=2.0 * n["ncr"] * float(rho[p]))
        S, K = _far(g, c.kw["k1"] if up else c.kw["k2"], 1.0 if up else -1.0, M)
        u, phi = (dens["u1"], dens["phi1"]) if up else (dens["u2"], dens["phi2"])
        cs = (0.5 if up else -0.5) * c.h * (2.0 * n["rho"])[:, None] * S
        ck = -0.5 * c.h * (2.0 * n["rho"] * n["speed"])[:, None] * K
        out.append(torch.einsum("mn,nmr->nr", cs, phi) + torch.einsum("mn,nmr->nr", ck, u))
    return torch.stack(out, 1)


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    inp = _inputs(case, seed, dev)
    N, M = case["N"], case["M"]
    if case["kind"] == "close" and N > 600:      # the Laplace modes' quadrature of all pairs takes too long
        return None
    curves = [_Curve(kw, dev) for kw in inp["kw"]]
    c = curves[0]
    if case["kind"] in ("solve", "batch"):
        got = [_field(q, inp["receivers"], _solve(q, inp["incidence"])) for q in curves]
        return got if case["kind"] == "batch" else got[0]
    if case["kind"] == "field":
        return _field(c, inp["receivers"], inp["densities"])
    l, m = _grid_pairs(c)
    if case["kind"] == "kernels":
        val, _ = _all_kernels(c, _take(c.nodes, l), _take(c.nodes, m), 1 << 15)
        out = torch.zeros((case["hi"] - case["lo"], 4, N, N), dtype=torch.complex128, device=dev)
        for k in range(4):
            out[:, k, l, m] = val[k][:, case["lo"]:case["hi"]].T
        return out
    corr = _corrections(c)
    g = c.pair(_take(c.nodes, l), _take(c.nodes, m))
    x = g["d2"] / g["rr"]
    near = torch.sqrt(((x.abs() + x.real) * 0.5).clamp(min=0.0)) < 8.0 * 2.0 * PI / M
    l, m = l[near], m[near]
    tgt = {k: torch.cat([c.nodes[k][l], c.nodes[k][corr[0]]]) for k in c.nodes}
    src = {k: torch.cat([c.nodes[k][m], corr[1][k]]) for k in c.nodes}
    val, _ = _all_kernels(c, tgt, src, 1 << 15)
    return torch.stack([v[:, case["lo"]:case["hi"]] for v in val], 1)
