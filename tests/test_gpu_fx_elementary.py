"""The sampling loops' exp, sin / cos and 1/sqrt (csrc/fxtrig.cuh), point by point through
pmlbie_selftest_elementary selectors 30 .. 32, against the host's extended precision.

Bars: the functions' stated errors plus the rounding of the result to a double --
exp 2^-55.7 + 2^-53 relative; sin and cos 2^-57.9 + 2^-54 absolute, plus |x| 2^-63 (the 64
bits of 1 / 2 pi) and 2^-61 (the fraction of a turn, cut at 2^-64 turns); 1/sqrt 2^-52
(about 1 ulp) relative.  sin(q)/q, at most 1, to 2^-51 and (sin q - q cos q)/q^3, at most
1/3, to 2^-50: their series below q = 1/2 to an ulp; above, the sine's rounding over q
and, of the difference, (2^-57.9 + 2^-53 q) 8 at q = 1/2.
"""
import numpy as np
import pytest

from test_gpu_elementary import _grid, _run

pytestmark = pytest.mark.gpu
LD = np.longdouble


def test_exp():
    x = np.concatenate([_grid(-707.0, 709.0, 1 << 18, 1), _grid(-1.0, 1.0, 1 << 17, 2),
                        # powers of two of either sign: shifts of the fraction, nothing left of it, all of it
                        *(s * 2.0 ** np.arange(-80, 10) for s in (-1, 1)),
                        # next to multiples of ln 2 / 256 (table entries) and of ln 2
                        *(np.arange(-2000, 2001) * (np.log(2) / 256) * (1 + d) for d in (-1e-15, 0, 1e-15)),
                        np.arange(-1000, 1001) * np.log(2), [0.0, -0.0, 1e-300, -1e-300, 5e-324]])
    got, ref = _run(30, x), np.exp(x.astype(LD))
    err = np.abs(got.astype(LD) - ref) / ref
    assert np.max(err) <= 2.0 ** -53 + 2.0 ** -55.7, (float(np.max(err)) * 2.0 ** 53, x[np.argmax(err)])
    assert np.all(_run(30, np.array([-709.0, -750.0, -1023.5, -1024.0, -1e4, -1e300, -np.inf])) == 0.0)
    assert np.all(_run(30, np.array([710.0, 750.0, 1023.5, 1024.0, 1e4, 1e300, np.inf])) == np.inf)


def test_sin_cos():
    x = np.concatenate([_grid(0.0, 8.0, 1 << 18, 3), _grid(0.0, 2.0 ** 20, 1 << 18, 4), _grid(0.0, 2.0 ** 40, 1 << 12, 5),
                        2.0 ** np.arange(-80, 41),
                        # next to the table's angles, half way between them, and the quadrants' ends
                        *(np.arange(0, 8193) * (np.pi / 1024) * (1 + d) for d in (-1e-15, 0, 1e-15)),
                        np.arange(0, 4001) * (np.pi / 2), [0.0, 1e-300, 5e-324]])
    got = _run(31, x)
    bar = 2.0 ** -54 + 2.0 ** -57.9 + x * 2.0 ** -63 + 2.0 ** -61
    for k, ref in enumerate((np.sin(x.astype(LD)), np.cos(x.astype(LD)))):
        err = np.abs(got[k::2].astype(LD) - ref)
        assert np.all(err <= bar), (k, float(np.max(err / bar)), x[np.argmax(err / bar)])


def test_rsqrt():
    rng = np.random.default_rng(6)
    x = np.concatenate([2.0 ** rng.uniform(-1021, 1023, 1 << 18), _grid(0.5, 8.0, 1 << 17, 7),
                        # every exponent, odd and even, at both ends of the significand
                        *(2.0 ** np.arange(-1022, 1024) * v for v in (1.0, 2 - 2.0 ** -52))])
    got, ref = _run(32, x), 1 / np.sqrt(x.astype(LD))
    err = np.abs(got.astype(LD) - ref) / ref
    assert np.max(err) <= 2.0 ** -52, (float(np.max(err)) * 2.0 ** 52, x[np.argmax(err)])
    # outside: NaN
    assert np.all(np.isnan(_run(32, np.array([0.0, -0.0, 5e-324, 2.0 ** -1023, -1.0, -np.inf, np.inf, np.nan]))))


def test_field_on_a_node_is_not_a_number():
    """The kernels are infinite there: every mode of that receiver, and of no other, is NaN."""
    import torch
    from paper_2412_11162_gb300 import Problem
    P = Problem(2 * np.pi, 3 * np.pi, 64, 32)
    node, m = P.nodes(), 20
    one = torch.ones((P.n_modes, P.N, 1), dtype=torch.complex128, device="cuda")
    rho, z = np.array([node["rho"][m], 0.7]), np.array([node["z"][m], 0.9])
    for region in ([0, 0], [1, 0]):
        got = P.field(rho, z, np.array(region), dict(u1=one, phi1=one, u2=one, phi2=one)).cpu().numpy()
        assert np.all(np.isnan(got[:, 0])) and np.all(np.isfinite(got[:, 1]))


def test_small_phase_quotients():
    q = np.concatenate([np.exp(_grid(np.log(1e-12), np.log(30.0), 1 << 18, 8)), _grid(0.0005, 2.0, 1 << 17, 9),
                        *(v * (1 + np.array([-1e-9, 0.0, 1e-9])) for v in (1e-3, 1e-2, 0.5))])
    x = q.astype(LD)
    s, k = np.zeros_like(x), np.zeros_like(x)
    ts, tk = np.ones_like(x), np.ones_like(x) / 3          # power series, all terms that count for q < 1
    for j in range(16):
        s, k = s + ts, k + tk
        ts = ts * -x * x / ((2 * j + 2) * (2 * j + 3))
        tk = tk * -x * x / ((2 * j + 2) * (2 * j + 5))
    big = x > 1
    s[big], k[big] = np.sin(x[big]) / x[big], (np.sin(x[big]) - x[big] * np.cos(x[big])) / x[big] ** 3
    for fn, ref, bar in ((33, s, 2.0 ** -51), (34, k, 2.0 ** -50)):
        err = np.abs(_run(fn, q).astype(LD) - ref)
        assert np.max(err) <= bar, (fn, float(np.max(err)) * 2.0 ** 53, q[np.argmax(err)])
