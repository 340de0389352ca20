"""The dense complex128 kernels of the solves, entry by entry: integer products there keep
bits relative to a row's and a column's largest entry, a double relative to the entry.

Bar for every entry of P A - L U: (8 sqrt(n) + 16) u of the entry of |L| |U| (u = 2^-53).
A complex multiply-add errs by at most (1 + sqrt 5) u of its terms, a sum of n of them by
4 sqrt(n) u with errors of independent signs, in the elimination and again in the test's
own product; a pivot's reciprocal and the product with it by 16 u.  Products A X against
the same bar times the entry of |A| |X|.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def bar(n):
    return (8 * n ** 0.5 + 16) * U


def matrices(n, seed):
    """Three matrices of order n: graded away from the diagonal as the modal kernels of
    high modes next to the axis are (down to 2^-90), with rows and columns of any scale
    (2^-40 .. 2^40), and plain."""
    rng = np.random.default_rng(seed)
    E = rng.standard_normal((3, n, n)) + 1j * rng.standard_normal((3, n, n))
    t = np.sort(rng.random(n))
    E[0] *= np.exp(-62.0 * np.abs(t[:, None] - t[None]))
    E[1] *= 2.0 ** rng.integers(-40, 41, n)[:, None] * 2.0 ** rng.integers(-40, 41, n)
    return E


# one panel, its sub-panels of 8 columns: none, remainders, all
@pytest.mark.parametrize("n", [7, 8, 9, 16, 17, 31, 32])
def test_factors_of_one_panel(n):
    check_factors(n)


# tensor-core updates of 64 x 32 tiles: trailing blocks of 1 .. 66 rows, whole tiles, several
# row blocks (of the three matrices two are updated together, then one)
@pytest.mark.parametrize("n", [33, 34, 48, 64, 65, 96, 97, 98, 130, 160, 258])
def test_factors_of_several_panels(n):
    check_factors(n)


def check_factors(n):
    import torch
    from paper_2412_11162_gb300 import binding as B
    A = matrices(n, n)
    F = torch.tensor(A.transpose(0, 2, 1).copy(), device="cuda")
    perm = torch.empty((3, n), dtype=torch.int32, device="cuda")
    B.pmlbie_selftest_lu(F, perm)
    F, perm = F.cpu().numpy().transpose(0, 2, 1), perm.cpu().numpy()
    for b in range(3):
        L, R = np.tril(F[b], -1) + np.eye(n), np.triu(F[b])
        assert np.max(np.abs(L)) <= 1 + 4 * U            # partial pivoting
        ratio = np.abs(A[b][perm[b]] - L @ R) / (np.abs(L) @ np.abs(R))
        assert np.max(ratio) <= bar(n), (b, np.max(ratio) / U, np.unravel_index(np.argmax(ratio), ratio.shape))


# row blocks of 128 and column chunks of 32 (of either half of the columns) with remainders,
# groups of 8 right-hand sides with remainders, one right-hand side; X of any scale from
# row to row
@pytest.mark.parametrize("n,waves", [(2, 2), (62, 2), (64, 3), (66, 8), (130, 9), (190, 16), (258, 17), (258, 1)])
def test_products(n, waves):
    import torch
    from paper_2412_11162_gb300 import binding as B
    A, rng = matrices(n, n), np.random.default_rng(waves)
    X = rng.standard_normal((3, n, waves)) + 1j * rng.standard_normal((3, n, waves))
    X *= 2.0 ** rng.integers(-40, 41, (3, n, 1))
    Y = torch.empty((3, n, waves), dtype=torch.complex128, device="cuda")
    B.pmlbie_selftest_product(torch.tensor(A.transpose(0, 2, 1).copy(), device="cuda"), torch.tensor(X, device="cuda"), Y)
    ratio = np.abs(Y.cpu().numpy() - A @ X) / (np.abs(A) @ np.abs(X))
    assert np.max(ratio) <= bar(n), (np.max(ratio) / U, np.unravel_index(np.argmax(ratio), ratio.shape))
