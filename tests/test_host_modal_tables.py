"""The tables of the operators in Legendre modes are rounded once: every entry
within half a unit of its last place of its value in extended precision (numpy's
long double; a hundredth of a unit for that value's own rounding).  The values
come another way than the library's: node to mode by inverting the modes at the
Gauss-Lobatto nodes, restrictions from the modes at nodes of the part.

Restrictions to small parts have entries down to 2^-68, what is left of sums of
modes of up to sqrt(17): nine products of up to 17 / 9 with some ten roundings
of 2^-64 each leave up to 1e-17 in them, and as much in the value compared
with."""
import numpy as np
import pytest

X = np.longdouble


def _modes(n, x):
    """(len(x), n): sqrt(2k+1) P_k at x in [-1, 1], and P_{n-1}, P_{n-1}'."""
    P = np.zeros((n + 1, len(x)), dtype=X)
    P[0], P[1] = 1, x
    for k in range(1, n):
        P[k + 1] = ((2 * k + 1) * x * P[k] - k * P[k - 1]) / X(k + 1)
    return (np.sqrt(2 * np.arange(n, dtype=X) + 1)[:, None] * P[:n]).T, P[n - 1], P[n - 2]


def _gll(p):
    inner = np.polynomial.legendre.Legendre.basis(p).deriv().roots() if p > 1 else np.zeros(0)
    x = np.sort(inner.real).astype(X)
    for _ in range(4):
        _, P, Q = _modes(p + 1, x)
        d = p * (x * P - Q) / (x * x - 1)
        x = x - d * (1 - x * x) / (2 * x * d - p * (p + 1) * P)
    return np.concatenate([[X(-1)], x, [X(1)]])


def _solve(A, B):
    """A^-1 B by Gauss-Jordan with row exchanges, in long double."""
    A, B = A.copy(), B.copy()
    for c in range(len(A)):
        r = c + int(np.argmax(np.abs(A[c:, c])))
        A[[c, r]], B[[c, r]] = A[[r, c]], B[[r, c]]
        B[c] /= A[c, c]
        A[c] /= A[c, c]
        for r in range(len(A)):
            if r != c:
                B[r] -= A[r, c] * B[c]
                A[r] -= A[r, c] * A[c]
    return B


def _rounded(got, want, left=0.0):
    unit = np.spacing(np.maximum(np.abs(want).astype(np.float64), 1e-3))
    assert (np.abs(got - want) <= X(0.51) * unit + left).all()


@pytest.mark.parametrize("p", range(1, 9))
def test_tables_of_a_degree(built_lib, p):
    E, O, K, s, q, _ = built_lib.modal_tables(p)
    n = p + 1
    W = _solve(_modes(n, _gll(p))[0], np.eye(n, dtype=X))
    _rounded(E, W[0::2, :E.shape[1]])
    _rounded(O, W[1::2, :O.shape[1]])
    k = np.arange(n)
    root = np.sqrt(X(2) * k + 1)
    lo = np.minimum.outer(k, k)
    _rounded(K, np.where((k[:, None] + k) % 2 == 0, 2 * np.outer(root, root) * lo * (lo + 1), X(0)))
    _rounded(s, root)
    _rounded(q, root * k * (k + 1))


@pytest.mark.parametrize("L", [0, 1, 2, 3, 8])
def test_restrictions(built_lib, L):
    x = _gll(8)
    fine = _modes(9, x)[0]
    for o in sorted({0, (1 << L) // 2, (1 << L) - 1}):
        R = built_lib.modal_tables(1, L, o)[5]
        coarse = _modes(9, (2 * o + 1 + x) / X(1 << L) - 1)[0]
        want = np.triu(_solve(fine, coarse))   # the rest is zero
        _rounded(R, want, 2e-17)
        assert (np.tril(R, -1) == 0).all()
