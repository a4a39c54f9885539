"""Newton steps of nearly real systems: both components of dx as accurate as the
double-double elimination makes them.

f_i = sum_j a_ij x_j + c_i with real a, c at points 2^-apart off the real axis:
J = A, and the exact step is A dx = -f in the real and in the imaginary parts
by themselves.  Bound per component of a part: elimination in double-double
errs by 2^-102 of |A^-1| |A| |dx|, times n steps and a growth of 8."""
from fractions import Fraction

import numpy as np
import pytest

import synth

from test_newton_int import newton

pytestmark = pytest.mark.gpu


def solve(A, b):
    """A x = b in rationals, one right-hand side per column."""
    n = len(A)
    M = [list(A[i]) + list(b[i]) for i in range(n)]
    for k in range(n):
        p = max(range(k, n), key=lambda i: abs(M[i][k]))
        M[k], M[p] = M[p], M[k]
        for i in range(k + 1, n):
            w = M[i][k] / M[k][k]
            if w:
                M[i] = M[i][:k] + [x - w * y for x, y in zip(M[i][k:], M[k][k:])]
    x = [None] * n
    for i in range(n - 1, -1, -1):
        x[i] = [(M[i][n + c] - sum((M[i][j] * x[j][c] for j in range(i + 1, n)), Fraction(0))) / M[i][i] for c in range(len(b[0]))]
    return x


@pytest.mark.parametrize("n", [11, 12, 20])
@pytest.mark.parametrize("apart", [14, 30, 60])
def test_both_components(n, apart):
    rng = np.random.Generator(np.random.PCG64(760 + n))
    polys = [[([j], [1]) for j in range(n)] + [([], [])] for _ in range(n)]
    coef = np.zeros((n * (n + 1), 4))
    coef[:, 0] = rng.uniform(-1.0, 1.0, len(coef))
    s = synth.from_monomials(n, polys, coef)
    pts = np.zeros((n, 2, 4))
    pts[..., 0] = rng.uniform(0.5, 1.0, (n, 2)) * rng.choice([-1.0, 1.0], (n, 2))
    pts[..., 2] = np.ldexp(rng.uniform(0.5, 1.0, (n, 2)), -apart)
    f, J, dx, lu, norms, x1 = newton(s, pts)
    A = coef.reshape(n, n + 1, 4)[:, :n, 0]
    assert np.array_equal(J[:, :, 0, 0], A) and np.all(J[:, :, 0, 1:] == 0.0)
    cond = np.abs(np.linalg.inv(A)) @ np.abs(A)
    for q in range(2):
        rhs = [[-(Fraction(float(f[i, q, 2 * c])) + Fraction(float(f[i, q, 2 * c + 1]))) for c in range(2)] for i in range(n)]
        exact = solve([[Fraction(float(a)) for a in row] for row in A], rhs)
        for c in range(2):
            bound = 8.0 * n * 2.0**-102 * (cond @ np.abs(dx[:, q, 2 * c]))
            for i in range(n):
                got = Fraction(float(dx[i, q, 2 * c])) + Fraction(float(dx[i, q, 2 * c + 1]))
                assert abs(float(got - exact[i][c])) <= bound[i], (q, c, i)


def test_real_systems_stay_real():
    n = 14
    rng = np.random.Generator(np.random.PCG64(770))
    polys = [[([j], [1]) for j in range(n)] + [([0, 1], [2, 1]), ([], [])] for _ in range(n)]
    coef = np.zeros((n * (n + 2), 4))
    coef[:, 0] = rng.uniform(-1.0, 1.0, len(coef))
    pts = np.zeros((n, 3, 4))
    pts[..., 0] = rng.uniform(0.5, 1.0, (n, 3))
    f, J, dx, lu, norms, x1 = newton(synth.from_monomials(n, polys, coef), pts)
    assert np.all(dx[..., 2:] == 0.0) and np.all(lu[..., 2:] == 0.0) and np.all(np.isfinite(dx))
