"""The Newton step's elimination on the integer pipes (csrc/newton_int.cu): the
smallest and largest systems it takes, sizes at the steps of its block sizes,
points it leaves to the double-double code (non-finite or huge entries) and
singular points, against the exact residual.

Tolerance: the backward error bound of the double-double Newton tests, 1e-28
(an entry's products and differences err by 2^-115 of their operands; n = 77
elimination steps of unit growth stay below 1e-31)."""
from fractions import Fraction

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def linear_plus_square(seed, n):
    """f_i = sum_j a_ij x_j + x_0^2 + c_i: J is A plus 2 x_0 in column 0."""
    rng = np.random.Generator(np.random.PCG64(seed))
    polys = [[([j], [1]) for j in range(n)] + [([0], [2]), ([], [])] for _ in range(n)]
    return synth.from_monomials(n, polys, synth.random_cdd(rng, n * (n + 2)))


def newton(s, pts):
    import torch

    import paper_1201_0499_gb300 as pkg

    ev = pkg.PolyEval(s, pkg.PE_DD, max_points=pts.shape[1])
    x = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
    f, J = ev.eval(x)
    dx, lu, norms = ev.newton(x)
    torch.cuda.synchronize()
    assert ev.status() == pkg.PE_OK
    ev.close()
    return [t.cpu().numpy() for t in (f, J, dx, lu, norms, x)]


def fr(v):
    return Fraction(float(v[0])) + Fraction(float(v[1])), Fraction(float(v[2])) + Fraction(float(v[3]))


def backward_error(f, J, dx, q):
    """max_i |J dx + f|_i / (|J| |dx| + |f|), J, f, dx as returned, exactly summed."""
    n = f.shape[0]
    d = [fr(dx[i, q]) for i in range(n)]
    res = 0.0
    for i in range(n):
        re, im = fr(f[i, q])
        for j in range(n):
            a, b = fr(J[i, j, q])
            re += a * d[j][0] - b * d[j][1]
            im += a * d[j][1] + b * d[j][0]
        res = max(res, float(abs(re)) + float(abs(im)))
    mod = np.hypot(J[:, :, q, 0], J[:, :, q, 2]).sum(1).max()
    return res / (mod * np.hypot(dx[:, q, 0], dx[:, q, 2]).max() + np.hypot(f[:, q, 0], f[:, q, 2]).max())


@pytest.mark.parametrize("n", [11, 12, 16, 17, 40, 41, 77, 79])
def test_sizes(n):
    s = linear_plus_square(700 + n, n)
    pts = synth.points(701 + n, n, 3)
    f, J, dx, lu, norms, x1 = newton(s, pts)
    assert np.all(np.isfinite(lu))
    for q in range(3 if n < 50 else 1):
        assert backward_error(f, J, dx, q) <= 1e-28
        assert norms[q, 1] == pytest.approx(np.hypot(dx[:, q, 0], dx[:, q, 2]).max(), rel=1e-12)
    assert np.allclose(x1[..., 0], pts[..., 0] + dx[..., 0], rtol=1e-13)


def test_points_left_to_the_double_double_elimination():
    n, P = 13, 7
    s = linear_plus_square(720, n)
    pts = synth.points(721, n, P)
    pts[0, 2, :2] = [np.ldexp(1.0, 230), 0.0]  # column 0 of J beyond the integer elimination
    pts[3, 4, 0] = np.nan
    f, J, dx, lu, norms, x1 = newton(s, pts)
    for q in (0, 1, 2, 3, 5, 6):
        assert backward_error(f, J, dx, q) <= 1e-28, q
    assert np.isnan(norms[4, 0]) and (np.isnan(norms[4, 1]) or norms[4, 1] != norms[4, 1])
    others = [q for q in range(P) if q not in (2, 4)]
    g = synth.points(721, n, P)
    same = newton(s, g)
    for a, b in zip((dx, x1), (same[2], same[5])):
        assert np.array_equal(a[:, others], b[:, others])


def test_singular_points_step_nowhere():
    """A zero column at one point only: x_5 enters as x_5^2 alone."""
    n, P = 12, 3
    rng = np.random.Generator(np.random.PCG64(730))
    polys = [[([j], [2 if j == 5 else 1]) for j in range(n)] + [([], [])] for _ in range(n)]
    s = synth.from_monomials(n, polys, synth.random_cdd(rng, n * (n + 1)))
    pts = synth.points(731, n, P)
    pts[5, 1] = 0.0
    f, J, dx, lu, norms, x1 = newton(s, pts)
    assert np.all(dx[:, 1] == 0.0) and np.isnan(norms[1, 1]) and np.array_equal(x1[:, 1], pts[:, 1])
    for q in (0, 2):
        assert backward_error(f, J, dx, q) <= 1e-28


@pytest.mark.parametrize("n", [12, 17, 41])
def test_factors_stay_where_each_step_puts_them(n):
    """out_J entry by entry: an exchange at step k moves the columns from k on
    and leaves the multipliers of earlier steps.  Tolerance: elimination in
    complex double errs by n growth 2^-53 max|J| / |pivot| in a multiplier,
    below 41 x 10 x 1.1e-16 x 1e3 = 5e-11; taken as 1e-9 of max|J|."""
    s = linear_plus_square(740 + n, n)
    f, J, dx, lu, norms, x1 = newton(s, synth.points(741 + n, n, 2))
    for q in range(2):
        a = J[:, :, q, 0] + 1j * J[:, :, q, 2]
        scale = np.abs(a).max()
        for k in range(n):
            p = k + int(np.argmax(np.abs(a[k:, k])))
            a[[k, p], k:] = a[[p, k], k:]
            a[k + 1:, k] /= a[k, k]
            a[k + 1:, k + 1:] -= np.outer(a[k + 1:, k], a[k, k + 1:])
        assert np.abs(lu[:, :, q, 0] + 1j * lu[:, :, q, 2] - a).max() <= 1e-9 * scale
