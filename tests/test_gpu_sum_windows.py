"""Windows of the evaluation from the monomials' values (csrc/kernels_sum.cu)
where the magnitudes of a polynomial's monomials differ: sums that an earlier
chunk formed and a later one outgrows, and derivatives whose terms are small
beside the polynomial's largest monomial.

Every entry of J against the exact oracle, relative to its own terms."""
import numpy as np
import pytest

import synth
from oracle import exact as E

from test_gpu_sum import evaluate, errors, inputs
from _util import tol

pytestmark = pytest.mark.gpu

PRECS = ["dd", "ddint", "f64", "qd"]


def scaled(rng, bits):
    """Coefficients near the unit circle times 2^-bits (one entry per monomial)."""
    c = synth.random_cdd(rng, len(bits))
    return c * np.ldexp(1.0, -np.asarray(bits))[:, None]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("growth", [40, 80, 150, 300])
@pytest.mark.parametrize("small", ["first", "last"])
@pytest.mark.parametrize("P", [3, 160])
def test_sums_outgrown_by_a_later_chunk(prec, growth, small, P):
    """Monomials go by falling k: 600 of two variables x_0 .. x_9, then 100 of
    one variable x_10 .. x_19, one kind 2^-growth times the other.  At few
    points a chunk holds 512 monomials, at 160 points 128.  Tolerance: the
    library's (a term keeps at least 72, 112, 224 bits: 2e-22, 2e-34, 4e-68)."""
    n, N = 20, 4
    rng = np.random.Generator(np.random.PCG64(960 + growth))
    polys, bits = [], []
    for _p in range(N):
        pairs = [([i, j], [a, b]) for i in range(10) for j in range(i + 1, 10) for a in range(1, 5) for b in range(1, 5)]
        pairs = [pairs[t] for t in sorted(rng.choice(len(pairs), size=600, replace=False))]
        polys.append(pairs + [([i], [a]) for i in range(10, 20) for a in range(1, 11)])
        bits += [growth if small == "first" else 0] * 600 + [0 if small == "first" else growth] * 100
    s = synth.from_monomials(n, polys, scaled(rng, bits))
    pts = synth.points(961 + growth, n, P)
    s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 962)
    f, J = evaluate(s_in, p_in, prec)
    ef, ej = errors(s_ref, p_ref, f, J, prec, [0, P - 1])
    assert ef <= tol(prec) and ej <= tol(prec), (ef, ej)


# Relative to its terms a derivative may lose: 2^-111 double-double, 2^-71
# double, 2^-223 quad-double by the window; its products 2^-109, 2^-77, 2^-219
# (x^256: 255 units of 2^-117, 2^-85, 2^-227); its rounding 2^-106, 2^-53, 2^-211.
CLOSE = {"dd": 2.0**-104, "ddint": 2.0**-104, "f64": 2.0**-52, "qd": 2.0**-210}


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("below", [30, 50, 55, 58, 59, 60, 61, 62, 63, 64, 65, 66, 67, 70, 90])
@pytest.mark.parametrize("m", [100, 300, 2000])
def test_many_tiny_terms_beside_a_small_one(prec, below, m):
    """d f / d x_0 has one term 2^-below and m of 2^-130, which only the floors
    of the window show, 256 units each; x_1 alone is of size 1.  m = 100: one
    chunk; 300: one chunk but for a slack of 17 bits; 2000: several."""
    n, P = 2, 2
    rng = np.random.Generator(np.random.PCG64(970))
    polys = [[([1], [1]), ([0], [1])] + [([0], [256])] * m]
    s = synth.from_monomials(n, polys, scaled(rng, [0, below] + [130] * m))
    pts = synth.points(971, n, P)
    s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 972)
    f, J = evaluate(s_in, p_in, prec)
    ef, ej = errors(s_ref, p_ref, f, J, prec, range(P))
    assert ef <= CLOSE[prec] and ej <= CLOSE[prec], (ef, ej)
