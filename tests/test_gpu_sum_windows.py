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
