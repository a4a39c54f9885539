"""Each component of f and J by itself, where its terms are far below the other
component's: a derivative that is one coefficient, points near the real axis.

Measure: |error of a component| over the sum of its terms' parts, (|re|, |im|)
pairs multiplied without cancellation ((a, b)(c, d) = (ac + bd, ad + bc)).
Bound: that of the general kernels, which compute components apart: a product
errs by 2^-102 (double-double) of its parts, a chain of 8 and a sum stay below
2^-98; in double 2^-52 each, 2^-48."""
import numpy as np
import pytest

import synth
from fractions import Fraction
from oracle import exact as E

from test_gpu_methods import evaluate
from test_gpu_sum import inputs, system

pytestmark = pytest.mark.gpu

BOUND = {"dd": 2.0**-98, "f64": 2.0**-48}


def pair(v):
    w = len(v) // 2
    return abs(sum(v[:w])), abs(sum(v[w:]))


def times(a, b):
    return a[0] * b[0] + a[1] * b[1], a[0] * b[1] + a[1] * b[0]


def part_scales(s, pts, q, p):
    """The measure's denominators: f [2], J [n, 2] of polynomial p at point q."""
    x = [pair(pts[v, q]) for v in range(s.n_vars)]
    f, J = np.zeros(2), np.zeros((s.n_vars, 2))
    for t in range(int(s.poly_ptr[p]), int(s.poly_ptr[p + 1])):
        vs = s.pos[s.mono_ptr[t]:s.mono_ptr[t + 1]]
        es = s.exp[s.mono_ptr[t]:s.mono_ptr[t + 1]]
        less, full = [], []
        for v, e in zip(vs, es):
            y = (1.0, 0.0)
            for _ in range(e - 1):
                y = times(y, x[v])
            less.append(y)
            full.append(times(y, x[v]))
        value = pair(s.coef[t])
        for y in full:
            value = times(value, y)
        f += value
        for j in range(len(vs)):
            d = pair(s.coef[t])
            for i in range(len(vs)):
                d = times(d, less[i] if i == j else full[i])
            J[vs[j]] += es[j] * np.array(d)
    return f, J


def component_error(got, exact, scale):
    w = len(got) // 2
    worst = 0.0
    for c in range(2):
        value = sum((Fraction(float(v)) for v in got[c * w:(c + 1) * w]), Fraction(0))
        d = float(abs(value - Fraction(exact[c]) * Fraction(2) ** exact[2]))
        worst = max(worst, d / scale[c] if scale[c] else (0.0 if d == 0.0 else np.inf))
    return worst


def worst_components(s, pts, f, J, points, polys):
    worst = 0.0
    for q in points:
        fx, Jx = E.evaluate_point(s, pts, q, polys)
        for p in polys:
            sf, sJ = part_scales(s, pts, q, p)
            worst = max(worst, component_error(f[p, q], fx[p], sf))
            for i, v in Jx[p].items():
                worst = max(worst, component_error(J[p, i, q], v, sJ[i]))
    return worst


@pytest.mark.parametrize("prec,apart", [("dd", 12), ("dd", 22), ("dd", 34), ("ddint", 12), ("ddint", 34), ("f64", 12)])
def test_derivatives_that_are_one_coefficient(prec, apart):
    """x_6 .. x_9 occur once per polynomial, as c x with components 2^-apart of
    each other: their derivatives are c, bit for bit, at any point."""
    import paper_1201_0499_gb300 as pkg

    n, N, P = 10, 3, 9
    base = system(1200, 6, N, 70, 2, 5, 3)
    rng = np.random.Generator(np.random.PCG64(1201))
    polys, coef, m = [], [], 0
    for p in range(N):
        mons = []
        for t in range(int(base.poly_ptr[p]), int(base.poly_ptr[p + 1])):
            mons.append((base.pos[base.mono_ptr[t]:base.mono_ptr[t + 1]].tolist(),
                         base.exp[base.mono_ptr[t]:base.mono_ptr[t + 1]].tolist()))
        coef += [c for c in base.coef[int(base.poly_ptr[p]):int(base.poly_ptr[p + 1])]]
        own = synth.random_cdd(rng, 4)
        own[:2, 2:] = np.ldexp(own[:2, 2:], -apart)
        own[2:, :2] = np.ldexp(own[2:, :2], -apart)
        polys.append(mons + [([6 + i], [1]) for i in range(4)])
        coef += [c for c in own]
    s = synth.from_monomials(n, polys, np.array(coef))
    pts = synth.points(1202, n, P)
    s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 1203)
    f, J = evaluate(s_in, p_in, prec, pkg.PE_FROM_VALUES)
    for p in range(N):
        for i in range(4):
            c = s_ref.coef[int(s.poly_ptr[p + 1]) - 4 + i]
            assert np.all(J[p, 6 + i] == (c[[0, 2]] if prec == "f64" else c)), (p, i)


@pytest.mark.parametrize("prec", ["dd", "f64"])
def test_constant_derivatives_have_no_negative_zeros(prec):
    """A sum that starts from 0: the zero parts of a coefficient come out as +0."""
    import paper_1201_0499_gb300 as pkg

    s = synth.from_monomials(2, [[([0], [1]), ([1], [2])]], np.array([[-0.0, -0.0, 2.0, -0.0], [1.0, 0.0, 1.0, 0.0]]))
    pts = synth.points(1260, 2, 5)
    s_in, p_in, _, _ = inputs(s, pts, prec, 1261)
    for flags in (pkg.PE_FROM_VALUES, pkg.PE_GENERAL_KERNELS):
        J = evaluate(s_in, p_in, prec, flags)[1]
        assert np.all(J[0, 0, :, J.shape[-1] // 2] == 2.0) and not np.any(np.signbit(J[0, 0]))


def run(s, pts, prec, flags):
    import torch

    import paper_1201_0499_gb300 as pkg
    from _util import pe_precision

    ev = pkg.PolyEval(s, pe_precision(prec), max_points=pts.shape[1], flags=flags)
    f, J = ev.eval(torch.from_numpy(np.ascontiguousarray(pts)).cuda())
    torch.cuda.synchronize()
    assert ev.status() == pkg.PE_OK
    ev.close()
    return f.cpu().numpy(), J.cpu().numpy()


def near_axis_case(kind, apart, seed, n=7, N=4, m=60, P=11):
    """A system and points with imaginary parts 2^-apart of the real ones, in
    the coefficients, the points, or both; points 4 and 9 on the unit circle."""
    s = system(seed, n, N, m, 0, 5, 3)
    pts = synth.points(seed + 1, n, P)
    circle = pts.copy()
    if "near" in kind[0]:
        s.coef[:, 2:] = np.ldexp(s.coef[:, 2:], -apart)
    elif kind[0] == "real":
        s.coef[:, 2:] = 0.0
    elif kind[0] == "imaginary":
        s.coef[:, :2] = 0.0
    if kind[1] == "near":
        pts[..., 2:] = np.ldexp(pts[..., 2:], -apart)
    else:
        pts[..., 2:] = 0.0
    pts[:, [4, 9]] = circle[:, [4, 9]]
    return s, pts


@pytest.mark.parametrize("prec", ["dd", "f64"])
@pytest.mark.parametrize("apart", [8, 16, 22])
@pytest.mark.parametrize("wanted", ["values", "own"])  # own: the library's choice
@pytest.mark.parametrize("kind", [("real", "near"), ("near", "near"), ("near", "real"), ("imaginary", "near"), ("any", "near")])
def test_near_the_axes(prec, apart, kind, wanted):
    import paper_1201_0499_gb300 as pkg

    s, pts = near_axis_case(kind, apart, 1210 + apart)
    s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 1211)
    f, J = run(s_in, p_in, prec, pkg.PE_FROM_VALUES if wanted == "values" else 0)
    assert worst_components(s_ref, p_ref, f, J, range(pts.shape[1]), [0, 3]) <= BOUND[prec]


@pytest.mark.parametrize("apart", [24, 31, 38])
def test_coefficients_far_apart_in_double(apart):
    """At real points and on the unit circle."""
    import paper_1201_0499_gb300 as pkg

    s, pts = near_axis_case(("real", "real"), 0, 1250)
    rng = np.random.Generator(np.random.PCG64(1252))
    s.coef[:, 0] = rng.uniform(0.5, 1.0, len(s.coef))
    s.coef[:, 2] = np.ldexp(rng.uniform(0.5, 1.0, len(s.coef)), -apart)
    s_in, p_in, s_ref, p_ref = inputs(s, pts, "f64", 1251)
    f, J = run(s_in, p_in, "f64", pkg.PE_FROM_VALUES)
    assert worst_components(s_ref, p_ref, f, J, range(pts.shape[1]), [0, 3]) <= BOUND["f64"]


def test_near_the_axes_in_a_batch():
    """One system of real coefficients among others; its near-real points."""
    import torch

    import paper_1201_0499_gb300 as pkg

    cases = [near_axis_case(k, 16, 1230 + i, n=5 + i, P=10 + i) for i, k in
             enumerate([("any", "near"), ("real", "near"), ("near", "real")])]
    ev = pkg.PolyEvalMany([s for s, _ in cases], [p.shape[1] for _, p in cases], pkg.PE_DD, pkg.PE_FROM_VALUES)
    fs, Js = ev.eval([torch.from_numpy(p).cuda() for _, p in cases])
    torch.cuda.synchronize()
    for (s, p), f, J in zip(cases, fs, Js):
        assert worst_components(s, p, f.cpu().numpy(), J.cpu().numpy(), range(p.shape[1]), [1]) <= BOUND["dd"]
    ev.close()


@pytest.mark.parametrize("prec", ["dd", "ddint", "f64", "qd"])
def test_real_points_of_real_systems(prec):
    """Imaginary parts are exact zeros, the real parts as accurate as ever."""
    import paper_1201_0499_gb300 as pkg

    s, pts = near_axis_case(("real", "real"), 0, 1240)
    pts[..., 2:] = 0.0
    s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 1241)
    if prec == "qd":  # no lower parts to the zeros
        s_in.coef[:, 4:] = 0.0
        p_in[..., 4:] = 0.0
    f, J = evaluate(s_in, p_in, prec, pkg.PE_FROM_VALUES)
    w = f.shape[-1] // 2
    assert np.all(f[..., w:] == 0.0) and np.all(J[..., w:] == 0.0)
    assert worst_components(s_ref, p_ref, f, J, [0, 10], [0]) <= (2.0**-195 if prec == "qd" else BOUND.get(prec, 2.0**-90))
