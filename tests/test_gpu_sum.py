"""The evaluation from the monomials' values (csrc/kernels_sum.cu): sizes at the
edges of its tiles (points), blocks (64 monomials) and lists, in the four
precisions, and the points it leaves to the general kernels.

Tolerances: the library's normwise ones (tests/_util.py).  They bound this
path: a value is a chain of at most 33 products here, each within 2^-112
(double-double; 2^-82 double, 2^-222 quad-double) of its modulus, and the sums
lose at most a unit of 2^-111 (2^-71, 2^-223) of the largest term.
"""
import numpy as np
import pytest

import synth
from oracle import exact as E

from _util import pe_precision, tol, widen

pytestmark = pytest.mark.gpu

PRECS = ["dd", "ddint", "f64", "qd"]


def system(seed, n, N, m, kmin, kmax, emax):
    rng = np.random.Generator(np.random.PCG64(seed))
    polys = []
    for _p in range(N):
        mons = []
        for _t in range(m):
            k = int(rng.integers(kmin, kmax + 1))
            pos = sorted(rng.choice(n, size=k, replace=False).tolist())
            mons.append((pos, rng.integers(1, emax + 1, size=k).tolist()))
        polys.append(mons)
    return synth.from_monomials(n, polys, synth.random_cdd(rng, N * m))


def inputs(s, pts, prec, seed):
    """(system, points) in the arrays of a precision, and for the oracle."""
    if prec == "qd":
        sq = s.to_qd(seed)
        pq = synth.widen_qd(np.random.Generator(np.random.PCG64(seed + 1)), pts)
        return sq, pq, sq, pq
    if prec == "f64":
        p = pts.copy()
        p[..., 1] = p[..., 3] = 0.0
        return s.as_fp64(), np.ascontiguousarray(pts[..., [0, 2]]), s.as_fp64(), p
    return s, pts, s, pts


def evaluate(s, pts, prec, general=False):
    import torch

    import paper_1201_0499_gb300 as pkg

    ev = pkg.PolyEval(s, pe_precision(prec), max_points=pts.shape[1])
    x = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
    f = torch.full((s.n_polys, pts.shape[1], pts.shape[2]), float("nan"), dtype=torch.float64, device="cuda")
    J = torch.full((s.n_polys, s.n_vars, pts.shape[1], pts.shape[2]), float("nan"), dtype=torch.float64, device="cuda")
    if general:  # the tuner times the general kernels and leaves their results
        ev.autotune(x, f, J)
    else:
        ev.eval(x, f, J)
    torch.cuda.synchronize()
    assert ev.status() == pkg.PE_OK
    ev.close()
    return f.cpu().numpy(), J.cpu().numpy()


def errors(s_ref, p_ref, f, J, prec, idx):
    if prec == "f64":
        f, J = widen(f), widen(J)
    return E.max_errors(s_ref, p_ref, f, J, idx)


SHAPES = [  # n, N, m, kmin, kmax, emax, P
    (1, 1, 1, 1, 1, 1, 1),
    (3, 2, 63, 0, 3, 2, 5),
    (5, 3, 64, 1, 5, 4, 4),
    (7, 2, 65, 1, 7, 9, 3),
    (40, 2, 130, 1, 3, 2, 9),   # variables that do not occur
    (6, 1, 257, 2, 6, 3, 2),
    (33, 1, 5, 33, 33, 1, 6),
    (70, 700, 6, 3, 6, 2, 7),   # many polynomials: runs that share a table
    (128, 2, 70, 20, 32, 4, 5),  # a large table: fewer points per tile
    (300, 1, 40, 2, 5, 12, 3),  # a table that outgrows shared memory in quad-double
]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("shape", SHAPES)
def test_edges(shape, prec):
    n, N, m, kmin, kmax, emax, P = shape
    s = system(900 + n, n, N, m, kmin, kmax, emax)
    pts = synth.points(901 + n, n, P, modulus_octaves=(-1, 0))
    s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 902)
    f, J = evaluate(s_in, p_in, prec)
    ef, ej = errors(s_ref, p_ref, f, J, prec, range(P) if N < 100 else [0, P - 1])
    assert ef <= tol(prec) and ej <= tol(prec), (ef, ej)


@pytest.mark.parametrize("prec", PRECS)
def test_points_left_to_the_general_kernels(prec):
    """Zero, real, imaginary, lopsided, tiny and non-finite coordinates among
    ordinary points: every finite point within the tolerance, non-finite
    results where the general kernels have them, and the ordinary points' bits
    independent of their neighbours."""
    n, P = 6, 23
    s = system(910, n, 4, 20, 0, 5, 4)
    plain = synth.points(911, n, P)
    pts = plain.copy()
    pts[2, 1] = 0.0                                    # x_2 = 0
    pts[:, 2] = 0.0                                    # the origin
    pts[:, 3, 2:] = 0.0                                # a real point
    pts[:, 6, :2] = 0.0                                # an imaginary point
    pts[1, 7] = [0.75, 0.0, np.ldexp(0.6, -70), 0.0]   # components far apart
    pts[4, 9] *= np.ldexp(1.0, -40)                    # a derivative far below the others' terms
    pts[0, 12] *= np.ldexp(1.0, 60)
    pts[3, 17, 0] = np.nan
    pts[5, 21, 2] = np.inf
    special = [1, 2, 3, 6, 7, 9, 12, 17, 21]
    finite = [q for q in range(P) if q not in (17, 21)]
    s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 912)
    if prec == "qd":  # the lower parts drawn for the plain points
        _, q_plain, _, _ = inputs(s, plain, prec, 912)
        p_in = q_plain.copy()
        p_in[..., [0, 1, 4, 5]] = pts
        for q in (1, 2, 3, 6, 7, 9, 12, 17, 21):
            p_in[:, q, [2, 3, 6, 7]] = 0.0
        p_ref = p_in
    else:
        q_plain = inputs(s, plain, prec, 912)[1]
    f, J = evaluate(s_in, p_in, prec)
    ef, ej = errors(s_ref, p_ref, f, J, prec, finite)
    assert ef <= tol(prec) and ej <= tol(prec), (ef, ej)
    fg, Jg = evaluate(s_in, p_in, prec, general=True)
    for q in (17, 21):
        assert np.array_equal(np.isfinite(f[:, q]), np.isfinite(fg[:, q]))
        assert np.array_equal(np.isfinite(J[:, :, q]), np.isfinite(Jg[:, :, q]))
    f0, J0 = evaluate(s_in, q_plain, prec)
    same = [q for q in range(P) if q not in special]
    assert np.array_equal(f[:, same], f0[:, same]) and np.array_equal(J[:, :, same], J0[:, :, same])


@pytest.mark.parametrize("prec", PRECS)
def test_batch_of_uneven_systems(prec):
    """Systems of one launch, some with points left to the general kernels and
    one without points."""
    import torch

    import paper_1201_0499_gb300 as pkg

    shapes = [(4, 3, 70, 0, 4, 3, 11), (9, 5, 12, 1, 6, 2, 5), (3, 2, 4, 1, 3, 5, 0), (12, 2, 129, 2, 9, 4, 21)]
    systems, points, refs = [], [], []
    for i, (n, N, m, kmin, kmax, emax, P) in enumerate(shapes):
        s = system(920 + i, n, N, m, kmin, kmax, emax)
        pts = synth.points(930 + i, n, P)
        if P > 2:
            pts[1, P - 2] = 0.0
        s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 940 + i)
        systems.append(s_in)
        points.append(p_in)
        refs.append((s_ref, p_ref))
    ev = pkg.PolyEvalMany(systems, [p.shape[1] for p in points], pe_precision(prec))
    fs, Js = ev.eval([torch.from_numpy(p).cuda() for p in points])
    torch.cuda.synchronize()
    for (s_ref, p_ref), f, J in zip(refs, fs, Js):
        if f.shape[1] == 0:
            continue
        ef, ej = errors(s_ref, p_ref, f.cpu().numpy(), J.cpu().numpy(), prec, range(f.shape[1]))
        assert ef <= tol(prec) and ej <= tol(prec), (ef, ej)
    ev.close()
