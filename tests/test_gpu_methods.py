"""Which kernels a handle evaluates with (the create flags PE_GENERAL_KERNELS and
PE_FROM_VALUES), and each of the two on the cases that the library's own choice
gives to the other.

Evaluation from values: every edge shape and the left-over points in every
precision.  General kernels: the launch, chunk, group, graph and agreement
tests that were written for them, and the n = 64 and n = 128 workloads."""
import numpy as np
import pytest

import synth
from oracle import exact as E

import test_gpu_batch as batch
import test_gpu_parity as parity
from test_gpu_sum import PRECS, SHAPES, errors, inputs, system
from _util import fp64_inputs, normwise_vs, pe_precision, scales, tol, widen

pytestmark = pytest.mark.gpu


def from_values(handle, prec, one_eval):
    """Whether an evaluation, of one monomial chunk, goes by the monomials'
    values, from the kernels it queues: the table and the sums, then the
    general kernels over the points left to them (their table, if exponents
    need one, and the sums; quad-double has no rounding pass there).  The
    general kernels alone are at most two (three in quad-double)."""
    import paper_1201_0499_gb300 as pkg

    pkg.polyeval_timing(handle, True)
    one_eval()
    kernels = pkg.polyeval_timing_read(handle)[2]
    pkg.polyeval_timing(handle, False)
    return kernels > (3 if prec == "qd" else 2)


def evaluate(s, pts, prec, flags, chunks=1):
    import torch

    import paper_1201_0499_gb300 as pkg

    P = pts.shape[1]
    ev = pkg.PolyEval(s, pe_precision(prec), max_points=P, flags=flags)
    pkg.polyeval_set_launch(ev.handle, P, chunks)
    f = torch.full((s.n_polys, P, pts.shape[2]), float("nan"), dtype=torch.float64, device="cuda")
    J = torch.full((s.n_polys, s.n_vars, P, pts.shape[2]), float("nan"), dtype=torch.float64, device="cuda")
    x = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
    by_values = from_values(ev.handle, prec, lambda: ev.eval(x, f, J))
    assert chunks > 1 or by_values == (flags == pkg.PE_FROM_VALUES)
    torch.cuda.synchronize()
    assert ev.status() == pkg.PE_OK
    ev.close()
    return f.cpu().numpy(), J.cpu().numpy()


def test_the_choice_and_its_flags():
    import torch

    import paper_1201_0499_gb300 as pkg

    def method(s, prec, flags):
        ev = pkg.PolyEval(s, pe_precision(prec), max_points=4, flags=flags)
        pkg.polyeval_set_launch(ev.handle, 4, 1)
        x = torch.ones((s.n_vars, 4, 2 if prec == "f64" else 8 if prec == "qd" else 4), dtype=torch.float64, device="cuda")
        m = from_values(ev.handle, prec, lambda: ev.eval(x))
        ev.close()
        return m

    dense = synth.config(2, n_points=1)[0]       # 64 monomials of 9 variables
    few = system(980, 50, 50, 8, 2, 2, 2)        # 8 monomials of 2
    both = pkg.PE_FROM_VALUES | pkg.PE_GENERAL_KERNELS
    for prec in PRECS:
        s = dense.as_fp64() if prec == "f64" else dense
        assert [method(s, prec, x) for x in (0, pkg.PE_FROM_VALUES, pkg.PE_GENERAL_KERNELS, both)] == [True, True, False, False]
    assert [method(few.as_fp64(), "f64", x) for x in (0, pkg.PE_FROM_VALUES, pkg.PE_GENERAL_KERNELS)] == [False, True, False]
    for flags, m in ((0, True), (pkg.PE_GENERAL_KERNELS, False)):
        many = pkg.PolyEvalMany([dense, dense], [5, 9], pkg.PE_DD, flags)
        x = [torch.ones((32, P, 4), dtype=torch.float64, device="cuda") for P in (5, 9)]
        assert from_values(many.handle, "dd", lambda: many.eval(x)) == m
        many.close()


# --------------------------------------------------------------------------
# evaluation from values
# --------------------------------------------------------------------------

@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("shape", SHAPES + [(70, 700, 6, 3, 6, 2, 50)])  # last: runs of two polynomials
def test_edges_from_values(shape, prec):
    import paper_1201_0499_gb300 as pkg

    n, N, m, kmin, kmax, emax, P = shape
    s = system(900 + n, n, N, m, kmin, kmax, emax)
    pts = synth.points(901 + n, n, P, modulus_octaves=(-1, 0))
    s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 902)
    f, J = evaluate(s_in, p_in, prec, pkg.PE_FROM_VALUES)
    assert np.all(np.isfinite(f)) and np.all(np.isfinite(J))
    ef, ej = errors(s_ref, p_ref, f, J, prec, range(P) if N < 100 else [0, P - 1])
    assert ef <= tol(prec) and ej <= tol(prec), (ef, ej)


def lopsided_points(pts):
    """Points left to the general kernels among ordinary ones (in place)."""
    pts[2, 1] = 0.0                                    # x_2 = 0
    pts[:, 2] = 0.0                                    # the origin
    pts[1, 7] = [0.75, 0.0, np.ldexp(0.6, -70), 0.0]   # components far apart
    pts[0, 12] *= np.ldexp(1.0, 60)
    pts[3, 17, 0] = np.nan
    pts[5, 21, 2] = np.inf
    return [1, 2, 7, 12, 17, 21]


def quad(pts, plain, special, seed):
    """The lower parts drawn for the plain points, none where pts differ."""
    out = synth.widen_qd(np.random.Generator(np.random.PCG64(seed)), plain)
    out[..., [0, 1, 4, 5]] = pts
    out[:, special] = 0.0
    out[:, special, :] = np.stack([pts[:, special, 0], pts[:, special, 1], 0 * pts[:, special, 0], 0 * pts[:, special, 0],
                                   pts[:, special, 2], pts[:, special, 3], 0 * pts[:, special, 0], 0 * pts[:, special, 0]], -1)
    return out


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("m,chunks", [(20, 1), (20, 3), (300, 1), (300, 3)])
def test_left_over_points_from_values(prec, m, chunks):
    """Ordinary points: the bits they have without the others.  The points left
    over: within the tolerance, and finite where the general kernels are; their
    sums in one part or added up from three."""
    import paper_1201_0499_gb300 as pkg

    n, P = 6, 23
    s = system(981, n, 4, m, 0, 5, 4)
    plain = synth.points(982, n, P)
    pts = plain.copy()
    special = lopsided_points(pts)
    s_in, p_plain, s_ref, _ = inputs(s, plain, prec, 983)
    if prec == "qd":
        p_in = p_ref = quad(pts, plain, special, 985)
        p_plain = quad(plain, plain, [], 985)
    else:
        _, p_in, _, p_ref = inputs(s, pts, prec, 983)
    f, J = evaluate(s_in, p_in, prec, pkg.PE_FROM_VALUES, chunks)
    f0, J0 = evaluate(s_in, p_plain, prec, pkg.PE_FROM_VALUES, chunks)
    fg, Jg = evaluate(s_in, p_in, prec, pkg.PE_GENERAL_KERNELS, chunks)
    same = [q for q in range(P) if q not in special]
    assert np.array_equal(f[:, same], f0[:, same]) and np.array_equal(J[:, :, same], J0[:, :, same])
    finite = [q for q in range(P) if q not in (17, 21)]
    for a, b in ((f, J), (fg, Jg)):
        ef, ej = errors(s_ref, p_ref, a, b, prec, finite)
        assert ef <= tol(prec) and ej <= tol(prec), (ef, ej)
    for q in (17, 21):
        assert np.array_equal(np.isfinite(f[:, q]), np.isfinite(fg[:, q]))
        assert np.array_equal(np.isfinite(J[:, :, q]), np.isfinite(Jg[:, :, q]))


@pytest.mark.parametrize("prec", PRECS)
def test_batch_with_left_over_points_from_values(prec):
    import torch

    import paper_1201_0499_gb300 as pkg

    shapes = [(6, 3, 70, 0, 4, 3, 23), (9, 5, 12, 1, 6, 2, 25), (12, 2, 129, 2, 9, 4, 22)]
    systems, points, refs = [], [], []
    for i, (n, N, m, kmin, kmax, emax, P) in enumerate(shapes):
        s = system(990 + i, n, N, m, kmin, kmax, emax)
        pts = synth.points(995 + i, n, P)
        pts[1, P - 2] = 0.0
        pts[0, 3] *= np.ldexp(1.0, 60)
        s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 999 + i)
        systems.append(s_in)
        points.append(p_in)
        refs.append((s_ref, p_ref))
    ev = pkg.PolyEvalMany(systems, [p.shape[1] for p in points], pe_precision(prec), pkg.PE_FROM_VALUES)
    x = [torch.from_numpy(p).cuda() for p in points]
    assert from_values(ev.handle, prec, lambda: ev.eval(x))
    fs, Js = ev.eval(x)
    torch.cuda.synchronize()
    for (s_ref, p_ref), f, J in zip(refs, fs, Js):
        ef, ej = errors(s_ref, p_ref, f.cpu().numpy(), J.cpu().numpy(), prec, range(f.shape[1]))
        assert ef <= tol(prec) and ej <= tol(prec), (ef, ej)
    ev.close()


# --------------------------------------------------------------------------
# general kernels
# --------------------------------------------------------------------------

@pytest.fixture
def general(monkeypatch):
    """Every handle that a test makes evaluates with the general kernels."""
    import paper_1201_0499_gb300 as pkg

    class One(pkg.PolyEval):
        def __init__(self, system, precision=pkg.PE_DD, max_points=1, flags=0):
            super().__init__(system, precision, max_points, flags | pkg.PE_GENERAL_KERNELS)

    class Many(pkg.PolyEvalMany):
        def __init__(self, systems, points_per_system, precision=pkg.PE_DD, flags=0):
            super().__init__(systems, points_per_system, precision, flags | pkg.PE_GENERAL_KERNELS)

    monkeypatch.setattr(pkg, "PolyEval", One)
    monkeypatch.setattr(pkg, "PolyEvalMany", Many)


@pytest.mark.parametrize("prec", ["dd", "qd"])
def test_general_every_launch(general, prec):
    parity.test_set_launch_every_choice(prec)


@pytest.mark.parametrize("prec", ["dd", "f64"])
@pytest.mark.parametrize("P", [1, 3, 5, 15])
def test_general_monomial_groups(general, prec, P):
    parity.test_monomial_groups_few_points(prec, P)


@pytest.mark.parametrize("prec", ["dd", "ddint"])
def test_general_autotune_then_eval(general, prec):
    parity.test_autotune_then_eval(prec)


def test_general_integer_products_agree_with_fp64(general):
    parity.test_integer_path_deterministic_and_close_to_fp64_dd()


def test_general_graph_replay(general):
    parity.test_cuda_graph_replay_matches_eager()


@pytest.mark.parametrize("prec", ["dd", "f64", "ddint", "qd"])
def test_general_batch_every_launch(general, prec):
    batch.test_batch_every_launch_choice(prec)


@pytest.mark.parametrize("prec", ["dd", "qd"])
def test_general_batch_graph_replay(general, prec):
    batch.test_batch_cuda_graph_replay_matches_eager(prec)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("cfg", [3, 5])
def test_general_at_the_large_shapes(general, prec, cfg):
    """The n = 64 and n = 128 workloads at 33 points: every output of the first,
    a middle and the last point against the C double-double oracle (itself
    within 1e-30), one row of each against the exact one; quad-double: the
    exact rows."""
    import torch

    import oracle
    import paper_1201_0499_gb300 as pkg

    s, pts = synth.config(cfg, n_points=33)
    idx = [0, 15, 32]
    s_in, p_in, s_ref, p_ref = inputs(s, pts, prec, 986)
    ev = pkg.PolyEval(s_in, pe_precision(prec), max_points=33)
    f, J = ev.eval(torch.from_numpy(np.ascontiguousarray(p_in)).cuda())
    torch.cuda.synchronize()
    assert ev.status() == pkg.PE_OK
    f, J = f.cpu().numpy(), J.cpu().numpy()
    if prec == "f64":
        f, J = widen(f), widen(J)
    if prec != "qd":
        sub = np.ascontiguousarray(pts[:, idx])
        so, po = fp64_inputs(s, sub) if prec == "f64" else (s, sub)
        Fo, Jo = oracle.dd_eval(so, po, threads=0)
        Sf, SJ = scales(s, sub)
        assert normwise_vs(f[:, idx], Fo, Sf) <= tol(prec)
        assert normwise_vs(J[:, :, idx], Jo, SJ) <= tol(prec)
    ef, ej = E.max_errors(s_ref, p_ref, f, J, idx[:1], polys=[s.n_polys - 1])
    assert ef <= tol(prec) and ej <= tol(prec), (ef, ej)
    ev.close()
