"""Workloads of the polynomial evaluator, each through the entry point a user's
program calls.

A case is one system shape (n variables, N = n polynomials of m monomials, k
variables per monomial, exponents 1..e), one precision and one number of
points.  `op` says which call:

  eval    f and the Jacobian at a batch of points, device in and out
  host    the same with host buffers (copies included)
  newton  one Newton step (evaluation and linear solve) per point
  many    a batch of systems of uneven shape in one call
  track   a square dense system solved by following all its paths

Points and coefficients lie on the unit circle (`spread` 0), or have moduli
log-uniform in 2^-s .. 2^s (points: within [0.5, 2)).
"""
import math

import numpy as np
import torch

import paper_1201_0499_gb300 as pkg

PRECISION = {"dd": pkg.PE_DD, "f64": pkg.PE_F64, "ddint": pkg.PE_DD_INT, "qd": pkg.PE_QD_INT}
WORDS = {"dd": 4, "f64": 2, "ddint": 4, "qd": 8}  # doubles per complex number


def listed():
    return [
        # One point of a tiny system: a single corrector evaluation inside a
        # user's own solver loop; launches and latency are all there is.
        dict(name="one_point_n16", op="eval", prec="dd", n=16, m=8, k=4, e=3, P=1, spread=0),
        # A handful of points of a middle-sized system (odd sizes): a tracker
        # following a few paths.
        dict(name="few_points_n33", op="eval", prec="dd", n=33, m=47, k=7, e=4, P=21, spread=0),
        # The n = 32 workload of the benchmark: the usual batch of points.
        dict(name="dd_n32", op="eval", prec="dd", n=32, m=64, k=9, e=5, P=1024, spread=0),
        # The same in quad-double, at a ragged number of points.
        dict(name="qd_n32", op="eval", prec="qd", n=32, m=64, k=9, e=5, P=777, spread=0),
        # The n = 64 workload with spread moduli, in plain complex double ...
        dict(name="f64_n64", op="eval", prec="f64", n=64, m=256, k=16, e=8, P=4096, spread=10),
        # ... and in double-double with products on the integer pipes.
        dict(name="ddint_n64", op="eval", prec="ddint", n=64, m=256, k=16, e=8, P=1500, spread=10),
        # Many variables, few of them in a monomial: sparse systems from
        # applications (each monomial touches k of n variables).
        dict(name="dd_sparse_n200", op="eval", prec="dd", n=200, m=24, k=3, e=2, P=500, spread=0),
        # The n = 128 workload of the benchmark, the largest, with as many
        # points as one pass of about a second takes.
        dict(name="dd_n128", op="eval", prec="dd", n=128, m=1024, k=32, e=4, P=1024, spread=0),
        # One Newton step at every point of the n = 32 workload.
        dict(name="newton_dd_n32", op="newton", prec="dd", n=32, m=64, k=9, e=5, P=1024, spread=0),
        # Host buffers in and out: a program that keeps its points on the host.
        dict(name="host_dd_n32", op="host", prec="dd", n=32, m=64, k=9, e=5, P=600, spread=0),
        # Systems of uneven shape, each at its own points, in one call.
        dict(name="many_dd", op="many", prec="dd", systems=24, n=96, m=256, k=20, e=6, P=160, spread=0),
        # Ten dense quadrics, all 1024 paths, in double-double.
        dict(name="track_dd_quadrics10", op="track", prec="dd", n=10, degree=2, spread=0),
    ]


def _products(c):
    """A measure of a case's work: complex products of the textbook method,
    scaled by what a precision costs."""
    w = {"dd": 1.0, "ddint": 0.3, "qd": 0.7, "f64": 0.2}[c["prec"]]
    if c["op"] == "track":
        return 0.0
    count = c["systems"] / 6.0 if c["op"] == "many" else 1.0
    return w * count * c["n"] * c["m"] * c["P"] * (6.0 * c["k"] + 10.0)


def draw(rng):
    """One more case: every call and precision, sizes over the listed ranges."""
    most = max(_products(c) for c in listed())

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["eval", "eval", "eval", "eval", "eval", "eval", "newton", "host", "many", "track"])
    if op == "track":
        return dict(op="track", prec=rng.choice(["dd", "f64", "ddint"]), n=rng.randint(6, 9), degree=2, spread=0)
    while True:
        n = log(10, 200)
        c = dict(op=op, prec=rng.choice(["dd", "f64", "ddint", "qd"]), n=n, m=log(8, 1024), k=min(log(2, 32), n),
                 e=rng.randint(1, 8), P=log(1, 4096), spread=rng.choice([0, 0, 10]))
        if op == "newton":
            c.update(n=min(n, 64), k=min(c["k"], min(n, 64)), prec=rng.choice(["dd", "f64", "ddint"]))
        if op == "many":
            c.update(systems=rng.randint(4, 32), n=log(12, 96), m=log(16, 256), P=log(8, 200))
            c["k"] = min(log(3, 20), c["n"])
        # outputs of at most 1.5 GB, Newton solves of at most a fraction of a second
        out = c["n"] * c["n"] * c["P"] * WORDS[c["prec"]] * 8 * c.get("systems", 1)
        solve = c["n"] ** 3 * c["P"] if op == "newton" else 0
        if _products(c) <= 0.5 * most and out <= 1.5e9 and solve <= 2.5e8:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class System:
    """The plain arrays the package compiles: monomials in compressed rows."""

    def __init__(self, n, poly_ptr, mono_ptr, pos, exp, coef):
        self.n_vars, self.n_polys = n, len(poly_ptr) - 1
        self.poly_ptr, self.mono_ptr, self.pos, self.exp, self.coef = poly_ptr, mono_ptr, pos, exp, coef


def _numbers(rng, size, words, moduli=None):
    """Complex numbers near the unit circle (or of the given moduli) as
    unevaluated sums of words/2 doubles per component, all parts in use."""
    angle = rng.random(size) * (2.0 * np.pi)
    out = np.zeros((size, words))
    for c, part in enumerate((np.cos(angle), np.sin(angle))):
        x = part if moduli is None else part * moduli
        for w in range(words // 2):
            out[:, c * (words // 2) + w] = x
            x = np.spacing(np.abs(x)) * (rng.random(size) - 0.5) * 0.5
    return out


def _moduli(rng, size, spread):
    return np.exp2(rng.uniform(-spread, spread, size)) if spread else None


def _system(rng, n, m, k, e, words, spread, k_of=None, m_of=None):
    """N = n polynomials.  k_of, m_of: sizes drawn per monomial, per polynomial."""
    ms = np.full(n, m) if m_of is None else m_of(n)
    M = int(ms.sum())
    ks = np.full(M, k) if k_of is None else k_of(M)
    kmax = int(ks.max())
    rank = np.argpartition(rng.random((M, n), dtype=np.float32), kmax - 1, axis=1)[:, :kmax]
    taken = np.arange(kmax)[None, :] < ks[:, None]
    rank = np.sort(np.where(taken, rank, n), axis=1)
    pos = rank[rank < n].astype(np.int32)
    exp = rng.integers(1, e + 1, pos.size).astype(np.int32)
    poly_ptr = np.concatenate([[0], np.cumsum(ms)]).astype(np.int64)
    mono_ptr = np.concatenate([[0], np.cumsum(ks)]).astype(np.int64)
    return System(n, poly_ptr, mono_ptr, pos, exp, _numbers(rng, M, words, _moduli(rng, M, spread)))


def _dense(rng, n, degree, words):
    """n polynomials with every monomial of total degree <= 2."""
    mons = [[]] + [[(i, 1)] for i in range(n)] + [[(i, 2)] for i in range(n)]
    mons += [[(i, 1), (j, 1)] for i in range(n) for j in range(i + 1, n)]
    assert degree == 2
    M = n * len(mons)
    ks = [len(t) for t in mons] * n
    return System(n, np.arange(n + 1, dtype=np.int64) * len(mons), np.concatenate([[0], np.cumsum(ks)]).astype(np.int64),
                  np.array([v for t in mons for v, _ in t] * n, dtype=np.int32),
                  np.array([a for t in mons for _, a in t] * n, dtype=np.int32), _numbers(rng, M, words))


def _points(rng, n, P, words, spread):
    moduli = np.exp2(rng.uniform(-1.0, 1.0, n * P)) if spread else None
    return _numbers(rng, n * P, words, moduli).reshape(n, P, words)


def _draw_inputs(case, seed):
    """(systems, points) on the host, from the seed alone."""
    rng = np.random.default_rng([seed, 1201])
    w = WORDS[case["prec"]]
    cw = max(w, 4)  # coefficients of plain double systems are given as double-doubles with zero low parts
    if case["op"] == "track":
        s = _dense(rng, case["n"], case["degree"], cw)
        if w == 2:
            s.coef[:, [1, 3]] = 0.0
        return [s], None
    if case["op"] == "many":
        # the sizes belong to the case; monomials, coefficients and points to the seed
        sizes = np.random.default_rng([case[v] for v in ("systems", "n", "m", "k", "e", "P")])
        systems, points = [], []
        for _ in range(case["systems"]):
            n = int(sizes.integers(8, case["n"] + 1))
            ms = sizes.integers(8, max(9, case["m"] + 1), n)
            top = min(n, case["k"])
            systems.append(_system(rng, n, 0, 0, case["e"], cw, case["spread"],
                                   k_of=lambda c: rng.integers(min(2, top), top + 1, c), m_of=lambda c: ms))
            points.append(_points(rng, n, int(sizes.integers(1, case["P"] + 1)), w, case["spread"]))
    else:
        systems = [_system(rng, case["n"], case["m"], case["k"], case["e"], cw, case["spread"])]
        points = [_points(rng, case["n"], case["P"], w, case["spread"])]
    if w == 2:
        for s in systems:
            s.coef[:, [1, 3]] = 0.0
    return systems, points


def prepare(case, seed):
    systems, points = _draw_inputs(case, seed)
    prec, w, op = PRECISION[case["prec"]], WORDS[case["prec"]], case["op"]
    st = dict(op=op)
    new = dict(dtype=torch.float64, device="cuda")
    if op == "track":
        paths = 2 ** case["n"]
        st["ev"] = pkg.PolyEval(systems[0], prec, max_points=paths)
        st["start"] = st["ev"].start_points(paths)
        return st
    if op == "many":
        st["ev"] = pkg.PolyEvalMany(systems, [p.shape[1] for p in points], prec)
        st["x"], st["f"], st["J"] = st["ev"].buffers()
        st["ev"].pack_points([torch.from_numpy(p).cuda() for p in points], st["x"])
        return st
    n, P = case["n"], case["P"]
    st["ev"] = pkg.PolyEval(systems[0], prec, max_points=P)
    if op == "host":
        st["P"] = P
        st["x"] = torch.from_numpy(points[0]).pin_memory()
        st["f"] = torch.empty((n, P, w), dtype=torch.float64).pin_memory()
        st["J"] = torch.empty((n, n, P, w), dtype=torch.float64).pin_memory()
        return st
    st["x"] = torch.from_numpy(points[0]).cuda()
    st["f"] = torch.empty((n, P, w), **new)
    st["J"] = torch.empty((n, n, P, w), **new)
    if op == "newton":
        st["work"] = torch.empty_like(st["x"])
        st["norms"] = torch.empty((P, 2), **new)
    return st


def run(st):
    op, ev = st["op"], st["ev"]
    if op == "track":
        x = st["start"].clone()
        status, t, _iterations = ev.track(x)
        return dict(x=x, t=t, status=status)
    if op == "many":
        ev.eval_buffers(st["x"], st["f"], st["J"])
        return dict(f=st["f"], J=st["J"])
    if op == "host":
        pkg.polyeval_eval_host(ev.handle, st["x"], st["P"], st["f"], st["J"])
        return dict(f=st["f"], J=st["J"])
    if op == "newton":  # the step works in place: keep the points for the next pass
        st["work"].copy_(st["x"])
        dx, lu, norms = ev.newton(st["work"], st["f"], st["J"], st["norms"])
        return dict(x=st["work"], dx=dx, lu=lu, norms=norms)
    f, J = ev.eval(st["x"], st["f"], st["J"])
    return dict(f=f, J=J)


# ---------------------------------------------------------------------------
# what a pass cannot do without, and its results in 64 bits
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: points, coefficients and exponent lists in, f and J out.  flops:
    a monomial's value takes k complex products, its k derivative sums and its
    value sum k + 1 complex additions (6 and 2 flops in the case's own
    precision, which takes several machine operations each)."""
    w = 8 * WORDS[case["prec"]]
    if case["op"] == "track":
        n, paths = case["n"], 2 ** case["n"]
        return {"bytes": 2.0 * w * n * paths, "flops": 8.0 * paths * (n * n * n + 4.0 * n * n * n)}
    if case["op"] == "many":  # sizes are drawn per system: expected values
        S, n, m, k, P = case["systems"], (8 + case["n"]) / 2, (8 + case["m"]) / 2, (2 + case["k"]) / 2, (1 + case["P"]) / 2
    else:
        S, n, m, k, P = 1, case["n"], case["m"], case["k"], case["P"]
    M = n * m
    flops = M * P * (6.0 * k + 2.0 * (k + 1))
    if case["op"] == "newton":
        flops += P * (8.0 / 3.0) * n ** 3
    return {"bytes": S * (w * P * (2 * n + n * n) + M * (w + 4.0 * k)), "flops": S * flops}


def _values(system, x):
    """f [N, P] and J [N, n, P] of complex128 points x [n, P], term by term."""
    n, P = x.shape
    h = system.coef.shape[1] // 2
    c = torch.from_numpy(system.coef[:, 0] + 1j * system.coef[:, h]).to(x.device)
    emax = int(system.exp.max())
    pw = torch.ones((emax + 1, n, P), dtype=x.dtype, device=x.device)
    for a in range(1, emax + 1):
        pw[a] = pw[a - 1] * x
    f = torch.zeros((system.n_polys, P), dtype=x.dtype, device=x.device)
    J = torch.zeros((system.n_polys, n, P), dtype=x.dtype, device=x.device)
    ks = np.diff(system.mono_ptr)
    for p in range(system.n_polys):
        rows = np.arange(system.poly_ptr[p], system.poly_ptr[p + 1])
        for k in np.unique(ks[rows]):
            every = rows[ks[rows] == k]
            for r in np.array_split(every, -(-len(every) * max(1, int(k)) * P // 20_000_000)):
                at = system.mono_ptr[r][:, None] + np.arange(k)[None, :]
                v = torch.from_numpy(system.pos[at].astype(np.int64)).to(x.device)
                a = torch.from_numpy(system.exp[at].astype(np.int64)).to(x.device)
                cr = c[torch.from_numpy(r).to(x.device)][:, None]
                left = [cr.expand(len(r), P)]
                for j in range(k):
                    left.append(left[-1] * pw[a[:, j], v[:, j]])
                f[p] += left[-1].sum(0)
                right = torch.ones_like(left[0])
                for j in range(k - 1, -1, -1):
                    d = a[:, j, None] * left[j] * pw[a[:, j] - 1, v[:, j]] * right
                    J[p].index_add_(0, v[:, j], d)
                    right = right * pw[a[:, j], v[:, j]]
    return f, J


def _laid_out(z, words):
    """A complex tensor as [..., words] doubles: leading parts, the rest zero."""
    out = torch.zeros(z.shape + (words,), dtype=torch.float64, device=z.device)
    out[..., 0] = z.real
    out[..., words // 2] = z.imag
    return out


def exact(case, seed):
    if case["op"] == "track":
        return None
    systems, points = _draw_inputs(case, seed)
    w = WORDS[case["prec"]]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    fs, Js = [], []
    for s, p in zip(systems, points):
        x = torch.from_numpy(p[..., 0] + 1j * p[..., w // 2]).to(dev)
        f, J = _values(s, x)
        fs.append(f)
        Js.append(J)
    if case["op"] == "newton":
        # the factors depend on the row exchanges taken and have no one value
        f, J = fs[0], Js[0]
        dx = torch.linalg.solve(J.permute(2, 0, 1), -f.t().unsqueeze(-1)).squeeze(-1).t()
        norms = torch.stack([f.abs().amax(0), dx.abs().amax(0)], -1)
        return dict(x=_laid_out(x + dx, w), dx=_laid_out(dx, w), lu=None, norms=norms)
    if case["op"] == "many":
        return dict(f=torch.cat([_laid_out(f, w).reshape(-1, w) for f in fs]),
                    J=torch.cat([_laid_out(J, w).reshape(-1, w) for J in Js]))
    f, J = _laid_out(fs[0], w), _laid_out(Js[0], w)
    return dict(f=f.cpu(), J=J.cpu()) if case["op"] == "host" else dict(f=f, J=J)
