"""Initial guess and first residual in FP64 as scaled integers.

The pass itself (test_pass_*): x and r against extended-precision sums, within
the bound of its arithmetic, over cancelling coefficients and the whole range
of the scale, and FP64 sums outside it.

The solves that start from it (test_guessed_solutions): masses solved from
Lagrange guesses through up to 14 earlier ones reach the residual asked for
(checked by the FP64 operator), agree with solves from a zero guess, and scale
with the source."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,n_mass", [((4, 4, 4, 6), 15), ((6, 2, 4, 10), 4), ((8, 6, 2, 4), 2)])
@pytest.mark.parametrize("inner", ["f64", "f32"])
def test_guessed_solutions(dims, n_mass, inner):
    from oracle import oracle as O
    from paper_1103_5103_gb300 import api, synth
    U = synth.gauge_field(dims, 0.4, seed=71)
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(U).cuda(), precs=("f64", "f32"))
    masses = [0.5 * 0.9 ** i for i in range(n_mass)]
    bs = [synth.point_source(dims), synth.gaussian_source(dims, seed=72)]

    def run(scale, guess):
        xs, st = api.multimass_solve(g, [torch.from_numpy(b * scale).cuda() for b in bs], masses,
                                     api.params(inner_prec=inner, outer_prec="f64", guess=guess, guess_max=15))
        assert max(s["true_relres"] for row in st for s in row) <= 1e-10
        return [[x.cpu().numpy() / scale for x in row] for row in xs]

    ref = run(1.0, api.GUESS_POLY)
    for b, row in zip(bs, ref):
        for m, x in zip(masses, row):
            assert O.true_relres(U, dims, b, x, m) <= 1.1e-10
    # two solutions of residual 1e-10: kappa form, ||(1 - kappa D)^-1|| <= (m + 4) / m < 40
    e = 40 if inner == "f64" else 10   # FP32 inner products of residuals of 1e-10 stay normal
    for other in (run(1.0, api.GUESS_ZERO), run(2.0 ** e, api.GUESS_POLY), run(2.0 ** -e, api.GUESS_POLY)):
        for b, row, orow in zip(bs, ref, other):
            for x, y in zip(row, orow):
                assert np.linalg.norm(x - y) <= 8e-9 * np.linalg.norm(b)


DIMS = (6, 4, 2, 10)   # 240 sites per parity: a ragged block
LD = np.longdouble


def _pass(k, xs, ys, b, c, d):
    """The pass on n_rhs vectors: xs, ys [k][rhs], b [rhs] canonical, c, d [rhs][k]."""
    from paper_1103_5103_gb300 import api, synth
    lat = api.Lattice(DIMS)
    g = api.Gauge(lat, torch.from_numpy(synth.gauge_field(DIMS, 0.5, seed=73)).cuda(), precs=("f64",))
    n = len(b)
    stride = (lat.spinor_bytes("f64") + 255) // 256 * 256

    def pack(rows):
        buf = torch.zeros(n * stride, dtype=torch.uint8, device="cuda")
        for r, v in enumerate(rows):
            lat.spinor_import(torch.from_numpy(np.ascontiguousarray(v)).cuda(), buf[r * stride:(r + 1) * stride], "f64", 0)
        return buf

    vecs = [pack(v) for v in xs] + [pack(v) for v in ys] + [pack(b)]
    outs = [torch.full((n * stride,), 255, dtype=torch.uint8, device="cuda") for _ in range(2)]
    api.vector_op(g, api.VEC_GUESS + k, "f64", n, stride, vecs + outs, [list(c[r]) + list(d[r]) for r in range(n)])
    res = []
    for o in outs:
        rows = []
        for r in range(n):
            t = torch.zeros(b[r].shape, dtype=torch.complex128, device="cuda")
            lat.spinor_export(o[r * stride:], t, "f64", 0)
            rows.append(t.cpu().numpy())
        res.append(rows)
    return res


def _inputs(k, seed, scale=1.0):
    from paper_1103_5103_gb300 import synth
    odd = synth.parity(DIMS) == 1

    def v(s):
        a = synth.gaussian_source(DIMS, seed=s) * scale
        a[odd] = 0
        return a
    return ([[v(seed + 10 * j + r) for r in range(2)] for j in range(k)],
            [[v(seed + 500 + 10 * j + r) for r in range(2)] for j in range(k)], [v(seed + 900 + r) for r in range(2)])


def _parts(z):
    return z.real.astype(LD), z.imag.astype(LD)


def _bound_and_sum(terms, extra, k):
    """Sum of coefficient times vector and of extra vectors, in extended
    precision, and the bound of the integer arithmetic: 4 k + 4 units of 2^-55
    of the largest term of each complex number, and one rounding."""
    want, big = [LD(0), LD(0)], LD(0)
    for w, z in terms + [(1.0, z) for z in extra]:
        p = [LD(w) * x for x in _parts(z)]
        big = np.maximum(big, np.maximum(np.abs(p[0]), np.abs(p[1])))
        want = [want[0] + p[0], want[1] + p[1]]
    return want, [(4 * k + 4) * LD(2.0) ** -55 * big + LD(2.0) ** -53 * np.abs(w) for w in want]


def _check(k, xs, ys, b, c, d):
    X, R = _pass(k, xs, ys, b, c, d)
    for r in range(len(b)):
        want, bound = _bound_and_sum([(c[r][j], xs[j][r]) for j in range(k)], [np.zeros_like(b[r])], k)
        for got, w, e in zip(_parts(X[r]), want, bound):
            assert np.all(np.abs(got - w) <= e)
        want, bound = _bound_and_sum([(d[r][j], ys[j][r]) for j in range(k)], [b[r], -X[r]], k)
        for got, w, e in zip(_parts(R[r]), want, bound):
            assert np.all(np.abs(got - w) <= e)


@pytest.mark.parametrize("k", [0, 1, 2, 15])
@pytest.mark.parametrize("kind", ["lagrange", "spread", "low", "high", "split"])
def test_pass_error_bound(k, kind):
    rng = np.random.default_rng(k)
    # extrapolation weights of equally spaced points: alternating, up to 6435 for 15
    import math
    lag = [(-1.0) ** j * math.comb(k, j + 1) for j in range(k)]
    c = [[w * (1 + 0.1 * r) for w in lag] for r in range(2)]
    d = [[0.0131 * w for w in row] for row in c]
    xs, ys, b = _inputs(k, 1000 + k)
    if kind == "spread":      # magnitudes over 120 binary orders, between and within the vectors, and zeros
        for v in xs + ys + [b]:
            for a in v:
                a *= 2.0 ** rng.integers(-60, 60, a.shape)
                a[::7] = 0
        c = [[w * 2.0 ** int(rng.integers(-60, 60)) for w in row] for row in c]
    elif kind in ("low", "high"):   # the ends of the scale: components 2^(-423..478), coefficients 2^(-200..201)
        s, t = (-415, -185) if kind == "low" else (470, 185)
        xs, ys, b = _inputs(k, 1000 + k, 2.0 ** s)
        c, d = ([[w * 2.0 ** t for w in row] for row in m] for m in (c, d))
    elif kind == "split":     # re and im 2^40 apart
        xs, ys = ([[a.real + 1j * 2.0 ** -40 * a.imag for a in v] for v in m] for m in (xs, ys))
    _check(k, xs, ys, b, c, d)


@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("where", ["x", "y", "b", "c", "d"])
@pytest.mark.parametrize("value", [2.0 ** -460, 2.0 ** 490, 5e-324, np.inf, -np.inf, np.nan])
def test_pass_outside_the_scale(k, where, value):
    """A component or coefficient outside the integers' range takes FP64 sums;
    the components beside it stay."""
    xs, ys, b = _inputs(k, 2000 + k)
    c, d = [[0.7] * k, [-1.3] * k], [[0.01] * k, [0.02] * k]
    small = 0 < value < 1
    if where == "c":
        c[1][0] = value
    elif where == "d":
        d[1][0] = value
    else:
        v = {"x": xs[0][1], "y": ys[0][1], "b": b[1]}[where]
        v[0, 2, 1] = value if small else 1.0 + 1j * value
    from paper_1103_5103_gb300 import synth
    with np.errstate(all="ignore"):
        X, R = _pass(k, xs, ys, b, c, d)
        even = synth.parity(DIMS) == 0   # what the pass works on: 0 inf would be NaN elsewhere
        X, R, b = ([a[even] for a in v] for v in (X, R, b))
        xs, ys = ([[a[even] for a in v] for v in m] for m in (xs, ys))
        for r in range(2):
            for got, terms, extra in ((X[r], [(c[r][j], xs[j][r]) for j in range(k)], []),
                                      (R[r], [(d[r][j], ys[j][r]) for j in range(k)], [b[r], -X[r]])):
                for part in (0, 1):
                    f = [LD(w) * _parts(z)[part] for w, z in terms] + [_parts(z)[part] for z in extra]
                    want, size = sum(f), sum(np.abs(t) for t in f)
                    g = _parts(got)[part].astype(np.float64)
                    w64 = want.astype(np.float64)
                    assert np.array_equal(np.isnan(g), np.isnan(w64)) and np.array_equal(np.isinf(g), np.isinf(w64))
                    ok = np.isfinite(w64)
                    assert np.array_equal(g[~ok], w64[~ok], equal_nan=True)
                    # FP64 sums, or the integers' bound, whose scale re and im share
                    other = sum(np.abs(LD(w) * _parts(z)[1 - part]) for w, z in terms + [(1.0, z) for z in extra])
                    other = np.where(np.isfinite(other.astype(np.float64)), other, 0)
                    assert np.all(np.abs(g - want)[ok] <= (4 * k + 4) * LD(2.0) ** -52 * (size + other)[ok] + LD(5e-324))
