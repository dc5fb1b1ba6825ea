"""The fixed-point FP64 hop (variant 6000) against an extended-precision
reference and against the FP64-pipe hop (variant 101).

Bound.  With 2^E the exponent of the largest component of a site's eight
neighbours, a transporter is off by at most: the conversion (two components
rounded down by one unit of 2^(E-58) each, times a link row of unit norm:
sqrt(6) 2^(E-57)), the dropped lo*lo products and the rounded low word (6/4
+ 1/2 units of 2^(E-56)) and the shifts to a larger scale (one unit each, at
most one per transporter): below 2^(E-54).  Eight of them: 2^(E-51), plus
the rounding of the result to FP64."""
import numpy as np
import pytest
import torch

from paper_1103_5103_gb300 import synth

pytestmark = pytest.mark.gpu

LD, CLD = np.longdouble, np.clongdouble
# v^dag of the projectors 1 - gamma_mu = v1 v1^dag + v2 v2^dag (Table 1)
V1 = [(1j, 0, 0, 1), (-1, 0, 0, 1), (0, -1j, 0, 1), (0, 1, 0, 1)]
V2 = [(0, 1j, 1, 0), (0, 1, 1, 0), (1j, 0, 1, 0), (1, 0, 1, 0)]


@pytest.fixture(scope="module")
def api():
    from paper_1103_5103_gb300 import api as A
    return A


def _shift(f, dims, mu, step):
    X, Y, Z, T = dims
    g = np.roll(f.reshape((T, Z, Y, X) + f.shape[1:]), -step, axis=3 - mu)
    if mu == 3:
        g = g.copy()
        g[T - 1 if step > 0 else 0] *= -1
    return g.reshape(f.shape)


def _reference(U, dims, psi, dagger):
    """D psi in extended precision, and the largest neighbour component of each site."""
    U, psi = U.astype(CLD), psi.astype(CLD)
    out = np.zeros_like(psi)
    big = np.zeros(psi.shape[0], dtype=LD)
    mag = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(1, 2))
    for mu in range(4):
        for step in (1, -1):
            plus = (step > 0) == dagger
            P = np.zeros((4, 4), dtype=CLD)
            for vd in (V1[mu], V2[mu]):
                v = np.array(vd, dtype=CLD)
                if plus:
                    v[:2] *= -1
                P += np.conj(v)[:, None] * v[None, :]
            f = (psi[:, :, None, :] * P[None, :, :, None]).sum(axis=1)
            if step > 0:
                f = _shift(f, dims, mu, 1)
                f = (U[mu][:, None, :, :] * f[:, :, None, :]).sum(axis=3)
            else:
                f = (np.conj(U[mu]).transpose(0, 2, 1)[:, None] * f[:, :, None, :]).sum(axis=3)
                f = _shift(f, dims, mu, -1)
            out += f
            big = np.maximum(big, np.abs(_shift(mag[:, None], dims, mu, step))[:, 0])
    return out, big


def _source(dims, kind):
    psi = synth.gaussian_source(dims, seed=11)
    n = np.arange(psi.shape[0])
    if kind == "sites":           # magnitudes over 80 binary orders from site to site
        psi = psi * (2.0 ** ((n * 37) % 81 - 40))[:, None, None]
    elif kind == "components":    # and over 40 within a site
        psi = psi * 2.0 ** ((np.arange(12).reshape(4, 3) * 17 + n[:, None, None]) % 41 - 20)
    elif kind == "point":
        psi = synth.point_source(dims, 2, 1, site=3)
    elif kind == "large":
        psi = psi * 2.0 ** 800
    elif kind == "small":
        psi = psi * 2.0 ** -780
    return psi


def _hop(api, lat, g, psi, variant, dagger=False, x=None, coef=1.0, nrhs=1):
    """Odd outputs from even inputs of nrhs copies of psi; returns the last, canonical."""
    stride = (lat.spinor_bytes("f64") + 255) // 256 * 256
    a = torch.zeros(nrhs * stride, dtype=torch.uint8, device="cuda")
    t = torch.from_numpy(np.ascontiguousarray(psi)).cuda()
    for r in range(nrhs):
        lat.spinor_import(t, a[r * stride:(r + 1) * stride], "f64", api.EVEN)
    xo = None
    if x is not None:
        xo = torch.zeros_like(a)
        for r in range(nrhs):
            lat.spinor_import(torch.from_numpy(x).cuda(), xo[r * stride:(r + 1) * stride], "f64", api.ODD)
    b = torch.zeros_like(a)
    api.hop_batch(g, a, b, nrhs, stride, coef, "f64", api.ODD, -variant if variant else 1, x=xo, dagger=dagger)
    out = torch.zeros_like(t)
    lat.spinor_export(b[(nrhs - 1) * stride:], out, "f64", api.ODD)
    return out.cpu().numpy()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 10), (4, 6, 6, 4)])
@pytest.mark.parametrize("kind", ["gauss", "sites", "components", "point", "large", "small"])
def test_error_bound_and_no_worse_than_fp64(api, dims, kind):
    U = synth.gauge_field(dims, 0.5, seed=21)
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(U).cuda(), precs=("f64",))
    psi = _source(dims, kind)
    odd = synth.parity(dims) == 1
    psi[odd] = 0
    for dagger in (False, True):
        want, big = _reference(U, dims, psi, dagger)
        err = {}
        for variant in (6000, 101):
            if variant == 101 and dagger:
                continue
            got = _hop(api, lat, g, psi, variant, dagger).astype(CLD)
            d = np.maximum(np.abs((got - want).real), np.abs((got - want).imag))[odd]
            if variant == 6000:
                bound = LD(2.0) ** -51 * big[odd, None, None] + LD(2.0) ** -53 * np.abs(want[odd])
                assert np.all(d <= bound), float((d / np.maximum(bound, LD(1e-300))).max())
            err[variant] = float(np.sqrt((np.abs(got - want)[odd] ** 2).sum()))
        if 101 in err:
            # no further off than the FP64 hop; a point source's few values, which
            # both hops all but round correctly, no further than one rounding
            once = 2.0 ** -53 * float(np.sqrt((np.abs(want)[odd] ** 2).sum()))
            assert err[6000] <= (max(err[101], once) if kind == "point" else err[101]), err


@pytest.mark.parametrize("nrhs", [1, 3, 5])
def test_batched_xpay_is_the_single_hop(api, nrhs):
    """Ragged last warps, the rhs order and the epilogue: every rhs of a batch
    equals the single hop bit for bit, whatever rhs_block asks for."""
    dims = (6, 4, 2, 10)   # 240 sites per parity
    U = synth.gauge_field(dims, 0.5, seed=22)
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(U).cuda(), precs=("f64",))
    psi, x = synth.gaussian_source(dims, seed=23), synth.gaussian_source(dims, seed=24)
    one = _hop(api, lat, g, psi, 6000, x=x, coef=-0.13)
    assert np.array_equal(_hop(api, lat, g, psi, 6000, x=x, coef=-0.13, nrhs=nrhs), one)
    for variant in (0, 6001, 6002):
        assert np.array_equal(_hop(api, lat, g, psi, variant, x=x, coef=-0.13, nrhs=nrhs), one)
    ref = _hop(api, lat, g, psi, 101, x=x, coef=-0.13)
    assert np.linalg.norm(one - ref) <= 1e-15 * np.linalg.norm(ref)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e300, 1e-290, 5e-324, 0.0])
def test_out_of_range_sites_take_the_fp64_path(api, value):
    """One even site holds a component outside the scale's range (or only
    zeros): its neighbours get what the FP64 transporters give, the rest stays."""
    dims = (4, 4, 6, 4)
    U = synth.gauge_field(dims, 0.5, seed=25)
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(U).cuda(), precs=("f64",))
    psi = synth.gaussian_source(dims, seed=26)
    even = np.flatnonzero(synth.parity(dims) == 0)
    psi[even] *= 1e-295 if value in (1e-290, 5e-324) else 1.0   # the rest as small: nothing hides the entry
    if value == 0.0:
        psi[even] = 0
        psi[even[7]] = 1.0
    else:
        psi[even[5]] = 0
        psi[even[5], 2, 1] = value
    got, ref = _hop(api, lat, g, psi, 6000), _hop(api, lat, g, psi, 101)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(np.isinf(got.real), np.isinf(ref.real)) and np.array_equal(np.isinf(got.imag), np.isinf(ref.imag))
    ok = np.isfinite(ref)
    scale = np.abs(ref[ok]).max()
    assert np.abs(got[ok] - ref[ok]).max() <= 2.0 ** -50 * scale + 1e-323
    if value == 0.0:
        assert np.array_equal(got == 0, ref == 0)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 10), (8, 8, 8, 8), (10, 14, 12, 16), (12, 14, 12, 16)])
@pytest.mark.parametrize("kind", ["gauss", "sites", "special"])
def test_canonical_application_is_the_internal_one(api, dims, kind):
    """wilson_dslash in FP64 reads and writes the canonical fields, with the
    directions of a site on four warps up to 760 chunks of 16 sites (10x14x12x16:
    840 chunks per parity, 2^4: one ragged chunk) and in one thread above.  It
    agrees with the same application from page-locked host fields, which goes
    through the layout passes and the internal hops: the sums differ by the
    order of their rescaling, four units of 2^(E-56) per hop."""
    U = synth.gauge_field(dims, 0.5, seed=31)
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(U).cuda(), precs=("f64",))
    psi = _source(dims, "gauss" if kind == "special" else kind)
    if kind == "special":
        psi[3, 2, 1], psi[5 % len(psi), 0, 0] = np.nan, 1e300
    dev = torch.from_numpy(np.ascontiguousarray(psi)).cuda()
    host = torch.from_numpy(np.ascontiguousarray(psi)).pin_memory()
    for op in (api.OP_HOP, api.OP_M, api.OP_MPREC):
        for f in (api.wilson_dslash, api.wilson_dslash_dag):
            a = torch.full_like(dev, float("nan"))
            b = torch.full_like(host, float("nan")).pin_memory()
            f(g, dev, a, 0.13, "f64", op)
            f(g, host, b, 0.13, "f64", op)
            torch.cuda.synchronize()
            a, b = a.cpu().numpy(), b.numpy()
            assert np.array_equal(np.isnan(a), np.isnan(b))
            ok = np.isfinite(b) & (np.abs(b) < 1e290)
            big = np.abs(b[ok]).max()
            assert np.abs(a[ok] - b[ok]).max() <= 2.0 ** -50 * big
            if op == api.OP_MPREC:
                assert np.all(a[synth.parity(dims) == 1] == 0)


def _separating_links(dims, kind):
    """Links that keep colours apart: unit, diagonal, or SU(2) on colours 0, 1."""
    U = synth.unit_gauge_field(dims)
    rng = np.random.default_rng(5)
    if kind == "diagonal":
        a = rng.uniform(-np.pi, np.pi, U.shape[:2] + (2,))
        for c, p in enumerate((a[..., 0], a[..., 1], -a[..., 0] - a[..., 1])):
            U[..., c, c] = np.exp(1j * p)
    elif kind == "block":
        q = rng.standard_normal(U.shape[:2] + (4,))
        q /= np.linalg.norm(q, axis=-1, keepdims=True)
        a, b = q[..., 0] + 1j * q[..., 1], q[..., 2] + 1j * q[..., 3]
        U[..., 0, 0], U[..., 0, 1], U[..., 1, 0], U[..., 1, 1] = a, b, -b.conj(), a.conj()
    return U


@pytest.mark.parametrize("kind", ["unit", "diagonal", "block"])
def test_colours_that_do_not_mix_keep_their_precision(api, kind):
    """Colours 2^-30 and 2^-60 of another (block: only colour 2 stands apart):
    each comes out to FP64 rounding of its own size, through every FP64
    operator.  Bound per colour: 8 transporters and the epilogue, some 20
    roundings each of at most the colour's own norm, twice for M_prec."""
    dims = (4, 6, 2, 8)
    U = _separating_links(dims, kind)
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(U).cuda(), precs=("f64",))
    psi = synth.gaussian_source(dims, seed=12) * (2.0 ** np.array([0, 0 if kind == "block" else -30, -60]))
    odd = synth.parity(dims) == 1
    dev, k = torch.from_numpy(psi).cuda(), 0.13
    even_in = psi.copy()
    even_in[odd] = 0

    def close(got, want):
        for c in range(3):
            e = np.sqrt((np.abs(got[..., c].astype(CLD) - want[..., c]) ** 2).sum())
            assert e <= 2.0 ** -48 * np.sqrt((np.abs(want[..., c]) ** 2).sum()), (c, float(e))

    for dagger, f in ((False, api.wilson_dslash), (True, api.wilson_dslash_dag)):
        D = _reference(U, dims, psi, dagger)[0]
        Doe = _reference(U, dims, even_in, dagger)[0]
        DD = _reference(U, dims, Doe, dagger)[0]
        mprec = even_in - LD(k) ** 2 * DD
        mprec[odd] = 0
        for op, want in ((api.OP_HOP, D), (api.OP_M, psi - LD(k) * D), (api.OP_MPREC, mprec)):
            a, b = torch.empty_like(dev), torch.empty_like(dev)
            f(g, dev, a, k, "f64", op)
            api.wilson_dslash_noalloc(g, dev, b, k, "f64", op, dagger=dagger)
            close(a.cpu().numpy(), want)
            close(b.cpu().numpy(), want)
        Doe[~odd] = 0
        close(_hop(api, lat, g, even_in, 0, dagger), Doe)             # rhs_block 1
        close(_hop(api, lat, g, even_in, 0, dagger, nrhs=3), Doe)


@pytest.mark.parametrize("exponent,fixed", [(-29, True), (-31, False)])
def test_where_colours_count_as_mixed(api, exponent, fixed):
    """The line at entries of 2^-30: rotations by 2^exponent in all three planes."""
    dims = (2, 2, 2, 2)
    th = 2.0 ** exponent
    R = np.eye(3)
    for i, j in ((0, 1), (0, 2), (1, 2)):
        P = np.eye(3)
        P[i, i] = P[j, j] = np.cos(th)
        P[i, j], P[j, i] = np.sin(th), -np.sin(th)
        R = R @ P
    # random links but for one
    U = synth.gauge_field(dims, 0.5, seed=33)
    U[2, 5] = R
    g = api.Gauge(api.Lattice(dims), torch.from_numpy(U).cuda(), precs=("f64",))
    assert (api.autotune(g, "f64", 1)[0] == 6000) == fixed
