"""Handles without the integer links of the fixed-point FP64 hop: every FP64
entry point works on the FP64 pipe and agrees with the handle that has them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DIMS = (6, 4, 2, 10)


@pytest.fixture(scope="module")
def api():
    from paper_1103_5103_gb300 import api as A
    return A


def _handles(api):
    """The same links with and without their integer copy."""
    from paper_1103_5103_gb300 import synth
    U = torch.from_numpy(synth.gauge_field(DIMS, 0.4, seed=81)).cuda()
    lat = api.Lattice(DIMS)
    a, b = (api.Gauge(lat, U) for _ in range(2))
    b.release_integer_links()
    return a, b


def test_operators_and_tuning(api):
    from paper_1103_5103_gb300 import synth
    g, p = _handles(api)
    assert api.autotune(g, "f64", 2)[0] == 6000
    # links released after tuning: the choice goes with them
    g2, _ = _handles(api)
    api.autotune(g2, "f64", 2)
    g2.release_integer_links()
    g2.release_integer_links()   # none left: no effect
    for h in (p, g2):
        assert api.autotune(h, "f64", 2)[0] in (101, 103, 201, 7101, 7102, 7201, 7202)
    psi = torch.from_numpy(synth.gaussian_source(DIMS, seed=82)).cuda()
    for op in (api.OP_HOP, api.OP_M, api.OP_MPREC):
        for f in (api.wilson_dslash, api.wilson_dslash_dag, api.wilson_dslash_noalloc):
            x, y = torch.empty_like(psi), torch.empty_like(psi)
            f(g, psi, x, 0.13, "f64", op)
            f(p, psi, y, 0.13, "f64", op)
            assert float((x - y).norm() / y.norm()) <= 1e-15
    n = p.lat.spinor_bytes("f64")
    a, b = torch.zeros(n, dtype=torch.uint8, device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda")
    with pytest.raises(api.WilsonError):
        api.hop_batch(p, a, b, 1, (n + 255) // 256 * 256, 1.0, "f64", api.ODD, -6000)


@pytest.mark.parametrize("kw", [dict(inner_prec="f64"), dict(inner_prec="f32"), dict(inner_prec="f16", inner_refine=1),
                                dict(inner_prec="f64", inner_solver=1), dict(inner_prec="f64", outer_blocks_per_sm=2),
                                dict(inner_prec="f64", mode=0), dict(inner_prec="f64", mode=2)])
def test_solves(api, kw):
    from paper_1103_5103_gb300 import synth
    g, p = _handles(api)
    bs = [torch.from_numpy(synth.gaussian_source(DIMS, seed=83)).cuda(), torch.from_numpy(synth.point_source(DIMS)).cuda()]
    ref, _ = api.multimass_solve(g, bs, [0.5, 0.2], api.params(**kw))
    xs, st = api.multimass_solve(p, bs, [0.5, 0.2], api.params(**kw))
    # then the handle that has solved with them loses them: nothing captured is reused
    g.release_integer_links()
    ys, _ = api.multimass_solve(g, bs, [0.5, 0.2], api.params(**kw))
    assert max(s["true_relres"] for row in st for s in row) <= 1e-10
    for row in zip(ref, xs, ys):
        for r, x, y in zip(*row):   # residual 1e-10 each, ||M^-1|| <= (m + 4) / m < 21
            assert float((x - r).norm() / r.norm()) <= 5e-9 and float((y - r).norm() / r.norm()) <= 5e-9


def test_multishift_and_gradient(api):
    from paper_1103_5103_gb300 import synth
    g, p = _handles(api)
    b = torch.from_numpy(synth.gaussian_source(DIMS, seed=84)).cuda()
    out = []
    for h in (g, p):
        xs = [torch.empty_like(b) for _ in range(3)]
        st = api.bicgstab_m_solve(h, b, xs, [0.2, 0.4, 0.7], api.params(outer_prec="f64"))
        assert max(s["true_relres"] for s in st) <= 1e-10
        dU, dm, _ = api.solve_backward(h, b, xs, [0.2, 0.4, 0.7], xs, api.params(inner_prec="f64"))
        out.append([torch.stack(xs), dU, torch.tensor(dm)])
    for a, c in zip(*out):
        assert float((a - c).norm() / a.norm()) <= 1e-8


def _holds(api, g):
    n = g.lat.spinor_bytes("f64")
    a, b = (torch.zeros(n, dtype=torch.uint8, device="cuda") for _ in range(2))
    try:
        api.hop_batch(g, a, b, 1, (n + 255) // 256 * 256, 1.0, "f64", api.ODD, -6000)
    except api.WilsonError:
        return False
    return True


def _calls(api, b):
    """Calls with their results, for handles that hold all precisions."""
    def mm(**kw):
        def f(g):
            xs, st = api.multimass_solve(g, [b], [0.5, 0.3, 0.2], api.params(**kw))
            assert max(s["true_relres"] for s in st[0]) <= 1e-10
            return torch.stack(xs[0])
        return f

    def mprec(g):
        x = torch.empty_like(b)
        api.wilson_dslash(g, b, x, 0.13, "f64", api.OP_MPREC)
        return x

    def shifts(g):
        xs = [torch.empty_like(b) for _ in range(2)]
        api.bicgstab_m_solve(g, b, xs, [0.2, 0.4], api.params(outer_prec="f64"))
        return torch.stack(xs)

    def gradient(g):
        return api.solve_backward(g, b, [b], [0.3], None, api.params(inner_prec="f64"))[0]

    return dict(refined=mm(inner_prec="f16", inner_refine=1, outer_blocks_per_sm=2), ssm=mm(inner_prec="f64", guess=2),
                mprec=mprec, shifts=shifts, gradient=gradient)


@pytest.mark.parametrize("name", ["refined", "ssm", "mprec", "shifts", "gradient"])
def test_out_of_memory_gives_the_integer_links_up(api, name):
    """Whichever allocation of a call fails: the integer links are released and
    the call goes on without them, as on a handle that never had them."""
    from paper_1103_5103_gb300 import synth
    U = torch.from_numpy(synth.gauge_field(DIMS, 0.4, seed=85)).cuda()
    lat = api.Lattice(DIMS)
    b = torch.from_numpy(synth.gaussian_source(DIMS, seed=86)).cuda()
    call = _calls(api, b)[name]
    ref = call(api.Gauge(lat, U))
    after = 0
    while True:
        g = api.Gauge(lat, U)
        g.fail_allocation(after)
        x = call(g)
        assert float((x - ref).norm() / ref.norm()) <= 1e-8, after
        if _holds(api, g):   # fewer allocations than that
            break
        after += 1
    assert after >= (1 if name == "mprec" else 10)
    # nothing left to release: reported, and the next call finds a clean state
    g = api.Gauge(lat, U)
    g.release_integer_links()
    g.fail_allocation(0)
    with pytest.raises(api.WilsonError) as e:
        call(g)
    assert e.value.status == api.WL_ERR_OOM
    assert float((call(g) - ref).norm() / ref.norm()) <= 1e-8


@pytest.mark.parametrize("call", ["dslash", "noalloc", "batch"])
def test_captured_operators_keep_the_integer_links(api, call):
    """A caller's graph reads the links when it is replayed: neither a failed
    allocation nor the release call takes them away."""
    from paper_1103_5103_gb300 import synth
    U = torch.from_numpy(synth.gauge_field(DIMS, 0.4, seed=87)).cuda()
    lat = api.Lattice(DIMS)
    g = api.Gauge(lat, U)
    b = torch.from_numpy(synth.gaussian_source(DIMS, seed=88)).cuda()
    n = (lat.spinor_bytes("f64") + 255) // 256 * 256
    a = torch.zeros(n, dtype=torch.uint8, device="cuda")
    lat.spinor_import(b, a, "f64", api.EVEN)
    x = torch.empty_like(b) if call != "batch" else torch.zeros_like(a)

    def run():
        if call == "batch":
            api.hop_batch(g, a, x, 1, n, 1.0, "f64", api.ODD)
        else:
            (api.wilson_dslash if call == "dslash" else api.wilson_dslash_noalloc)(g, b, x, 0.13, "f64", api.OP_MPREC)

    run()   # workspace and addresses before the capture
    torch.cuda.synchronize()
    want = x.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    with pytest.raises(api.WilsonError):
        g.release_integer_links()
    g.fail_allocation(0)
    with pytest.raises(api.WilsonError) as e:
        api.multimass_solve(g, [b], [0.5], api.params(inner_prec="f64"))
    assert e.value.status == api.WL_ERR_OOM and _holds(api, g)
    x.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, want)
