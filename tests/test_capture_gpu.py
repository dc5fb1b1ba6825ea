"""An operator application captured into a graph after other calls of the same
handle: a route that needs workspace the earlier calls did not need allocates
it under capture."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 6), (8, 16, 16, 18)])   # below and above 16384 sites per parity
@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "df"])
@pytest.mark.parametrize("warm", [True, False])
def test_first_use_of_a_route_under_capture(dims, prec, warm):
    from paper_1103_5103_gb300 import api, synth
    lat = api.Lattice(dims)
    U = torch.from_numpy(synth.gauge_field(dims, 0.5, seed=95)).cuda()
    psi = torch.from_numpy(synth.gaussian_source(dims, seed=96)).cuda()
    g = api.Gauge(lat, U, precs=(prec,))
    want = {}
    for op in (api.OP_HOP, api.OP_M, api.OP_MPREC):
        want[op] = torch.empty_like(psi)
        api.wilson_dslash(g, psi, want[op], 0.13, prec, op)
    torch.cuda.synchronize()
    for op in want:
        h = api.Gauge(lat, U, precs=(prec,))   # no workspace yet
        x = torch.empty_like(psi)
        if warm:
            api.wilson_dslash(h, psi, x, 0.13, prec, api.OP_M)
            torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            api.wilson_dslash(h, psi, x, 0.13, prec, op)
        x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(x, want[op]), op
