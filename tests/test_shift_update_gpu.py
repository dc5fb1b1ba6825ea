"""The fixed-point shift updates of the FP64 multi-shift solver: a source
scaled by a power of two scales every vector of the recursion, exactly in
FP64, across the range that the integers take (a site component outside
2^(-423..478) takes the FP64 products), so the solution scales with it up to
rounding; sparse and dense sources, an odd number of sites per block."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (6, 2, 4, 10)])
@pytest.mark.parametrize("source", ["z2", "point"])
def test_scaled_source(dims, source):
    from oracle import oracle as O
    from paper_1103_5103_gb300 import api, synth
    U = synth.gauge_field(dims, 0.4, seed=61)
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(U).cuda(), precs=("f64",))
    b = synth.z2_source(dims, seed=62) if source == "z2" else synth.point_source(dims)
    shadow = torch.from_numpy(synth.gaussian_source(dims, seed=63)).cuda()   # of one size: <shadow, r>^2 stays normal
    masses = [0.1, 0.2, 0.35, 0.6]

    def run(scale):
        xs = [torch.empty(b.shape, dtype=torch.complex128, device="cuda") for _ in masses]
        st = api.bicgstab_m_solve(g, torch.from_numpy(b * scale).cuda(), xs, masses,
                                  api.params(outer_prec="f64", shadow=shadow))
        assert max(s["true_relres"] for s in st) <= 1e-10
        return [x.cpu().numpy() / scale for x in xs]

    ref = run(1.0)
    for m, x in zip(masses, ref):
        assert O.true_relres(U, dims, b, x, m) <= 1.1e-10
    # 2^-300 and 2^300: integers; 2^-410: residuals leave the range on the way;
    # 2^-440: FP64 products throughout (||b||^2 = 2^-880 is still normal)
    for e in (-300, 300, -410, -440):
        for a, x in zip(ref, run(2.0 ** e)):
            # both solve to a relative residual of 1e-10; ||M^-1|| <= 1 / m = 10
            assert np.linalg.norm(x - a) <= 2e-9 * np.linalg.norm(b), e
