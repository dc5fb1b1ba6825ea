"""multimass_solve leaves the odd half of a call's sources out only where it is
exactly zero: an odd part whose squares underflow counts.  The norm of a
double-float vector is summed in FP32, where entries below 2.6e-23 square to
zero; here the even entries are about 2^-60 (8.7e-19) and the odd ones 2^-20
of them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mixed", [False, True])
def test_small_odd_part(mixed):
    from paper_1103_5103_gb300 import api, synth
    dims, scale = (4, 6, 4, 8), 2.0 ** -60
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(synth.gauge_field(dims, 0.4, seed=91)).cuda())
    odd = synth.parity(dims) == 1
    b = synth.gaussian_source(dims, seed=92)
    b[odd] *= 2.0 ** -20
    even = b.copy()
    even[odd] = 0
    # mixed: beside a source that has no odd part
    bs = [torch.from_numpy(b).cuda()] + ([torch.from_numpy(even).cuda()] if mixed else [])
    ref, _ = api.multimass_solve(g, bs, [0.5, 0.3], api.params(inner_prec="f64", tol=1e-12))
    xs, _ = api.multimass_solve(g, [t * scale for t in bs], [0.5, 0.3], api.params(inner_prec="f64", outer_prec="df"))
    for row, rrow in zip(xs, ref):
        for x, r in zip(row, rrow):
            # to the solve's tolerance of 1e-10, with ||M^-1|| <= (m + 4) / m < 15; without
            # b_o the odd half would be off by 2^-20 = 9.5e-7 of ||b||
            assert float((x / scale - r).norm()) <= 3e-9 * np.linalg.norm(b)
