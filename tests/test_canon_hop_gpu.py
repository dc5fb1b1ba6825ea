"""wilson_dslash in FP32, FP16 and double-float: the hop that stores to the
canonical field against the layout passes, which page-locked host fields
still take: the same values bit for bit, below, at and above the sizes where
M_prec changes its route (16384 sites per parity, 8x16x16x16; in double-float
8192, 8x16x16x8)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 10), (8, 16, 16, 8), (8, 16, 16, 10), (8, 16, 16, 16),
                                  (8, 16, 16, 18)])
@pytest.mark.parametrize("prec", ["f32", "f16", "df"])
def test_canonical_store_equals_export(dims, prec):
    from paper_1103_5103_gb300 import api, synth
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(synth.gauge_field(dims, 0.5, seed=41)).cuda(), precs=(prec,))
    psi = synth.gaussian_source(dims, seed=42)
    psi[1] *= 1e-40   # below FP16's and FP32's range
    dev = torch.from_numpy(psi).cuda()
    host = torch.from_numpy(psi).pin_memory()
    for op in (api.OP_HOP, api.OP_M, api.OP_MPREC):
        for f in (api.wilson_dslash, api.wilson_dslash_dag):
            a = torch.full_like(dev, float("nan"))
            b = torch.full_like(host, float("nan")).pin_memory()
            f(g, dev, a, 0.13, prec, op)
            f(g, host, b, 0.13, prec, op)
            torch.cuda.synchronize()
            assert np.array_equal(a.cpu().numpy(), b.numpy()), (op, f)
