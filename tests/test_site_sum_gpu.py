"""The two-level block reduction of the vector kernels at the edge between its
one-level and two-level forms (1024 blocks of 128 sites) and above: ||a||^2
and the inner products of the x, r update against FP64 sums of the same data.

Bounds: FP64 data, n = 24 Vh terms in tree order, below 64 eps relative;
FP32 data, 24 terms per site and 128 sites in FP32, (24 + 12) 2^-24 relative
for a sum of squares."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# Vh = 131072 (1024 blocks), 131136 (1025: a last group of one), 163840 (1280)
LATTICES = [(16, 16, 16, 64), (1366, 4, 6, 8), (16, 16, 32, 40)]


@pytest.mark.parametrize("dims", LATTICES)
@pytest.mark.parametrize("prec,tol", [("f64", 64 * 2.0 ** -53), ("f32", 36 * 2.0 ** -24)])
def test_sums_at_the_edge_of_two_levels(dims, prec, tol):
    from paper_1103_5103_gb300 import api, synth
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(synth.unit_gauge_field(dims)).cuda(), precs=(prec,))
    V, nrhs = lat.volume, 2
    stride = (lat.spinor_bytes(prec) + 255) // 256 * 256
    gen = torch.Generator(device="cuda").manual_seed(5)
    odd = torch.from_numpy(synth.parity(dims) == 1).cuda()

    def batch():
        buf = torch.zeros(nrhs * stride, dtype=torch.uint8, device="cuda")
        vals = []
        for r in range(nrhs):
            t = torch.view_as_complex(torch.randn((V, 4, 3, 2), dtype=torch.float64, device="cuda", generator=gen))
            if prec == "f32":
                t = t.to(torch.complex64).to(torch.complex128)
            t[odd] = 0
            lat.spinor_import(t, buf[r * stride:(r + 1) * stride], prec, api.EVEN)
            vals.append(t)
        return buf, vals

    a, av = batch()
    for _ in range(2):   # the second call finds the tickets reset
        got = api.vector_op(g, api.VEC_NORM2, prec, nrhs, stride, [a])
        for r in range(nrhs):
            want = float((av[r].abs() ** 2).sum())
            assert abs(got[r] - want) <= tol * want
    # omega = 1 and t = 0, so r = s: <rhat, s> and ||s||^2
    (x, _), (p, _), (s, sv), (r_, _), (rh, hv) = (batch() for _ in range(5))
    t = torch.zeros_like(s)
    dots = api.vector_op(g, api.VEC_XR, prec, nrhs, stride, [x, p, s, t, r_, rh], [(0, 1, 0)] * nrhs)
    for r in range(nrhs):
        d = complex(torch.vdot(hv[r].reshape(-1), sv[r].reshape(-1)))
        n = float((sv[r].abs() ** 2).sum())
        size = float(hv[r].abs().square().sum().sqrt() * sv[r].abs().square().sum().sqrt())
        assert abs(dots[3 * r] - d.real) <= tol * size and abs(dots[3 * r + 1] - d.imag) <= tol * size
        assert abs(dots[3 * r + 2] - n) <= tol * n
