"""Initial guess and first residual in FP64 as scaled integers: masses solved
from Lagrange guesses through up to 14 earlier ones reach the residual asked
for (checked by the FP64 operator), agree with solves from a zero guess, and
scale with the source."""
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
