"""The number of inner iterations between two looks at the solver state
(whole captured blocks, then single captured iterations) changes nothing in a
solve: solutions and iteration counts are those of one iteration per look,
and a solve cut off by max_iter ends after the same whole blocks when it is
repeated."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inner,solver", [("f32", "SOLVER_BICGSTAB"), ("f16", "SOLVER_BICGSTAB"), ("f64", "SOLVER_CG")])
def test_groups_change_no_result(inner, solver):
    from paper_1103_5103_gb300 import api, synth
    dims = (8, 4, 6, 8)
    lat = api.Lattice(dims)
    g = api.Gauge(lat, torch.from_numpy(synth.gauge_field(dims, 0.3, seed=51)).cuda(), precs=("f64", "f32", "f16", "df"))
    bs = [torch.from_numpy(synth.z2_source(dims, seed=52 + r)).cuda() for r in range(2)]

    def run(**kw):
        xs, st = api.multimass_solve(g, bs, [0.4, 0.1], api.params(inner_prec=inner, inner_solver=getattr(api, solver), **kw),
                                     check=False)
        return np.stack([x.cpu().numpy() for row in xs for x in row]), [s["iterations"] for row in st for s in row]

    x1, it1 = run(graph_iters=1)
    for k in (3, 8, 50):
        x, it = run(graph_iters=k)
        assert it == it1 and np.array_equal(x, x1), k
    a, ita = run(graph_iters=8, max_iter=12)
    b, itb = run(graph_iters=8, max_iter=12)
    assert ita == itb and max(ita) > 12 and np.array_equal(a, b)
