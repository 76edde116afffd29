"""A second, larger solve on one handle: the deflation vectors move to a larger buffer, and what the handle
keeps between solves (the instantiated graphs of the inner iteration) must follow them.  Its results are
those of a fresh handle."""
import numpy as np
import pytest

import synthgraphs as sg
from tests.gpu_util import dev_graph, need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name,precond,opts", [("rmat12", 0, {}), ("grid151x140", 1, {}), ("er4000", 0, {"reorder": 0})])
def test_second_solve_with_more_pairs_matches_a_fresh_handle(name, precond, opts, prec):
    need_gpu()
    import paper_1710_07080_gb300 as isira
    g = {"rmat12": lambda: sg.rmat(12), "grid151x140": lambda: sg.grid2d(151, 140),
         "er4000": lambda: sg.erdos_renyi(4000, 8.0, seed=2)}[name]()
    rp, ci = dev_graph(g)
    P = isira.ISIRA_FP64 if prec == "fp64" else isira.ISIRA_MIXED
    u0 = torch.from_numpy(sg.start_vector(g.n, 1)).cuda()
    with isira.Solver(rp, ci, precision=P, precond=precond, **opts) as a:
        a.solve(3, tol=1e-9, u0=u0)
        lam3 = a.eigpairs()[0]
        a.solve(7, tol=1e-9, u0=u0)
        lam, vec, res = a.eigpairs()
        its = a.stats()["inner_iters"]
    with isira.Solver(rp, ci, precision=P, precond=precond, **opts) as b:
        b.solve(7, tol=1e-9, u0=u0)
        lam_b, vec_b, res_b = b.eigpairs()
        assert b.stats()["inner_iters"] == its
    assert torch.equal(lam, lam_b) and torch.equal(vec, vec_b)
    np.testing.assert_allclose(lam[:3].numpy(), lam3.numpy(), rtol=1e-9)
    assert float(res.max()) < 1e-9
