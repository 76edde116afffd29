"""The second relabelling of mesh-like graphs whose numbering has no locality (multilevel
preconditioner; random geometric graphs): rows keep their entries' order and clusters their members',
so the V-cycle and the operator are bit for bit those of the same graph without it (a handle with
the diagonal preconditioner builds the same hierarchy lazily and is never relabelled again), and whole
solves, default start vectors and users' trimmed vertices do not change."""
import numpy as np
import pytest

import synthgraphs as sg
from tests.gpu_util import dev_graph, need_gpu, orthonormal_columns, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,weighted,opts", [(700, False, {}), (20011, False, {"trim_index": 5}), (30000, True, {}),
                                             (90001, False, {})])
def test_relabelled_handle_gives_the_same_results(n, weighted, opts):
    need_gpu()
    import paper_1710_07080_gb300 as isira
    g = sg.rgg(n, 12.0, seed=3)
    rp, ci = dev_graph(g)
    w = torch.from_numpy(sg.edge_weights(g, 4)).cuda() if weighted else None
    rng = np.random.default_rng(n)
    x = torch.from_numpy(rng.standard_normal(g.n)).cuda()
    V = torch.from_numpy(orthonormal_columns(g.n, 3, 5)).cuda()
    with isira.Solver(rp, ci, weights=w, precond=1, **opts) as a, isira.Solver(rp, ci, weights=w, precond=0, **opts) as b:
        assert a.stats()["trim_index"] == b.stats()["trim_index"]
        for t in (x, x.float()):
            ya, la, ca = a.precond_apply(t)
            yb, lb, cb = b.precond_apply(t)
            assert (la, ca) == (lb, cb)
            assert torch.equal(ya, yb)
        # the operator: the same row sums; its global sums are taken in another order
        za, zb = a.apply_operator(x, 0.01, V), b.apply_operator(x, 0.01, V)
        assert float((za - zb).abs().max()) <= 1e-12 * float(zb.abs().max())
        assert torch.equal(a.apply_operator(x, 0.0), b.apply_operator(x, 0.0))


def test_solve_with_default_start_vector_matches():
    need_gpu()
    import paper_1710_07080_gb300 as isira
    g = sg.rgg(20500, 12.0, seed=9)
    rp, ci = dev_graph(g)
    lam = [isira.solve(rp, ci, 4, tol=1e-11, precond=pc).eigvals.numpy() for pc in (1, 0)]
    np.testing.assert_allclose(lam[0], lam[1], rtol=1e-9)
