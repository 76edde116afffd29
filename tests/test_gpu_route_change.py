"""A whole FP64 solve whose inner solves change from the one-launch kernel to launches per iteration as vectors
lock (a grid near the row limit, twelve pairs): eigenvalues against the closed form, and a converged inner
solve at a rank above 8 against the launches."""
import numpy as np
import pytest

import synthgraphs as sg
from tests.gpu_util import dev_graph, need_gpu, orthonormal_columns, torch

pytestmark = pytest.mark.gpu


def test_solve_across_both_paths_matches_closed_form():
    need_gpu()
    import paper_1710_07080_gb300 as isira
    nx, ny, k = 173, 171, 12
    g = sg.grid2d(nx, ny)
    rp, ci = dev_graph(g)
    with isira.Solver(rp, ci, precision=isira.ISIRA_FP64, precond=0) as s:
        taken = [s.inner_route(c, isira.ISIRA_FP64)["one_launch_ctas"] > 0 for c in range(k)]
        assert any(taken) and not all(taken)
        s.solve(k, tol=1e-10, u0=torch.from_numpy(sg.start_vector(g.n, 1)).cuda())
        lam, vec, res = s.eigpairs()
    ev = [2 - 2 * np.cos(np.pi * np.arange(m) / m) for m in (nx, ny)]
    closed = np.sort((ev[0][:, None] + ev[1][None, :]).ravel())[1:k + 1]
    np.testing.assert_allclose(lam.numpy(), closed, rtol=1e-9)
    assert float(res.max()) < 1e-9


@pytest.mark.parametrize("n,c", [(12000, 20), (16000, 31), (25000, 8)])
def test_converged_solve_matches_launches(n, c):
    need_gpu()
    import paper_1710_07080_gb300 as isira
    g = sg.watts_strogatz(n, 10, 0.1, seed=4)
    rp, ci = dev_graph(g)
    r = np.random.default_rng(n).standard_normal(g.n)
    V = orthonormal_columns(g.n, c, 7)
    r -= r.mean()
    r -= V @ (V.T @ r)
    r = torch.from_numpy(r / np.linalg.norm(r)).cuda()
    tau, z = 1e-10, {}
    for graph in (1, 0):
        with isira.Solver(rp, ci, precision=isira.ISIRA_FP64, precond=0, inner_graph=graph) as s:
            assert (s.inner_route(c, isira.ISIRA_FP64)["one_launch_ctas"] > 0) == bool(graph)
            z[graph], its, rel = s.inner_solve(r, V=torch.from_numpy(V).cuda(), tau=tau, precision=isira.ISIRA_FP64)
            assert rel <= tau and its < 5000
    # both have a relative preconditioned residual of tau; the operator's condition on this graph (a random graph of
    # degree 10, smallest positive eigenvalue above 0.1) is below 1000
    np.testing.assert_allclose(z[1].cpu().numpy(), z[0].cpu().numpy(), rtol=0,
                               atol=1000 * tau * float(z[0].abs().max()))
