"""The one-launch inner solve of small graphs (inner_cluster.cu) against the three-launch solve
(inner_graph = 0), which the oracle pins elsewhere: the same MINRES iterates to rounding, over the
edges of its tiles (slices of 32 rows, the steps of the CTA count, the last partial slice), deflation
ranks on both sides of the warps per CTA, weights, a user's trimmed vertex and both precisions."""
import numpy as np
import pytest

import synthgraphs as sg
from tests.gpu_util import dev_graph, need_gpu, orthonormal_columns, torch

pytestmark = pytest.mark.gpu

GRAPHS = {
    "path3": lambda: sg.path(3), "path33": lambda: sg.path(33), "complete65": lambda: sg.complete(65),
    "cycle256": lambda: sg.cycle(256), "grid257": lambda: sg.grid2d(257, 1 + 1), "grid31x33": lambda: sg.grid2d(31, 33),
    "er2049": lambda: sg.erdos_renyi(2060, 8.0, seed=3), "ws4097": lambda: sg.watts_strogatz(4097, 10, 0.1, seed=4),
    "er17000": lambda: sg.erdos_renyi(17000, 8.0, seed=5), "grid175x175": lambda: sg.grid2d(175, 175),
    "ws79999": lambda: sg.watts_strogatz(79999, 10, 0.1, seed=6),
}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("c,weighted,opts", [(0, False, {}), (1, False, {"trim_index": 2}), (7, True, {}),
                                             (31, False, {"drop_rank1": 1})])
def test_one_launch_solve_matches_three_launches(prec, name, c, weighted, opts):
    need_gpu()
    import paper_1710_07080_gb300 as isira
    g = GRAPHS[name]()
    if c > g.n - 2:
        pytest.skip("more columns than the graph has")
    rp, ci = dev_graph(g)
    w = torch.from_numpy(sg.edge_weights(g, 2)).cuda() if weighted else None
    P = isira.ISIRA_FP64 if prec == "fp64" else isira.ISIRA_MIXED
    rng = np.random.default_rng(c + g.n)
    r = rng.standard_normal(g.n)
    r = torch.from_numpy((r - r.mean()) / np.linalg.norm(r)).cuda()
    V = torch.from_numpy(orthonormal_columns(g.n, c, 7)).cuda() if c else None
    sigma = 0.001 if c else 0.0
    out = {}
    for graph in (1, 0):
        with isira.Solver(rp, ci, weights=w, precision=P, precond=0, inner_graph=graph, **opts) as s:
            out[graph] = s.inner_solve(r, sigma=sigma, V=V, tau=1e-12, max_it=6, precision=P)
            z2 = s.inner_solve(r, sigma=sigma, V=V, tau=1e-12, max_it=6, precision=P)[0]
            assert torch.equal(out[graph][0], z2)                    # deterministic, nothing left over from a solve
            if graph:
                assert s.stats()["kernel_launches"] > 0
    z1, its1, rel1 = out[1]
    z0, its0, rel0 = out[0]
    # six iterations: rounding is amplified by a few units each, so a thousand roundings bound the difference
    # (a two- or three-vertex graph ends at its exact solution earlier, in either path)
    u = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    scale = float(z0.abs().max())
    np.testing.assert_allclose(z1.cpu().numpy(), z0.cpu().numpy(), rtol=0, atol=1000 * u * max(scale, 1e-30))
    if rel0 > 1e4 * u:
        assert its1 == its0
        assert abs(rel1 - rel0) <= 1e4 * u


def test_profiling_keeps_results_and_counts_iterations():
    need_gpu()
    import paper_1710_07080_gb300 as isira
    g = sg.grid2d(40, 37)
    rp, ci = dev_graph(g)
    u0 = torch.from_numpy(sg.start_vector(g.n, 1)).cuda()
    with isira.Solver(rp, ci) as s:
        s.solve(3, tol=1e-9, u0=u0)
        lam = s.eigpairs()[0]
        s.set_profiling(True)
        s.solve(3, tol=1e-9, u0=u0)
        st = s.stats()
        assert torch.equal(lam, s.eigpairs()[0])
        assert st["inner_phase1_timed"] == st["inner_iters"] > 0
        assert st["inner_phase1_ms"] > 0 and st["inner_phase2_ms"] > 0
