"""The Gram matrix of the deflation vectors and its inverse, through the inner solve that uses them: ranks
around the steps of the kernel's layout (several segments to an entry, one, two entries to a thread; the
factor and the inverse in the tile's place) against the FP64 oracle's inner solve."""
import numpy as np
import pytest

import oracle
import synthgraphs as sg
from tests.gpu_util import dev_graph, need_gpu, orthonormal_columns, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c", [1, 2, 15, 16, 22, 23, 26, 27, 30, 31])
@pytest.mark.parametrize("n", [130, 4001])
def test_inner_solve_matches_oracle_at_every_layout(n, c):
    need_gpu()
    import paper_1710_07080_gb300 as isira
    g = sg.watts_strogatz(n, 10, 0.1, seed=3)
    rp, ci = dev_graph(g)
    V = orthonormal_columns(g.n, c, 7)
    r = np.random.default_rng(c).standard_normal(g.n)
    r = (r - r.mean()) / np.linalg.norm(r)
    with isira.Solver(rp, ci, precision=isira.ISIRA_FP64, precond=0, inner_graph=0) as s:
        st = s.stats()
        z, its, _ = s.inner_solve(torch.from_numpy(r).cuda(), sigma=0.001, V=torch.from_numpy(V).cuda(), tau=1e-12,
                                  max_it=6, precision=isira.ISIRA_FP64)
    z_or, its_or, _ = oracle.inner_solve(g.row_ptr, g.col_idx, st["trim_index"], 0.001, st["delta"], V, r, tau=1e-12,
                                         max_it=6)
    # six iterations in FP64: rounding is amplified by a few units each, so a thousand roundings bound the difference
    z = z.cpu().numpy()
    z_or = z_or - z_or.mean()
    assert its == its_or
    np.testing.assert_allclose(z, z_or, rtol=0, atol=1000 * 2.0 ** -53 * np.abs(z_or).max())
