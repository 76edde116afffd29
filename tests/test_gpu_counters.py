"""Counters of single inner solves driven from the host: the same call counts the same launches every time,
whatever the host had enqueued beyond the stop."""
import numpy as np
import pytest

import synthgraphs as sg
from tests.gpu_util import dev_graph, need_gpu, orthonormal_columns, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,precond", [("rmat12", 0), ("grid151x140", 1)])
def test_equal_calls_count_equally(name, precond):
    need_gpu()
    import paper_1710_07080_gb300 as isira
    g = sg.rmat(12) if name == "rmat12" else sg.grid2d(151, 140)
    rp, ci = dev_graph(g)
    r = np.random.default_rng(1).standard_normal(g.n)
    r = torch.from_numpy((r - r.mean()) / np.linalg.norm(r)).cuda()
    V = torch.from_numpy(orthonormal_columns(g.n, 3, 2)).cuda()
    with isira.Solver(rp, ci, precond=precond) as s:
        seen = set()
        for _ in range(8):
            a = s.stats()
            _, its, _ = s.inner_solve(r, sigma=0.001, V=V)
            b = s.stats()
            d = {f: b[f] - a[f] for f in ("spmv_launches", "kernel_launches", "inner_iters", "inner_solves")}
            assert d["spmv_launches"] == d["inner_iters"] == its > 0 and d["inner_solves"] == 1
            seen.add(d["kernel_launches"])
        assert len(seen) == 1
        if precond == 0:
            assert seen == {3 * its + 4}             # Gram matrix, start (two launches), result
