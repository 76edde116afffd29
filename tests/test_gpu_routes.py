"""Which path an inner solve takes (isira_inner_route), on both sides of every line: the row limits, the
lines that the gathers touch, long rows, the CTA count's steps, gathers from a staged copy, and the second
numbering of mesh-like graphs.  The tests that compare the paths' results rely on these."""
import pytest

import synthgraphs as sg
from tests.gpu_util import dev_graph, need_gpu

pytestmark = pytest.mark.gpu


def route(g, prec, c=0, **opts):
    need_gpu()
    import paper_1710_07080_gb300 as isira
    rp, ci = dev_graph(g)
    P = isira.ISIRA_FP64 if prec == "fp64" else isira.ISIRA_MIXED
    with isira.Solver(rp, ci, precision=P, **{"precond": 0, **opts}) as s:
        return s.inner_route(c, P)


@pytest.mark.parametrize("prec,n,ctas", [("mixed", 256, 1), ("mixed", 257, 2), ("mixed", 2049, 16), ("mixed", 80000, 16),
                                         ("mixed", 80001, 0), ("fp64", 64, 1), ("fp64", 65, 2), ("fp64", 513, 16),
                                         ("fp64", 30720, 16), ("fp64", 30721, 0)])
def test_row_limits_and_cta_counts(prec, n, ctas):
    assert route(sg.cycle(n), prec)["one_launch_ctas"] == ctas


@pytest.mark.parametrize("make,prec,ctas,staged", [
    (lambda: sg.erdos_renyi(12347, 8.0, seed=1), "mixed", 16, 1),     # more lines than the copy moves
    (lambda: sg.erdos_renyi(17000, 8.0, seed=5), "mixed", 16, 1),
    (lambda: sg.grid2d(112, 88), "mixed", 16, 0),                     # fewer
    (lambda: sg.erdos_renyi(12347, 8.0, seed=1), "fp64", 16, 0),
    (lambda: sg.watts_strogatz(79999, 10, 0.1, seed=6), "mixed", 16, 0),
    (lambda: sg.erdos_renyi(60000, 8.0, seed=5), "mixed", 0, 0),      # too many lines for 16 SMs
    (lambda: sg.rmat(12), "mixed", 0, 0),                             # rows above 64 neighbours
])
def test_lines_and_long_rows(make, prec, ctas, staged):
    r = route(make(), prec)
    assert (r["one_launch_ctas"], r["staged"]) == (ctas, staged)


@pytest.mark.parametrize("make,prec,ranks", [
    (lambda: sg.grid2d(63, 63), "fp64", {0: 16, 8: 16, 31: 16}),
    (lambda: sg.grid2d(126, 126), "fp64", {0: 16, 16: 16, 31: 16}),
    (lambda: sg.grid2d(173, 173), "fp64", {0: 16, 4: 16, 12: 0, 31: 0}),      # 16 SMs against 152 from here on
    (lambda: sg.erdos_renyi(30000, 8.0, seed=5), "fp64", {0: 16, 2: 16, 10: 0, 31: 0}),
    (lambda: sg.watts_strogatz(30000, 20, 0.1, seed=5), "fp64", {0: 0, 8: 0, 31: 0}),
    (lambda: sg.grid2d(279, 279), "mixed", {0: 16, 31: 16}),
    (lambda: sg.watts_strogatz(68000, 10, 0.1, seed=6), "mixed", {0: 16, 31: 16}),
    (lambda: sg.watts_strogatz(79999, 10, 0.1, seed=6), "mixed", {0: 16, 8: 16, 9: 0, 31: 0}),   # little L1 left
])
def test_ranks_at_which_one_launch_pays(make, prec, ranks):
    g = make()
    for c, ctas in ranks.items():
        assert route(g, prec, c)["one_launch_ctas"] == ctas, c


@pytest.mark.parametrize("opts", [{"inner_graph": 0}, {"precond": 1}, {"reorder": 0}, {"sell": 0}])
def test_options_that_keep_launches_per_iteration(opts):
    assert route(sg.grid2d(40, 37), "mixed", **opts)["one_launch_ctas"] == 0


@pytest.mark.parametrize("make,opts,renumbered", [
    (lambda: sg.rgg(20011, 12.0, seed=3), {"precond": 1, "trim_index": 5}, 1),
    (lambda: sg.rgg(90001, 12.0, seed=3), {"precond": 1}, 1),
    (lambda: sg.rgg(20011, 12.0, seed=3), {"precond": 0}, 0),
    (lambda: sg.rgg(20011, 12.0, seed=3), {"precond": 1, "reorder": 0}, 0),
    (lambda: sg.grid2d(151, 140), {"precond": 1}, 0),
])
def test_second_numbering(make, opts, renumbered):
    assert route(make(), "mixed", **opts)["renumbered"] == renumbered


def test_arguments():
    need_gpu()
    import paper_1710_07080_gb300 as isira
    rp, ci = dev_graph(sg.path(5))
    with isira.Solver(rp, ci) as s:
        for c, prec in ((-1, 1), (32, 1), (0, 2)):
            with pytest.raises(isira.IsiraError) as e:
                s.inner_route(c, prec)
            assert e.value.status == isira.ISIRA_ERR_INVALID_ARG
