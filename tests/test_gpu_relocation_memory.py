"""The second numbering of mesh-like graphs is an extra: where device memory for its copy runs out, create
goes on with the first numbering, with the same results.  Every allocation of the renumbering is refused
in turn (alloc_hook)."""
import numpy as np
import pytest

import synthgraphs as sg
from tests import alloc_hook
from tests.gpu_util import dev_graph, need_gpu, torch

pytestmark = pytest.mark.gpu

@pytest.fixture(scope="module")
def hooked(tmp_path_factory):
    need_gpu()
    import paper_1710_07080_gb300 as isira
    mp = pytest.MonkeyPatch()
    alloc_hook.install(isira, alloc_hook.build(tmp_path_factory.mktemp("alloc")), mp)
    yield isira
    mp.undo()


@pytest.mark.parametrize("weighted", [False, True])
def test_create_goes_on_without_memory_for_the_second_copy(hooked, weighted):
    isira, lib = hooked, hooked.lib
    g = sg.rgg(20011, 12.0, seed=3)
    rp, ci = dev_graph(g)
    w = torch.from_numpy(sg.edge_weights(g, 4)).cuda() if weighted else None
    x = torch.from_numpy(np.random.default_rng(1).standard_normal(g.n)).cuda()

    def make(refuse):
        lib.test_alloc_reset(refuse)
        s = isira.Solver(rp, ci, weights=w, precision=isira.ISIRA_FP64, precond=1)
        calls = lib.test_alloc_calls()
        lib.test_alloc_reset(-1)
        return s, calls

    s, total = make(-1)
    assert s.inner_route(0, isira.ISIRA_FP64)["renumbered"] == 1
    y = s.precond_apply(x)[0]
    s.close()
    # the renumbering's allocations: from the last three index arrays and a row pointer in a row to the end
    s, _ = make(-1)
    s.close()
    lib.test_alloc_reset(-1)
    with isira.Solver(rp, ci, weights=w, precision=isira.ISIRA_FP64, precond=1):
        sizes = [lib.test_alloc_size(i) for i in range(total)]
    idx, row = 4 * g.n, 8 * (g.n + 1)
    first = max(i for i in range(total - 3) if sizes[i:i + 4] == [idx, idx, idx, row])
    entries = [i for i in range(first, total) if sizes[i] >= 4 * g.nnz]
    assert len(entries) == (5 if weighted else 2)              # the CSR and the sliced copy, with the weights
    for refuse in range(first, total):
        s, _ = make(refuse)
        assert s.inner_route(0, isira.ISIRA_FP64)["renumbered"] == 0
        assert torch.equal(s.precond_apply(x)[0], y)
        s.close()
    with pytest.raises(isira.IsiraError) as e:                 # the first numbering itself cannot do without
        make(first - 1)
    assert e.value.status == isira.ISIRA_ERR_OOM
    lib.test_alloc_reset(-1)
