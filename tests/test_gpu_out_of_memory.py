"""Component calls that take buffers on first use: when device memory runs out at any of their allocations
the call says so, and the same call after it, with memory again, is right (nothing half built is used)."""
import numpy as np
import pytest

import synthgraphs as sg
from tests import alloc_hook
from tests.gpu_util import dev_graph, need_gpu, orthonormal_columns, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hooked(tmp_path_factory):
    need_gpu()
    import paper_1710_07080_gb300 as isira
    mp = pytest.MonkeyPatch()
    alloc_hook.install(isira, alloc_hook.build(tmp_path_factory.mktemp("alloc")), mp)
    yield isira
    mp.undo()


@pytest.mark.parametrize("entry", ["precond", "apply", "inner", "solve"])
def test_call_after_one_without_memory_is_right(hooked, entry):
    isira, lib = hooked, hooked.lib
    g = sg.rmat(11) if entry == "solve" else sg.grid2d(40, 37)
    rp, ci = dev_graph(g)
    rng = np.random.default_rng(1)
    x = torch.from_numpy(rng.standard_normal(g.n)).cuda()
    V = torch.from_numpy(orthonormal_columns(g.n, 3, 2)).cuda()
    u0 = torch.from_numpy(sg.start_vector(g.n, 1)).cuda()

    def call(s):                                   # FP32 on an FP64 handle: every buffer of the call is new
        if entry == "precond":
            return s.precond_apply(x.float())[0]
        if entry == "apply":
            return s.apply_operator(x.float(), 0.1, V)
        if entry == "inner":
            return s.inner_solve(x / x.norm(), V=V, max_it=20, precision=isira.ISIRA_MIXED)[0]
        s.solve(2, tol=1e-8, u0=u0)
        s.solve(5, tol=1e-8, u0=u0)                # larger buffers for the deflation vectors
        return s.eigpairs()[0]

    lib.test_alloc_reset(-1)
    with isira.Solver(rp, ci, precision=isira.ISIRA_FP64, precond=0) as s:
        lib.test_alloc_reset(-1)
        want = call(s)
        calls = lib.test_alloc_calls()
    assert calls > 0
    for refuse in range(calls):
        with isira.Solver(rp, ci, precision=isira.ISIRA_FP64, precond=0) as s:
            lib.test_alloc_reset(refuse)
            with pytest.raises(isira.IsiraError) as e:
                call(s)
            assert e.value.status == isira.ISIRA_ERR_OOM
            lib.test_alloc_reset(-1)
            assert torch.equal(call(s), want)
