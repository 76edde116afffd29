"""isira_apply_operator_noalloc after two calls raced on its scratch (which its contract forbids): the
racing calls' own results are lost, a later call that runs alone must be right.  A race can leave the
arrival counter of the reduction at any value, so the test sets one (in a copy of the translation unit
with an entry for it) instead of racing."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle
import synthgraphs as sg
from tests.gpu_util import dev_graph, need_gpu, orthonormal_columns, torch

pytestmark = pytest.mark.gpu

POKE = """
#include "noalloc.cu"
extern "C" __attribute__((visibility("default"))) int test_set_counter(unsigned v) {
    double* p = nullptr;
    if (na_scratch(&p) != cudaSuccess) return 1;
    return cudaMemcpy(p + kNaCounter, &v, sizeof(v), cudaMemcpyHostToDevice) == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def poked(tmp_path_factory):
    need_gpu()
    from paper_1710_07080_gb300 import _build as b
    d = tmp_path_factory.mktemp("noalloc")
    src, so = d / "poke.cu", d / "poke.so"
    src.write_text(POKE)
    subprocess.check_call([b._nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", "-cudart", "static", "-o", str(so),
                           str(src)])
    lib = C.CDLL(os.fspath(so))
    P, I, D, I64 = C.c_void_p, C.c_int, C.c_double, C.c_int64
    lib.isira_apply_operator_noalloc.argtypes = [I64, I64, P, P, I64, I, D, D, I, I, P, P, P, P]
    lib.test_set_counter.argtypes = [C.c_uint]
    return lib


@pytest.mark.parametrize("left", [1, 7, 1000])
@pytest.mark.parametrize("nx,ny", [(8, 9), (200, 181)])
def test_call_after_a_race_is_right(poked, nx, ny, left):
    import paper_1710_07080_gb300 as isira
    g = sg.grid2d(nx, ny)
    rp, ci = dev_graph(g)
    c, sigma, delta, trim = 3, 0.37, 8.0, 5
    rng = np.random.default_rng(left)
    V = orthonormal_columns(g.n, c, 4)
    Vc = torch.from_numpy(V).cuda().t().contiguous()
    assert poked.test_set_counter(left) == 0
    for call in range(3):
        x = rng.standard_normal(g.n)
        x[trim] = 0.0
        xt = torch.from_numpy(x).cuda()
        y = torch.full_like(xt, float("nan"))
        torch.cuda.synchronize()
        st = poked.isira_apply_operator_noalloc(g.n, g.nnz, rp.data_ptr(), ci.data_ptr(), trim, isira.ISIRA_FP64, sigma,
                                                delta, 0, c, Vc.data_ptr(), xt.data_ptr(), y.data_ptr(), None)
        assert st == isira.ISIRA_OK
        if call == 0:
            continue                                # its counter was not zero: lost, as after a race
        ref = np.insert(oracle.trimmed_apply(g.row_ptr, g.col_idx, trim, sigma, delta, V, np.delete(x, trim)), trim, 0.0)
        np.testing.assert_allclose(y.cpu().numpy(), ref, rtol=0, atol=1e-12 * np.abs(ref).max())
