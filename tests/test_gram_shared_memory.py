"""The Gram kernel's shared memory at its highest deflation rank stays within the 48 KB that a launch may
take without opting in: an opt-in is a property of the function on one device, so a kernel that needs it
fails on a second device of the process.  The compiler states the static part."""
import re
import subprocess

from paper_1710_07080_gb300 import _build as b

UNIT = """
#include "inner_impl.cuh"
namespace isira {
template __global__ void k_gram<float>(InnerArgs<float>, double*, double*, double*, int);
template __global__ void k_gram<double>(InnerArgs<double>, double*, double*, double*, int);
}
"""


def test_gram_kernel_needs_no_shared_memory_opt_in(tmp_path):
    src = tmp_path / "gram.cu"
    src.write_text(UNIT)
    out = subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-Xptxas", "-v", "-I", b.CSRC, "-c", str(src), "-o",
                          str(tmp_path / "gram.o")], check=True, capture_output=True, text=True)
    text = out.stdout + out.stderr
    smem = [int(m.group(1)) for m in re.finditer(r"Compiling entry function '\w*k_gram\w*'.*?(\d+) bytes smem", text, re.S)]
    assert len(smem) == 2
    assert max(smem) + 8 * 31 * (128 + 1) <= 48 * 1024
