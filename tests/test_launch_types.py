"""A kernel launched through a chain takes its arguments by implicit conversion: a pointer of another type
or without its const is a compile error, as in a plain launch."""
import os
import subprocess

import pytest

from paper_2012_12686_gb300 import build

SOURCE = """
#include "kernels.cuh"
__global__ void kernel(float2*, const double*, const int*, size_t) {}
cudaError_t call(adorym::Chain& s, float2* a, const float2* ca, double* b, int* c, int n) {
  return s.launch(kernel, 1, 32, 0, ARGS);
}
"""


@pytest.mark.parametrize("args,accepted", [
    ("a, b, c, n", True),                  # added const, int to size_t: what a plain launch accepts
    ("a, nullptr, nullptr, 3", True),
    ("b, a, c, n", False),                 # two pointers swapped
    ("a, c, b, n", False),
    ("ca, b, c, n", False),                # const taken away
    ("a, b, n, n", False),                 # an integer for a pointer
])
def test_argument_types(tmp_path, args, accepted):
    src = tmp_path / "launch.cu"
    src.write_text(SOURCE.replace("ARGS", args))
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, "-c", str(src), "-o",
                        str(tmp_path / "launch.o")], capture_output=True, text=True,
                       env=dict(os.environ, TMPDIR=str(tmp_path)))
    assert (r.returncode == 0) == accepted, r.stderr
