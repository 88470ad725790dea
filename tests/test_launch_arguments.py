"""launch_chained checks a launch's arguments against the kernel's parameters when
it is compiled, as the <<< >>> syntax does: a pointer of another type, a dropped
const or an integer in a pointer's place is an error, not a cast."""
import os
import subprocess

import pytest

from helpers import ROOT
from paper_2608_10139_gb300 import build

SOURCE = """
#include <cstdint>
#include "common.cuh"
__global__ void k(const int64_t* in, int64_t n, int32_t* out) { if (n > 0) out[0] = static_cast<int32_t>(in[0]); }
cudaError_t launch(const int64_t* wide, int32_t* narrow, const int32_t* fixed, int n, cudaStream_t s) {
  return launch_chained(k, dim3(1), 32, 0, s, 1, %s);
}
"""


def _compiles(tmp_path, arguments):
    src = tmp_path / "launch.cu"
    src.write_text(SOURCE % arguments)
    cmd = [build.nvcc()] + build.ARCH + build.FLAGS + ["-c", str(src), "-o", os.devnull]
    return subprocess.run(cmd, capture_output=True, text=True, cwd=ROOT)


@pytest.mark.parametrize("arguments,ok", [("wide, n, narrow", True), ("nullptr, n, nullptr", True),
                                          ("narrow, n, narrow", False), ("wide, n, fixed", False),
                                          ("n, n, narrow", False), ("wide, n", False)])
def test_arguments_are_checked(tmp_path, arguments, ok):
    r = _compiles(tmp_path, arguments)
    assert (r.returncode == 0) == ok, r.stderr
    if not ok:
        assert "launch_chained" in r.stderr
