"""A launch that the runtime refuses (more threads than a block may have) is reported once, by the launch helper's
return value, and does not stay behind as the calling thread's last error, which the host program's next check would find."""
import subprocess

import pytest

from paper_2509_24014_b200 import build

pytestmark = pytest.mark.gpu   # (without a device every error check fails)

SOURCE = """
#include <cstdio>
#include "internal.h"
__global__ void nothing(int) {}
int main() {
  cudaGetLastError();
  const cudaError_t e = sparsed::launch_overlapped(nothing, 1, %d, 4096, 0, nullptr, 1);
  std::printf("%%d %%d\\n", static_cast<int>(e), static_cast<int>(cudaPeekAtLastError()));
}
"""


def test_a_refused_launch_leaves_no_error_behind(tmp_path):
    for resident in (0, 2):   # launched as usual; allowed to overlap
        src, exe = tmp_path / f"refused{resident}.cu", tmp_path / f"refused{resident}"
        src.write_text(SOURCE % resident)
        subprocess.run([build._nvcc(), *build.ARCH_FLAGS, "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)],
                       check=True, capture_output=True, timeout=300)
        out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout.split()
        assert int(out[0]) != 0 and int(out[1]) == 0, out
