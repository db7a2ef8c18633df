"""The exponential that the selection from Q and K takes off the exponential unit (exp2_by_polynomial in scoring.cu),
against 2^x in 64 bits: its stated error over every f it reduces to, at exponents from end to end, and the values that the
scores' -inf, inf and NaN depend on."""
import ctypes
import math
import os
import subprocess

import pytest
import torch

from paper_2509_24014_b200 import build

pytestmark = pytest.mark.gpu
# Running error bound of the six fmas (half a unit of each sum, half a unit of each coefficient, both times the powers of
# |f| that follow): 8.52e-8 of the result at f = -1/2, where it is largest; and 1.9e-9 for the polynomial itself.
BOUND = 8.52e-8 + 1.9e-9


@pytest.fixture(scope="module")
def exp2(tmp_path_factory):
    folder = tmp_path_factory.mktemp("exp2")
    src, lib = folder / "exp2.cu", folder / "exp2.so"
    src.write_text('#include "scoring.cu"\n'
                   "__global__ void evaluate(const float2* x, float2* y, int n) {\n"
                   "  const int i = blockIdx.x * blockDim.x + threadIdx.x;\n"
                   "  if (i < n) y[i] = sparsed::exp2_by_polynomial(x[i]);\n}\n"
                   'extern "C" int run(const float* x, float* y, int pairs, void* stream) {\n'
                   "  evaluate<<<(pairs + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(\n"
                   "      reinterpret_cast<const float2*>(x), reinterpret_cast<float2*>(y), pairs);\n"
                   "  return cudaGetLastError();\n}\n")
    subprocess.run(["nvcc", *build.ARCH_FLAGS, *build.COMMON_FLAGS, "-shared", "-I", build.CSRC, str(src), "-o", str(lib)],
                   check=True, capture_output=True, timeout=600)
    run = ctypes.CDLL(str(lib)).run
    run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]

    def evaluate(x):
        assert x.dtype == torch.float32 and x.is_contiguous() and x.numel() % 2 == 0
        y = torch.full_like(x, float("nan"))
        assert run(x.data_ptr(), y.data_ptr(), x.numel() // 2, torch.cuda.current_stream().cuda_stream) == 0
        return y

    return evaluate


@pytest.mark.parametrize("n", [-126, -125, -61, -1, 0, 1, 64, 126])
def test_error_bound(exp2, n):
    x = (torch.arange(-(1 << 23), (1 << 23) + 2, device="cuda") * 2.0 ** -24).float() + n   # [n - 1/2, n + 1/2]
    x = x[(x >= n - 0.5) & (x <= n + 0.5) & (x >= -126.0)]   # (normal results)
    x = x[: x.numel() // 2 * 2].contiguous()
    ref = torch.exp2(x.double())
    assert ((exp2(x).double() - ref).abs() <= BOUND * ref).all()


def test_ends_of_the_range(exp2):
    inf, nan = math.inf, math.nan
    x = torch.tensor([-inf, -1e30, -200.0, -127.0, 128.0, 200.0, 1e30, inf, nan, -nan, 0.0, -0.0], device="cuda")
    y = exp2(x).tolist()
    assert y[:4] == [0.0] * 4 and y[4:8] == [inf] * 4 and math.isnan(y[8]) and math.isnan(y[9]) and y[10:] == [1.0, 1.0]
    x = torch.tensor([-126.75, -126.5, -126.25, 127.25], device="cuda")   # no normal results: 0, denormal ones
    y = exp2(x).tolist()
    assert y[0] == 0.0 and all(abs(a - 2.0 ** b) <= 2.0 ** -149 for a, b in zip(y[1:3], (-126.5, -126.25)))
    assert abs(y[3] / 2.0 ** 127.25 - 1.0) <= BOUND
