"""The library's own functions of one float against 64-bit values, compiled here from its header."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_20225_b200", "csrc")
SOURCE = """
#include "rdf_math.cuh"
__global__ void kernel(const float* x, float* y, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = tanh_select(x[i]);
}
extern "C" int run(const float* x, float* y, int n, void* stream) {
    kernel<<<296, 256, 0, (cudaStream_t)stream>>>(x, y, n);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("math")
    (d / "t.cu").write_text(SOURCE)
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
                    "-shared", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cu")], check=True, capture_output=True)
    fn = ctypes.CDLL(str(d / "t.so")).run
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]

    def call(x):
        y = torch.empty_like(x)
        assert fn(x.data_ptr(), y.data_ptr(), x.numel(), torch.cuda.current_stream().cuda_stream) == 0
        return y
    return call


def test_tanh_select_over_its_range(run):
    """Every 97th float from the smallest normal one to 64 (both branches, the saturated end) and all of them around the
    switch at 0.55.  The quotient is within 2 units in the last place, the exponential within 2, and above 0.55 the
    difference from 1 makes at most twice that of them: 4 units of 2^-24 on a value of at least 0.5, 4.8e-7."""
    bits = np.concatenate([np.arange(0x00800000, 0x42800000, 97), np.arange(0x3F0CCCCD - 20000, 0x3F0CCCCD + 20000)]).astype(np.int32)
    x = torch.from_numpy(bits).cuda().view(torch.float32)
    for s in (x, -x):
        want = torch.tanh(s.double())
        err = ((run(s).double() - want).abs() / want.abs()).max().item()
        print("tanh_select: largest relative error", err, "tanhf", ((torch.tanh(s).double() - want).abs() / want.abs()).max().item())
        assert err <= 4.8e-7


def test_tanh_select_special_values(run):
    x = torch.tensor([0.0, -0.0, float("inf"), -float("inf"), 1e38, -1e38, 88.8, 44.5, float("nan"), 1e-45], device="cuda")
    y = run(x)
    assert torch.equal(y[:8], torch.tensor([0.0, -0.0, 1.0, -1.0, 1.0, -1.0, 1.0, 1.0], device="cuda"))
    assert torch.isnan(y[8]) and 0.0 <= y[9] <= 1e-44
    assert bool(torch.signbit(y[1])) and not bool(torch.signbit(y[0]))
