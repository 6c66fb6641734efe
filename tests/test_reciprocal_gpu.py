"""The reciprocal of the weight schedule (recip in csrc/gka_common.cuh) against the quotient in 64 bits, over every fp32 number of
the range that it is used on."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2511_21016_b200 import build

pytestmark = pytest.mark.gpu

SOURCE = """
#include "gka_common.cuh"
__global__ void recip_kernel(float *y, unsigned first, unsigned n) {
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = gka::recip(__uint_as_float(first + i));
}
extern "C" int recip_all(float *y, unsigned first, unsigned n) {
    recip_kernel<<<(n + 255) / 256, 256>>>(y, first, n);
    return (int)cudaDeviceSynchronize();
}
"""


def test_reciprocal_is_within_one_unit_in_the_last_place(tmp_path):
    src, lib = tmp_path / "recip.cu", tmp_path / "recip.so"
    src.write_text(SOURCE)
    flags = [f for f in build.NVCC_FLAGS if f not in ("-Xptxas", "-v")]
    subprocess.check_call([build._nvcc(), *flags, "-I", build.CSRC, "-shared", str(src), "-o", str(lib)])
    first, last = (int(np.float32(v).view(np.uint32)) for v in (2.0, 4.0))
    n = last - first + 1
    y = torch.zeros(n, device="cuda")
    torch.cuda.synchronize()
    fn = ctypes.CDLL(os.fspath(lib)).recip_all
    fn.argtypes = [ctypes.c_void_p, ctypes.c_uint, ctypes.c_uint]
    assert fn(y.data_ptr(), first, n) == 0
    got = y.cpu().numpy()
    exact = 1.0 / np.arange(first, last + 1, dtype=np.uint32).view(np.float32).astype(np.float64)
    ulps = np.abs(got.astype(np.float64) - exact) / np.spacing(exact.astype(np.float32)).astype(np.float64)
    # 1/2 unit from the last rounding, and the step's own error (relative 2^-46: 2^-22 units) on top; a neighbouring power of two
    # halves the unit on one side, hence the bound that the function states
    print("reciprocal: largest error %.4f units in the last place" % ulps.max())
    assert ulps.max() <= 1.0
