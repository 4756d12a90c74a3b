"""The columns' 1 / sqrt(q) (Markstein's corrections of the hardware's
approximation) against CUDA's 1.0f / sqrtf(q), for every float from 1 to 2^30,
which q = |d|^2 in mm^2 is: no result off by more than its last bit, and no more
than 60 of the 251,658,241 off by that (as the comment beside it says), so that
P^T's step vectors are P's."""
import ctypes as C
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = r"""
#include "pcas_internal.cuh"
__global__ void k_compare(unsigned lo, unsigned hi, unsigned long long* out) {
    unsigned long long off = 0, far = 0;
    for (unsigned long long b = lo + 2ull * (blockIdx.x * blockDim.x + threadIdx.x); b <= hi;
         b += 2ull * gridDim.x * blockDim.x) {
        const unsigned b1 = b + 1 <= hi ? (unsigned)b + 1 : (unsigned)b;
        const float2 q = make_float2(__uint_as_float((unsigned)b), __uint_as_float(b1));
        const float2 r = pcas::inv_sqrt2(q);
        const int d[2] = {__float_as_int(r.x) - __float_as_int(1.0f / sqrtf(q.x)),
                          b1 != (unsigned)b ? __float_as_int(r.y) - __float_as_int(1.0f / sqrtf(q.y)) : 0};
        for (int e = 0; e < 2; e++) {
            off += d[e] != 0;
            far += d[e] > 1 || d[e] < -1;
        }
    }
    atomicAdd(out, off);
    atomicAdd(out + 1, far);
}
extern "C" int compare(unsigned lo, unsigned hi, unsigned long long* out) {
    k_compare<<<1216, 256>>>(lo, hi, out);
    return (int)cudaDeviceSynchronize();
}
"""


def test_every_float(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1102_1712_gb300 import build as B
    src, so = tmp_path / "compare.cu", tmp_path / "compare.so"
    src.write_text(SOURCE)
    subprocess.check_call([B.nvcc(), *B.CFLAGS, "-I", B.CSRC, "-shared", "-o", os.fspath(so), os.fspath(src)])
    L = C.CDLL(os.fspath(so))
    out = torch.zeros(2, dtype=torch.int64, device="cuda")
    assert L.compare(C.c_uint(0x3f800000), C.c_uint(0x4e800000), C.c_void_p(out.data_ptr())) == 0
    off, far = out.tolist()
    assert far == 0 and off <= 60, (off, far)
