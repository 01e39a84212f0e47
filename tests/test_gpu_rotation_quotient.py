"""The quotients of the rotation kernels by a shared reciprocal are those of the division, bit for bit: random
mantissas over exponents of -400 to 400, and every pair of edge mantissas (powers of two, their neighbours,
all ones, halfway patterns) with both signs. The kernel's own function is compiled from its source."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = """
#include "fm_rotation.cu"
void fm_internal_set_error(const char *) {}
__global__ void k_compare(const double *a, const double *b, double *q, double *d, long long n) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    q[i] = quotient(a[i], b[i], 1.0 / b[i]);
    d[i] = __ddiv_rn(a[i], b[i]);
}
extern "C" __attribute__((visibility("default"))) int compare(const double *a, const double *b, double *q, double *d, long long n) {
    k_compare<<<(unsigned)((n + 255) / 256), 256>>>(a, b, q, d, n);
    return (int)cudaDeviceSynchronize();
}
"""


def _operands():
    rng = np.random.default_rng(0)
    n = 1 << 22
    def mant(k):
        return 1.0 + rng.integers(0, 1 << 52, k) * 2.0 ** -52
    a = np.ldexp(mant(n), rng.integers(-400, 401, n)) * rng.choice([-1.0, 1.0], n)
    b = np.ldexp(mant(n), rng.integers(-400, 401, n))
    bits = [0, 1, 2, (1 << 52) - 1, (1 << 52) - 2, 1 << 51, (1 << 51) - 1, (1 << 51) + 1, 1 << 26, (1 << 26) - 1, (1 << 26) + 1,
            0x5555555555555, 0xAAAAAAAAAAAAA, 0x5555555555556]
    bits += [int(v) for v in rng.integers(0, 1 << 52, 50)]
    edge = np.array([1.0 + v * 2.0 ** -52 for v in bits])
    edge = np.concatenate([np.ldexp(edge, e) for e in (-300, -1, 0, 1, 300)])
    ea, eb = (v.ravel() for v in np.meshgrid(np.concatenate([edge, -edge, [0.0]]), edge))
    # quotients close to halfway between two doubles: a = b q rounded, for random q
    q = mant(n)
    return np.concatenate([a, ea, b * q]), np.concatenate([b, eb, b])


def test_quotient_rounds_like_the_division(tmp_path):
    src, lib = tmp_path / "q.cu", str(tmp_path / "q.so")
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", "-o", lib, str(src)], check=True)
    a, b = (torch.from_numpy(v).cuda() for v in _operands())
    q, d = torch.empty_like(a), torch.empty_like(a)
    torch.cuda.synchronize()
    fn = ctypes.CDLL(lib).compare
    fn.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_longlong]
    assert fn(a.data_ptr(), b.data_ptr(), q.data_ptr(), d.data_ptr(), a.numel()) == 0
    assert torch.isfinite(d).all() and torch.equal(q, d)
