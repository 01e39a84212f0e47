"""Device memory that making a problem takes beside what the problem keeps: the keys in pair order (4 bytes a
point pair), the sort's two buffers (8 bytes) and its histograms (256 counters per 4,096 point pairs and the
scan's, under 0.3 bytes) for an input in any order, nothing for one in pair order. The library takes such
memory from the device's default pool, whose high-water mark the driver keeps."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu

USED_MEM_HIGH = 8   # CU_MEMPOOL_ATTR_USED_MEM_HIGH


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("shuffled", [False, True])
def test_scratch_of_a_new_problem(storage, shuffled):
    build.build()
    n, n_cams = 4_000_001, 9
    torch.zeros(1, device="cuda")
    cuda = ctypes.CDLL("libcuda.so.1")
    pool = ctypes.c_void_p()
    assert cuda.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0

    def high(reset=False):
        v = ctypes.c_uint64(0)
        f = cuda.cuMemPoolSetAttribute if reset else cuda.cuMemPoolGetAttribute
        assert f(pool, USED_MEM_HIGH, ctypes.byref(v)) == 0
        return v.value

    a = np.linspace(0.0, 1.0, n_cams)
    R = np.stack([np.array([[np.cos(x), 0, np.sin(x)], [0, 1, 0], [-np.sin(x), 0, np.cos(x)]]) for x in a])
    t = np.random.default_rng(0).normal(size=(n_cams, 3))
    ci = np.arange(n_cams - 1, dtype=np.int32)
    g = torch.Generator(device="cuda")
    g.manual_seed(0)
    pid = torch.arange(n, device="cuda") * (n_cams - 1) // n
    if shuffled:
        pid = pid[torch.randperm(n, generator=g, device="cuda")]
    pid = pid.to(torch.int32)
    x1, x2 = (torch.rand(n, 2, generator=g, device="cuda") - 0.5 for _ in range(2))
    torch.cuda.synchronize()
    high(reset=True)
    before = high()
    with fm.Problem(R, t, ci, ci + 1, pid, x1, x2, options=fm.default_options(storage=storage)) as p:
        took = high() - before
        assert p.info()["input_was_sorted"] == (0 if shuffled else 1)
    assert took <= (12.3 * n + 65536 if shuffled else 0)
    assert took >= (12 * n if shuffled else 0)   # the mark counts what the library takes
