"""Reading the parameters and the first call of the quadratic form while the host has no memory to give: they
need none, and no exception may leave the C boundary. The library is linked again from the built objects with
a fake of the C++ allocation that refuses what is above a limit, once one is set."""
import os
import subprocess
import sys

import pytest

from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = """
#include <new>
extern "C" {
void *__real__Znwm(unsigned long n);
__attribute__((visibility("default"))) unsigned long fake_new_limit = 0;
void *__wrap__Znwm(unsigned long n) {
    if (fake_new_limit && n > fake_new_limit) throw std::bad_alloc();
    return __real__Znwm(n);
}
}
"""

CALLER = """
import ctypes, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import scenegen
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import binding
lib = binding.load_library(sys.argv[2])
sc = scenegen.make_scene("ring16", seed=2)
with fm.Problem(sc.R_init, sc.t_init, sc.cam_i, sc.cam_j, sc.pair_id, sc.x1, sc.x2) as p:
    R, c = p.get_params()
    limit = ctypes.c_ulong.in_dll(lib, "fake_new_limit")
    limit.value = int(sys.argv[3])
    a = p.get_params()
    p.preaggregate()
    limit.value = 0
    np.testing.assert_array_equal(a[0], R)
    np.testing.assert_array_equal(a[1], c)
"""


@pytest.mark.parametrize("limit", [512, 16])   # 16 cameras: 1.5 KB of parameters; 16 bytes: a list of one pointer
def test_reading_without_host_memory(tmp_path, limit):
    build.build()
    (tmp_path / "fake.cc").write_text(FAKE)
    subprocess.run(["g++", "-O1", "-fPIC", "-c", str(tmp_path / "fake.cc"), "-o", str(tmp_path / "fake.o")], check=True)
    objs = [os.path.join(build.BUILD_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    lib = str(tmp_path / "libfastmap_fake.so")
    subprocess.run([build._nvcc(), *build.ARCH, "-shared", "-Xlinker", "--wrap=_Znwm", "-o", lib, *objs,
                    str(tmp_path / "fake.o")], check=True)
    r = subprocess.run([sys.executable, "-c", CALLER, ROOT, lib, str(limit)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
