"""The quadratic form where its persistent kernel cannot be had: a copy of the library whose query for resident
blocks fails (linked from the built objects with a fake of that call) must step through the launches, with
the same bits as the persistent kernel, and a second form must not take the memory again."""
import os
import subprocess
import sys

import pytest

from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
QUERY = "cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags"
FAKE = """#include <stddef.h>
int __wrap_%s(int *n, const void *f, int t, size_t s, unsigned g) { *n = 0; return 1; /* cudaErrorInvalidValue */ }
""" % QUERY

CALLER = """
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import scenegen
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import binding
binding.load_library(sys.argv[2])
sc = scenegen.make_scene("ring16", seed=2)
with fm.Problem(sc.R_init, sc.t_init, sc.cam_i, sc.cam_j, sc.pair_id, sc.x1, sc.x2) as p:
    p.irls_preaggregate(0.1)
    held = p.info()["device_bytes"]
    p.step_quadratic(11)
    p.preaggregate()
    p.step_quadratic(2)
    assert p.info()["device_bytes"] == held
    np.savez(sys.argv[3], *p.get_poses(), p.loss_grad()[1])
"""


def test_steps_without_the_persistent_kernel(tmp_path):
    import numpy as np
    build.build()
    (tmp_path / "fake.c").write_text(FAKE)
    subprocess.run(["gcc", "-O1", "-fPIC", "-c", str(tmp_path / "fake.c"), "-o", str(tmp_path / "fake.o")], check=True)
    objs = [os.path.join(build.BUILD_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    lib = str(tmp_path / "libfastmap_fake.so")
    subprocess.run([build._nvcc(), *build.ARCH, "-shared", "-Xlinker", "--wrap=" + QUERY, "-o", lib, *objs,
                    str(tmp_path / "fake.o")], check=True)
    out = []
    for k, path in enumerate((build.LIB, lib)):
        out.append(str(tmp_path / f"{k}.npz"))
        r = subprocess.run([sys.executable, "-c", CALLER, ROOT, path, out[-1]], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
    a, b = (np.load(f) for f in out)
    for k in a.files:
        np.testing.assert_array_equal(a[k], b[k])
