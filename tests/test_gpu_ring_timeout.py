"""A wait of the FP16 ring kernel that runs out is reported on every tank whose
cells it may have left unstepped.  The library is built once more with ring
waits that all give up at once; one step of it then has to end with
LBM_FS_ETIMEOUT on each tank of a batch, and on a single tank."""
import os
import subprocess
import sys

import pytest

from paper_1201_0351_gb300 import build

pytestmark = pytest.mark.gpu

CHILD = """
import sys
from paper_1201_0351_gb300 import build, inputs as I, lbm_fs
build.build = lambda *a, **k: sys.argv[1]

def tank(n):
    flags, fill, rho = I.hydrostatic_tank(n, n, n, lambda X, Y: 0.6 * n + 0.4, 1e-5, 1.0, 0)
    return I.Scenario("t", n, n, n, 0, 0.7, (0.0, 0.0, -1e-5), (0.0, 0.0, 0.0), 1.0, 1e-2, flags, fill, rho, [], 0)

def code(t):
    try:
        t.sync()
    except lbm_fs.LbmFsError as e:
        return e.code
    return 0

sim = lbm_fs.Simulation(tank(24), storage="f16s")
sim.step(1)
assert code(sim) == lbm_fs.LBM_FS_ETIMEOUT, code(sim)
bt = lbm_fs.Batch([tank(n) for n in (24, 40, 17, 64)], storage="f16s")
bt.step(1)
codes = [code(t) for t in bt.tanks]
assert codes == [lbm_fs.LBM_FS_ETIMEOUT] * 4, codes
# (the double storage has no such waits)
sim = lbm_fs.Simulation(tank(16), storage="f64")
sim.step(1)
assert code(sim) == 0
print("reported")
"""


def _variant(out_dir):
    """the library with the FP16 unit's ring waits giving up at once"""
    build.build()
    obj = os.path.join(out_dir, "kernels_f16s.o")
    lib = os.path.join(out_dir, "libgb300_lbmfs.so")
    src = os.path.join(build.CSRC, "kernels_f16s.cu")
    subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, "-DLBMFS_RING_POLLS=0", "-c", src, "-o", obj], check=True)
    rest = [os.path.join(build.OUT_DIR, u.replace(".cu", ".o")) for u in build.UNITS if u != "kernels_f16s.cu"]
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-o", lib, obj, *rest], check=True)
    return lib


def test_every_tank_reports_a_ring_wait_that_runs_out(tmp_path):
    lib = _variant(str(tmp_path))
    r = subprocess.run([sys.executable, "-c", CHILD, lib], cwd=build.ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "reported" in r.stdout, r.stdout + r.stderr
