"""The ring of cached normals when a wait for its copies gives up: the pass
reports SDPD_E_TIMEOUT, waits for what is on its way and leaves, and the
process goes on computing.  The library is linked once more with the pair
passes built so that every such wait gives up at once (the copies themselves
arrive as always), and run in a process of its own."""
import os
import subprocess
import sys

import pytest

from paper_2002_03120_gb300 import build

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu

RUN = """
import sys
import numpy as np
from paper_2002_03120_gb300 import binding as B, build, cases
build.LIB = sys.argv[1]
case = cases.poiseuille_si(nx=12, ny=25, nz=12)
sim = B.Sim(case, precision=B.SDPD_PREC_SPLIT)
sim.set_force_mode(0)
try:
    sim.step(2)
except B.SdpdError as e:
    assert e.code == 7, e                      # SDPD_E_TIMEOUT
else:
    raise AssertionError("no timeout reported")
sim.close()
sim = B.Sim(case, precision=B.SDPD_PREC_SPLIT)
sim.set_force_mode(0)
sim.set_noise_cache(0)                         # no ring on this path
sim.step(2)
assert np.isfinite(sim.state()["F"]).all()
sim.close()
print("done")
"""


def test_a_wait_that_gives_up_is_reported(tmp_path):
    need_gpu()
    build.build()
    obj, lib = str(tmp_path / "k_pairs.o"), str(tmp_path / "libsdpd_no_tries.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-DRING_TRIES=0", "-c",
                    os.path.join(build.CSRC, "k_pairs.cu"), "-o", obj], check=True)
    others = [os.path.join(build.OUT, s.replace(".cu", ".o")) for s in build.SOURCES if s != "k_pairs.cu"]
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-o", lib, obj, *others], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RUN, lib], cwd=root, capture_output=True, text=True, timeout=120,
                       env={**os.environ, "PYTHONPATH": root})
    assert r.returncode == 0 and r.stdout.strip() == "done", r.stdout + r.stderr
