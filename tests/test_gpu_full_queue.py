"""GPU: segments that find no place in the record queue of the round-based paths.  The reserve
below the queue's end rules that out, so the library is built here with a queue of 512
slots and no reserve.  The network path tallies such segments with the tables, in place, and
counts them; the table rounds refuse the launch."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2512_01283_gb300 import build as B

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# one launch in a process of its own (a process holds one build of the library)
PROGRAM = """
import sys
import numpy as np
from paper_2512_01283_gb300 import mcrt as M
from paper_2512_01283_gb300 import workloads as W
library, optics, n_cam, out = sys.argv[1], sys.argv[2], int(sys.argv[3]), sys.argv[4]
M.LIB_PATH = library
# one size bin: the tables of a packet's size, which the network's tally takes, are the mixture's
model = dict(W.disk(n=12, tau_mid=20.0), optics=W.table_optics(n_bins=1))
run = dict(W.disk_run(1500, n_cam=8, npix=4), cameras=W.inclination_cameras(n_cam, 4))
m = M.Model(model)
if optics == "surrogate":
    s = M.Surrogate(m, seed=3)
    m.set_surrogate(s, -1.0)  # every evaluation from the tables
try:
    st = M.launch(m, run, optics=optics)
    S, A = m.tallies(n_cam)
    np.savez(out, S=S, A=A, overflow=st["tally_overflow"], scatterings=st["scatterings"], error="")
except Exception as e:
    np.savez(out, error=str(e))
"""


@pytest.fixture(scope="module")
def libraries(tmp_path_factory):
    """The library as built, and the one whose queue runs over."""
    B.build()
    d = tmp_path_factory.mktemp("queue")
    obj, lib = str(d / "mcrt_api.o"), str(d / "libmcrt.so")
    src = os.path.join(B.CSRC, "mcrt_api.cu")
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-DMCRT_REC_LIMIT=512", "-c", src, "-o", obj], check=True)
    others = [os.path.join(B.OUT_DIR, f.replace(".cu", ".o")) for f in B.SOURCES if f != "mcrt_api.cu"]
    subprocess.run([B._nvcc(), *B.ARCH, "-shared", "-o", lib, obj, *others, "-cudart", "static"], check=True)
    return B.LIB, lib, d


def launch(library, optics, n_cam, out):
    subprocess.run([sys.executable, "-c", PROGRAM, library, optics, str(n_cam), str(out)], check=True, cwd=ROOT,
                   timeout=300)
    return np.load(str(out) + ".npz")


# The same trajectories, every contribution within some 50 FP32 operations of 2^-24 each of the
# other kernel's: 3e-6 of the tally's norm, 1e-5 as for the in-place rows.
@pytest.mark.parametrize("n_cam", [1, 3, 16])
def test_network_path_tallies_what_finds_no_place(libraries, n_cam):
    whole, short, d = libraries
    a = launch(whole, "surrogate", n_cam, d / ("whole%d" % n_cam))
    b = launch(short, "surrogate", n_cam, d / ("short%d" % n_cam))
    assert a["error"] == "" and b["error"] == ""
    assert a["overflow"] == 0 and b["overflow"] > 0
    assert a["scatterings"] == b["scatterings"]
    assert np.linalg.norm(a["S"]) > 0
    assert np.linalg.norm(b["S"] - a["S"]) <= 1e-5 * np.linalg.norm(a["S"])
    assert np.linalg.norm(b["A"] - a["A"]) <= 1e-9 * np.linalg.norm(a["A"])


def test_table_rounds_refuse_a_queue_that_ran_over(libraries):
    whole, short, d = libraries
    assert launch(whole, "tables", 3, d / "wholet")["error"] == ""
    assert "tally queue overflow" in str(launch(short, "tables", 3, d / "shortt")["error"])
