"""GPU: the in-place source tally adds a warp's staged rows together (4 values per camera and
segment); camera counts around the widths at which the rows' split over the lanes changes,
in both precisions, against the FP64 oracle's tally."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2512_01283_gb300 import build as B
from paper_2512_01283_gb300 import mcrt as M
from paper_2512_01283_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    O.build()


def cameras(n):
    """Cameras off the grid axes."""
    out = []
    for k in range(n):
        a, i = 0.2 + 0.7 * k, 0.3 + 0.15 * k
        out.append(W.camera((np.sin(i) * np.cos(a), np.sin(i) * np.sin(a), np.cos(i)), (4, 4), (2.0, 2.0)))
    return out


# FP64: the two sides differ by summation order and by the operations' rounding (1e-9, the
# bound of the FP64 parity tests).  FP32: a contribution is some 50 FP32 operations, each within
# 2^-24 of its result, so 50 * 2^-24 = 3e-6 of the tally's norm, and one in 1e5 packets takes
# another path at a rounding (measured trace match 0.99999): 2000 packets, 1e-5.
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 1e-5)])
@pytest.mark.parametrize("n_cam", [1, 2, 3, 7, 8, 9, 16])
def test_in_place_rows_against_the_oracle(n_cam, precision, tol):
    model = W.rayleigh_sphere(n=8, tau=2.0)
    run = {"sources": [{"type": "point", "pos": (0.03, -0.02, 0.01), "luminosity": 1.0, "n_packets": 2000}],
           "cameras": cameras(n_cam), "seed": 11, "roulette_threshold": 1e-4, "roulette_survival": 0.1}
    m = M.Model(model)
    M.launch(m, run, precision=precision)
    S, A = m.tallies(n_cam)
    m.close()
    ref = O.transport(model, run)
    R = np.asarray(ref["S"]).reshape(S.shape)
    assert np.linalg.norm(R) > 0
    assert np.linalg.norm(S - R) <= tol * np.linalg.norm(R)
    # every camera and Stokes component lands in its own place
    for k in range(n_cam):
        assert np.linalg.norm(S[:, k, 0] - R[:, k, 0]) <= tol * np.linalg.norm(R[:, k, 0])
