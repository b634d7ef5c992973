"""GPU: prepared tables of the smallest, odd and largest numbers of bins and angles (blocks of
256 threads, 32 lanes of bins): every packet of an FP64 run ends as the FP64 oracle's does."""
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


# Without a field all of a packet's arithmetic is FP64 on both sides: 1e-9, as for the other
# FP64 traces.  Thermal packets carry the luminosity that the mean of alpha1 gives.
@pytest.mark.parametrize("n_bins,n_theta,n_ktheta", [(1, 2, 2), (3, 256, 257), (5, 258, 31), (32, 721, 721)])
def test_tables_of_any_size(n_bins, n_theta, n_ktheta):
    model = dict(W.disk(n=8, tau_mid=3.0), bfield=None)
    tabs, w, _ = W.synthetic_bins(n_bins, n_theta)
    model["optics"] = {"model": "table", "mueller": tabs, "bin_weight": w, "kext": W.kext_dipole(0.3, n=n_ktheta)}
    run = dict(W.disk_run(600, n_cam=1, npix=4))
    ref = O.transport(model, dict(run, n_trace=600))["trace"]
    m = M.Model(model)
    got = np.zeros((600, 16))
    M.launch(m, run, precision="fp64", trace=got, n_trace=600)
    m.close()
    assert np.array_equal(got[:, 12], ref[:, 12])
    assert np.all(np.abs(got[:, :4] - ref[:, :4]) <= 1e-9 * ref[:, :1])
