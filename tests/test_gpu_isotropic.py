"""GPU: the kernels for isotropic extinction against the general ones, which take over when the
extinction table holds a dichroism, here of 1e-30 (the sphere, which absorbs nothing, absorbs
that much of the light's polarization)."""
import numpy as np
import pytest

from paper_2512_01283_gb300 import build as B
from paper_2512_01283_gb300 import mcrt as M
from paper_2512_01283_gb300 import workloads as W

pytestmark = pytest.mark.gpu
N = 4000


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def run(model, alpha2, precision, inline):
    model = dict(model, optics=dict(model["optics"], kext=W.kext_constant(alpha2)))
    r = dict(W.disk_run(N, n_cam=3, npix=8))
    r["sources"] = r["sources"][:1] if model["emissivity"] is None else r["sources"]
    n = sum(s["n_packets"] for s in r["sources"])
    m = M.Model(model)
    trace = np.zeros((n, 16))
    M.launch(m, r, precision=precision, trace=trace, n_trace=n, inline_tally=inline)
    S, A = m.tallies(3)
    m.close()
    return trace, S, A


# FP64: the general kernels turn Q and U into the grain frame and back, a few roundings per
# segment, 1e-9 as for the traces against the oracle; FP32: 1e-4 for 99.9 % of the packets, as there.
@pytest.mark.parametrize("precision,tol,share", [("fp64", 1e-9, 1.0), ("fp32", 1e-4, 0.999)])
@pytest.mark.parametrize("kind,inline", [("sphere", False), ("disk", False), ("disk", True), ("refined", False),
                                         ("refined", True)])
def test_isotropic_kernels_match_the_general_ones(kind, inline, precision, tol, share):
    model = (W.rayleigh_sphere(n=12, tau=3.0) if kind == "sphere" else
             W.disk(n=16, tau_mid=30.0) if kind == "disk" else W.disk_refined(n=16, factor=2, tau_mid=30.0))
    a, Sa, Aa = run(model, 0.0, precision, inline)
    b, Sb, Ab = run(model, 1e-30, precision, inline)
    scale = np.abs(b[:, :1]) + 1e-300
    same = (a[:, 12] == b[:, 12]) & (np.abs(a[:, :4] - b[:, :4]) <= tol * scale).all(axis=1)
    assert same.mean() >= share
    if share == 1.0:
        assert np.linalg.norm(Sa - Sb) <= tol * np.linalg.norm(Sb)
        assert np.linalg.norm(Aa - Ab) <= (1e-28 if kind == "sphere" else tol * np.linalg.norm(Ab))
