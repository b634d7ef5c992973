"""GPU: the source and absorbed tallies of the FP32 kernels for isotropic extinction, table rounds
and in place, against the general kernels' (a packet's trace, which test_gpu_isotropic.py
compares, holds no path integral)."""
import numpy as np
import pytest

from paper_2512_01283_gb300 import workloads as W
from test_gpu_isotropic import built, run  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


# A packet whose trace agrees to 1e-4 adds along the same path with Stokes vectors that agree as
# well; one that went another way adds up to ten times the mean packet's share, on both sides.
@pytest.mark.parametrize("kind", ["sphere", "disk", "refined"])
@pytest.mark.parametrize("inline", [False, True])
def test_isotropic_tallies_match_the_general_ones(kind, inline):
    model = (W.rayleigh_sphere(n=12, tau=3.0) if kind == "sphere" else
             W.disk(n=16, tau_mid=30.0) if kind == "disk" else W.disk_refined(n=16, factor=2, tau_mid=30.0))
    a, Sa, Aa = run(model, 0.0, "fp32", inline)
    b, Sb, Ab = run(model, 1e-30, "fp32", inline)
    scale = np.abs(b[:, :1]) + 1e-300
    other = 1.0 - ((a[:, 12] == b[:, 12]) & (np.abs(a[:, :4] - b[:, :4]) <= 1e-4 * scale).all(axis=1)).mean()
    assert other <= 1e-3
    bound = 1e-4 + 20.0 * other
    for k in range(Sa.shape[1]):
        assert np.abs(Sb[:, k]).sum() > 0
        assert np.abs(Sa[:, k] - Sb[:, k]).sum() <= bound * np.abs(Sb[:, k]).sum()
    assert np.abs(Aa - Ab).sum() <= (1e-25 if kind == "sphere" else bound * np.abs(Ab).sum())
