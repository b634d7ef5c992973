"""GPU: a ray's result is the same however many lanes of a warp share it.  The middle column of
an image with an odd width holds the same rays at every width, so images on either side of the
lines between 8, 4 and 1 lanes per ray have it alike, bit for bit."""
import numpy as np
import pytest

from paper_2512_01283_gb300 import build as B
from paper_2512_01283_gb300 import mcrt as M
from paper_2512_01283_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# 128 rows each: one column; FP64 on either side of 2048 and 8192 rays; FP32 of 12288 and 40960
WIDTHS = [1, 15, 17, 63, 65, 95, 97, 319, 321]


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("model", ["disk", "refined", "dipole"])
def test_a_ray_does_not_depend_on_the_lanes_that_share_it(precision, model):
    mod = (W.disk(n=12) if model == "disk" else
           W.disk_refined(n=16, factor=2) if model == "refined" else W.spheroid_sphere(n=16))
    if model == "dipole":
        mod["emissivity"] = np.ones_like(mod["kappa_abs"])
    # one packet: its additions to a cell come in the same order for every camera
    run = W.center_source_run(1, pos=(0.1, 0.0, 0.0))
    cams = [W.camera((0.31, -0.42, 0.77), (w, 128), (2.1, 1.9)) for w in WIDTHS]
    m = M.Model(mod)
    M.launch(m, dict(run, cameras=cams), precision=precision)
    cols = []
    for k, w in enumerate(WIDTHS):
        out = np.zeros((4, 128, w))
        m.image(k, out)
        cols.append(out[:, :, w // 2])
    m.close()
    assert np.abs(cols[0][:2]).max(axis=1).min() > 0
    for w, col in zip(WIDTHS[1:], cols[1:]):
        assert np.array_equal(col, cols[0]), w
