"""GPU: an FP32 image reads a cell's source with the cell's record up to 2^17 rays, after it beyond.
The middle column of an image with an odd width holds the same rays at every width, so images on
either side of that line have it alike, bit for bit."""
import numpy as np
import pytest

from paper_2512_01283_gb300 import build as B
from paper_2512_01283_gb300 import mcrt as M
from paper_2512_01283_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WIDTHS = [1, 1023, 1025]  # of 128 rows: 2^17 rays lie between the last two


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


@pytest.mark.parametrize("model", ["disk", "refined", "sphere", "absorbing"])
def test_images_on_both_sides_of_the_line_agree(model):
    mod = (W.disk(n=12) if model == "disk" else W.disk_refined(n=16, factor=2) if model == "refined" else
           W.rayleigh_sphere(n=12, tau=2.0) if model == "sphere" else W.dichroic_slab(n=12, emissivity=1.0))
    # one packet: its additions to a cell come in the same order for every camera
    run = W.center_source_run(1, pos=(0.1, 0.2, 0.3))
    cams = [W.camera((0.31, -0.42, 0.77), (w, 128), (2.1, 1.9)) for w in WIDTHS]
    m = M.Model(mod)
    M.launch(m, dict(run, cameras=cams), precision="fp32")
    cols = []
    for k, w in enumerate(WIDTHS):
        out = np.zeros((4, 128, w))
        m.image(k, out)
        cols.append(out[:, :, w // 2])
    m.close()
    assert np.abs(cols[0][:2]).max(axis=1).min() > 0
    for col in cols[1:]:
        assert np.array_equal(col, cols[0])
