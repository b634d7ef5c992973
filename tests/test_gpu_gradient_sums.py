"""GPU: the sum over a batch's rows in the BF16 gradient, on batches of equal rows.  A row adds the
product of two BF16 numbers to a weight's gradient, 16 bits, and a tile of 16 or 32 equal rows
the same times a power of two: an FP32 sum of n tiles is exact up to n = 256 and in error by at
most n / 2 roundings of 2^-24 beyond.  The batch's mean has a power of two in place of its size,
so the gradient of 2^k equal rows is that of 16 of them.  A weight of the first layer takes two
products, of the input's high and low part, so its sums round from the first tile on."""
import numpy as np
import pytest

from test_gpu_surrogate import inputs, sur  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


# tiles in the longest FP32 sum: 4 sums up to 256 tiles (2048 rows: 128 tiles of 16 in 128 blocks; 8192: 256 of 32
# in 152, 38 blocks to a sum), 16 beyond (152 blocks: 10 in the fullest, of 14 tiles at 2^16 rows and 216 at 2^20)
@pytest.mark.parametrize("n,tiles", [(128, 8), (2048, 32), (8192, 76), (1 << 16, 140), (1 << 20, 2160)])
def test_equal_rows_give_the_gradient_of_sixteen(sur, n, tiles):  # noqa: F811
    s, _ = sur
    u = np.repeat(inputs(1), n, axis=0)
    t = np.repeat(np.linspace(-0.5, 0.5, 20, dtype=np.float32)[None, :], n, axis=0)
    many, few = s.grad(u, t)[1], s.grad(u[:16], t[:16])[1]
    for layer, (a, b) in enumerate(zip(many, few)):
        for which, (x, y) in enumerate(zip(a, b)):
            terms = 2 * tiles if layer == 0 and which == 0 else (0 if tiles <= 256 else tiles)
            # the longest sum's error; twice 2^-24 more where the first layer's sixteen rows round too
            bound = (terms / 2 + (2 if layer == 0 and which == 0 else 0)) * U
            # high and low part may differ in sign: the parts' sum is at most 1 + 2^-7 of the entry
            assert (np.abs(x.astype(np.float64) - y) <= 1.01 * bound * np.abs(y)).all(), (layer, which)
