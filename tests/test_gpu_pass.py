"""GPU: the gradient kernel at the edges of its tiles of 16 and 32 rows (one row, ragged last
tiles, the last batch of a tile per SM of 152 and the first beyond, more tiles than SMs) against
the FP64 passes with the same BF16 storage points."""
import numpy as np
import pytest

from test_gpu_surrogate import bf16_passes_reference, inputs, sur  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


# What is left against the reference is the FP32 summation order and the BF16 roundings it
# flips: 1e-2 in norm per layer, as for the gradients of 1024 rows.
@pytest.mark.parametrize("n", [1, 15, 16, 17, 33, 2432, 2433, 4896, 9750])
def test_gradients_of_any_batch(sur, n):  # noqa: F811
    s, _ = sur
    rng = np.random.default_rng(n)
    u = inputs(n)
    t = rng.normal(scale=0.3, size=(n, 20)).astype(np.float32)
    w = rng.uniform(0.5, 2.0, size=20).astype(np.float32)
    loss, grads = s.grad(u, t, w)
    rloss, rgrads = bf16_passes_reference(s.get_params(), u, t.astype(np.float64), w.astype(np.float64))
    assert abs(loss - rloss) < 1e-2 * rloss
    assert not grads[0][0][:, 7:].any() and not grads[4][0][20:].any() and not grads[4][1][20:].any()
    for li, ((gW, gb), (rW, rb)) in enumerate(zip(grads, rgrads)):
        if li == 0:
            gW, rW = gW[:, :7], rW[:, :7]
        if li == 4:
            gW, rW, gb, rb = gW[:20], rW[:20], gb[:20], rb[:20]
        assert np.linalg.norm(gW - rW) < 1e-2 * np.linalg.norm(rW), li
        assert np.linalg.norm(gb - rb) < 1e-2 * np.linalg.norm(rb), li
