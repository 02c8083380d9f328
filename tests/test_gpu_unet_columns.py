"""The column-form convolution (k_conv_tma) at the edges of its range: blocks
that end inside the grid along x, and every form of the input layer (x
neighbours folded into channels or not, one or both halves of a 32-channel
stage), against the oracle."""
import pytest

from test_gpu_unet import _compare, _gpu, _oracle, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,F", [
    ((24, 32, 104), 3),      # 624 bricks, folded, one half; 24 is no multiple of 16
    ((24, 32, 104), 8),      # folded, both halves
    ((24, 32, 104), 12),     # 27 taps, one half
    ((24, 32, 104), 20),     # 27 taps, both halves
    ((8, 128, 80), 3),       # 640 bricks, fewer planes than a block holds
    ((152, 16, 32), 3),      # 608 bricks, the fewest; one column in y
])
def test_columns_match_oracle(n, F):
    """Logits, loss and gradients within the tolerances of the other paths."""
    theta, x, y = _problem(n, 33, F=F)
    zo, lo, go = _oracle(theta, x, y)
    z, loss, g = _gpu(theta, x, y, n, "tcgen05", F=F)
    _compare(z, zo.reshape(-1), g, go, loss, lo, F, "%s F=%d" % (n, F))
