"""The sin^2 stencil's convolution on rows of every length and alignment."""
import numpy as np
import pytest

import oracle as O
from paper_2208_05524_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nz", [1, 3, 7, 8, 9, 15, 16, 17, 23, 29, 40])
@pytest.mark.parametrize("off", [0, 1, 5])
def test_conv3_rows(nz, off):
    """W equals the oracle's integer convolution with the labels `off` bytes
    into their allocation and bytes of other value around them."""
    from paper_2208_05524_gb300 import vesis
    n, h = (9, 11, nz), 0.25
    s = synth.single_ion(n=8, h=h)
    s["n"] = np.array(n)
    s["origin"] = -0.5 * np.array(n) * h
    sc = O.surface_constants(s, O.params(kernel="sin2", sin2_lambda=2.0))
    S = vesis.System(s, kernel="sin2", sin2_lambda=2.0)
    G = int(np.prod(n))
    chi0 = synth.random_labels(n, seed=nz)
    buf = torch.full((G + 16,), 255, dtype=torch.uint8, device="cuda")
    chi = buf[off:off + G]
    chi.copy_(torch.from_numpy(chi0.reshape(-1)))
    W = torch.full((G + 8,), -1, dtype=torch.int32, device="cuda")
    S.surface_weights(chi, W[:G])
    assert np.array_equal(W[:G].cpu().numpy().astype(np.int64), O.conv3(chi0, sc["k3"]).reshape(-1))
    assert bool((W[G:] == -1).all()) and bool((buf[off + G:] == 255).all())
