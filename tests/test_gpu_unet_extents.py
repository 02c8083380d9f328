"""The network on grids with long planes: offsets past 32 bits in elements.
The element-wise bounds are those of the other network tests."""
import numpy as np
import pytest

from oracle import unet as N
from test_gpu_unet import _elementwise

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _net(F, seed):
    from paper_2208_05524_gb300 import vesis
    net = vesis.Net(F)
    net.set_params(N.init_params(F, seed=seed).astype(np.float32))
    return net


def _need(gigabytes):
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < gigabytes * 1e9:
        pytest.skip("needs %d GB of device memory" % gigabytes)


def test_planes_past_two_gigaelements():
    """8 planes of 8320 x 8192 cells x 32 channels (2.2e9 elements each): the
    far corner's logits against those of a small crop there (the same path;
    the network sees less than 64 cells around a cell)."""
    _need(160)
    n, c, m = (8, 8320, 8192), 512, 64
    net = _net(1, 41)
    g = torch.Generator(device="cuda").manual_seed(41)
    x = torch.randn(int(np.prod(n)), device="cuda", generator=g)
    part = torch.empty(8 * c * c, device="cuda")
    net.forward(x, n, crop=(0, n[1] - c, n[2] - c, 8, c, c), logits=part)
    want = part.view(8, c, c)[:, m:, m:].cpu().numpy()
    whole = torch.empty(int(np.prod(n)), device="cuda")
    net.forward(x, n, logits=whole)
    got = whole.view(n)[:, n[1] - c + m:, n[2] - c + m:].cpu().numpy()
    net.close()
    del x, whole
    torch.cuda.empty_cache()
    _elementwise(got, want, "far corner")
