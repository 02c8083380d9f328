"""The network on grids whose planes or rows are long: offsets past 32 bits in
elements, and rows of more work items than one launch dimension holds.  The
element-wise bounds are those of the other network tests."""
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


def test_training_on_long_rows():
    """Gradients on 8 x 8 rows of 1,048,640 cells made of two equal halves
    against those of one half (the loss is a mean; the seam is 1e-4 of the
    cells)."""
    _need(80)
    L = 524320
    net = _net(1, 42)
    g = torch.Generator(device="cuda").manual_seed(42)
    x = torch.randn(8, 8, L, device="cuda", generator=g)
    y = (x > 0.3).to(torch.uint8)
    l1, g1 = net.loss_grad(x.reshape(-1), y.reshape(-1), (8, 8, L), grad=True)
    x2, y2 = torch.cat([x, x], 2).reshape(-1), torch.cat([y, y], 2).reshape(-1)
    l2, g2 = net.loss_grad(x2, y2, (8, 8, 2 * L), grad=True)
    net.close()
    del x, y, x2, y2
    torch.cuda.empty_cache()
    assert abs(l1 - l2) <= 1e-3 * abs(l1)
    a, b = N.unpack(g1.astype(np.float64), 1), N.unpack(g2.astype(np.float64), 1)
    for k in a:
        for i in range(2):
            _elementwise(b[k][i], a[k][i], "%s[%d]" % (k, i))
