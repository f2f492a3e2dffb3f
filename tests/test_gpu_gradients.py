"""The order of the network's gradient sums: fixed for bias gradients and, below 16,384 pixels, for weight
gradients, so that they have the same bits on every run."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle.unet as U  # noqa: E402
from paper_2211_05009_gb300 import binding as B  # noqa: E402
from tests.test_gpu_warmstart import _setup  # noqa: E402


def gradients(n, dev, H, W, runs):
    out = []
    for _ in range(runs):  # launched directly, captured, replayed
        B.lbm_net_zero_grads(n)
        B.lbm_net_backward(n, *dev, H, W)
        g = torch.empty(B.lbm_net_param_count(n), dtype=torch.float32, device="cuda")
        B.lbm_net_get_grads(n, g)
        out.append(g.cpu().numpy())
    return out


def tensors(width):
    """(offset, length, is a bias) of every parameter tensor."""
    off = 0
    for ci, co in U.conv_list(width):
        for sz, bias in ((co * ci * 9, False), (co, True)):
            yield off, sz, bias
            off += sz


@pytest.mark.parametrize("width,H,W", [(4, 16, 128),     # fewer pixels than a block at the deep levels
                                       (12, 112, 128),   # 14,336 pixels: the longest sums in one slice
                                       (4, 64, 192),     # no channels-last path at 192, 96, 48 columns
                                       (4, 128, 128)])   # 16,384 pixels: weight gradients in four slices at level 0
def test_gradients_repeat_bit_for_bit(width, H, W):
    n, _, _, dev = _setup(width=width, H=H, W=W, backend=3)
    try:
        first, *rest = gradients(n, dev, H, W, 6)
        assert np.isfinite(first).all()
        for g in rest:
            for off, sz, bias in tensors(width):
                if bias or H * W < 16384:
                    assert np.array_equal(g[off:off + sz], first[off:off + sz]), (off, sz)
    finally:
        B.lbm_net_destroy(n)


@pytest.mark.parametrize("H,W", [(16, 128), (48, 128), (160, 256)])
def test_head_bias_gradient_is_summed_in_its_stated_order(H, W):
    """dL/d(out) formed here in FP32 as the library forms it, 256 running sums over every 256th pixel and
    a tree over them: the same bits."""
    n, _, _, dev = _setup(width=4, H=H, W=W, backend=3)
    try:
        out = torch.empty(3, H, W, dtype=torch.float32, device="cuda")
        B.lbm_net_forward(n, dev[0], H, W, out)
        got = gradients(n, dev, H, W, 1)[0][-3:]
    finally:
        B.lbm_net_destroy(n)
    out, (base, tgt, mask) = out.cpu().numpy(), (d.cpu().numpy() for d in dev[1:])
    f = np.float32
    err = (base + out) - tgt
    count = mask.sum(dtype=np.float64)
    mean = f((mask * err[0]).sum(dtype=np.float64) / count)
    err[0] -= mean
    dz = (f(2) * (mask * err)) * f(1.0 / (3.0 * count))
    for c in range(3):
        s = np.zeros(256, dtype=f)
        for row in dz[c].reshape(-1, 256):
            s += row
        o = 128
        while o:
            s[:o] += s[o:2 * o]
            o //= 2
        assert got[c] == s[0], (c, got[c], s[0])
