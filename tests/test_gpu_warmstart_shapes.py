"""The default network back end at image shapes whose levels mix its two convolution paths (channels-last
boxes, explicit im2col), several tile cuts and channel padding, against the network oracle: forward and
gradients to twice the scale of the BF16 rounding's own effect (the oracle with against without it;
flips of rounded operands compound with depth), the loss to 1e-3."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle.unet as U  # noqa: E402
from paper_2211_05009_gb300 import binding as B  # noqa: E402
from tests.test_gpu_warmstart import _setup  # noqa: E402


@pytest.mark.parametrize("width,H,W", [(4, 16, 128),    # one pixel row at the deepest level
                                       (4, 48, 384),    # 384, 192, 96, 48, 24 wide
                                       (4, 128, 48),    # 48 .. 3 wide: no channels-last level
                                       (12, 80, 128)])  # both paths; channels padded to 64, 128, 192
def test_network_at_shape_matches_oracle(width, H, W):
    n, p, (x, base, tgt, mask), (dx, dbase, dtgt, dmask) = _setup(width=width, H=H, W=W, backend=3)
    try:
        got = torch.empty(3, H, W, dtype=torch.float32, device="cuda")
        B.lbm_net_forward(n, dx, H, W, got)
        out, cache = U.forward(p, width, x, rnd=True)
        out_x, cache_x = U.forward(p, width, x, rnd=False)
        assert np.linalg.norm(got.double().cpu().numpy() - out) < 2.0 * np.linalg.norm(out - out_x)
        B.lbm_net_zero_grads(n)
        grads = []
        for _ in range(2):  # gradients add up
            loss = B.lbm_net_backward(n, dx, dbase, dtgt, dmask, H, W)
            g = torch.empty(B.lbm_net_param_count(n), dtype=torch.float32, device="cuda")
            B.lbm_net_get_grads(n, g)
            grads.append(g.double().cpu().numpy())
        ref_loss, gout = U.loss_and_grad(out, base, tgt, mask)
        ref = U.backward(p, width, cache, gout, rnd=True)
        assert abs(loss - ref_loss) < 1e-3 * ref_loss
        exact = U.backward(p, width, cache_x, U.loss_and_grad(out_x, base, tgt, mask)[1], rnd=False)
        off = 0
        for ci, co in U.conv_list(width):
            for sz in (co * ci * 9, co):
                a, b, e = grads[0][off:off + sz], ref[off:off + sz], exact[off:off + sz]
                assert np.linalg.norm(a - b) < 2.0 * max(np.linalg.norm(b - e), 1e-2 * np.linalg.norm(b)), (ci, co, sz)
                off += sz
        assert np.linalg.norm(grads[0] - ref) < 2.0 * np.linalg.norm(ref - exact)
        assert np.linalg.norm(grads[1] - 2 * grads[0]) < 1e-5 * np.linalg.norm(grads[0])
    finally:
        B.lbm_net_destroy(n)
