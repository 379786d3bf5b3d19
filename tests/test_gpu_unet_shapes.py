"""The warm-start network's convolution kernels at the shapes the configured
network does not reach: odd channel counts (no aligned pairs), images that are
not square and end inside a tile, tiles of either side, and layers too wide
for their channels to be staged at once.  Each layer against the oracle's
products of the device's own stored inputs (tolerances and teacher forcing as
in test_gpu_unet.py)."""
import numpy as np
import pytest

from oracle import unet as ou
from test_gpu_unet import _case, _flips, _layer_levels, ms, rel, unpack  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,width,H,W", [(2, 2, 8, 8), (3, 3, 16, 48), (2, 5, 40, 24),
                                              (2, 6, 296, 280), (2, 256, 8, 16)])
def test_each_layer(ms, levels, width, H, W):  # noqa: F811
    net, spec, params, x, t, xd, td = _case(ms, levels, width, max(H, W), 5)
    x, xd, td = x[:H, :W], xd[:H, :W].contiguous(), td[:H, :W].contiguous()
    net.keep_intermediates(True)
    y, _, g = net.gradients(xd, td)
    assert rel(net.forward(xd).cpu().numpy(), y.cpu().numpy()) == 0.0
    got = unpack(spec, g)
    level, shapes = _layer_levels(levels), spec.conv_shapes()
    for k, (co, ci) in enumerate(shapes):
        h, w = H >> level[k], W >> level[k]
        a_in = net.layer_tensor(k, "in", (h, w, ci)).astype(np.float64)
        dz = net.layer_tensor(k, "grad", (h, w, co)).astype(np.float64)
        assert rel(got[k]["w"], ou.conv3x3_grad_weight(a_in, dz)) <= 5e-3, k
        assert rel(got[k]["b"], dz.sum(axis=(0, 1))) <= 5e-3, k
        if k == len(shapes) - 1:   # FP32 sums of bfloat16 products
            want = ou.conv3x3(a_in, ou.bf16(params[k]["w"]), params[k]["b"])[..., 0] + x[..., 0]
            assert rel(y.cpu().numpy(), want) <= 1e-5
            continue
        out = net.layer_tensor(k, "out", (h, w, co)).astype(np.float64)
        want = ou.conv3x3(a_in, ou.bf16(params[k]["w"]), params[k]["b"])
        assert _flips(out, ou.bf16(np.maximum(want, 0.0)))[1] <= 1.0 + 1e-9, k
        if level[k + 1] == level[k] and shapes[k + 1][1] == co:
            dz_next = net.layer_tensor(k + 1, "grad", (h, w, shapes[k + 1][0]))
            dx = ou.conv3x3_grad_input(dz_next.astype(np.float64), ou.bf16(params[k + 1]["w"]))
            assert _flips(dz, ou.bf16(dx * (out > 0)))[1] <= 1.0 + 1e-9, k
    net.close()
