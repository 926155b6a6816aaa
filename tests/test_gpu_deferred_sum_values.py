"""Residual sums that the pointwise layer behind them forms, against the elementwise pass: the stage that ends with the sum hands out what that pass stores, and one with a 1x1 layer behind whose
weights pick one channel each hands out what the layer stored and read.  Beyond 4 M elements the same bits; at any size the same values where an operand is not a number."""
import numpy as np
import pytest

import stage_inputs as si

pytestmark = pytest.mark.gpu

L = si.Layer


def _sum_net(c, bn, relu):
    net = []
    for _ in range(2):
        net.append(L("conv", 16, c, 1, 1, 0, -1, -1))
        if bn:
            net.append(L("bn", c, c, 0, 1, 0, len(net) - 1, -1))
    net.append(L("add", c, c, 0, 1, 0, len(net) - 1, 1 if bn else 0))
    return net + ([L("relu", c, c, 0, 1, 0, len(net) - 1, -1)] if relu else [])


def _forward(net, params, x, h, w, B):
    """Output of one forward, and the layer that the profile names for the sum (None: a pass of its own)."""
    import torch
    import paper_2408_08015_b200 as P
    last = len(net) - 1
    hdl = P.asteroid_stage_create(net, 0, last, h, w, B, 1, dtype=P.AST_BF16)
    try:
        P.asteroid_stage_import_state(hdl, np.ascontiguousarray(params, np.float32))
        _, shp = P.asteroid_stage_output_elems(hdl)
        y = torch.empty((B,) + shp, device="cuda", dtype=torch.bfloat16)
        P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        add = next(i for i, l in enumerate(net) if l.op == "add")
        into = P.asteroid_stage_profile(hdl, add, B)["fused_into"] if add < last else -1
        return y.reshape(-1, shp[2]), into
    finally:
        P.asteroid_stage_destroy(hdl)


def _both(c, c_out, h, w, B, bn, relu, odd):
    """The sum by the elementwise pass, its picked channels, and the output of the layer that forms it."""
    import torch
    net = _sum_net(c, bn, relu)
    last = len(net) - 1
    x = torch.randn(B, h, w, 16, generator=torch.Generator().manual_seed(3))
    flat = x.reshape(-1, 16)
    for i, v in enumerate(odd):
        flat[i * 97 % flat.shape[0]] = v
    x = x.to("cuda", torch.bfloat16)
    params = si.init_params(net, 0, last, 7)
    if bn:
        params = si.randomize_bn(params, net, 0, last, 7)
    else:                                          # one sign, so that minus infinity in gives it in every channel
        params = np.abs(params)
    whole, _ = _forward(net, params, x, h, w, B)
    channels = (np.arange(c_out) * 5 + 3) % c      # 5 and the channel counts have no common factor
    pick = np.zeros((c_out, c), np.float32)
    pick[np.arange(c_out), channels] = 1.0
    picked, into = _forward(net + [L("conv", c, c_out, 1, 1, 0, last, -1)], np.concatenate([params, pick.ravel()]), x, h, w, B)
    assert into == last + 1
    return whole, channels, picked


# more than 4 M elements; every map leaves a last tile partly filled, 264 channels a last chunk
@pytest.mark.parametrize("c, c_out, h, w, B", [(256, 64, 61, 935, 1), (264, 56, 57013, 1, 1), (128, 64, 100, 190, 3), (512, 64, 40, 977, 1)])
@pytest.mark.parametrize("relu", [False, True])
def test_large_sums_to_the_bit(c, c_out, h, w, B, relu):
    import torch
    whole, channels, picked = _both(c, c_out, h, w, B, True, relu, [])
    assert whole.shape[0] * c > 1 << 22
    assert torch.equal(whole[:, channels], picked)


# inputs that are not numbers, and minus infinity: a ReLU makes numbers of the sums (anything else would spread over the layer's products).  One large sum, two small ones
@pytest.mark.parametrize("c, c_out, h, w, B", [(256, 64, 61, 935, 1), (64, 24, 16, 16, 4), (64, 32, 131, 127, 2)])
def test_sums_of_what_is_not_a_number(c, c_out, h, w, B):
    import torch
    whole, channels, picked = _both(c, c_out, h, w, B, False, True, (float("nan"), -float("inf")))
    assert bool(torch.isfinite(whole).all())
    assert torch.equal(whole[:, channels], picked)
