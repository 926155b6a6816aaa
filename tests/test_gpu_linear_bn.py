"""A linear layer with a BatchNorm (and an activation) behind it: the BatchNorm takes the layer's bias out again with the mean, so the bias has no gradient.
The zero is judged on the scale of the other parameters' gradients."""
import pytest

import stage_inputs as si
from harness import ALL, CONTRACT, bf16_store, compare, gpu_round, make_inputs, oracle_round

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("act", [None, "relu", "relu6"])
def test_linear_in_front_of_bn(act, bf16):
    L, c, hid, B = si.Layer, 24, 40, 64
    net = [L("gap", c, c, 0, 1, 0, -1, -1), L("linear", c, hid, 1, 1, 0, 0, -1), L("bn", hid, hid, 0, 1, 0, 1, -1)]
    if act:
        net.append(L(act, hid, hid, 0, 1, 0, 2, -1))
    net.append(L("linear", hid, 16, 1, 1, 0, len(net) - 1, -1))
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, 3, 3, B, 2, "mse", 47, bf16)
    params = si.randomize_bn(params, net, 0, last, 47)
    plain = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params)
    mirror = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params, store=bf16_store) if bf16 else None
    gpu = gpu_round(net, 0, last, 3, 3, B, 2, "mse", xs, tg, params, bf16)
    compare(gpu, plain, net, 0, last, 2e-2 if bf16 else 1e-4, mirror=mirror, allow=ALL if bf16 else (CONTRACT,), case="linear_bn/%s" % act)
