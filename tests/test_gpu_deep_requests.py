"""Pointwise layers whose operands are requested several steps ahead: input gradients of 128 channels and more at reductions that end inside a 32-channel chunk, with fewer steps than
slots, several tiles a CTA and a last one partly filled, with and without an activation behind the BatchNorm (whose gradient then is not stored masked: the layer is the last); residual sums of more than 4 M
elements that the layer behind forms as it loads, and ones that it does not (three column tiles, a short reduction)."""
import pytest

import stage_inputs as si
from harness import ALL, CONTRACT, bf16_store, compare, gpu_round, kernels, make_inputs, oracle_round

pytestmark = pytest.mark.gpu

L = si.Layer


def _check(net, h, w, B, case, act):
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, B, 1, "mse", 59, True)
    params = si.randomize_bn(params, net, 0, last, 59)
    plain = oracle_round(net, 0, last, B, 1, "mse", xs, tg, params)
    mirror = oracle_round(net, 0, last, B, 1, "mse", xs, tg, params, store=bf16_store) if act else None
    gpu = gpu_round(net, 0, last, h, w, B, 1, "mse", xs, tg, params, True)
    compare(gpu, plain, net, 0, last, 2e-2, mirror=mirror, allow=ALL if act else (CONTRACT,), case="deep/%s" % case)


def _ahead(found, bwd):
    """Of the register-operand pointwise kernels of one direction: which request several steps ahead (their last template argument)."""
    if not found:
        pytest.skip("no kernel records from the profiler")
    names = [k["name"] for k in found if "pw_mma_kernel<%s," % ("true" if bwd else "false") in k["name"]]
    return [n.split("pw_mma_kernel<")[1].split(">")[0].endswith("true") for n in names]


# several column blocks, and one: forwards of long reductions and several tiles a CTA, whose operand the layer before has just written
@pytest.mark.parametrize("c, c_out, h, w, B", [(128, 512, 28, 28, 32), (256, 512, 25, 20, 40), (256, 64, 95, 100, 6)])
def test_forwards_request_one_step_ahead(c, c_out, h, w, B):
    net = [L("conv", 16, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 0, -1), L("relu", c, c, 0, 1, 0, 1, -1), L("conv", c, c_out, 1, 1, 0, 2, -1), L("bn", c_out, c_out, 0, 1, 0, 3, -1)]
    xs, tg, params, _ = make_inputs(net, 0, 4, h, w, B, 1, "mse", 59, True)
    with kernels() as found:
        gpu_round(net, 0, 4, h, w, B, 1, "mse", xs, tg, params, True)
    assert _ahead(found, False) == [False, False]


# 5 pixels: one tile; 1 000: single and partly filled ones; 19 594: several a CTA
@pytest.mark.parametrize("h, w, B", [(1, 5, 1), (25, 20, 2), (101, 97, 2)])
@pytest.mark.parametrize("c_in, c_out", [(32, 128), (64, 136), (72, 168), (64, 264), (48, 520)])
@pytest.mark.parametrize("act", [None, "relu6"])
def test_input_gradients(c_in, c_out, h, w, B, act):
    net = [L("conv", c_in, c_out, 1, 1, 0, -1, -1), L("bn", c_out, c_out, 0, 1, 0, 0, -1)] + ([L(act, c_out, c_out, 0, 1, 0, 1, -1)] if act else [])
    if act and h * w * B < 50:
        pytest.skip("masks of five values a channel")
    _check(net, h, w, B, "%d_%d_%d_%s" % (c_in, c_out, h * w * B, act), act)


# formed by the layer: 256 -> 64 and 264 -> 40 on 16 510 pixels; not: 256 -> 136 (more columns than a CTA takes), 128 -> 64 on 33 020
@pytest.mark.parametrize("c, c_out, B", [(256, 64, 1), (264, 40, 1), (256, 136, 1), (128, 64, 2)])
@pytest.mark.parametrize("relu", [False, True])
def test_large_sums(c, c_out, B, relu):
    net = [L("conv", 16, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 0, -1), L("conv", 16, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 2, -1), L("add", c, c, 0, 1, 0, 3, 1)]
    net += [L("relu", c, c, 0, 1, 0, 4, -1)] if relu else []
    net += [L("conv", c, c_out, 1, 1, 0, len(net) - 1, -1), L("bn", c_out, c_out, 0, 1, 0, len(net), -1)]
    _check(net, 130, 127, B, "sum_%d_%d_%s" % (c, c_out, relu), relu)
