"""Pointwise layers on maps of 50 000 pixels and more, where the tensor-memory kernels take over from the register-operand ones: the pipeline with resident
weights, for as many channels as fit; for 192 to 256 channels on both sides the streaming kernel (forward, and a backward that needs no transform)
and the one-tile kernel (a backward that does).  392 tiles of 128 pixels, the last one ragged.  And the pipelined weight gradient on channel
sub-ranges, which begins beyond 4 096 pixels: four of 128 channels, two of 192 where a quarter is no multiple of 64.  Activation-free stages, held to the plain float64
oracle at the bfloat16 contract (2e-2) on every tensor."""
import pytest

import stage_inputs as si
from harness import CONTRACT, compare, gpu_round, make_inputs, oracle_round, summary

pytestmark = pytest.mark.gpu

H, W = 227, 221                                    # 50 167 pixels


def _check(c_in, c_out, bn, H, W):
    net = si.single_unit_net("conv", c_in, c_out, bn=bn)
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, H, W, 1, 1, "mse", 19, True)
    params = si.randomize_bn(params, net, 0, last, 19)
    plain = oracle_round(net, 0, last, 1, 1, "mse", xs, tg, params)
    gpu = gpu_round(net, 0, last, H, W, 1, 1, "mse", xs, tg, params, True)
    print(summary(compare(gpu, plain, net, 0, last, 2e-2, allow=(CONTRACT,), case="pw_large/%d_%d_%s" % (c_in, c_out, "bn" if bn else "plain"))))


@pytest.mark.parametrize("bn", [False, True], ids=["plain", "bn"])
@pytest.mark.parametrize("c_in, c_out", [(64, 256), (128, 256), (256, 128), (72, 232), (256, 256), (192, 256), (256, 192), (224, 256), (200, 256)])
def test_pointwise_on_a_large_map(c_in, c_out, bn):
    _check(c_in, c_out, bn, H, W)


@pytest.mark.parametrize("c_in, c_out", [(128, 512), (512, 128), (128, 384), (384, 128)])
def test_weight_gradient_on_channel_sub_ranges(c_in, c_out):
    _check(c_in, c_out, True, 67, 63)              # 4 221 pixels
