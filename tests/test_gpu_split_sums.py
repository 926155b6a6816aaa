"""Sums of the weight gradients' partials: blocks of eight warps from 64 blocks of 128 outputs and 17 partials on, blocks of 32 warps below.  Gradients of 60, 64
and 67.5 blocks; maps that leave 33 partials, 65 (one more than eight warps request at once) and one per multiprocessor.  A partial that is left out or
taken twice changes a gradient by about one over the square root of their number, a multiple of the contract's 2e-2."""
import pytest

import stage_inputs as si
from harness import CONTRACT, compare, gpu_round, make_inputs, oracle_round, summary

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h, w", [(67, 63), (97, 85), (149, 131)])
@pytest.mark.parametrize("c_in, c_out", [(64, 120), (64, 128), (120, 72)])
def test_split_sums(c_in, c_out, h, w):
    net = si.single_unit_net("conv", c_in, c_out, bn=True)
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, 1, 1, "mse", 41, True)
    params = si.randomize_bn(params, net, 0, last, 41)
    plain = oracle_round(net, 0, last, 1, 1, "mse", xs, tg, params)
    gpu = gpu_round(net, 0, last, h, w, 1, 1, "mse", xs, tg, params, True)
    print(summary(compare(gpu, plain, net, 0, last, 2e-2, allow=(CONTRACT,), case="split_sums/%d_%d_%d" % (c_in, c_out, h * w))))
