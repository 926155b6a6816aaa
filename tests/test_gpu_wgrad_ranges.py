"""Pixel ranges of the pointwise weight gradient on small maps: one, two, four or eight to a cluster, the last two where every warp of a range has a group of 16
pixels (512 and 1024 pixels).  Maps at those limits, one pixel below and above, gradients of one block of 32 x 32 and of several; with a BatchNorm
(coefficients formed by the kernel).  A range left out or taken twice changes a gradient by at least a third, the contract is 2e-2."""
import pytest

import stage_inputs as si
from harness import CONTRACT, MIRROR, bf16_store, compare, gpu_round, make_inputs, oracle_round

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h, w", [(7, 73), (16, 32), (19, 27), (31, 33), (32, 32), (25, 41)])
@pytest.mark.parametrize("c_in, c_out", [(24, 32), (72, 40), (40, 136)])
def test_wgrad_ranges(c_in, c_out, h, w):
    net = si.single_unit_net("conv", c_in, c_out, bn=True)
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, 1, 2, "mse", 43, True)
    params = si.randomize_bn(params, net, 0, last, 43)
    plain = oracle_round(net, 0, last, 1, 2, "mse", xs, tg, params)
    mirror = oracle_round(net, 0, last, 1, 2, "mse", xs, tg, params, store=bf16_store)
    gpu = gpu_round(net, 0, last, h, w, 1, 2, "mse", xs, tg, params, True)
    compare(gpu, plain, net, 0, last, 2e-2, mirror=mirror, allow=(CONTRACT, MIRROR), case="wgrad_ranges/%d_%d_%d" % (c_in, c_out, h * w))
