"""The register-operand pointwise kernels at the edges of their tiles: channel counts that are no whole chunk or column tile, maps of a few
pixels, one pixel past a tile, reductions that are split over warps, coefficients that are still sums when the next kernel reads
them.  Activation-free stages, held to the plain float64 oracle at the bfloat16 contract (2e-2) on every tensor."""
import pytest

import stage_inputs as si
from harness import CONTRACT, compare, gpu_round, make_inputs, oracle_round, summary

pytestmark = pytest.mark.gpu


def _chain(*channels):
    """1x1 convs with BatchNorm one after another (no activation)."""
    net = []
    for c_in, c_out in zip(channels, channels[1:]):
        net.append(si.Layer("conv", c_in, c_out, 1, 1, 0, len(net) - 1, -1))
        net.append(si.Layer("bn", c_out, c_out, 0, 1, 0, len(net) - 1, -1))
    return net


CASES = {
    # name: (channels, h, w, micro-batch)
    "smallest": ((8, 8), 3, 3, 8),
    "one_pixel_past_a_tile": ((24, 40), 43, 3, 1),                   # 129 pixels
    "chunk_tail_column_tail": ((40, 200, 24), 9, 7, 3),              # 40 = 32 + 8, 200 = 6 chunks + 8
    "persistent_many_tiles": ((32, 56, 16), 61, 57, 5),              # 17 385 pixels, several tiles per CTA, 56 = 32 + 24 columns
    "persistent_two_tiles_high": ((16, 96, 72), 80, 79, 4),
    "split_reduction_over_eight_warps": ((960, 24), 5, 3, 4),
    "split_reduction_ragged": ((328, 88), 11, 5, 7),                 # 11 chunks over the warps
    "wide_on_both_sides": ((648, 520), 7, 7, 3),
    "tiny_map_wide": ((1032, 1000), 2, 2, 5),
}


@pytest.mark.parametrize("name", list(CASES))
def test_pointwise_edges(name):
    channels, h, w, B = CASES[name]
    net = _chain(*channels)
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, B, 2, "mse", 17, True)
    params = si.randomize_bn(params, net, 0, last, 17)
    plain = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params)
    gpu = gpu_round(net, 0, last, h, w, B, 2, "mse", xs, tg, params, True)
    r = compare(gpu, plain, net, 0, last, 2e-2, allow=(CONTRACT,), case="pw_edges/%s" % name)
    print(name, summary(r))
