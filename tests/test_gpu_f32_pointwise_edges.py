"""The float32 pointwise kernels at the edges of their tiles: channel counts that are no whole column tile or chunk, maps of a few pixels, one
pixel past a tile, reductions split over warps, pixel ranges that end inside a group, gradients cut into several clusters.
Activation-free stages, held to the plain float64 oracle at the float32 contract (1e-4) on every tensor."""
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
    "smallest": ((4, 4), 3, 3, 8),
    "one_pixel_past_a_tile": ((24, 40), 43, 3, 1),
    "chunk_tail_column_tail": ((20, 100, 28), 9, 7, 3),
    "many_tiles_per_block": ((16, 52, 12), 121, 107, 5),
    "reduction_over_two_warps": ((36, 24, 44), 17, 13, 5),
    "reduction_over_four_warps": ((324, 88, 64), 11, 5, 7),
    "wide_on_both_sides": ((200, 260), 7, 7, 3),
    "long_reduction": ((1284, 20), 3, 3, 8),
    "several_clusters": ((48, 16), 75, 70, 4),
    "ranges_left_empty": ((24, 144, 24), 28, 28, 1),
    "thin_gradient_in_narrow_tiles": ((144, 24), 75, 70, 4),
}


@pytest.mark.parametrize("name", list(CASES))
def test_f32_pointwise_edges(name):
    channels, h, w, B = CASES[name]
    net = _chain(*channels)
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, B, 2, "mse", 29, False)
    params = si.randomize_bn(params, net, 0, last, 29)
    plain = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params)
    gpu = gpu_round(net, 0, last, h, w, B, 2, "mse", xs, tg, params, False)
    r = compare(gpu, plain, net, 0, last, 1e-4, allow=(CONTRACT,), case="f32_pw_edges/%s" % name)
    print(name, summary(r))
