"""The 3x3 and 5x5 depthwise kernels at the edges of their strips: maps narrower and shorter than a strip, widths that strips cover exactly and
one more, odd and even maps at stride 2, channel counts that split unevenly over the blocks, several strips per thread, with and
without the units that leave sums behind or take them.  Activation-free, held to the plain float64 oracle on every tensor."""
import pytest

import stage_inputs as si
from harness import ALL, CONTRACT, bf16_store, compare, gpu_round, make_inputs, oracle_round, summary

pytestmark = pytest.mark.gpu


def _net(c, stride, around, k):
    """Depthwise conv with BatchNorm; `around`: between two 1x1 convs with BatchNorm (coefficients pending on both sides)."""
    L, net = si.Layer, []

    def push(op, ci, co, k, st, pad):
        net.append(L(op, ci, co, k, st, pad, len(net) - 1, -1))

    if around:
        push("conv", 16, c, 1, 1, 0)
        push("bn", c, c, 0, 1, 0)
    push("dwconv", c, c, k, stride, k // 2)
    push("bn", c, c, 0, 1, 0)
    if around:
        push("conv", c, 24, 1, 1, 0)
        push("bn", 24, 24, 0, 1, 0)
    return net


CASES = {
    # name: (channels, stride, h, w, micro-batch, between pointwise layers)
    "one_column": (8, 1, 6, 1, 3, True),
    "narrower_than_a_strip": (8, 1, 1, 3, 9, True),
    "one_strip": (24, 1, 7, 4, 4, True),
    "one_past_a_strip": (24, 1, 5, 9, 4, True),
    "uneven_channel_split": (72, 1, 14, 14, 3, True),
    "many_channels": (1000, 1, 7, 7, 2, True),
    "several_strips_per_thread": (24, 1, 181, 134, 5, True),
    "alone": (40, 1, 11, 13, 3, False),
    "s2_smallest": (8, 2, 1, 1, 24, True),
    "s2_two_rows": (8, 2, 2, 3, 6, True),
    "s2_odd": (24, 2, 9, 13, 4, True),
    "s2_even_exact": (72, 2, 12, 16, 3, True),
    "s2_even_one_past": (136, 2, 14, 14, 2, True),
    "s2_several_strips_per_thread": (24, 2, 233, 151, 5, True),
    "s2_alone": (40, 2, 10, 11, 3, False),
}


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("k", [3, 5])
@pytest.mark.parametrize("name", list(CASES))
def test_depthwise_edges(name, k, bf16):
    c, stride, h, w, B, around = CASES[name]
    net = _net(c, stride, around, k)
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, B, 2, "mse", 23, bf16)
    params = si.randomize_bn(params, net, 0, last, 23)
    plain = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params)
    # maps of a few pixels: the gradients in front of a BatchNorm nearly vanish, and what is left of them is the storage rounding
    mirror = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params, store=bf16_store) if bf16 else None
    gpu = gpu_round(net, 0, last, h, w, B, 2, "mse", xs, tg, params, bf16)
    r = compare(gpu, plain, net, 0, last, 2e-2 if bf16 else 1e-4, mirror=mirror, allow=ALL if bf16 else (CONTRACT,), case="dw%d_edges/%s" % (k, name))
    print(name, k, summary(r))
