"""Residual sums formed by the pointwise layer that reads them: with and without a ReLU, one operand or both with pending coefficients, channel
counts that leave a tail in the last chunk, maps for one tile, for several tiles per block and for the split reduction, sums read again by a later
sum.  Held to the plain float64 oracle, or to the rounding of bfloat16 storage."""
import pytest

import stage_inputs as si
from harness import ALL, CONTRACT, bf16_store, compare, gpu_round, make_inputs, oracle_round, summary

pytestmark = pytest.mark.gpu


def _net(c, wide, relu, projected):
    """Two residual blocks: x -> 1x1 -> BN -> 1x1 -> BN, + x (or + 1x1 -> BN of x), [ReLU], and a 1x1 layer at the end."""
    L, net = si.Layer, []

    def push(op, ci, co, src, add_from=-1):
        net.append(L(op, ci, co, 1 if op == "conv" else 0, 1, 0, src, add_from))
        return len(net) - 1

    top = push("bn", c, c, push("conv", 16, c, -1))
    for block in range(2):
        other = top
        if projected and block == 0:
            other = push("bn", c, c, push("conv", c, c, top))
        last = push("bn", wide, wide, push("conv", c, wide, top))
        last = push("bn", c, c, push("conv", wide, c, last))
        top = push("add", c, c, last, other)
        if relu:
            top = push("relu", c, c, top)
    push("conv", c, 24, top)
    return net


CASES = {
    # name: (channels, inner channels, relu, projected, h, w, micro-batch)
    "plain": (24, 48, False, False, 9, 7, 3),
    "relu": (32, 40, True, False, 11, 5, 2),
    "both_pending_tail": (40, 16, True, True, 13, 9, 3),
    "persistent_tiles": (24, 32, False, False, 151, 139, 2),
    "split_reduction": (328, 24, False, True, 7, 7, 4),
    "one_pixel_maps": (64, 64, True, False, 1, 1, 32),
}


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("name", list(CASES))
def test_deferred_add_edges(name, bf16):
    c, wide, relu, projected, h, w, B = CASES[name]
    net = _net(c, wide, relu, projected)
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, B, 2, "mse", 37, bf16)
    params = si.randomize_bn(params, net, 0, last, 37)
    plain = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params)
    mirror = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params, store=bf16_store) if bf16 else None
    gpu = gpu_round(net, 0, last, h, w, B, 2, "mse", xs, tg, params, bf16)
    r = compare(gpu, plain, net, 0, last, 2e-2 if bf16 else 1e-4, mirror=mirror, allow=ALL if bf16 else (CONTRACT,), outlier_frac=2e-3 if bf16 else 0.0,
                case="deferred_add/%s" % name)
    print(name, summary(r))
