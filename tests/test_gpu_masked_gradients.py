"""Gradients stored as the activation in front lets them through, by the kernels that take that unit's sums: pointwise -> depthwise -> pointwise with an
activation behind each BatchNorm, at channel counts and maps that end inside a tile, stride 1 and 2, with a residual sum at the end and without; every other kind
of layer as the one whose gradient arrives masked; and a residual sum whose operand has an activation of its own: the pointwise layer behind the sum takes that
operand's sums, but the gradient it writes is the other operand's too and must not be masked."""
import pytest

import stage_inputs as si
from harness import ALL, CONTRACT, bf16_store, compare, gpu_round, make_inputs, oracle_round

pytestmark = pytest.mark.gpu

CASES = {
    # name: (c_in, c_mid, c_out, stride, h, w, micro-batch)
    "small": (8, 32, 8, 1, 3, 7, 6),
    "one_column": (16, 40, 16, 1, 9, 1, 8),
    "ragged": (24, 72, 24, 1, 13, 11, 5),
    "wide": (160, 320, 160, 1, 7, 7, 3),
    "large_map": (16, 96, 16, 1, 61, 67, 2),
    "s2_odd": (24, 104, 32, 2, 13, 9, 5),
    "s2_even": (32, 192, 64, 2, 14, 14, 3),
}


def _check(net, h, w, B, bf16, case):
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, B, 2, "mse", 37, bf16)
    params = si.randomize_bn(params, net, 0, last, 37)
    plain = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params)
    mirror = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params, store=bf16_store) if bf16 else None
    gpu = gpu_round(net, 0, last, h, w, B, 2, "mse", xs, tg, params, bf16)
    compare(gpu, plain, net, 0, last, 2e-2 if bf16 else 1e-4, mirror=mirror, allow=ALL if bf16 else (CONTRACT,), case=case)


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("act", ["relu6", "relu"])
@pytest.mark.parametrize("name", list(CASES))
def test_masked_gradients(name, act, bf16):
    c_in, c, c_out, stride, h, w, B = CASES[name]
    L, net = si.Layer, []

    def push(op, ci, co, k=0, st=1, pad=0, src=None, add=-1):
        net.append(L(op, ci, co, k, st, pad, len(net) - 1 if src is None else src, add))

    for op, args in (("conv", (c_in, c, 1)), ("dwconv", (c, c, 3, stride, 1)), ("conv", (c, c_out, 1))):
        push(op, *args)
        push("bn", args[1], args[1])
        if len(net) < 6:
            push(act, args[1], args[1])
    if stride == 1 and c_in == c_out:
        push("add", c_out, c_out, add=-1)
    _check(net, h, w, B, bf16, "masked/%s/%s" % (name, act))


READERS = {
    # name: (layer, k, stride, c_in, c_out): the layer whose output gradient the pointwise layer behind it stores masked
    "depthwise_7x7": ("dwconv", 7, 1, 24, 24),
    "depthwise_7x7_s2": ("dwconv", 7, 2, 24, 24),
    "depthwise_5x5": ("dwconv", 5, 1, 24, 24),
    "columns_3x3": ("conv", 3, 1, 4, 24),
    "columns_3x3_s2": ("conv", 3, 2, 4, 24),
    "dense_3x3": ("conv", 3, 1, 64, 64),
    "zero_insertion_3x3": ("conv", 3, 2, 64, 64),
    "plain_3x3": ("conv", 3, 1, 24, 40),
    "strided_pointwise": ("conv", 1, 2, 24, 40),
}


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("name", list(READERS))
def test_readers_of_masked_gradients(name, bf16):
    op, k, stride, c_in, c = READERS[name]
    L, B, h, w = si.Layer, 3, 14, 12
    net = [L("conv", 16, c_in, 1, 1, 0, -1, -1), L("bn", c_in, c_in, 0, 1, 0, 0, -1), L("relu6", c_in, c_in, 0, 1, 0, 1, -1),
           L(op, c_in, c, k, stride, (k - 1) // 2, 2, -1), L("bn", c, c, 0, 1, 0, 3, -1), L("relu6", c, c, 0, 1, 0, 4, -1),
           L("conv", c, 24, 1, 1, 0, 5, -1), L("bn", 24, 24, 0, 1, 0, 6, -1)]
    _check(net, h, w, B, bf16, "masked_readers/%s" % name)


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("act", ["relu6", "relu"])
@pytest.mark.parametrize("skip", ["input", "activated"])
def test_gradient_of_both_operands_is_not_masked(skip, act, bf16):
    L, c = si.Layer, 24
    net = []
    if skip == "activated":
        net += [L("conv", c, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 0, -1), L(act, c, c, 0, 1, 0, 1, -1)]
    x = len(net) - 1
    net += [L("conv", c, c, 1, 1, 0, x, -1), L("bn", c, c, 0, 1, 0, x + 1, -1), L(act, c, c, 0, 1, 0, x + 2, -1), L("add", c, c, 0, 1, 0, x + 3, x),
            L("conv", c, 40, 1, 1, 0, x + 4, -1), L("bn", 40, 40, 0, 1, 0, x + 5, -1)]
    _check(net, 13, 11, 4, bf16, "masked_operand/%s_%s" % (skip, act))
