"""Gradients stored as the activation in front lets them through, by the kernels that take that unit's sums: pointwise -> depthwise -> pointwise with an
activation behind each BatchNorm, at channel counts and maps that end inside a tile, stride 1 and 2, with the residual sum (whose other operand's gradient must
not be masked) and without."""
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
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, B, 2, "mse", 37, bf16)
    params = si.randomize_bn(params, net, 0, last, 37)
    plain = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params)
    mirror = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params, store=bf16_store) if bf16 else None
    gpu = gpu_round(net, 0, last, h, w, B, 2, "mse", xs, tg, params, bf16)
    compare(gpu, plain, net, 0, last, 2e-2 if bf16 else 1e-4, mirror=mirror, allow=ALL if bf16 else (CONTRACT,), case="masked/%s/%s" % (name, act))
