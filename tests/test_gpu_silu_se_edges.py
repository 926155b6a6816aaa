"""The SiLU and squeeze-excite passes at the edges of their cuts: maps of one pixel, fewer pixels than a block holds side by side, more channel
vectors than threads, odd channel counts, gates too wide for shared memory, and the pairs that are fused (SiLU in front of the gate, BatchNorm in
front of SiLU) beside those that are not.  Held to the plain float64 oracle, or to the rounding of bfloat16 storage."""
import pytest

import stage_inputs as si
from harness import ALL, CONTRACT, bf16_store, compare, gpu_round, make_inputs, oracle_round, summary

pytestmark = pytest.mark.gpu

CASES = {
    # name: (channels, hidden units, layers behind the conv, h, w, micro-batch)
    "one_pixel": (16, 4, ("bn", "silu", "se"), 1, 1, 32),
    "few_pixels": (24, 6, ("bn", "silu", "se"), 3, 3, 4),
    "ragged_runs": (40, 10, ("bn", "silu", "se"), 37, 29, 3),
    "more_vectors_than_threads": (2056, 4, ("bn", "silu", "se"), 3, 2, 8),
    "wide_gate": (800, 40, ("bn", "silu", "se"), 4, 4, 4),
    "silu_alone": (48, 0, ("bn", "silu"), 15, 11, 5),
    "silu_without_batchnorm": (48, 0, ("silu",), 9, 7, 3),
    "gate_without_silu": (40, 8, ("bn", "se"), 13, 9, 4),
}


def _net(c, k, ops):
    net = [si.Layer("conv", 16, c, 1, 1, 0, -1, -1)]
    for op in ops:
        net.append(si.Layer(op, c, c, k if op == "se" else 0, 1, 0, len(net) - 1, -1))
    return net


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("name", list(CASES))
def test_silu_se_edges(name, bf16):
    c, k, ops, h, w, B = CASES[name]
    net = _net(c, k, ops)
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, B, 2, "mse", 31, bf16)
    params = si.randomize_bn(params, net, 0, last, 31)
    plain = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params)
    mirror = oracle_round(net, 0, last, B, 2, "mse", xs, tg, params, store=bf16_store) if bf16 else None
    gpu = gpu_round(net, 0, last, h, w, B, 2, "mse", xs, tg, params, bf16)
    r = compare(gpu, plain, net, 0, last, 2e-2 if bf16 else 1e-4, mirror=mirror, allow=ALL if bf16 else (CONTRACT,), case="silu_se_edges/%s" % name)
    print(name, summary(r))
