"""Pointwise layers whose operands are requested several steps ahead.  Input gradients: reductions that end inside a 32-channel chunk, several tiles a CTA and a last one partly filled, CTAs of
four and of eight warps, one and several column blocks, with a residual's addend, with the sums of a BatchNorm in front, with and without an activation that the gradient was not stored behind (the
layer is the last).  Residual sums of more than 4 M elements that the layer behind forms as it loads.  And layers just outside these rules.  Each test reads from a profile which form ran."""
import pytest

import stage_inputs as si
from harness import ALL, CONTRACT, bf16_store, compare, gpu_round, kernels, make_inputs, oracle_round

pytestmark = pytest.mark.gpu

L = si.Layer


def _check(net, h, w, B, case, act):
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, B, 1, "mse", 59, True)
    params = si.randomize_bn(params, net, 0, last, 59)
    plain = oracle_round(net, 0, last, B, 1, "mse", xs, tg, params)
    mirror = oracle_round(net, 0, last, B, 1, "mse", xs, tg, params, store=bf16_store) if act else None
    gpu = gpu_round(net, 0, last, h, w, B, 1, "mse", xs, tg, params, True)
    compare(gpu, plain, net, 0, last, 2e-2, mirror=mirror, allow=ALL if act else (CONTRACT,), case="deep/%s" % case)


def _ahead(found, bwd):
    """Of the register-operand pointwise kernels of one direction: which request several steps ahead (their last template argument)."""
    if not found:
        pytest.skip("no kernel records from the profiler")
    names = [k["name"] for k in found if "pw_mma_kernel<%s," % ("true" if bwd else "false") in k["name"]]
    return [n.split("pw_mma_kernel<")[1].split(">")[0].endswith("true") for n in names]


# several column blocks, and one: forwards of long reductions and several tiles a CTA, whose operand the layer before has just written
@pytest.mark.parametrize("c, c_out, h, w, B", [(128, 512, 28, 28, 32), (256, 512, 25, 20, 40), (256, 64, 95, 100, 6)])
def test_forwards_request_one_step_ahead(c, c_out, h, w, B):
    net = [L("conv", 16, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 0, -1), L("relu", c, c, 0, 1, 0, 1, -1), L("conv", c, c_out, 1, 1, 0, 2, -1), L("bn", c_out, c_out, 0, 1, 0, 3, -1)]
    xs, tg, params, _ = make_inputs(net, 0, 4, h, w, B, 1, "mse", 59, True)
    with kernels() as found:
        gpu_round(net, 0, 4, h, w, B, 1, "mse", xs, tg, params, True)
    assert _ahead(found, False) == [False, False]


def _net(c_in, c_out, act, where):
    """A 1x1 layer with BatchNorm [and an activation]; "behind" another one, whose BatchNorm sums its input gradient takes; in a "block", whose residual gradient it adds as well."""
    net = []

    def unit(ci, co, src, op):
        net.extend([L("conv", ci, co, 1, 1, 0, src, -1), L("bn", co, co, 0, 1, 0, len(net), -1)])
        if op:
            net.append(L(op, co, co, 0, 1, 0, len(net) - 1, -1))
        return len(net) - 1

    top = unit(16, c_in, -1, "relu") if where else -1
    last = unit(c_in, c_out, top, act)
    if where == "block":
        last = unit(c_out, c_in, last, None)
        net.append(L("add", c_in, c_in, 0, 1, 0, last, top))
    return net


GRADIENTS = {
    # columns (c_in), reduction (c_out), activation, where, h, w, micro-batch: several steps ahead?, threads of a CTA, column blocks, fewest tiles of a CTA
    "eight_warps": (256, 144, None, None, 209, 79, 1, True, 256, 4, 3),
    "eight_warps_long": (128, 528, None, "behind", 53, 67, 5, True, 256, 2, 1),
    "four_warps": (64, 176, None, None, 57013, 1, 1, True, 128, 1, 3),
    "four_warps_chunk_tail": (64, 152, None, "behind", 57013, 1, 1, True, 128, 1, 3),
    "four_warps_blocks": (192, 528, None, "behind", 20011, 1, 1, True, 128, 3, 3),
    "column_tail": (184, 272, None, None, 20011, 1, 1, True, 128, 3, 3),
    "one_block_column_tail": (56, 128, None, "behind", 101, 113, 5, True, 128, 1, 3),
    "addend": (64, 144, "relu", "block", 101, 113, 5, True, 128, 1, 3),
    "activation": (256, 264, "relu", None, 171, 193, 1, True, 128, 4, 6),
    "activation_relu6": (320, 272, "relu6", "behind", 171, 193, 1, True, 128, 5, 8),
    "activation_short": (512, 128, "relu", None, 28, 28, 32, True, 128, 8, 10),
    "activation_eight_warps": (256, 144, "relu", None, 209, 79, 1, True, 256, 4, 3),
    # one step ahead: rows that split sectors on smaller maps, short reductions, one tile a CTA
    "split_sectors_activation": (256, 136, "relu", None, 109, 92, 1, False, 256, 4, 2),
    "split_sectors_small": (256, 136, None, None, 25, 1000, 1, False, 128, 4, 5),
    "short": (64, 120, None, None, 57013, 1, 1, False, 128, 1, 3),
    "one_tile": (64, 128, None, None, 13, 1000, 1, False, 256, 1, 1),
}


@pytest.mark.parametrize("name", list(GRADIENTS))
def test_input_gradients(name):
    c_in, c_out, act, where, h, w, B, ahead, threads, blocks, tiles = GRADIENTS[name]
    net = _net(c_in, c_out, act, where)
    with kernels() as found:
        _check(net, h, w, B, name, bool(act or where))
    got = [k for k in found if "pw_mma_kernel<true," in k["name"] and k["grid"][1] == blocks and ", 8, 4, " in k["name"]]
    assert _ahead(found, True).count(True) == int(ahead)
    mine = next(k for k in got if _ahead([k], True) == [ahead])
    assert mine["block"][0] == threads and -(-h * w * B // (threads // 2)) >= tiles * mine["grid"][0]


SUMS = {
    # channels of the sum, columns of the layer behind, h, w, micro-batch: formed by that layer?
    "tile_tail": (256, 64, 61, 935, 1, True),
    "chunk_tail_column_tail": (264, 56, 57013, 1, 1, True),
    "long": (512, 64, 40, 977, 1, True),
    "four_chunks": (128, 64, 100, 119, 5, True),
    "columns_of_three_CTAs": (256, 136, 130, 127, 1, False),
    "blocks_of_48_columns": (264, 40, 130, 127, 1, False),
    "fewer_tiles_than_CTAs": (128, 64, 130, 127, 2, False),
    "short": (120, 64, 57013, 1, 1, False),
}


@pytest.mark.parametrize("name", list(SUMS))
@pytest.mark.parametrize("relu", [False, True])
def test_large_sums(name, relu):
    c, c_out, h, w, B, formed = SUMS[name]
    net = [L("conv", 16, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 0, -1), L("conv", 16, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 2, -1), L("add", c, c, 0, 1, 0, 3, 1)]
    net += [L("relu", c, c, 0, 1, 0, 4, -1)] if relu else []
    net += [L("conv", c, c_out, 1, 1, 0, len(net) - 1, -1), L("bn", c_out, c_out, 0, 1, 0, len(net), -1)]
    assert c * h * w * B > 1 << 22
    with kernels() as found:
        _check(net, h, w, B, "sum_%s_%s" % (name, relu), relu)
    assert _ahead(found, False).count(True) == int(formed)
