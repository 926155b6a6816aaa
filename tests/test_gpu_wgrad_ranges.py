"""Pixel ranges of the pointwise weight gradient on small maps: a partial each where the gradient has few blocks, else one, two, four or eight to a cluster, four
from 512 pixels and eight from 1024 on (a group of 16 pixels for every warp of a range).  With a BatchNorm (coefficients formed by the kernel).  A
range left out or taken twice changes a gradient by about a quarter or more, the contract is 2e-2."""
import pytest

import stage_inputs as si
from harness import CONTRACT, MIRROR, bf16_store, compare, gpu_round, make_inputs, oracle_round

pytestmark = pytest.mark.gpu


# below 512 pixels clusters of two, at 512 and 513 of four, from 1023 on 15 or 16 partials
FEW_BLOCKS = [(ci, co, h, w) for ci, co in ((24, 32), (72, 40), (40, 136)) for h, w in ((7, 73), (16, 32), (19, 27), (31, 33), (32, 32), (25, 41))]
MORE_BLOCKS = [
    # 24 and 30 blocks of 32 x 32: one range
    (64, 384, 11, 11), (160, 192, 9, 14),
    # clusters of two, four (up to 1023 pixels) and eight
    (64, 384, 8, 16), (160, 192, 7, 73), (64, 384, 16, 32), (64, 384, 28, 36), (160, 192, 31, 33), (64, 384, 32, 32), (160, 192, 25, 41), (64, 384, 26, 40),
    # 75 blocks of 64 x 64: one range whatever the map
    (320, 960, 7, 9), (960, 320, 13, 11),
]


@pytest.mark.parametrize("c_in, c_out, h, w", FEW_BLOCKS + MORE_BLOCKS)
def test_wgrad_ranges(c_in, c_out, h, w):
    net = si.single_unit_net("conv", c_in, c_out, bn=True)
    last = len(net) - 1
    xs, tg, params, _ = make_inputs(net, 0, last, h, w, 1, 2, "mse", 43, True)
    params = si.randomize_bn(params, net, 0, last, 43)
    plain = oracle_round(net, 0, last, 1, 2, "mse", xs, tg, params)
    mirror = oracle_round(net, 0, last, 1, 2, "mse", xs, tg, params, store=bf16_store)
    gpu = gpu_round(net, 0, last, h, w, 1, 2, "mse", xs, tg, params, True)
    compare(gpu, plain, net, 0, last, 2e-2, mirror=mirror, allow=(CONTRACT, MIRROR), case="wgrad_ranges/%d_%d_%d" % (c_in, c_out, h * w))


def test_error_of_four_ranges():
    """Four ranges of 784 pixels are no further from the sum in 64 bits than eight ranges were with warps and ranges added one after the other: 7.57e-8 in the
    2-norm, over these seeds, with a standard error of 0.02e-8.  (Four added one after the other: 7.82e-8.)"""
    import numpy as np
    import torch
    import paper_2408_08015_b200 as P
    ci, co, B, h, w = 64, 384, 4, 14, 14
    net = si.single_unit_net("conv", ci, co)
    errors = []
    for seed in range(8):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(B, h, w, ci, generator=gen, device="cuda").to(torch.bfloat16)
        dy = torch.randn(B, h, w, co, generator=gen, device="cuda").to(torch.bfloat16)
        y, dx, G = torch.empty_like(dy), torch.empty_like(x), np.zeros(ci * co, np.float32)
        hdl = P.asteroid_stage_create(net, 0, 0, h, w, B, 1, dtype=P.AST_BF16)
        try:
            P.asteroid_stage_import_state(hdl, G)
            sp = torch.cuda.current_stream().cuda_stream
            P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr(), sp)
            P.asteroid_stage_backward(hdl, 0, dy.data_ptr(), dx.data_ptr(), sp)
            P.asteroid_stage_accumulate(hdl, 0, sp)
            P.asteroid_stage_export_state(hdl, grad_accum=G)
        finally:
            P.asteroid_stage_destroy(hdl)
        want = (dy.double().view(-1, co).T @ x.double().view(-1, ci)).cpu().numpy()
        errors.append(np.linalg.norm(G.reshape(co, ci) - want) / np.linalg.norm(want))
    assert np.mean(errors) <= 7.57e-8, errors
