"""The passes at the ends of a call: the cross-entropy head with rows that fit the registers its threads keep and longer ones, the pool's backward by vectors
and by channels, reductions over maps of a few pixels."""
import numpy as np
import pytest

import stage_inputs as si
from harness import ALL, CONTRACT, bf16_store, compare, gpu_round, make_inputs, oracle_round

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("rows,classes", [(1, 1), (3, 7), (16, 1000), (5, 2047), (5, 2048), (5, 2049), (2, 6000)])
def test_cross_entropy_rows(rows, classes, bf16):
    import torch
    import paper_2408_08015_b200 as P
    gen = torch.Generator(device="cuda").manual_seed(rows * 7919 + classes)
    x = (3 * torch.randn(rows, classes, generator=gen, device="cuda")).to(torch.bfloat16 if bf16 else torch.float32)
    t = torch.randint(0, classes, (rows,), generator=gen, device="cuda", dtype=torch.int32)
    t[0] = classes - 1
    dx, loss = torch.empty_like(x), torch.zeros(1, device="cuda")
    P.asteroid_loss_softmax_xent(x.data_ptr(), t.data_ptr(), rows, classes, P.AST_BF16 if bf16 else P.AST_F32, dx.data_ptr(), loss.data_ptr())
    x64 = x.double()
    ref = (torch.softmax(x64, 1) - torch.nn.functional.one_hot(t.long(), classes)) / rows
    want = torch.nn.functional.cross_entropy(x64, t.long()).item()
    # float32: a sum of `classes` terms of rounded exponentials (2 ulp each) and a division; bfloat16: the rounding to 8 significant bits, 2^-8, on top
    eps = 2.0 ** -24
    tol = (classes ** 0.5 + 8) * 2 * eps + (2.0 ** -8 if bf16 else 0)
    assert ((dx.double() - ref).abs() <= tol * ref.abs() + 4 * eps / rows).all()
    assert abs(loss.item() - want) <= (classes ** 0.5 + 8) * 4 * eps * max(want, 1.0)


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("c,h,w,B", [(8, 1, 1, 12), (12, 3, 2, 5), (24, 7, 7, 4), (20, 5, 3, 3), (328, 2, 2, 6)])
def test_pool_and_small_reductions(c, h, w, B, bf16):
    L = si.Layer
    net = [L("conv", 16, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 0, -1), L("gap", c, c, 0, 1, 0, 1, -1), L("linear", c, 40, 1, 1, 0, 2, -1)]
    xs, tg, params, _ = make_inputs(net, 0, 3, h, w, B, 2, "xent", 31, bf16)
    params = si.randomize_bn(params, net, 0, 3, 31)
    plain = oracle_round(net, 0, 3, B, 2, "xent", xs, tg, params)
    mirror = oracle_round(net, 0, 3, B, 2, "xent", xs, tg, params, store=bf16_store) if bf16 else None
    gpu = gpu_round(net, 0, 3, h, w, B, 2, "xent", xs, tg, params, bf16)
    compare(gpu, plain, net, 0, 3, 2e-2 if bf16 else 1e-4, mirror=mirror, allow=ALL if bf16 else (CONTRACT,), case="small_passes/%d_%d_%d_%d" % (c, h, w, B))
