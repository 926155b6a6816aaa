"""The pool's backward with buffers of the caller's at any address of an element: dy where the pool is the stage's last layer, dx where it is the first.
Channel counts of whole vectors, so that the aligned call takes the vector kernel; both forms divide and round alike, so they agree to the bit."""
import numpy as np
import pytest

import stage_inputs as si

pytestmark = pytest.mark.gpu


def _at(t, offset):
    """A copy of t that begins `offset` elements behind a 16-byte boundary."""
    import torch
    flat = torch.empty(t.numel() + offset, dtype=t.dtype, device=t.device)[offset:]
    assert flat.data_ptr() % 16 == offset * t.element_size() % 16
    return flat.copy_(t.reshape(-1))


def _round(net, B, h, w, bf16, x, dy, off):
    import torch
    import paper_2408_08015_b200 as P
    last = len(net) - 1
    hdl = P.asteroid_stage_create(net, 0, last, h, w, B, 1, dtype=P.AST_BF16 if bf16 else P.AST_F32)
    try:
        P.asteroid_stage_import_state(hdl, si.randomize_bn(si.init_params(net, 0, last, 5), net, 0, last, 5))
        tensors = [_at(t, off.get(k, 0)) for k, t in (("x", x), ("y", torch.zeros_like(dy)), ("dy", dy), ("dx", torch.zeros_like(x)))]
        xd, yd, dyd, dxd = [t.data_ptr() for t in tensors]
        P.asteroid_stage_forward(hdl, 0, xd, yd)
        P.asteroid_stage_backward(hdl, 0, dyd, dxd)
        P.asteroid_stage_accumulate(hdl, 0)
        G = np.empty(P.asteroid_stage_param_count(hdl), np.float32)
        P.asteroid_stage_export_state(hdl, grad_accum=G)
        torch.cuda.synchronize()
        return tensors[1].clone(), tensors[3].clone(), G
    finally:
        P.asteroid_stage_destroy(hdl)


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("offset", [1, 2, 3, 7])
@pytest.mark.parametrize("where", ["last", "first"])
def test_pool_backward_addresses(where, offset, bf16):
    import torch
    L, c, B, h, w = si.Layer, 24, 5, 7, 6
    if where == "last":
        net = [L("conv", 16, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 0, -1), L("gap", c, c, 0, 1, 0, 1, -1)]
        c_in, out, off = 16, c, {"y": offset, "dy": offset}
    else:
        net = [L("gap", c, c, 0, 1, 0, -1, -1), L("linear", c, 40, 1, 1, 0, 0, -1)]
        c_in, out, off = c, 40, {"x": offset, "dx": offset}
    gen = torch.Generator(device="cuda").manual_seed(3)
    dt = torch.bfloat16 if bf16 else torch.float32
    x = torch.randn(B, h, w, c_in, generator=gen, device="cuda").to(dt)
    dy = torch.randn(B, 1, 1, out, generator=gen, device="cuda").to(dt)
    want, got = _round(net, B, h, w, bf16, x, dy, {}), _round(net, B, h, w, bf16, x, dy, off)
    assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1]) and np.array_equal(want[2], got[2])
    assert want[1].abs().max() > 0 and np.abs(want[2]).max() > 0
