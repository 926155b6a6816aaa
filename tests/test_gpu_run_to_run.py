"""The same backward gives the same gradients, bit for bit, on every run.  Each kernel that takes channel sums or depthwise weight gradients is
given an output gradient with two entries of +-2^60 at far-away pixels among entries of about 1: the large ones cancel exactly, and
a sum that rounded on the way (a double keeps 53 bits) would hold what the order of its additions left of the small ones."""
import numpy as np
import pytest
import torch

import stage_inputs as si

pytestmark = pytest.mark.gpu

B, H, W, RUNS = 16, 32, 32, 24
L = si.Layer


def _net(kind, c):
    conv, bn = L("conv", c, c, 1, 1, 0, -1, -1), L("bn", c, c, 0, 1, 0, 0, -1)
    if kind == "own_pass":                                       # the stage's last BatchNorm: a reduction of its own over dy
        return [conv, bn]
    if kind == "pointwise":                                      # ... by the pointwise layer behind it
        return [conv, bn, L("conv", c, c, 1, 1, 0, 1, -1)]
    if kind == "silu":
        return [conv, bn, L("silu", c, c, 0, 1, 0, 1, -1)]
    k = int(kind[-1])
    return [conv, bn, L("dwconv", c, c, k, 1, (k - 1) // 2, 1, -1)]


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("kind", ["own_pass", "pointwise", "depthwise3", "depthwise5", "silu"])
def test_gradients_do_not_depend_on_the_order_of_additions(kind, bf16):
    import paper_2408_08015_b200 as P
    c = 32
    net = _net(kind, c)
    last = len(net) - 1
    n = si.param_count(net, 0, last)
    dt, tdt = (P.AST_BF16, torch.bfloat16) if bf16 else (P.AST_F32, torch.float32)
    gen = torch.Generator(device="cuda").manual_seed(11)
    x = torch.ones(B, H, W, c, device="cuda", dtype=tdt)         # the same everywhere: what is large cancels behind every layer
    x[:, 0] = torch.randn(B, W, c, generator=gen, device="cuda").to(tdt)
    dy = torch.randn(B, H, W, c, generator=gen, device="cuda").to(tdt)
    dy[1, 16, 16] = 2.0 ** 60
    dy[B - 2, 16, 16] = -2.0 ** 60
    y, dx = torch.empty_like(x), torch.empty_like(x)
    hdl = P.asteroid_stage_create(net, 0, last, H, W, B, 1, dtype=dt)
    try:
        params = np.ascontiguousarray(si.init_params(net, 0, last, 4), np.float32)
        first = None
        for run in range(RUNS):
            P.asteroid_stage_import_state(hdl, params)
            sp = torch.cuda.current_stream().cuda_stream
            P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr(), sp)
            P.asteroid_stage_backward(hdl, 0, dy.data_ptr(), dx.data_ptr(), sp)
            g = np.empty(n, np.float32)
            P.asteroid_stage_export_state(hdl, micro_grad=g)
            P.asteroid_stage_accumulate(hdl, 0, sp)
            P.asteroid_stage_step(hdl, 0.0, 0.0, sp)
            got = (g, dx.float().cpu().numpy())
            assert np.isfinite(got[0]).all()
            first = first or got
            for a, b in zip(first, got):
                np.testing.assert_array_equal(a, b, err_msg="run %d" % run)
    finally:
        P.asteroid_stage_destroy(hdl)


@pytest.mark.parametrize("kind", ["own_pass", "pointwise", "depthwise3"])
@pytest.mark.parametrize("exp", [-130, -80, -55, -33, -10, 10, 30, 60, 100])
def test_sums_of_every_magnitude(kind, exp):
    """beta's gradient against float64 for output gradients of about 2^exp, from where partial sums are subnormal to near the largest float.  A
    block's partial sum is a chain of float32 additions, each off by 2^-24 of what it holds: 2^-16 of the sum of magnitudes covers chains of 256."""
    import paper_2408_08015_b200 as P
    c = 32
    net = _net(kind, c)
    last = len(net) - 1
    gen = torch.Generator(device="cuda").manual_seed(12)
    x = torch.randn(B, H, W, c, generator=gen, device="cuda")
    dy = torch.randn(B, H, W, c, generator=gen, device="cuda") * torch.tensor(2.0, device="cuda").pow(exp / 2) * torch.tensor(2.0, device="cuda").pow(exp / 2)
    params = np.ascontiguousarray(si.init_params(net, 0, last, 4), np.float32)
    off, tail = {}, 0
    for i, name, shape in si.param_layout(net, 0, last):
        off[name, i] = (tail, shape)
        tail += int(np.prod(shape))
    y, dx = torch.empty_like(x), torch.empty_like(x)
    hdl = P.asteroid_stage_create(net, 0, last, H, W, B, 1, dtype=P.AST_F32)
    try:
        P.asteroid_stage_import_state(hdl, params)
        sp = torch.cuda.current_stream().cuda_stream
        P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr(), sp)
        P.asteroid_stage_backward(hdl, 0, dy.data_ptr(), dx.data_ptr(), sp)
        g = np.empty(tail, np.float32)
        P.asteroid_stage_export_state(hdl, micro_grad=g)
    finally:
        P.asteroid_stage_destroy(hdl)
    d = dy.double()
    if kind != "own_pass":
        o, shape = off["weight", last]
        w = torch.from_numpy(params[o:o + int(np.prod(shape))].astype(np.float64)).cuda()
        conv = torch.nn.grad.conv2d_input
        if kind == "pointwise":
            d = d.reshape(-1, c) @ w.reshape(c, c)
        else:
            d = conv((B, c, H, W), w.reshape(c, 1, 3, 3), d.permute(0, 3, 1, 2), padding=1, groups=c).permute(0, 2, 3, 1).reshape(-1, c)
    d = d.reshape(-1, c)
    o, _ = off["beta", 1]
    err = np.abs(g[o:o + c] - d.sum(0).cpu().numpy())
    # and a subnormal result is a multiple of 2^-149
    assert (err <= 2.0 ** -16 * d.abs().sum(0).cpu().numpy() + B * H * W * 2.0 ** -150).all(), (err, d.sum(0))


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_what_is_not_finite_stays_so(value):
    import paper_2408_08015_b200 as P
    c = 32
    net = _net("own_pass", c)
    x = torch.randn(B, H, W, c, device="cuda")
    dy = torch.randn(B, H, W, c, device="cuda")
    dy[3, 5, 7, 4] = value
    y, dx = torch.empty_like(x), torch.empty_like(x)
    hdl = P.asteroid_stage_create(net, 0, 1, H, W, B, 1, dtype=P.AST_F32)
    try:
        P.asteroid_stage_import_state(hdl, np.ascontiguousarray(si.init_params(net, 0, 1, 4), np.float32))
        P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr())
        P.asteroid_stage_backward(hdl, 0, dy.data_ptr(), dx.data_ptr())
        g = np.empty(si.param_count(net, 0, 1), np.float32)
        P.asteroid_stage_export_state(hdl, micro_grad=g)
    finally:
        P.asteroid_stage_destroy(hdl)
    beta = g[c * c + c:]
    assert beta[4] == value or (np.isnan(value) and np.isnan(beta[4]))
    assert np.isfinite(np.delete(beta, 4)).all()


@pytest.mark.parametrize("samples", [4096, 4097])
def test_more_samples_than_the_sums_have_room_for(samples):
    """The SiLU backward adds at least one partial sum a sample; beyond what the words of a sum have room for the sums are taken by a pass of their own.
    Against float64 autograd, at the float32 contract."""
    import paper_2408_08015_b200 as P
    c = 8
    net = _net("silu", c)
    n = si.param_count(net, 0, 2)
    params = np.ascontiguousarray(si.init_params(net, 0, 2, 6), np.float32)
    gen = torch.Generator(device="cuda").manual_seed(13)
    x, dy = (torch.randn(samples, 1, 1, c, generator=gen, device="cuda") for _ in range(2))
    y, dx = torch.empty_like(x), torch.empty_like(x)
    hdl = P.asteroid_stage_create(net, 0, 2, 1, 1, samples, 1, dtype=P.AST_F32)
    try:
        P.asteroid_stage_import_state(hdl, params)
        P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr())
        P.asteroid_stage_backward(hdl, 0, dy.data_ptr(), dx.data_ptr())
        g = np.empty(n, np.float32)
        P.asteroid_stage_export_state(hdl, micro_grad=g)
    finally:
        P.asteroid_stage_destroy(hdl)
    p = torch.from_numpy(params.astype(np.float64)).cuda()
    w, gamma, beta = (t.clone().requires_grad_() for t in (p[:c * c].reshape(c, c), p[c * c:c * c + c], p[c * c + c:]))
    xd = x.double().reshape(samples, c).requires_grad_()
    out = torch.nn.functional.silu(torch.nn.functional.batch_norm(xd @ w.T, None, None, gamma, beta, training=True, eps=1e-5))
    out.backward(dy.double().reshape(samples, c))
    ref = torch.cat([w.grad.reshape(-1), gamma.grad, beta.grad]).cpu().numpy()
    for got, want in ((g[:c * c], ref[:c * c]), (g[c * c:], ref[c * c:]), (dx.reshape(samples, c).cpu().numpy(), xd.grad.cpu().numpy()),
                      (y.reshape(samples, c).cpu().numpy(), out.detach().cpu().numpy())):
        assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()
