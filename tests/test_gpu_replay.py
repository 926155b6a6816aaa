"""Calls repeated with the same slot and buffers are replayed from graphs; calls with new buffers are not, nor calls made while the caller
captures.  Both must give the same rounds: outputs, gradients, losses, BatchNorm estimates and parameters, on the default stream and on another,
with more distinct buffers than graphs are kept, and after a new state has been imported."""
import numpy as np
import pytest

import paper_2408_08015_b200 as P
import stage_inputs as si

pytestmark = pytest.mark.gpu

ROUNDS, B, M, H, W = 6, 3, 3, 13, 11


def _run(fresh, own_stream):
    """ROUNDS training rounds; `fresh`: every call gets buffers of its own."""
    import torch

    net = si.block_net(16, 6)
    last = len(net) - 1
    n = si.param_count(net, 0, last)
    rng = np.random.default_rng(5)
    params = (rng.standard_normal(n) * 0.2).astype(np.float32)
    dev = torch.device("cuda")
    h = P.asteroid_stage_create(net, 0, last, H, W, B, M, dtype=P.AST_F32, slots=2)
    P.asteroid_stage_import_state(h, params)
    oh, ow, oc = si.out_shape(net, 0, last, H, W)[last]
    xs = [torch.from_numpy(rng.standard_normal((B, H, W, 16)).astype(np.float32)).to(dev) for _ in range(M)]
    ts = [torch.from_numpy(rng.standard_normal((B, oh, ow, oc)).astype(np.float32)).to(dev) for _ in range(M)]
    fixed = [(x.clone(), torch.empty_like(ts[0]), torch.empty_like(ts[0]), torch.empty_like(x)) for x in xs]
    loss = torch.zeros(ROUNDS, M, device=dev)
    st = torch.cuda.Stream() if own_stream else torch.cuda.default_stream()
    torch.cuda.synchronize()
    out, keep = [], []
    with torch.cuda.stream(st):
        raw = st.cuda_stream
        for r in range(ROUNDS):
            if r == 4:
                torch.cuda.synchronize()
                P.asteroid_stage_import_state(h, params * np.float32(0.5))
            for m in range(M):
                x, y, dy, dx = fixed[m] if not fresh else (xs[m].clone(), torch.empty_like(ts[0]), torch.empty_like(ts[0]), torch.empty_like(xs[0]))
                keep.append((x, y, dy, dx))
                P.asteroid_stage_forward(h, m, x.data_ptr(), y.data_ptr(), raw)
                P.asteroid_loss_mse(y.data_ptr(), ts[m].data_ptr(), y.numel(), P.AST_F32, dy.data_ptr(), loss[r, m:].data_ptr(), raw)
                P.asteroid_stage_backward(h, m, dy.data_ptr(), dx.data_ptr(), raw)
                P.asteroid_stage_accumulate(h, m, raw)
                out.append((y.clone(), dx.clone()))
            P.asteroid_stage_step(h, 0.05, 0.9, raw)
    torch.cuda.synchronize()
    res = [t.cpu().numpy() for p in out for t in p] + [loss.cpu().numpy()]
    state = [np.empty(n, np.float32) for _ in range(2)]
    P.asteroid_stage_export_state(h, *state)
    res += state
    P.asteroid_stage_destroy(h)
    return res


@pytest.mark.parametrize("own_stream", [False, True], ids=["default_stream", "own_stream"])
def test_replayed_calls_equal_direct_ones(own_stream):
    a, b = _run(False, own_stream), _run(True, own_stream)
    assert len(a) == len(b)
    for x, y in zip(a, b):
        np.testing.assert_allclose(x, y, rtol=1e-5, atol=1e-6)


def test_more_buffers_than_graphs():
    """Forty buffer sets, each used four times in turn: graphs come and go, every call still computes its own input."""
    import torch

    net = si.single_unit_net("conv", 16, 24, bn=True)
    last = len(net) - 1
    rng = np.random.default_rng(6)
    h = P.asteroid_stage_create(net, 0, last, 5, 5, 2, 1, dtype=P.AST_F32)
    P.asteroid_stage_import_state(h, (rng.standard_normal(si.param_count(net, 0, last)) * 0.3).astype(np.float32))
    dev = torch.device("cuda")
    sets = [(torch.randn(2, 5, 5, 16, device=dev), torch.empty(2, 5, 5, 24, device=dev), torch.randn(2, 5, 5, 24, device=dev), torch.empty(2, 5, 5, 16, device=dev))
            for _ in range(40)]
    first = {}
    for rep in range(4):
        for i, (x, y, dy, dx) in enumerate(sets):
            for _ in range(3 if i % 7 == 0 else 1):
                y.zero_()
                dx.zero_()
                P.asteroid_stage_forward(h, 0, x.data_ptr(), y.data_ptr(), torch.cuda.current_stream().cuda_stream)
                P.asteroid_stage_backward(h, 0, dy.data_ptr(), dx.data_ptr(), torch.cuda.current_stream().cuda_stream)
                P.asteroid_stage_accumulate(h, 0, torch.cuda.current_stream().cuda_stream)
                P.asteroid_stage_step(h, 0.0, 0.0, torch.cuda.current_stream().cuda_stream)
                got = (y.clone(), dx.clone())
                if i not in first:
                    first[i] = got
                torch.testing.assert_close(got[0], first[i][0], rtol=1e-5, atol=1e-6)
                torch.testing.assert_close(got[1], first[i][1], rtol=1e-5, atol=1e-6)
    P.asteroid_stage_destroy(h)
