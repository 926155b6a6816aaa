"""A captured round needs nothing but the state it was captured from: whatever ran on the stage before a replay, and was dropped again by an import
of the state, leaves no trace in the replayed round."""
import numpy as np
import pytest
import torch

import stage_inputs as si

pytestmark = pytest.mark.gpu

B, M, H, W = 3, 2, 12, 10


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("dropped", ["forward", "backward"])
def test_replay_after_an_import_that_drops_calls(bf16, dropped):
    import paper_2408_08015_b200 as P
    net = si.block_net(16, 6)
    last = len(net) - 1
    n = si.param_count(net, 0, last)
    dt, tdt = (P.AST_BF16, torch.bfloat16) if bf16 else (P.AST_F32, torch.float32)
    params = np.ascontiguousarray(si.init_params(net, 0, last, 3), np.float32)
    gen = torch.Generator(device="cuda").manual_seed(3)
    x, dy = ([torch.randn(B, H, W, 16, generator=gen, device="cuda").to(tdt) for _ in range(M)] for _ in range(2))
    y, dx = ([torch.empty_like(t) for t in x] for _ in range(2))
    hdl = P.asteroid_stage_create(net, 0, last, H, W, B, M, dtype=dt)

    def micro(m, sp):
        P.asteroid_stage_forward(hdl, m, x[m].data_ptr(), y[m].data_ptr(), sp)
        P.asteroid_stage_backward(hdl, m, dy[m].data_ptr(), dx[m].data_ptr(), sp)

    def round_(sp):
        for m in range(M):
            micro(m, sp)
            P.asteroid_stage_accumulate(hdl, m, sp)
        P.asteroid_stage_step(hdl, 0.05, 0.9, sp)

    def result():
        torch.cuda.synchronize()
        w, v = np.empty(n, np.float32), np.empty(n, np.float32)
        P.asteroid_stage_export_state(hdl, params=w, momentum=v)
        return [w, v] + [t.float().cpu().numpy() for t in y + dx]

    try:
        P.asteroid_stage_import_state(hdl, params)
        round_(torch.cuda.current_stream().cuda_stream)          # first-use set-up
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            round_(torch.cuda.current_stream().cuda_stream)
        P.asteroid_stage_import_state(hdl, params)
        g.replay()
        want = result()
        micro(0, torch.cuda.current_stream().cuda_stream)        # a backward nobody accumulates ...
        if dropped == "forward":
            P.asteroid_stage_accumulate(hdl, 0, torch.cuda.current_stream().cuda_stream)
            P.asteroid_stage_forward(hdl, 0, x[0].data_ptr(), y[0].data_ptr(), torch.cuda.current_stream().cuda_stream)
        P.asteroid_stage_import_state(hdl, params)               # ... and which the import drops
        g.replay()
        for a, b in zip(want, result()):
            np.testing.assert_array_equal(a, b)
    finally:
        P.asteroid_stage_destroy(hdl)


def test_accumulate_without_a_backward_is_refused():
    """... whatever micro-batch it names: -1 is also what stands for none."""
    import paper_2408_08015_b200 as P
    net = si.block_net(16, 6)
    last = len(net) - 1
    x = torch.randn(B, H, W, 16, device="cuda")
    y, dx = torch.empty_like(x), torch.empty_like(x)
    hdl = P.asteroid_stage_create(net, 0, last, H, W, B, M)
    try:
        P.asteroid_stage_import_state(hdl, np.ascontiguousarray(si.init_params(net, 0, last, 3), np.float32))
        for mb in (-1, 0, M):
            with pytest.raises(P.binding.AsteroidError) as e:
                P.asteroid_stage_accumulate(hdl, mb)
            assert e.value.code == P.AST_ERR_ORDER
        P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr())
        P.asteroid_stage_backward(hdl, 0, y.data_ptr(), dx.data_ptr())
        P.asteroid_stage_accumulate(hdl, 0)
        for mb in (-1, 0, 1):
            with pytest.raises(P.binding.AsteroidError) as e:
                P.asteroid_stage_accumulate(hdl, mb)
            assert e.value.code == P.AST_ERR_ORDER
    finally:
        P.asteroid_stage_destroy(hdl)
