"""Order of a traced backward's kernels: a trace keeps every kernel on the caller's stream, each layer's weight gradient in front of its input gradient."""
import json

import pytest

import stage_inputs as si

pytestmark = pytest.mark.gpu


def test_order_of_a_traced_backward(tmp_path):
    import torch
    from torch.profiler import ProfilerActivity, profile
    import paper_2408_08015_b200 as P
    L, c, B, h, w = si.Layer, 64, 4, 14, 14
    net = []
    for _ in range(3):
        net += [L("conv", c, c, 1, 1, 0, len(net) - 1, -1), L("bn", c, c, 0, 1, 0, len(net), -1), L("relu", c, c, 0, 1, 0, len(net) + 1, -1)]
    hdl = P.asteroid_stage_create(net, 0, len(net) - 1, h, w, B, 1, dtype=P.AST_BF16)
    try:
        P.asteroid_stage_import_state(hdl, si.init_params(net, 0, len(net) - 1, 0))
        x = torch.randn(B, h, w, c, device="cuda").to(torch.bfloat16)
        y, dy, dx = torch.empty_like(x), torch.randn_like(x), torch.empty_like(x)
        sp = torch.cuda.current_stream().cuda_stream
        P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr(), sp)
        torch.cuda.synchronize()
        P.asteroid_trace_start()
        with profile(activities=[ProfilerActivity.CUDA], acc_events=True) as p:
            P.asteroid_stage_backward(hdl, 0, dy.data_ptr(), dx.data_ptr(), sp)
            torch.cuda.synchronize()
        P.asteroid_trace_stop()
    finally:
        P.asteroid_stage_destroy(hdl)
    p.export_chrome_trace(str(tmp_path / "t.json"))
    events = sorted((e["ts"], e["name"]) for e in json.load(open(tmp_path / "t.json"))["traceEvents"] if e.get("cat") == "kernel")
    if not events:
        pytest.skip("no kernel records from the profiler")
    order = ["w" if "wgrad" in n else "d" for _, n in events if "wgrad" in n or "pw_mma" in n]
    assert "".join(order) == "wdwdwd", order
