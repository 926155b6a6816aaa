"""The profile call times the launches a round makes: as many kernels as a direct forward and backward, and a residual sum that a pointwise layer forms
as it loads is no pass of its own in either."""
import numpy as np
import pytest
import torch

import stage_inputs as si

pytestmark = pytest.mark.gpu

PASSES = 10                                        # warm-up and timed rounds of one profile call


@pytest.mark.parametrize("bf16", [False, True], ids=["f32", "bf16"])
@pytest.mark.parametrize("net", ["mobilenetv2_stage", "resnet50_c2c3"])
def test_profile_launches_what_a_round_launches(net, bf16):
    import paper_2408_08015_b200 as P
    net = si.stage_net_mbv2_4blocks() if net == "mobilenetv2_stage" else si.resnet50_c2c3_net()
    last, B, H, W = len(net) - 1, 4, 28, 28
    dt, tdt = (P.AST_BF16, torch.bfloat16) if bf16 else (P.AST_F32, torch.float32)
    hdl = P.asteroid_stage_create(net, 0, last, H, W, B, 1, dtype=dt)
    try:
        P.asteroid_stage_import_state(hdl, np.ascontiguousarray(si.init_params(net, 0, last, 0), np.float32))
        x = torch.randn(B, H, W, net[0].c_in, device="cuda").to(tdt)
        _, shp = P.asteroid_stage_output_elems(hdl)
        y = torch.empty((B,) + shp, device="cuda", dtype=tdt)
        dy, dx = torch.randn_like(y), torch.empty_like(x)
        n0 = P.asteroid_launch_count()
        P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr())
        P.asteroid_stage_backward(hdl, 0, dy.data_ptr(), dx.data_ptr())
        n1 = P.asteroid_launch_count()
        recs = [P.asteroid_stage_profile(hdl, l, B) for l in range(last + 1)]
        assert P.asteroid_launch_count() - n1 == PASSES * (n1 - n0)
        deferred = [l for l in range(last + 1) if net[l].op == "add" and recs[l]["fused_into"] >= 0]
        if not bf16 or net[0].c_in == 24:          # MobileNetV2's sums in front of a pointwise layer, and all of float32's
            assert deferred
        for l in deferred:
            conv = recs[l]["fused_into"]
            assert net[conv].op == "conv" and net[conv].k == 1 and recs[l]["t_f_ms"] == 0 and recs[l]["alg_bytes_f"] == 0
            e = 2 if bf16 else 4
            p = B * si.out_shape(net, 0, last, H, W)[l][0] * si.out_shape(net, 0, last, H, W)[l][1]
            assert recs[conv]["alg_bytes_f"] == e * p * (3 * net[conv].c_in + net[conv].c_out) + recs[conv]["w_l_bytes"]
    finally:
        P.asteroid_stage_destroy(hdl)
