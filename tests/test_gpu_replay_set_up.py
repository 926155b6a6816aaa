"""A call that is repeated with the same slot and buffers is captured by the library.  That must not disturb a capture of the caller's own that is
open at the time, on another stream of the same thread or in another thread."""
import threading

import numpy as np
import pytest
import torch

import stage_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["same_thread", "other_thread"])
def test_repeated_calls_beside_an_open_capture(where):
    import paper_2408_08015_b200 as P
    net = si.block_net(16, 6)
    last = len(net) - 1
    x = torch.randn(2, 8, 8, 16, device="cuda")
    y, dy, dx = torch.empty_like(x), torch.randn_like(x), torch.empty_like(x)
    hdl = P.asteroid_stage_create(net, 0, last, 8, 8, 2, 1)
    work, other = torch.cuda.Stream(), torch.cuda.Stream()
    a, b = torch.ones(1000, device="cuda"), torch.zeros(1000, device="cuda")
    errors = []

    def calls():
        try:
            for _ in range(5):
                P.asteroid_stage_forward(hdl, 0, x.data_ptr(), y.data_ptr(), work.cuda_stream)
                P.asteroid_stage_backward(hdl, 0, dy.data_ptr(), dx.data_ptr(), work.cuda_stream)
                P.asteroid_stage_accumulate(hdl, 0, work.cuda_stream)
                P.asteroid_stage_step(hdl, 0.0, 0.0, work.cuda_stream)
        except Exception as e:                                   # reported by the main thread
            errors.append(e)

    try:
        P.asteroid_stage_import_state(hdl, np.ascontiguousarray(si.init_params(net, 0, last, 2), np.float32))
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(other):
            g.capture_begin(capture_error_mode="global")
            b.add_(a)
            if where == "same_thread":
                calls()
            else:
                t = threading.Thread(target=calls)
                t.start()
                t.join()
            b.add_(a)
            g.capture_end()
        assert not errors, errors
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert (b == 2).all() and torch.isfinite(dx).all()
    finally:
        P.asteroid_stage_destroy(hdl)
