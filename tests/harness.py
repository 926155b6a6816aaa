"""Shared test harness: run one HPP-Round on the oracle and on the CUDA library from the same
seeded inputs, and compare tensor by tensor.  Imported by tests and the smoke check only."""
import contextlib
import json
import os
import tempfile

import numpy as np

import stage_inputs as si


def make_inputs(net, first, last, h, w, B, M, loss, seed, bf16):
    c_in = net[first].c_in
    shp = si.out_shape(net, first, last, h, w)[last]
    cast = si.round_to_bf16 if bf16 else (lambda a: a)
    xs = [cast(si.normal(seed, 100000 + m, (B, h, w, c_in)).astype(np.float32)) for m in range(M)]
    if loss == "mse":
        tg = [cast(si.normal(seed, 200000 + m, (B,) + shp).astype(np.float32)) for m in range(M)]
    else:
        tg = [si.labels(seed, 300000 + m, B, shp[2]) for m in range(M)]
    params = si.init_params(net, first, last, seed)
    return xs, tg, params, shp


def default_order(M):
    return [("F", m) for m in range(M)] + [("B", m) for m in range(M)]


def bf16_store(a):
    """Rounding applied at storage points, and to the operands of dense contractions, when mirroring
    bfloat16 activation storage with bfloat16 tensor-core inputs."""
    return si.round_to_bf16(np.asarray(a, np.float32)).astype(np.float64)


def oracle_round(net, first, last, B, M, loss, xs, tg, params, lr=0.01, mu=0.9, order=None, momentum0=None, rounds=1,
                 store=None):
    import oracle as O
    st = O.Stage(net, first, last, B, M, params, store=store, operand=store)
    if momentum0 is not None:
        off = 0
        for k in st.v:
            n = st.v[k].size
            st.v[k] = np.asarray(momentum0[off:off + n], dtype=np.float64).reshape(st.v[k].shape)
            off += n
    res = None
    for _ in range(rounds):
        ys, out = {}, {}
        for kind, m in (order or default_order(M)):
            if kind == "F":
                ys[m] = st.forward(m, xs[m])
            else:
                if loss == "mse":
                    Lm, dy = O.mse_loss(ys[m], tg[m])
                else:
                    Lm, dy = O.softmax_xent_loss(ys[m].reshape(B, -1), tg[m])
                if store is not None:
                    dy = store(dy)
                dx = st.backward(m, dy)
                st.accumulate(m)
                out[m] = (ys[m], dx, Lm)
        G = st.flat_grad_accum().copy()
        st.step(lr, mu)
        res = {"y": [out[m][0] for m in range(M)], "dx": [out[m][1] for m in range(M)],
               "loss": [out[m][2] for m in range(M)], "G": G, "w": st.flat_params().copy(), "v": st.flat_momentum().copy()}
    return res


def gpu_round(net, first, last, h, w, B, M, loss, xs, tg, params, bf16, lr=0.01, mu=0.9, order=None,
              slots=0, need_dx=1, momentum0=None, rounds=1, stream=None, export_micro=False):
    import torch
    import paper_2408_08015_b200 as P
    dev = torch.device("cuda:0")
    tdt = torch.bfloat16 if bf16 else torch.float32
    dt = P.AST_BF16 if bf16 else P.AST_F32
    hdl = P.asteroid_stage_create(net, first, last, h, w, B, M, dtype=dt, slots=slots, need_input_grad=need_dx)
    try:
        P.asteroid_stage_import_state(hdl, np.ascontiguousarray(params, np.float32),
                                      None if momentum0 is None else np.ascontiguousarray(momentum0, np.float32))
        n_out, shp = P.asteroid_stage_output_elems(hdl)
        xd = [torch.from_numpy(x).to(dev, tdt).contiguous() for x in xs]
        if loss == "mse":
            td = [torch.from_numpy(t).to(dev, tdt).contiguous() for t in tg]
        else:
            td = [torch.from_numpy(np.asarray(t, np.int32)).to(dev) for t in tg]
        yd = [torch.empty((B,) + shp, device=dev, dtype=tdt) for _ in range(M)]
        dyd = [torch.empty((B,) + shp, device=dev, dtype=tdt) for _ in range(M)]
        dxd = [torch.zeros_like(x) for x in xd]
        lossd = torch.zeros(M, device=dev, dtype=torch.float32)
        sp = 0 if stream is None else stream.cuda_stream
        torch.cuda.synchronize()
        micro = {}
        for _ in range(rounds):
            for kind, m in (order or default_order(M)):
                if kind == "F":
                    P.asteroid_stage_forward(hdl, m, xd[m].data_ptr(), yd[m].data_ptr(), sp)
                else:
                    lp = lossd.data_ptr() + 4 * m
                    if loss == "mse":
                        P.asteroid_loss_mse(yd[m].data_ptr(), td[m].data_ptr(), n_out, dt, dyd[m].data_ptr(), lp, sp)
                    else:
                        P.asteroid_loss_softmax_xent(yd[m].data_ptr(), td[m].data_ptr(), B, shp[2], dt, dyd[m].data_ptr(), lp, sp)
                    P.asteroid_stage_backward(hdl, m, dyd[m].data_ptr(), dxd[m].data_ptr() if need_dx else None, sp)
                    if export_micro:
                        gm = np.empty(P.asteroid_stage_param_count(hdl), np.float32)
                        P.asteroid_stage_export_state(hdl, micro_grad=gm)
                        micro[m] = gm
                    P.asteroid_stage_accumulate(hdl, m, sp)
            n = P.asteroid_stage_param_count(hdl)
            G = np.empty(n, np.float32)
            P.asteroid_stage_export_state(hdl, grad_accum=G)
            P.asteroid_stage_step(hdl, lr, mu, sp)
        wv, vv = np.empty(n, np.float32), np.empty(n, np.float32)
        P.asteroid_stage_export_state(hdl, params=wv, momentum=vv)
        torch.cuda.synchronize()
        return {"y": [t.float().cpu().numpy() for t in yd], "dx": [t.float().cpu().numpy() for t in dxd],
                "loss": lossd.cpu().numpy().tolist(), "G": G, "w": wv, "v": vv, "g": micro}
    finally:
        P.asteroid_stage_destroy(hdl)


@contextlib.contextmanager
def kernels():
    """The kernels that run inside the block, in the order of their starts: a list of {"name", "grid", "block"} that is filled when the block ends (empty where the profiler has no records)."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    found = []
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA], acc_events=True) as p:
        yield found
        torch.cuda.synchronize()
    with tempfile.TemporaryDirectory() as d:
        path = os.path.join(d, "trace.json")
        p.export_chrome_trace(path)
        with open(path) as f:
            events = [e for e in json.load(f)["traceEvents"] if e.get("cat") == "kernel"]
    for e in sorted(events, key=lambda e: e["ts"]):
        found.append({"name": e["name"], "grid": e["args"]["grid"], "block": e["args"]["block"]})


def rel_err(a, b, floor=0.0):
    a = np.asarray(a, np.float64).ravel()
    b = np.asarray(b, np.float64).ravel()
    return float(np.abs(a - b).max() / max(np.abs(b).max(), floor, 1e-300))


PARITY_LOG = os.environ.get("ASTEROID_PARITY_LOG")       # file for the records of `compare`, if wanted


def _log_records(case, records):
    """One JSON line per compared tensor, appended to the file that ASTEROID_PARITY_LOG names."""
    if not case or not PARITY_LOG:
        return
    with open(PARITY_LOG, "a") as f:
        for r in records:
            f.write(json.dumps(dict(case=case, **r)) + "\n")


CONTRACT, MIRROR, CALIBRATED = "contract", "mirror", "calibrated"
# Calibrated criterion: factors by which a tensor's error against the plain oracle may exceed the mirroring oracle's own
# (max-norm, L2).  Measured over all deep bfloat16 cases of this suite the ratios have median 0.99 / 1.00; tensors of at
# least 1000 elements stay below 1.33 / 1.08, while the ratio of two error norms over a few dozen elements (BatchNorm
# parameters of narrow layers, the 3x3x3 stem) scatters up to 2.4 / 1.7.
CAL_BIG, CAL_SMALL, CAL_SIZE = (1.5, 1.15), (3.0, 2.0), 1000
ALL = (CONTRACT, MIRROR, CALIBRATED)


def compare(gpu, plain, net, first, last, tol, need_dx=True, mirror=None, allow=(CONTRACT,), outlier_frac=0.0, outlier_cap=0.05,
            case=None, contract_kinds=("y", "loss")):
    """Judges every tensor of a round (each y_m, dx_m, loss_m; accumulated gradient, momentum and weights, parameter
    tensor by parameter tensor) and returns {"records": [...], "counts": {criterion: n}, kind: worst contract error}.

    `plain` is the round of the plain float64 oracle: the contract.  The metric is max|gpu-ref| / max|ref| per tensor;
    parameter tensors use a denominator floored at 1% of the largest entry of their kind, so that a tensor whose
    true value vanishes (a beta gradient in front of another BatchNorm) is judged on the scale of its siblings.

    A tensor passes by the first criterion it meets; `allow` lists the ones a test accepts; tensors of the kinds in
    `contract_kinds` (by default the activations y and the losses) must meet the contract whatever `allow` says:
      contract    error against `plain` <= tol.
      mirror      (diagnostic; needs `mirror`, the float64 oracle that rounds at the bfloat16 storage points and rounds
                  the operands of dense contractions) error against `mirror` <= tol, where up to `outlier_frac` of the
                  elements may exceed tol but never `outlier_cap`.  ReLU/ReLU6 masks are decisions taken on stored
                  values; this oracle takes them on the same rounded values the library sees.
      calibrated  (diagnostic) the library is no further from `plain` than the storage format alone puts the
                  mirroring oracle: max-norm error <= 1.5x and L2 error <= 1.15x the mirror's own (3x / 2x for tensors of fewer
                  than 1000 elements, where a ratio of two error norms is itself noisy).
    """
    records, counts, worst = [], {CONTRACT: 0, MIRROR: 0, CALIBRATED: 0}, {}

    def norms(a, b, floor):
        scale = max(np.abs(b).max(), floor, 1e-300)
        err = np.abs(a - b) / scale
        l2 = float(np.linalg.norm(a - b) / max(np.linalg.norm(b), floor * np.sqrt(b.size), 1e-300))
        return err, l2

    def note(kind, name, a, p, m, floor=0.0):
        must_contract = kind in contract_kinds
        a = np.asarray(a, np.float64).ravel()
        p = np.asarray(p, np.float64).ravel()
        assert np.isfinite(a).all(), "%s: non-finite values" % name
        err_p, l2_p = norms(a, p, floor)
        rec = {"tensor": name, "kind": kind, "n": int(a.size), "err_plain": float(err_p.max()), "l2_plain": l2_p}
        ok = None
        if rec["err_plain"] <= tol:
            ok = CONTRACT
        if m is not None:
            m = np.asarray(m, np.float64).ravel()
            err_m, l2_m = norms(a, m, floor)
            mp, l2_mp = norms(m, p, floor)
            bad = int((err_m > tol).sum())
            rec.update(err_mirror=float(err_m.max()), l2_mirror=l2_m, mirror_vs_plain=float(mp.max()), l2_mirror_vs_plain=l2_mp,
                       outliers=bad)
            if ok is None and (bad == 0 or (bad <= outlier_frac * err_m.size and float(err_m.max()) <= outlier_cap)):
                ok = MIRROR
            cm, cl = CAL_BIG if a.size >= CAL_SIZE else CAL_SMALL
            if ok is None and rec["err_plain"] <= cm * rec["mirror_vs_plain"] and l2_p <= cl * l2_mp:
                ok = CALIBRATED
        rec["criterion"] = ok or "FAIL"
        records.append(rec)
        accepted = (CONTRACT,) if must_contract else allow
        if ok in accepted:
            counts[ok] += 1
            worst[kind] = max(worst.get(kind, 0.0), rec["err_plain"])
            return None
        return "%s: %s (accepted: %s) %s" % (name, rec["criterion"], "/".join(accepted), {k: ("%.3e" % v if isinstance(v, float) else v)
                                                                                         for k, v in rec.items() if k not in ("tensor", "kind")})

    fails = []
    M_ = mirror
    for m in range(len(plain["y"])):
        fails.append(note("y", "y[%d]" % m, gpu["y"][m], plain["y"][m], M_ and M_["y"][m]))
        if need_dx:
            fails.append(note("dx", "dx[%d]" % m, gpu["dx"][m], plain["dx"][m], M_ and M_["dx"][m]))
        fails.append(note("loss", "loss[%d]" % m, [gpu["loss"][m]], [plain["loss"][m]], M_ and [M_["loss"][m]]))
    for kind in ("G", "v", "w"):
        kmax = np.abs(plain[kind]).max()
        off = 0
        for i, pname, shape in si.param_layout(net, first, last):
            n = int(np.prod(shape))
            sl = slice(off, off + n)
            off += n
            fails.append(note(kind, "%s[%d.%s]" % (kind, i, pname), gpu[kind][sl], plain[kind][sl], M_ and M_[kind][sl], floor=1e-2 * kmax))
    _log_records(case, records)
    fails = [f for f in fails if f]
    assert not fails, "%d tensors fail:\n%s" % (len(fails), "\n".join(fails[:12]))
    worst["records"] = records
    worst["counts"] = counts
    return worst


def summary(worst):
    """Short printable form of compare's result."""
    return {k: ("%.2e" % v if isinstance(v, float) else v) for k, v in worst.items() if k != "records"}


def sampled_round_check(net, first, last, h, w, B, M, loss, bf16, sample, tol, seed=0, need_dx=1, lr=0.01, mu=0.9,
                        outlier_frac=0.0, allow=(CONTRACT,), case=None, contract_kinds=("y", "loss")):
    """Full-size round on the GPU (all M micro-batches); the oracle computes only the micro-batches
    in `sample` (micro-batches are independent given the weights: BatchNorm statistics are per
    micro-batch), and the rest of the round is checked through what holds at any size:
    G is the float32 running sum of the per-micro-batch gradients in backward order (bit-exact),
    v = G/M and w = w0 - lr*v from zero momentum."""
    xs, tg, params, _ = make_inputs(net, first, last, h, w, B, M, loss, seed, bf16)
    gpu = gpu_round(net, first, last, h, w, B, M, loss, xs, tg, params, bf16, lr=lr, mu=mu, need_dx=need_dx, export_micro=True)
    acc = np.zeros_like(gpu["G"])
    for m in range(M):
        acc = acc + gpu["g"][m]                      # float32, same order as the library
    assert np.array_equal(acc, gpu["G"]), "accumulated gradient is not the running float32 sum of the micro-batch gradients"
    v_expect = gpu["G"].astype(np.float64) / M
    assert np.abs(gpu["v"] - v_expect).max() <= 1e-6 * max(np.abs(v_expect).max(), 1e-30)
    w_expect = params.astype(np.float64) - lr * v_expect
    assert np.abs(gpu["w"] - w_expect).max() <= 2e-7 * np.abs(w_expect).max()
    S = len(sample)
    sx, st = [xs[m] for m in sample], [tg[m] for m in sample]
    plain = oracle_round(net, first, last, B, S, loss, sx, st, params, lr=lr, mu=mu)
    mirror = oracle_round(net, first, last, B, S, loss, sx, st, params, lr=lr, mu=mu, store=bf16_store) if bf16 else None
    Gs = np.sum([gpu["g"][m].astype(np.float64) for m in sample], axis=0)
    sub = {"y": [gpu["y"][m] for m in sample], "dx": [gpu["dx"][m] for m in sample], "loss": [gpu["loss"][m] for m in sample],
           "G": Gs, "v": Gs / S, "w": params.astype(np.float64) - lr * Gs / S}
    return compare(sub, plain, net, first, last, tol, need_dx=need_dx != 0, mirror=mirror, allow=allow, outlier_frac=outlier_frac, case=case,
                   contract_kinds=contract_kinds)
