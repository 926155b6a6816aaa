"""The work a user of the stage library has it do, as cases that can be prepared, run and compared.

One pass is one HPP-Round of a stage through the public calls: forward of every micro-batch with its loss head, backward
and accumulation of every micro-batch, one SGD-momentum update.  A case names a network of `stage_inputs`, the part of it the
stage holds, the image size, the micro-batch size, the micro-batches per round, the storage type, the order of the
calls and how they are issued:

  net, parts, part   layer range: the whole network, or part `part` of its cut into `parts` stages at block boundaries
                     (MobileNetV2 only; the cut minimises the largest stage's multiply-adds at the reference image size)
  size_h, size_w     height and width of the WHOLE network's input image (a part sees the map that reaches it)
  batch, micro       samples per micro-batch, micro-batches per round
  dtype              "f32" or "bf16" (storage of activations and activation gradients)
  resident           micro-batches that may wait for their backward: `micro` = all forwards first, fewer = 1F1B order with
                     that many activation slots (what a stage of a running pipeline does)
  issue              "calls": every call of the round is made from the host, as a pipeline runtime does that receives each
                     micro-batch from its neighbour; "graph": the round was captured once into a CUDA graph and is
                     replayed, as a single-GPU training loop does

A stage that starts at layer 0 of a whole classifier network computes no input gradient; a stage that ends with the
classifier has the softmax cross-entropy head, every other one the MSE head.
"""
import math
import random

import numpy as np
import torch

import paper_2408_08015_b200 as P
import stage_inputs as si
from paper_2408_08015_b200.dp import grad_tensor

LR, MOMENTUM = 0.01, 0.9
NETS = {
    "inverted_residual": lambda: si.block_net(16, 6),
    "mobilenetv2_stage": si.stage_net_mbv2_4blocks,
    "mobilenetv2": si.mobilenetv2_net,
    "resnet50_c2c3": si.resnet50_c2c3_net,
    "efficientnet_b1_stage": si.efficientnet_b1_stage_net,
}
CUT_SIZE = 224                # image size the cut of MobileNetV2 into parts is computed for


def _case(net, size, batch, micro, dtype="bf16", parts=1, part=0, resident=0, issue="calls", name=None):
    h, w = size
    c = {"net": net, "parts": parts, "part": part, "size_h": h, "size_w": w, "batch": batch, "micro": micro, "dtype": dtype,
         "resident": resident or micro, "issue": issue}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest round in use: one inverted-residual block in float32 on a 32x32 map (launches and host time)
        _case("inverted_residual", (32, 32), 8, 4, "f32", name="block_f32"),
        # one of six stages of MobileNetV2 on a device that gets few samples of each micro-batch: small maps, many launches,
        # calls issued one by one in the order of a pipeline stage with three resident micro-batches
        _case("mobilenetv2", (224, 224), 4, 8, parts=6, part=2, resident=3, name="mbv2_6th_b4_1f1b"),
        # the same cut's 7x7 / 14x14 stage, replayed from a graph
        _case("mobilenetv2", (224, 224), 4, 8, parts=6, part=4, issue="graph", name="mbv2_6th_late_b4_graph"),
        # second half of MobileNetV2 with the classifier and the cross-entropy head
        _case("mobilenetv2", (224, 224), 16, 8, parts=2, part=1, name="mbv2_half_head_b16"),
        # a stage on an odd-sized map with an odd micro-batch (an uneven data-parallel share), 1F1B with two slots
        _case("mobilenetv2_stage", (57, 45), 5, 3, resident=2, name="mbv2_stage_ragged"),
        # the same stage in float32
        _case("mobilenetv2_stage", (56, 56), 8, 4, "f32", name="mbv2_stage_f32"),
        # four inverted-residual blocks at 56x56, the ordinary single-GPU stage, replayed from a graph
        _case("mobilenetv2_stage", (56, 56), 32, 8, issue="graph", name="mbv2_stage_b32_graph"),
        # a whole MobileNetV2 on small images of an odd size: maps down to 4x3
        _case("mobilenetv2", (115, 96), 8, 2, name="mbv2_small_images_b8"),
        # a whole MobileNetV2 on 224x224 images
        _case("mobilenetv2", (224, 224), 16, 4, name="mbv2_imagenet_b16"),
        # squeeze-excite, SiLU and 5x5 depthwise
        _case("efficientnet_b1_stage", (56, 56), 32, 8, name="effnet_stage_b32"),
        # dense bottlenecks: a small odd share, and the largest round
        _case("resnet50_c2c3", (45, 43), 6, 2, name="resnet_ragged_b6"),
        _case("resnet50_c2c3", (56, 56), 32, 8, name="resnet_b32"),
    ]


def draw(rng):
    """A case of the listed ranges: any network, part, order and issue; image sizes odd and even from a quarter of the usual
    area or less up to the usual one, micro-batches of 1 to 32 samples, 1 to 8 of them per round.  BatchNorm keeps at least 64
    values a channel, and no case costs more than the largest listed one."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    net = rng.choice(sorted(NETS))
    low, top = {"inverted_residual": (14, 64), "mobilenetv2": (96, 224)}.get(net, (14, 56))
    size = (log_int(low, top), log_int(low, top))
    dtype = "f32" if net in ("inverted_residual", "mobilenetv2_stage") and rng.random() < 0.5 else "bf16"
    # the parts a pipeline of 2 to 6 stages has; of the two halves the one with the head (the other is the whole network's)
    parts, part = rng.choice([(1, 0), (2, 1), (3, 1), (3, 2)] + [(4, i) for i in range(4)] + [(6, i) for i in range(6)]) if net == "mobilenetv2" else (1, 0)
    batch, micro = log_int(1, 32), rng.randint(1, 8)
    if net == "mobilenetv2" and parts == 1:
        micro = (micro + 1) // 2
    c = _case(net, size, batch, micro, dtype, parts, part, rng.randint(1, micro), rng.choice(["calls", "calls", "graph"]))
    while c["batch"] > 1 and _cost(c) > _cost_limit():
        c["batch"] //= 2
    while c["batch"] * _smallest_map(c) < 64:
        c["batch"] += 1
    return c


class _Plan:
    """Layer range, input map and output shape of a case's stage."""

    def __init__(self, c):
        self.net = NETS[c["net"]]()
        self.image = (c["size_h"], c["size_w"])
        self.first, self.last = 0, len(self.net) - 1
        if c["parts"] > 1:
            self.first, self.last = si.partition_units(self.net, si.mobilenetv2_units(), c["parts"], CUT_SIZE, CUT_SIZE)[c["part"]]
        shapes = si.out_shape(self.net, 0, len(self.net) - 1, c["size_h"], c["size_w"])
        self.h, self.w, self.c_in = shapes[self.first - 1]
        self.shapes = {i: shapes[i] for i in range(self.first, self.last + 1)}
        self.out = shapes[self.last]
        classifier = c["net"] == "mobilenetv2"
        self.need_dx = not (classifier and self.first == 0)
        self.xent = classifier and self.last == len(self.net) - 1


def _macs_and_conv_elems(plan):
    """Multiply-adds and raw conv outputs of one sample."""
    macs = si.forward_macs(plan.net, 0, plan.last, *plan.image)
    convs = [i for i in plan.shapes if plan.net[i].op in ("conv", "dwconv", "linear")]
    elems = sum(int(np.prod(plan.shapes[i])) for i in convs)
    skipped = 0 if plan.need_dx else macs[plan.first]          # the first conv of a network has no input gradient
    return sum(macs[i] for i in convs), skipped, elems


def work(case):
    """Operations: two per multiply-add of every conv and linear layer, forward, input gradient and weight gradient.  Bytes:
    inputs, targets, outputs and input gradients once; every raw conv output written and read in the forward and read in the
    backward, its gradient written and read (BatchNorm's statistics, and the two sums of its backward, stand between a
    tensor and its consumer, and the tensors of a round are larger than the chip's memories); parameters, momentum and
    gradients of the update."""
    p = _Plan(case)
    macs, skipped, elems = _macs_and_conv_elems(p)
    n, e = case["batch"] * case["micro"], (4 if case["dtype"] == "f32" else 2)
    n_in, n_out = p.h * p.w * p.c_in, int(np.prod(p.out))
    params = si.param_count(p.net, p.first, p.last)
    io = n_in * (2 if p.need_dx else 1) + n_out * (1 if p.xent else 2)
    return {"bytes": float(n * e * (io + 5 * elems) + 4 * params * (2 * case["micro"] + 5)), "flops": 2.0 * n * (3 * macs - skipped)}


def tolerance(case):
    return {"rel": 3e-2} if case["dtype"] == "bf16" else {"rel": 1e-4}


def _smallest_map(case):
    p = _Plan(case)
    return min(h * w for i, (h, w, _) in p.shapes.items() if p.net[i].op == "bn")


def _cost(case):
    """A round's time in arbitrary units: float32 runs on the vector units, bfloat16 contractions on the tensor cores."""
    w = work(case)
    return w["bytes"] + w["flops"] * (3.0 if case["dtype"] == "f32" else 0.02)


def _cost_limit():
    return _cost(listed()[-1])


class _State:
    def __init__(self, case, seed):
        p = self.plan = _Plan(case)
        B, M = case["batch"], case["micro"]
        self.micro, self.resident, self.bf16 = M, case["resident"], case["dtype"] == "bf16"
        self.batch, self.classes = B, p.out[2]
        self.dtype = P.AST_BF16 if self.bf16 else P.AST_F32
        dt = torch.bfloat16 if self.bf16 else torch.float32
        dev = torch.device("cuda", torch.cuda.current_device())
        gen = torch.Generator(device=dev)
        gen.manual_seed(int(seed))
        normal = lambda *shape: torch.randn(shape, generator=gen, device=dev).to(dt)   # noqa: E731
        self.x = [normal(B, p.h, p.w, p.c_in) for _ in range(M)]
        if p.xent:
            self.t = [torch.randint(0, p.out[2], (B,), generator=gen, device=dev, dtype=torch.int32) for _ in range(M)]
        else:
            self.t = [normal(B, *p.out) for _ in range(M)]
        self.y = [torch.empty((B,) + tuple(p.out), device=dev, dtype=dt) for _ in range(M)]
        self.dy = [torch.empty_like(y) for y in self.y]
        self.dx = [torch.empty_like(x) for x in self.x] if p.need_dx else []
        self.loss = torch.zeros(M, device=dev)
        self.handle = P.asteroid_stage_create(p.net, p.first, p.last, p.h, p.w, B, M, dtype=self.dtype, slots=self.resident, need_input_grad=int(p.need_dx))
        P.asteroid_stage_import_state(self.handle, _parameters(p, seed))
        self.arena = grad_tensor(self.handle)      # the accumulated gradients, where a data-parallel group sums them
        self.grad = torch.empty_like(self.arena)
        self.graph = None
        if case["issue"] == "graph":
            _round(self)                                # first-use set-up happens outside the capture
            torch.cuda.synchronize()
            self.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(self.graph, capture_error_mode="thread_local"):
                _round(self)
            torch.cuda.synchronize()

    def __del__(self):
        self.graph = None
        if getattr(self, "handle", None) is not None:
            P.asteroid_stage_destroy(self.handle)
            self.handle = None


def _parameters(p, seed):
    """Flat parameter vector: Kaiming-uniform weights; BatchNorms as in a network under training, each channel with a scale and an
    offset of its own.  One channel in eight is off; the others lie well inside the linear region of their activation.  (With
    offsets of 0 a bfloat16 comparison says nothing: an activation at its kink is decided by the last bit, 0.2 % of them
    by any reordering of a sum, and the input gradients of two correct implementations then differ by 6 % a layer.)"""
    rng = np.random.default_rng(int(seed))

    def uniform(n, lo, hi):
        return np.float32(lo) + np.float32(hi - lo) * rng.random(n, dtype=np.float32)

    flat = []
    for i, name, shape in si.param_layout(p.net, p.first, p.last):
        n, layer = int(np.prod(shape)), p.net[i]
        if name in ("weight", "w1", "w2"):
            fan_in = {"conv": layer.k * layer.k * layer.c_in, "dwconv": layer.k * layer.k}.get(layer.op, shape[-1])
            flat.append(uniform(n, -1, 1) * np.float32(math.sqrt(6 / fan_in)))
        elif name in ("gamma", "beta"):
            role = _bn_role(p.net, i)
            if name == "gamma":
                flat.append(uniform(n, *{"activation": (0.4, 0.6), "residual": (0.1, 0.2)}.get(role, (0.3, 0.5))))
            elif role == "activation":
                flat.append(np.where(rng.random(n) < 0.125, uniform(n, -6.0, -5.0), uniform(n, 2.7, 3.3)))
            else:
                flat.append(uniform(n, *{"shortcut": (1.3, 1.7), "residual": (-0.2, 0.2)}.get(role, (-0.5, 0.5))))
        else:
            flat.append(np.zeros(n, np.float32))
    return np.concatenate(flat)


def _bn_role(net, i):
    """What follows the BatchNorm at layer i: a ReLU or ReLU6; a residual sum with a ReLU, whose other operand is the projection
    shortcut's BatchNorm or the block's input; anything else."""
    if i + 1 < len(net) and net[i + 1].op in ("relu", "relu6"):
        return "activation"
    for j in range(i + 1, min(i + 4, len(net) - 1)):
        if net[j].op == "add" and net[j + 1].op == "relu" and i in (net[j].src, net[j].add_from):
            return "shortcut" if net[net[j].src + net[j].add_from - i].op == "bn" else "residual"
    return "plain"


def prepare(case, seed):
    return _State(case, seed)


def _forward(s, m, stream):
    P.asteroid_stage_forward(s.handle, m, s.x[m].data_ptr(), s.y[m].data_ptr(), stream)
    loss = s.loss.data_ptr() + 4 * m
    if s.plan.xent:
        P.asteroid_loss_softmax_xent(s.y[m].data_ptr(), s.t[m].data_ptr(), s.batch, s.classes, s.dtype, s.dy[m].data_ptr(), loss, stream)
    else:
        P.asteroid_loss_mse(s.y[m].data_ptr(), s.t[m].data_ptr(), s.y[m].numel(), s.dtype, s.dy[m].data_ptr(), loss, stream)


def _backward(s, m, stream):
    P.asteroid_stage_backward(s.handle, m, s.dy[m].data_ptr(), s.dx[m].data_ptr() if s.dx else None, stream)
    P.asteroid_stage_accumulate(s.handle, m, stream)


def _round(s):
    stream = torch.cuda.current_stream().cuda_stream
    for m in range(s.micro):
        if m >= s.resident:                             # 1F1B: the oldest resident micro-batch makes room
            _backward(s, m - s.resident, stream)
        _forward(s, m, stream)
    for m in range(max(0, s.micro - s.resident), s.micro):
        _backward(s, m, stream)
    s.grad.copy_(s.arena)                               # what a training loop logs or clips by, and a group reduces
    P.asteroid_stage_step(s.handle, LR, MOMENTUM, stream)


def run(state):
    if state.graph is not None:
        state.graph.replay()
    else:
        _round(state)
    return {"y": state.y, "dx": state.dx, "loss": state.loss, "grad": state.grad}
