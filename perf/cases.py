"""What a user of this library has it do, as cases that can be timed.

A case is a dict of plain values.  "step" cases train (or score) a whole network through `Model`: the layer list, the
cuts, the micro-batches and the fp32 buffers are the user's, a pass is one step.  "conv", "bn" and "update" cases are the
single-op entry points, for callers that bring their own training loop.  `listed()` names the standing ones, `draw(rng)`
gives more of the same ranges; both directions run in every case that has two.
"""
import math

import torch

import paper_1911_05146_b200 as hpf
from paper_1911_05146_b200 import ADD, BN, BNRELU, CONV, HEAD, MAXPOOL, RELU

EPS = 1e-5


# ---- layer lists: (kind, src0, src1, c_in, c_out, ksize, stride, pad, eps) -----------------------------------------
def _conv(ops, src, ci, co, k, s=1):
    ops.append((CONV, src, -1, ci, co, k, s, k // 2, 0.0))
    return len(ops) - 1


def _same(ops, kind, src, c, src1=-1):
    ops.append((kind, src, src1, c, c, 0, 1, 0, EPS if kind in (BN, BNRELU) else 0.0))
    return len(ops) - 1


def _pool(ops, src, c, k, s, pad):
    ops.append((MAXPOOL, src, -1, c, c, k, s, pad, 0.0))
    return len(ops) - 1


def _bottlenecks(ops, t, c, widths, outs, blocks):
    """Pre-activation bottleneck stages; every stage but the first starts with a stride of 2."""
    for stage, (w, co, count) in enumerate(zip(widths, outs, blocks)):
        for b in range(count):
            s = 2 if stage and not b else 1
            v = _conv(ops, _same(ops, BNRELU, t, c), c, w, 1, s)
            v = _conv(ops, _same(ops, BNRELU, v, w), w, w, 3)
            v = _conv(ops, _same(ops, BNRELU, v, w), w, co, 1)
            short = t if b else _conv(ops, t, c, co, 1, s)
            t, c = _same(ops, ADD, v, co, short), co
    return _same(ops, BNRELU, t, c), c


def _net(case):
    """The case's layer list: v2 = pre-activation bottlenecks on small maps (depth 9n+2), v2k = the same with the Keras
    example's widths, v1 = post-activation basic blocks (depth 6n+2), vgg16, imagenet = 7x7 stem and 3x3 max-pool."""
    ops, n = [], case["n"]
    if case["net"] in ("v2", "v2k"):
        widths = (16, 32, 64) if case["net"] == "v2" else (16, 64, 128)
        t, c = _bottlenecks(ops, _conv(ops, -1, 3, 16, 3), 16, widths, (64, 128, 256), (n, n, n))
    elif case["net"] == "v1":
        t, c = _same(ops, BNRELU, _conv(ops, -1, 3, 16, 3), 16), 16
        for w in (16, 32, 64):
            for b in range(n):
                s = 2 if w != c else 1
                v = _same(ops, BNRELU, _conv(ops, t, c, w, 3, s), w)
                v = _same(ops, BN, _conv(ops, v, w, w, 3), w)
                short = t if s == 1 else _conv(ops, t, c, w, 1, s)
                t, c = _same(ops, RELU, _same(ops, ADD, v, w, short), w), w
    elif case["net"] == "vgg16":
        t, c = -1, 3
        for w, k in zip((64, 128, 256, 512, 512), (2, 2, 3, 3, 3)):
            for _ in range(k):
                t, c = _same(ops, RELU, _conv(ops, t, c, w, 3), w), w
            t = _pool(ops, t, c, 2, 2, 0)
        for _ in range(2):
            t, c = _same(ops, RELU, _conv(ops, t, c, 4096, 1), 4096), 4096
    else:
        t = _conv(ops, -1, 3, 64, 7, 2)
        blocks = (3, 8, 36, 3) if n == 36 else (3, 4, n, 3)
        t, c = _bottlenecks(ops, _pool(ops, t, 64, 3, 2, 1), 64, (64, 128, 256, 512), (256, 512, 1024, 2048), blocks)
    ops.append((HEAD, t, -1, c, _classes(case), 0, 1, 0, 0.0))
    return ops


def _classes(case):
    return 1000 if case["net"] == "imagenet" else 10


def _map_sizes(ops, size):
    """Side of every layer's output map."""
    out = []
    for kind, src, _, _, _, k, s, pad, _ in ops:
        h = size if src < 0 else out[src]
        out.append(1 if kind == HEAD else (h + 2 * pad - k) // s + 1 if kind in (CONV, MAXPOOL) else h)
    return out


def _weights(op):
    kind, _, _, ci, co, k = op[:6]
    return co * k * k * ci if kind == CONV else co * ci if kind == HEAD else ci if kind in (BN, BNRELU) else 0


def _biases(op):
    return op[4] if op[0] == HEAD else op[3] if op[0] in (BN, BNRELU) else 0


# ---- the cases -------------------------------------------------------------------------------------------------------
def _step(name, net, n, size, batch, micro, parts, mode):
    return {"name": name, "kind": "step", "net": net, "n": n, "size": size, "batch": batch, "micro": micro, "parts": parts, "mode": mode}


def _layer(name, k, stride, c_in, c_out, size, batch, path):
    return {"name": name, "kind": "conv", "ksize": k, "stride": stride, "c_in": c_in, "c_out": c_out, "size": size, "batch": batch, "path": path}


def listed():
    return [
        # the first thing anybody runs: the smallest network, where launches and latency are all there is
        _step("step_resnet11_b8", "v2", 1, 32, 8, 2, 2, "average"),
        # a short network on maps and micro-batches that divide nothing evenly, trained with the fused update
        _step("step_resnet29_ragged", "v2", 3, 27, 42, 3, 3, "sgd"),
        # the everyday training run on small images: gradient average and momentum update in one call
        _step("step_resnet110_b128", "v2", 12, 32, 128, 4, 4, "sgd"),
        # the network the method was made for: too deep for anything but partitions and micro-batches
        _step("step_resnet1001_b128", "v2", 111, 32, 128, 8, 8, "average"),
        # large images, wide layers, a thousand classes
        _step("step_resnet152_b64", "imagenet", 36, 224, 64, 4, 4, "average"),
        # no batch norm, wide 3x3 convolutions, large fully connected layers
        _step("step_vgg16_b128", "vgg16", 0, 32, 128, 4, 4, "sgd"),
        # a data loader's pinned host batch in, the loss back on the host, every step
        _step("step_resnet110v1_host_b128", "v1", 18, 32, 128, 4, 4, "host"),
        # scoring a large batch: forward only, logits and losses read
        _step("score_resnet182_wide_b256", "v2k", 20, 32, 256, 4, 4, "forward"),
        # one layer's forward, data gradient and weight gradient in a caller's own loop: bound by the tensor cores
        _layer("conv3x3_128_16x16_b128", 3, 1, 128, 128, 16, 128, 0),
        # the same, bound by memory, in the single-pass precision such callers may choose
        _layer("conv1x1_64to256_56x56_b64", 1, 1, 64, 256, 56, 64, 2),
        # batch norm with ReLU, forward and backward, of an activation larger than the L2 cache
        {"name": "bnrelu_256_56x56_b64", "kind": "bn", "rows": 64 * 56 * 56, "channels": 256},
        # the update of a model of 60 M parameters from four micro-batches' gradients
        {"name": "update_60m", "kind": "update", "micro": 4, "params": 60185128},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["step"] * 8 + ["conv"] * 2 + ["bn", "update"])
    if what == "conv":
        k = rng.choice((1, 3))
        case = _layer("", k, rng.choice((1, 1, 2)) if k == 1 else 1, rng.choice((16, 32, 48, 64, 96, 128, 256, 512)),
                      rng.choice((16, 32, 48, 64, 96, 128, 256, 512)), _log(rng, 4, 56), _log(rng, 4, 128), rng.choice((0, 2)))
    elif what == "bn":
        case = {"kind": "bn", "rows": _log(rng, 200, 200704), "channels": rng.choice((16, 32, 64, 96, 128, 256))}
    elif what == "update":
        case = {"kind": "update", "micro": rng.choice((1, 2, 3, 4, 8)), "params": _log(rng, 100_000, 30_000_000)}
    else:
        largest = work(next(c for c in listed() if c["name"] == "step_resnet1001_b128"))
        while True:
            net = rng.choice(("v2", "v2", "v2", "v2k", "v1", "vgg16", "imagenet"))
            n = {"vgg16": 0, "imagenet": rng.choice((6, 23, 36)), "v1": _log(rng, 1, 18)}.get(net) or (_log(rng, 1, 111) if net != "vgg16" else 0)
            size = rng.choice((96, 128, 161, 192, 224)) if net == "imagenet" else 32 if net == "vgg16" else rng.choice((32, 32, 32, 24, 28, 27, 40))
            micro, parts = rng.choice((1, 2, 3, 4, 8)), rng.randint(1, 8)
            case = _step("", net, n, size, micro * _log(rng, 2, 64), micro, parts, rng.choice(("average", "sgd", "sgd", "host", "forward")))
            w = work(case)
            if len(_net(case)) * micro <= 2337 * 8 and 1e6 <= w["bytes"] <= largest["bytes"] / 2 and w["flops"] <= 2 * largest["flops"] and case["batch"] <= 256:
                break
    case.pop("name", None)
    return case


# ---- inputs ----------------------------------------------------------------------------------------------------------
_streams = []


def _kept_streams(n):
    """A program makes its streams once and orders every model's steps on them."""
    while len(_streams) < n:
        _streams.append(torch.cuda.Stream())
    return _streams[:n]


def _draw_params(ops, normal):
    """Flat parameters: He-normal weights, batch norm scales around 1 and shifts around 0, head biases 0.  A weight in
    front of a batch norm only grows under plain SGD (its gradient is orthogonal to it): twice He's size, as some way into
    training."""
    gain = 2.0 if any(op[0] in (BN, BNRELU) for op in ops) else 1.0
    scale, shift, counts = [], [], []
    for op in ops:
        kind, _, _, ci, _, k = op[:6]
        norm = kind in (BN, BNRELU)
        he = math.sqrt(2.0 / (ci * max(k, 1) ** 2)) * (gain if kind == CONV else 1.0)
        for count, s, m in ((_weights(op), 0.1 if norm else he, 1.0 if norm else 0.0), (_biases(op), 0.1 if norm else 0.0, 0.0)):
            if count:
                scale.append(s), shift.append(m), counts.append(count)
    counts = torch.tensor(counts, device="cuda")
    spread = lambda v: torch.repeat_interleave(torch.tensor(v, device="cuda"), counts)  # noqa: E731
    return spread(scale) * normal(int(counts.sum())) + spread(shift)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    normal = lambda *shape: torch.randn(*shape, generator=g, device="cuda")  # noqa: E731
    s = {"case": case}
    if case["kind"] == "step":
        ops, B, M, P, size = _net(case), case["batch"], case["micro"], case["parts"], case["size"]
        model = hpf.Model(ops, (B, size, size, 3), [p * len(ops) // P for p in range(1, P)], M)
        s["params"] = _draw_params(ops, normal)
        s["avg"] = torch.empty(model.num_params(), device="cuda")
        slots = torch.empty((M, model.num_params()), device="cuda")
        ws = torch.empty(model.workspace_bytes(), dtype=torch.uint8, device="cuda")
        s["x"], s["labels"] = normal(B, size, size, 3), torch.randint(_classes(case), (B,), generator=g, device="cuda", dtype=torch.int32)
        if case["mode"] == "host":
            s["x"], s["labels"] = s["x"].cpu().pin_memory(), s["labels"].cpu().pin_memory()
        if case["mode"] == "sgd":
            s["velocity"] = torch.zeros_like(s["avg"])
        torch.cuda.synchronize()
        model.bind(s["params"], slots, s["avg"], ws, _kept_streams(3 * model.num_stream_slots()))
        s["model"] = model
        inside = lambda p, *shape: ws[p - ws.data_ptr():][:4 * math.prod(shape)].view(torch.float32).reshape(shape)  # noqa: E731
        s["losses"] = inside(model.loss_slots_ptr(), M)
        s["logits"] = [inside(p, *shape) for p, shape in (model.tensor_ptr(len(ops) - 1, m) for m in range(M))]
    elif case["kind"] == "conv":
        N, H, C, K, R, st = (case[k] for k in ("batch", "size", "c_in", "c_out", "ksize", "stride"))
        Q = (H - 1) // st + 1
        s["args"] = (N, H, H, C, K, R, st, R // 2, case["path"])
        s["x"], s["dy"] = normal(N, H, H, C), normal(N, Q, Q, K)
        s["w"] = normal(K, R, R, C) * math.sqrt(2.0 / (C * R * R))
        s["y"], s["dx"], s["dw"] = torch.empty_like(s["dy"]), torch.empty_like(s["x"]), torch.empty_like(s["w"])
        s["wprep"] = torch.empty(4 * s["w"].numel(), device="cuda")
        s["scratch"] = torch.zeros(hpf.conv_scratch_bytes(*s["args"][:8]), dtype=torch.uint8, device="cuda")
        hpf.conv_prepare_weights(s["w"], s["wprep"], C, K, R)
    elif case["kind"] == "bn":
        rows, C = case["rows"], case["channels"]
        s["x"], s["dy"], s["shortcut"] = 3.0 * normal(rows, C) + 1.0, normal(rows, C), normal(rows, C)
        s["gamma"], s["beta"] = 1.0 + 0.1 * normal(C), 0.1 * normal(C)
        s["y"], s["dx"] = torch.empty_like(s["x"]), torch.empty_like(s["x"])
        s["stats"], s["dgamma"], s["dbeta"] = torch.empty(2 * C, device="cuda"), torch.empty(C, device="cuda"), torch.empty(C, device="cuda")
        s["scratch"] = torch.zeros(hpf.bnrelu_scratch_bytes(rows, C), dtype=torch.uint8, device="cuda")
    else:
        M, G = case["micro"], case["params"]
        s["slots"], s["params"], s["velocity"], s["avg"] = normal(M, G), normal(G), 0.1 * normal(G), torch.empty(G, device="cuda")
    return s


# ---- one pass --------------------------------------------------------------------------------------------------------
def run(s):
    case = s["case"]
    if case["kind"] == "step":
        model = s["model"]
        if case["mode"] == "host":
            return {"loss": model.step_host(s["x"], s["labels"]), "grad": s["avg"]}
        if case["mode"] == "forward":
            model.forward(s["x"], s["labels"])
            return {"losses": s["losses"], "logits": s["logits"]}
        model.forward_backward(s["x"], s["labels"])
        if case["mode"] == "sgd":
            model.sgd_momentum_step(s["velocity"], 1e-3, 0.9, 1e-4)
            return {"losses": s["losses"], "grad": s["avg"], "params": s["params"], "velocity": s["velocity"]}
        model.grad_average()
        return {"losses": s["losses"], "grad": s["avg"]}
    if case["kind"] == "conv":
        hpf.conv_fwd(s["x"], s["w"], s["wprep"], s["y"], *s["args"], s["scratch"])
        hpf.conv_dgrad(s["dy"], s["w"], s["wprep"], s["dx"], *s["args"], s["scratch"])
        hpf.conv_wgrad(s["x"], s["dy"], s["dw"], *s["args"], s["scratch"])
        return {"y": s["y"], "dx": s["dx"], "dw": s["dw"]}
    if case["kind"] == "bn":
        rows, C = case["rows"], case["channels"]
        hpf.bnrelu_fwd(s["x"], s["gamma"], s["beta"], EPS, s["y"], s["stats"], rows, C, s["scratch"])
        hpf.bnrelu_bwd(s["x"], s["dy"], s["gamma"], s["beta"], s["stats"], s["dx"], s["shortcut"], 0, s["dgamma"], s["dbeta"], rows, C, s["scratch"])
        return {"y": s["y"], "stats": s["stats"], "dx": s["dx"], "dgamma": s["dgamma"], "dbeta": s["dbeta"]}
    hpf.sgd_momentum_flat(s["slots"], s["avg"], s["params"], s["velocity"], case["micro"], case["params"], 1e-4, 0.9, 1e-4)
    return {"avg": s["avg"], "params": s["params"], "velocity": s["velocity"]}


def work(case):
    """Steps: every layer's output is written once and read once, its gradient as well (a convolution that only feeds a
    residual sum shares the sum's), parameters are read each way and every micro-batch's gradients written and read."""
    if case["kind"] == "conv":
        N, H, C, K, R = (case[k] for k in ("batch", "size", "c_in", "c_out", "ksize"))
        Q = (H - 1) // case["stride"] + 1
        x, y, w = N * H * H * C, N * Q * Q * K, K * R * R * C
        sampled = N * Q * Q * C                       # a strided 1x1 reads its samples only
        return {"bytes": 4.0 * (sampled + w + y + y + w + x + w), "flops": 6.0 * y * R * R * C}
    if case["kind"] == "bn":
        return {"bytes": 4.0 * case["rows"] * case["channels"] * 5, "flops": 15.0 * case["rows"] * case["channels"]}
    if case["kind"] == "update":
        return {"bytes": 4.0 * case["params"] * (case["micro"] + 5), "flops": case["params"] * (case["micro"] + 6.0)}
    ops, B = _net(case), case["batch"]
    size = _map_sizes(ops, case["size"])
    both = 0 if case["mode"] == "forward" else 1
    summed = {o[1] for o in ops if o[0] == ADD} | {o[2] for o in ops if o[0] == ADD}
    values = flops = params = 0
    for i, op in enumerate(ops):
        out = B * size[i] ** 2 * op[4]
        params += _weights(op) + _biases(op)
        if not (op[0] == CONV and i in summed):
            values += out
        if op[0] in (CONV, HEAD):
            flops += 2.0 * out * max(op[5], 1) ** 2 * op[3] * (1 if not both else 2 if op[1] < 0 else 3)
    update = {"forward": 0, "sgd": 5}.get(case["mode"], 1)
    return {"bytes": 4.0 * (B * case["size"] ** 2 * 3 + values * (2 + 2 * both) + params * (1 + both * (1 + 2 * case["micro"]) + update)), "flops": flops}


def tolerance(case):
    """Sums of fp32 products in another order differ by about 1e-5.  A whole step's gradients differ by more: the derivative
    of ReLU is a step, so a pre-activation within rounding of zero may fall on either side and moves its element of the
    gradient by all of it, the more so the deeper the network; and weight gradients take TF32 operands (11 bits)."""
    if case["kind"] == "conv":
        return {"rel": 5e-5, "max": 1e-3} if case["path"] == 0 else {"rel": 1e-3, "max": 1e-2}
    if case["kind"] == "bn":
        return {"rel": 1e-3, "max": 0.99}
    if case["kind"] == "update":
        return {"rel": 1e-6, "max": 1e-5}
    if case["mode"] == "forward":
        return {"rel": 5e-5, "max": 1e-3}
    return {"rel": 1e-2, "max": 0.9}
