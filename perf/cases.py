"""The work that a user of this library has it do, as cases that can be timed.

Three kinds, one per public entry point that does device work:

``train``   a run of consecutive ``Trainer.step`` calls on device-resident minibatches, ``flush``, and the
            last minibatch's loss (``get_loss``): what a training loop does between two log lines.
``gemm``    ``lp_gemm_bf16``: the three contractions of one fully connected layer (forward, delta, G) on the
            caller's buffers.
``xent``    ``lp_softmax_xent_static``: loss and output gradient of a batch of logits, as in a validation pass.

``listed()`` are the named cases, ``draw(rng)`` one more of the same ranges.  Networks are written as text:
``widths`` of a fully connected network, or ``plan`` of a VGG-type one ("P" = 2x2 max pool), or ``net`` = "sample"
for the strided 5x5 / 3x3 four-layer network, each with the image size ``hw``.
"""
import math

import numpy as np
import torch

from paper_2108_06629_b200 import binding
from paper_2108_06629_b200 import inputs


def _train(name, batch, stages, steps, lr, momentum=0.0, widths="", act="relu", plan="", fcs="", net="", hw=0, delays="",
           input="f32", schedule="layerpipe", recompute=False):
    return dict(name=name, kind="train", widths=widths, act=act, plan=plan, fcs=fcs, net=net, hw=hw, batch=batch, stages=stages,
                delays=delays, steps=steps, lr=lr, momentum=momentum, input=input, schedule=schedule, recompute=recompute)


VGG16 = "64,64,P,128,128,P,256,256,256,P,512,512,512,P,512,512,512,P"


def listed():
    mlp4 = dict(widths="784,256,256,256,10", batch=32, stages=4, delays="3,2,1,0", lr=0.01)
    small = dict(plan="64,64,P,128,128,P,256,256,P", fcs="512,10", hw=32, stages=7, lr=0.002)
    return [
        # a digit classifier trained online: one minibatch, then its loss (latency of a single step)
        _train("mlp4_784_one", steps=1, **mlp4),
        # the same network in its training loop: launch-bound, minibatches in flight
        _train("mlp4_784", steps=32, **mlp4),
        # features of a tabular set, nothing a multiple of a tile: GELU, momentum, bf16 inputs, batch 100
        _train("mlp_ragged", widths="1003,777,515,131", act="gelu", batch=100, stages=3, steps=16, lr=0.001, momentum=0.9,
               input="bf16"),
        # wide layers on a small batch: weights and optimiser state stream from memory
        _train("mlp8_4096", widths=",".join(["4096"] * 8 + ["1000"]), act="gelu", batch=256, stages=8, delays="7,6,5,4,3,2,1,0",
               steps=8, lr=0.001, momentum=0.9),
        # the largest network: tensor-bound contractions
        _train("mlp16_8192", widths=",".join(["8192"] * 17), act="gelu", batch=2048, stages=9, steps=4, lr=0.01),
        # a small convolutional network on 32 x 32 images
        _train("vgg_small_32", batch=128, steps=16, **small),
        # the same with the backward pass as one task per layer, bf16 images and half the batch
        _train("vgg_small_32_fused_b", batch=64, steps=16, input="bf16", schedule="fused_b", **small),
        # VGG-16 on full-size images
        _train("vgg16_224", plan=VGG16, fcs="4096,4096,1000", hw=224, batch=64, stages=9, steps=4, lr=0.001),
        # strided 5x5 / 3x3 convolutions of 3 to 128 channels
        _train("sample4_224", net="sample", hw=224, batch=32, stages=3, steps=8, lr=0.0005),
        # the contractions of one layer in isolation: ragged, and large
        dict(name="gemm_ragged", kind="gemm", batch=250, n_in=1000, n_out=513),
        dict(name="gemm_4096", kind="gemm", batch=1024, n_in=4096, n_out=4096),
        # validation loss of one large batch over 1000 classes
        dict(name="xent_8192_1000", kind="xent", batch=8192, classes=1000),
    ]


# ---- drawn cases ----------------------------------------------------------------------------------------
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_mlp(rng):
    depth = rng.randint(2, 10)
    base = _log_int(rng, 64, 8192)
    widths = [max(8, min(8192, int(base * rng.uniform(0.4, 1.4)))) for _ in range(depth)] + [rng.randint(2, 1000)]
    if rng.random() < 0.5:                      # half of them as people mostly size layers
        widths = [max(16, w // 16 * 16) for w in widths[:-1]] + widths[-1:]
    batch = _log_int(rng, 1, 2048)
    steps = rng.choice([1, 4, 8, 16] if batch >= 32 else [1, 4])     # (a long run on a few samples a step amplifies every rounding)
    while depth > 1 and sum(a * b for a, b in zip(widths, widths[1:])) > 2.5e8:
        widths.pop(1)
        depth -= 1
    while steps > 1 and 6.0 * batch * steps * sum(a * b for a, b in zip(widths, widths[1:])) > 1e13:
        steps //= 2
    return _train("", widths=",".join(map(str, widths)), act=rng.choice(["relu", "gelu"]), batch=batch,
                  stages=rng.randint(1, depth), steps=steps, lr=0.001, momentum=rng.choice([0.0, 0.9]),
                  input=rng.choice(["f32", "bf16"]), schedule=rng.choice(["layerpipe", "layerpipe", "fused_b"]))


def _draw_conv(rng):
    hw = rng.choice([16, 32, 48, 56, 64, 96, 112, 160, 224])
    batch = rng.choice([32, 64, 96, 128] if hw <= 64 else [32, 64])
    c = rng.choice([16, 32, 48, 64])
    plan, h = [], hw
    for _ in range(rng.randint(1, 4)):
        plan += [str(c)] * rng.randint(1, 3) + ["P"]
        c = min(512, c * rng.choice([1, 2, 2]))
        h //= 2
        if h % 2:
            break
    most = max(2, 60000000 // (int(plan[-2]) * h * h))            # rows of the first fully connected matrix
    fcs = [min(most, f) for f in [rng.randint(50, 2000)] * rng.randint(0, 1)] + [min(most, rng.randint(2, 500))]
    steps = 2 if hw > 112 else rng.choice([2, 4, 8])
    return _train("", plan=",".join(plan), fcs=",".join(map(str, fcs)), hw=hw, batch=batch, stages=rng.randint(2, 8), steps=steps,
                  lr=0.0005, momentum=rng.choice([0.0, 0.0, 0.9]), input=rng.choice(["f32", "bf16"]),
                  schedule=rng.choice(["layerpipe", "layerpipe", "fused_b"]), recompute=rng.random() < 0.25)


def draw(rng):
    kind = rng.choice(["mlp", "mlp", "mlp", "conv", "conv", "conv", "sample", "gemm", "gemm", "xent"])
    if kind == "mlp":
        c = _draw_mlp(rng)
    elif kind == "conv":
        c = _draw_conv(rng)
    elif kind == "sample":
        c = _train("", net="sample", hw=rng.choice([32, 64, 96, 128, 160, 192, 224, 256]), batch=rng.choice([32, 64]),
                   stages=rng.randint(1, 5), steps=rng.choice([2, 4, 8]), lr=0.0005, momentum=rng.choice([0.0, 0.9]),
                   input=rng.choice(["f32", "bf16"]))
    elif kind == "gemm":
        c = dict(kind="gemm", batch=_log_int(rng, 1, 4096), n_in=_log_int(rng, 16, 8192), n_out=_log_int(rng, 8, 8192))
    else:
        c = dict(kind="xent", batch=_log_int(rng, 1, binding.LP_XENT_STATIC_MAX_BATCH), classes=_log_int(rng, 2, 4000))
    c.pop("name", None)
    return c


# ---- networks -------------------------------------------------------------------------------------------
def _ints(text):
    return [int(t) for t in text.split(",")]


def _layers(case):
    if case["widths"]:
        return inputs.mlp(_ints(case["widths"]), case["act"])
    if case["net"] == "sample":
        return inputs.sample_net(case["hw"])
    return inputs.vgg(case["hw"], [t if t == "P" else int(t) for t in case["plan"].split(",")], _ints(case["fcs"]), case["act"])


def _in_state(trainer, host, pitch):
    """The fp32 master of the matrix `host` as a tensor over the trainer's workspace.  All state of a handle lives in
    that workspace, every buffer on a 256-byte boundary; the master is the first buffer that starts with the
    initial values (a bias vector has its version ring behind it, which starts with the same ones)."""
    rows, cols = host.shape
    base = (-trainer.workspace.data_ptr()) % 256
    ws = trainer.workspace[base:base + trainer.workspace_bytes // 256 * 256].view(torch.float32)
    at = torch.nonzero(ws[::64] == float(host[0, 0])).reshape(-1) * 64
    key = torch.from_numpy(host[0, :8].copy()).to(ws.device)
    for off in at.tolist():
        if off + (rows - 1) * pitch + cols <= ws.numel() and torch.equal(ws[off:off + key.numel()], key):
            return ws.as_strided((rows, cols), (pitch, 1), ws.storage_offset() + off)
    raise RuntimeError("a layer's master weights are not in the workspace")


def _initial(layers, normal):
    """He-normal weights, small biases, on the host as lp_create takes them."""
    W0, b0 = [], []
    for l in layers:
        shape = inputs.weight_shape(l)
        w = torch.empty(shape, pin_memory=True)
        w.copy_(normal(*shape) * math.sqrt(2.0 / np.prod(shape[1:])))
        W0.append(w.numpy())
        b0.append((0.05 * normal(l["n_out"])).cpu().numpy())
    return W0, b0


def _minibatches(case, layers, normal, gen):
    shape = inputs.input_shape(layers, case["batch"])
    x = [normal(*shape).to(torch.bfloat16 if case["input"] == "bf16" else torch.float32) for _ in range(case["steps"])]
    y = [torch.randint(0, inputs.n_classes(layers), (case["batch"],), generator=gen, device="cuda", dtype=torch.int32)
         for _ in range(case["steps"])]
    return x, y


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device=dev)

    def rows_of(n, cols, scale):                    # bf16 matrix with its rows on 16-byte boundaries
        m = torch.zeros(n, (cols + 7) // 8 * 8, dtype=torch.bfloat16, device=dev)
        m[:, :cols] = normal(n, cols) * scale
        return m

    if case["kind"] == "gemm":
        B, I, O = case["batch"], case["n_in"], case["n_out"]
        up4 = lambda x: (x + 3) // 4 * 4            # noqa: E731
        return dict(kind="gemm", B=B, I=I, O=O, a=rows_of(B, I, 1.0), w=rows_of(O, I, math.sqrt(2.0 / I)), d=rows_of(B, O, 1.0 / B),
                    z=torch.zeros(B, up4(O), device=dev), e=torch.zeros(B, up4(I), device=dev), g=torch.zeros(O, up4(I), device=dev))
    if case["kind"] == "xent":
        B, C = case["batch"], case["classes"]
        return dict(kind="xent", C=C, logits=2.0 * normal(B, C),
                    labels=torch.randint(0, C, (B,), generator=gen, device=dev, dtype=torch.int32),
                    delta=torch.zeros(B, (C + 7) // 8 * 8, dtype=torch.bfloat16, device=dev), loss=torch.zeros(1, device=dev))

    layers = _layers(case)
    W0, b0 = _initial(layers, normal)
    bf16 = case["input"] == "bf16"
    tr = binding.Trainer(layers, case["batch"], case["stages"], delays=_ints(case["delays"]) if case["delays"] else None,
                         lr=case["lr"], momentum=case["momentum"], W0=W0, b0=b0,
                         schedule=binding.LP_SCHED_FUSED_B if case["schedule"] == "fused_b" else binding.LP_SCHED_LAYERPIPE,
                         input_dtype=binding.LP_BF16 if bf16 else binding.LP_F32,
                         flags=binding.LP_RECOMPUTE if case["recompute"] else 0)
    weights = []
    for i, l in enumerate(layers):
        w = W0[i].reshape(l["n_out"], -1)
        conv = l["kind"] == "conv"
        # a first layer with few channels is stored as one row of R*S*C values per filter, others one row per tap
        one_row = not conv or (i == 0 and w.shape[1] <= (64 if (l["R"], l["S"], l["stride"], l["pad"]) == (3, 3, 1, 1) else 128))
        w = w if one_row else w.reshape(-1, l["n_in"])
        weights.append(_in_state(tr, w, (w.shape[1] + 7) // 8 * 8))
        weights.append(_in_state(tr, b0[i].reshape(1, -1), l["n_out"]))
    x, y = _minibatches(case, layers, normal, gen)
    return dict(kind="train", trainer=tr, x=x, y=y, weights=weights, done=0)


def run(state):
    if state["kind"] == "gemm":
        B, I, O, a, w, d, z, e, g = (state[k] for k in ("B", "I", "O", "a", "w", "d", "z", "e", "g"))
        binding.lp_gemm_bf16(0, B, O, I, a, a.stride(0), w, w.stride(0), z, z.stride(0))
        binding.lp_gemm_bf16(1, B, I, O, d, d.stride(0), w, w.stride(0), e, e.stride(0))
        binding.lp_gemm_bf16(2, O, I, B, d, d.stride(0), a, a.stride(0), g, g.stride(0))
        return dict(z=z[:, :O], e=e[:, :I], g=g[:, :I])
    if state["kind"] == "xent":
        rc = binding.lp_softmax_xent_static(state["logits"], state["labels"], state["delta"], state["loss"], state["C"])
        if rc != binding.LP_OK:
            raise binding.LayerPipeError(rc, "lp_softmax_xent_static")
        return dict(delta=state["delta"], loss=state["loss"])
    tr = state["trainer"]
    for x, y in zip(state["x"], state["y"]):
        tr.step(x, y)
    tr.flush()
    state["done"] += len(state["x"])
    return dict(weights=state["weights"], loss=tr.get_loss(state["done"] - 1))


# ---- the same results in 64 bits --------------------------------------------------------------------------
def exact(case, seed):
    """What `run` returns after one pass on a new state, in float64 torch without any rounding of what is stored.  Training runs of
    fully connected networks whose delays are given (or do not matter, with one step); None for the others: two runs
    of a convolutional network part after a step, and a planned network's delays are the library's to say."""
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    if case["kind"] == "gemm":
        s = prepare(case, seed)
        a, w, d = s["a"][:, :s["I"]].double(), s["w"][:, :s["I"]].double(), s["d"][:, :s["O"]].double()
        return dict(z=a @ w.T, e=d @ w, g=d.T @ a)
    if case["kind"] == "xent":
        s = prepare(case, seed)
        B, C = s["logits"].shape
        rows, labels = torch.arange(B, device="cuda"), s["labels"].long()
        logp = torch.log_softmax(s["logits"].double(), 1)
        delta = torch.zeros(s["delta"].shape, dtype=torch.float64, device="cuda")
        delta[:, :C] = logp.exp() / B
        delta[rows, labels] -= 1.0 / B
        return dict(delta=delta, loss=-logp[rows, labels].mean().reshape(1))
    if not case["widths"] or not (case["delays"] or case["steps"] == 1):
        return None
    layers = _layers(case)
    W0, b0 = _initial(layers, normal)
    xs, ys = _minibatches(case, layers, normal, gen)
    delays = _ints(case["delays"]) if case["delays"] else [0] * len(layers)
    W = [[torch.from_numpy(w).cuda().double()] for w in W0]        # per layer: every version so far
    b = [[torch.from_numpy(v).cuda().double()] for v in b0]
    mW, mb = [torch.zeros_like(w[0]) for w in W], [torch.zeros_like(v[0]) for v in b]
    gelu = case["act"] == "gelu"
    loss = 0.0
    for n, (x, y) in enumerate(zip(xs, ys)):
        v = [max(0, n - d) for d in delays]
        a, z = [x.double()], []
        for l in range(len(layers)):
            z.append(a[l] @ W[l][v[l]].T + b[l][v[l]])
            if l + 1 < len(layers):
                a.append(torch.nn.functional.gelu(z[l]) if gelu else z[l].clamp_min(0.0))
        logp = torch.log_softmax(z[-1], 1)
        rows = torch.arange(len(y), device="cuda")
        loss = float(-logp[rows, y.long()].mean())
        d = logp.exp()
        d[rows, y.long()] -= 1.0
        d /= len(y)
        for l in reversed(range(len(layers))):
            mW[l] = case["momentum"] * mW[l] + d.T @ a[l]
            mb[l] = case["momentum"] * mb[l] + d.sum(0)
            if l > 0:
                below = z[l - 1]
                slope = (0.5 * (1.0 + torch.erf(below / math.sqrt(2.0))) + below * torch.exp(-0.5 * below * below) / math.sqrt(2.0 * math.pi)
                         if gelu else (below > 0).double())
                d = (d @ W[l][v[l]]) * slope
            W[l].append(W[l][-1] - case["lr"] * mW[l])
            b[l].append(b[l][-1] - case["lr"] * mb[l])
    return dict(weights=[t for l in range(len(layers)) for t in (W[l][-1], b[l][-1].reshape(1, -1))], loss=loss)


# ---- what a pass cannot do without ------------------------------------------------------------------------
def work(case):
    if case["kind"] == "gemm":
        B, I, O = case["batch"], case["n_in"], case["n_out"]
        return {"bytes": 2 * (B * I + O * I + B * O) + 4 * (B * O + B * I + O * I), "flops": 6 * B * I * O}
    if case["kind"] == "xent":
        B, C = case["batch"], case["classes"]
        return {"bytes": B * C * (4 + 2) + 4 * B, "flops": 8 * B * C}
    layers, B = _layers(case), case["batch"]
    flops = 0
    nbytes = B * int(np.prod(inputs.input_shape(layers, 1))) * (2 if case["input"] == "bf16" else 4)
    for i, l in enumerate(layers):
        params = int(np.prod(inputs.weight_shape(l)))
        if l["kind"] == "conv":
            ho, wo = inputs.conv_out_hw(l)
            outs, macs = B * ho * wo * l["n_out"], B * ho * wo * params
        else:
            outs, macs = B * l["n_out"], B * params
        flops += 2 * macs * (3 if i > 0 else 2)
        # bf16 weights into forward and delta, fp32 master (and momentum) read and written, a new bf16 version
        nbytes += params * (2 + (2 if i > 0 else 0) + 8 + (8 if case["momentum"] else 0) + 2)
        # activations written, read by the next layer and by the backward pass; the gradient written and read
        nbytes += 2 * outs * 5
    return {"bytes": case["steps"] * nbytes, "flops": case["steps"] * flops}


def tolerance(case):
    """About four times what was seen: against 64-bit sums (gemm, xent), or between two runs whose initial weights
    differ in their last bit (train), which moves some bf16 roundings as another order of the sums does."""
    if case["kind"] == "gemm":                      # the accumulator is truncated once per 16 terms: 1.1e-9 a term
        rel = 2e-6 + 4.4e-9 * max(case["batch"], case["n_in"], case["n_out"])
        return {"rel": rel, "max": 5 * rel}
    if case["kind"] == "xent":                      # 3e-5 of the bf16 results land on the other side of a rounding boundary
        return {"rel": max(3e-5, 8e-3 / math.sqrt(case["batch"] * case["classes"])), "max": 2e-2}
    if case["steps"] == 1:                          # seen: 1.4e-4
        return {"rel": 5e-4, "max": 3e-3}
    if not case["widths"]:                          # ReLU gates and pooling winners flip: 4e-3, single weights 3e-2
        return {"rel": 1.5e-2, "max": 1.2e-1}
    if case["batch"] < 64:                          # 2e-3, 9e-3
        return {"rel": 8e-3, "max": 5e-2}
    return {"rel": 5e-4, "max": 2e-3}               # 1e-4, 4e-4
