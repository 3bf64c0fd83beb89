"""Workloads for timing the whole DP-SGD step through the public entry points.

A case is a model (layer shapes), a batch size, an input type and the way the step is launched.  `prepare` draws the
step's inputs on the GPU and makes the plan (and, for recorded steps, the CUDA graph) that a training program keeps;
`run` is one step.  The families:

  mlp    dense layers with T = 1; optionally followed by the parameter update of every tensor (noise folded into it)
  cnn    convolutions handed over as patch matrices, then dense layers
  maps   convolutions handed over as feature maps with dL/dZ channel-major, as back-propagation has them, then dense layers
  seq    attention projections, feed-forward and recurrent gate layers applied at T positions; global or per-layer clipping
  block  one pre-norm transformer block: two LayerNorms, four projections, two feed-forward layers
  layer  a single dense layer applied at T positions

Inputs: activations ~ N(0, 1) (ReLU of it behind a non-linearity), dL/dZ ~ N(0, v) with v such that the per-example norms
spread over a factor of sixteen around the clipping threshold C = 1, so that about half of the examples are clipped, as
thresholds are chosen in practice.  sigma = 0.05, the paper's setting.
"""
import math

import torch

import paper_2009_03106_b200 as dp

C, SIGMA, SEED = 1.0, 0.05, 17
LR, BETA1, BETA2, EPS, ADAM_STEP = 1e-3, 0.9, 0.999, 1e-8, 100


# ---------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest step in use: a two-layer MLP at batch 32, one launch, all latency
        dict(name="mlp_b32_f32", kind="mlp", dtype="f32", B=32, widths="784-256-10", update="none"),
        # the MNIST-sized MLP at batch 128
        dict(name="mlp_b128_f32", kind="mlp", dtype="f32", B=128, widths="784-1000-1000-10", update="none"),
        # a wide classifier head (fully connected layers on top of a feature extractor), step and Adam update: the
        # parameters, not the inputs, are the bulk of the bytes
        dict(name="mlp_wide_adam_bf16", kind="mlp", dtype="bf16", B=256, widths="4096-4096-1000", update="adam"),
        # the 32 x 32 CNN at batch 128 from patch matrices, both input types, as a recorded step
        dict(name="cnn_f32", kind="cnn", dtype="f32", B=128, size=32, channels="3-32-64-128", head="256-10"),
        dict(name="cnn_bf16", kind="cnn", dtype="bf16", B=128, size=32, channels="3-32-64-128", head="256-10"),
        # the same CNN as back-propagation hands it over (feature maps, channel-major gradients)
        dict(name="maps_f32", kind="maps", dtype="f32", B=128, size=32, channels="3-32-64-128", strides="1-1-1", pool=1,
             head="256-10"),
        # a deeper convolution stack that halves its maps by stride, up to 256 channels
        dict(name="maps_strided_bf16", kind="maps", dtype="bf16", B=64, size=32, channels="3-64-128-256-256",
             strides="1-2-2-1", pool=0, head="10"),
        # the sequence model: four projections, feed-forward in and out, recurrent gates
        dict(name="seq_bf16", kind="seq", dtype="bf16", B=128, T=256, d=512, d_ff=2048, clip="global"),
        # a text model on 300-dimensional word vectors: sentence length and widths that fit no tile; per-layer thresholds
        dict(name="seq_ragged_bf16", kind="seq", dtype="bf16", B=50, T=77, d=300, d_ff=1100, clip="per_layer"),
        # the sequence model in fp32
        dict(name="seq_f32", kind="seq", dtype="f32", B=32, T=128, d=512, d_ff=2048, clip="global"),
        # a transformer block with its LayerNorm parameters
        dict(name="block_bf16", kind="block", dtype="bf16", B=128, T=256, d=512, d_ff=2048),
        # the largest: one feed-forward layer of a long-sequence model
        dict(name="layer_long_bf16", kind="layer", dtype="bf16", B=256, T=512, d_in=1024, d_out=4096),
    ]


MOST_FLOPS = 1.3e12       # a drawn case costs no more than the largest listed one


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A layer width: mostly a multiple of 16, sometimes of 4 (300), sometimes anything."""
    w = _log_int(rng, lo, hi)
    u = rng.random()
    m = 16 if u < 0.6 else 4 if u < 0.85 else 1
    return max(m, w // m * m)


def draw(rng):
    while True:
        kind = rng.choice(["mlp", "mlp", "cnn", "maps", "maps", "seq", "seq", "block", "layer", "layer"])
        dtype = rng.choice(["f32", "bf16", "bf16"])
        if kind == "mlp":
            n = rng.randint(2, 4)
            widths = [_width(rng, 128, 4096) for _ in range(n)] + [rng.choice([2, 10, 100, 1000])]
            c = dict(kind=kind, dtype=dtype, B=_log_int(rng, 16, 512), widths="-".join(map(str, widths)),
                     update=rng.choice(["none", "none", "sgd", "adam"]))
        elif kind == "cnn":
            ch = [rng.choice([1, 3])] + [rng.choice([16, 32, 48, 64]), rng.choice([32, 64, 96]), rng.choice([64, 128, 160])]
            c = dict(kind=kind, dtype=dtype, B=_log_int(rng, 16, 256), size=rng.choice([28, 32, 48]),
                     channels="-".join(map(str, ch)), head=rng.choice(["256-10", "100", "120-84-10"]))
        elif kind == "maps":
            n = rng.randint(2, 4)
            ch, strides = [rng.choice([1, 3, 16])], []
            for _ in range(n):
                ch.append(min(256, max(16, ch[-1]) * rng.choice([1, 2, 2, 4])))
                strides.append(rng.choice([1, 1, 2]))
            c = dict(kind=kind, dtype=dtype, B=_log_int(rng, 16, 256), size=rng.choice([14, 28, 32, 56]),
                     channels="-".join(map(str, ch)), strides="-".join(map(str, strides)), pool=rng.choice([0, 1]),
                     head=rng.choice(["10", "256-10"]))
        elif kind == "seq":
            d = _width(rng, 64, 1024)
            c = dict(kind=kind, dtype=dtype, B=_log_int(rng, 16, 256), T=_log_int(rng, 16, 512), d=d,
                     d_ff=_width(rng, 2 * d, 4 * d), clip=rng.choice(["global", "global", "per_layer"]))
        elif kind == "block":
            d = _width(rng, 64, 1024)
            c = dict(kind=kind, dtype=dtype, B=_log_int(rng, 16, 256), T=_log_int(rng, 16, 512), d=d, d_ff=4 * d)
        else:
            c = dict(kind=kind, dtype=dtype, B=_log_int(rng, 16, 1024), T=_log_int(rng, 16, 2048),
                     d_in=_width(rng, 128, 4096), d_out=_width(rng, 128, 4096))
        w = work(c)
        # fp32 work costs several times as much as bf16 work
        if w["flops"] * (6 if dtype == "f32" else 1) <= MOST_FLOPS and w["bytes"] <= 1.3e9:
            return c


# ---------------------------------------------------------------------------------------------------------------
# shapes
# ---------------------------------------------------------------------------------------------------------------
def _ints(text):
    return [int(v) for v in str(text).split("-")]


def _shapes(case):
    """The layers of a case: dicts with kind (dense / norm / conv), T, d_in, d_out, bias, relu (input behind a
    non-linearity) and, for convolutions, c (input channels), size, stride."""
    dense = lambda T, i, o, bias=True, relu=False: dict(kind="dense", T=T, d_in=i, d_out=o, bias=bias, relu=relu)   # noqa: E731
    kind = case["kind"]
    if kind == "mlp":
        w = _ints(case["widths"])
        return [dense(1, i, o, True, k > 0) for k, (i, o) in enumerate(zip(w, w[1:]))]
    if kind in ("cnn", "maps"):
        ch, size, out = _ints(case["channels"]), case["size"], []
        strides = _ints(case["strides"]) if kind == "maps" else [1] * (len(ch) - 1)
        pool = case["pool"] if kind == "maps" else 1
        for i, o, s in zip(ch, ch[1:], strides):
            o_size = (size + 2 - 3) // s + 1
            out.append(dict(kind="conv", T=o_size * o_size, d_in=9 * i, d_out=o, bias=True, relu=True, c=i, size=size, stride=s))
            size = o_size // 2 if pool and o_size >= 8 else o_size
        # without pooling between the convolutions the maps are averaged before the head
        w = [ch[-1] * size * size if pool else ch[-1]] + _ints(case["head"])
        return out + [dense(1, i, o, True, True) for i, o in zip(w, w[1:])]
    T = case["T"]
    if kind == "layer":
        return [dense(T, case["d_in"], case["d_out"])]
    d, ff = case["d"], case["d_ff"]
    attn = [dense(T, d, d, False) for _ in range(4)]
    ffn = [dense(T, d, ff), dense(T, ff, d, True, True)]
    if kind == "seq":
        return attn + ffn + [dense(T, d, 4 * d)]
    norm = dict(kind="norm", T=T, d_in=d, d_out=d, bias=True, relu=False)
    return [norm] + attn + [norm] + ffn


def _params(y):
    return y["d_out"] * (1 if y["kind"] == "norm" else y["d_in"]) + (y["d_out"] if y["bias"] else 0)


def work(case):
    """Inputs once, outputs once; for the update its state in and out.  Flops: the cheaper exact norm form per layer
    and the clipped-sum product."""
    B, es = case["B"], 4 if case["dtype"] == "f32" else 2
    n_bytes, flops = 8.0 * B, 0.0
    for y in _shapes(case):
        T, i, o = y["T"], y["d_in"], y["d_out"]
        n_in = y["c"] * y["size"] ** 2 if y["kind"] == "conv" and case["kind"] == "maps" else T * i
        n_bytes += B * (n_in + T * o) * es + 4.0 * _params(y)
        if case.get("update", "none") != "none":
            n_bytes += 4.0 * _params(y) * (3 if case["update"] == "sgd" else 7)
        if y["kind"] == "norm":
            flops += 4.0 * B * T * o
        else:
            flops += 2.0 * B * T * i * o
            flops += 2.0 * B * (i + o) if T == 1 else min(float(B) * T * (T + 1) * (i + o), 2.0 * B * T * i * o)
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    # fp32: sums of 1e2 .. 1e5 products in fp32 (or three tf32 products per term); bf16: one bf16 rounding of a
    # clipped operand.  The noise is part of the outputs.
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 4e-3}


# ---------------------------------------------------------------------------------------------------------------
# inputs, plan, step
# ---------------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    B, shapes = case["B"], _shapes(case)
    randn = lambda *s: torch.randn(*s, generator=gen, device=dev)                                   # noqa: E731
    # E ||G_i||^2 = sum over layers of T d_out (d_in E[a^2] + bias) v: v puts it at C^2
    total = 0.0
    for y in shapes:
        a2 = 0.5 if y["relu"] else 1.0
        total += y["T"] * y["d_out"] * ((a2 if y["kind"] == "norm" else y["d_in"] * a2) + (1.0 if y["bias"] else 0.0))
    spread = torch.exp((torch.rand(B, generator=gen, device=dev) * 2 - 1) * math.log(4.0)) * (C / math.sqrt(total))
    mixed = case["kind"] in ("maps", "block")
    layers = []
    for y in shapes:
        T, i, o = y["T"], y["d_in"], y["d_out"]
        Z = (randn(B, T, o) * spread[:, None, None]).to(dtype)
        if y["kind"] == "conv":
            X = torch.relu(randn(B, y["c"], y["size"], y["size"]))
            if mixed:
                layers.append(dp.ModelLayer(dp.DPCLIP_KIND_CONV, X.to(dtype), Z.transpose(1, 2).contiguous(), y["bias"],
                                            conv=(3, 3, y["stride"], 1), z_channel_major=True))
                continue
            A = torch.nn.functional.unfold(X, 3, padding=1, stride=y["stride"]).transpose(1, 2).to(dtype).contiguous()
        elif y["kind"] == "norm":
            A = torch.nn.functional.layer_norm(randn(B, T, i), (i,)).to(dtype)
        else:
            A = randn(B, T, i)
            A = (torch.relu(A) if y["relu"] else A).to(dtype)
        if mixed:
            kind = dp.DPCLIP_KIND_ELEMENTWISE if y["kind"] == "norm" else dp.DPCLIP_KIND_DENSE
            layers.append(dp.ModelLayer(kind, A, Z, y["bias"]))
        else:
            layers.append(dp.Layer(A, Z, y["bias"]))
    plan = dp.ModelPlan(layers) if mixed else dp.StepPlan(layers)
    state = {"plan": plan, "kind": case["kind"], "graph": None, "update": case.get("update", "none"), "B": B,
             "C_layer": [C / math.sqrt(len(shapes))] * len(shapes) if case.get("clip") == "per_layer" else None}
    if case["kind"] in ("cnn", "maps"):
        # many small launches: a training program records them.  The capture stream comes from the other of torch's
        # two stream pools (32 streams each, handed out in rotation), so that it is never one of the plan's own streams.
        plan.run_streams(C, SIGMA, SEED, branches=4)
        torch.cuda.synchronize()
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"], stream=torch.cuda.Stream(priority=-1)):
            plan.run_streams(C, SIGMA, SEED, branches=4)
    if state["update"] != "none":
        sums = [g for gs in zip(plan.gW, plan.gb) for g in gs]
        theta = [randn(g.numel()) * 0.02 for g in sums]
        m = [randn(g.numel()) * 1e-3 for g in sums]
        v = [torch.rand(g.numel(), generator=gen, device=dev) * 1e-5 + 1e-6 for g in sums]
        state.update(sums=[g.view(-1) for g in sums], theta=theta, m=m, v=v)
    return state


def run(state):
    plan = state["plan"]
    out = {"gW": plan.gW, "gb": plan.gb, "clip": plan.clip, "norms": plan.norms}
    if state["graph"] is not None:
        state["graph"].replay()
    elif state["C_layer"] is not None:
        out["clip"] = dp.dpclip_step_per_layer(plan, state["C_layer"], SIGMA, SEED)
        out["norms"] = plan.sq_layers
    elif state["update"] != "none":
        plan.run(C, 0.0, SEED)                      # the noise belongs to the update
        for k, (theta, m, v, g) in enumerate(zip(state["theta"], state["m"], state["v"], state["sums"])):
            if state["update"] == "adam":
                dp.dpclip_dp_adam_step(theta, m, v, g, 1.0 / state["B"], C, SIGMA, SEED, k, LR, BETA1, BETA2, EPS, ADAM_STEP)
            else:
                dp.dpclip_dp_sgd_step(theta, g, 1.0 / state["B"], C, SIGMA, SEED, k, LR)
        out["theta"] = state["theta"]
        if state["update"] == "adam":
            out["m"], out["v"] = state["m"], state["v"]
    elif state["kind"] == "block":
        plan.run_streams(C, SIGMA, SEED, branches=4)
    else:
        plan.run(C, SIGMA, SEED)
    return out
