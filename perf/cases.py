"""Workloads of the AGZO library as a training program runs them, one dict per workload.

A program that trains with AGZO does one of four things with the library:

  step     one whole iteration through agzo_step over resident activations: subspace extraction, the
           in-place passes, the scalar, the fused restore-and-update.  The forwards belong to the
           caller's model; here the losses are already on the device and the callback has nothing to do.
  hook     the same iteration with extraction called from forward hooks: one call per group of layers
           that read the same activations, layer descriptors made on the spot (the activation tensors
           of a forward are new every time), then the passes over all layers.
  dense    the parameters that are not matrices of a linear layer (norm vectors, an embedding table),
           perturbed with a dense Gaussian direction: +eps, -2 eps, then the update.
  static   extraction for one layer without a workspace, for callers that cannot allocate.

Layers are either the seven linear layers of transformer blocks ("hidden" > 0) or a stack of square
layers ("width" > 0).  Weights are bf16, fp32, or an fp32 master with a bf16 compute copy ("pair").
With "shared", q/k/v read one activation buffer and gate/up another, as in a transformer block;
without it every layer has activations of its own.
"""
import math

import torch

from paper_2601_17261_b200 import binding as B

EPS, LR = 1e-3, 1e-6


def _case(name, op, **kw):
    c = {"op": op, "blocks": 0, "hidden": 0, "q_out": 0, "kv_out": 0, "inter": 0, "width": 0, "layers": 0,
         "tokens": 0, "rank": 1, "K": 3, "mode": 0, "weights": "bf16", "acts": "bf16", "shared": True,
         "vectors": 0, "vector": 0, "table": 0}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _blocks(n, hidden, q_out, kv_out, inter):
    return {"blocks": n, "hidden": hidden, "q_out": q_out, "kv_out": kv_out, "inter": inter}


SMALL = (1024, 2048, 1024, 3072)      # the 0.6B-shaped block of workloads.py
MEDIUM = (2048, 2048, 1024, 6144)     # the 1.7B-shaped block
LARGE = (4096, 4096, 1024, 12288)     # the 8B-shaped block


def listed():
    return [
        # one fp32 linear layer on a least-squares problem: the smallest complete step, all latency
        _case("one_layer_f32", "step", layers=1, width=256, tokens=512, rank=4, weights="f32", acts="f32"),
        # an 8-layer MLP with fp32 masters and bf16 compute copies
        _case("mlp_pair", "step", layers=8, width=1024, tokens=4096, rank=8, weights="pair", shared=False),
        # whole layer set of a small model, every layer with activations of its own
        _case("set_0p6b_r8", "step", **_blocks(28, *SMALL), tokens=8192, rank=8, shared=False),
        # whole layer set of a medium model as its blocks run: shared inputs, a batch trimmed to its real length
        _case("set_1p7b_r4_ragged", "step", **_blocks(28, *MEDIUM), tokens=11873, rank=4),
        # part of a large model's layer set at the rank and token count of the benchmark's headline row
        _case("set_8b_r16", "step", **_blocks(10, *LARGE), tokens=16384, rank=16, shared=False),
        # the largest rank
        _case("set_8b_r64", "step", **_blocks(6, *LARGE), tokens=16384, rank=64),
        # rank 1, one-sided difference, 16 sequences of a classification task: the method as printed
        _case("set_8b_r1_short", "step", **_blocks(8, *LARGE), tokens=4811, rank=1, mode=1),
        # extraction inside the forward, long batches of a large model
        _case("hooks_8b_r16", "hook", **_blocks(2, *LARGE), tokens=16384, rank=16),
        # extraction inside the forward, a handful of short sequences: many small calls
        _case("hooks_0p6b_r8_short", "hook", **_blocks(4, *SMALL), tokens=613, rank=8),
        # fp32 training: weights and activations in fp32
        _case("set_f32_r8", "step", **_blocks(2, *SMALL), tokens=4000, rank=8, weights="f32", acts="f32"),
        # norm vectors and an embedding table
        _case("vectors_and_table", "dense", vectors=56, vector=1024, table=65536 * 1024),
        # one layer, no workspace
        _case("static_layer", "static", layers=1, width=2048, tokens=4096, rank=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "step", "hook", "hook", "dense", "static"])
    K = rng.choice([3, 3, 3, 1])
    if op == "dense":
        return _case(None, op, vectors=rng.randint(1, 80), vector=_log(rng, 100, 6000), table=_log(rng, 1 << 16, 1 << 26),
                     weights=rng.choice(["bf16", "bf16", "f32"]))
    if op == "static":
        return _case(None, op, layers=1, width=_log(rng, 128, 2048), tokens=_log(rng, 256, 4096), rank=rng.randint(1, 16),
                     K=K, acts=rng.choice(["bf16", "f32"]))
    rank = rng.choice([1, 2, 3, 4, 6, 8, 8, 12, 16, 16, 24, 32, 64])
    if op == "step" and rng.random() < 0.4:          # a stack of square layers
        width = _log(rng, 128, 2048)
        if rng.random() < 0.75:
            width = (width + 7) // 8 * 8
        weights = rng.choice(["f32", "pair", "bf16"])
        return _case(None, op, layers=rng.randint(1, 12), width=width, tokens=_log(rng, 256, 8192), rank=rank, K=K,
                     mode=rng.choice([0, 0, 1]), weights=weights, acts="f32" if weights == "f32" else "bf16", shared=False)
    shape = rng.choice([SMALL, SMALL, MEDIUM, MEDIUM, LARGE])
    tokens = _log(rng, 300, 16384)
    n = rng.randint(1, 28 if shape is SMALL else 12 if shape is MEDIUM else 5)
    f32 = shape is SMALL and rng.random() < 0.25
    if f32:
        n, tokens = min(n, 3), min(tokens, 4096)
    if op == "hook":
        n = min(n, 6)
    return _case(None, op, **_blocks(n, *shape), tokens=tokens, rank=rank, K=K, mode=rng.choice([0, 0, 1]),
                 weights="f32" if f32 else "bf16", acts="f32" if f32 else "bf16", shared=op == "hook" or rng.random() < 0.7)


def _layers(case):
    """(d_in, d_out, group) of every linear layer; layers of a group read the same activations."""
    out = []
    if case["width"]:
        return [(case["width"], case["width"], i) for i in range(case["layers"])]
    h, q, kv, inter = case["hidden"], case["q_out"], case["kv_out"], case["inter"]
    for b in range(case["blocks"]):
        block = [(h, q, 0), (h, kv, 0), (h, kv, 0), (q, h, 1), (h, inter, 2), (h, inter, 2), (inter, h, 3)]
        for i, (di, do, g) in enumerate(block):
            out.append((di, do, 4 * b + g if case["shared"] else 7 * b + i))
    return out


def _dtype(name):
    return torch.float32 if name == "f32" else torch.bfloat16


def _views(shapes, dtype, dev):
    """Tensors of these shapes in one buffer (a flat parameter buffer), each start at a multiple of 128 elements."""
    at, total = [], 0
    for rows, cols in shapes:
        at.append(total)
        total += (rows * cols + 127) // 128 * 128
    flat = torch.zeros(total, dtype=dtype, device=dev)
    return flat, [flat[a:a + r * c].view(r, c) for a, (r, c) in zip(at, shapes)]


def _activations(m, d, gen, dtype, dev):
    """N(0, 1) tokens with a dominant low-rank part of ten times the variance, as workloads.py plants it."""
    p = min(64, max(4, d // 32))
    x = torch.empty(m, d, dtype=dtype, device=dev)
    basis = torch.randn(p, d, generator=gen, device=dev) * math.sqrt(10.0 / d)
    for t in range(0, m, 4096):
        n = min(4096, m - t)
        c = torch.randn(n, p, generator=gen, device=dev)
        x[t:t + n] = torch.addmm(torch.randn(n, d, generator=gen, device=dev), c, basis)
    return x


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    state = {"case": case, "seed": 7919 * seed + 1}
    state["losses"] = 2.0 + 1e-3 * torch.randn(2, generator=gen, device=dev, dtype=torch.float64)
    state["ghat"] = torch.zeros(1, device=dev)
    if case["op"] == "dense":
        dt = _dtype(case["weights"])
        sizes = [case["vector"]] * case["vectors"] + [case["table"]]
        flat, views = _views([(1, n) for n in sizes], dt, dev)
        flat.normal_(0.0, 0.02, generator=gen)
        state.update(flat=flat, params=[v.view(-1) for v in views], ctx=B.Context(dev.index, 4096))
        return state
    specs = _layers(case)
    r = min(case["rank"], case["tokens"])
    X, per_layer = {}, []
    for di, _, g in specs:
        if g not in X:
            X[g] = _activations(case["tokens"], di, gen, _dtype(case["acts"]), dev)
        per_layer.append(X[g])
    flat_v, V = _views([(r, di) for di, _, _ in specs], torch.float32, dev)
    state.update(X=per_layer, groups=[g for _, _, g in specs], flat_v=flat_v, V=V, r=r)
    if case["op"] == "static":
        state["flag"] = torch.zeros(1, dtype=torch.int32, device=dev)
        return state
    flat_w, W = _views([(do, di) for di, do, _ in specs], torch.float32 if case["weights"] == "pair" else _dtype(case["weights"]), dev)
    flat_w.normal_(0.0, 0.02, generator=gen)
    W16 = [None] * len(specs)
    if case["weights"] == "pair":
        flat_16, W16 = _views([(do, di) for di, do, _ in specs], torch.bfloat16, dev)
        flat_16.copy_(flat_w)
        state["flat_w16"] = flat_16
    layers = [B.make_layer(W=w, W16=w16, X=x, V=v, r=r, layer_id=i)
              for i, (w, w16, x, v) in enumerate(zip(W, W16, per_layer, V))]
    state.update(flat_w=flat_w, layers=layers, arr=B.layer_array(layers), ctx=B.agzo_create(layers, dev.index))
    return state


def _forward(phase, slot, stream):
    """The caller's forward: its loss is on the device already."""


def _run_dense(s):
    ctx, seed = s["ctx"], s["seed"]
    for i, w in enumerate(s["params"]):
        B.agzo_perturb_dense(ctx, w, seed, i, EPS)
    for i, w in enumerate(s["params"]):
        B.agzo_perturb_dense(ctx, w, seed, i, -2 * EPS)
    B.agzo_ghat(ctx, s["losses"][0:1], s["losses"][1:2], EPS, 0, s["ghat"])
    for i, w in enumerate(s["params"]):
        B.agzo_perturb_dense(ctx, w, seed, i, EPS)
        B.agzo_perturb_dense(ctx, w, seed, i, -LR, s["ghat"])
    return {"w": s["flat"], "ghat": s["ghat"]}


def _run_hook(s):
    case, ctx, seed = s["case"], s["ctx"], s["seed"]
    i, n = 0, len(s["layers"])
    while i < n:          # one call per group of layers that read the same activations
        j = i
        while j < n and s["groups"][j] == s["groups"][i]:
            j += 1
        group = [B.make_layer(X=s["X"][k], V=s["V"][k], r=s["r"], layer_id=k) for k in range(i, j)]
        B.agzo_extract_subspace(ctx, group, seed, case["K"])
        i = j
    arr = s["arr"]
    B.agzo_perturb(ctx, s["layers"], seed, EPS, arr=arr)
    if case["mode"] == 0:
        B.agzo_perturb(ctx, s["layers"], seed, -2 * EPS, arr=arr)
    B.agzo_ghat(ctx, s["losses"][0:1], s["losses"][1:2], EPS, case["mode"], s["ghat"])
    B.agzo_restore_update(ctx, s["layers"], seed, EPS, LR, case["mode"], s["ghat"], arr=arr)


def run(state):
    case = state["case"]
    state["seed"] += 1                     # every iteration draws new directions
    if case["op"] == "dense":
        return _run_dense(state)
    if case["op"] == "static":
        B.agzo_extract_subspace_static(state["X"][0], state["V"][0], state["r"], case["K"], state["seed"], 0, state["flag"])
        return {"v": state["flat_v"], "flag": state["flag"]}
    if case["op"] == "hook":
        _run_hook(state)
    else:
        B.agzo_step(state["ctx"], state["layers"], seed=state["seed"], eps=EPS, lr=LR, K=case["K"], mode=case["mode"],
                    loss_fn=_forward, d_losses2=state["losses"], d_ghat=state["ghat"], arr=state["arr"])
    out = {"v": state["flat_v"], "w": state["flat_w"], "ghat": state["ghat"]}
    if "flat_w16" in state:
        out["w16"] = state["flat_w16"]
    return out


def work(case):
    """Activations read once, bases written once, weights read and written once per in-place pass (the
    caller's forward runs between the passes)."""
    if case["op"] == "dense":
        n = case["vectors"] * case["vector"] + case["table"]
        return {"bytes": 3 * 2 * n * (4 if case["weights"] == "f32" else 2), "flops": 3 * 2 * n}
    specs = _layers(case)
    m, r = case["tokens"], min(case["rank"], case["tokens"])
    x = {g: m * di * (4 if case["acts"] == "f32" else 2) for di, _, g in specs}
    v = sum(4 * r * di for di, _, _ in specs)
    flops = sum(2 * (2 * case["K"] + 1) * m * di * r + 4 * (case["K"] + 1) * di * r * r for di, _, _ in specs)
    if case["op"] == "static":
        return {"bytes": sum(x.values()) + v, "flops": flops}
    n = sum(di * do for di, do, _ in specs)
    passes = 3 - case["mode"]
    per_weight = {"bf16": 4 * passes, "f32": 8 * passes, "pair": 6 * (passes - 1) + 10}[case["weights"]]
    return {"bytes": sum(x.values()) + v * (1 + passes) + n * per_weight, "flops": flops + passes * n * 2 * (r + 1)}


def tolerance(case):
    """About four times what the library's tensor-core and fp32 kernels differ by on the same inputs: bases
    1.2e-5 up to rank 16 and 3.2e-5 at rank 64 (single entries 9e-5 and 1.2e-3); bf16 weights 5e-5, where the few
    that round the other way are off by one step of the grid (7.8e-3) in a pass."""
    if case["op"] == "static" or (case["weights"] == "f32" and case["op"] != "dense"):
        return {"rel": 5e-5, "max": 1e-3} if case["rank"] <= 16 else {"rel": 1.5e-4, "max": 5e-3}
    if case["weights"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 2e-4, "max": 5e-2}
