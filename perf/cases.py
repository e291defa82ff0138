"""What a user of this package has it do, as cases that can be timed and compared.

A case is one DP-SGD step on GPT-2-style shapes: per-example norms of every block linear, the LM
head and the embedding tables (plus the cross term of a tied head, or biases and LayerNorm
parameters), clip factors, the clipped sum of every parameter tensor and its Gaussian noise.  Every
layer has tensors of its own, as after a real backward pass.
"""
import math

import torch

from paper_2609_40335_b200 import binding as dp
from paper_2609_40335_b200 import pipeline

V_GPT2 = 50257


def _case(name, **kw):
    """mode: "step" = pipeline.dp_step call by call; "graph" = one replay of pipeline.StepGraph;
    "sums" = dp_step without noise, which is what a rank hands to the exchange."""
    c = dict(dtype="bf16", d_model=768, blocks=12, square=False, V=V_GPT2, head=True, tied=False,
             positions=False, full=False, sigma=0.8, mode="step")
    c.update(kw)
    return dict({"name": name}, **c) if name else c


def listed():
    return [
        # the smallest step there is: one fp32 linear layer and a 1000-row table; launches and latency
        _case("tiny_f32", B=4, T=16, dtype="f32", d_model=64, blocks=1, square=True, V=1000, head=False,
              sigma=1.0),
        # fp32 activations and gradients, DistilGPT2 shape, a small batch
        _case("distil_f32", B=8, T=128, dtype="f32", blocks=6),
        # the few examples per step that remain on each GPU when memory is short; GPT-2 small with a
        # tied head, an odd sequence length
        _case("micro_tied_graph", B=3, T=77, tied=True, mode="graph"),
        # DistilGPT2, untied head, an ordinary fine-tuning batch
        _case("distil_untied", B=32, T=128, blocks=6),
        # the same step on one rank of a data-parallel job: the sums leave before any noise is drawn
        _case("distil_sums", B=32, T=128, blocks=6, mode="sums"),
        # every parameter of DistilGPT2 (biases, LayerNorm, position table), ragged batch and length
        _case("distil_full_ragged", B=21, T=203, blocks=6, positions=True, full=True),
        # GPT-2 small with a tied head
        _case("small_tied", B=32, T=128, tied=True),
        # GPT-2 small with a position table, captured once and replayed: the flagship workload
        _case("small_positions_graph", B=64, T=256, positions=True, mode="graph"),
        # GPT-2 small at its full context: some layers take the DIRECT norm
        _case("small_context", B=6, T=1024, positions=True),
        # GPT-2 medium: a small batch of short sequences (parameters dominate), of long ones, and the largest
        _case("medium_short", B=16, T=128, d_model=1024, blocks=24, sigma=1.0),
        _case("medium_long", B=16, T=512, d_model=1024, blocks=24, sigma=1.0),
        _case("medium_large", B=64, T=512, d_model=1024, blocks=24, sigma=1.0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["untied", "tied", "positions", "full", "sums", "graph", "f32", "tiny"])
    kw = dict(B=log_int(1, 96), T=log_int(16, 1024), d_model=64 * log_int(1, 16), blocks=log_int(1, 24),
              V=log_int(500, V_GPT2), sigma=round(rng.uniform(0.5, 1.2), 2))
    if kind in ("tied", "graph"):
        kw["tied"] = kind == "tied" or rng.random() < 0.5
    if kind in ("positions", "full"):
        kw["positions"] = True
    if kind == "full":
        kw["full"] = True
        kw["blocks"] = min(kw["blocks"], 12)
    if kind in ("sums", "graph"):
        kw["mode"] = kind
    if kind == "f32":
        kw.update(dtype="f32", B=min(kw["B"], 16), T=min(kw["T"], 256), blocks=min(kw["blocks"], 6))
    if kind == "tiny":
        kw.update(dtype=rng.choice(["f32", "bf16"]), B=log_int(1, 8), T=log_int(8, 64), blocks=1, square=True,
                  d_model=64 * rng.randint(1, 3), V=log_int(500, 5000), head=False)
    top = work(listed()[-1])
    while True:
        c = _case(None, **kw)
        w = work(c)
        small = c["dtype"] == "bf16" or w["flops"] <= 0.02 * top["flops"]     # fp32 products cost more
        if small and w["bytes"] <= 0.5 * top["bytes"] and w["flops"] <= 0.5 * top["flops"]:
            return c
        kw["B"], kw["blocks"] = max(1, kw["B"] // 2), max(1, kw["blocks"] * 3 // 4)


def _shapes(case):
    d = case["d_model"]
    block = [(d, d)] if case["square"] else [(d, 3 * d), (d, d), (d, 4 * d), (4 * d, d)]
    return block * case["blocks"]


def prepare(case, seed):
    dev = "cuda"
    B, T, V, d = case["B"], case["T"], case["V"], case["d_model"]
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))

    def normal(cols, std, ld=None):
        t = torch.empty(B, T, ld or cols, dtype=dtype, device=dev)
        return t.normal_(0.0, std, generator=g)

    # activations N(0,1), output gradients N(0, 1e-4), the head's pitch padded to a multiple of 8
    linears = [dp.Linear(normal(i, 1.0), normal(o, 1e-2), d=i, p=o) for i, o in _shapes(case)]
    lm = None
    if case["head"]:
        lm = dp.Linear(normal(d, 1.0), normal(V, 1e-2, ld=(V + 7) // 8 * 8), d=d, p=V)
    # token ids by a Zipf law (s = 1.1), as natural text has them
    w = torch.arange(1, V + 1, device=dev, dtype=torch.float64) ** -1.1
    cdf = torch.cumsum(w, 0) / w.sum()
    u = torch.rand(B * T, generator=g, device=dev, dtype=torch.float64)
    ids = torch.searchsorted(cdf, u, right=True).clamp_(max=V - 1).to(torch.int32).view(B, T)
    pos = None
    if case["positions"]:
        pos = torch.arange(T, dtype=torch.int32, device=dev).repeat(B, 1).contiguous()
    per_example = dict(dtype=torch.float32, device=dev)
    ds = pipeline.DeviceStep(
        B=B, T=T, V=V, C=1.0, sigma=case["sigma"], tied=case["tied"], positions=case["positions"],
        linears=linears, lm=lm, ids=ids, pos_ids=pos, G_emb=normal(d, 1e-2), d_model=d,
        sq=torch.zeros(B, **per_example), clip=torch.zeros(B, **per_example),
        norms=torch.zeros(B, **per_example),
        cross=torch.zeros(B, **per_example) if case["tied"] else None,
        dev_status=torch.zeros(1, dtype=torch.int32, device=dev))
    if case["full"]:                    # two LayerNorms per block, a final one, and every bias
        for _ in range(2 * case["blocks"] + 1):
            gn = normal(d, 1e-2)
            ds.vectors += [dp.Vector(gn, normal(d, 1.0), p=d), dp.Vector(gn, None, p=d)]
        ds.vectors += [dp.Vector(l.G, None, p=l.p) for l in linears]
    pipeline.allocate(ds)
    # the gradients of the blocks, and those of the vectors, live in one flat buffer each, as sharded
    # optimisers keep them (every tensor on a 16-byte boundary)
    flat = {}
    for kind in ("linear", "vector"):
        names = [n for n in ds.outs if n.startswith(kind)]
        if names:
            sizes = [(ds.outs[n].numel() + 3) // 4 * 4 for n in names]
            flat[kind] = torch.zeros(sum(sizes), **per_example)
            at = 0
            for n, size in zip(names, sizes):
                ds.outs[n] = flat[kind][at:at + ds.outs[n].numel()].view(ds.outs[n].shape)
                at += size
    out = {"sq": ds.sq, "norms": ds.norms, "clip": ds.clip, "dev_status": ds.dev_status, **flat}
    out.update({n: t for n, t in ds.outs.items() if n in ("wte", "lm_head", "wpe")})
    state = {"ds": ds, "out": out, "mode": case["mode"], "seed": int(seed)}
    if case["mode"] == "graph":
        state["graph"] = pipeline.StepGraph(ds, seed=int(seed), first_step=0)
    return state


def run(state):
    if state["mode"] == "graph":
        state["graph"].replay()
    else:
        pipeline.dp_step(state["ds"], seed=state["seed"], step=1, noise=state["mode"] == "step")
    return state["out"]


def work(case):
    """Every input read once and every output written once; the symmetric half of each Gram product
    (or the DIRECT product where that is smaller) and the clipped sums."""
    B, T, V, d = case["B"], case["T"], case["V"], case["d_model"]
    es = 4 if case["dtype"] == "f32" else 2
    layers = _shapes(case) + ([(d, V)] if case["head"] else [])
    read = sum(es * B * T * (i + o) for i, o in layers) + es * B * T * d + 4 * B * T
    flops = sum(min(B * T * (T + 1) * (i + o), 2 * B * T * i * o) + 2 * B * T * i * o for i, o in layers)
    flops += 6 * B * T * d
    params = sum(i * o for i, o in layers) + (0 if case["tied"] else V * d)
    if case["positions"]:
        params += pipeline.WPE_ROWS * d
    if case["full"]:
        norms = 2 * case["blocks"] + 1
        read += 2 * es * B * T * d * norms
        params += 2 * d * norms + sum(o for _, o in _shapes(case))
    if case["tied"]:
        flops += 2 * B * T * T * d
    return {"bytes": read + 4 * params + 12 * B, "flops": flops}


def tolerance(case):
    """About four times what the path differed by from the plain fp32 kernels, which sum in another
    order: squared norms 3.6e-6 (bf16 inputs), 1.5e-5 (fp32 inputs as two bf16 terms) and rounding
    only (fp32 too small for that); clipped sums 1.65e-3 (largest 9e-3: one bf16 rounding of R_i * g)
    and 8.5e-6.  Noise of standard deviation sigma hides the rounding of a sum whose norm is about
    sqrt(B) (C = 1) spread over the parameters: measured 3e-5 at 4 096 of them, 7e-7 at 14 million."""
    if case["dtype"] == "f32":
        return {"rel": 6e-5, "max": 1.5e-4} if case["T"] >= 32 else {"rel": 1e-5, "max": 4e-5}
    if case["mode"] == "sums":
        return {"rel": 7e-3, "max": 4e-2}
    linear = sum(i * o for i, o in _shapes(case)) + (case["V"] * case["d_model"] if case["head"] else 0)
    rel = max(1.5e-5, 7e-3 * math.sqrt(case["B"] / linear) / case["sigma"])
    return {"rel": rel, "max": 6 * rel}
