"""The work this framework is measured on: one pass through its public runners for each case.

A case is one transformer sub-layer (self-attention, the same with low-rank adapters, feed-forward, cross-attention)
at one shape, dtype and set of options, either as a training step (forward and backward) or as the forward alone.
The listed cases are the repository's own workloads (``fbl_inputs.configs``) and generic shapes beside them; ``draw``
gives more of the same kinds over the ranges a user has.  Inputs are drawn on the GPU from the seed: activations and
output gradients N(0, 1), weights N(0, w_std^2), norm gains around 1.
"""
from __future__ import annotations

import math

import torch

from fbl_inputs import CONFIGS, MLP_CONFIGS, XATTN_CONFIGS, LayerConfig, MlpConfig, XattnConfig
from paper_2607_21624_b200 import LayerRunner
from paper_2607_21624_b200.binding import TENSOR, _check, lib
from paper_2607_21624_b200.lora import ADAPTER, LoraRunner
from paper_2607_21624_b200.mlp import MLP_TENSOR, MlpRunner
from paper_2607_21624_b200.xattn import XattnRunner

# A drawn case's largest flop count: well inside the time of the largest listed case for what runs at tensor-core
# rates, and about the fp32 listed case's for fp32, for less than a tile of tokens and for single-head keys of width 64.
DRAW_FLOPS, DRAW_FLOPS_SMALL = 2.0e12, 1.2e10


def _layer(name, cfg, mode="step", boundary=False, rank=0):
    return {"name": name, "kind": "lora" if rank else "layer", "mode": mode, "boundary": boundary, "rank": rank,
            "batch": cfg.batch, "seq": cfg.seq, "d_model": cfg.d_model, "heads": cfg.n_q_heads, "kv_heads": cfg.n_kv_heads,
            "head_dim": cfg.head_dim, "dtype": cfg.dtype, "norm": cfg.norm, "causal": cfg.causal, "bias": cfg.has_bias,
            "residual": cfg.residual, "rope": cfg.rope_base, "w_std": cfg.w_std}


def _mlp(name, cfg, mode="step", boundary=False):
    return {"name": name, "kind": "mlp", "mode": mode, "boundary": boundary, "batch": cfg.batch, "seq": cfg.seq,
            "d_model": cfg.d_model, "d_ff": cfg.d_ff, "dtype": cfg.dtype, "norm": cfg.norm, "act": cfg.act,
            "bias": cfg.has_bias, "residual": cfg.residual, "w_std": cfg.w_std}


def _xattn(name, cfg, mode="step", boundary=False):
    return {"name": name, "kind": "xattn", "mode": mode, "boundary": boundary, "batch": cfg.batch, "seq": cfg.seq,
            "seq_kv": cfg.seq_kv, "d_model": cfg.d_model, "d_mem": cfg.d_mem, "heads": cfg.n_q_heads,
            "kv_heads": cfg.n_kv_heads, "head_dim": cfg.head_dim, "dtype": cfg.dtype, "norm": cfg.norm,
            "bias": cfg.has_bias, "residual": cfg.residual, "w_std": cfg.w_std}


def listed():
    return [
        # the smallest workload: one 64-token fp32 sequence, where launches and host work are all there is
        _layer("tiny fp32 step", CONFIGS[1]),
        # a short prompt through one layer of a small decoder, forward only: fewer tokens than one compute tile
        _layer("short prompt forward", LayerConfig("p", 1, 50, 768, 12, 12, 64, "bf16", "layernorm", True, True, True, 1e-5, 0, 0.02), mode="forward"),
        # a small decoder's training step inside a program that keeps its activations row-major: X and dY are packed,
        # Y and dX unpacked in every pass
        _layer("gpt2-small step row-major", CONFIGS[2], boundary=True),
        # an image encoder's step: ragged 197-token sequences, many of them, no mask
        _layer("vit-base step", CONFIGS[3]),
        # grouped-query decoder with long sequences
        _layer("llama1b gqa step", CONFIGS[4]),
        # the largest: one 8192-token sequence, heads of 128
        _layer("llama7b long step", CONFIGS[5]),
        # prompts of odd length through a multi-query decoder layer with rotary embedding, forward only
        _layer("multi-query forward", LayerConfig("q", 4, 777, 1024, 16, 1, 64, "bf16", "rmsnorm", True, False, True, 1e-5, 0, 0.02, 0.0, 10000.0), mode="forward"),
        # adapter fine-tuning at 512 tokens with frozen weights: rank 16, rotary embedding
        _layer("adapters rank 16 step", LayerConfig("l", 4, 512, 2048, 32, 8, 64, "bf16", "rmsnorm", True, False, True, 1e-5, 0, 0.02, 0.0, 10000.0), rank=16),
        # full-precision training of the image encoder on a few images
        _layer("vit-base fp32 step", LayerConfig("f", 4, 197, 768, 12, 12, 64, "fp32", "layernorm", False, True, True, 1e-6, 0, 0.02)),
        # feed-forward halves: the small decoder's with biases, the larger one's gated
        _mlp("gpt2-small mlp step", MLP_CONFIGS["gpt2"]),
        _mlp("llama1b gated mlp step", MLP_CONFIGS["llama1b"]),
        # a speech decoder's cross-attention over 1500 encoder positions
        _xattn("whisper-large cross step", XATTN_CONFIGS["whisper-large"]),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        kind = rng.choices(["layer", "lora", "mlp", "xattn"], [5, 2, 3, 2])[0]
        fp32 = rng.random() < 0.2
        case = {"kind": kind, "mode": "forward" if rng.random() < 0.3 else "step", "boundary": rng.random() < 0.25,
                "batch": _log_int(rng, 1, 64), "seq": _log_int(rng, 8, 8192), "dtype": "fp32" if fp32 else "bf16",
                "norm": rng.choice(["layernorm", "rmsnorm"]), "bias": rng.random() < 0.5, "residual": rng.random() < 0.5,
                "w_std": 0.02}
        if kind == "mlp":
            case["d_model"] = 64 * _log_int(rng, 2, 64)
            case["d_ff"] = 64 * max(2, int(case["d_model"] / 64 * rng.choice([2, 2.6875, 4])))
            case["act"] = rng.choice(["gelu", "swiglu"])
        else:
            hd = rng.choice([32, 64, 128] if fp32 else [64, 64, 128])
            heads = _log_int(rng, 2, 4096 // hd)
            kv = heads if rng.random() < 0.5 else rng.choice([k for k in range(1, heads + 1) if heads % k == 0])
            # mostly the model's width over its heads, sometimes a width of its own
            d_model = heads * hd if rng.random() < 0.75 and heads * hd >= 128 else 64 * _log_int(rng, 2, 64)
            case.update(d_model=d_model, heads=heads, kv_heads=kv, head_dim=hd)
            if kind == "xattn":
                case["seq_kv"] = _log_int(rng, 8, 4096)
                case["d_mem"] = d_model if rng.random() < 0.7 else 64 * _log_int(rng, 2, 32)
            else:
                case["causal"] = rng.random() < 0.7
                case["rope"] = 10000.0 if rng.random() < 0.4 else 0.0
                case["rank"] = rng.choice([4, 8, 16, 32, 64]) if kind == "lora" else 0
        small = fp32 or case["batch"] * case["seq"] < 128 or case["batch"] * case.get("seq_kv", 128) < 128 or \
            case.get("kv_heads", 2) * case.get("head_dim", 64) < 128
        if work(case)["flops"] <= (DRAW_FLOPS_SMALL if small else DRAW_FLOPS) and case["batch"] * case["seq"] <= 32768:
            return case


def _config(c):
    eps = 1e-5
    if c["kind"] == "mlp":
        return MlpConfig("case", c["batch"], c["seq"], c["d_model"], c["d_ff"], c["dtype"], c["norm"], c["act"], c["bias"],
                         c["residual"], eps, 0, c["w_std"])
    if c["kind"] == "xattn":
        return XattnConfig("case", c["batch"], c["seq"], c["seq_kv"], c["d_model"], c["d_mem"], c["heads"], c["kv_heads"],
                           c["head_dim"], c["dtype"], c["norm"], c["bias"], c["residual"], eps, 0, c["w_std"])
    return LayerConfig("case", c["batch"], c["seq"], c["d_model"], c["heads"], c["kv_heads"], c["head_dim"], c["dtype"],
                       c["norm"], c["causal"], c["bias"], c["residual"], eps, 0, c["w_std"], 0.0, c["rope"])


def prepare(case, seed):
    cfg = _config(case)
    kind, step, rank = case["kind"], case["mode"] == "step", case.get("rank", 0)
    gen = torch.Generator(device="cuda").manual_seed(seed)

    if kind == "mlp":
        run, ids = MlpRunner(cfg), MLP_TENSOR
        mats = [m for m in MlpRunner.IN_MATS.items() if m[0] in run.buf]
        shape = lambda name: run._shape(MlpRunner.IN_MATS[name])
        vecs = {"b1": 0, "bg": 0, "b2": 0}
    else:
        run = LoraRunner(cfg, rank) if kind == "lora" else XattnRunner(cfg) if kind == "xattn" else LayerRunner(cfg)
        ids, mats, shape = TENSOR, list(run.MATS.items()), run._shape
        vecs = {"bq": 0, "bk": 0, "bv": 0, "bo": 0}
    stream = torch.cuda.current_stream().cuda_stream
    normal = lambda size, std: torch.randn(size, generator=gen, device="cuda").mul_(std).to(run.tdtype)
    row_major = {}
    for name, tid in mats:
        rm = normal(shape(name), cfg.w_std if name.startswith("W") else 1.0)
        run.plan.pack(ids[tid], rm.data_ptr(), run.buf[name].data_ptr(), stream)
        if case["boundary"] and name in ("X", "dY"):
            row_major[name] = rm
    for name, mean in {"gamma": 1.0, "beta": 0.0, **vecs}.items():
        v = run.vec[name]
        v.copy_(torch.randn(v.numel(), generator=gen, device="cuda") * (0.1 if name in ("gamma", "beta") else cfg.w_std) + mean)
    if kind == "lora":
        run.buf["A_all"].zero_()
        run.buf["B_all"].zero_()
        for name, which in ADAPTER.items():
            rm = normal(run._adapter_shape(name), 0.05)
            _check(lib().fbl_lora_pack(run.plan._h, which, rm.data_ptr(), run.buf[name[0] + "_all"].data_ptr(), stream))

    # the pass's outputs: the runner's own buffers
    tiled = lambda name: run.buf[name].view(run.tdtype)
    out = {}
    if not step:
        out["Y"] = tiled("Y")
    elif kind == "lora":                 # weights and norm are frozen: adapters and input receive gradients
        out.update({"Y": tiled("Y"), "dX": tiled("dX")})
        w = 64 if case["dtype"] == "bf16" else 32                         # columns of a panel
        da = tiled("dA_all").view(-1, cfg.d_model, w)                     # [panels, rows, w]
        db = tiled("dB_all").view(-1, 192, w)
        col = 0
        for i, (k, n) in enumerate((("q", cfg.d_q), ("k", cfg.d_kv), ("v", cfg.d_kv))):
            for p in range(-(-rank // w)):
                out["dA%s%d" % (k, p)] = da[i * 64 // w + p, :, :min(w, rank - p * w)]
            out["dB" + k] = db[col // w:(col + n) // w, 64 * i:64 * i + rank]
            col += n
    else:
        out.update({name: tiled(name) for name in run.OUT_MATS if name in run.buf})
        out["dgamma"] = run.vec["dgamma"]
        if cfg.norm == "layernorm":
            out["dbeta"] = run.vec["dbeta"]
        if cfg.has_bias and kind == "mlp":
            out.update({n: run.vec[n] for n in ("db1", "db2") + (("dbg",) if cfg.gated else ())})
        elif cfg.has_bias:
            # without the rotation the key bias shifts every score of a row alike, so its gradient is zero and what
            # comes back is rounding noise that no two implementations share
            out.update({n: run.vec[n] for n in ("dbq", "dbv", "dbo") + (("dbk",) if cfg.rope_base > 0 else ())})
    state = {"run": run, "call": run.step if step else run.forward, "out": out, "boundary": case["boundary"], "step": step}
    if case["boundary"]:
        state.update(ids=(ids["X"], ids["X"] if kind == "mlp" else ids["DY"]), rm=row_major)
        for name in ("Y", "dX") if step else ("Y",):
            state["rm"][name] = torch.empty(shape("X"), dtype=run.tdtype, device="cuda")
            out[name] = state["rm"][name]
    torch.cuda.synchronize()
    return state


def run(state):
    if not state["boundary"]:
        state["call"]()
        return state["out"]
    r, rm, (x_id, dy_id) = state["run"], state["rm"], state["ids"]
    stream = torch.cuda.current_stream().cuda_stream
    r.plan.pack(x_id, rm["X"].data_ptr(), r.buf["X"].data_ptr(), stream)
    if state["step"]:
        r.plan.pack(dy_id, rm["dY"].data_ptr(), r.buf["dY"].data_ptr(), stream)
    state["call"]()
    r.plan.unpack(x_id, r.buf["Y"].data_ptr(), rm["Y"].data_ptr(), stream)
    if state["step"]:
        r.plan.unpack(x_id, r.buf["dX"].data_ptr(), rm["dX"].data_ptr(), stream)
    return state["out"]


def work(case):
    c = case
    step, e = c["mode"] == "step", 4 if c["dtype"] == "fp32" else 2
    n, d = c["batch"] * c["seq"], c["d_model"]
    if c["kind"] == "mlp":
        weights = (3 if c["act"] == "swiglu" else 2) * d * c["d_ff"]
        flops = 2.0 * n * weights * (3 if step else 1)
        elements = n * d * (4 if step else 2) + weights * (2 if step else 1)
        return {"bytes": float(e * elements), "flops": flops}
    dq, dkv = c["heads"] * c["head_dim"], c["kv_heads"] * c["head_dim"]
    if c["kind"] == "xattn":
        nk, dm, pairs = c["batch"] * c["seq_kv"], c["d_mem"], float(c["seq"]) * c["seq_kv"]
        weights, memory = 2 * d * dq + 2 * dm * dkv, nk * dm
        proj = 4.0 * n * d * dq + 4.0 * nk * dm * dkv
    else:
        pairs = c["seq"] * (c["seq"] + 1) / 2 if c["causal"] else float(c["seq"]) ** 2
        weights, memory = 2 * d * dq + 2 * d * dkv, 0
        proj = 2.0 * n * weights
    one = 2.0 * c["batch"] * dq * pairs                       # one of the two attention products
    rank = c.get("rank", 0)
    if rank:
        adapters = rank * (3 * d + dq + 2 * dkv)
        flops = (2 if step else 1) * proj + (6 if step else 2) * one + 2.0 * n * adapters * (3 if step else 1)
        elements = n * d * (4 if step else 2) + weights + adapters * (2 if step else 1)
    else:
        flops = (3 if step else 1) * proj + (6 if step else 2) * one
        elements = n * d * (4 if step else 2) + (weights + memory) * (2 if step else 1)
    return {"bytes": float(e * elements), "flops": flops}


def tolerance(case):
    # bf16: results and the tensors between the kernels are rounded to 8 bits, each step adding 2e-3 or so
    return {"rel": 2e-5} if case["dtype"] == "fp32" else {"rel": 1e-2}
