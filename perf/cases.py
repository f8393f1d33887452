"""What is measured when this framework's speed is measured.

Each case is one piece of work that a training program gives to the library through its public entry
points (the ``ZeroLock`` object, or the C calls through their thin binding): whole optimizer steps of the
decoupled per-chunk update, the forward of a chunk, and the single operations that a program can call by
themselves (attention forward and backward, the three products of a linear layer, the fused local
objective, the head fused with it). Sizes are those of the model configurations of this repository (tiny
fp32, GPT-2-small, Llama 1.1B, 3B and 7B shapes), and `draw` gives others of the same ranges, odd ones
among them.

    kind "step"     `steps` optimizer steps of a model of a few layers cut into K chunks, the losses read
                    after each one, then every trained tensor copied out (what a program does before it
                    evaluates or exports its weights)
    kind "forward"  the forward of one chunk, h_out = f_k(h_in), as evaluation and the pipeline use it
    kind "attn"     one layer's causal attention, forward and backward
    kind "linear"   one linear layer: forward (with RoPE for a Llama QKV projection, else bias and
                    residual), the gradient at its input, and the weight gradient accumulated in fp32
    kind "loss"     the fused local objective over given logits
    kind "head"     the frozen head fused with the local objective, in row slices
"""
import ctypes
import math
import types

import torch

from paper_2608_07974_gb300 import binding

LLAMA, GPT2 = binding.ZL_ARCH_LLAMA, binding.ZL_ARCH_GPT2
LR, B1, B2, EPS, WD = 1e-3, 0.9, 0.999, 1e-8, 0.01
ALPHA = 0.5


# ------------------------------------------------------------------------------------------------
# The cases
# ------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: the tiny fp32 model (4 layers, d 128), where launches and latency count
        step("step-tiny-f32", LLAMA, "f32", layers=4, d=128, heads=4, kv=4, ff=344, vocab=512, K=2, B=4, S=64, steps=8),
        # GPT-2-small blocks (LayerNorm, biases, GELU, tied 50257-word head), 8 x 512 tokens, two chunks
        step("step-gpt2", GPT2, "bf16", layers=4, d=768, heads=12, kv=12, ff=3072, vocab=50257, K=2, B=8, S=512, steps=3),
        # the paper's own setting, LoRA rank 4 on a 1.1B-shaped model (GQA 32/4), two micro-batches per window
        step("step-1b-lora", LLAMA, "bf16", layers=2, d=2048, heads=32, kv=4, ff=5632, vocab=32000, K=2, B=4, S=1024,
             steps=2, lora=4, accum=2),
        # the largest: one 7B-shaped layer as a chunk of its own, full fine-tune, 2 x 1024 tokens
        step("step-7b-layer", LLAMA, "bf16", layers=1, d=4096, heads=32, kv=32, ff=11008, vocab=32000, K=1, B=2, S=1024,
             steps=2),
        # evaluation / pipeline direction: the forward of a two-layer chunk of the 3B shape (head dim 100)
        dict(name="forward-3b", kind="forward", layers=2, d=3200, heads=32, kv=32, ff=8640, B=2, S=2048),
        # one layer's attention: GPT-2-small, the 7B shape, and the 1.1B shape at its longest sequence
        dict(name="attn-gpt2", kind="attn", B=8, S=512, H=12, Hkv=12, hd=64),
        dict(name="attn-7b", kind="attn", B=2, S=1024, H=32, Hkv=32, hd=128),
        dict(name="attn-1b-long", kind="attn", B=4, S=2048, H=32, Hkv=4, hd=64),
        # a small ragged batch through one GPT-2 projection, and the 7B QKV projection with its rotation
        dict(name="linear-small", kind="linear", N=203, din=768, dout=2304, S=203, hd=0),
        dict(name="linear-7b-qkv", kind="linear", N=2048, din=4096, dout=12288, S=1024, hd=128),
        # the local objective over a GPT-2 batch of logits, and the 1.1B head in slices of 1024 rows
        dict(name="loss-gpt2", kind="loss", N=4096, V=50257, alpha=ALPHA, kl_dir=0),
        dict(name="head-1b", kind="head", N=4096, d=2048, V=32000, rows=1024, alpha=ALPHA, kl_dir=0),
    ]


def step(name, arch, dtype, layers, d, heads, kv, ff, vocab, K, B, S, steps, lora=0, accum=1):
    return dict(name=name, kind="step", arch=arch, dtype=dtype, layers=layers, d=d, heads=heads, kv=kv, ff=ff, vocab=vocab,
                K=K, B=B, S=S, steps=steps, lora=lora, accum=accum)


def _log(rng, lo, hi, multiple=1):
    """A whole number spread over the logarithm of [lo, hi], a multiple of `multiple`."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(multiple, int(round(v / multiple)) * multiple)


def draw(rng):
    kind = rng.choice(["step", "step", "forward", "attn", "attn", "linear", "linear", "loss", "head"])
    if kind == "step":
        arch = rng.choice([LLAMA, GPT2])
        hd = rng.choice([64, 64, 128])
        heads = _log(rng, 4, 16)
        K = rng.choice([1, 2])
        kv = heads if arch == GPT2 else rng.choice([k for k in (1, 2, 4, heads) if heads % k == 0])
        lora = rng.choice([0, 0, 0, 4]) if arch == LLAMA else 0
        c = step("", arch, "bf16", layers=K * rng.choice([1, 2]), d=heads * hd, heads=heads, kv=kv,
                 ff=_log(rng, 2.5 * heads * hd, 4 * heads * hd, 8), vocab=_log(rng, 1000, 50257), K=K, B=rng.randint(1, 8),
                 S=_log(rng, 48, 512), steps=2, lora=lora, accum=rng.choice([1, 1, 2]))
        del c["name"]
        return c
    if kind == "forward":
        hd = rng.choice([64, 100, 128])
        heads = _log(rng, 4, 32)
        return dict(kind=kind, layers=rng.choice([1, 2]), d=heads * hd // 8 * 8 if heads * hd % 8 == 0 else 2 * heads * hd,
                    heads=heads if heads * hd % 8 == 0 else 2 * heads, kv=heads if heads * hd % 8 == 0 else 2 * heads,
                    ff=_log(rng, 2.5 * heads * hd, 3 * heads * hd, 8), B=rng.randint(1, 4), S=_log(rng, 33, 1024))
    if kind == "attn":
        hd = rng.choice([64, 64, 128, 128, 100])
        H = rng.choice([4, 8, 12, 16, 32])
        S = _log(rng, 33, 4096)
        return dict(kind=kind, B=max(1, min(16, rng.randint(2048, 8192) // S)), S=S, H=H,
                    Hkv=rng.choice([h for h in (1, 2, 4, H, H) if H % h == 0]), hd=hd)
    if kind == "linear":
        hd = rng.choice([0, 0, 64, 128])
        S = _log(rng, 32, 1024)
        return dict(kind=kind, N=S * rng.randint(1, 4), din=_log(rng, 768, 8192, 8),
                    dout=_log(rng, 768, 8192, hd if hd else 8), S=S, hd=hd)
    if kind == "loss":
        return dict(kind=kind, N=_log(rng, 64, 4096), V=_log(rng, 1000, 50257), alpha=rng.choice([0.3, 0.5, 0.5, 1.0]),
                    kl_dir=rng.choice([0, 0, 1]))
    return dict(kind=kind, N=_log(rng, 256, 4096), d=_log(rng, 512, 2048, 64), V=_log(rng, 4000, 32000),
                rows=rng.choice([256, 512, 1024, 2048]), alpha=rng.choice([0.5, 0.5, 1.0]), kl_dir=0)


# ------------------------------------------------------------------------------------------------
# Inputs, all drawn on the device from the seed
# ------------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 + int(seed))


def _randn(g, *shape, std=1.0):
    return torch.randn(*shape, device="cuda", generator=g).mul_(std)


def _bf(x):
    return x.to(torch.bfloat16)


def _token_ids(g, n, V):
    """Token ids with the heavy head of natural text: P(id) ~ 1 / (id + 1)."""
    u = torch.rand(n, device="cuda", generator=g, dtype=torch.float64)
    return (torch.exp(u * math.log(V + 1.0)) - 1.0).long().clamp_(0, V - 1).to(torch.int32)


def _next_labels(ids):
    """Next-token labels of [B, S] ids; the last position of each row lies outside the loss."""
    lab = torch.full_like(ids, -1)
    lab[:, :-1] = ids[:, 1:]
    return lab


def _layer_shapes(c):
    """The trained tensors of a layer (name suffix, shape), weights [out, in]."""
    d, hd, ff = c["d"], c["d"] // c["heads"], c["ff"]
    qkv = (c["heads"] + 2 * c["kv"]) * hd
    if c["arch"] == LLAMA:
        return [("attn_norm.weight", (d,)), ("wqkv", (qkv, d)), ("wo", (d, d)), ("ffn_norm.weight", (d,)),
                ("w1", (2 * ff, d)), ("w2", (d, ff))]
    return [("attn_norm.weight", (d,)), ("attn_norm.bias", (d,)), ("wqkv", (qkv, d)), ("bqkv", (qkv,)), ("wo", (d, d)),
            ("bo", (d,)), ("ffn_norm.weight", (d,)), ("ffn_norm.bias", (d,)), ("w1", (ff, d)), ("b1", (ff,)),
            ("w2", (d, ff)), ("b2", (d,))]


MATRICES = ("wqkv", "wo", "w1", "w2")


def _model(c, g):
    """fp32 parameters by name; the matrices hold values of the compute type."""
    rnd = (lambda x: x.to(torch.bfloat16).float()) if c["dtype"] == "bf16" else (lambda x: x)
    P = {"tok_emb": rnd(_randn(g, c["vocab"], c["d"], std=0.02 if c["arch"] == GPT2 else 0.5))}
    if c["arch"] == GPT2:
        P["pos_emb"] = rnd(_randn(g, c["S"], c["d"], std=0.02))
        P["norm_f.bias"] = _randn(g, c["d"], std=0.02)
    else:
        P["lm_head"] = rnd(_randn(g, c["vocab"], c["d"], std=0.02))
    P["norm_f.weight"] = 1.0 + _randn(g, c["d"], std=0.1)
    for l in range(c["layers"]):
        for s, shape in _layer_shapes(c):
            x = _randn(g, *shape, std=0.02 if s in MATRICES else 0.2 if s[0] == "b" else 0.1)
            P["layers.%d.%s" % (l, s)] = rnd(x) if s in MATRICES else x + 1.0 if s.endswith("norm.weight") else x
            if c["lora"] and s in MATRICES:
                P["layers.%d.%s.lora_a" % (l, s)] = rnd(_randn(g, c["lora"], shape[1], std=0.02))
                P["layers.%d.%s.lora_b" % (l, s)] = rnd(_randn(g, shape[0], c["lora"], std=0.02))
    return P


def _trained(c):
    """(name, shape) of every tensor that a step updates."""
    out = []
    for l in range(c["layers"]):
        for s, shape in _layer_shapes(c):
            n = "layers.%d.%s" % (l, s)
            if not c["lora"]:
                out.append((n, shape))
            elif s in MATRICES:
                out += [(n + ".lora_a", (c["lora"], shape[1])), (n + ".lora_b", (shape[0], c["lora"]))]
    return out


def _batches(c, g):
    got = []
    for _ in range(c["steps"]):
        ids = _token_ids(g, c["B"] * c["S"], c["vocab"]).view(c["B"], c["S"])
        got.append((ids, _next_labels(ids)))
    return got


def _bounds(c):
    return [c["layers"] * k // c["K"] for k in range(c["K"] + 1)]


def _forward_case(c):
    """A forward case as a model: a small vocabulary, since the chunk starts from hidden states."""
    return dict(c, arch=LLAMA, dtype="bf16", vocab=256, K=1, lora=0, accum=1, steps=0)


def _inputs(c, seed):
    g = _gen(seed)
    if c["kind"] == "step":
        return dict(P=_model(c, g), batches=_batches(c, g))
    if c["kind"] == "forward":
        return dict(P=_model(_forward_case(c), g), h=_bf(_randn(g, c["B"] * c["S"], c["d"])))
    if c["kind"] == "attn":
        N, W = c["B"] * c["S"], (c["H"] + 2 * c["Hkv"]) * c["hd"]
        return dict(qkv=_bf(_randn(g, N, W)), dout=_bf(_randn(g, N, c["H"] * c["hd"], std=0.1)))
    if c["kind"] == "linear":
        i = dict(x=_bf(_randn(g, c["N"], c["din"])), w=_bf(_randn(g, c["dout"], c["din"], std=0.02)),
                 dy=_bf(_randn(g, c["N"], c["dout"], std=0.1)), dw=_randn(g, c["dout"], c["din"], std=0.1),
                 bias=_randn(g, c["dout"], std=0.02))
        if c["hd"]:   # the rotation's (cos, sin) table
            a = torch.outer(torch.arange(c["S"], dtype=torch.float64),
                            10000.0 ** (-2.0 * torch.arange(c["hd"] // 2, dtype=torch.float64) / c["hd"]))
            i["cs"] = torch.stack([a.cos(), a.sin()], -1).float().cuda()
        else:
            i["res"] = _bf(_randn(g, c["N"], c["dout"]))
        return i
    lab = _token_ids(g, c["N"], c["V"])
    lab[torch.rand(c["N"], device="cuda", generator=g) < 0.01] = -1
    ld = (c["V"] + 127) // 128 * 128
    if c["kind"] == "loss":
        z = _randn(g, c["N"], ld, std=2.0)
        return dict(z=_bf(z), t=_bf(0.8 * z + _randn(g, c["N"], ld, std=1.2)), lab=lab)
    n = _randn(g, c["N"], c["d"])
    W = _randn(g, ld, c["d"], std=1.0 / math.sqrt(c["d"]))
    W[c["V"]:] = 0
    return dict(n=_bf(n), tn=_bf(0.8 * n + _randn(g, c["N"], c["d"], std=0.6)), W=_bf(W), lab=lab)


# ------------------------------------------------------------------------------------------------
# prepare and run
# ------------------------------------------------------------------------------------------------
# zl_get_param into device memory: the binding's wrapper copies to the host, the C call takes either.
_abi = ctypes.CDLL(binding.LIB_PATH)
_abi.zl_get_param.argtypes = [ctypes.c_void_p, ctypes.c_char_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]


def _engine(c, P):
    dims = types.SimpleNamespace(arch=c["arch"], n_layers=c["layers"], d_model=c["d"], n_heads=c["heads"], n_kv_heads=c["kv"],
                                 d_ff=c["ff"], vocab=c["vocab"], max_seq=c["S"], norm_eps=1e-5, rope_theta=10000.0)
    eng = binding.ZeroLock(dims, c["K"], _bounds(c), dtype=c["dtype"], alpha=ALPHA, lr=LR, beta1=B1, beta2=B2, eps=EPS,
                           weight_decay=WD, accum_m=c["accum"], max_live_chunks=2 if c["K"] > 1 else 0, lora_rank=c["lora"],
                           lora_scale=16.0 / c["lora"] if c["lora"] else 1.0)
    eng.load(P)
    return eng


def prepare(case, seed):
    c, i = case, _inputs(case, seed)
    s = dict(case=case, **i)
    if c["kind"] == "step":
        s["eng"] = _engine(c, s.pop("P"))
        s["out"] = {n: torch.empty(shape, device="cuda") for n, shape in _trained(c)}
    elif c["kind"] == "forward":
        s["eng"] = _engine(_forward_case(c), s.pop("P"))
        s["out"] = torch.empty_like(i["h"])
    elif c["kind"] == "attn":
        s["o"] = torch.empty_like(i["dout"])
        s["lse"] = torch.empty(c["B"], c["H"], c["S"], device="cuda")
        s["dqkv"] = torch.empty_like(i["qkv"])
    elif c["kind"] == "linear":
        s["y"], s["dx"] = torch.empty_like(i["dy"]), torch.empty_like(i["x"])
    elif c["kind"] == "loss":
        s["dz"] = torch.empty_like(i["z"])
    else:
        s["dn"] = torch.empty_like(i["n"])
    if c["kind"] in ("loss", "head"):
        s["rl"], s["loss"] = torch.empty(c["N"], device="cuda"), torch.empty(1, device="cuda")
    return s


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "step":
        losses = [s["eng"].step(ids, lab) for ids, lab in s["batches"]]
        for n, t in s["out"].items():
            if _abi.zl_get_param(s["eng"].ctx, n.encode(), 0, t.data_ptr(), t.numel() * 4, 1) != binding.ZL_OK:
                raise RuntimeError(binding.last_error())
        return dict(losses=losses, weights=s["out"])
    stream = torch.cuda.current_stream().cuda_stream
    if c["kind"] == "forward":
        binding.zl_forward_chunk(s["eng"].ctx, 1, s["h"], None, s["out"], c["B"], c["S"])
        binding.zl_join(s["eng"].ctx)
        return s["out"]
    if c["kind"] == "attn":
        binding.zl_op_attention(1, s["qkv"], s["o"], s["lse"], c["B"], c["S"], c["H"], c["Hkv"], c["hd"], stream)
        binding.zl_op_attention_bwd(1, s["qkv"], s["o"], s["dout"], s["lse"], s["dqkv"], c["B"], c["S"], c["H"], c["Hkv"],
                                    c["hd"], stream)
        return dict(out=s["o"], lse=s["lse"], dqkv=s["dqkv"])
    if c["kind"] == "linear":
        N, din, dout = c["N"], c["din"], c["dout"]
        if c["hd"]:   # the first two thirds (queries and keys) are rotated
            binding.zl_op_qkv_rope(1, N, dout, din, s["x"], s["w"], s["y"], s["cs"], c["S"], c["hd"], _rot_cols(c), None, stream)
        else:
            binding.zl_op_gemm_ex(1, 0, N, dout, din, s["x"], s["w"], s["y"], s["bias"], s["res"], 0, stream)
        binding.zl_op_gemm(1, 1, N, din, dout, s["dy"], s["w"], s["dx"], stream)
        binding.zl_op_gemm(1, 2, dout, din, N, s["dy"], s["x"], s["dw"], stream)
        return dict(y=s["y"], dx=s["dx"], dw=s["dw"])
    if c["kind"] == "loss":
        binding.zl_op_local_loss(1, s["z"], s["t"] if c["alpha"] < 1 else None, s["lab"], c["N"], c["V"], s["z"].shape[1],
                                 c["alpha"], c["kl_dir"], s["dz"], s["rl"], s["loss"], stream)
        return dict(dz=s["dz"], row_loss=s["rl"], loss=s["loss"])
    binding.zl_op_head_loss(1, s["n"], s["tn"] if c["alpha"] < 1 else None, s["W"], s["lab"], c["N"], c["d"], c["V"],
                            s["W"].shape[0], c["alpha"], c["kl_dir"], c["rows"], s["dn"], s["rl"], s["loss"], stream)
    return dict(dn=s["dn"], row_loss=s["rl"], loss=s["loss"])


def _rot_cols(c):
    return c["dout"] // c["hd"] * 2 // 3 * c["hd"]


# ------------------------------------------------------------------------------------------------
# The work that a pass cannot do without
# ------------------------------------------------------------------------------------------------
def work(case):
    c = case
    if c["kind"] in ("step", "forward"):
        m = _forward_case(c) if c["kind"] == "forward" else c
        N, d, hd = c["B"] * c["S"], c["d"], c["d"] // c["heads"]
        mats = sum(a * b for s, (a, b) in ((s, sh) for s, sh in _layer_shapes(m) if s in MATRICES)) * c["layers"]
        attn = 2.0 * c["B"] * c["heads"] * c["S"] ** 2 * hd * c["layers"]     # causal forward, two products
        if c["kind"] == "forward":
            return dict(bytes=2.0 * mats + 4.0 * N * d, flops=2.0 * N * mats + attn)
        n_tr = sum(math.prod(sh) for _, sh in _trained(c))
        head = 2.0 * N * c["vocab"] * d
        flops = N * mats * (4.0 if c["lora"] else 6.0) + 3.5 * attn + (2 * c["K"] + 1) * head
        updates = c["steps"] // c["accum"]
        state = (26.0 if c["dtype"] == "bf16" else 24.0) * n_tr * updates + 4.0 * n_tr
        frozen = (2.0 if c["dtype"] == "bf16" else 4.0) * (c["vocab"] * d + (mats if c["lora"] else 0)) * c["steps"]
        return dict(bytes=state + frozen, flops=c["steps"] * flops)
    if c["kind"] == "attn":
        N, W, A = c["B"] * c["S"], (c["H"] + 2 * c["Hkv"]) * c["hd"], c["H"] * c["hd"]
        return dict(bytes=2.0 * N * (2 * W + 2 * A) + 4.0 * N * c["H"], flops=7.0 * c["B"] * c["H"] * c["S"] ** 2 * c["hd"])
    if c["kind"] == "linear":
        N, i, o = c["N"], c["din"], c["dout"]
        return dict(bytes=2.0 * (2 * N * i + (2 if c["hd"] else 3) * N * o + i * o) + 8.0 * i * o, flops=6.0 * N * i * o)
    t = c["alpha"] < 1
    if c["kind"] == "loss":
        return dict(bytes=(6.0 if t else 4.0) * c["N"] * c["V"], flops=0.0)
    return dict(bytes=2.0 * ((3 if t else 2) * c["N"] * c["d"] + c["V"] * c["d"]),
                flops=(6.0 if t else 4.0) * c["N"] * c["V"] * c["d"])


def tolerance(case):
    """About four times what bf16 rounding (fp32: another order of the sums) makes of each kind's results,
    as measured against the 64-bit results of `exact`."""
    c = case
    if c["kind"] == "step":
        return {"rel": 1e-5, "max": 5e-3} if c["dtype"] == "f32" else {"rel": 2.5e-2, "max": 0.9}
    # (worst relative error seen: steps 7e-3 in bf16 and 2e-6 in fp32, a two-layer forward 6.4e-3, head 3.1e-3, attention 2.4e-3,
    # linear 2.1e-3, loss 1.8e-3)
    return {"forward": {"rel": 2.5e-2, "max": 0.3}, "head": {"rel": 1.2e-2, "max": 0.3}, "attn": {"rel": 1e-2, "max": 0.3},
            "linear": {"rel": 8e-3, "max": 0.1}, "loss": {"rel": 8e-3, "max": 0.1}}[c["kind"]]


# ------------------------------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ------------------------------------------------------------------------------------------------
def _norm64(c, x, w, b):
    if c["arch"] == LLAMA:
        return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-5) * w
    x = x - x.mean(-1, keepdim=True)
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-5) * w + b


def _rot64(x, S):
    """Rotate-half RoPE of x [B, h, S, hd]."""
    half = x.shape[-1] // 2
    a = torch.outer(torch.arange(S, dtype=torch.float64, device=x.device),
                    10000.0 ** (-torch.arange(half, dtype=torch.float64, device=x.device) / half))
    x1, x2 = x[..., :half], x[..., half:]
    return torch.cat([x1 * a.cos() - x2 * a.sin(), x2 * a.cos() + x1 * a.sin()], -1)


def _attn64(qkv, B, S, H, Hkv, hd, rope):
    """Causal attention of [B*S, (H + 2 Hkv) hd]; returns [B*S, H hd] and the log-sum-exp [B, H, S]."""
    x = qkv.view(B, S, H + 2 * Hkv, hd).permute(0, 2, 1, 3)
    q, k, v = x[:, :H], x[:, H:H + Hkv], x[:, H + Hkv:]
    if rope:
        q, k = _rot64(q, S), _rot64(k, S)
    k, v = k.repeat_interleave(H // Hkv, 1), v.repeat_interleave(H // Hkv, 1)
    s = (q @ k.transpose(-1, -2)) / math.sqrt(hd)
    s = s.masked_fill(torch.ones(S, S, dtype=torch.bool, device=s.device).triu(1), -math.inf)
    lse = torch.logsumexp(s, -1)
    return ((s - lse[..., None]).exp() @ v).permute(0, 2, 1, 3).reshape(B * S, H * hd), lse


def _layer64(c, P, l, x):
    p = lambda s: P.get("layers.%d.%s" % (l, s))  # noqa: E731

    def lin(x, s, bias):
        w, b = p(s), p(bias)
        if c["lora"]:
            w = w + 16.0 / c["lora"] * p(s + ".lora_b") @ p(s + ".lora_a")
        return x @ w.T if b is None else x @ w.T + b
    B, S, H, ff = c["B"], c["S"], c["heads"], c["ff"]
    qkv = lin(_norm64(c, x, p("attn_norm.weight"), p("attn_norm.bias")), "wqkv", "bqkv")
    a, _ = _attn64(qkv, B, S, H, c["kv"], c["d"] // H, c["arch"] == LLAMA)
    x = x + lin(a, "wo", "bo")
    u = lin(_norm64(c, x, p("ffn_norm.weight"), p("ffn_norm.bias")), "w1", "b1")
    u = torch.nn.functional.silu(u[:, :ff]) * u[:, ff:] if c["arch"] == LLAMA else torch.nn.functional.gelu(u, approximate="tanh")
    return x + lin(u, "w2", "b2")


def _loss64(z, t, lab, alpha, kl_dir=0):
    """Per-row local objective (0 outside the loss set) and its mean over the loss set."""
    lp = torch.log_softmax(z, -1)
    ok = lab >= 0
    row = -alpha * lp.gather(1, lab.clamp(min=0).long()[:, None])[:, 0]
    if alpha < 1:
        lq = torch.log_softmax(t, -1)
        kl = (lp.exp() * (lp - lq)).sum(-1) if kl_dir == 0 else (lq.exp() * (lq - lp)).sum(-1)
        row = row + (1 - alpha) * kl
    row = torch.where(ok, row, torch.zeros_like(row))
    return row, row.sum() / ok.sum()


def _steps64(c, i):
    P = {n: t.double() for n, t in i["P"].items()}
    head = P["lm_head"] if c["arch"] == LLAMA else P["tok_emb"]
    readout = lambda h: _norm64(c, h, P["norm_f.weight"], P.get("norm_f.bias")) @ head.T  # noqa: E731
    rnd = (lambda x: x.to(torch.bfloat16).double()) if c["dtype"] == "bf16" else (lambda x: x)
    chunks, names = _bounds(c), [n for n, _ in _trained(c)]
    grad = {n: torch.zeros_like(P[n]) for n in names}
    m, v = {n: torch.zeros_like(P[n]) for n in names}, {n: torch.zeros_like(P[n]) for n in names}
    losses, t = [], 0
    for k, (ids, lab) in enumerate(i["batches"]):
        h = P["tok_emb"][ids.view(-1).long()]
        if c["arch"] == GPT2:
            h = h + P["pos_emb"][: c["S"]].repeat(c["B"], 1)
        # the forward reads the matrices in the compute type, the update works on the 32-bit master
        use = {n: (rnd(x) if n.split(".")[-1] in MATRICES + ("lora_a", "lora_b") else x) for n, x in P.items()}
        losses.append([])
        for a, b in zip(chunks, chunks[1:]):
            mine = [n for n in names if a <= int(n.split(".")[1]) < b]
            leaf = {n: use[n].detach().clone().requires_grad_() for n in mine}
            with torch.no_grad():
                teacher = readout(h)
            y = h
            for l in range(a, b):
                y = _layer64(c, {**use, **leaf}, l, y)
            _, loss = _loss64(readout(y), teacher, lab.view(-1), ALPHA)
            for n, dg in zip(mine, torch.autograd.grad(loss, [leaf[n] for n in mine])):
                grad[n] += dg / c["accum"]
            losses[-1].append(float(loss.detach()))
            h = y.detach()
        if (k + 1) % c["accum"] == 0:
            t += 1
            for n in names:
                m[n].mul_(B1).add_(grad[n], alpha=1 - B1)
                v[n].mul_(B2).addcmul_(grad[n], grad[n], value=1 - B2)
                P[n] = P[n] * (1 - LR * WD) - LR / (1 - B1 ** t) * m[n] / ((v[n] / (1 - B2 ** t)).sqrt() + EPS)
                grad[n].zero_()
    return dict(losses=losses, weights={n: P[n] for n in names})


def exact(case, seed):
    c, i = case, _inputs(case, seed)
    if c["kind"] == "step":
        return _steps64(c, i)
    if c["kind"] == "forward":
        m, P, h = _forward_case(c), {n: t.double() for n, t in i["P"].items()}, i["h"].double()
        for l in range(c["layers"]):
            h = _layer64(m, P, l, h)
        return h
    if c["kind"] == "attn":
        x = i["qkv"].double().requires_grad_()
        o, lse = _attn64(x, c["B"], c["S"], c["H"], c["Hkv"], c["hd"], False)
        (dx,) = torch.autograd.grad(o, x, i["dout"].double())
        return dict(out=o.detach(), lse=lse.detach(), dqkv=dx)
    if c["kind"] == "linear":
        x, w, dy = i["x"].double(), i["w"].double(), i["dy"].double()
        y = x @ w.T
        if c["hd"]:
            n, hd, S = _rot_cols(c), c["hd"], c["S"]
            r = y[:, :n].reshape(-1, S, n // hd, hd).transpose(1, 2)
            y = torch.cat([_rot64(r, S).transpose(1, 2).reshape(-1, n), y[:, n:]], 1)
        else:
            y = y + i["bias"].double() + i["res"].double()
        return dict(y=y, dx=dy @ w, dw=i["dw"].double() + dy.T @ x)
    V, lab = c["V"], i["lab"]
    if c["kind"] == "loss":
        z = i["z"][:, :V].double().requires_grad_()
        row, loss = _loss64(z, i["t"][:, :V].double(), lab, c["alpha"], c["kl_dir"])
        (dz,) = torch.autograd.grad(loss, z)
        dz = torch.nn.functional.pad(dz, (0, i["z"].shape[1] - V))
        return dict(dz=dz, row_loss=row.detach(), loss=loss.detach()[None])
    W = i["W"][:V].double()
    n = i["n"].double().requires_grad_()
    row, loss = _loss64(n @ W.T, i["tn"].double() @ W.T, lab, c["alpha"], c["kl_dir"])
    (dn,) = torch.autograd.grad(loss, n)
    return dict(dn=dn, row_loss=row.detach(), loss=loss.detach()[None])
