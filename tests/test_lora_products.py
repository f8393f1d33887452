"""LoRA's products folded into the base products (bf16): ranks around one and two k blocks of 64, ragged token
counts, head dims with and without the rotation in the epilogue, both architectures, against the oracle in fp32
on the same bf16-rounded weights."""
import pytest
import torch

import synth
from tests.gpu_common import cosine, engine_for, fro_rel, oracle_for, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arch,rank,heads,kv,hd,batch,seq", [
    (synth.ARCH_LLAMA, 4, 4, 2, 64, 3, 67), (synth.ARCH_LLAMA, 16, 2, 2, 128, 2, 130), (synth.ARCH_LLAMA, 20, 4, 4, 64, 1, 40),
    (synth.ARCH_LLAMA, 70, 4, 1, 64, 2, 64), (synth.ARCH_LLAMA, 8, 4, 4, 50, 2, 33), (synth.ARCH_GPT2, 4, 4, 4, 64, 5, 51)])
def test_lora_gradients(arch, rank, heads, kv, hd, batch, seq):
    d = synth.ModelDims(arch, 2, heads * hd, heads, kv, 328, 640, 256)
    w = synth.Workload("lora-products", d, "bf16", batch=batch, seq=seq, K=2, steps=1, seed=77)
    P = synth.make_params(d, w.seed)
    P.update(synth.make_lora_params(d, w.seed, rank, b_std=0.05))
    P = {n: (synth.round_bf16(t) if t.dim() == 2 else t) for n, t in P.items()}
    kw = dict(accum_m=2, lora_rank=rank, lora_scale=16.0 / rank)   # a window of two: the gradients stay readable
    eng = engine_for(w, **kw)
    eng.load(P)
    ids, labels = synth.make_batch(w, 0)
    losses = eng.step(ids.cuda(), labels.cuda())
    orc = oracle_for(w, P, dtype=torch.float32, **kw)
    h = eng.embed(ids.cuda()).float().cpu().view(batch, seq, -1)
    for k in (1, 2):
        L, g, _ = orc.local_grad(k, h, labels)
        assert rel(losses[k - 1], L) <= 2e-2
        for n in orc.chunk_names(k):
            assert cosine(eng.get(n, 1), g[n]) >= 0.999, (k, n)
        h = eng.forward_chunk(k, h.view(batch * seq, -1).to(torch.bfloat16).cuda(), None, batch, seq)
        h = h.float().cpu().view(batch, seq, -1)
    eng.close()


# Token counts on the other side of the rank-16 kernels' lines: 32 rows a CTA (the last one ragged), and the tokens
# shared by clusters of eight and of four.
@pytest.mark.parametrize("batch,seq", [(10, 251), (5, 255), (3, 200)])
def test_lora_gradients_many_tokens(batch, seq):
    test_lora_gradients(synth.ARCH_LLAMA, 16, 2, 1, 64, batch, seq)


# Where the product does not rotate (head dim 50) the forward forms the same products as where it does (64): a RoPE pass and the
# head padding's two copies more, and nothing twice.
def test_lora_forward_launches():
    from paper_2608_07974_gb300 import binding
    counts = []
    for hd in (64, 50):
        d = synth.ModelDims(synth.ARCH_LLAMA, 1, 4 * hd, 4, 4, 328, 640, 64)
        w = synth.Workload("lora-launches", d, "bf16", batch=2, seq=64, K=1, steps=1, seed=7)
        P = synth.make_params(d, w.seed)
        P.update(synth.make_lora_params(d, w.seed, 8, b_std=0.05))
        eng = engine_for(w, lora_rank=8, lora_scale=2.0)
        eng.load({n: (synth.round_bf16(t) if t.dim() == 2 else t) for n, t in P.items()})
        h = torch.randn(128, 4 * hd, device="cuda").to(torch.bfloat16)
        n0 = binding.zl_kernel_launches()
        eng.forward_chunk(1, h, None, 2, 64)
        counts.append(binding.zl_kernel_launches() - n0)
        eng.close()
    assert counts[1] - counts[0] == 3, counts


# The product with the LoRA term as further k blocks under every kind of plan (tiles of 64, 128, 256, CTA pairs with an odd tile row
# at the end, splits whose last share is the term alone), both modes, with the rotation in the epilogue and without.
@pytest.mark.parametrize("tile", ["64:1", "128:1:0", "128:1:1", "256:1:0", "256:1:1", "64:4", "128:4:0", "128:4:1", "256:3:1"])
@pytest.mark.parametrize("rank,hd", [(16, 64), (70, 64), (16, 50), (70, 128)])
def test_lora_every_plan(monkeypatch, tile, rank, hd):
    batch, seq = 3, 107   # 321 tokens: three tile rows
    d = synth.ModelDims(synth.ARCH_LLAMA, 1, 4 * hd, 4, 2, 328, 640, 128)
    w = synth.Workload("lora-plans", d, "bf16", batch=batch, seq=seq, K=1, steps=1, seed=79)
    P = synth.make_params(d, w.seed)
    P.update(synth.make_lora_params(d, w.seed, rank, b_std=0.05))
    P = {n: (synth.round_bf16(t) if t.dim() == 2 else t) for n, t in P.items()}
    kw = dict(accum_m=2, lora_rank=rank, lora_scale=1.0)   # the term is about a third of the layer's output
    eng = engine_for(w, **kw)
    eng.load(P)
    ids, labels = synth.make_batch(w, 0)
    monkeypatch.setenv("ZL_GEMM_TILE", tile)
    loss = eng.step(ids.cuda(), labels.cuda())[0]
    h = eng.embed(ids.cuda())
    y = eng.forward_chunk(1, h, None, batch, seq)
    monkeypatch.delenv("ZL_GEMM_TILE")
    orc = oracle_for(w, P, dtype=torch.float32, **kw)
    h = h.float().cpu().view(batch, seq, -1)
    L, g, ref = orc.local_grad(1, h, labels)
    # about ten roundings to bf16 (2^-8 / sqrt(3) of a value in the mean, at most half of it on average) lie before each gradient,
    # four before each output: 7e-3 and 5e-3; a wrong or missing term is 0.1 to 1
    assert rel(loss, L) <= 1e-3
    assert fro_rel(y.float().cpu().view(batch, seq, -1) - h, ref - h) <= 1e-2
    for n in orc.chunk_names(1):
        assert fro_rel(eng.get(n, 1), g[n]) <= 1.5e-2, n
    eng.close()
