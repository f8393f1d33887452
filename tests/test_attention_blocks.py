"""The tcgen05 attention at the edges of its 128-row blocks and of its head deal (GPU), against fp32 autograd."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import paper_2608_07974_gb300 as pkg
    pkg.build()
    from paper_2608_07974_gb300 import binding
    return binding


# One block exactly, one row more and one less, a last block of one row; grouped heads whose dK / dV kernel takes
# all query heads of a KV head in one CTA.
@pytest.mark.parametrize("Bb,S,H,Hkv,hd", [(2, 127, 2, 2, 64), (2, 128, 2, 2, 128), (1, 129, 2, 1, 128), (3, 256, 3, 3, 64),
                                           (1, 257, 2, 2, 64), (1, 385, 2, 2, 128), (16, 200, 32, 8, 64),
                                           (40, 129, 32, 8, 128), (16, 257, 32, 4, 128), (8, 641, 64, 8, 64)])
def test_attention_block_edges(B, Bb, S, H, Hkv, hd):
    g = torch.Generator(device="cuda").manual_seed(S + 7 * H + hd)
    W = (H + 2 * Hkv) * hd
    qkv = torch.randn(Bb * S, W, device="cuda", generator=g).to(torch.bfloat16)
    dout = torch.randn(Bb * S, H * hd, device="cuda", generator=g).to(torch.bfloat16)
    out = torch.full((Bb * S, H * hd), float("nan"), device="cuda", dtype=torch.bfloat16)
    lse = torch.full((Bb, H, S), float("nan"), device="cuda")
    dqkv = torch.full_like(qkv, float("nan"))
    B.zl_op_attention(B.ZL_DTYPE_BF16, qkv, out, lse, Bb, S, H, Hkv, hd)
    B.zl_op_attention_bwd(B.ZL_DTYPE_BF16, qkv, out, dout, lse, dqkv, Bb, S, H, Hkv, hd)
    torch.cuda.synchronize()
    x = qkv.float().requires_grad_(True)
    t = x.view(Bb, S, H + 2 * Hkv, hd).transpose(1, 2)
    k, v = (t[:, a:a + Hkv].repeat_interleave(H // Hkv, 1) for a in (H, H + Hkv))
    s = (t[:, :H] @ k.transpose(-1, -2)) / hd ** 0.5
    s = s.masked_fill(torch.ones(S, S, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    ref = (torch.softmax(s, -1) @ v).transpose(1, 2).reshape(Bb * S, H * hd)
    (gx,) = torch.autograd.grad(ref, x, dout.float())
    # P, dS and the results are rounded to bf16 (2^-9 relative each, independent errors): well under 1% in norm
    assert float((lse - torch.logsumexp(s, -1)).abs().max()) <= 1e-5 * S ** 0.5
    assert float((out.float() - ref).norm() / ref.norm()) <= 1e-2
    for lo, hi in ((0, H * hd), (H * hd, (H + Hkv) * hd), ((H + Hkv) * hd, W)):
        assert float((dqkv[:, lo:hi].float() - gx[:, lo:hi]).norm() / gx[:, lo:hi].norm()) <= 1e-2, (lo, hi)
    again = torch.empty_like(dqkv)
    B.zl_op_attention_bwd(B.ZL_DTYPE_BF16, qkv, out, dout, lse, again, Bb, S, H, Hkv, hd)
    assert torch.equal(again, dqkv)   # fixed summation order


# The forward's 64-key blocks: two keys (with one dQ and dK are exactly zero and have no relative error), a block exactly, one key more and less, an odd and an even number of them.
@pytest.mark.parametrize("S,hd", [(2, 64), (63, 128), (64, 64), (65, 128), (191, 64), (193, 64), (193, 128)])
def test_attention_key_blocks(B, S, hd):
    test_attention_block_edges(B, 2, S, 2, 1, hd)


# Grouped heads whose dK / dV kernel takes one or several query heads of a KV head in one CTA and sums the partials afterwards
# (with 152 SMs: 1 of 2, 2 of 4, 2 of 8, 4 of 8).
@pytest.mark.parametrize("Bb,S,H,Hkv,hd", [(1, 257, 2, 1, 128), (16, 385, 8, 2, 64), (8, 513, 16, 2, 64), (8, 641, 16, 2, 128)])
def test_attention_head_shares(B, Bb, S, H, Hkv, hd):
    test_attention_block_edges(B, Bb, S, H, Hkv, hd)


@pytest.mark.parametrize("S,hd", [(300, 64), (450, 128)])
def test_attention_moving_maximum(B, S, hd):
    """Scores that grow with the key's position: the running maximum moves, and O is rescaled, in every block."""
    g = torch.Generator(device="cuda").manual_seed(S)
    q, k, v = (torch.randn(S, 2, hd, device="cuda", generator=g) for _ in range(3))
    q[..., 0] = 1.0
    k[..., 0] = torch.arange(S, device="cuda").float()[:, None] * (0.4 * hd ** 0.5)   # 0.4 a key, 26 a block (> 8 in log2)
    qkv = torch.cat([q, k, v], 1).reshape(S, 6 * hd).to(torch.bfloat16)
    out, lse = torch.empty(S, 2 * hd, device="cuda", dtype=torch.bfloat16), torch.empty(1, 2, S, device="cuda")
    B.zl_op_attention(B.ZL_DTYPE_BF16, qkv, out, lse, 1, S, 2, 2, hd)
    t = qkv.double().view(S, 6, hd).transpose(0, 1)
    s = (t[:2] @ t[2:4].transpose(-1, -2)) / hd ** 0.5
    s = s.masked_fill(torch.ones(S, S, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    ref = (torch.softmax(s, -1) @ t[4:]).transpose(0, 1).reshape(S, 2 * hd)
    # fp32 scores of up to 0.4 S carry errors of 2^-24 of their terms; P and the result are rounded to bf16
    assert float((lse[0].double() - torch.logsumexp(s, -1)).abs().max()) <= 0.4 * S * hd * 2.0 ** -23
    assert float((out.double() - ref).norm() / ref.norm()) <= 1e-2


@pytest.mark.parametrize("S,hd", [(100, 64), (128, 128), (129, 128), (300, 64)])
def test_attention_first_maximum(B, S, hd):
    """A row's largest probability among its first 128 keys is 1, which bf16 holds, also where the key lies in the second 64: one
    key there outweighs the first by 2^0.1 to 2^7.6, less than what moves the running maximum."""
    key, D = 64 + (S - 64) // 2 if S < 128 else 90, 16
    g = torch.Generator(device="cuda").manual_seed(S)
    q, k = torch.zeros(S, 2, hd, device="cuda"), torch.zeros(S, 2, hd, device="cuda")
    q[..., 0] = torch.linspace(0.1, 7.6, S, device="cuda")[:, None] * 0.6931 * hd ** 0.5 / D   # log2 units over the first key
    k[key, :, 0] = D
    q[..., 1], k[..., 1] = -30.0, hd ** 0.5       # every key but two: e^-30 of the first
    k[0, :, 1] = k[key, :, 1] = 0.0
    v = 1.0 + torch.rand(S, 2, hd, device="cuda", generator=g)
    qkv = torch.cat([q, k, v], 1).reshape(S, 6 * hd).to(torch.bfloat16)
    out, lse = torch.empty(S, 2 * hd, device="cuda", dtype=torch.bfloat16), torch.empty(1, 2, S, device="cuda")
    B.zl_op_attention(B.ZL_DTYPE_BF16, qkv, out, lse, 1, S, 2, 2, hd)
    t = qkv.double().view(S, 6, hd).transpose(0, 1)
    s = (t[:2] @ t[2:4].transpose(-1, -2)) / hd ** 0.5
    s = s.masked_fill(torch.ones(S, S, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    ref = (torch.softmax(s, -1) @ t[4:]).transpose(0, 1)[key:]
    # bf16 rounds by at most 2^-8 of a value's power of two: the result once, and the first key's probability once, a share w2 of
    # the result (times a value of at most 2); fp32 sums and exponentials stay below 1e-5
    w2 = torch.softmax(s, -1)[:, key:, 0].transpose(0, 1)[..., None]
    got = out.double().view(S, 2, hd)[key:]
    bound = 2.0 ** (torch.floor(torch.log2(ref)) - 8) + 2.0 ** -8 * w2 * 2.0 + 1e-5
    assert bool(((got - ref).abs() <= bound).all()), float(((got - ref).abs() / bound).max())


# The launch counter: one kernel forward and two backward (one each in fp32), a reduction where a KV head's query heads lie in
# several CTAs, two and four copies more where heads are padded to 64 or 128.
@pytest.mark.parametrize("dt,Bb,S,H,Hkv,hd,fwd,bwd", [(1, 2, 100, 4, 4, 64, 1, 2), (1, 1, 257, 2, 1, 128, 1, 3), (1, 40, 129, 32, 8, 128, 1, 2),
                                                      (1, 8, 513, 16, 2, 64, 1, 3), (1, 2, 100, 4, 4, 50, 3, 6), (0, 2, 100, 4, 2, 64, 1, 1)])
def test_attention_launch_count(B, dt, Bb, S, H, Hkv, hd, fwd, bwd):
    td = torch.bfloat16 if dt else torch.float32
    qkv, out = torch.randn(Bb * S, (H + 2 * Hkv) * hd, device="cuda").to(td), torch.empty(Bb * S, H * hd, device="cuda", dtype=td)
    lse, n0 = torch.empty(Bb, H, S, device="cuda"), B.zl_kernel_launches()
    B.zl_op_attention(dt, qkv, out, lse, Bb, S, H, Hkv, hd)
    n1 = B.zl_kernel_launches()
    B.zl_op_attention_bwd(dt, qkv, out, torch.randn_like(out), lse, torch.empty_like(qkv), Bb, S, H, Hkv, hd)
    torch.cuda.synchronize()
    assert (n1 - n0, B.zl_kernel_launches() - n1) == (fwd, bwd)


@pytest.mark.parametrize("hd,fwd,bwd", [(64, 1, 2), (50, 3, 6)])
def test_attention_profile_count(B, hd, fwd, bwd):
    """The step's profile counts the same launches."""
    import synth
    from tests.gpu_common import engine_for
    d = synth.ModelDims(synth.ARCH_GPT2, 1, 4 * hd, 4, 4, 256, 300, 64)
    w = synth.Workload("attn-profile", d, "bf16", batch=2, seq=64, K=1, steps=1, seed=3)
    eng = engine_for(w)
    eng.load(synth.make_params(d, w.seed))
    ids, labels = (t.cuda() for t in synth.make_batch(w, 0))
    eng.step(ids, labels)
    B.zl_profile(eng.ctx, True)
    eng.step(ids, labels)
    p = B.zl_profile_read(eng.ctx)
    eng.close()
    assert (p["attn_fwd"]["launches"], p["attn_bwd"]["launches"]) == (fwd, bwd)
