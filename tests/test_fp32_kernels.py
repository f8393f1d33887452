"""The fp32 CUDA-core kernels at the edges of their tiles, splits and head-dim classes (GPU), against float64."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import paper_2608_07974_gb300 as pkg
    pkg.build()
    from paper_2608_07974_gb300 import binding
    return binding


# Tiles of 32 with K in 1, 2 or 4 shares (the last one short), tiles of 64, ragged rows and columns, and rows that
# are not a multiple of 16 bytes (the plain kernel).
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("M,N,K", [(32, 32, 64), (256, 128, 344), (256, 384, 128), (100, 36, 260), (4, 4, 4), (36, 1200, 512),
                                   (1300, 1236, 68), (33, 35, 37), (256, 688, 128), (64, 64, 1028)])
def test_fp32_gemm(B, mode, M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + 3 * N + 7 * K)
    shp = {0: ((M, K), (N, K)), 1: ((M, K), (K, N)), 2: ((K, M), (K, N))}[mode]
    a, b = (torch.randn(*s, device="cuda", generator=g) for s in shp)
    c0 = torch.randn(M, N, device="cuda", generator=g)
    bias, c = torch.randn(N, device="cuda", generator=g), c0.clone()
    p = {0: lambda: a.double() @ b.double().T, 1: lambda: a.double() @ b.double(), 2: lambda: a.double().T @ b.double()}[mode]()
    if mode == 2:
        B.zl_op_gemm(0, 2, M, N, K, a, b, c)
        ref = c0.double() + p
    else:
        B.zl_op_gemm_ex(0, mode, M, N, K, a, b, c, bias, c0, 0)
        ref = p + bias.double() + c0.double()
    # an fp32 sum of K unit-variance products: at most K rounding errors of 2^-24 of a partial sum of about sqrt(K)
    assert float((c - ref).abs().max()) <= 2.0 ** -24 * 4 * (K + 8) ** 0.5 * max(8.0, K ** 0.5)
    assert float((c - ref).norm() / ref.norm()) <= 1e-6


@pytest.mark.parametrize("Bb,S,H,Hkv,hd", [(4, 64, 4, 4, 32), (1, 31, 2, 1, 30), (2, 33, 4, 2, 34), (1, 65, 3, 3, 64),
                                           (2, 96, 4, 1, 66), (1, 100, 2, 2, 128), (1, 1, 2, 2, 2)])
def test_fp32_attention(B, Bb, S, H, Hkv, hd):
    g = torch.Generator(device="cuda").manual_seed(S + 7 * H + hd)
    W = (H + 2 * Hkv) * hd
    qkv, dout = torch.randn(Bb * S, W, device="cuda", generator=g), torch.randn(Bb * S, H * hd, device="cuda", generator=g)
    out, dqkv = torch.full_like(dout, float("nan")), torch.full_like(qkv, float("nan"))
    lse = torch.full((Bb, H, S), float("nan"), device="cuda")
    B.zl_op_attention(0, qkv, out, lse, Bb, S, H, Hkv, hd)
    B.zl_op_attention_bwd(0, qkv, out, dout, lse, dqkv, Bb, S, H, Hkv, hd)
    torch.cuda.synchronize()
    x = qkv.double().requires_grad_(True)
    t = x.view(Bb, S, H + 2 * Hkv, hd).transpose(1, 2)
    k, v = (t[:, a:a + Hkv].repeat_interleave(H // Hkv, 1) for a in (H, H + Hkv))
    s = (t[:, :H] @ k.transpose(-1, -2)) / hd ** 0.5
    s = s.masked_fill(torch.ones(S, S, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    ref = (torch.softmax(s, -1) @ v).transpose(1, 2).reshape(Bb * S, H * hd)
    (gx,) = torch.autograd.grad(ref, x, dout.double())
    # fp32 sums of up to max(S, hd) terms and expf (2 ulp): a few 1e-7 relative to the values' scale
    assert float((lse - torch.logsumexp(s, -1).detach()).abs().max()) <= 1e-5
    assert float((out - ref.detach()).abs().max()) <= 1e-5 * max(1.0, float(ref.detach().abs().max()))
    assert float((dqkv - gx).abs().max()) <= 1e-5 * max(1.0, float(gx.abs().max()))


# Rows off 16 bytes take single loads, the others 16-byte ones: the same values in the same order.
@pytest.mark.parametrize("S,H,Hkv,hd", [(65, 4, 2, 32), (40, 2, 2, 64)])
def test_fp32_attention_alignment(B, S, H, Hkv, hd):
    g = torch.Generator(device="cuda").manual_seed(S)
    W = (H + 2 * Hkv) * hd
    qkv, dout = torch.randn(S, W, device="cuda", generator=g), torch.randn(S, H * hd, device="cuda", generator=g)
    res = []
    for off in (0, 1):
        def at(t):
            b = torch.empty(t.numel() + off, device="cuda")
            b[off:].copy_(t.flatten())
            return b[off:].view(t.shape)
        q, d, lse = at(qkv), at(dout), torch.empty(1, H, S, device="cuda")
        out, dqkv = at(dout), at(qkv)
        B.zl_op_attention(0, q, out, lse, 1, S, H, Hkv, hd)
        B.zl_op_attention_bwd(0, q, out, d, lse, dqkv, 1, S, H, Hkv, hd)
        res.append((out.clone(), lse, dqkv.clone()))
    for a, b in zip(*res):
        assert torch.equal(a, b)


def _f32_attention(B, qkv, dout, S, H, Hkv, hd):
    out, dqkv, lse = torch.empty_like(dout), torch.empty_like(qkv), torch.empty(1, H, S, device="cuda")
    B.zl_op_attention(0, qkv, out, lse, 1, S, H, Hkv, hd)
    B.zl_op_attention_bwd(0, qkv, out, dout, lse, dqkv, 1, S, H, Hkv, hd)
    return out.view(S, H, hd), lse[0].T, dqkv.view(S, H + 2 * Hkv, hd)


# A row whose first keys all have NaN scores (a whole group of eight, or of the row's length) is NaN, whatever follows.
@pytest.mark.parametrize("nan_keys", [1, 8, 16, 40])
@pytest.mark.parametrize("hd", [32, 66, 128])
def test_fp32_attention_keeps_nan(B, nan_keys, hd):
    S, H, Hkv = 70, 2, 1
    g = torch.Generator(device="cuda").manual_seed(hd)
    qkv, dout = torch.randn(S, (H + 2) * hd, device="cuda", generator=g), torch.randn(S, H * hd, device="cuda", generator=g)
    qkv[:nan_keys, H * hd] = float("nan")
    out, lse, _ = _f32_attention(B, qkv, dout, S, H, Hkv, hd)
    assert bool(out.isnan().all()) and bool(lse.isnan().all())


# NaN or Inf in one token's query, key, value or output gradient reaches the rows that read it and, causally, no others: the
# rest is what it is without (first and last rows of 32-row tiles and of the sequence).
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("S,t,hd", [(70, 3, 32), (70, 31, 30), (70, 32, 64), (70, 69, 32), (64, 63, 128), (33, 32, 66)])
@pytest.mark.parametrize("where", ["q", "k", "v", "dout"])
def test_fp32_attention_causal_nonfinite(B, where, S, t, hd, bad):
    H, Hkv, h = 4, 2, 1   # query head 1 and KV head 0, which heads 0 and 1 read
    g = torch.Generator(device="cuda").manual_seed(S + t + hd)
    qkv, dout = torch.randn(S, (H + 2 * Hkv) * hd, device="cuda", generator=g), torch.randn(S, H * hd, device="cuda", generator=g)
    clean = [x.clone() for x in _f32_attention(B, qkv, dout, S, H, Hkv, hd)]
    if where == "dout":
        dout[t, h * hd + 1] = bad
    else:
        qkv[t, {"q": h, "k": H, "v": H + Hkv}[where] * hd + 1] = bad
    out, lse, dqkv = _f32_attention(B, qkv, dout, S, H, Hkv, hd)
    i = torch.arange(S, device="cuda")
    # rows of (out, lse, dQ) of the heads, and of (dK, dV) of the KV heads, that the bad row may reach
    none, later, own, upto = i < 0, i >= t, i == t, i <= t
    heads = [h] if where in ("q", "dout") else [0, 1]
    o, l, dq, dk, dv = {"q": (own, own, own, upto, upto), "k": (later, later, later, i >= 0, i >= 0), "v": (later, none, later, i >= 0, none),
                        "dout": (none, none, own, upto, upto)}[where]
    for name, got, ref, hs, rows in (("out", out, clean[0], heads, o), ("lse", lse, clean[1], heads, l), ("dq", dqkv[:, :H], clean[2][:, :H], heads, dq),
                                     ("dk", dqkv[:, H:H + Hkv], clean[2][:, H:H + Hkv], [0], dk),
                                     ("dv", dqkv[:, H + Hkv:], clean[2][:, H + Hkv:], [0], dv)):
        may = torch.zeros(got.shape[:2], dtype=torch.bool, device="cuda")
        may[:, hs] = rows[:, None]
        assert torch.equal(got[~may], ref[~may]), name
    if bad != bad:   # (an infinite key may also be a score of -inf, a weight of zero)
        assert bool(out[o][:, heads].isnan().any(-1).all()) and bool(dqkv[dq][:, heads].isnan().any(-1).all())


# Heads of 32 are rotated inside the fp32 attention kernels: training steps against the float64 oracle, with the
# loss and per-tensor tolerances of the other fp32 parity tests (1e-4).
@pytest.mark.parametrize("seq,kv", [(50, 2), (33, 1), (31, 4)])
def test_fp32_rotated_attention(seq, kv):
    import synth
    from tests.gpu_common import engine_for, fro_rel, oracle_for, rel
    w = synth.Workload("rot-f32", synth.ModelDims(synth.ARCH_LLAMA, 2, 128, 4, kv, 344, 300, 64), "f32", batch=3, seq=seq, K=2,
                       steps=2, lr=1e-4, seed=seq)
    P = synth.make_params(w.dims, w.seed)
    eng, orc = engine_for(w), oracle_for(w, P)
    eng.load(P)
    for s in range(w.steps):
        ids, labels = synth.make_batch(w, s)
        for a, b in zip(eng.step(ids.cuda(), labels.cuda()), orc.step(ids, labels)):
            assert rel(a, b) <= 1e-4
    for n in orc.trainable_names():
        assert fro_rel(eng.get(n), orc.P[n]) <= 1e-4, n
    eng.close()
