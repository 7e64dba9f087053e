"""The branches of the kernels' dispatch at the sizes where they can go wrong,
through the C ABI, against plain products and the oracle's definitions."""
import numpy as np
import pytest

import workloads as wl
from oracle import tadm_oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2609_37924_gb300 import tadm
    return tadm


def bf16_tensor(shape, seed, std=1.0):
    bits = wl.normal(seed, 99, int(np.prod(shape)), 0.0, std, "bf16").reshape(shape)
    return torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda(), O.widen(bits)


# fp32 outputs leave through TMA stores of 32 x 32 boxes (N % 4 == 0 and
# ldc % 4 == 0: TMA clips to 16 bytes, not to elements), otherwise row by row:
# ragged edges, padding columns that must stay untouched, an odd stride
@pytest.mark.parametrize("M,N,K,ldc", [(33, 300, 72, 304), (33, 301, 72, 304), (33, 301, 72, 301),
                                       (257, 260, 136, 260), (130, 36, 64, 40), (1, 4, 8, 4), (1, 1, 8, 4)])
def test_gemm_fp32_store_edges(T, M, N, K, ldc):
    A, a = bf16_tensor((M, K), 1)
    B, b = bf16_tensor((N, K), 2)
    flat = torch.full((M * ldc + 8,), 7.0, dtype=torch.float32, device="cuda")
    C = flat[:M * ldc].view(M, ldc)
    T.tadm_gemm(A, B, C[:, :N], dtype=1)
    got = C.cpu().numpy().astype(np.float64)
    # fp32 accumulation of K exact bf16 products
    assert np.abs(got[:, :N] - a @ b.T).max() <= 1e-5 * np.abs(a).max() * np.abs(b).max() * np.sqrt(K)
    assert (got[:, N:] == 7.0).all() and (flat[M * ldc:] == 7.0).all().item()


# bf16 outputs likewise (N % 8 == 0 and ldc % 8 == 0), on both tile kernels:
# columns past N of a wider matrix are the caller's
@pytest.mark.parametrize("M", [33, 257])
@pytest.mark.parametrize("N,K,ldc", [(301, 72, 304), (300, 136, 304), (304, 64, 312), (36, 64, 40), (260, 64, 264), (1, 8, 8),
                                     (301, 72, 301)])
def test_gemm_bf16_store_edges(T, M, N, K, ldc):
    A, a = bf16_tensor((M, K), 8)
    B, b = bf16_tensor((N, K), 9)
    flat = torch.full((M * ldc + 8,), 7.0, dtype=torch.bfloat16, device="cuda")
    C = flat[:M * ldc].view(M, ldc)
    T.tadm_gemm(A, B, C[:, :N], dtype=1)
    got, ref = C.cpu().to(torch.float64).numpy(), a @ b.T
    # fp32 accumulation of K exact bf16 products, then one rounding to 8 bits
    assert (np.abs(got[:, :N] - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5 * np.abs(a).max() * np.abs(b).max() * np.sqrt(K)).all()
    assert (got[:, N:] == 7.0).all() and (flat[M * ldc:] == 7.0).all().item()


def _nucleus_ok(logits, mask, top_p, u, tok, tol=2e-5):
    """tok is the inverse-CDF draw of the nucleus, up to fp32 rounding of the cumulative mass at its edges."""
    q = np.exp(logits.astype(np.float64) - np.delete(logits, mask).max())
    q[mask] = 0.0
    desc = np.sort(q)[::-1]
    c = np.cumsum(desc)
    for p in (top_p, top_p * (1 + tol), top_p * (1 - tol)):
        tau = desc[min(np.searchsorted(c, p * c[-1] * (1 - 1e-12)), len(desc) - 1)]
        n = np.where(q >= tau, q, 0.0)
        cum = np.cumsum(n)
        if n[tok] > 0 and cum[tok] - n[tok] - tol * cum[-1] <= u * cum[-1] <= cum[tok] + tol * cum[-1]:
            return True
    return False


# the shared-memory sampler: rows that are no multiple of 4 (scalar loads), one
# segment per warp and a tail, more equal tokens than the collected bracket
# holds, near one-hot rows, top_p = 1; more drawing rows than blocks
@pytest.mark.parametrize("V,R,top_p", [(30, 400, 0.9), (1001, 300, 0.9), (4100, 64, 1.0), (30522, 40, 0.9),
                                       (51200, 24, 0.5)])
def test_remdm_nucleus_draws(T, V, R, top_p):
    B, first, mask, seed, step = 2, 3, V - 1, 77, 4
    rng = np.random.default_rng(V)
    logits = (rng.standard_normal((B * R, V)) * rng.choice([0.3, 3.0], (B * R, 1))).astype(np.float32)
    logits[first] = 0.5                                   # all equal
    logits[first + 1] += np.where(np.arange(V) == V // 2, 60.0, 0.0).astype(np.float32)
    logits[first + 2, : V // 2] = -np.inf
    z = np.full((B, R), mask, np.int32)
    zt = torch.from_numpy(z).cuda()
    act = torch.empty(B * R, dtype=torch.int32, device="cuda")
    T.tadm_remdm_update(zt, torch.from_numpy(logits).cuda(), first, mask, 0.0, 1.0, top_p, seed, step, act)
    got, u = zt.cpu().numpy(), wl.remdm_uniforms(seed, step, B, R)
    assert (got[:, :first] == mask).all()
    for b in range(B):
        for r in range(first, R):
            assert _nucleus_ok(logits[b * R + r], mask, top_p, u[b, r, 2], got[b, r]), (b, r, got[b, r])


# more positions than one scan of the actions takes (32768), with drawing rows in
# every part of it and several per block: each draws once, the others keep their token
def test_remdm_many_positions(T):
    B, R, V, mask, top_p, seed, step = 9, 7400, 30, 29, 0.9, 79, 3
    rng = np.random.default_rng(9)
    logits = rng.standard_normal((B * R, V)).astype(np.float32)
    z = rng.integers(0, mask, (B, R)).astype(np.int32)
    z[rng.random((B, R)) < 1 / 24] = mask
    zt = torch.from_numpy(z).cuda()
    act = torch.empty(B * R, dtype=torch.int32, device="cuda")
    T.tadm_remdm_update(zt, torch.from_numpy(logits).cuda(), 0, mask, 0.0, 1.0, top_p, seed, step, act)
    got, u = zt.cpu().numpy(), wl.remdm_uniforms(seed, step, B, R)
    assert (got[z != mask] == z[z != mask]).all()
    rows = np.argwhere(z == mask)
    assert (rows[:, 0] * R + rows[:, 1] > 2 * 32768).any() and len(rows) > 2 * 304
    for b, r in rows:
        assert _nucleus_ok(logits[b * R + r], mask, top_p, u[b, r, 2], got[b, r]), (b, r, got[b, r])


# a NaN logit holds no mass and is never drawn; a row without any mass (every
# weight e^(l - max) is 0 or NaN) draws nothing and ends (token -1)
@pytest.mark.parametrize("V", [1001, 30522])
def test_remdm_rows_with_nan_and_inf(T, V):
    B, R, mask, top_p, seed, step = 1, 48, V - 1, 0.5, 78, 2
    rng = np.random.default_rng(V)
    logits = (0.5 * rng.standard_normal((R, V))).astype(np.float32)
    logits[:, 5::97] = np.nan
    logits[3] = -np.inf
    logits[4, 7] = np.inf
    zt = torch.full((B, R), mask, dtype=torch.int32, device="cuda")
    act = torch.empty(R, dtype=torch.int32, device="cuda")
    T.tadm_remdm_update(zt, torch.from_numpy(logits).cuda(), 0, mask, 0.0, 1.0, top_p, seed, step, act)
    got, u = zt.cpu().numpy()[0], wl.remdm_uniforms(seed, step, B, R)[0, :, 2]
    assert got[3] == got[4] == -1
    for r in set(range(R)) - {3, 4}:
        assert _nucleus_ok(np.where(np.isnan(logits[r]), -np.inf, logits[r]), mask, top_p, u[r], got[r]), (r, got[r])


def f32_tensor(shape, seed):
    x = wl.normal(seed, 98, int(np.prod(shape)), 0.0, 1.0, "f32").reshape(shape)
    return torch.from_numpy(x).cuda(), x.astype(np.float64)


# fp32 GEMM: 16- and 32-row tiles, 16-byte and 4-byte copies, K shorter than a
# stage, K ending inside a stage's 64 columns, one row and one column
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (17, 65, 4), (15, 64, 68), (33, 130, 257), (31, 2000, 132), (700, 900, 260),
                                   (300, 1100, 30)])
def test_gemm_f32_tiles(T, M, N, K):
    A, a = f32_tensor((M, K), 3)
    B, b = f32_tensor((N, K), 4)
    C = torch.empty((M, N), dtype=torch.float32, device="cuda")
    T.tadm_gemm(A, B, C, dtype=0)
    # sums of K fp32 products of N(0, 1) values: error below K 2^-24 |a| |b|
    assert np.abs(C.cpu().numpy() - a @ b.T).max() <= 2.0 ** -24 * (K + 4) * np.abs(a).max() * np.abs(b).max()


# fp32 attention: rows around the 16-row block, keys around the 64-key tile,
# an odd key stride (scalar loads), causal, windows that leave whole tiles out
@pytest.mark.parametrize("hd,Hq,Hkv,rows,ctx,causal,window,pad", [
    (32, 2, 1, 1, 0, False, 0, 0), (64, 2, 2, 17, 47, False, 0, 0), (64, 4, 2, 16, 48, True, 0, 3),
    (128, 2, 1, 33, 95, True, 20, 1), (64, 2, 2, 40, 200, False, 70, 0), (32, 4, 4, 130, 0, True, 1, 2)])
def test_attention_f32_tiles(T, hd, Hq, Hkv, rows, ctx, causal, window, pad):
    B, n = 2, ctx + rows
    stride = n + pad
    q, qa = f32_tensor((B, Hq, rows, hd), 5)
    k, ka = f32_tensor((B, Hkv, stride, hd), 6)
    v, va = f32_tensor((B, Hkv, hd, stride), 7)
    o = torch.empty((B * rows, Hq * hd), dtype=torch.float32, device="cuda")
    T.tadm_attention(q, k, v, o, Hq, Hkv, rows, ctx, causal, 0, window=window)
    pos, key = ctx + np.arange(rows)[:, None], np.arange(n)[None, :]
    see = np.ones((rows, n), bool)
    if causal:
        see &= key <= pos
    if window:
        see &= pos - key < window
    got = o.cpu().numpy().reshape(B, rows, Hq, hd)
    for b in range(B):
        for h in range(Hq):
            g = h // (Hq // Hkv)
            s = np.where(see, qa[b, h] @ ka[b, g, :n].T / np.sqrt(hd), -np.inf)
            p = np.exp(s - s.max(1, keepdims=True))
            ref = (p / p.sum(1, keepdims=True)) @ va[b, g, :, :n].T
            assert np.abs(got[b, :, h] - ref).max() < 2e-5     # fp32 scores of magnitude ~5, sums of n terms


# split-K reductions of every epilogue (QKV per head row, GLU, fusion gate /
# hidden / output, paired-attention gate, add, up) at row counts around their
# 8-row blocks, both head widths, QK-norm, and the paired-attention kernels
@pytest.mark.parametrize("hd,fusion,qk_norm,batch,rows", [(128, "gated_mlp", False, 3, 11), (64, "gated_mlp", True, 1, 1),
                                                          (128, "paired_attn", True, 2, 24), (64, "paired_attn", False, 5, 32),
                                                          (128, "paired_attn", False, 1, 17)])
def test_few_row_steps_match_the_oracle(T, hd, fusion, qk_norm, batch, rows):
    m = wl.ModelConfig(vocab=1024, d_model=1024, n_heads=1024 // hd, n_kv_heads=512 // hd, head_dim=hd, ffn=2048, n_anchor=1,
                       n_denoise=1, fusion=fusion, fusion_rank=256, fusion_heads=4, dtype="bf16", qk_norm=qk_norm,
                       qkv_split=hd == 128)
    host = wl.make_weights(m, seed=3, affine_std=0.05)
    tm = T.TadmModel(m, T.upload_weights(m, host), max_batch=batch, max_rows=rows)
    w = wl.Workload("t", m, batch=batch, prompt_len=0, gen_len=rows, steps_per_block=4, K=4)
    z0, z1 = (wl.random_canvas(w, batch, rows, f, s) for f, s in ((0.9, 1), (0.4, 2)))
    cache = tm.new_cache(batch, rows)
    logits = torch.empty((batch * rows, m.vocab), dtype=torch.float32, device="cuda")
    tm.tadm_reset(batch)
    tm.tadm_anchor_forward(torch.from_numpy(z0).cuda(), 4, cache)
    tm.tadm_denoise_step(torch.from_numpy(z1).cuda(), 3, 4, 0, cache, logits=logits)
    tm.tadm_sync_status()
    o = O.Oracle(m, host)
    sess = o.new_session(batch)
    ref = o.denoise_logits(sess, z1, o.anchor_forward(sess, z0)).reshape(batch * rows, m.vocab)
    rel = np.linalg.norm(logits.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert rel < 1.5e-2, rel          # bf16 operands, two layers and the fusion
    tm.close()


# pipelined hd-64 attention (launches of more 128-row tiles than SMs; P in
# tensor memory): odd row counts, tiles with idle softmax warps, a context,
# causal limits inside and between key tiles, a KV group of two heads, few keys
@pytest.mark.parametrize("B,Hq,Hkv,rows,ctx,causal", [(4, 12, 12, 450, 0, False), (7, 12, 12, 129, 40, False),
                                                      (4, 16, 16, 333, 70, True), (16, 20, 10, 40, 24, False),
                                                      (3, 16, 8, 500, 131, True), (40, 4, 4, 100, 0, True)])
def test_attention_pipelined_hd64(T, B, Hq, Hkv, rows, ctx, causal):
    hd, n = 64, ctx + rows
    stride = (n + 7) // 8 * 8
    assert ((Hq // Hkv) * rows + 127) // 128 * Hkv * B > torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator(device="cuda").manual_seed(rows)
    q = (2.0 * torch.randn((B, Hq, rows, hd), generator=g, device="cuda")).to(torch.bfloat16)
    k = torch.randn((B, Hkv, stride, hd), generator=g, device="cuda").to(torch.bfloat16)
    v = torch.randn((B, Hkv, hd, stride), generator=g, device="cuda").to(torch.bfloat16)
    o = torch.full((B * rows, Hq * hd), float("nan"), dtype=torch.bfloat16, device="cuda")
    T.tadm_attention(q, k, v, o, Hq, Hkv, rows, ctx, causal, 1)
    rep = Hq // Hkv
    kd, vd = k[:, :, :n].double().repeat_interleave(rep, 1), v[..., :n].double().transpose(2, 3).repeat_interleave(rep, 1)
    s = q.double() @ kd.transpose(2, 3) / 8.0
    if causal:
        pos = ctx + torch.arange(rows, device="cuda")[:, None]
        s = s.masked_fill(torch.arange(n, device="cuda")[None, :] > pos, -float("inf"))
    ref = (torch.softmax(s, -1) @ vd).transpose(1, 2).reshape(B * rows, Hq * hd)
    err = (o.double() - ref).abs()
    assert torch.isfinite(o.float()).all()
    # bf16 P (relative 2^-9 each, at most 2^-8 of the largest |V|) and the bf16 result
    assert (err <= 2.0 ** -8 * ref.abs() + 2.0 ** -8 * v.float().abs().max()).all()


# GLU projections on 192-wide pair tiles (96 gate and 96 up columns; FFN widths
# whose last round of 256-wide tiles is nearly empty): a width that 96 divides
# and one it does not, both activations, ragged rows
@pytest.mark.parametrize("ffn,glu,rows", [(10752, "swiglu", 130), (10112, "geglu", 255)])
def test_glu_192_wide_tiles(T, ffn, glu, rows):
    m = wl.ModelConfig(vocab=512, d_model=256, n_heads=4, n_kv_heads=4, head_dim=64, ffn=ffn, glu=glu, n_anchor=1,
                       n_denoise=1, fusion="none", dtype="bf16")
    host = wl.make_weights(m, seed=5, affine_std=0.05)
    tm = T.TadmModel(m, T.upload_weights(m, host), max_batch=1, max_rows=rows)
    w = wl.Workload("t", m, batch=1, prompt_len=0, gen_len=rows, steps_per_block=4, K=4)
    z = wl.random_canvas(w, 1, rows, 0.5, 1)
    cache = tm.new_cache(1, rows)
    logits = torch.empty((rows, m.vocab), dtype=torch.float32, device="cuda")
    tm.tadm_reset(1)
    tm.tadm_anchor_forward(torch.from_numpy(z).cuda(), 4, cache)
    tm.tadm_denoise_step(torch.from_numpy(z).cuda(), 3, 4, 0, cache, logits=logits)
    tm.tadm_sync_status()
    o = O.Oracle(m, host)
    sess = o.new_session(1)
    ref = np.asarray(o.denoise_logits(sess, z, o.anchor_forward(sess, z))).reshape(rows, m.vocab)
    rel = np.linalg.norm(logits.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert rel < 1.5e-2, rel           # bf16 operands, two layers
    tm.close()


# fp32 GEMM, head and attention: a row's results do not depend on how many rows
# the launch has: 16- and 32-row GEMM tiles, block- and warp-per-row reduction of the head's tiles, one
# or several attention blocks (equal to the last bit: a sampler compares
# confidences that may be that close)
@pytest.mark.parametrize("rows", [1, 60, 100, 1024])
def test_f32_rows_alone(T, rows):
    g = torch.Generator(device="cuda").manual_seed(3)
    d, vocab, M = 64, 4165, 1100
    x = torch.randn((M, d), generator=g, device="cuda")
    w = torch.randn((vocab, d), generator=g, device="cuda") * 0.3
    scratch = torch.empty(T.tadm_head_scratch_size(M, vocab, 0), dtype=torch.uint8, device="cuda")
    conf, tok = torch.empty(M, device="cuda"), torch.empty(M, dtype=torch.int32, device="cuda")
    T.tadm_head_confidence(x, w, vocab - 1, conf, tok, scratch, 0)
    conf2, tok2 = torch.empty(rows, device="cuda"), torch.empty(rows, dtype=torch.int32, device="cuda")
    T.tadm_head_confidence(x[:rows], w, vocab - 1, conf2, tok2, scratch, 0)
    assert torch.equal(conf[:rows], conf2) and torch.equal(tok[:rows], tok2)
    p = torch.softmax((x.double() @ w.double().T)[:, :-1], -1)
    assert (conf / p.max(-1).values.float() - 1).abs().max() < 1e-4    # logits of 64 terms, exponentiated


@pytest.mark.parametrize("hd", [32, 64, 128])
def test_attention_f32_row_alone(T, hd):
    g = torch.Generator(device="cuda").manual_seed(4)
    n, rows = 137, 33
    k = torch.randn((1, 2, n + 3, hd), generator=g, device="cuda")
    v = torch.randn((1, 2, hd, n + 3), generator=g, device="cuda")
    q = torch.randn((1, 4, rows, hd), generator=g, device="cuda")
    o = torch.empty((rows, 4 * hd), device="cuda")
    T.tadm_attention(q, k, v, o, 4, 2, rows, n - rows, False, 0)
    for r in (0, 15, 32):
        one = torch.empty((1, 4 * hd), device="cuda")
        T.tadm_attention(q[:, :, r:r + 1].contiguous(), k, v, one, 4, 2, 1, n - 1, False, 0)
        assert torch.equal(o[r:r + 1], one)


# a key outside a row's causal or window range leaves the row alone, whatever its V holds
@pytest.mark.parametrize("causal,window", [(True, 0), (False, 40)])
def test_attention_f32_masked_v(T, causal, window):
    g = torch.Generator(device="cuda").manual_seed(5)
    rows, hd = 100, 64
    q, k = (torch.randn((1, 1, rows, hd), generator=g, device="cuda") for _ in range(2))
    v = torch.randn((1, 1, hd, rows), generator=g, device="cuda")
    bad = 99 if causal else 0
    v[..., bad] = float("inf")
    o = torch.empty((rows, hd), device="cuda")
    T.tadm_attention(q, k, v, o, 1, 1, rows, 0, causal, 0, window=window)
    free = torch.arange(rows, device="cuda") < 99 if causal else torch.arange(rows, device="cuda") >= window
    assert torch.isfinite(o[free]).all() and not torch.isfinite(o[~free]).any()
