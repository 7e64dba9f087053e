"""Results of few-row steps to the last bit.

Every kernel of a step sums in an order of its own, and a bf16 model rounds its
operands again after each of them, so another order of one fp32 sum moves the
results of the layers behind it by more than that sum's rounding.  The digests
in ``golden/step_bits.json`` (SHA-256, first 16 hex digits, recorded on a
GB300) pin the orders that parity with the oracle cannot tell apart; a change
of order is to be seen here and not in a user's tokens.
"""
import hashlib
import json
import os

import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "step_bits.json")

# d 512, two layers; rank 256 and four mixer heads as in the post-train model
BASE = dict(vocab=1024, d_model=512, n_heads=4, n_kv_heads=2, head_dim=128, ffn=1024, n_anchor=1, n_denoise=1,
            fusion_rank=256, fusion_heads=4, dtype="bf16")
STEPS = {  # name: (model, batch, rows)
    "paired_2688": (dict(fusion="paired_attn"), 21, 128),
    "paired_64": (dict(fusion="paired_attn"), 2, 32),
    "paired_256": (dict(fusion="paired_attn"), 8, 32),
    "qk_norm_64": (dict(qk_norm=True), 2, 32),
    "qk_norm_hd64_96": (dict(qk_norm=True, n_heads=8, n_kv_heads=4, head_dim=64), 3, 32),
}


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2609_37924_gb300 import tadm
    return tadm


def sha(t):
    return hashlib.sha256(t.contiguous().view(torch.uint8).cpu().numpy().tobytes()).hexdigest()[:16]


def digests(T, name):
    """Anchor latent, paired-attention row scales and fused latent of one refresh and one reverse step."""
    over, batch, rows = STEPS[name]
    m = wl.ModelConfig(**{**BASE, **over})
    tm = T.TadmModel(m, T.upload_weights(m, wl.make_weights(m, seed=5, affine_std=0.05)), max_batch=batch, max_rows=rows)
    w = wl.Workload("bits", m, batch=batch, prompt_len=0, gen_len=rows, steps_per_block=4, K=4)
    z0, z1 = (torch.from_numpy(wl.random_canvas(w, batch, rows, f, s)).cuda() for f, s in ((0.9, 1), (0.4, 2)))
    M, d = batch * rows, m.d_model
    cache = tm.new_cache(batch, rows)
    fused = torch.empty((M, d), dtype=torch.float32, device="cuda")
    tm.tadm_reset(batch)
    tm.tadm_anchor_forward(z0, 4, cache)
    tm.tadm_denoise_step(z1, 3, 4, 0, cache, fused=fused)
    tm.tadm_sync_status()
    out = {"h": sha(cache[:4 * M * d]), "fused": sha(fused)}
    if m.fusion == "paired_attn":            # s_C and s_H follow the latent in the cache, each padded to 256 bytes
        at, pad = (4 * M * d + 255) // 256 * 256, (4 * M + 255) // 256 * 256
        out["scales"] = sha(torch.cat([cache[at:at + 4 * M], cache[at + pad:at + pad + 4 * M]]))
    tm.close()
    return out


# s_C and s_H of 1024 and more rows (one warp adds a row's squares); the gate of
# a split GEMM (its products added in column order; 2688 rows leave the mixer's
# GEMMs unsplit); the K slices of the mixer's GEMMs of few rows; the squares of
# QK-norm behind a split QKV projection (column by column)
@pytest.mark.parametrize("name,what", [("paired_2688", "scales"), ("paired_2688", "fused"), ("paired_64", "fused"),
                                       ("paired_256", "fused"), ("qk_norm_64", "h"), ("qk_norm_hd64_96", "h")])
def test_step_bits(T, name, what):
    with open(GOLDEN) as f:
        assert digests(T, name)[what] == json.load(f)[name][what]
