"""GPU parity of forwards of more than 128 rows (prefill chunks, large batches): the CTA-pair GEMM and the
attention over chunks of several query tiles, against the oracle's forward. Bound: 3e-2 in max-relative error, the
parity bound of the bf16 path."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_24211_b200 import binding as scd
from test_gpu_session import MID_BF16_D64, MID_BF16_D128_GQA, SMALL_BF16, _models, _rel

pytestmark = pytest.mark.gpu

WIDE_GQA4 = dict(n_layers=2, d_model=576, n_heads=8, n_kv_heads=2, head_dim=64, d_ffn=832, vocab_out=1000,
                 vocab_in=1010, dtype="bf16", rope_base=10000.0, rms_eps=1e-5)   # tiles of 256 that end inside a run of 32


@pytest.mark.parametrize("shape,page,P,B,M,min_ctx", [
    (MID_BF16_D64, 64, 130, 1, 3, 512),        # 129 prompt rows: one more than the weight-streaming kernel takes
    (MID_BF16_D64, 64, 258, 1, 129, 512),      # 257 rows: a second x tile with one row; a window of two query tiles
    (MID_BF16_D64, 128, 258, 1, 129, -1),      # the same through the mma.sync attention kernel, part after part
    (MID_BF16_D128_GQA, 64, 700, 1, 65, 512),  # two query heads per KV head: 64 positions per query tile
    (WIDE_GQA4, 64, 161, 3, 43, 512),          # 480 prompt rows, 129 window rows of three sequences
    (WIDE_GQA4, 128, 2700, 1, 5, 512),         # two passes over the prompt (2560 rows at most), the second over a context
    (SMALL_BF16, 16, 150, 2, 70, 512),         # head_dim 32: no tensor-core attention
    (MID_BF16_D64, 64, 70, 1, 65, 512),        # a second window tile with one row, eight warps, 64 dims: window last
    (dict(MID_BF16_D128_GQA, n_kv_heads=MID_BF16_D128_GQA["n_heads"]), 64, 200, 1, 128, 512),   # 128 dims: window first
    (MID_BF16_D64, 64, 300, 2, 64, 512),       # four warps, a full window tile, a ring that wraps
])
def test_many_rows_match_oracle(shape, page, P, B, M, min_ctx):
    gm, om = _models(shape, max_seq=P + M + 9, seed=17, std=0.06, page=page, n_streams=B)
    rng = np.random.default_rng(P)
    prompt = rng.integers(0, shape["vocab_in"], size=(B, P)).astype(np.int32)
    sess = scd.Session(gm, scd.decode_config(batch=B, window_L=M, allowed_hi=shape["vocab_out"]))
    sess.scd_session_attention_min_ctx(min_ctx)
    sess.scd_prefill(prompt, n_new=M + 4)
    ids = np.concatenate([prompt[:, -1:], rng.integers(0, shape["vocab_in"], size=(B, M - 1))], axis=1).astype(np.int32)
    logits, hidden = sess.scd_forward_window(torch.from_numpy(ids).cuda(), want_hidden=True)
    for b in range(B):
        om.forward(prompt[b, :-1], 0, stream=b)
        ref_logits, ref_hidden = om.forward(ids[b], P - 1, stream=b, want_hidden=True)
        assert _rel(hidden[b].cpu().numpy(), ref_hidden) <= 3e-2
        assert _rel(logits[b].cpu().numpy(), ref_logits) <= 3e-2
    again = sess.scd_forward_window(torch.from_numpy(ids).cuda())
    assert torch.equal(again, logits)          # cut tiles are added up in a fixed order


@pytest.mark.parametrize("L", [16, 32])
def test_step_of_many_rows_reads_only_the_sampled_ids(L):
    """A decoding step of 160 rows (the weight-streaming GEMM) and of 320 (CTA pairs) computes the logits of the
    allowed ids and of the end-of-row id alone; they are those of the explicit forward over the whole vocabulary. Only where a tile's sum over K is cut differs: fp32
    sums of 576 terms in another order, 1e-5 of the largest logit."""
    shape, B, P = WIDE_GQA4, 5, 40
    gm, _ = _models(shape, max_seq=P + 80, seed=5, std=0.06, page=64)
    rng = np.random.default_rng(2)
    cond = rng.integers(0, shape["vocab_in"], size=(B, P)).astype(np.int32)
    cfg = scd.decode_config(batch=B, window_L=L, top_k=50, cfg_lambda=1.0, seed=4, allowed_lo=100, allowed_hi=613,
                            row_period=9, eol_id=901)
    sess = scd.Session(gm, cfg)
    prompts = np.concatenate([cond, np.full_like(cond, 1)])
    sess.scd_prefill(prompts, n_new=60)
    drafts = sess.scd_debug_read("drafts").copy()
    ids = np.concatenate([prompts[:, -1:], np.tile(drafts[:, :L - 1], (2, 1))], axis=1).astype(np.int32)
    want = sess.scd_forward_window(torch.from_numpy(np.ascontiguousarray(ids)).cuda()).cpu().numpy()
    sess.scd_step()
    got = sess.scd_debug_read("logits")
    for lo, hi in ((100, 613), (901, 902)):
        assert _rel(got[:, :, lo:hi], want[:, :, lo:hi]) <= 1e-5


TINY_F32 = dict(n_layers=2, d_model=128, n_heads=4, n_kv_heads=2, head_dim=32, d_ffn=208, vocab_out=300, vocab_in=310,
                dtype="f32", rope_base=10000.0, rms_eps=1e-5)


@pytest.mark.parametrize("over,P,B,M", [
    (dict(), 5, 1, 1),                                                       # one row
    (dict(head_dim=96, n_heads=2, n_kv_heads=1), 40, 1, 17),                 # a second tile with one row
    (dict(d_model=130, d_ffn=206), 37, 2, 16),                               # K not a multiple of four: scalar loads
    (dict(d_model=1100, d_ffn=1030, head_dim=64, n_heads=4, n_kv_heads=4), 20, 1, 19),   # rows longer than one piece in shared memory
    (dict(head_dim=128, n_heads=3, n_kv_heads=3, d_ffn=600), 300, 1, 33),    # ten key tiles over eight warps
    (dict(d_ffn=2048, vocab_out=5000), 130, 2, 64),                          # enough columns for four per warp
])
def test_fp32_layers_match_oracle(over, P, B, M):
    """The fp32 path against the oracle. Bound 2e-5 of the largest value: fp32 sums of up to 2048 terms, two layers
    (one sum's error is about sqrt(2048) 2^-24 = 3e-6 of its magnitude)."""
    shape = dict(TINY_F32, **over)
    gm, om = _models(shape, max_seq=P + M + 9, seed=19, std=0.05, n_streams=B)
    rng = np.random.default_rng(P)
    prompt = rng.integers(0, shape["vocab_in"], size=(B, P)).astype(np.int32)
    sess = scd.Session(gm, scd.decode_config(batch=B, window_L=M, allowed_hi=shape["vocab_out"]))
    sess.scd_prefill(prompt, n_new=M + 4)
    ids = np.concatenate([prompt[:, -1:], rng.integers(0, shape["vocab_in"], size=(B, M - 1))], axis=1).astype(np.int32)
    logits, hidden = sess.scd_forward_window(torch.from_numpy(ids).cuda(), want_hidden=True)
    for b in range(B):
        if P > 1:
            om.forward(prompt[b, :-1], 0, stream=b)
        ref_logits, ref_hidden = om.forward(ids[b], P - 1, stream=b, want_hidden=True)
        assert _rel(hidden[b].cpu().numpy(), ref_hidden) <= 2e-5
        assert _rel(logits[b].cpu().numpy(), ref_logits) <= 2e-5


@pytest.mark.parametrize("B,M", [(1, 40), (2, 256)])
def test_swiglu_where_the_exponential_is_large(B, M):
    """silu(g) u with g down to -88.5, where 1 + exp(-g) passes 2^126, and u large enough for the product to matter: the
    weight-streaming kernel (40 rows) and the CTA-pair kernel (512). One layer without attention output, embeddings of +-1.
    Bound 1e-4 of the largest value: g is good to 2e-5 absolute (64 fp32 terms), the product is kept in two bf16 planes."""
    d, F = 64, 128
    shape = dict(n_layers=1, d_model=d, n_heads=1, n_kv_heads=1, head_dim=64, d_ffn=F, vocab_out=64, vocab_in=64, dtype="bf16",
                 rope_base=10000.0, rms_eps=1e-5)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    bf = dict(device="cuda", dtype=torch.bfloat16)
    gate = torch.linspace(-20.0, 20.0, F, device="cuda")
    gate[::16] = torch.tensor([-87.5, -88.0, -88.5, -87.5, -80.0, -88.0, -88.5, -60.0], device="cuda")
    up = torch.where(gate < -50.0, torch.full_like(gate, 3e37), torch.ones_like(gate))
    w = {"tok_emb": torch.ones(64, d, **bf), "final_norm": torch.ones(d, **bf), "lm_head": torch.zeros(64, d, **bf)}
    w["tok_emb"][1::2, d // 2:] = -1.0                 # odd tokens: g = u = 0
    w.update(attn_norm=[torch.ones(d, **bf)], ffn_norm=[torch.ones(d, **bf)], wo=[torch.zeros(d, 64, **bf)])
    for k in ("wq", "wk", "wv"):
        w[k] = [torch.zeros(64, d, **bf)]
    w["w_gate"] = [(gate / d).to(torch.bfloat16)[:, None].expand(F, d).contiguous()]
    w["w_up"] = [(up / d).to(torch.bfloat16)[:, None].expand(F, d).contiguous()]
    w["w_down"] = [(torch.rand(d, F, generator=g, device="cuda") * 0.2 - 0.1).to(torch.bfloat16)]
    model = scd.Model(shape, w, max_seq=M + 8)
    sess = scd.Session(model, scd.decode_config(batch=B, window_L=M, allowed_hi=64))
    sess.scd_prefill(np.zeros((B, 1), dtype=np.int32), n_new=M)
    ids = (torch.arange(B * M, device="cuda", dtype=torch.int32) % 64).reshape(B, M)
    _, hidden = sess.scd_forward_window(ids, want_hidden=True)
    h = w["tok_emb"][ids.long()].double()
    n = h / (h.square().mean(-1, keepdim=True) + 1e-5).sqrt()
    gd, ud = n @ w["w_gate"][0].double().T, n @ w["w_up"][0].double().T
    want = h + (gd / (1.0 + torch.exp(-gd)) * ud) @ w["w_down"][0].double().T
    assert (hidden.double() - want).abs().max() <= 1e-4 * want.abs().max()


@pytest.mark.parametrize("d,F,V,B,M", [
    (576, 832, 1000, 3, 86),        # 258 rows: a second x tile with two; weight tiles that end inside a run of 32 columns
    (1024, 2816, 4000, 4, 256),     # 1024 rows: every tile of the layer cut between pairs
    (256, 512, 40000, 2, 200),      # LM head of more tiles than pairs: whole ones and cut ones
    (4096, 256, 64, 2, 150),        # two tiles, each cut into many parts
    (64, 64, 8, 2, 129),            # one K block
])
def test_pair_gemm_against_64_bits(d, F, V, B, M):
    """One layer without attention output, so that the forward is the norm and the three GEMMs of the CTA-pair kernel in
    front of and behind known values. Gate, up and down multiply both bf16 planes of their input: 16 bits, 7.6e-6 of a value,
    which sums of many terms average; one plane alone would be off by 1e-3. Bound 1e-4 of the largest sum. The logits take
    the hidden state that came out, rounded to bf16 once: only fp32 sums differ, 2e-6 of the sum of magnitudes."""
    shape = dict(n_layers=1, d_model=d, n_heads=1, n_kv_heads=1, head_dim=64, d_ffn=F, vocab_out=V, vocab_in=512, dtype="bf16",
                 rope_base=10000.0, rms_eps=1e-5)
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    def mat(*dims, std=0.05):
        return (torch.randn(*dims, generator=g, device="cuda") * std).to(torch.bfloat16)
    def gain():
        return (1.0 + 0.4 * (torch.rand(d, generator=g, device="cuda") - 0.5)).to(torch.bfloat16)
    w = dict(tok_emb=mat(512, d, std=1.0), final_norm=gain(), lm_head=mat(V, d), attn_norm=[gain()], ffn_norm=[gain()],
             wq=[mat(64, d)], wk=[mat(64, d)], wv=[mat(64, d)], wo=[torch.zeros(d, 64, device="cuda", dtype=torch.bfloat16)],
             w_gate=[mat(F, d)], w_up=[mat(F, d)], w_down=[mat(d, F)])
    sess = scd.Session(scd.Model(shape, w, max_seq=M + 8), scd.decode_config(batch=B, window_L=M, allowed_hi=V))
    sess.scd_prefill(np.zeros((B, 1), dtype=np.int32), n_new=M)
    ids = torch.randint(0, 512, (B, M), generator=g, device="cuda", dtype=torch.int32)
    logits, hidden = sess.scd_forward_window(ids, want_hidden=True)
    h = w["tok_emb"][ids.long()].double()
    n = h / (h.square().mean(-1, keepdim=True) + 1e-5).sqrt() * w["ffn_norm"][0].double()
    gd, ud = n @ w["w_gate"][0].double().T, n @ w["w_up"][0].double().T
    down = (gd / (1.0 + torch.exp(-gd)) * ud) @ w["w_down"][0].double().T
    assert (hidden.double() - h - down).abs().max() <= 1e-4 * down.abs().max()
    x = (hidden * w["final_norm"].float()).to(torch.bfloat16).double()
    inv = 1.0 / (hidden.double().square().mean(-1, keepdim=True) + 1e-5).sqrt()
    head = w["lm_head"].double().T
    assert (logits.double() - (x @ head) * inv).abs().max() <= 2e-6 * ((x.abs() @ head.abs()) * inv).max()
    again, hidden2 = sess.scd_forward_window(ids, want_hidden=True)
    assert torch.equal(again, logits) and torch.equal(hidden2, hidden)
