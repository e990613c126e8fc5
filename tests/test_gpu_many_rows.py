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
