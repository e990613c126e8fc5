"""The work that programs using this library have it do, as cases that can be timed and compared.

Four kinds, all through the public binding:
  verify    scd_verify on logits the caller holds: the sampler alone (a host with its own decoder);
  window    scd_forward_window on a session that holds a context: one teacher-forced window pass;
  prefill   scd_prefill of a prompt, then the logits of its last token: the time to the first token;
  generate  scd_prefill, scd_generate to the end, then the logits behind the last token: a whole request.

Models are the shapes of `synth.WORKLOADS` with random weights. The weights of the session kinds carry a
successor rule: every token has one of CYCLE classes, visible as a direction in its embedding, and the LM
head gives the next class's token PEAK units of logit over the rest, as a trained model does where it is
sure. So the sampled tokens and the number of iterations do not hang on the last bits of a logit, and the
other ids keep the spread of a random model for top-k, top-p and guidance to work on. A draft that is one
class off stays so as the window moves: a forward commits one token, as on the random-weight models of
the benchmark, except behind a forced end-of-row token, where it commits a whole window. Output projections
are scaled by 1 / sqrt(2 n_layers), the usual initialisation of deep decoders.
"""
import math

import numpy as np
import torch

from paper_2510_24211_b200 import binding as scd
from paper_2510_24211_b200 import synth

CYCLE = 8
PEAK = 22.0

MODES = {"ar": scd.SCD_MODE_AR, "sjd": scd.SCD_MODE_SJD, "mc": scd.SCD_MODE_SCD_MC,
         "gs": scd.SCD_MODE_SCD_GS, "alpha": scd.SCD_MODE_ALPHA}


def _verify(name, batch, L, V, top_k, top_p, lam, mode):
    return dict(name=name, kind="verify", batch=batch, L=L, V=V, top_k=top_k, top_p=top_p, cfg_lambda=lam, mode=mode)


def _session(name, kind, model, mode="mc", batch=1, prompt=1, n_new=0, **over):
    w = synth.WORKLOADS[model]
    c = dict(name=name, kind=kind, model=model, mode=mode, batch=batch, prompt=prompt, n_new=n_new,
             n_layers=w["n_layers"], n_kv_heads=w["n_kv_heads"], L=w["window_L"], top_k=w["top_k"],
             top_p=w.get("top_p", 0.0), cfg_lambda=w["cfg_lambda"], row_period=w["row_period"], page=128)
    c.update(over)
    return c


def listed():
    return [
        # the sampler on one image window (the verify-only workload): the smallest call, all latency
        _verify("verify_image", 1, 32, 16384, 2000, 0.0, 0.0, "mc"),
        # the same for a full serving batch with guidance: two logit rows are read per window row
        _verify("verify_batch8_cfg", 8, 32, 16384, 2000, 0.0, 2.0, "mc"),
        # a video window with nucleus sampling over the whole vocabulary
        _verify("verify_video_nucleus", 1, 64, 64000, 0, 0.8, 0.0, "mc"),
        # the Gumbel-sharing coupling: a race over the vocabulary for every row
        _verify("verify_gumbel", 2, 32, 16384, 2000, 0.0, 0.0, "gs"),
        # a small fp32 decoder from a class token to a whole 16 x 16 grid: launches and host work
        _session("generate_tiny", "generate", "tiny", n_new=256),
        # class-conditional image tokens: a small bf16 decoder, guidance pair, latency-bound kernels
        _session("generate_class_image", "generate", "llamagen_xl", n_new=96),
        # text-to-image on a 7B-shaped decoder, two rows of the grid: weight streaming
        _session("generate_text_image", "generate", "lumina_7b", prompt=120, n_new=98),
        # the same model one token at a time (the vanilla path, and the tail of any serving mix)
        _session("generate_autoregressive", "generate", "lumina_7b", mode="ar", prompt=57, n_new=24),
        # one window late in a text-to-image generation
        _session("window_text_image_late", "window", "lumina_7b", prompt=2301),
        # four guided sequences at once: 256 window rows, the most that one pass over the weights carries
        _session("window_image_batch4", "window", "janus_like", batch=4, prompt=333),
        # one window late in a video generation: the KV cache is as large as the weights of several layers
        _session("window_video_late", "window", "video_4b", prompt=9001),
        # the first-frame prefix of a video: the compute-bound end
        _session("prefill_video", "prefill", "video_4b", prompt=2560),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("verify", "window", "window", "prefill", "generate", "generate"))
    if kind == "verify":
        batch = _log_int(rng, 1, 8)
        V = _log_int(rng, 1000, 65536)
        top_p = rng.choice((0.0, 0.0, 0.8, 0.95))
        c = _verify("", batch, _log_int(rng, 4, 128 if batch * V <= 131072 else 32), V,
                    0 if top_p else min(V, _log_int(rng, 50, 4000)), top_p, rng.choice((0.0, 2.0, 3.0)),
                    rng.choice(("mc", "mc", "mc", "sjd", "alpha", "gs", "ar")))
        del c["name"]
        return c
    model = rng.choice(("tiny", "llamagen_xl", "llamagen_xl", "lumina_7b", "janus_like", "video_4b", "video_4b_top_p"))
    w = synth.WORKLOADS[model]
    bf16 = w["dtype"] == "bf16"
    lam = rng.choice((0.0, w["cfg_lambda"] or 2.0))
    S = 2 if lam else 1
    mode = rng.choice(("mc", "mc", "mc", "sjd", "gs", "alpha", "ar"))
    batch = rng.choice((1, 1, 1, 2, 3, 4))
    L = 1 if mode == "ar" else _log_int(rng, 4, 128 if bf16 else 32)
    while S * batch * L > 256:
        L //= 2
    rep = rng.choice((1, 1, 2, 4))
    if rep * L > 128 or w["n_heads"] % rep:
        rep = 1
    video = model.startswith("video")
    most = 9001 if video else 2301 if bf16 else 512
    n_new = 0
    if kind == "window":
        prompt = _log_int(rng, 2, most // batch)
    elif kind == "prefill":
        prompt = _log_int(rng, 16, min(most, 2560) // (S * batch))
    else:
        prompt = rng.choice((1, _log_int(rng, 2, 256)))
        n_new = _log_int(rng, 8, 96 * 64 // max(64, S * batch * L) if bf16 else 256)
        if mode == "ar":
            n_new = min(n_new, 32)
    c = _session("", kind, model, mode=mode, batch=batch, prompt=prompt, n_new=n_new,
                 n_layers=_log_int(rng, 2, w["n_layers"]), n_kv_heads=w["n_heads"] // rep, L=L,
                 top_k=0 if w.get("top_p") else _log_int(rng, 16, w["top_k"]), cfg_lambda=lam,
                 row_period=rng.choice((0, w["row_period"], rng.randint(9, 49))), page=rng.choice((64, 128)))
    del c["name"]
    return c


def _shape(c):
    s = dict(synth.WORKLOADS[c["model"]])
    s.update(n_layers=c["n_layers"], n_kv_heads=c["n_kv_heads"])
    return s


def _streams(c):
    return 2 if c["cfg_lambda"] else 1


def _rows(c):
    return 1 if c["mode"] == "ar" else c["L"]


def _weights(shape, seed):
    w = synth.make_weights(shape, seed=seed, device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 1)
    d, lo, hi = shape["d_model"], shape["allowed_lo"], shape["allowed_hi"]
    for k in ("wo", "w_down"):
        for t in w[k]:
            t.mul_((2 * shape["n_layers"]) ** -0.5)
    emb = w["tok_emb"].float() * 50.0
    cls = torch.randint(0, CYCLE, (shape["vocab_in"],), generator=g, device="cuda")
    ids = lo + torch.randperm(hi - lo, generator=g, device="cuda")[:CYCLE]
    cls[ids] = torch.arange(CYCLE, device="cuda")
    dirs = torch.randn(CYCLE, d, generator=g, device="cuda")
    emb += dirs[cls]
    w["tok_emb"] = emb.to(w["tok_emb"].dtype)
    head = w["lm_head"][ids].float() + dirs.roll(1, 0) * (PEAK * 3.0 ** 0.5 / d)
    w["lm_head"][ids] = head.to(w["lm_head"].dtype)
    return w


def prepare(case, seed):
    c = case
    if c["kind"] == "verify":
        B, L, V, S = c["batch"], _rows(c), c["V"], _streams(c)
        p, q = synth.verify_logits(seed, 0, B, L, V, device="cuda", streams=S)
        if S == 2:                     # the unconditional logits resemble the conditional ones
            p[1] = 0.5 * p[0] + 0.5 * p[1]
        cfg = scd.decode_config(mode=MODES[c["mode"]], batch=B, window_L=L, top_k=c["top_k"], top_p=c["top_p"],
                                cfg_lambda=c["cfg_lambda"], seed=seed, allowed_hi=V, alpha=0.5)
        kept = q
        if c["top_p"]:                 # drafts come from the truncated draft distribution: its likely ids
            kept = torch.where(q >= q.amax(-1, keepdim=True) - 1.0, q, torch.full_like(q, float("-inf")))
        drafts = synth.draft_ids_from_logits(kept, c["top_k"], seed)
        ws = torch.empty(scd.scd_verify_workspace_bytes(cfg, V), dtype=torch.uint8, device="cuda")
        positions = torch.arange(B, device="cuda", dtype=torch.int64) * 17 + 5
        return dict(kind="verify", cfg=cfg, p=p, q=q, drafts=drafts, positions=positions, ws=ws)
    shape = _shape(c)
    B, S, L, P, V = c["batch"], _streams(c), _rows(c), c["prompt"], shape["vocab_out"]
    model = scd.Model(shape, _weights(shape, seed), max_seq=P + c["n_new"] + L + 8, kv_page_tokens=c["page"])
    cfg = scd.decode_config(mode=MODES[c["mode"]], batch=B, window_L=L, temperature=shape["temperature"],
                            top_k=c["top_k"], top_p=c["top_p"], cfg_lambda=c["cfg_lambda"], seed=seed,
                            allowed_lo=shape["allowed_lo"], allowed_hi=shape["allowed_hi"],
                            row_period=c["row_period"], eol_id=shape["eol_id"], alpha=0.5)
    sess = scd.Session(model, cfg)
    cond, uncond = synth.make_prompt(dict(shape, prompt_len=P), batch=B, seed=seed)
    prompts = np.concatenate([cond, uncond]) if S == 2 else cond
    state = dict(kind=c["kind"], sess=sess, prompts=prompts, n_new=c["n_new"])
    if c["kind"] == "window":
        sess.scd_prefill(prompts, n_new=L)
        rng = np.random.default_rng(seed + 7)
        more = rng.integers(shape["allowed_lo"], shape["allowed_hi"], size=(B, L - 1)).astype(np.int32)
        ids = np.concatenate([prompts[:, -1:], np.tile(more, (S, 1))], axis=1)
        state["ids"] = torch.from_numpy(np.ascontiguousarray(ids)).cuda()
    return state


def run(state):
    if state["kind"] == "verify":
        return scd.scd_verify(state["cfg"], state["p"], state["q"], state["drafts"], state["positions"], 3,
                              workspace=state["ws"])
    sess = state["sess"]
    if state["kind"] == "window":
        return sess.scd_forward_window(state["ids"])
    sess.scd_prefill(state["prompts"], n_new=state["n_new"])
    if state["kind"] == "prefill":
        last = torch.from_numpy(state["prompts"][:, -1:].copy()).cuda()
        return sess.scd_forward_window(last)
    tokens, _ = sess.scd_generate()
    last = torch.from_numpy(np.tile(tokens[:, -1:], (sess.S, 1))).cuda()
    return tokens, sess.scd_forward_window(last)


def _forward_work(c, shape, rows, ctx, positions):
    """One decoder pass over `rows` rows per stream-sequence on `ctx` committed positions that leaves logits
    of `positions` rows: every weight, cache entry and logit once; every contraction of it."""
    es = 4 if shape["dtype"] == "f32" else 2
    d, dq, dkv = shape["d_model"], shape["n_heads"] * shape["head_dim"], shape["n_kv_heads"] * shape["head_dim"]
    seqs = _streams(c) * c["batch"]
    layer = d * (dq + 2 * dkv) + dq * d + 3 * d * shape["d_ffn"]
    params = shape["n_layers"] * layer
    kv = 2 * shape["n_layers"] * dkv * es * seqs * (ctx + 2 * rows)
    att = 4 * shape["n_layers"] * dq * seqs * rows * (ctx + (rows + 1) / 2)
    head = shape["vocab_out"] * d if positions else 0
    return (es * (params + head) + kv + 4 * seqs * positions * shape["vocab_out"],
            2.0 * seqs * (rows * params + positions * head) + att)


def _iterations(c):
    """Forwards that the successor rule needs for n_new tokens: one each, but a row's end carries a window."""
    p, n, L = c["row_period"], c["n_new"], _rows(c)
    if L == 1 or p == 0 or n <= p:
        return n
    return p - 1 + math.ceil((n - p + 1) * max(1, p - L + 1) / p)


def _sampler_bytes(c, ids, rows):
    """Target rows and the draft row read, the post-processed row kept for the next iteration written."""
    return 4 * c["batch"] * rows * ids * (_streams(c) + 2)


def work(case):
    c = case
    if c["kind"] == "verify":
        return {"bytes": 4 * c["batch"] * _rows(c) * c["V"] * (_streams(c) + 1), "flops": 0}
    shape = _shape(c)
    if c["kind"] == "window":
        b, f = _forward_work(c, shape, _rows(c), c["prompt"] - 1, _rows(c))
        return {"bytes": b, "flops": f}
    b, f = _forward_work(c, shape, 1, c["prompt"] + c["n_new"] - 1, 1)       # the logits behind the last token
    if c["prompt"] > 1:
        pb, pf = _forward_work(c, shape, c["prompt"] - 1, 0, 0)
        b, f = b + pb, f + pf
    if c["n_new"]:
        L, n = _rows(c), _iterations(c)
        ids = shape["allowed_hi"] - shape["allowed_lo"]
        gb, gf = _forward_work(c, dict(shape, vocab_out=ids), L, c["prompt"] + c["n_new"] / 2, L)
        b, f = b + n * (gb + _sampler_bytes(c, ids, L)), f + n * gf
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Integers are exact. Logits: about four times the largest difference seen between two orders of the same
    fp32 sums (bf16: other K slices of the GEMMs or the other attention kernel, 1.9e-3 and 9e-3 over 60 cases;
    fp32: a torch evaluation in 32 against 64 bits, 2.5e-7 and 2.5e-5 at 257 tokens)."""
    if case["kind"] == "verify":
        return "exact"
    return {"rel": 7.5e-3, "max": 4e-2} if synth.WORKLOADS[case["model"]]["dtype"] == "bf16" else {"rel": 2e-6, "max": 2e-4}
