"""What a session holds on the device: activation buffers for its window and, only once a prompt asks for them, for wide
passes over it; prefills that have no memory for wide passes take narrow ones."""
import gc

import numpy as np
import pytest
import torch

from paper_2510_24211_b200 import binding as scd
from paper_2510_24211_b200 import synth

pytestmark = pytest.mark.gpu

# the SwiGLU output of a pass alone takes 131 KB per row: 17 MB for 128 rows, 184 MB for 1408 (half of 2599, in whole 128s)
SHAPE = dict(n_layers=1, d_model=256, n_heads=4, n_kv_heads=4, head_dim=64, d_ffn=32768, vocab_out=512, vocab_in=512,
             dtype="bf16", rope_base=10000.0, rms_eps=1e-5)
MB = 1 << 20


@pytest.fixture(scope="module")
def model():
    w = synth.make_weights(SHAPE, seed=3, device="cuda")
    m = scd.Model(SHAPE, w, max_seq=3000)
    s = _session(m)                                    # (the kernels of both paths are loaded from here on)
    _logits(s, 2600)
    _logits(s, 100)
    s.close()
    yield m
    m.close()


def _session(m, batch=1, L=8):
    return scd.Session(m, scd.decode_config(batch=batch, window_L=L, top_k=20, seed=1, allowed_hi=512))


def _logits(s, P):
    prompt = np.random.default_rng(P).integers(0, 512, size=(s.B, P)).astype(np.int32)
    s.scd_prefill(prompt, n_new=16)
    return s.scd_forward_window(torch.arange(5, device="cuda", dtype=torch.int32).repeat(s.B, 1) + 7)


def _free():
    torch.cuda.synchronize()
    gc.collect()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_session_grows_with_its_prompts(model):
    before = _free()
    s = _session(model)
    held = before - _free()
    assert held <= 64 * MB
    short = _logits(s, 100)
    assert before - _free() <= held + 8 * MB
    long = _logits(s, 2600)
    assert before - _free() >= held + 184_000_000
    # neither the buffers' size nor what was in them shows in the results
    fresh = _session(model)
    assert torch.equal(_logits(fresh, 2600), long) and torch.equal(_logits(s, 100), short)
    assert torch.equal(_logits(s, 700), _logits(fresh, 700))
    s.close()
    fresh.close()
    assert before - _free() <= 8 * MB


def test_prefill_without_room_for_wide_passes(model):
    s = _session(model)
    want = _logits(s, 2600)
    s.close()
    s = _session(model)
    block = torch.empty(_free() - 160 * MB, dtype=torch.uint8, device="cuda")
    try:
        got = _logits(s, 2600)                         # passes of 128 rows
    finally:
        del block
        torch.cuda.empty_cache()
    # the parity bound of the bf16 path
    assert (got - want).abs().max() <= 3e-2 * want.abs().max()
    assert torch.equal(_logits(s, 2600), want)         # there is room now
    s.close()


def test_explicit_forward_under_capture_allocates_its_scratch(model):
    """200 rows go through the CTA-pair kernel where the weights ask for it; its scratch is not there yet."""
    s = _session(model, batch=2)
    ids = torch.arange(200, device="cuda", dtype=torch.int32).reshape(2, 100)
    prompt = np.arange(20, dtype=np.int32).reshape(2, 10)
    s.scd_prefill(prompt, n_new=120)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = s.scd_forward_window(ids)
    g.replay()
    torch.cuda.synchronize()
    got = out.clone()
    # a longer prompt puts larger buffers in place of those that the graph uses, which are still there
    _logits(s, 1400)
    s.scd_prefill(prompt, n_new=120)
    want = s.scd_forward_window(ids)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got, want) and torch.equal(out, want)
    s.close()
