"""GPU parity of the fused verify-and-redraft kernel against the CPU oracle, through the C ABI.

Bit-exact comparison of accept counts, accept flags, committed ids and next drafts on the same
fp32 logits and the same Philox key."""
import os

import numpy as np
import pytest
import torch

import oracle
from helpers import oracle_verify
from paper_2510_24211_b200 import binding as scd
from paper_2510_24211_b200 import synth

pytestmark = pytest.mark.gpu
MODES = {"ar": scd.SCD_MODE_AR, "sjd": scd.SCD_MODE_SJD, "scd": scd.SCD_MODE_SCD_MC,
         "alpha": scd.SCD_MODE_ALPHA, "gs": scd.SCD_MODE_SCD_GS}


def _run_case(mode, B, L, V, iteration, seed, temperature=1.0, top_k=0, lam=0.0, lo=0, hi=None,
              row_period=0, eol_id=0, q_present=True, quantise=None, pos_base=1000, alpha=1.0, top_p=0.0):
    hi = V if hi is None else hi
    S = 2 if lam != 0.0 else 1
    p, q = synth.verify_logits(seed, iteration, B, L, V, device="cuda", streams=S)
    if quantise:
        p = torch.round(p / quantise) * quantise      # many exact ties
        q = torch.round(q / quantise) * quantise
    if mode == "ar":
        p = p[:, :, :1].contiguous()
        q = q[:, :1].contiguous()
    Lk = p.shape[2]
    qm = q.clone()
    qm[..., :lo] = float("-inf")
    qm[..., hi:] = float("-inf")
    drafts = synth.draft_ids_from_logits(qm / temperature, top_k, seed * 100 + iteration)
    positions = torch.tensor([pos_base + 37 * b + iteration for b in range(B)], dtype=torch.int64,
                             device="cuda")
    cfg = scd.decode_config(mode=MODES[mode], batch=B, window_L=L, temperature=temperature,
                            top_k=top_k, cfg_lambda=lam, seed=seed, allowed_lo=lo, allowed_hi=hi,
                            row_period=row_period, eol_id=eol_id, alpha=alpha, top_p=top_p)
    got = scd.scd_verify(cfg, p, q if q_present else None, drafts, positions, iteration)
    torch.cuda.synchronize()
    n_commit, committed, next_drafts, flags = [t.cpu().numpy() for t in got]
    want = oracle_verify(mode, p.cpu().numpy(), q.cpu().numpy() if q_present else None,
                         drafts.cpu().numpy(), positions.cpu().numpy(), iteration, seed, temperature,
                         top_k, lam, lo, hi, row_period, eol_id, alpha, top_p)
    assert np.array_equal(n_commit, want["n_commit"]), (n_commit, want["n_commit"])
    assert np.array_equal(flags[:, :Lk], want["flags"])
    for b in range(B):
        a = int(n_commit[b])
        assert np.array_equal(committed[b, :a], want["committed"][b, :a])
    if mode != "ar":
        assert np.array_equal(next_drafts, want["next_drafts"])
    return n_commit


def test_noise_matches_oracle_bitwise():
    pos = torch.arange(0, 1_000_000, dtype=torch.int64, device="cuda") * 7 + 3
    got = scd.scd_noise_u24(0xDEADBEEF12345678, oracle.NOISE_RESIDUAL, 5, pos, 77, 2).cpu().numpy()
    idx = np.concatenate([np.arange(0, 2000), np.random.default_rng(0).integers(0, 1_000_000, 3000)])
    for i in idx:
        assert int(got[i]) == oracle.noise_u24(0xDEADBEEF12345678, oracle.NOISE_RESIDUAL, 5,
                                               int(pos[i]), 77, 2)
    hist = np.bincount(got.astype(np.int64) >> 18, minlength=64)
    chi2 = ((hist - 1e6 / 64) ** 2 / (1e6 / 64)).sum()
    assert chi2 < 63 + 5 * np.sqrt(126)


@pytest.mark.parametrize("B", [1, 2, 8])
def test_verify_workload_shape(B):
    # the verify-only workload: L = 32, V = 16384, temperature 1, top-k 2000
    iters = int(os.environ.get("SCD_VERIFY_ITERS", "12" if B < 8 else "4"))
    accepted = []
    for seed in (0, 1, 2):
        for it in range(iters):
            accepted.append(_run_case("scd", B, 32, 16384, it, seed, top_k=2000))
    mean_a = float(np.concatenate(accepted).mean())
    assert 1.0 <= mean_a <= 32.0


@pytest.mark.parametrize("mode", ["scd", "sjd", "ar"])
def test_verify_modes_small_ragged(mode):
    # ragged vocabulary (not a multiple of the CTA width), short window
    for it in range(6):
        _run_case(mode, 3, 5, 1000, it, seed=4, top_k=50)
        _run_case(mode, 2, 7, 33, it, seed=5, top_k=0)


@pytest.mark.parametrize("alpha", [0.0, 0.3, 0.75, 1.0])
def test_verify_alpha_coupling(alpha):
    # Algorithm 5: rows beyond the committed prefix keep the coupled redraft with probability alpha
    for it in range(8):
        _run_case("alpha", 3, 12, 1000, it, seed=21, top_k=50, alpha=alpha)
        _run_case("alpha", 2, 9, 257, it, seed=22, top_k=0, lam=1.5, alpha=alpha)


def test_verify_gumbel_sharing_coupling():
    # Algorithm 7: verify as Algorithm 1, redraft and fresh rows by the shared-noise Gumbel race
    for it in range(6):
        _run_case("gs", 3, 12, 1000, it, seed=31, top_k=50)
        _run_case("gs", 2, 9, 257, it, seed=32, top_k=0, lam=1.5, temperature=0.8)
        _run_case("gs", 2, 12, 777, it, seed=33, top_k=40, lo=10, hi=700, row_period=5, eol_id=720,
                  pos_base=0)
    _run_case("gs", 2, 8, 300, 0, seed=34, top_k=20, q_present=False)
    _run_case("gs", 1, 32, 16384, 1, seed=35, top_k=2000)
    _run_case("gs", 2, 6, 1500, 2, seed=36, top_k=100, quantise=0.5)     # equal weights: ties in the race


@pytest.mark.parametrize("top_p", [0.8, 0.3, 0.999, 1e-4])
def test_verify_nucleus_truncation(top_p):
    # top-p after top-k (and alone), on p and on the raw draft rows; ties from quantised logits
    for it in range(4):
        _run_case("scd", 2, 8, 4099, it, seed=41, top_k=300, top_p=top_p)
        _run_case("scd", 2, 8, 1000, it, seed=42, top_k=0, lam=1.5, temperature=0.8, top_p=top_p)
        _run_case("scd", 1, 6, 1500, it, seed=43, top_k=0, quantise=0.5, top_p=top_p)
    _run_case("gs", 2, 8, 777, 0, seed=44, top_k=0, top_p=top_p)
    _run_case("sjd", 2, 8, 777, 1, seed=45, top_k=50, top_p=top_p)
    _run_case("ar", 3, 1, 2048, 2, seed=46, top_k=0, top_p=top_p)
    _run_case("scd", 1, 64, 64000, 0, seed=47, top_k=0, top_p=top_p)      # the video setting's shape


def test_verify_cfg_temperature_and_allowed_range():
    for it in range(5):
        _run_case("scd", 2, 8, 4099, it, seed=7, temperature=0.7, top_k=300, lam=3.0, lo=101, hi=3000)
        _run_case("scd", 1, 16, 2048, it, seed=8, temperature=1.3, top_k=100, lam=1.5)


def test_verify_fresh_rows_and_forced_tokens():
    for it in range(4):
        _run_case("scd", 2, 12, 777, it, seed=9, top_k=40, q_present=False)
        _run_case("scd", 2, 12, 777, it, seed=10, top_k=40, lo=10, hi=700, row_period=5, eol_id=720,
                  pos_base=0)


def test_verify_ties_and_topk_edges():
    for it in range(4):
        _run_case("scd", 2, 6, 1500, it, seed=11, top_k=100, quantise=0.5)
        _run_case("scd", 1, 6, 600, it, seed=12, top_k=1)          # greedy: one-hot rows
        _run_case("scd", 1, 6, 600, it, seed=13, top_k=600)        # k = n: no threshold
        _run_case("scd", 1, 6, 600, it, seed=14, top_k=5000)       # k > n


@pytest.mark.parametrize("B,L,V,top_k,top_p,lam", [
    (2, 8, 300, 20, 0.0, 0.0), (3, 5, 2634, 20, 0.0, 2.0), (1, 12, 1643, 1, 0.0, 0.0), (2, 8, 800, 150, 0.5, 0.0),
    (2, 80, 9000, 900, 0.0, 0.0),                                        # more candidates than are selected by counting
    (1, 3, 131073, 500, 0.0, 0.0),
])
def test_verify_threshold_at_signed_zeros(B, L, V, top_k, top_p, lam):
    """+0 and -0 are one logit: both are at the threshold, or neither is. Half of the ids at -1, the rest at zero, with the
    minus sign on most of them in the target rows and on few in the draft rows."""
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    S = 2 if lam else 1
    r = torch.rand(B, L, V, generator=g, device="cuda")
    at_zero = torch.rand(B, L, V, generator=g, device="cuda") < 0.5
    def row(minus):
        return torch.where(at_zero, torch.where(r < minus, -0.0, 0.0), -1.0)
    q = row(0.2)
    for it, p0 in enumerate((row(0.8), row(0.0), row(1.0))):
        p = p0[None].repeat(S, 1, 1, 1).contiguous()
        drafts = torch.argmax((q + r * at_zero > -1.0).to(torch.int32), dim=-1).to(torch.int32)
        positions = torch.arange(B, device="cuda", dtype=torch.int64) * 300 + 9
        cfg = scd.decode_config(mode=scd.SCD_MODE_SCD_MC, batch=B, window_L=L, top_k=top_k, top_p=top_p, cfg_lambda=lam, seed=8,
                                allowed_hi=V)
        n_commit, committed, next_drafts, flags = [t.cpu().numpy() for t in scd.scd_verify(cfg, p, q, drafts, positions, it)]
        want = oracle_verify("scd", p.cpu().numpy(), q.cpu().numpy(), drafts.cpu().numpy(), positions.cpu().numpy(), it, 8,
                             top_k=top_k, top_p=top_p, cfg_lambda=lam)
        assert (want["flags"] == 1).all()              # the same distribution twice
        assert np.array_equal(n_commit, want["n_commit"]) and np.array_equal(flags, want["flags"])
        assert np.array_equal(next_drafts, want["next_drafts"]) and np.array_equal(committed, want["committed"])


def test_verify_large_vocab_and_max_window():
    _run_case("scd", 1, 64, 64000, 0, seed=15, top_k=1000)
    _run_case("scd", 1, 256, 512, 1, seed=16, top_k=20)


def test_verify_rejects_bad_arguments():
    cfg = scd.decode_config(batch=1, window_L=4, allowed_hi=10)
    p = torch.zeros(1, 1, 4, 10, device="cuda")
    d = torch.zeros(1, 4, dtype=torch.int32, device="cuda")
    pos = torch.zeros(1, dtype=torch.int64, device="cuda")
    for bad in (dict(window_L=0), dict(window_L=257), dict(batch=0), dict(temperature=0.0),
                dict(allowed_hi=11), dict(allowed_lo=10), dict(mode=9), dict(row_period=3, eol_id=10),
                dict(mode=scd.SCD_MODE_ALPHA, alpha=1.5), dict(mode=scd.SCD_MODE_ALPHA, alpha=-0.1)):
        kw = dict(batch=1, window_L=4, allowed_hi=10)
        kw.update(bad)
        with pytest.raises(scd.ScdError) as e:
            scd.scd_verify(scd.decode_config(**kw), p, None, d, pos, 0,
                           workspace=torch.zeros(1 << 16, dtype=torch.uint8, device="cuda"))
        assert e.value.code == scd.SCD_ERR_ARG
    # the context is still usable
    scd.scd_verify(cfg, p, None, d, pos, 0)
    torch.cuda.synchronize()


def test_verify_draft_without_mass_is_rejected():
    """Drafts that have no mass under p (outside its top-k; some outside q's as well, which X ~ q rules
    out but a caller can hand in): never accepted, the row's output comes from the residual."""
    B, L, V, top_k, seed = 2, 6, 2000, 20, 51
    p, q = synth.verify_logits(seed, 0, B, L, V, device="cuda")
    drafts = torch.argmin(p[0] + q, dim=-1).to(torch.int32)          # far below both thresholds
    drafts[0, 1] = torch.argmax(q[0, 1]).to(torch.int32)              # one ordinary row in between
    positions = torch.tensor([300, 900], dtype=torch.int64, device="cuda")
    cfg = scd.decode_config(mode=scd.SCD_MODE_SCD_MC, batch=B, window_L=L, top_k=top_k, seed=seed, allowed_hi=V)
    got = [t.cpu().numpy() for t in scd.scd_verify(cfg, p, q, drafts, positions, 3)]
    want = oracle_verify("scd", p.cpu().numpy(), q.cpu().numpy(), drafts.cpu().numpy(), positions.cpu().numpy(),
                         3, seed, 1.0, top_k)
    assert np.array_equal(got[0], want["n_commit"]) and np.array_equal(got[3], want["flags"])
    assert np.array_equal(got[2], want["next_drafts"])
    assert (got[3][:, 0] == 0).all() and (got[0] == 1).all()         # row 0 of both sequences rejects
    for b in range(B):
        assert got[1][b, 0] == want["committed"][b, 0] and got[1][b, 0] != drafts[b, 0].item()


@pytest.mark.parametrize("mode,B,L,V,kw", [
    ("scd", 2, 80, 9000, dict(top_k=900)),                               # one CTA per row, read again from L2; short lists
    ("scd", 2, 80, 9000, dict(top_k=3000, quantise=8.0)),                # lists and candidates overflow (ties)
    ("sjd", 2, 80, 9000, dict()),                                        # no truncation: warps work on their whole ranges
    ("alpha", 2, 80, 9000, dict(top_p=0.9, quantise=2.0, alpha=0.4)),    # nucleus among ties
    ("scd", 2, 80, 9000, dict(top_p=0.9999999)),                         # the nucleus ends among the lightest weights
    ("scd", 1, 5, 9000, dict(top_p=0.7, top_k=1500, lam=2.0, temperature=1.3)),   # both truncations, guidance, clusters of 8
    ("gs", 2, 80, 5000, dict(top_k=300, lo=7, hi=4901)),
    ("gs", 1, 3, 16385, dict()),                                         # a race over every id
    ("ar", 3, 1, 65536, dict(top_k=2000)),
    ("scd", 1, 3, 131073, dict(top_k=500)),                              # rows too long for a cluster
    ("gs", 1, 3, 131073, dict(top_p=0.6)),
])
def test_verify_rows_at_the_edges_of_the_dispatch(mode, B, L, V, kw):
    _run_case(mode, B, L, V, iteration=2, seed=21, **kw)


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1000])
@pytest.mark.parametrize("L,V,top_k", [(3, 3000, 0), (3, 3000, 2500), (80, 3000, 0), (80, 9000, 0), (3, 20000, 4000)])
def test_verify_nucleus_that_ends_among_close_weights(L, V, top_k, n):
    """The nucleus ends in a run of n ids whose weights lie within 1 % of each other (one step of the search), distinct or in
    pairs: up to 256 are selected by counting, more are divided again."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    def row():
        x = torch.rand(2, L, V, generator=g, device="cuda") * 4.0 - 12.0
        at = torch.rand(2, L, V, generator=g, device="cuda").argsort(dim=-1)
        x.scatter_(-1, at[..., :n + 20], torch.cat([torch.linspace(-3.0, -2.99, n, device="cuda"), torch.linspace(-1.0, 0.0, 20, device="cuda")]).expand(2, L, -1).contiguous())
        return x
    p, q = row()[None].contiguous(), row()
    p[0, 1, :, 1::2] = p[0, 1, :, 0::2]                # sequence 1: weights in pairs
    drafts = torch.argmax(q, dim=-1).to(torch.int32)
    positions = torch.arange(2, device="cuda", dtype=torch.int64) * 300 + 9
    for mode, top_p in (("scd", 0.5 if n < 200 else 0.75), ("sjd", 0.9)):
        cfg = scd.decode_config(mode=MODES[mode], batch=2, window_L=L, top_k=top_k, top_p=top_p, seed=8, allowed_hi=V)
        got = [t.cpu().numpy() for t in scd.scd_verify(cfg, p, q, drafts, positions, 4)]
        want = oracle_verify(mode, p.cpu().numpy(), q.cpu().numpy(), drafts.cpu().numpy(), positions.cpu().numpy(), 4, 8, top_k=top_k, top_p=top_p)
        assert np.array_equal(got[0], want["n_commit"]) and np.array_equal(got[3], want["flags"])
        assert np.array_equal(got[2], want["next_drafts"]) and np.array_equal(got[1], want["committed"])


@pytest.mark.parametrize("B,L,V", [(1, 5, 2303), (1, 3, 20000), (2, 80, 9000), (4, 20, 40)])
@pytest.mark.parametrize("top_k,top_p", [(0, 0.8), (30, 0.8), (30, 0.0), (0, 0.0)])
def test_verify_rows_without_mass(B, L, V, top_k, top_p):
    """Rows whose logits are all -inf, in the target, in the draft, or in both, between ordinary ones: nothing is drawn from
    them and nothing depends on what the nucleus leaves undefined there."""
    p, q = synth.verify_logits(9, 1, B, L, V, device="cuda")
    p[0, :, 1::3] = float("-inf")
    q[:, 1::2] = float("-inf")
    drafts = torch.argmax(torch.where(torch.isinf(q), p[0], q), dim=-1).to(torch.int32)
    positions = torch.arange(B, device="cuda", dtype=torch.int64) * 300 + 9
    cfg = scd.decode_config(mode=scd.SCD_MODE_SCD_MC, batch=B, window_L=L, top_k=top_k, top_p=top_p, seed=8, allowed_hi=V)
    got = [t.cpu().numpy() for t in scd.scd_verify(cfg, p, q, drafts, positions, 4)]
    want = oracle_verify("scd", p.cpu().numpy(), q.cpu().numpy(), drafts.cpu().numpy(), positions.cpu().numpy(), 4, 8, top_k=top_k, top_p=top_p)
    assert np.array_equal(got[0], want["n_commit"]) and np.array_equal(got[3], want["flags"])
    assert np.array_equal(got[2], want["next_drafts"]) and np.array_equal(got[1], want["committed"])


@pytest.mark.parametrize("V,L,B,top_k,top_p", [(9000, 80, 2, 700, 0.0), (9000, 80, 2, 0, 0.8), (9001, 80, 2, 300, 0.0), (4000, 6, 1, 300, 0.0)])
def test_verify_bound_from_an_unlucky_sample(V, L, B, top_k, top_p):
    """The bound that the lists start from is estimated from ids at fixed places of each warp's range: here exactly those
    hold the largest logits, so that the bound is above the threshold and the lists are built again."""
    p, q = synth.verify_logits(3, 1, B, L, V, device="cuda")
    C = 1 if B * L > 74 else 8
    n = 2 * -(-V // (C * 16 * 256))                    # pieces of 128 ids per warp
    v = torch.arange(V, device="cuda")
    sampled = ((v // 128 % n == n // 4) & (v % 4 == 1)) | ((v // 128 % n == n - 1 - n // 4) & (v % 4 == 2))
    p[..., sampled] += 6.0
    q[..., sampled] += 6.0
    p[..., 0], q[..., 0] = float("-inf"), float("-inf")
    drafts = synth.draft_ids_from_logits(q, top_k, 5)
    positions = torch.arange(B, device="cuda", dtype=torch.int64) + 9
    cfg = scd.decode_config(mode=scd.SCD_MODE_SCD_MC, batch=B, window_L=L, top_k=top_k, top_p=top_p, seed=8, allowed_hi=V)
    n_commit, committed, next_drafts, flags = [t.cpu().numpy() for t in scd.scd_verify(cfg, p, q, drafts, positions, 4)]
    want = oracle_verify("scd", p.cpu().numpy(), q.cpu().numpy(), drafts.cpu().numpy(), positions.cpu().numpy(), 4, 8,
                         top_k=top_k, top_p=top_p)
    assert np.array_equal(n_commit, want["n_commit"]) and np.array_equal(flags, want["flags"])
    assert np.array_equal(next_drafts, want["next_drafts"])
    for b in range(B):
        assert np.array_equal(committed[b, :n_commit[b]], want["committed"][b, :n_commit[b]])


@pytest.mark.parametrize("B,L,V,top_k", [(1, 32, 16384, 2000), (3, 8, 1001, 50)])
def test_verify_reads_what_the_kernel_in_front_wrote(B, L, V, top_k):
    """The call's kernels start before the caller's last kernel is done: inputs copied into the same buffers right in front
    of every call give what each set gives by itself."""
    cfg = scd.decode_config(mode=scd.SCD_MODE_SCD_MC, batch=B, window_L=L, top_k=top_k, seed=8, allowed_hi=V)
    sets, want = [], []
    for i in range(3):
        p, q = synth.verify_logits(3 + i, 1, B, L, V, device="cuda")
        sets.append((p, q, synth.draft_ids_from_logits(q, top_k, 5 + i), torch.arange(B, device="cuda", dtype=torch.int64) * 7 + 9 * i))
        torch.cuda.synchronize()
        want.append([t.clone() for t in scd.scd_verify(cfg, *sets[-1], 4)])
        torch.cuda.synchronize()
    into = [torch.empty_like(t) for t in sets[0]]
    got = []
    for n in range(30):
        for a, b in zip(into, sets[n % 3]):
            a.copy_(b)
        got.append(scd.scd_verify(cfg, *into, 4))
    for n in range(30):
        assert all(torch.equal(a, b) for a, b in zip(got[n], want[n % 3]))


@pytest.mark.parametrize("V,top_k,top_p", [(300, 4, 0.0), (1000, 20, 0.0), (4000, 30, 0.0), (9000, 0, 0.3)])
def test_verify_gumbel_after_many_rejections(V, top_k, top_p):
    """A rejected row draws from its residual and then enters the Gumbel race, both through the same per-warp sums. Here
    every row rejects (drafts without mass), the lists are short, and the rows that enter the window sit at forced
    end-of-row positions, so that the race follows the draw at once; the same call again and again gives the oracle's answer."""
    B, L, seed, eol = 4, 15, 61, 299                   # L odd, row_period 2: ordinary rows at even positions enter odd ones
    p, q = synth.verify_logits(seed, 0, B, L, V, device="cuda")
    drafts = torch.argmin(p[0][..., :290] + q[..., :290], dim=-1).to(torch.int32)
    positions = torch.arange(B, device="cuda", dtype=torch.int64) * 10 + 100
    cfg = scd.decode_config(mode=scd.SCD_MODE_SCD_GS, batch=B, window_L=L, top_k=top_k, top_p=top_p, seed=seed, allowed_hi=V,
                            row_period=2, eol_id=eol)
    for it in range(4):
        want = oracle_verify("gs", p.cpu().numpy(), q.cpu().numpy(), drafts.cpu().numpy(), positions.cpu().numpy(), it, seed,
                             top_k=top_k, top_p=top_p, row_period=2, eol_id=eol)
        assert (want["flags"][:, ::2] == 0).all()      # (the forced positions have the one id, which is not the draft)
        for n_commit, committed, next_drafts, flags in [scd.scd_verify(cfg, p, q, drafts, positions, it) for _ in range(50)]:
            assert np.array_equal(n_commit.cpu().numpy(), want["n_commit"]) and np.array_equal(flags.cpu().numpy(), want["flags"])
            assert np.array_equal(next_drafts.cpu().numpy(), want["next_drafts"])
            assert np.array_equal(committed.cpu().numpy()[:, 0], want["committed"][:, 0])


def _dispatch(rows, n):
    """CTAs per row and ids per warp, as the launcher chooses them."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ids = lambda C: -(-max(n, 4) // (C * 16))
    C = 1
    while C < 8 and ids(C) > 128 and (rows * C * 2 <= sms or (rows * C * 2 <= 2 * sms and ids(C) > 256)):
        C *= 2
    while C < 8 and ids(C) > 1024:
        C *= 2
    return C, -(-ids(C) // 32) * 32


@pytest.mark.parametrize("B,L,V,C_want", [(1, 64, 64000, 4), (1, 8, 65536, 8), (2, 40, 20000, 2), (2, 80, 9000, 1)])
@pytest.mark.parametrize("unlucky", ["all", "one"])
@pytest.mark.parametrize("top_p", [0.0, 0.9])
def test_verify_lists_built_again_in_clusters(B, L, V, C_want, unlucky, top_p):
    """The bound of the lists comes from ids at fixed places of each warp's range. Here exactly those (of every CTA of a row, or
    of its first one) hold the largest logits, too few of them for the truncation: the bound is above the threshold, and all
    CTAs of the cluster build their lists again."""
    C, ids = _dispatch(B * L, V)
    assert C == C_want and ids > 256                   # read again from L2, not kept in registers
    g = torch.Generator(device="cuda")
    g.manual_seed(V)
    v = torch.arange(V, device="cuda")
    n, at = ids // 128, v % ids
    sampled = (at // 128 == n // 4) & (v % 4 == 1) | (at // 128 == n - 1 - n // 4) & (v % 4 == 2)
    sampled &= at < 128 * n
    if unlucky == "one":
        sampled &= v < 16 * ids
    n_sampled = int(sampled.sum())
    p = torch.rand(1, B, L, V, generator=g, device="cuda")
    q = (p[0] + 0.2 * torch.rand(B, L, V, generator=g, device="cuda")).contiguous()
    p[..., sampled] += 3.0
    q[..., sampled] += 3.0
    top_k = 0 if top_p else 2 * n_sampled
    # the bound of an unlucky CTA against the threshold of the row
    mine = p[0, 0, 0, : 16 * ids][sampled[: 16 * ids]].sort(descending=True).values
    if top_p:
        w = torch.exp(p[0, 0, 0].double())
        order = w.sort(descending=True).values
        theta = order[int((order.cumsum(0) < top_p * w.sum()).sum())]
        assert torch.exp(mine[int(0.28 * len(mine))].double()) > theta and torch.exp(mine[-1].double()) > 2.0 * theta
    else:
        e = top_k / V * len(mine)
        assert mine[min(len(mine) - 1, int(e + 4 * e ** 0.5) + 4)] > p[0, 0, 0].sort(descending=True).values[top_k - 1]
    drafts = torch.argmax(q, dim=-1).to(torch.int32)
    positions = torch.arange(B, device="cuda", dtype=torch.int64) * 300 + 9
    cfg = scd.decode_config(mode=scd.SCD_MODE_SCD_MC, batch=B, window_L=L, top_k=top_k, top_p=top_p, seed=8, allowed_hi=V)
    got = [t.cpu().numpy() for t in scd.scd_verify(cfg, p, q, drafts, positions, 4)]
    want = oracle_verify("scd", p.cpu().numpy(), q.cpu().numpy(), drafts.cpu().numpy(), positions.cpu().numpy(), 4, 8, top_k=top_k, top_p=top_p)
    assert np.array_equal(got[0], want["n_commit"]) and np.array_equal(got[3], want["flags"])
    assert np.array_equal(got[2], want["next_drafts"]) and np.array_equal(got[1], want["committed"])


@pytest.mark.parametrize("B,L,V", [(1, 64, 64000), (1, 8, 65536), (1, 64, 45001), (2, 80, 9000)])
@pytest.mark.parametrize("draft", ["none", "flat", "peaked"])
@pytest.mark.parametrize("top_p", [0.8, 0.99])
def test_verify_nucleus_of_flat_rows(B, L, V, draft, top_p):
    """Rows so flat that no list holds the nucleus (1000, 512, 704 and 576 ids per warp, lists of 384): the target row's weights
    take the place of the lists, unless the list of a peaked draft row is in the way of more than 768. Row 1 is peaked."""
    C, ids = _dispatch(B * L, V)
    assert ids > 384 + 100
    g = torch.Generator(device="cuda")
    g.manual_seed(V + L)
    p = 0.3 * torch.randn(1, B, L, V, generator=g, device="cuda")
    p[:, :, 1] *= 20.0
    q = (p[0] + 0.1 * torch.randn(B, L, V, generator=g, device="cuda")) * (20.0 if draft == "peaked" else 1.0)
    drafts = torch.argmax(q, dim=-1).to(torch.int32)
    positions = torch.arange(B, device="cuda", dtype=torch.int64) * 300 + 9
    for mode in ("scd", "sjd"):
        cfg = scd.decode_config(mode=MODES[mode], batch=B, window_L=L, top_p=top_p, seed=8, allowed_lo=3, allowed_hi=V - 2)
        qx = None if draft == "none" else q
        got = [t.cpu().numpy() for t in scd.scd_verify(cfg, p, qx, drafts, positions, 4)]
        want = oracle_verify(mode, p.cpu().numpy(), None if qx is None else q.cpu().numpy(), drafts.cpu().numpy(),
                             positions.cpu().numpy(), 4, 8, top_p=top_p, lo=3, hi=V - 2)
        assert np.array_equal(got[0], want["n_commit"]) and np.array_equal(got[3], want["flags"])
        assert np.array_equal(got[2], want["next_drafts"])
        for b in range(B):
            assert np.array_equal(got[1][b, :got[0][b]], want["committed"][b, :got[0][b]])
