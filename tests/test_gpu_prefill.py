"""Causal attention over the whole prompt (Eq. 1 for every position) on the GPU against the CPU checker, and the
compression path fed by the row log-sum-exp that this attention returns.

Bars.  lse: |gpu - ref| <= 2e-4 (fp32 sums of fp32 exponentials; the score bar of 1e-3 relative leaves room for
it).  O: the probabilities enter the second product rounded to bf16 (relative 2^-9 each, as in every tensor-core
attention kernel) and O is rounded to bf16 once at the store (2^-9 of |O|), so element-wise
|gpu - ref| <= 1e-2 |ref| + 2^-8 max|V| of the unit; the measured error is a small fraction of that.
"""
import numpy as np
import pytest
import torch

import paper_2407_08454_b200 as kvm
from paper_2407_08454_b200 import synth_inputs as si

pytestmark = pytest.mark.gpu

LSE_ATOL = 2e-4


def _run(cfg, d):
    p = kvm.make_params(cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.seq, cfg.head_dim, cfg.torch_dtype,
                        budget=cfg.budget)
    Q, K, V = d["Q"].cuda(), d["K"].cuda(), d["V"].cuda()
    O = torch.full_like(Q, 7.0)
    lse = torch.full(Q.shape[:3], -3.0, dtype=torch.float32, device="cuda")
    stats = kvm.new_stats("cuda")
    kvm.kvm_prefill_attend(p, Q, K, V, O, lse, stats)
    torch.cuda.synchronize()
    assert kvm.read_stats(stats).status == 0
    return p, Q, K, V, O, lse


def _check(O, lse, refO, ref_lse, V, G):
    g_lse = lse.cpu().numpy().astype(np.float64)
    assert np.abs(g_lse - ref_lse).max() <= LSE_ATOL
    gO = O.float().cpu().numpy().astype(np.float64)
    vmax = np.abs(V.float().numpy()).max(axis=(2, 3))                      # per (batch entry, KV head)
    tol = 1e-2 * np.abs(refO) + 2.0 ** -8 * np.repeat(vmax, G, axis=1)[:, :, None, None]
    excess = np.abs(gO - refO) / tol
    assert excess.max() <= 1.0, excess.max()
    return float(excess.max())


@pytest.mark.parametrize("S,D,Hq,Hkv,B", [(640, 128, 4, 2, 1), (300, 64, 2, 2, 2), (1024, 128, 8, 2, 1), (129, 128, 1, 1, 1),
                                          (77, 64, 4, 1, 1),
                                          (1100, 64, 40, 8, 1)])      # 360 work items: several per CTA, ragged last tile
def test_prefill_attention_matches_the_checker_elementwise(S, D, Hq, Hkv, B):
    from oracle import kvmo
    cfg = si.CONFIGS["C1"].scaled(seq=S, head_dim=D, n_q_heads=Hq, n_kv_heads=Hkv, batch=B, seed=31)
    d = si.make_layer(cfg)
    _, _, _, _, O, lse = _run(cfg, d)
    refO, ref_lse = kvmo.prefill_attend(d["Q"], d["K"], d["V"])
    _check(O, lse, refO, ref_lse, d["V"], Hq // Hkv)


@pytest.mark.parametrize("S,D,Hq,Hkv,B,logit_std", [
    (300, 128, 150, 150, 1, 4.0),     # neighbouring tiles of a head, an odd number of them, the last one ragged
    (513, 64, 57, 19, 2, 4.0),        # ... of groups of three; one row in the last tile
    (257, 64, 160, 20, 1, 4.0),       # two heads of a group
    (128, 128, 240, 120, 1, 4.0),     # one key tile per item
    (1700, 128, 32, 8, 1, 4.0),       # items of 28 steps, several per CTA
    (640, 128, 80, 80, 1, -1.0),      # nearly one-hot rows: the reference moves often
])
def test_two_query_tiles_at_a_time_match_the_checker_elementwise(S, D, Hq, Hkv, B, logit_std):
    from oracle import kvmo
    T = (S + 127) // 128
    assert B * Hq * (T + 1) >= 3 * 148                        # (the sizes from which on tiles go in pairs)
    cfg = si.CONFIGS["C1"].scaled(seq=S, head_dim=D, n_q_heads=Hq, n_kv_heads=Hkv, batch=B, seed=33, logit_std=logit_std)
    d = si.make_layer(cfg)
    _, _, _, _, O, lse = _run(cfg, d)
    refO, ref_lse = kvmo.prefill_attend(d["Q"], d["K"], d["V"])
    if logit_std > 0:
        _check(O, lse, refO, ref_lse, d["V"], Hq // Hkv)
    else:                                                     # (logits of magnitude 100s: lse relative to them, as below)
        assert np.abs(lse.cpu().numpy() - ref_lse).max() <= 1e-5 * np.abs(ref_lse).max() + LSE_ATOL
        tol = 1e-2 * np.abs(refO) + 2.0 ** -8 * np.abs(d["V"].float().numpy()).max()
        assert (np.abs(O.float().cpu().numpy() - refO) <= tol).all()


@pytest.mark.parametrize("S,D,Hq,Hkv,pairs", [
    (100, 64, 256, 256, False),       # one tile a head: no pair
    (128, 128, 456, 152, True),       # ... whose output is written the pairs' way (half of a block idle in every item)
    (100, 64, 256, 128, True),        # two heads of a group
    (250, 128, 148, 148, True),       # two tiles, a pair for every CTA
    (250, 64, 166, 166, False),       # ... and a second one for few
    (129, 128, 192, 64, False),
    (255, 64, 231, 231, True),
    (500, 64, 99, 33, False),         # four tiles: the longest pair and a short one
    (500, 128, 99, 33, True),
    (385, 64, 114, 114, True),
    (300, 64, 111, 111, True),        # three: the first one alone, twice per CTA
    (640, 64, 74, 74, True),          # five
])
def test_tiles_go_in_pairs_where_that_is_faster(S, D, Hq, Hkv, pairs):
    from parity import launched
    cfg = si.CONFIGS["C1"].scaled(seq=S, head_dim=D, n_q_heads=Hq, n_kv_heads=Hkv, seed=34)
    d = si.make_layer(cfg)
    p, Q, K, V, O, lse = _run(cfg, d)
    names = launched(lambda: kvm.kvm_prefill_attend(p, Q, K, V, O, lse))
    assert len(names) == 1 and ("prefill_pair_kernel" in names[0]) == pairs
    G = Hq // Hkv
    causal = torch.ones(S, S, dtype=torch.bool, device="cuda").tril()
    L = (Q[0].double() @ K[0].repeat_interleave(G, 0).double().transpose(-1, -2) / np.sqrt(D)).masked_fill(~causal, float("-inf"))
    refO = torch.softmax(L, -1) @ V[0].repeat_interleave(G, 0).double()
    _check(O, lse, refO[None].cpu().numpy(), torch.logsumexp(L, -1)[None].cpu().numpy(), d["V"], G)


@pytest.mark.parametrize("S,D,Hq,Hkv", [(2000, 64, 64, 32), (2000, 128, 64, 32), (1900, 64, 39, 39), (1900, 128, 39, 39)])
def test_two_tiles_at_a_time_repeat_themselves_bit_for_bit(S, D, Hq, Hkv):
    """The logits of a tile's next step land on the columns that its weights are read from: products that overtook one another
    would show as results that differ from run to run (hundreds of blocks' items, 15 steps each, under other work's noise)."""
    g = torch.Generator(device="cuda").manual_seed(S + D)
    Q, K, V = (torch.randn(1, h, S, D, generator=g, device="cuda").bfloat16() for h in (Hq, Hkv, Hkv))
    p = kvm.make_params(1, Hq, Hkv, S, D, torch.bfloat16)
    O, lse, O2, lse2 = torch.empty_like(Q), torch.empty(1, Hq, S, device="cuda"), torch.empty_like(Q), torch.empty(1, Hq, S, device="cuda")
    kvm.kvm_prefill_attend(p, Q, K, V, O, lse)
    for _ in range(50):
        kvm.kvm_prefill_attend(p, Q, K, V, O2, lse2)
        assert torch.equal(O, O2) and torch.equal(lse, lse2)


@pytest.mark.parametrize("D", [64, 128])
def test_large_values_stay_finite_when_a_maximum_grows(D):
    """A late key's logit is 10.5 (log2 units) above the others' and every value is 1e36: weights above 2^8 of a reference that
    was not moved would sum to more than fp32 holds."""
    H, Hkv, S = 160, 80, 256                                  # (two tiles at a time: 160 x 3 >= 3 x 148)
    Q, K = torch.zeros(1, H, S, D, device="cuda"), torch.zeros(1, Hkv, S, D, device="cuda")
    Q[..., 0] = 1.0
    K[:, :, 130, 0] = 10.5 * np.log(2.0) * np.sqrt(D)
    V = torch.full((1, Hkv, S, D), 1e36, device="cuda").bfloat16()
    O, lse = torch.empty(1, H, S, D, dtype=torch.bfloat16, device="cuda"), torch.empty(1, H, S, device="cuda")
    kvm.kvm_prefill_attend(kvm.make_params(1, H, Hkv, S, D, torch.bfloat16), Q.bfloat16(), K.bfloat16(), V, O, lse)
    # (a weighted mean of equal values: one rounding to bf16, one neighbour)
    assert ((O.double() - V[0, 0, 0, 0].double()).abs() <= 2.0 ** -7 * 1e36).all()


@pytest.mark.parametrize("H,Hkv,S,D", [(256, 128, 300, 64), (240, 30, 461, 64), (232, 116, 586, 64), (154, 154, 732, 128)])
def test_two_tiles_at_a_time_are_no_less_precise_than_one(H, Hkv, S, D):
    """The same heads all together and few at a time (which one tile at a time is the kernel for): the error of O against
    64 bits, over all rows, is no larger."""
    cfg = si.CONFIGS["C1"].scaled(seq=S, head_dim=D, n_q_heads=H, n_kv_heads=Hkv, seed=29)
    Q, K, V = (si.make_layer(cfg)[k].cuda() for k in "QKV")
    G, T = H // Hkv, (S + 127) // 128
    n = max(u for u in range(1, Hkv) if Hkv % u == 0 and u * G * (T + 1) < 444)
    assert H * (T + 1) >= 444

    def attend(Q, K, V):
        O, lse = torch.empty_like(Q), torch.empty(Q.shape[:3], device="cuda")
        kvm.kvm_prefill_attend(kvm.make_params(1, Q.shape[1], K.shape[1], S, D, torch.bfloat16), Q, K, V, O, lse)
        return O
    together = attend(Q, K, V)
    few = torch.cat([attend(*(t[:, i * k:(i + n) * k].contiguous() for t, k in ((Q, G), (K, 1), (V, 1))))
                     for i in range(0, Hkv, n)], 1)
    causal = torch.ones(S, S, dtype=torch.bool, device="cuda").tril()
    err = np.zeros(2)
    for u in range(Hkv):
        L = (Q[0, u * G:(u + 1) * G].double() @ K[0, u].double().T / np.sqrt(D)).masked_fill(~causal, float("-inf"))
        ref = torch.softmax(L, -1) @ V[0, u].double()
        err += [(O[0, u * G:(u + 1) * G].double() - ref).square().sum().item() for O in (together, few)]
    assert err[0] <= err[1]


def test_prefill_attention_with_unscaled_logits_and_a_custom_scale():
    """Nearly one-hot rows (logits of standard deviation in the tens) move the reference maximum often."""
    from oracle import kvmo
    cfg = si.CONFIGS["C1"].scaled(seq=512, n_q_heads=2, n_kv_heads=2, seed=32, logit_std=-1.0)
    d = si.make_layer(cfg)
    p = kvm.make_params(1, 2, 2, 512, 128, torch.bfloat16, softmax_scale=0.05)
    Q, K, V = d["Q"].cuda(), d["K"].cuda(), d["V"].cuda()
    O, lse = torch.empty_like(Q), torch.empty(1, 2, 512, device="cuda")
    kvm.kvm_prefill_attend(p, Q, K, V, O, lse)
    torch.cuda.synchronize()
    refO, ref_lse = kvmo.prefill_attend(d["Q"], d["K"], d["V"], 0.05)
    g_lse = lse.cpu().numpy().astype(np.float64)
    assert np.abs(g_lse - ref_lse).max() <= 1e-5 * np.abs(ref_lse).max() + LSE_ATOL    # logits of magnitude 100s
    gO = O.float().cpu().numpy().astype(np.float64)
    assert (np.abs(gO - refO) <= 1e-2 * np.abs(refO) + 2.0 ** -8 * np.abs(d["V"].float().numpy()).max()).all()


def test_compression_fed_by_the_attention_kernels_lse_matches_the_checker():
    """The production order: prefill attention -> its lse -> kvm_compress_with_lse (no row pass)."""
    from oracle import kvmo
    from parity import Case, _chain, f32, kv_error, score_excess, KV_TOL
    S = 1000
    cfg = si.CONFIGS["C1"].scaled(seq=S, n_q_heads=4, n_kv_heads=2, seed=33)
    d = si.make_layer(cfg)
    p, Q, K, V, O, lse = _run(cfg, d)
    case = Case(d["Q"], d["K"], d["V"], budget=0.5)
    comp = kvm.Compressor(p, want_scores=True)
    kvm.kvm_compress_with_lse(p, Q, K, V, lse, comp.K_out, comp.V_out, comp.out_len, comp.out_pos, comp.scores, None,
                              comp.ws)
    torch.cuda.synchronize()
    ref = kvmo.scores(d["Q"], d["K"])
    g_scores = comp.scores.cpu().numpy().reshape(2, S)
    assert score_excess(g_scores, ref.reshape(2, S)) <= 1.0
    sim = torch.empty(1, 2, S, device="cuda")
    ratio = torch.empty(2, device="cuda")
    kvm.kvm_layer_ratio(p, K, ratio, sim, comp.ws)
    cap, n_r, n_h = kvm.kvm_sizes(p)
    ch = _chain(case, g_scores.astype(np.float64), sim.cpu().numpy().reshape(2, S).astype(np.float64), cap, n_r, n_h)
    g_len = comp.out_len.cpu().numpy().reshape(2)
    assert np.array_equal(g_len, ch["out_len"])
    g_pos = comp.out_pos.cpu().numpy().reshape(2, cap)
    rK, rV = kvmo.merge(d["K"][0], d["V"][0], ch["set_start"], ch["pivot"], ch["out_len"], f32(5.0), True)
    for u in range(2):
        n = g_len[u]
        assert np.array_equal(g_pos[u, :n], ch["pivot"][u, :n])
        assert kv_error(comp.K_out[0, u, :n].float().cpu().numpy(), rK[u, :n]) <= KV_TOL
        assert kv_error(comp.V_out[0, u, :n].float().cpu().numpy(), rV[u, :n]) <= KV_TOL
    # the same scores as the library's own two-pass path, to the score bar
    own = torch.empty_like(comp.scores)
    kvm.kvm_score(p, Q, K, None, own, comp.ws)
    torch.cuda.synchronize()
    assert score_excess(g_scores, own.cpu().numpy().reshape(2, S).astype(np.float64)) <= 1.0


def test_prefill_attention_full_c1_layer_sampled_heads_and_twice_identical():
    """The benchmark's shape and launch configuration: every head through the library, two heads against the
    checker in full, two runs bit-identical, untouched memory around the outputs."""
    from oracle import kvmo
    cfg = si.CONFIGS["C1"]
    d = si.make_layer(cfg)
    p, Q, K, V, O, lse = _run(cfg, d)
    O2, lse2 = torch.empty_like(O), torch.empty_like(lse)
    kvm.kvm_prefill_attend(p, Q, K, V, O2, lse2)
    torch.cuda.synchronize()
    assert torch.equal(O, O2) and torch.equal(lse, lse2)
    assert torch.isfinite(O.float()).all() and torch.isfinite(lse).all()
    for h in (0, 31):
        refO, ref_lse = kvmo.prefill_attend(d["Q"][:, h:h + 1], d["K"][:, h:h + 1], d["V"][:, h:h + 1])
        _check(O[:, h:h + 1], lse[:, h:h + 1], refO, ref_lse, d["V"][:, h:h + 1], 1)


def test_prefill_attention_rejects_what_it_does_not_support():
    p = kvm.make_params(1, 2, 2, 256, 64, torch.float32)
    x = torch.zeros(1, 2, 256, 64, device="cuda")
    with pytest.raises(kvm.KvmError) as e:
        kvm.kvm_prefill_attend(p, x, x, x, x, torch.zeros(1, 2, 256, device="cuda"))
    assert e.value.status == -7          # KVM_E_UNSUPPORTED
