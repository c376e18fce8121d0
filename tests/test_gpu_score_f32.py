"""The fp32 score passes (three-plane tensor-core products) against fp64 at the edges of their tiles and of their
split of the work."""
import math

import pytest
import torch

import paper_2407_08454_b200 as kvm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,S,D", [
    (1, 1, 1, 1, 64),          # one token
    (1, 2, 1, 128, 128),       # one full tile, group of two
    (2, 3, 3, 129, 64),        # one token past a tile, batch
    (1, 6, 2, 257, 128),       # group of three over three tiles: the column pass wraps to the next head mid-item
    (1, 1, 1, 2300, 128),      # one head: an item is cut into the most pieces
    (1, 16, 8, 1500, 64),      # several items per CTA, cut at both ends
    (4, 128, 64, 700, 64),     # too many rows for cut items: whole ones
])
def test_scores_and_row_lse_against_fp64(B, Hq, Hkv, S, D):
    g = torch.Generator().manual_seed(S + D)
    Q = (torch.randn(B, Hq, S, D, generator=g) * 4).cuda()
    K = torch.randn(B, Hkv, S, D, generator=g).cuda()
    p = kvm.make_params(B, Hq, Hkv, S, D, torch.float32, budget=1.0, recent_ratio=0.0, heavy_ratio=0.0)
    ws = torch.full((kvm.kvm_workspace_bytes(p),), 255, dtype=torch.uint8, device="cuda")      # NaN patterns
    scores = torch.full((B, Hkv, S), float("nan"), device="cuda")
    lse = torch.full((B, Hq, S), float("nan"), device="cuda")
    kvm.kvm_score(p, Q, K, None, scores, ws)
    kvm.kvm_row_lse(p, Q, K, lse, ws)
    with_lse = torch.full_like(scores, float("nan"))
    kvm.kvm_score(p, Q, K, lse, with_lse, ws)
    c = 1.0 / math.sqrt(D)
    # a logit is D / 16 accumulations of exact products and one addition, each off by at most 2^-23 of |q||k| c (plus as
    # much again for the rounding of the scale, the exponent and the log-sum-exp, all below 2^-23 of 64 + |q||k| c)
    qk = c * Q.norm(dim=-1).max().item() * K.norm(dim=-1).max().item()
    delta = 2.0 ** -23 * ((D / 16 + 1) * qk + 3 * (64 + qk))
    G = Hq // Hkv
    mask = torch.triu(torch.ones(S, S, dtype=torch.bool, device="cuda"), 1)
    for b in range(B):
        for u in {0, Hkv // 2, Hkv - 1}:
            L = (Q[b, u * G:(u + 1) * G].double() @ K[b, u].double().T * c).masked_fill(mask, float("-inf"))
            ref_lse = torch.logsumexp(L, -1)
            ref = torch.exp(L - ref_lse[..., None]).sum(-2).mean(0)
            assert (lse[b, u * G:(u + 1) * G].double() - ref_lse).abs().max().item() <= delta
            for got in (scores, with_lse):
                # every term of a column sum is off by at most exp(2 delta) - 1; fp32 sums of positive terms add 2^-17
                assert ((got[b, u].double() - ref).abs() / ref).max().item() <= 2.1 * delta + 2.0 ** -17


@pytest.mark.parametrize("Hq,Hkv,S,D,joined", [
    (1, 1, 130, 64, False),        # two states a row, one step a CTA
    (4, 4, 512, 128, False),       # four states, one step
    (4, 4, 512, 64, True),         # ... of half the channels
    (8, 4, 1024, 64, False),       # five, two steps
    (1, 1, 700, 128, True),        # six, one step
    (32, 32, 389, 64, True),       # two, three steps
    (32, 32, 700, 128, True),      # two, five steps
])
def test_row_states_are_joined_by_a_launch_where_steps_would_read_many(Hq, Hkv, S, D, joined):
    """A launch between the passes costs a small call more than its steps' few reads; both forms give the same bits as the
    column pass fed with the row log-sum-exp (which joins the states by a kernel of its own) to the rounding of the units."""
    from parity import launched
    g = torch.Generator().manual_seed(S)
    Q, K = torch.randn(1, Hq, S, D, generator=g).cuda(), torch.randn(1, Hkv, S, D, generator=g).cuda()
    p = kvm.make_params(1, Hq, Hkv, S, D, torch.float32, budget=1.0, recent_ratio=0.0, heavy_ratio=0.0)
    ws = torch.empty(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    scores, with_lse, lse = torch.empty(1, Hkv, S, device="cuda"), torch.empty(1, Hkv, S, device="cuda"), torch.empty(1, Hq, S, device="cuda")
    kvm.kvm_score(p, Q, K, None, scores, ws)
    kvm.kvm_row_lse(p, Q, K, lse, ws)
    kvm.kvm_score(p, Q, K, lse, with_lse, ws)
    # (log2 units to natural and back: two roundings of a number below 64, 2^-24 of it each)
    assert ((scores - with_lse).abs() <= 2.0 ** -17 * with_lse).all()
    names = launched(lambda: kvm.kvm_score(p, Q, K, None, scores, ws))
    assert sum("join_states_kernel" in n for n in names) == int(joined) and sum("score_f32_kernel" in n for n in names) == 2


def _reference(Q, K, allowed):
    L = (Q.double() @ K.double().transpose(-1, -2) / math.sqrt(Q.shape[-1])).masked_fill(~allowed, float("-inf"))
    return torch.nan_to_num(torch.softmax(L, -1)).sum(-2)          # (rows without any key weigh nothing)


@pytest.mark.parametrize("S,D", [(300, 64), (1000, 128)])
def test_keys_at_the_lowest_value_get_no_weight(S, D):
    """Key rows filled with the type's lowest value, as masks are: their logits overflow to -inf, their weight is zero and
    the other keys' scores are what they are without them, also where a query's first keys are all masked."""
    g = torch.Generator().manual_seed(S)
    Q = torch.randn(1, 4, S, D, generator=g).abs().cuda() + 0.1
    K = torch.randn(1, 4, S, D, generator=g).cuda()
    masked = torch.zeros(4, S, dtype=torch.bool, device="cuda")
    masked[0, 3], masked[1, 40:170], masked[2, :40], masked[3, :200] = True, True, True, True
    K[0][masked] = torch.finfo(torch.float32).min
    p = kvm.make_params(1, 4, 4, S, D, torch.float32, budget=1.0, recent_ratio=0.0, heavy_ratio=0.0)
    ws = torch.empty(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    scores, lse, with_lse = (torch.empty(1, 4, S, device="cuda") for _ in range(3))
    kvm.kvm_score(p, Q, K, None, scores, ws)
    kvm.kvm_row_lse(p, Q, K, lse, ws)
    kvm.kvm_score(p, Q, K, lse, with_lse, ws)
    causal = torch.ones(S, S, dtype=torch.bool, device="cuda").tril()
    for u in range(4):
        ref = _reference(Q[0, u], K[0, u].masked_fill(masked[u, :, None], 0.0), causal & ~masked[u])
        dead = masked[u] & (torch.arange(S, device="cuda") >= masked[u].logical_not().nonzero()[0])
        for got in (scores[0, u], with_lse[0, u]):
            assert (got[dead] == 0).all()
            live = ~masked[u]
            assert ((got[live].double() - ref[live]).abs() <= 1e-4 * ref[live]).all()


def test_a_nan_query_reaches_only_the_keys_before_it():
    Q, K = (torch.randn(1, 1, 700, 64, generator=torch.Generator().manual_seed(s)).cuda() for s in (1, 2))
    Q[0, 0, 333, 5] = float("nan")
    p = kvm.make_params(1, 1, 1, 700, 64, torch.float32, budget=1.0, recent_ratio=0.0, heavy_ratio=0.0)
    ws = torch.empty(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    scores = torch.empty(1, 1, 700, device="cuda")
    kvm.kvm_score(p, Q, K, None, scores, ws)
    assert torch.isnan(scores[0, 0, :334]).all()
    ref = _reference(torch.nan_to_num(Q[0, 0]), K[0, 0], torch.ones(700, 700, dtype=torch.bool, device="cuda").tril())
    assert ((scores[0, 0, 334:].double() - ref[334:]).abs() <= 1e-4 * ref[334:]).all()
