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
