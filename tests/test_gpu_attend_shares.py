"""Decode attention where the rows are split over the blocks: shares that cut units anywhere, groups of every size,
empty units, rows that no block of rows divides, against fp64."""
import pytest
import torch

import paper_2407_08454_b200 as kvm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("B,G,Hkv,rows,D", [
    (1, 1, 1, 1, 128),         # one row
    (1, 3, 2, 15, 64),         # less than a 16-row block
    (2, 5, 2, 65, 128),        # one row past a stage
    (1, 8, 1, 700, 64),        # one unit over many blocks
    (1, 9, 3, 333, 128),       # more query heads than one pass takes
    (3, 2, 37, 97, 64),        # more units than blocks need, shares cut in the middle of units
    (1, 1, 300, 70, 128),      # more units than SMs
    (1, 1, 600, 129, 64),      # many short units: small blocks, one row past two groups' rounds
    (3, 2, 70, 200, 128),      # ... for two query heads
    (1, 8, 200, 150, 64),      # as many units for eight: equal shares
    (4, 4, 100, 3, 64),        # many units of a row or two: shares whose ends fall between units' rows
    (1, 2, 1100, 30, 128),     # several units per share, most of each for the unit itself
])
def test_attend_against_fp64(B, G, Hkv, rows, D, dtype):
    g = torch.Generator().manual_seed(rows * G + D)
    q = (torch.randn(B, Hkv * G, D, generator=g) * 3).to(dtype).cuda()
    K = torch.randn(B, Hkv, rows, D, generator=g).to(dtype).cuda()
    V = torch.randn(B, Hkv, rows, D, generator=g).to(dtype).cuda()
    n = torch.randint(0, rows + 1, (B, Hkv), generator=g, dtype=torch.int32)
    n.view(-1)[-1] = rows
    p = kvm.make_params(B, Hkv * G, Hkv, rows, D, dtype, budget=1.0, recent_ratio=0.0, heavy_ratio=0.0)
    ws = torch.full((kvm.kvm_workspace_bytes(p),), 255, dtype=torch.uint8, device="cuda")
    for length in (None, n):
        Kc, Vc = K.clone(), V.clone()
        dead = (torch.arange(rows) >= (n[..., None] if length is not None else torch.full_like(n, rows)[..., None]))
        Kc[dead.cuda()], Vc[dead.cuda()] = float("nan"), float("nan")      # rows past a unit's length may hold anything
        out = torch.full((B, Hkv * G, D), 7.0, device="cuda")
        kvm.kvm_attend(p, q, Kc, Vc, rows, None if length is None else length.cuda(), out, ws)
        L = (q.double().view(B, Hkv, G, D) @ K.double().transpose(-1, -2)) / D ** 0.5
        L = L.masked_fill(dead.cuda()[:, :, None], float("-inf"))
        ref = torch.nan_to_num(torch.softmax(L, -1)) @ V.double()
        # a logit of at most ~20 is off by (D + few) * 2^-24 of |q||k| c; weights and sums add 2^-20 of the largest value
        qk = (q.double().norm(dim=-1).max() * K.double().norm(dim=-1).max() / D ** 0.5).item()
        tol = (2 * (D / 16 + 4) * 2.0 ** -23 * qk + 2.0 ** -20) * V.double().abs().max().item()
        assert (out.double().view_as(ref) - ref).abs().max().item() <= tol


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("G,Hkv,rows,D", [(1, 2, 300, 64), (4, 3, 2000, 128), (2, 200, 333, 64), (8, 150, 400, 128)])
def test_attend_with_infinite_values(G, Hkv, rows, D, dtype):
    """An infinite value in a row that has any weight makes its channel infinite, and no other."""
    g = torch.Generator().manual_seed(rows + G)
    q = torch.randn(1, Hkv * G, D, generator=g).to(dtype).cuda()
    K = torch.randn(1, Hkv, rows, D, generator=g).to(dtype).cuda()
    V = torch.randn(1, Hkv, rows, D, generator=g).to(dtype).cuda()
    V[0, 0, 0, 3], V[0, 1, rows - 1, 5], V[0, -1, rows // 2, D - 1] = float("inf"), float("-inf"), float("inf")
    V[0, -1, 7, D - 1], V[0, -1, rows // 3, 0], V[0, -1, rows // 3 + 1, 0] = float("inf"), float("inf"), float("-inf")
    p = kvm.make_params(1, Hkv * G, Hkv, rows, D, dtype, budget=1.0, recent_ratio=0.0, heavy_ratio=0.0)
    ws = torch.empty(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    out = torch.empty(1, Hkv * G, D, device="cuda")
    kvm.kvm_attend(p, q, K, V, rows, None, out, ws)
    L = (q.double().view(1, Hkv, G, D) @ K.double().transpose(-1, -2)) / D ** 0.5
    ref = (torch.softmax(L, -1) @ V.double()).view_as(out)
    for test in (torch.isposinf, torch.isneginf, torch.isnan):
        assert torch.equal(test(out), test(ref)) and test(ref).any()
    fine = torch.isfinite(ref)
    assert (out.double() - ref)[fine].abs().max().item() <= 1e-4      # |V| is below 5: fp32 sums, logits off by ~1e-5


@pytest.mark.parametrize("dtype,step", [(torch.bfloat16, 128), (torch.float32, 64)])
def test_attend_at_the_end_of_the_value_range(dtype, step):
    """Two rows of a unit have weight, a stage of rows apart in the same lanes' hands, the later one 2^7.5 times the
    earlier one's: weights are taken relative to a reference that is not below any logit, so that values near the largest
    number do not overflow on the way."""
    q = torch.zeros(1, 1, 64, dtype=dtype, device="cuda")
    q[..., 0] = 8.0
    K = torch.zeros(1, 1, 2048, 64, dtype=dtype, device="cuda")
    K[..., 0] = -1000.0
    K[0, 0, 0, 0], K[0, 0, step, 0] = 0.0, 5.1875
    V = torch.full_like(K, 3e38)
    p = kvm.make_params(1, 1, 1, 2048, 64, dtype, budget=1.0, recent_ratio=0.0, heavy_ratio=0.0)
    ws = torch.empty(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    out = torch.empty(1, 1, 64, device="cuda")
    kvm.kvm_attend(p, q, K, V, 2048, None, out, ws)
    assert ((out.double() / V[0, 0, 0].double() - 1).abs() <= 2.0 ** -18).all()
