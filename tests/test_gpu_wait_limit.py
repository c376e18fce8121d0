"""The give-up path of the bounded device waits (failure detection without a fault).

Every wait on an mbarrier has a limit; in the score kernels, when one runs out the kernel stops
touching tensor memory, writes NaN for the work items it could not finish, reports KVM_E_DEVICE_TIMEOUT through
kvm_stats, frees its tensor memory and returns.  Nothing in the shipped library can make a wait run out, so
this test uses a second build of the same sources (never loaded by the package) in which the limit is two
milliseconds of SM clocks and the TMA producer of one block leaves out its first stage: the barrier of that stage is
never armed, the MMA warp's wait for it gives up, and the kernel must come back by itself.  No trap, no unbounded
loop, no bad address is involved.  The eviction rule is used so that what runs after the score step (the
conserved tokens are gathered by index) does not depend on the values of the scores.
"""
import ctypes

import numpy as np
import pytest
import torch

import paper_2407_08454_b200 as kvm
from paper_2407_08454_b200 import build
from paper_2407_08454_b200 import synth_inputs as si

pytestmark = pytest.mark.gpu


def test_a_wait_that_runs_out_is_reported_and_the_next_call_is_correct():
    from oracle import kvmo
    from parity import SCORE_ATOL, SCORE_RTOL, f32
    lib = ctypes.CDLL(build.build_waittest())
    cfg = si.CONFIGS["C1"].scaled(seq=1024, n_q_heads=4, n_kv_heads=4, seed=77)     # 8 tiles: the longest items have 4 stages
    d = si.make_layer(cfg)
    Q, K, V = d["Q"].cuda(), d["K"].cuda(), d["V"].cuda()
    p = kvm.make_params(cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.seq, cfg.head_dim, cfg.torch_dtype,
                        budget=0.5, set_rule=kvm.KVM_SETS_CONSERVED_ONLY)
    cap, _, _ = kvm.kvm_sizes(p)
    ws = torch.empty(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    Ko = torch.zeros(cfg.batch, cfg.n_kv_heads, cap, cfg.head_dim, dtype=Q.dtype, device="cuda")
    Vo = torch.zeros_like(Ko)
    out_len = torch.zeros(cfg.batch, cfg.n_kv_heads, dtype=torch.int32, device="cuda")
    out_pos = torch.zeros(cfg.batch, cfg.n_kv_heads, cap, dtype=torch.int32, device="cuda")
    scores = torch.zeros(cfg.batch, cfg.n_kv_heads, cfg.seq, device="cuda")
    stats = kvm.new_stats("cuda")
    vp = ctypes.c_void_p
    rc = lib.kvm_compress(ctypes.byref(p), vp(Q.data_ptr()), vp(K.data_ptr()), vp(V.data_ptr()), vp(Ko.data_ptr()),
                          vp(Vo.data_ptr()), vp(out_len.data_ptr()), vp(out_pos.data_ptr()), vp(scores.data_ptr()),
                          vp(stats.data_ptr()), vp(ws.data_ptr()), ctypes.c_size_t(ws.numel()),
                          vp(torch.cuda.current_stream().cuda_stream))
    assert rc == 0                                  # nothing is known on the host when the call returns
    torch.cuda.synchronize()                        # the kernels came back by themselves
    assert kvm.read_stats(stats).status == -9       # KVM_E_DEVICE_TIMEOUT
    assert torch.isnan(scores).any()                # what could not be finished is marked, not made up
    # the context is intact: the shipped library computes the same layer correctly right afterwards
    good = torch.empty_like(scores)
    kvm.kvm_score(p, Q, K, None, good, ws)
    torch.cuda.synchronize()
    ref = kvmo.scores(d["Q"].double().numpy(), d["K"].double().numpy(), f32(1.0 / np.sqrt(np.float32(cfg.head_dim))))
    g = good.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= SCORE_RTOL * np.abs(ref) + SCORE_ATOL)


def _ptrs(*tensors):
    return [ctypes.c_void_p(0 if t is None else t.data_ptr()) for t in tensors]


def test_a_piece_that_gave_up_marks_every_row_and_score_that_depends_on_it():
    """Every step is a piece of its own here (4 heads x 8 tiles, 144 steps) and block 1 gives up its only one: in the row
    pass the first of the two pieces of query tile 1, in the column pass the first piece of key tile 6.  The row's other
    piece is good; joined, the row is still NaN, and with it the scores of every key that its queries see."""
    lib = ctypes.CDLL(build.build_waittest())
    g = torch.Generator().manual_seed(5)
    Q, K = ((torch.randn(1, 4, 1024, 128, generator=g) * s).bfloat16().cuda() for s in (2, 1))
    p = kvm.make_params(1, 4, 4, 1024, 128, torch.bfloat16)
    ws = torch.zeros(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    scores, lse, good_scores, good_lse = (torch.zeros(1, 4, 1024, device="cuda") for _ in range(4))
    size, st = ctypes.c_size_t(ws.numel()), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.kvm_score(ctypes.byref(p), *_ptrs(Q, K, None, scores, ws), size, st) == 0
    assert lib.kvm_row_lse(ctypes.byref(p), *_ptrs(Q, K, lse, ws), size, st) == 0
    torch.cuda.synchronize()
    kvm.kvm_score(p, Q, K, None, good_scores, ws)
    kvm.kvm_row_lse(p, Q, K, good_lse, ws)
    bad_lse, bad_scores = torch.zeros_like(lse, dtype=torch.bool), torch.zeros_like(scores, dtype=torch.bool)
    bad_lse[0, 0, 128:256] = True
    bad_scores[0, 0, :256] = True
    bad_scores[0, 0, 768:896] = True
    for got, good, bad in ((lse, good_lse, bad_lse), (scores, good_scores, bad_scores)):
        assert torch.equal(torch.isnan(got), bad)
        assert torch.equal(got[~bad], good[~bad])


@pytest.mark.parametrize("H,S,dtype", [(300, 500, torch.bfloat16), (750, 200, torch.float32)])
def test_after_a_give_up_every_item_of_the_block_is_marked(H, S, dtype):
    """More items per block than the passes have buffers to join an item's parts in.  Block 1 gives up at its first step:
    every row (key) of every item it has a step of is NaN, none keeps what was in memory before, and the other blocks'
    are those of the library.  bf16: items stay whole here and are dealt back and forth, longest first; fp32: block c takes
    the steps from c q on."""
    lib = ctypes.CDLL(build.build_waittest())
    D, T, P = 64, (S + 127) // 128, 148
    g = torch.Generator(device="cuda").manual_seed(S)
    Q, K = ((torch.randn(1, H, S, D, generator=g, device="cuda") * s).to(dtype) for s in (2, 1))
    p = kvm.make_params(1, H, H, S, D, dtype)
    ws = torch.zeros(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    scores, lse = (torch.full((1, H, S), 5.0, device="cuda") for _ in range(2))
    good_scores, good_lse = torch.empty_like(scores), torch.empty_like(lse)
    kvm.kvm_row_lse(p, Q, K, good_lse, ws)
    kvm.kvm_score(p, Q, K, good_lse, good_scores, ws)
    kvm.kvm_row_lse(p, Q, K, good_lse, ws)                        # (finite states in the workspace)
    size, st = ctypes.c_size_t(ws.numel()), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.kvm_row_lse(ctypes.byref(p), *_ptrs(Q, K, lse, ws), size, st) == 0
    assert lib.kvm_score(ctypes.byref(p), *_ptrs(Q, K, good_lse, scores, ws), size, st) == 0
    torch.cuda.synchronize()
    bad_rows, bad_keys = (torch.zeros(H, T * 128, dtype=torch.bool) for _ in range(2))
    if dtype == torch.bfloat16:
        for f in range(H * T // P + 1):
            k = f * P + (P - 2 if f & 1 else 1)
            if k < H * T:
                bad_rows[k % H, (T - 1 - k // H) * 128:(T - k // H) * 128] = True
                bad_keys[k % H, k // H * 128:(k // H + 1) * 128] = True
    else:
        tri = T * (T + 1) // 2
        q = -(-H * tri // P)
        for h in range(H):
            for n in range(T):                                    # an item of n + 1 steps that starts at step s of the pass
                s = h * tri + n * (n + 1) // 2
                if s < 2 * q and s + n + 1 > q:
                    bad_rows[h, n * 128:(n + 1) * 128] = True
                    bad_keys[h, (T - 1 - n) * 128:(T - n) * 128] = True
    for got, good, bad in ((lse, good_lse, bad_rows), (scores, good_scores, bad_keys)):
        bad = bad[None, :, :S].cuda()
        assert bad.any() and torch.equal(torch.isnan(got), bad)
        assert torch.equal(got[~bad], good[~bad])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("U,G,rows,bad", [
    (4, 4, 512, [0]),              # clusters: block 1 holds rows of unit 0
    (300, 4, 600, [2, 3]),         # equal shares: block 1 holds all rows of units 2 and 3
    (200, 4, 3000, [1, 2]),        # ... the end of unit 1 and the beginning of unit 2
])
def test_the_decode_attention_kernels_also_come_back_and_mark_their_units(U, G, rows, bad, dtype):
    """Block 1 leaves out its first stage: the units that it holds rows of are NaN, the others are the library's."""
    lib = ctypes.CDLL(build.build_waittest())
    g = torch.Generator().manual_seed(U)
    q, K, V = (torch.randn(1, h, n, 64, generator=g).to(dtype).cuda() for h, n in ((U * G, 1), (U, rows), (U, rows)))
    p = kvm.make_params(1, U * G, U, rows, 64, dtype, budget=1.0, recent_ratio=0.0, heavy_ratio=0.0)
    ws = torch.zeros(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    out, good = (torch.full((U, G, 64), 5.0, device="cuda") for _ in range(2))
    size, st = ctypes.c_size_t(ws.numel()), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.kvm_attend(ctypes.byref(p), *_ptrs(q, K, V), ctypes.c_int32(rows), *_ptrs(None, out, ws), size, st) == 0
    torch.cuda.synchronize()                        # the kernels came back by themselves
    kvm.kvm_attend(p, q.squeeze(2).contiguous(), K, V, rows, None, good, ws)
    assert torch.isfinite(good).all() and torch.isnan(out[bad]).all()
    rest = [u for u in range(U) if u not in bad]
    assert torch.equal(out[rest], good[rest])


def test_the_prefill_attention_kernel_also_comes_back_and_reports():
    """Same build, the attention kernel: its producer leaves out the fourth V tile of every work item that has one,
    the MMA thread's wait for it runs out, the kernel returns, the status is set, the rows that were in hand are NaN
    and the work items that never needed that tile are complete."""
    from oracle import kvmo
    lib = ctypes.CDLL(build.build_waittest())
    cfg = si.CONFIGS["C1"].scaled(seq=1024, n_q_heads=4, n_kv_heads=4, seed=78)     # 8 query tiles per head, one per CTA
    d = si.make_layer(cfg)
    Q, K, V = d["Q"].cuda(), d["K"].cuda(), d["V"].cuda()
    p = kvm.make_params(cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.seq, cfg.head_dim, cfg.torch_dtype)
    O = torch.zeros_like(Q)
    lse = torch.zeros(1, 4, 1024, device="cuda")
    stats = kvm.new_stats("cuda")
    vp = ctypes.c_void_p
    rc = lib.kvm_prefill_attend(ctypes.byref(p), vp(Q.data_ptr()), vp(K.data_ptr()), vp(V.data_ptr()), vp(O.data_ptr()),
                                vp(lse.data_ptr()), vp(stats.data_ptr()), vp(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()                        # the kernel came back by itself
    assert kvm.read_stats(stats).status == -9       # KVM_E_DEVICE_TIMEOUT
    bad = torch.isnan(lse)
    assert bad[:, :, 3 * 128:].all()                # query tiles 3..7 need a fourth V tile: marked, not made up
    assert not bad[:, :, :3 * 128].any()            # tiles 0..2 never needed it
    refO, ref_lse = kvmo.prefill_attend(d["Q"][:, :, :384], d["K"][:, :, :384], d["V"][:, :, :384])
    assert np.abs(lse[:, :, :384].cpu().numpy() - ref_lse).max() <= 2e-4
    # the context is intact: the shipped library computes the same layer correctly right afterwards
    kvm.kvm_prefill_attend(p, Q, K, V, O, lse)
    torch.cuda.synchronize()
    refO, ref_lse = kvmo.prefill_attend(d["Q"], d["K"], d["V"])
    assert torch.isfinite(lse).all() and np.abs(lse.cpu().numpy() - ref_lse).max() <= 2e-4


def test_after_a_give_up_of_the_two_tile_attention_every_row_of_the_block_is_marked():
    """450 pairs of tiles: every block's first one is the longest (tiles 4 and 5 of a head), whose fourth V tile never comes, so
    that every row of every block's items is marked and none keeps what was in memory before."""
    lib = ctypes.CDLL(build.build_waittest())
    H, S, D = 150, 700, 64
    g = torch.Generator(device="cuda").manual_seed(79)
    Q, K, V = (torch.randn(1, H, S, D, generator=g, device="cuda").bfloat16() for _ in range(3))
    p = kvm.make_params(1, H, H, S, D, torch.bfloat16)
    O, lse, stats = torch.zeros_like(Q), torch.zeros(1, H, S, device="cuda"), kvm.new_stats("cuda")
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.kvm_prefill_attend(ctypes.byref(p), *_ptrs(Q, K, V, O, lse, stats), st) == 0
    torch.cuda.synchronize()                        # the kernel came back by itself
    assert kvm.read_stats(stats).status == -9       # KVM_E_DEVICE_TIMEOUT
    # (a block's first pair: the rows of tile 4 too, whose group had its four steps' logits but not the fourth product)
    assert torch.isnan(lse).all() and torch.isnan(O).all()
    kvm.kvm_prefill_attend(p, Q, K, V, O, lse)      # the context is intact
    torch.cuda.synchronize()
    assert torch.isfinite(lse).all() and torch.isfinite(O).all()
