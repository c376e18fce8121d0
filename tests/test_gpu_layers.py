"""Layer stacks that go through the kernels together against the same layers one by one."""
import pytest
import torch

import paper_2407_08454_b200 as kvm
from paper_2407_08454_b200 import binding
from paper_2407_08454_b200 import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,S,Hq,Hkv,D,dtype", [
    (1, 300, 4, 2, 64, "bf16"),
    (3, 389, 4, 4, 128, "bf16"),
    (9, 257, 8, 2, 128, "bf16"),      # more layers than go together
    (5, 1500, 16, 2, 64, "bf16"),     # column items cut across layers
    (2, 300, 4, 2, 64, "f32"),        # fp32 tensors: layer by layer
])
def test_layers_together_match_layers_alone(n, S, Hq, Hkv, D, dtype, monkeypatch):
    cfg = si.CONFIGS["C1"].scaled(seq=S, head_dim=D, n_q_heads=Hq, n_kv_heads=Hkv, dtype=dtype, seed=S + n)
    layers = [tuple(si.make_layer(cfg, l)[k].cuda() for k in "QKV") for l in range(n)]
    eps = [0.6 + 0.3 * l / n for l in range(n)]
    kw = dict(budget=cfg.budget)
    p = kvm.make_params(1, Hq, Hkv, S, D, cfg.torch_dtype, **kw)
    one, many = kvm.kvm_workspace_bytes(p), binding.kvm_layers_workspace_bytes(p, n)
    assert many >= one and (many > one) == (dtype == "bf16" and n > 1)
    together, _ = kvm.compress_layers(p, layers, eps)
    monkeypatch.setattr(binding, "kvm_layers_workspace_bytes", lambda p, n: one)      # one layer's: no room for more
    alone, _ = kvm.compress_layers(p, layers, eps)
    for l, (Q, K, V) in enumerate(layers):
        ref = kvm.Compressor(kvm.make_params(1, Hq, Hkv, S, D, cfg.torch_dtype, sim_threshold=eps[l], **kw))(Q, K, V)
        assert all(torch.equal(getattr(alone[l], k), getattr(ref, k)) for k in ("out_len", "out_pos", "K_out", "V_out"))
        # together the column sums may be added in other pieces: scores that tie to fp32 rounding may change places, and
        # with them a token be conserved or not.  A row that has the same pivot in both results, as its two neighbours
        # have, is the same set (the similarities are the same) and has to be the same bits.
        got, rows, same = together[l], 0, 0
        assert (got.out_len - ref.out_len).abs().max() <= 2
        for h in range(Hkv):
            a, b = (c.out_pos[0, h, :int(c.out_len[0, h])].tolist() for c in (got, ref))
            triples = {t: i for i, t in enumerate(zip([-1] + b, b, b[1:] + [S]))}
            pairs = [(i, triples[t]) for i, t in enumerate(zip([-1] + a, a, a[1:] + [S])) if t in triples]
            rows, same = rows + len(b), same + len(pairs)
            x, y = (torch.tensor(ix, device="cuda") for ix in zip(*pairs))
            assert torch.equal(got.K_out[0, h, x], ref.K_out[0, h, y]) and torch.equal(got.V_out[0, h, x], ref.V_out[0, h, y])
        assert same >= 0.97 * rows


def _call_layers(name, p, layers, outs, ws, eps=None):
    """kvm_compress_layers or kvm_compress_layers_filled on the caller's buffers (K_out, V_out, out_len, out_pos per layer)."""
    import ctypes
    array = ctypes.c_void_p * len(layers)
    q, k, v = (array(*[l[i].data_ptr() for l in layers]) for i in range(3))
    ko, vo, ln, pos = (array(*[o[i].data_ptr() for o in outs]) for i in range(4))
    binding._call(name, p, len(layers), eps and (ctypes.c_float * len(layers))(*eps), q, k, v, ko, vo, ln, pos, None,
                  ws.data_ptr(), ws.nbytes, binding._stream(None))


def _dirty_outputs(n, Hkv, cap, D, dtype):
    def full(shape, dt):
        t = torch.empty(shape, dtype=dt, device="cuda")
        t.view(torch.uint8).fill_(0xFF)
        return t
    return [(full((1, Hkv, cap, D), dtype), full((1, Hkv, cap, D), dtype), full((1, Hkv), torch.int32),
             full((1, Hkv, cap), torch.int32)) for _ in range(n)]


@pytest.mark.parametrize("n,S,Hkv,D,dtype,rules", [
    (3, 389, 4, 128, "bf16", {}),                     # layers together; the last tile's share of the rows is cut
    (9, 1500, 8, 128, "bf16", {}),                    # two groups of layers, megabytes each
    (2, 33, 3, 64, "f32", {}),                        # two tiles, capacity 16
    (2, 700, 2, 64, "bf16", {"set_rule": kvm.KVM_SETS_CONSERVED_ONLY}),     # a gather instead of the merge
    (2, 640, 2, 128, "bf16", {"weight_rule": kvm.KVM_WEIGHT_SET_SIGMA}),
])
def test_rows_past_a_units_length_are_zero(n, S, Hkv, D, dtype, rules, monkeypatch):
    """kvm_compress_layers_filled zeroes what lies past the lengths, kvm_compress_layers leaves it, both give the same rows; the
    buffers start as 0xFF bytes, those that compress_layers allocates too."""
    cfg = si.CONFIGS["C1"].scaled(seq=S, head_dim=D, n_q_heads=Hkv, n_kv_heads=Hkv, dtype=dtype, seed=S)
    layers = [tuple(si.make_layer(cfg, l)[k].cuda() for k in "QKV") for l in range(n)]
    p = kvm.make_params(1, Hkv, Hkv, S, D, cfg.torch_dtype, **rules)
    cap = kvm.kvm_sizes(p)[0]
    ws = torch.empty(binding.kvm_layers_workspace_bytes(p, n), dtype=torch.uint8, device="cuda")
    filled, left = (_dirty_outputs(n, Hkv, cap, D, cfg.torch_dtype) for _ in range(2))
    _call_layers("kvm_compress_layers_filled", p, layers, filled, ws)
    _call_layers("kvm_compress_layers", p, layers, left, ws)
    empty = torch.empty
    with monkeypatch.context() as m:
        m.setattr(torch, "empty", lambda *a, **k: empty(*a, **k).view(torch.uint8).fill_(0xFF).view(k["dtype"]))
        out, _ = kvm.compress_layers(p, layers)
    for (ko, vo, ln, pos), (lko, lvo, lln, lpos), c, (Q, K, V) in zip(filled, left, out, layers):
        assert 0 < int(ln.min()) < cap and torch.equal(ln, lln)
        rest = torch.arange(cap, device="cuda") >= ln[..., None]
        for t, u in ((ko, lko), (vo, lvo), (pos, lpos)):
            assert torch.equal(t[~rest], u[~rest])
            assert not t[rest].any() and (u[rest].view(torch.uint8) == 0xFF).all()
        assert all(torch.equal(a, b) for a, b in ((c.K_out, ko), (c.V_out, vo), (c.out_len, ln), (c.out_pos, pos)))
        if n == 2:                                    # (alone: the same bits; its buffers start at zero)
            ref = kvm.Compressor(p)(Q, K, V)
            assert all(torch.equal(getattr(c, k), getattr(ref, k)) for k in ("K_out", "V_out", "out_len", "out_pos"))


@pytest.mark.parametrize("S,Hkv,D,dtype,rules", [
    (700, 2, 64, torch.bfloat16, {"set_rule": kvm.KVM_SETS_CONSERVED_ONLY}),
    (129, 3, 128, torch.float32, {"set_rule": kvm.KVM_SETS_CONSERVED_ONLY}),
    (500, 2, 128, torch.bfloat16, {"weight_rule": kvm.KVM_WEIGHT_PIVOT_ONLY}),
])
def test_gathered_layers_are_zero_past_their_length_without_further_launches(S, Hkv, D, dtype, rules):
    from parity import launched
    p = kvm.make_params(1, Hkv, Hkv, S, D, dtype, **rules)
    # (neighbours alike, so that there are fewer sets than rows)
    layers = [tuple(torch.randn(1, Hkv, S // 8 + 1, D, device="cuda").repeat_interleave(8, 2)[:, :, :S].to(dtype).contiguous()
                    for _ in "QKV") for _ in range(3)]
    cap = kvm.kvm_sizes(p)[0]
    ws = torch.empty(binding.kvm_layers_workspace_bytes(p, 3), dtype=torch.uint8, device="cuda")
    outs = _dirty_outputs(3, Hkv, cap, D, dtype)
    filled = launched(lambda: _call_layers("kvm_compress_layers_filled", p, layers, outs, ws))
    other = _dirty_outputs(3, Hkv, cap, D, dtype)
    assert filled == launched(lambda: _call_layers("kvm_compress_layers", p, layers, other, ws))
    for (ko, vo, n, pos), (Q, K, V) in zip(outs, layers):
        ref = kvm.Compressor(p)(Q, K, V)              # (its buffers start at zero)
        assert int(n.max()) < cap and torch.equal(n, ref.out_len)
        assert torch.equal(ko, ref.K_out) and torch.equal(vo, ref.V_out) and torch.equal(pos, ref.out_pos)


@pytest.mark.parametrize("as_handle", [False, True])
def test_on_a_stream_that_is_not_the_current_one(as_handle):
    """The ratios are read when the kernels are through, the results and the freed workspace belong to the current stream."""
    n, H, S, D = 3, 4, 600, 64
    layers = [tuple(torch.randn(1, H, S // 8, D, device="cuda").repeat_interleave(8, 2).bfloat16() for _ in "QKV") for _ in range(n)]
    p = kvm.make_params(1, H, H, S, D, torch.bfloat16)
    want, ratios = kvm.compress_layers(p, layers)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(50_000_000)                 # (the kernels begin some 25 ms after the call)
    got, got_ratios = kvm.compress_layers(p, layers, stream=s.cuda_stream if as_handle else s)
    scratch = [torch.full((1 << 20,), -1, dtype=torch.int32, device="cuda") for _ in range(16)]      # (the freed workspace's memory, among others)
    assert got_ratios == ratios and s.query()
    for a, b in zip(got, want):
        assert all(torch.equal(getattr(a, k), getattr(b, k)) for k in ("K_out", "V_out", "out_len", "out_pos"))
    del scratch


def test_a_layer_that_is_dropped_is_freed():
    p = kvm.make_params(1, 4, 4, 1024, 128, torch.bfloat16)
    layers = [tuple(torch.randn(1, 4, 1024, 128, device="cuda").bfloat16() for _ in "QKV") for _ in range(4)]
    out, _ = kvm.compress_layers(p, layers)
    size = sum(t.nbytes for t in (out[0].K_out, out[0].V_out, out[0].out_pos))
    kept, before = out[2].K_out.clone(), torch.cuda.memory_allocated()
    del out[0]
    assert before - torch.cuda.memory_allocated() >= size
    assert torch.equal(out[1].K_out, kept)
