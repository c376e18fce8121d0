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
        # together the column sums may be added in other pieces: scores that tie to fp32 rounding may change places
        assert torch.equal(together[l].out_len, ref.out_len) or (together[l].out_len - ref.out_len).abs().max() <= 2
        same = (together[l].out_pos == ref.out_pos).float().mean().item()
        assert same >= 0.99
        if torch.equal(together[l].out_pos, ref.out_pos):
            assert torch.equal(together[l].K_out, ref.K_out) and torch.equal(together[l].V_out, ref.V_out)


def test_a_layer_that_is_dropped_is_freed():
    p = kvm.make_params(1, 4, 4, 1024, 128, torch.bfloat16)
    layers = [tuple(torch.randn(1, 4, 1024, 128, device="cuda").bfloat16() for _ in "QKV") for _ in range(4)]
    out, _ = kvm.compress_layers(p, layers)
    size = sum(t.nbytes for t in (out[0].K_out, out[0].V_out, out[0].out_pos))
    kept, before = out[2].K_out.clone(), torch.cuda.memory_allocated()
    del out[0]
    assert before - torch.cuda.memory_allocated() >= size
    assert torch.equal(out[1].K_out, kept)
