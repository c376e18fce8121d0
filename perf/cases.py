"""The work that users of this package have it do, as measurable cases.

A case is a dict of plain values.  `listed()` gives the standing ones, `draw(rng)` one more of the same ranges,
`prepare(case, seed)` makes what a program holds before the call, `run(state)` is one pass through the public entry
points, `work(case)` the bytes and operations the pass cannot do without, and `tolerance(case)` how far another correct
implementation at the same precision may be off.

Five operations:

  compress  one layer's cache is compressed after its prefill (`Compressor`, i.e. kvm_compress): scores, merging sets,
            pivots, weighted merge
  prefill   the prefill attention of a layer followed by the compression that reuses its row log-sum-exp
            (kvm_prefill_attend, kvm_compress_with_lse)
  decode    one decode step of attention over a compressed cache whose units hold different numbers of rows (kvm_attend)
  layers    a stack of layers with one similarity threshold each (`compress_layers`)
  host      a layer whose tensors live in pinned host memory (kvm_compress_host)
"""
import math

import torch

import paper_2407_08454_b200 as kvm

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
RULES = {
    "merge": {},                                                                        # the method itself
    "average": {"weight_rule": kvm.KVM_WEIGHT_AVERAGE, "pivot_rule": kvm.KVM_PIVOT_LAST},  # average-weighted merging
    "evict": {"set_rule": kvm.KVM_SETS_CONSERVED_ONLY},                                 # conserved tokens only
}


def _case(op, batch, n_q_heads, n_kv_heads, seq, head_dim, dtype="bf16", budget=0.5, rule="merge", restart=0.0,
          layers=1, **name):
    return {**name, "op": op, "batch": batch, "n_q_heads": n_q_heads, "n_kv_heads": n_kv_heads, "seq": seq,
            "head_dim": head_dim, "dtype": dtype, "budget": budget, "rule": rule, "restart": restart, "layers": layers}


def listed():
    return [
        # the smallest layer in use, in fp32: launches and host work
        _case("compress", 1, 4, 4, 512, 64, dtype="f32", name="compress-tiny-f32"),
        # an fp32 layer of ordinary size, grouped queries, a length that no tile divides
        _case("compress", 1, 16, 8, 2999, 128, dtype="f32", name="compress-f32-ragged"),
        # a short prompt on a Llama2-7B-shaped layer
        _case("compress", 1, 32, 32, 389, 128, name="compress-short"),
        # the headline workload: one Llama2-7B-shaped layer, 4k tokens, 50 % budget
        _case("compress", 1, 32, 32, 4096, 128, name="compress-7b-4k"),
        # the same layer for four sequences at the 35 % budget
        _case("compress", 4, 32, 32, 4096, 128, budget=0.35, name="compress-7b-batch"),
        # a Mistral-7B-shaped layer with a 32k-token prompt: the largest
        _case("compress", 1, 32, 8, 32768, 128, name="compress-gqa-32k"),
        # the production path: attention of the prefill, then the compression fed by it
        _case("prefill", 1, 32, 32, 4096, 128, name="prefill-7b-4k"),
        # the same with head dimension 64, grouped queries and a ragged length, 35 % budget
        _case("prefill", 1, 32, 8, 10007, 64, budget=0.35, name="prefill-gqa-d64-ragged"),
        # one decode step over one sequence's compressed cache: latency
        _case("decode", 1, 32, 32, 4096, 128, name="decode-7b-4k"),
        # a decode step of a serving batch with grouped queries and long caches: bandwidth
        _case("decode", 8, 32, 8, 32768, 128, name="decode-gqa-batch"),
        # a stack of layers, thresholds chosen layer by layer, keys with many short runs
        _case("layers", 1, 32, 8, 2048, 128, restart=1.0 / 64.0, layers=8, name="layers-gqa-2k"),
        # the headline layer from and to host memory
        _case("host", 1, 32, 32, 4096, 128, name="host-7b-4k"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    op = rng.choices(["compress", "prefill", "decode", "layers", "host"], [9, 3, 4, 2, 2])[0]
    dtype = "f32" if op in ("compress", "decode") and rng.random() < 0.25 else "bf16"
    budget = rng.choice([0.5, 0.35])
    rule = rng.choices(["merge", "average", "evict"], [6, 1, 1])[0] if op == "compress" else "merge"
    restart = rng.choice([0.0, 0.0, 1.0 / 64.0])
    while True:
        batch = _log_int(rng, 1, 8)
        n_kv_heads, group = _log_int(rng, 1, 40), rng.choice([1, 1, 2, 4, 8])
        seq = _log_int(rng, 256, 4096 if dtype == "f32" and op == "compress" else 32768)
        layers = rng.randint(2, 8) if op == "layers" else 1
        rows = batch * n_kv_heads * seq * layers           # key rows; `group` times as many query rows
        if n_kv_heads * group > 64 or rows * group > 1 << 20:
            continue
        pairs = rows * group * seq                         # logits (twice the causal half), by the cost of one each
        if op == "decode" or pairs * (16 if dtype == "f32" else 2 if op == "prefill" else 1) <= 32 * 32768 ** 2:
            break
    return _case(op, batch, n_kv_heads * group, n_kv_heads, seq, rng.choice([64, 128, 128]), dtype=dtype,
                 budget=budget, rule=rule, restart=restart, layers=layers)


def _params(case):
    return kvm.make_params(case["batch"], case["n_q_heads"], case["n_kv_heads"], case["seq"], case["head_dim"],
                           DTYPES[case["dtype"]], budget=case["budget"], **RULES[case["rule"]])


def _ar1(g, shape, rho, restart):
    """AR(1) over the token axis (dim 2), unit variance per channel; restarts from N(0,1) with probability `restart`."""
    B, H, S, _ = shape
    x = torch.randn(shape, generator=g, device="cuda")
    a = torch.full((B, H, S, 1), rho, device="cuda")
    if restart > 0.0:
        a[torch.rand((B, H, S, 1), generator=g, device="cuda") < restart] = 0.0
    a[:, :, 0] = 0.0
    x *= (1.0 - a * a).sqrt()
    k = 1
    while k < S and rho ** k > 1e-7:           # x_t = a_t x_{t-1} + u_t by doubling
        x[:, :, k:] = torch.addcmul(x[:, :, k:], a[:, :, k:], x[:, :, :-k])
        a[:, :, k:] = a[:, :, k:] * a[:, :, :-k]
        a[:, :, :k] = 0.0
        k *= 2
    return x


def _keys_and_scales(case, g, S):
    """Keys as real prefill caches show them: neighbours similar, channels of unequal scale, two outlier channels."""
    B, Hkv, D = case["batch"], case["n_kv_heads"], case["head_dim"]
    rho = 0.85 + 0.13 * torch.rand((), generator=g, device="cuda").item() if case["budget"] < 0.425 else 0.95
    s = torch.exp(0.5 * torch.randn((1, Hkv, 1, D), generator=g, device="cuda"))
    out = torch.rand((1, Hkv, 1, D), generator=g, device="cuda").topk(2).indices
    gain = torch.ones_like(s).scatter_(-1, out, 10.0)
    s = s * gain
    return (_ar1(g, (B, Hkv, S, D), rho, case["restart"]) * s).to(DTYPES[case["dtype"]]), s, gain, rho


def _queries(case, g, S, sk, gain, rho):
    """Queries on the same outlier channels, scaled per head so that the logits have standard deviation 4."""
    B, Hq, D = case["batch"], case["n_q_heads"], case["head_dim"]
    G = Hq // case["n_kv_heads"]
    sq = torch.exp(0.5 * torch.randn((1, Hq, 1, D), generator=g, device="cuda")) * gain.repeat_interleave(G, 1)
    sq = sq * (4.0 * math.sqrt(D) / (sq * sk.repeat_interleave(G, 1)).square().sum(-1, keepdim=True).sqrt())
    return (_ar1(g, (B, Hq, S, D), rho, 0.0) * sq).to(DTYPES[case["dtype"]])


def _layer(case, g):
    K, sk, gain, rho = _keys_and_scales(case, g, case["seq"])
    Q = _queries(case, g, case["seq"], sk, gain, rho)
    V = torch.randn(K.shape, generator=g, device="cuda").to(K.dtype)
    return Q, K, V


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    op, p = case["op"], _params(case)
    st = {"op": op, "p": p}
    if op == "decode":
        cap = kvm.kvm_sizes(p)[0]
        K, sk, gain, rho = _keys_and_scales(case, g, cap)
        st.update(K=K, V=torch.randn(K.shape, generator=g, device="cuda").to(K.dtype), rows=cap)
        st["q"] = _queries(case, g, 1, sk, gain, rho).squeeze(2).contiguous()
        st["len"] = torch.randint(cap // 2, cap + 1, K.shape[:2], generator=g, device="cuda", dtype=torch.int32)
        st["out"] = torch.empty(st["q"].shape, dtype=torch.float32, device="cuda")
        st["ws"] = torch.empty(kvm.kvm_workspace_bytes(p), dtype=torch.uint8, device="cuda")
        return st
    if op == "layers":
        st["layers"] = [_layer(case, g) for _ in range(case["layers"])]
        st["eps"] = (0.6 + 0.3 * torch.rand(case["layers"], generator=g, device="cuda")).tolist()
        return st
    Q, K, V = _layer(case, g)
    if op == "host":
        cap = kvm.kvm_sizes(p)[0]
        st.update(Q=Q.cpu().pin_memory(), K=K.cpu().pin_memory(), V=V.cpu().pin_memory())
        st["K_out"] = torch.zeros(K.shape[0], K.shape[1], cap, K.shape[3], dtype=K.dtype).pin_memory()
        st["V_out"] = torch.zeros_like(st["K_out"]).pin_memory()
        st["out_len"] = torch.zeros(K.shape[:2], dtype=torch.int32).pin_memory()
        st["out_pos"] = torch.zeros(K.shape[0], K.shape[1], cap, dtype=torch.int32).pin_memory()
        # (rows past a unit's length are copied out as the staging buffer holds them: zeros here)
        st["dev"] = torch.zeros(kvm.kvm_host_staging_bytes(p), dtype=torch.uint8, device="cuda")
        return st
    st.update(Q=Q, K=K, V=V, comp=kvm.Compressor(p))
    if op == "prefill":
        st["O"] = torch.empty_like(Q)
        st["lse"] = torch.empty(Q.shape[:3], dtype=torch.float32, device="cuda")
    return st


def _outputs(c):
    return {"K_out": c.K_out, "V_out": c.V_out, "out_len": c.out_len, "out_pos": c.out_pos}


def run(st):
    op, p = st["op"], st["p"]
    if op == "compress":
        return _outputs(st["comp"](st["Q"], st["K"], st["V"]))
    if op == "prefill":
        c = st["comp"]
        kvm.kvm_prefill_attend(p, st["Q"], st["K"], st["V"], st["O"], st["lse"])
        kvm.kvm_compress_with_lse(p, st["Q"], st["K"], st["V"], st["lse"], c.K_out, c.V_out, c.out_len, c.out_pos,
                                  None, None, c.ws)
        return {"O": st["O"], "lse": st["lse"], **_outputs(c)}
    if op == "decode":
        kvm.kvm_attend(p, st["q"], st["K"], st["V"], st["rows"], st["len"], st["out"], st["ws"])
        return st["out"]
    if op == "layers":
        out, ratios = kvm.compress_layers(p, st["layers"], st["eps"])
        return {"layers": [_outputs(c) for c in out], "ratios": ratios}
    kvm.kvm_compress_host(p, st["Q"], st["K"], st["V"], st["K_out"], st["V_out"], st["out_len"], st["out_pos"],
                          st["dev"])
    torch.cuda.current_stream().synchronize()      # the results are in host memory: the caller reads them next
    return {k: st[k] for k in ("K_out", "V_out", "out_len", "out_pos")}


def work(case):
    B, Hq, Hkv, S, D = (case[k] for k in ("batch", "n_q_heads", "n_kv_heads", "seq", "head_dim"))
    e = 2 if case["dtype"] == "bf16" else 4
    cap, n_recent, n_heavy = kvm.kvm_sizes(_params(case))
    if case["op"] == "decode":
        rows = B * Hkv * 0.75 * cap                # lengths are uniform over the upper half of the capacity
        return {"bytes": rows * 2 * D * e + B * Hq * D * (e + 4), "flops": 4.0 * D * rows * (Hq // Hkv)}
    product = 2.0 * D * B * Hq * S * (S + 1) / 2   # the causal half of Q K^T
    # Q, K, V in; at least the conserved rows of K and V, and their positions, out
    moved = (B * Hq * S * D + 2 * B * Hkv * S * D + 2 * B * Hkv * (n_recent + n_heavy) * D) * e
    moved += 4 * B * Hkv * (n_recent + n_heavy)
    products = 2                                   # the row log-sum-exp, then the column sums
    if case["op"] == "prefill":
        products = 3                               # attention's two, then the column sums
        moved += B * Hq * S * (D * e + 4)
    return {"bytes": float(moved * case["layers"]), "flops": product * products * case["layers"]}


def tolerance(case):
    if case["op"] == "decode":
        return {"rel": 2e-5}                       # fp32 arithmetic on the stored values
    # merged rows: one rounding to the storage type; positions and lengths: scores that tie to fp32 rounding
    return {"rel": 1e-2 if case["dtype"] == "bf16" else 1e-5, "differ": 2e-3}
