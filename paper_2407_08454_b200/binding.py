"""Thin ctypes binding of libkvm.so: argument marshalling only.

Function names and argument order follow include/kvm.h.  Tensors are torch CUDA
tensors (device memory and the current stream come from torch); every step of
the compression path runs inside the library's kernels.  There is no CPU path:
loading fails loudly when the shared library is missing.
"""
from __future__ import annotations

import ctypes
import os
from dataclasses import dataclass
from typing import Optional

import torch

_PKG = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_PKG, "libkvm.so")

KVM_BF16, KVM_F32 = 0, 1
KVM_OK = 0
KVM_PIVOT_MAX_SCORE, KVM_PIVOT_LAST, KVM_PIVOT_KEY = 0, 1, 2
KVM_WEIGHT_GAUSSIAN, KVM_WEIGHT_AVERAGE, KVM_WEIGHT_PIVOT_ONLY, KVM_WEIGHT_SET_SIGMA = 0, 1, 2, 3
KVM_SETS_ADJACENT, KVM_SETS_CONSERVED_ONLY, KVM_SETS_ANCHOR = 0, 1, 2
EXPORTS = (
    "kvm_sizes", "kvm_workspace_bytes", "kvm_score", "kvm_row_lse", "kvm_segment", "kvm_merge_compact", "kvm_compress",
    "kvm_compress_with_lse", "kvm_compress_layers", "kvm_compress_layers_filled", "kvm_layers_workspace_bytes",
    "kvm_host_staging_bytes", "kvm_compress_host", "kvm_score_static", "kvm_layer_ratio", "kvm_attend",
    "kvm_output_perturbation", "kvm_prefill_attend", "kvm_status_string",
    "kvm_version",
)
KVM_STATIC_SCORE_ROWS = 1 << 20


class KvmParams(ctypes.Structure):
    """Mirror of `kvm_params`."""
    _fields_ = [
        ("batch", ctypes.c_int32), ("n_q_heads", ctypes.c_int32), ("n_kv_heads", ctypes.c_int32),
        ("seq", ctypes.c_int32), ("head_dim", ctypes.c_int32), ("dtype", ctypes.c_int32),
        ("budget", ctypes.c_float), ("recent_ratio", ctypes.c_float), ("heavy_ratio", ctypes.c_float),
        ("sim_threshold", ctypes.c_float), ("sigma", ctypes.c_float), ("softmax_scale", ctypes.c_float),
        ("causal", ctypes.c_int32), ("scale_v_by_set_size", ctypes.c_int32), ("enforce_budget", ctypes.c_int32),
        ("pivot_rule", ctypes.c_int32), ("weight_rule", ctypes.c_int32), ("set_rule", ctypes.c_int32),
        ("pivot_key", ctypes.c_void_p),
    ]


class KvmStats(ctypes.Structure):
    """Mirror of `kvm_stats` (24 + 8 bytes)."""
    _fields_ = [
        ("status", ctypes.c_int32), ("units_budget_rule", ctypes.c_int32), ("near_threshold", ctypes.c_int32),
        ("min_out_len", ctypes.c_int32), ("max_out_len", ctypes.c_int32), ("_pad", ctypes.c_int32),
        ("sum_out_len", ctypes.c_int64),
    ]


class KvmError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {status_string(status)} ({status})")


_lib = None
_F = {}          # entry points of the loaded library, argument types declared

_P, _I, _Z = ctypes.c_void_p, ctypes.c_int32, ctypes.c_size_t
_PARAMS = ctypes.POINTER(KvmParams)
# Argument types as in include/kvm.h: with them declared, pointers pass as plain integers (a ctypes object per argument
# costs more than the call).
_ARGTYPES = {
    "kvm_sizes": (_PARAMS, ctypes.POINTER(_I), ctypes.POINTER(_I), ctypes.POINTER(_I)),
    "kvm_workspace_bytes": (_PARAMS, ctypes.POINTER(_Z)),
    "kvm_host_staging_bytes": (_PARAMS, ctypes.POINTER(_Z)),
    "kvm_score": (_PARAMS, _P, _P, _P, _P, _P, _Z, _P),
    "kvm_row_lse": (_PARAMS, _P, _P, _P, _P, _Z, _P),
    "kvm_score_static": (_PARAMS, _P, _P, _P, _P),
    "kvm_segment": (_PARAMS, _P, _P, _P, _P, _P, _P, _P, _P, _P, _Z, _P),
    "kvm_layer_ratio": (_PARAMS, _P, _P, _P, _P, _Z, _P),
    "kvm_attend": (_PARAMS, _P, _P, _P, _I, _P, _P, _P, _Z, _P),
    "kvm_prefill_attend": (_PARAMS, _P, _P, _P, _P, _P, _P, _P),
    "kvm_output_perturbation": (_PARAMS,) + (_P,) * 11 + (_Z, _P),
    "kvm_merge_compact": (_PARAMS,) + (_P,) * 9 + (_Z, _P),
    "kvm_compress": (_PARAMS,) + (_P,) * 10 + (_Z, _P),
    "kvm_compress_with_lse": (_PARAMS,) + (_P,) * 11 + (_Z, _P),
    "kvm_compress_layers": (_PARAMS, _I) + (_P,) * 10 + (_Z, _P),
    "kvm_compress_layers_filled": (_PARAMS, _I) + (_P,) * 10 + (_Z, _P),
    "kvm_layers_workspace_bytes": (_PARAMS, _I, ctypes.POINTER(_Z)),
    "kvm_compress_host": (_PARAMS,) + (_P,) * 8 + (_Z, _P),
}


def lib() -> ctypes.CDLL:
    """Load libkvm.so (built by paper_2407_08454_b200.build).  Raises if it is absent."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise FileNotFoundError(
                f"{LIB_PATH} is missing: run `python -m paper_2407_08454_b200.build` (needs nvcc). "
                "There is no fallback path.")
        L = ctypes.CDLL(LIB_PATH)
        L.kvm_status_string.restype = ctypes.c_char_p
        L.kvm_status_string.argtypes = [ctypes.c_int]
        for name in EXPORTS:
            getattr(L, name)
        # (a handle of its own: whoever takes lib() declares or converts arguments as they like)
        own = ctypes.CDLL(LIB_PATH)
        for name, types in _ARGTYPES.items():
            fn = getattr(own, name)
            fn.argtypes = types
            _F[name] = fn
        _lib = L
    return _lib


def _call(name: str, p: KvmParams, *args) -> None:
    if _lib is None:
        lib()
    rc = _F[name](p, *args)
    if rc != KVM_OK:
        raise KvmError(rc, name)


def status_string(status: int) -> str:
    return lib().kvm_status_string(int(status)).decode()


def make_params(batch: int, n_q_heads: int, n_kv_heads: int, seq: int, head_dim: int, dtype,
                budget: float = 0.5, recent_ratio: float = -1.0, heavy_ratio: float = -1.0,
                sim_threshold: float = 0.75, sigma: float = 5.0, softmax_scale: float = 0.0, causal: int = 1,
                scale_v_by_set_size: int = 1, enforce_budget: int = 1, pivot_rule: int = 0, weight_rule: int = 0,
                set_rule: int = 0, pivot_key: Optional[torch.Tensor] = None) -> KvmParams:
    """`pivot_key` ([batch, n_kv_heads, seq] fp32 CUDA tensor) must stay alive while the parameters are in use."""
    if isinstance(dtype, torch.dtype):
        dtype = {torch.bfloat16: KVM_BF16, torch.float32: KVM_F32}[dtype]
    key_ptr = None
    if pivot_key is not None:
        assert pivot_key.is_cuda and pivot_key.dtype == torch.float32 and pivot_key.is_contiguous()
        assert tuple(pivot_key.shape) == (batch, n_kv_heads, seq)
        key_ptr = pivot_key.data_ptr()
    return KvmParams(batch, n_q_heads, n_kv_heads, seq, head_dim, int(dtype), budget, recent_ratio, heavy_ratio,
                     sim_threshold, sigma, softmax_scale, causal, scale_v_by_set_size, enforce_budget,
                     pivot_rule, weight_rule, set_rule, key_ptr)


def _ptr(t: Optional[torch.Tensor]) -> Optional[int]:
    if t is None:
        return None
    assert t.is_contiguous(), "tensors must be contiguous"
    return t.data_ptr()


# The current stream's handle without the Stream object around it.
_device, _raw_stream = torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream


def _stream(stream) -> int:
    if stream is None:
        if not torch.cuda.is_initialized():
            torch.cuda.init()
        return _raw_stream(_device())
    return stream.cuda_stream if hasattr(stream, "cuda_stream") else int(stream)


def kvm_version() -> int:
    return int(lib().kvm_version())


def kvm_sizes(p: KvmParams):
    cap, nr, nh = ctypes.c_int32(), ctypes.c_int32(), ctypes.c_int32()
    _call("kvm_sizes", p, cap, nr, nh)
    return cap.value, nr.value, nh.value


def kvm_workspace_bytes(p: KvmParams) -> int:
    n = ctypes.c_size_t()
    _call("kvm_workspace_bytes", p, n)
    return n.value


def kvm_layers_workspace_bytes(p: KvmParams, n_layers: int) -> int:
    n = ctypes.c_size_t()
    _call("kvm_layers_workspace_bytes", p, n_layers, n)
    return n.value


def kvm_host_staging_bytes(p: KvmParams) -> int:
    n = ctypes.c_size_t()
    _call("kvm_host_staging_bytes", p, n)
    return n.value


def kvm_score(p: KvmParams, Q, K, lse_in, scores, ws, stream=None) -> None:
    _call("kvm_score", p, _ptr(Q), _ptr(K), _ptr(lse_in), _ptr(scores), _ptr(ws), ws.nbytes, _stream(stream))


def kvm_row_lse(p: KvmParams, Q, K, lse_out, ws, stream=None) -> None:
    _call("kvm_row_lse", p, _ptr(Q), _ptr(K), _ptr(lse_out), _ptr(ws), ws.nbytes, _stream(stream))


def kvm_score_static(p: KvmParams, Q, K, scores, stream=None) -> None:
    """kvm_score on the library's built-in scratch: for callers that cannot allocate a workspace.
    batch * n_q_heads * seq must not exceed KVM_STATIC_SCORE_ROWS (fp32) or an eighth of it (bf16); calls on one
    device must not overlap."""
    _call("kvm_score_static", p, _ptr(Q), _ptr(K), _ptr(scores), _stream(stream))


def kvm_segment(p: KvmParams, K, scores, set_id, set_start, pivot, out_len, sim_out, stats, ws, stream=None) -> None:
    _call("kvm_segment", p, _ptr(K), _ptr(scores), _ptr(set_id), _ptr(set_start), _ptr(pivot), _ptr(out_len),
          _ptr(sim_out), _ptr(stats), _ptr(ws), ws.nbytes, _stream(stream))


def kvm_layer_ratio(p: KvmParams, K, ratio, sim_out, ws, stream=None) -> None:
    _call("kvm_layer_ratio", p, _ptr(K), _ptr(ratio), _ptr(sim_out), _ptr(ws), ws.nbytes, _stream(stream))


def kvm_attend(p: KvmParams, q, K, V, rows: int, length, out, ws, stream=None) -> None:
    _call("kvm_attend", p, _ptr(q), _ptr(K), _ptr(V), rows, _ptr(length), _ptr(out), _ptr(ws), ws.nbytes,
          _stream(stream))


def kvm_prefill_attend(p: KvmParams, Q, K, V, O, lse, stats=None, stream=None) -> None:
    """Causal attention over the whole prompt: O [B,Hq,S,D] bf16 and the rows' natural-log log-sum-exp [B,Hq,S]."""
    _call("kvm_prefill_attend", p, _ptr(Q), _ptr(K), _ptr(V), _ptr(O), _ptr(lse), _ptr(stats), _stream(stream))


def kvm_output_perturbation(p: KvmParams, q, K, V, K_c, V_c, len_c, out_full, out_comp, err, ref, ws,
                            stream=None) -> None:
    _call("kvm_output_perturbation", p, _ptr(q), _ptr(K), _ptr(V), _ptr(K_c), _ptr(V_c), _ptr(len_c), _ptr(out_full),
          _ptr(out_comp), _ptr(err), _ptr(ref), _ptr(ws), ws.nbytes, _stream(stream))


def kvm_merge_compact(p: KvmParams, K, V, set_start, pivot, out_len, K_out, V_out, out_size, ws, stream=None) -> None:
    _call("kvm_merge_compact", p, _ptr(K), _ptr(V), _ptr(set_start), _ptr(pivot), _ptr(out_len), _ptr(K_out),
          _ptr(V_out), _ptr(out_size), _ptr(ws), ws.nbytes, _stream(stream))


def kvm_compress(p: KvmParams, Q, K, V, K_out, V_out, out_len, out_pos, scores_out, stats, ws, stream=None) -> None:
    _call("kvm_compress", p, _ptr(Q), _ptr(K), _ptr(V), _ptr(K_out), _ptr(V_out), _ptr(out_len), _ptr(out_pos),
          _ptr(scores_out), _ptr(stats), _ptr(ws), ws.nbytes, _stream(stream))


def kvm_compress_with_lse(p: KvmParams, Q, K, V, lse_in, K_out, V_out, out_len, out_pos, scores_out, stats, ws,
                          stream=None) -> None:
    _call("kvm_compress_with_lse", p, _ptr(Q), _ptr(K), _ptr(V), _ptr(lse_in), _ptr(K_out), _ptr(V_out),
          _ptr(out_len), _ptr(out_pos), _ptr(scores_out), _ptr(stats), _ptr(ws), ws.nbytes, _stream(stream))


def kvm_compress_host(p: KvmParams, Q, K, V, K_out, V_out, out_len, out_pos, dev, stream=None) -> None:
    """Q..out_pos are HOST tensors (pin them for asynchronous copies); `dev` is a device byte buffer."""
    _call("kvm_compress_host", p, _ptr(Q), _ptr(K), _ptr(V), _ptr(K_out), _ptr(V_out), _ptr(out_len), _ptr(out_pos),
          _ptr(dev), dev.nbytes, _stream(stream))


# ----------------------------------------------------------------------------- convenience
def new_stats(device) -> torch.Tensor:
    """Zeroed device buffer laid out as `kvm_stats`."""
    return torch.zeros(ctypes.sizeof(KvmStats), dtype=torch.uint8, device=device)


def read_stats(buf: torch.Tensor) -> KvmStats:
    return KvmStats.from_buffer_copy(bytes(buf.cpu().numpy().tobytes()))


@dataclass
class Compressed:
    K_out: torch.Tensor
    V_out: torch.Tensor
    out_len: torch.Tensor
    out_pos: torch.Tensor
    scores: Optional[torch.Tensor]
    cap: int


class Compressor:
    """Owns the workspace and output buffers for one problem shape and calls kvm_compress."""

    def __init__(self, p: KvmParams, device="cuda", want_scores: bool = False):
        self.p = p
        self.cap, self.n_recent, self.n_heavy = kvm_sizes(p)
        U = p.batch * p.n_kv_heads
        dt = torch.bfloat16 if p.dtype == KVM_BF16 else torch.float32
        self.ws = torch.empty(kvm_workspace_bytes(p), dtype=torch.uint8, device=device)
        self.K_out = torch.zeros(p.batch, p.n_kv_heads, self.cap, p.head_dim, dtype=dt, device=device)
        self.V_out = torch.zeros_like(self.K_out)
        self.out_len = torch.zeros(U, dtype=torch.int32, device=device).view(p.batch, p.n_kv_heads)
        self.out_pos = torch.zeros(p.batch, p.n_kv_heads, self.cap, dtype=torch.int32, device=device)
        self.scores = (torch.empty(p.batch, p.n_kv_heads, p.seq, dtype=torch.float32, device=device)
                       if want_scores else None)

    def __call__(self, Q, K, V, stats=None, stream=None) -> Compressed:
        kvm_compress(self.p, Q, K, V, self.K_out, self.V_out, self.out_len, self.out_pos, self.scores, stats,
                     self.ws, stream)
        return Compressed(self.K_out, self.V_out, self.out_len, self.out_pos, self.scores, self.cap)


def compress_layers(p: KvmParams, layers, sim_thresholds=None, device="cuda", stream=None):
    """Compress a stack of layers, each an (Q, K, V) triple of CUDA tensors of the shape `p` describes, with one
    similarity threshold per layer (Section 3.2: thresholds chosen layer by layer), through kvm_compress_layers_filled.
    Returns, per layer, a `Compressed` holding the outputs, and the layer's compression ratio mean(out_len) / S.
    `stream`: the one the kernels run on, after what the current stream has been given so far; the results are there when
    the function returns."""
    # (the GPU waits for this function: whatever its results do not need is left until the kernels are enqueued, and the
    # addresses are worked out from the bases)
    n = len(layers)
    B, H, cap, D = p.batch, p.n_kv_heads, kvm_sizes(p)[0], p.head_dim
    units, dtype = B * H, torch.bfloat16 if p.dtype == KVM_BF16 else torch.float32
    # A layer's rows and positions are one allocation (a layer that the caller drops is freed); what lies past the lengths is
    # zeroed by the merge; the lengths of all layers are read back together.
    kv_bytes = units * cap * D * (2 if p.dtype == KVM_BF16 else 4)
    blobs = [torch.empty(2 * kv_bytes + 4 * units * cap, dtype=torch.uint8, device=device) for _ in range(n)]
    out_len = torch.empty((n, B, H), dtype=torch.int32, device=device)
    ws = torch.empty(kvm_layers_workspace_bytes(p, n), dtype=torch.uint8, device=device)
    array = ctypes.c_void_p * n

    for layer in layers:
        assert len(layer) == 3 and all([t.is_contiguous() for t in layer]), "tensors must be contiguous"
    q, k, v = (array(*[layer[i].data_ptr() for layer in layers]) for i in range(3))
    eps = None
    if sim_thresholds is not None:
        assert len(sim_thresholds) == n
        eps = (ctypes.c_float * n)(*[float(e) for e in sim_thresholds])
    bases, len_base = [b.data_ptr() for b in blobs], out_len.data_ptr()
    handle, other = _stream(stream), None
    if stream is not None and handle != _stream(None):
        # (the buffers are the current stream's: what it last did with their memory comes before the kernels, and the
        # workspace is not handed out again before they are through)
        other = torch.cuda.ExternalStream(handle, device=out_len.device)
        other.wait_stream(torch.cuda.current_stream(out_len.device))
        for t in (*blobs, out_len, ws):
            t.record_stream(other)
    _call("kvm_compress_layers_filled", p, n, eps, q, k, v, array(*bases), array(*[b + kv_bytes for b in bases]),
          array(*range(len_base, len_base + 4 * n * units, 4 * units)), array(*[b + 2 * kv_bytes for b in bases]), None,
          ws.data_ptr(), ws.nbytes, handle)
    out = []
    for blob, lengths in zip(blobs, out_len.unbind(0)):
        K_out, V_out = blob[:2 * kv_bytes].view(dtype).view(2, B, H, cap, D).unbind(0)
        out.append(Compressed(K_out, V_out, lengths, blob[2 * kv_bytes:].view(torch.int32).view(B, H, cap), None, cap))
    if other is not None:
        other.synchronize()
    ratios = (out_len.cpu().float().mean((1, 2)) / p.seq).tolist()      # the one read-back of the call
    return out, ratios
