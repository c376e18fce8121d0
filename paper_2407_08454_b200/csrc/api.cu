// C ABI of the kvm library: host-side validation, workspace carving, dispatch.
// All checks run before anything is enqueued; nothing here allocates device memory or synchronises.
#include <math.h>
#include <string.h>

#include <mutex>

#include "score_plan.cuh"

namespace kvm {
namespace {

inline size_t align_up(size_t x, size_t a = 256) { return (x + a - 1) / a * a; }

int derive(const kvm_params* p, Dims& d) {
    if (!p) return KVM_E_NULL;
    if (p->dtype != KVM_BF16 && p->dtype != KVM_F32) return KVM_E_DTYPE;
    if (p->batch < 1 || p->n_q_heads < 1 || p->n_kv_heads < 1 || p->seq < 1) return KVM_E_SHAPE;
    if (p->n_q_heads % p->n_kv_heads != 0) return KVM_E_SHAPE;
    if (p->head_dim != 64 && p->head_dim != 128) return KVM_E_SHAPE;
    if (p->seq > KVM_MAX_SEQ) return KVM_E_SHAPE;
    if ((long long)p->batch * p->n_q_heads > 65535) return KVM_E_SHAPE;
    if (!(p->budget > 0.f && p->budget <= 1.f)) return KVM_E_PARAM;
    if (!isfinite(p->sim_threshold)) return KVM_E_PARAM;
    if (!isfinite(p->softmax_scale)) return KVM_E_PARAM;
    if (p->causal != 1) return KVM_E_UNSUPPORTED;
    const bool half_budget = p->budget >= 0.425f;
    const float recent = p->recent_ratio < 0.f ? (half_budget ? 0.17f : 0.08f) : p->recent_ratio;
    const float heavy = p->heavy_ratio < 0.f ? (half_budget ? 0.12f : 0.02f) : p->heavy_ratio;
    if (!(recent >= 0.f && recent <= 1.f) || !(heavy >= 0.f && heavy <= 1.f)) return KVM_E_PARAM;
    d.B = p->batch; d.Hq = p->n_q_heads; d.Hkv = p->n_kv_heads; d.G = d.Hq / d.Hkv;
    d.S = p->seq; d.D = p->head_dim; d.U = d.B * d.Hkv; d.dtype = p->dtype;
    const int C = (int)floor((double)p->budget * (double)d.S);
    d.n_r = (int)floor((double)recent * (double)d.S);
    d.n_h = (int)floor((double)heavy * (double)d.S);
    d.enforce = p->enforce_budget ? 1 : 0;
    d.cap = d.enforce ? C : d.S;
    if (p->pivot_rule < KVM_PIVOT_MAX_SCORE || p->pivot_rule > KVM_PIVOT_KEY) return KVM_E_PARAM;
    if (p->weight_rule < KVM_WEIGHT_GAUSSIAN || p->weight_rule > KVM_WEIGHT_SET_SIGMA) return KVM_E_PARAM;
    if (p->set_rule < KVM_SETS_ADJACENT || p->set_rule > KVM_SETS_ANCHOR) return KVM_E_PARAM;
    if (p->set_rule == KVM_SETS_ANCHOR && (p->enforce_budget || p->seq > KVM_ANCHOR_MAX_SEQ)) return KVM_E_UNSUPPORTED;
    d.pivot_rule = p->pivot_rule; d.weight_rule = p->weight_rule; d.set_rule = p->set_rule;
    d.pivot_key = p->pivot_key;
    if (p->set_rule != KVM_SETS_CONSERVED_ONLY && p->weight_rule == KVM_WEIGHT_GAUSSIAN &&
        (!(p->sigma > 0.f) || !isfinite(p->sigma)))
        return KVM_E_PARAM;
    if (d.set_rule == KVM_SETS_CONSERVED_ONLY) {
        d.pivot_rule = KVM_PIVOT_MAX_SCORE; d.weight_rule = KVM_WEIGHT_PIVOT_ONLY; d.pivot_key = nullptr;
        if ((long long)d.cap < (long long)d.n_r + d.n_h) return KVM_E_PARAM;   // the kept tokens must fit
    } else {
        if (d.pivot_rule == KVM_PIVOT_KEY && !d.pivot_key) return KVM_E_NULL;
        // (pivot_key is read with scalar loads: no alignment beyond a float's is asked of it)
        if (d.pivot_rule == KVM_PIVOT_KEY && ((uintptr_t)d.pivot_key & 3u)) return KVM_E_ALIGN;
        // the forced cuts alone (first token, recent window, each heavy hitter and its right neighbour) must fit
        if (d.enforce && (long long)d.cap < 1LL + d.n_r + 2LL * d.n_h) return KVM_E_PARAM;
    }
    if (d.cap < 1) return KVM_E_PARAM;
    d.scale = p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf((float)d.D);
    d.eps = p->sim_threshold;
    d.sigma = p->sigma;
    d.scale_v = p->scale_v_by_set_size ? 1 : 0;
    return KVM_OK;
}

// scratch of the score step: the bf16 path's side tensor, and what cut items leave (row states, partial column sums)
inline size_t score_bytes(const Dims& d) {
    return d.dtype == KVM_BF16 ? score_tc_scratch_bytes(d) : score_f32_scratch_bytes(d);
}

struct Workspace {
    float* lse;         // score scratch
    float* scores;      // [U,S]
    float* sim;         // [U,S]
    int32_t* set_start; // [U,cap+1]
    int32_t* set_id;    // [U,S]
    float* merge_part;  // partial sums of sets that cross token tiles
    float* attend_part; // per-chunk online-softmax states of the decode-step attention
    size_t bytes;
};

Workspace carve(const Dims& d, void* base) {
    Workspace w;
    size_t off = 0;
    auto take = [&](size_t n) { size_t o = off; off += align_up(n); return (char*)base + o; };
    w.lse = (float*)take(score_bytes(d));
    w.scores = (float*)take((size_t)d.U * d.S * sizeof(float));
    w.sim = (float*)take((size_t)d.U * d.S * sizeof(float));
    w.set_start = (int32_t*)take((size_t)d.U * (d.cap + 1) * sizeof(int32_t));
    w.set_id = (int32_t*)take((size_t)d.U * d.S * sizeof(int32_t));
    w.merge_part = (float*)take(merge_scratch_floats(d) * sizeof(float));
    w.attend_part = (float*)take(attend_scratch_floats(d) * sizeof(float));
    w.bytes = off;
    return w;
}

inline bool misaligned(const void* p) { return ((uintptr_t)p & 15u) != 0; }

int check_ws(const Dims& d, void* ws, size_t ws_bytes, Workspace& w) {
    if (!ws) return KVM_E_WORKSPACE;
    if (misaligned(ws)) return KVM_E_ALIGN;
    w = carve(d, ws);
    if (ws_bytes < w.bytes) return KVM_E_WORKSPACE;
    return KVM_OK;
}

// One layer's tensors as the kernels take them.
Layers one_layer(const Dims& d, const void* Q, const void* K, const void* V = nullptr, void* K_out = nullptr,
                 void* V_out = nullptr, int32_t* out_len = nullptr, int32_t* pivot = nullptr) {
    Layers L = {};
    L.n = 1; L.U = d.U; L.H = d.B * d.Hq;
    L.Q[0] = Q; L.K[0] = K; L.V[0] = V; L.K_out[0] = K_out; L.V_out[0] = V_out;
    L.out_len[0] = out_len; L.pivot[0] = pivot; L.eps[0] = d.eps;
    return L;
}

// sim_out (nullable): where the neighbour-key similarities are wanted, which the score step produces on the side.
cudaError_t run_score(const Dims& d, const Layers& L, const float* lse_in, float* scores, const Workspace& w,
                      kvm_stats* stats, cudaStream_t st, float* sim_out = nullptr, ScorePart* parts = nullptr) {
    // fp32 tensors enter the tensor cores as exact sums of three bf16 planes: rounding them would not hold the
    // score tolerance
    return d.dtype == KVM_BF16 ? launch_score_tc(d, L, lse_in, w.lse, scores, stats, st, sim_out, nullptr, parts)
                               : launch_score_f32(d, L.Q[0], L.K[0], lse_in, w.lse, scores, stats, st, sim_out, nullptr, parts);
}

// The whole chain over the layers in L (d: the layers together, a batch of n times a layer's).
int run_chain(const Dims& d, const Layers& L, const float* lse_in, float* scores, const Workspace& w, kvm_stats* stats,
              cudaStream_t st) {
    const bool want_sim = d.set_rule == KVM_SETS_ADJACENT;
    ScorePart parts;
    if (run_score(d, L, lse_in, scores, w, stats, st, want_sim ? w.sim : nullptr, &parts) != cudaSuccess) return KVM_E_CUDA;
    if (d.set_rule == KVM_SETS_ANCHOR)
        if (launch_anchor_runs(d, L.K[0], w.sim, (float*)w.set_id, st) != cudaSuccess) return KVM_E_CUDA;
    if (launch_segment(d, L, scores, parts, w.sim, w.set_id, w.set_start, stats, st) != cudaSuccess) return KVM_E_CUDA;
    const cudaError_t e =
        d.weight_rule == KVM_WEIGHT_PIVOT_ONLY
            ? launch_gather(d, L.K[0], L.V[0], w.set_start, L.pivot[0], L.out_len[0], L.K_out[0], L.V_out[0], nullptr, L.zero_rest ? L.pivot[0] : nullptr, st)
            : launch_merge(d, L, w.set_start, w.set_id, nullptr, w.merge_part, w.sim, w.scores, stats, st);
    return e == cudaSuccess ? KVM_OK : KVM_E_CUDA;
}

// How many layers of a stack go through the kernels together.  A layer whose score pass gives a CTA few steps loses most
// of its time to the launches, the passes' start and drain and the last, half-empty round (32 query / 8 KV heads x 2048
// tokens, about 30 steps per CTA: 78 us a layer); together the layers share them.  As many go together as give a CTA about
// 300 steps (us a layer of 8, alone / together: 3 steps 31.9 / 12.8, 8 42.5 / 25.9 and 38.7 / 16.0, 30 71.0 / 47.1, 46 96 / 73,
// 65 124 / 99; what is shared, about 25 us, stays the same while the rest grows).  The variants beside the method, and fp32
// tensors, run layer by layer.
int layers_together(const Dims& d, int n_layers) {
    if (d.dtype != KVM_BF16 || d.set_rule != KVM_SETS_ADJACENT ||
        (d.weight_rule != KVM_WEIGHT_GAUSSIAN && d.weight_rule != KVM_WEIGHT_AVERAGE))
        return 1;
    const long long T = (d.S + 127) / 128, steps = (long long)d.B * d.Hq * T * (T + 1) / 2 / 148 + 1;
    long long n = 300 / steps;
    if (n > (long long)(65535 / (d.B * d.Hq))) n = 65535 / (d.B * d.Hq);      // (grid dimensions)
    if (n > n_layers) n = n_layers;
    return (int)(n < 1 ? 1 : n > MAX_LAYERS ? MAX_LAYERS : n);
}
Dims times_batch(Dims d, int n) {
    d.B *= n;
    d.U *= n;
    return d;
}

}  // namespace
}  // namespace kvm

using namespace kvm;

extern "C" {

int kvm_version(void) { return KVM_VERSION; }

const char* kvm_status_string(int s) {
    switch (s) {
        case KVM_OK: return "ok";
        case KVM_E_NULL: return "a required pointer is NULL";
        case KVM_E_SHAPE: return "unsupported shape";
        case KVM_E_DTYPE: return "unknown dtype";
        case KVM_E_PARAM: return "parameter out of range or capacity too small for the conserved tokens";
        case KVM_E_ALIGN: return "pointer not 16-byte aligned";
        case KVM_E_WORKSPACE: return "workspace missing or too small";
        case KVM_E_UNSUPPORTED: return "unsupported request";
        case KVM_E_CUDA: return "CUDA runtime error";
        case KVM_E_DEVICE_TIMEOUT: return "a bounded device-side wait gave up";
        case KVM_E_STATIC_LIMIT:
            return "batch * n_q_heads * seq exceeds the built-in scratch of kvm_score_static (KVM_STATIC_SCORE_ROWS rows in fp32, an eighth of that in bf16)";
        default: return "unknown status";
    }
}

int kvm_sizes(const kvm_params* p, int32_t* cap, int32_t* n_recent, int32_t* n_heavy) {
    Dims d;
    const int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (cap) *cap = d.cap;
    if (n_recent) *n_recent = d.n_r;
    if (n_heavy) *n_heavy = d.n_h;
    return KVM_OK;
}

int kvm_workspace_bytes(const kvm_params* p, size_t* bytes) {
    Dims d;
    const int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!bytes) return KVM_E_NULL;
    *bytes = carve(d, nullptr).bytes;
    return KVM_OK;
}

int kvm_score(const kvm_params* p, const void* Q, const void* K, const float* lse_in, float* scores, void* ws,
              size_t ws_bytes, void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!Q || !K || !scores) return KVM_E_NULL;
    if (misaligned(Q) || misaligned(K) || misaligned(scores) || (lse_in && misaligned(lse_in))) return KVM_E_ALIGN;
    Workspace w;
    if ((rc = check_ws(d, ws, ws_bytes, w)) != KVM_OK) return rc;
    return run_score(d, one_layer(d, Q, K), lse_in, scores, w, nullptr, (cudaStream_t)cuda_stream) == cudaSuccess ? KVM_OK
                                                                                                    : KVM_E_CUDA;
}

int kvm_row_lse(const kvm_params* p, const void* Q, const void* K, float* lse_out, void* ws, size_t ws_bytes,
                void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!Q || !K || !lse_out) return KVM_E_NULL;
    if (misaligned(Q) || misaligned(K) || misaligned(lse_out)) return KVM_E_ALIGN;
    Workspace w;
    if ((rc = check_ws(d, ws, ws_bytes, w)) != KVM_OK) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const cudaError_t e = d.dtype == KVM_BF16
                              ? launch_score_tc(d, one_layer(d, Q, K), nullptr, w.lse, nullptr, nullptr, st, nullptr, lse_out)
                              : launch_score_f32(d, Q, K, nullptr, w.lse, nullptr, nullptr, st, nullptr, lse_out);
    return e == cudaSuccess ? KVM_OK : KVM_E_CUDA;
}

int kvm_segment(const kvm_params* p, const void* K, const float* scores, int32_t* set_id, int32_t* set_start,
                int32_t* pivot, int32_t* out_len, float* sim_out, kvm_stats* stats, void* ws, size_t ws_bytes,
                void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!K || !scores || !set_start || !pivot || !out_len) return KVM_E_NULL;
    if (misaligned(K) || misaligned(scores)) return KVM_E_ALIGN;
    Workspace w;
    if ((rc = check_ws(d, ws, ws_bytes, w)) != KVM_OK) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    float* sim = sim_out ? sim_out : w.sim;
    if (d.set_rule == KVM_SETS_ANCHOR) {
        // (the workspace's set-id region is free until the segment kernel writes it: scratch for the key norms)
        if (launch_anchor_runs(d, K, sim, (float*)w.set_id, st) != cudaSuccess) return KVM_E_CUDA;
    } else if (d.set_rule == KVM_SETS_ADJACENT || sim_out) {
        if (launch_similarity(d, K, sim, st) != cudaSuccess) return KVM_E_CUDA;
    }
    if (launch_segment(d, one_layer(d, nullptr, K, nullptr, nullptr, nullptr, out_len, pivot), const_cast<float*>(scores), ScorePart{},
                       sim, set_id, set_start, stats, st) != cudaSuccess)
        return KVM_E_CUDA;
    return KVM_OK;
}

int kvm_layer_ratio(const kvm_params* p, const void* K, float* ratio, float* sim_out, void* ws, size_t ws_bytes,
                    void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!K || !ratio) return KVM_E_NULL;
    if (misaligned(K)) return KVM_E_ALIGN;
    Workspace w;
    if ((rc = check_ws(d, ws, ws_bytes, w)) != KVM_OK) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    float* sim = sim_out ? sim_out : w.sim;
    if (launch_similarity(d, K, sim, st) != cudaSuccess) return KVM_E_CUDA;
    return launch_set_ratio(d, sim, ratio, st) == cudaSuccess ? KVM_OK : KVM_E_CUDA;
}

int kvm_prefill_attend(const kvm_params* p, const void* Q, const void* K, const void* V, void* O, float* lse,
                       kvm_stats* stats, void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (d.dtype != KVM_BF16) return KVM_E_UNSUPPORTED;
    if (!Q || !K || !V || !O || !lse) return KVM_E_NULL;
    if (misaligned(Q) || misaligned(K) || misaligned(V) || misaligned(O)) return KVM_E_ALIGN;
    return launch_prefill_attend(d, Q, K, V, O, lse, stats, (cudaStream_t)cuda_stream) == cudaSuccess ? KVM_OK
                                                                                                     : KVM_E_CUDA;
}

int kvm_attend(const kvm_params* p, const void* q, const void* K, const void* V, int32_t rows, const int32_t* len,
               float* out, void* ws, size_t ws_bytes, void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!q || !K || !V || !out) return KVM_E_NULL;
    if (rows < 1 || rows > d.S) return KVM_E_SHAPE;
    if (misaligned(q) || misaligned(K) || misaligned(V) || misaligned(out)) return KVM_E_ALIGN;
    Workspace w;
    if ((rc = check_ws(d, ws, ws_bytes, w)) != KVM_OK) return rc;
    return launch_attend(d, q, K, V, rows, len, out, w.attend_part, (cudaStream_t)cuda_stream) == cudaSuccess
               ? KVM_OK
               : KVM_E_CUDA;
}

int kvm_output_perturbation(const kvm_params* p, const void* q, const void* K, const void* V, const void* K_c,
                            const void* V_c, const int32_t* len_c, float* out_full, float* out_comp, float* err,
                            float* ref, void* ws, size_t ws_bytes, void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!q || !K || !V || !K_c || !V_c || !len_c || !out_full || !out_comp || !err || !ref) return KVM_E_NULL;
    if (misaligned(q) || misaligned(K) || misaligned(V) || misaligned(K_c) || misaligned(V_c) ||
        misaligned(out_full) || misaligned(out_comp))
        return KVM_E_ALIGN;
    Workspace w;
    if ((rc = check_ws(d, ws, ws_bytes, w)) != KVM_OK) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (launch_attend(d, q, K, V, d.S, nullptr, out_full, w.attend_part, st) != cudaSuccess) return KVM_E_CUDA;
    if (launch_attend(d, q, K_c, V_c, d.cap, len_c, out_comp, w.attend_part, st) != cudaSuccess) return KVM_E_CUDA;
    return launch_perturbation(d, out_full, out_comp, err, ref, st) == cudaSuccess ? KVM_OK : KVM_E_CUDA;
}

int kvm_merge_compact(const kvm_params* p, const void* K, const void* V, const int32_t* set_start,
                      const int32_t* pivot, const int32_t* out_len, void* K_out, void* V_out, int32_t* out_size,
                      void* ws, size_t ws_bytes, void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!K || !V || !set_start || !pivot || !out_len || !K_out || !V_out) return KVM_E_NULL;
    if (misaligned(K) || misaligned(V) || misaligned(K_out) || misaligned(V_out)) return KVM_E_ALIGN;
    Workspace w;
    if ((rc = check_ws(d, ws, ws_bytes, w)) != KVM_OK) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (d.weight_rule == KVM_WEIGHT_PIVOT_ONLY)
        return launch_gather(d, K, V, set_start, pivot, out_len, K_out, V_out, out_size, nullptr, st) == cudaSuccess
                   ? KVM_OK
                   : KVM_E_CUDA;
    if (launch_token_sets(d, set_start, out_len, w.set_id, st) != cudaSuccess) return KVM_E_CUDA;
    // (the similarity and score regions of the workspace are free here: scratch for the per-set bandwidths)
    const Layers L = one_layer(d, nullptr, K, V, K_out, V_out, const_cast<int32_t*>(out_len), const_cast<int32_t*>(pivot));
    return launch_merge(d, L, set_start, w.set_id, out_size, w.merge_part, w.sim, w.scores, nullptr, st) == cudaSuccess
               ? KVM_OK
               : KVM_E_CUDA;
}

int kvm_compress(const kvm_params* p, const void* Q, const void* K, const void* V, void* K_out, void* V_out,
                 int32_t* out_len, int32_t* out_pos, float* scores_out, kvm_stats* stats, void* ws,
                 size_t ws_bytes, void* cuda_stream) {
    return kvm_compress_with_lse(p, Q, K, V, nullptr, K_out, V_out, out_len, out_pos, scores_out, stats, ws,
                                 ws_bytes, cuda_stream);
}

int kvm_compress_with_lse(const kvm_params* p, const void* Q, const void* K, const void* V, const float* lse_in,
                          void* K_out, void* V_out, int32_t* out_len, int32_t* out_pos, float* scores_out,
                          kvm_stats* stats, void* ws, size_t ws_bytes, void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!Q || !K || !V || !K_out || !V_out || !out_len || !out_pos) return KVM_E_NULL;
    if (misaligned(Q) || misaligned(K) || misaligned(V) || misaligned(K_out) || misaligned(V_out) ||
        (scores_out && misaligned(scores_out)) || (lse_in && misaligned(lse_in)))
        return KVM_E_ALIGN;
    Workspace w;
    if ((rc = check_ws(d, ws, ws_bytes, w)) != KVM_OK) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    return run_chain(d, one_layer(d, Q, K, V, K_out, V_out, out_len, out_pos), lse_in, scores_out ? scores_out : w.scores, w,
                     stats, st);
}

int kvm_layers_workspace_bytes(const kvm_params* p, int32_t n_layers, size_t* bytes) {
    Dims d;
    const int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!bytes) return KVM_E_NULL;
    if (n_layers < 1) return KVM_E_SHAPE;
    *bytes = 0;
    for (int n = 1; n <= layers_together(d, n_layers); ++n) {      // (a smaller last group may be split differently)
        const size_t b = carve(times_batch(d, n), nullptr).bytes;
        if (b > *bytes) *bytes = b;
    }
    return KVM_OK;
}

static int compress_layers(int zero_rest, const kvm_params* p, int32_t n_layers, const float* sim_thresholds, const void* const* Q,
                        const void* const* K, const void* const* V, void* const* K_out, void* const* V_out,
                        int32_t* const* out_len, int32_t* const* out_pos, kvm_stats* stats, void* ws,
                        size_t ws_bytes, void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (n_layers < 1) return KVM_E_SHAPE;
    if (!Q || !K || !V || !K_out || !V_out || !out_len || !out_pos) return KVM_E_NULL;
    Workspace w;
    if ((rc = check_ws(d, ws, ws_bytes, w)) != KVM_OK) return rc;
    for (int32_t l = 0; l < n_layers; ++l) {       // everything is checked before the first layer is enqueued
        if (!Q[l] || !K[l] || !V[l] || !K_out[l] || !V_out[l] || !out_len[l] || !out_pos[l]) return KVM_E_NULL;
        if (misaligned(Q[l]) || misaligned(K[l]) || misaligned(V[l]) || misaligned(K_out[l]) || misaligned(V_out[l]))
            return KVM_E_ALIGN;
        if (sim_thresholds && !isfinite(sim_thresholds[l])) return KVM_E_PARAM;
    }
    const int together = layers_together(d, n_layers);
    for (int32_t l0 = 0; l0 < n_layers;) {
        int n = n_layers - l0 < together ? n_layers - l0 : together;
        while (n > 1 && carve(times_batch(d, n), nullptr).bytes > ws_bytes) --n;
        Layers L = one_layer(d, nullptr, nullptr);
        L.n = n;
        L.zero_rest = zero_rest;
        for (int i = 0; i < n; ++i) {
            L.Q[i] = Q[l0 + i]; L.K[i] = K[l0 + i]; L.V[i] = V[l0 + i];
            L.K_out[i] = K_out[l0 + i]; L.V_out[i] = V_out[l0 + i];
            L.out_len[i] = out_len[l0 + i]; L.pivot[i] = out_pos[l0 + i];
            L.eps[i] = sim_thresholds ? sim_thresholds[l0 + i] : d.eps;
        }
        const Dims dn = times_batch(d, n);
        const Workspace wn = carve(dn, ws);
        rc = run_chain(dn, L, nullptr, wn.scores, wn, stats, (cudaStream_t)cuda_stream);
        if (rc != KVM_OK) return rc;
        l0 += n;
    }
    return KVM_OK;
}

int kvm_compress_layers(const kvm_params* p, int32_t n_layers, const float* sim_thresholds, const void* const* Q,
                        const void* const* K, const void* const* V, void* const* K_out, void* const* V_out,
                        int32_t* const* out_len, int32_t* const* out_pos, kvm_stats* stats, void* ws,
                        size_t ws_bytes, void* cuda_stream) {
    return compress_layers(0, p, n_layers, sim_thresholds, Q, K, V, K_out, V_out, out_len, out_pos, stats, ws, ws_bytes, cuda_stream);
}
int kvm_compress_layers_filled(const kvm_params* p, int32_t n_layers, const float* sim_thresholds, const void* const* Q,
                        const void* const* K, const void* const* V, void* const* K_out, void* const* V_out,
                        int32_t* const* out_len, int32_t* const* out_pos, kvm_stats* stats, void* ws,
                        size_t ws_bytes, void* cuda_stream) {
    return compress_layers(1, p, n_layers, sim_thresholds, Q, K, V, K_out, V_out, out_len, out_pos, stats, ws, ws_bytes, cuda_stream);
}

// The groups of units that kvm_compress_host's pipeline takes one after the other.
namespace {

constexpr int kHostChunksMax = 6;
// (us a call for a Llama2-7B-shaped layer of 4096 tokens, 101 MB in, in one run: equal quarters 2223; ratio 0.7 2242, 0.6 2201,
// 0.5 2136, 0.4 2166, 0.3 2236; over several boxes quarters 2203-2225, ratio 0.5 2124-2190.  15 heads x 2 x 488 x 64, 5.6 MB
// in: quarters 387; ratio 0.5 with groups of at least 3 MB 285, 2 MB 209, 1 MB 226)
constexpr double kHostRatio = 0.5;
constexpr long long kHostMinBytes = 2ll << 20;

// Cuts U units of `unit_bytes` input each into groups: group c is units [first[c], first[c + 1]).  What the pipeline's end
// costs is the last group's kernels and copy out, with nothing left to overlap them, so every group is kHostRatio of the one
// before it; none is copied in with less than kHostMinBytes (shorter copies do not reach the link's rate, and a group
// costs a dozen launches and copies).
int host_groups(int U, size_t unit_bytes, int* first) {
    const long long total = (long long)U * (long long)unit_bytes;
    int n = 1;
    double w = 1.0, sum = 1.0;                 // weights 1, r, r^2, ...
    while (n < kHostChunksMax && n < U) {
        const double w2 = w * kHostRatio;
        if ((double)total * w2 / (sum + w2) < (double)kHostMinBytes) break;
        w = w2;
        sum += w;
        ++n;
    }
    double acc = 0.0, wi = 1.0;
    first[0] = 0;
    for (int c = 0; c < n; ++c, wi *= kHostRatio) {
        acc += wi;
        int e = (int)(acc / sum * U + 0.5);
        const int lo = first[c] + 1, hi = U - (n - 1 - c);
        e = e < lo ? lo : e > hi ? hi : e;
        first[c + 1] = c + 1 == n ? U : e;
    }
    return n;
}

// A group of units as a layer of its own: one batch entry, nu KV heads.
kvm_params group_params(const kvm_params* p, const Dims& d, int u0, int nu) {
    kvm_params pc = *p;
    pc.batch = 1;
    pc.n_kv_heads = nu;
    pc.n_q_heads = nu * d.G;
    if (pc.pivot_key) pc.pivot_key += (size_t)u0 * d.S;
    return pc;
}
size_t host_unit_bytes(const Dims& d) { return (size_t)(d.G + 2) * d.S * d.D * (d.dtype == KVM_BF16 ? 2 : 4); }

}  // namespace

int kvm_host_staging_bytes(const kvm_params* p, size_t* bytes) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!bytes) return KVM_E_NULL;
    const size_t e = d.dtype == KVM_BF16 ? 2 : 4;
    size_t off = 0;
    off += align_up((size_t)d.B * d.Hq * d.S * d.D * e);        // Q
    off += 2 * align_up((size_t)d.U * d.S * d.D * e);           // K, V
    off += 2 * align_up((size_t)d.U * d.cap * d.D * e);         // K_out, V_out
    off += align_up((size_t)d.U * sizeof(int32_t));             // out_len
    off += align_up((size_t)d.U * d.cap * sizeof(int32_t));     // out_pos
    // The groups' kernels run one after the other in one workspace.  A group can need more than the whole layer: its score
    // passes may be cut where the layer's are not, and then leave partial results.
    size_t ws = carve(d, nullptr).bytes;
    int first[kHostChunksMax + 1];
    const int n = host_groups(d.U, host_unit_bytes(d), first);
    for (int c = 0; c < n; ++c) {
        const kvm_params pc = group_params(p, d, first[c], first[c + 1] - first[c]);
        Dims dc;
        if ((rc = derive(&pc, dc)) != KVM_OK) return rc;
        const size_t b = carve(dc, nullptr).bytes;
        if (b > ws) ws = b;
    }
    *bytes = off + ws;
    return KVM_OK;
}

// Streams and events of kvm_compress_host's copy/compute pipeline: created once per device on first use,
// kept until the process exits.
namespace {

constexpr int kPipeDevices = 64;

struct HostPipe {
    bool ready = false;
    cudaStream_t compute = nullptr, d2h = nullptr;
    cudaEvent_t start = nullptr, end = nullptr, h2d[kHostChunksMax] = {}, done[kHostChunksMax] = {};
};
HostPipe g_pipe[kPipeDevices];
std::mutex g_pipe_mu;      // held while a call enqueues: calls on one device share the events

HostPipe* host_pipe_for_current_device() {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kPipeDevices) return nullptr;
    HostPipe& hp = g_pipe[dev];
    if (hp.ready) return &hp;
    bool ok = cudaStreamCreateWithFlags(&hp.compute, cudaStreamNonBlocking) == cudaSuccess &&
              cudaStreamCreateWithFlags(&hp.d2h, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&hp.start, cudaEventDisableTiming) == cudaSuccess &&
              cudaEventCreateWithFlags(&hp.end, cudaEventDisableTiming) == cudaSuccess;
    for (int i = 0; ok && i < kHostChunksMax; ++i)
        ok = cudaEventCreateWithFlags(&hp.h2d[i], cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&hp.done[i], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) return nullptr;
    hp.ready = true;
    return &hp;
}

}  // namespace

int kvm_compress_host(const kvm_params* p, const void* Q, const void* K, const void* V, void* K_out, void* V_out,
                      int32_t* out_len, int32_t* out_pos, void* dev, size_t dev_bytes, void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!Q || !K || !V || !K_out || !V_out || !out_len || !out_pos) return KVM_E_NULL;
    size_t need = 0;
    kvm_host_staging_bytes(p, &need);
    if (!dev || dev_bytes < need) return KVM_E_WORKSPACE;
    if (misaligned(dev)) return KVM_E_ALIGN;
    const size_t e = d.dtype == KVM_BF16 ? 2 : 4;
    const size_t rowQ = (size_t)d.G * d.S * d.D * e, rowK = (size_t)d.S * d.D * e;       // bytes per unit
    const size_t rowO = (size_t)d.cap * d.D * e, rowP = (size_t)d.cap * sizeof(int32_t);
    char* b = (char*)dev;
    size_t off = 0;
    auto take = [&](size_t n) { char* q = b + off; off += align_up(n); return q; };
    char* dQ = take(rowQ * d.U); char* dK = take(rowK * d.U); char* dV = take(rowK * d.U);
    char* dKo = take(rowO * d.U); char* dVo = take(rowO * d.U);
    char* dL = take((size_t)d.U * sizeof(int32_t)); char* dP = take(rowP * d.U);
    char* ws = b + off;
    const size_t ws_bytes = dev_bytes - off;
    cudaStream_t st = (cudaStream_t)cuda_stream;

    // Units are independent and contiguous in every tensor, so the layer is cut into groups of units and
    // the three stages run as a pipeline: host-to-device copies on the caller's stream, kernels on a second
    // stream, device-to-host copies on a third.  The caller's stream waits for the last copy out.
    std::lock_guard<std::mutex> lock(g_pipe_mu);
    HostPipe* hp = host_pipe_for_current_device();
    if (!hp) return KVM_E_CUDA;
    int first[kHostChunksMax + 1];
    const int nch = host_groups(d.U, host_unit_bytes(d), first);
    auto ok = [](cudaError_t err) { return err == cudaSuccess; };
    // every group is validated before anything is enqueued, so a refusal leaves no copy in flight
    for (int c = 0; c < nch; ++c) {
        const kvm_params pc = group_params(p, d, first[c], first[c + 1] - first[c]);
        Dims dc;
        size_t need_c = 0;
        if ((rc = derive(&pc, dc)) != KVM_OK) return rc;
        if ((rc = kvm_workspace_bytes(&pc, &need_c)) != KVM_OK) return rc;
        if (need_c > ws_bytes) return KVM_E_WORKSPACE;
    }
    if (!ok(cudaEventRecord(hp->start, st)) || !ok(cudaStreamWaitEvent(hp->compute, hp->start, 0)) ||
        !ok(cudaStreamWaitEvent(hp->d2h, hp->start, 0)))
        return KVM_E_CUDA;
    // From here on work is in flight on the library's streams: whatever happens, the caller's stream is made
    // to wait for all of it before the call returns, so that an error return never leaves copies writing the
    // caller's buffers behind its back.
    int status = KVM_OK;
    for (int c = 0; c < nch && status == KVM_OK; ++c) {
        const int u0 = first[c], nu = first[c + 1] - u0;
        const kvm_params pc = group_params(p, d, u0, nu);
        if (!ok(cudaMemcpyAsync(dQ + rowQ * u0, (const char*)Q + rowQ * u0, rowQ * nu, cudaMemcpyHostToDevice, st)) ||
            !ok(cudaMemcpyAsync(dK + rowK * u0, (const char*)K + rowK * u0, rowK * nu, cudaMemcpyHostToDevice, st)) ||
            !ok(cudaMemcpyAsync(dV + rowK * u0, (const char*)V + rowK * u0, rowK * nu, cudaMemcpyHostToDevice, st)) ||
            !ok(cudaEventRecord(hp->h2d[c], st)) || !ok(cudaStreamWaitEvent(hp->compute, hp->h2d[c], 0))) {
            status = KVM_E_CUDA;
            break;
        }
        rc = kvm_compress(&pc, dQ + rowQ * u0, dK + rowK * u0, dV + rowK * u0, dKo + rowO * u0, dVo + rowO * u0,
                          (int32_t*)dL + u0, (int32_t*)(dP + rowP * u0), nullptr, nullptr, ws, ws_bytes, hp->compute);
        if (rc != KVM_OK) {
            status = rc;
            break;
        }
        if (!ok(cudaEventRecord(hp->done[c], hp->compute)) || !ok(cudaStreamWaitEvent(hp->d2h, hp->done[c], 0)) ||
            !ok(cudaMemcpyAsync((char*)K_out + rowO * u0, dKo + rowO * u0, rowO * nu, cudaMemcpyDeviceToHost, hp->d2h)) ||
            !ok(cudaMemcpyAsync((char*)V_out + rowO * u0, dVo + rowO * u0, rowO * nu, cudaMemcpyDeviceToHost, hp->d2h)) ||
            !ok(cudaMemcpyAsync(out_len + u0, (int32_t*)dL + u0, (size_t)nu * sizeof(int32_t), cudaMemcpyDeviceToHost,
                                hp->d2h)) ||
            !ok(cudaMemcpyAsync((char*)out_pos + rowP * u0, dP + rowP * u0, rowP * nu, cudaMemcpyDeviceToHost, hp->d2h)))
            status = KVM_E_CUDA;
    }
    // join: the copy-out stream follows the compute stream, the caller's stream follows the copy-out stream
    if (!ok(cudaEventRecord(hp->done[0], hp->compute)) || !ok(cudaStreamWaitEvent(hp->d2h, hp->done[0], 0)) ||
        !ok(cudaEventRecord(hp->end, hp->d2h)) || !ok(cudaStreamWaitEvent(st, hp->end, 0)))
        return KVM_E_CUDA;
    return status;
}

// ---------------------------------------------------------------------------
// kvm_score without a caller workspace, for callers that may not allocate.
// The scratch is part of the library image; see the declaration in kvm.h.
namespace {

constexpr int kMaxDevices = KVM_MAX_DEVICES;

// The row pass's output for up to KVM_STATIC_SCORE_ROWS fp32 rows, and room for what cut work items leave (for 2^17 bf16
// rows at most 0.6 MiB over all shapes; the fp32 path's share the 4 MiB).  In HOST code this name is only a stand-in
// for the device symbol; its device address comes from cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned char g_static_score_scratch[(size_t)KVM_STATIC_SCORE_ROWS * sizeof(float) + (5u << 18)];

void* g_static_ptr[kMaxDevices];   // device address of the array, per device; set once

// One-time set-up for the current device.  Returns nullptr if the runtime refuses.
void* static_scratch_for_current_device() {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    void* ptr = __atomic_load_n(&g_static_ptr[dev], __ATOMIC_ACQUIRE);
    if (ptr) return ptr;
    if (cudaGetSymbolAddress(&ptr, g_static_score_scratch) != cudaSuccess || !ptr) return nullptr;
    __atomic_store_n(&g_static_ptr[dev], ptr, __ATOMIC_RELEASE);   // racing first calls store the same value
    return ptr;
}

}  // namespace

int kvm_score_static(const kvm_params* p, const void* Q, const void* K, float* scores, void* cuda_stream) {
    Dims d;
    int rc = derive(p, d);
    if (rc != KVM_OK) return rc;
    if (!Q || !K || !scores) return KVM_E_NULL;
    if (misaligned(Q) || misaligned(K) || misaligned(scores)) return KVM_E_ALIGN;
    // 32 bytes per query row for bf16 tensors; fp32 ones need 4 where work items stay whole, and what fits the array
    // where they are split (so that both entry points run the same plan)
    if ((unsigned long long)d.B * d.Hq * d.S > (unsigned long long)KVM_STATIC_SCORE_ROWS / (d.dtype == KVM_BF16 ? 8 : 1))
        return KVM_E_STATIC_LIMIT;
    if (score_bytes(d) > sizeof(g_static_score_scratch)) return KVM_E_STATIC_LIMIT;
    unsigned char* base = (unsigned char*)static_scratch_for_current_device();
    if (!base) return KVM_E_CUDA;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // The array keeps the previous call's contents.  Nothing in it has to start at zero: the row pass rewrites
    // every row this call's column pass reads.
    Workspace w;
    w.lse = (float*)base;
    w.scores = nullptr;
    w.sim = nullptr;
    w.set_start = nullptr;
    w.set_id = nullptr;
    w.merge_part = nullptr;
    w.attend_part = nullptr;
    w.bytes = sizeof(g_static_score_scratch);
    return run_score(d, one_layer(d, Q, K), nullptr, scores, w, nullptr, st) == cudaSuccess ? KVM_OK : KVM_E_CUDA;
}

}  // extern "C"
