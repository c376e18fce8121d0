// One decode step of attention over a cache whose units may have different
// lengths (Eq. 1: O_t = softmax(q_t K^T / sqrt(d)) V), and the output
// perturbation |O_t - O_t*| of Definition 2.1 between the full and the
// compressed cache.
//
// Bandwidth-bound: K and V rows are read once from HBM.  What it takes to get there:
//   - the query heads of a KV head share a row's one way through shared memory (up to eight at a time; one block per
//     query head read everything G times through L2: 206 us against 72 us on 8 x 32/8 heads x 12288 rows on average);
//   - one persistent block per SM takes an equal share of all the rows there are (lengths differ; the shares are cut by
//     a prefix sum over the units' lengths, so that no SM idles while another finishes a long unit; a unit counts as
//     many rows more as a block could take in the time that starting and joining it costs);
//   - the rows come by bulk copies into a ring of 16 KB + 16 KB stages, 128 KB in flight per SM, issued by a warp of
//     its own; eight warps compute.
// A group of LPR lanes owns four rows of a stage.  Its products (rows x heads) are summed across the lanes by a
// transposing butterfly that leaves each lane one (row, head) to exponentiate; the weights come back by shuffle for
// the second product.  The weights' reference is never below a logit (no weight exceeds 1, as with the plain running maximum)
// and moves only when it is: to 8 above the new maximum (log2 units), so that a slowly growing maximum moves it seldom.
// A unit's rows that fall into several blocks' shares leave partial states (weighted V sum, maximum, sum), combined in a
// fixed order by a second kernel: results are reproducible.
// Two more forms, for few units (clusters) and for many short ones (small blocks), below; Scratch::choose says which is when.
#include <mutex>
#include <type_traits>

#include "tc_common.cuh"

namespace kvm {
namespace {

using namespace tc;

constexpr int ATT_WARPS = 8;                // computing warps; one more issues the copies
constexpr int ATT_NT = (ATT_WARPS + 1) * 32;
constexpr int ATT_STAGES = 4;
constexpr int ATT_STAGE_BYTES = 16384;      // of K, and as much of V
constexpr int ATT_MIN_SHARE = 64;           // fewest rows a block is given (bounds the number of pieces)
// What an item costs a block beside its rows, about 3 us, in rows at a block's part of the bandwidth.  (Counted by rows
// alone, 160 units of up to 3 rows fell to 4 blocks, 40 each: 64 us, 12 so.)
constexpr int ATT_ITEM_BYTES = 131072;
__host__ __device__ constexpr int item_rows(int D, int elem) { return ATT_ITEM_BYTES / (2 * D * elem); }
constexpr int RPI = 4;                      // rows of a stage per lane group
constexpr float LOG2E = 1.4426950408889634f;
constexpr float REF_STEP = 8.f;             // room above the maximum that the reference is set with (log2 units)

// Weight of a partial state with maximum m when the overall maximum is M (an empty state has m = -inf).
__device__ __forceinline__ float rescale(float m, float M) { return m == -INFINITY ? 0.f : exp2f(m - M); }
// The block's walk over the items of its share.  Item = (unit, group of GH query heads), in that order.  Shares are cut in
// a list in which an item with rows is `pad` entries for itself, then one for each of its rows.
struct Item {
    unsigned long long start;    // entries of all items before this one
    int id, n;                   // item, rows of its unit
    int off, cnt;                // this block's part: rows [off, off + cnt)
};
struct Work {
    const int32_t* len;
    int rows, HG, items, pad;
    unsigned long long q, f, f_end;      // entries per block; what is left of this block's share: [f, f_end)
    __device__ __forceinline__ int rows_of(int item) const { return len ? max(0, min(__ldg(len + item / HG), rows)) : rows; }
    __device__ __forceinline__ int entries(int n) const { return n > 0 ? n + pad : 0; }
    // moves to the rows of item `it` that belong to the share (skipping items without any); false when the share is done
    __device__ __forceinline__ bool settle(Item& it) {
        while (f < f_end && it.id < items) {
            const unsigned long long r0 = it.start + pad, end = it.start + entries(it.n);
            if (end > f) {
                if (f < r0) f = r0;
                if (f >= f_end) return false;
                it.off = (int)(f - r0);
                it.cnt = (int)(min(end, f_end) - f);
                return true;
            }
            it.start = end;
            if (++it.id < items) it.n = rows_of(it.id);
        }
        return false;
    }
};

// This block's share, cut by a prefix sum over the items' rows (all threads of the block; false: nothing to do).
struct ShareSmem {
    unsigned long long wsum[ATT_WARPS + 1], start;
    int id;
};
__device__ __forceinline__ bool take_share(Work& w, Item& it, ShareSmem& sh) {
    const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
    const int E = (w.items + ATT_NT - 1) / ATT_NT, i0 = min(w.items, (int)threadIdx.x * E), i1 = min(w.items, i0 + E);
    unsigned long long mine = 0;
    for (int i = i0; i < i1; ++i) mine += w.entries(w.rows_of(i));
    unsigned long long inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xffffffffu, inc, o);
        if (wl >= o) inc += t;
    }
    if (wl == 31) sh.wsum[warp] = inc;
    __syncthreads();
    unsigned long long total = 0, before = inc - mine;
#pragma unroll
    for (int x = 0; x <= ATT_WARPS; ++x) {
        if (x < warp) before += sh.wsum[x];
        total += sh.wsum[x];
    }
    w.q = max((total + gridDim.x - 1) / gridDim.x, (unsigned long long)ATT_MIN_SHARE);
    w.f = min(total, w.q * blockIdx.x);
    w.f_end = min(total, w.f + w.q);
    if (w.f == w.f_end) return false;
    if (before <= w.f && w.f < before + mine) {                    // true in exactly one thread
        unsigned long long st = before;
        int id = i0, n = w.entries(w.rows_of(id));
        while (st + n <= w.f) { st += n; n = w.entries(w.rows_of(++id)); }
        sh.start = st;
        sh.id = id;
    }
    __syncthreads();
    it.start = sh.start; it.id = sh.id; it.n = w.rows_of(it.id);
    return true;
}

// Copies complete on their own; the copying thread, which has issued k stages, stays until its last ones have landed (the
// wait is bounded like the others), so that a block whose other warps gave up does not hand its shared memory back under a
// copy in flight.
__device__ __forceinline__ void drain(uint64_t* full, uint32_t k) {
    for (uint32_t s = 0; s < ATT_STAGES && s < k; ++s) {
        const uint32_t parity = ((k - 1 - s) / ATT_STAGES) & 1;
        const long long t0 = clock64();
        while (!mbar_try(&full[s], parity) && clock64() - t0 <= WAIT_LIMIT_CLOCKS) {}
    }
}

// Piece end: the warps' states (sm_m, sm_l, sm_acc [warp][GH][D]) in a fixed order -> the piece's state of `heads` heads at
// dst: per head D weighted sums, the maximum and the sum.
template <int D, int GH>
__device__ __forceinline__ void store_piece(const float (*sm_m)[GH], const float (*sm_l)[GH], const float* sm_acc, bool bad,
                                            float* dst, int heads) {
    for (int i = threadIdx.x; i < heads * D; i += ATT_WARPS * 32) {
        const int h = i / D;
        float M = -INFINITY, L = 0.f, o = 0.f;
#pragma unroll
        for (int x = 0; x < ATT_WARPS; ++x) M = fmaxf(M, sm_m[x][h]);
#pragma unroll
        for (int x = 0; x < ATT_WARPS; ++x) {
            const float a = rescale(sm_m[x][h], M);
            L = fmaf(sm_l[x][h], a, L);
            o = fmaf(sm_acc[(x * GH + h) * D + i % D], a, o);
        }
        dst[h * (D + 2) + i % D] = bad ? NAN : o;
        if (i % D == 0) { dst[h * (D + 2) + D] = M; dst[h * (D + 2) + D + 1] = L; }
    }
}
// Where a piece's state goes; the block that holds the item's first row also tells how many pieces the item has.
__device__ __forceinline__ float* piece_slot(const Work& w, const Item& it, float* part, int32_t* pieces, int max_pieces,
                                             int state_floats) {
    const unsigned long long r0 = it.start + w.pad;
    const int first = (int)(r0 / w.q);
    if (threadIdx.x == 0 && (int)blockIdx.x == first) pieces[it.id] = (int)((r0 + it.n - 1) / w.q) - first + 1;
    return part + ((size_t)it.id * max_pieces + (blockIdx.x - first)) * state_floats;
}

// ------------------------------------------------------------------ short caches: a cluster per item
// Where an item's rows divided over a few blocks take about as long as an equal share, the blocks of an item are a
// thread-block cluster: each takes a slice of the item's rows and the states are joined through distributed shared
// memory, without a second kernel (32 heads x 1536 rows on average: 12.0 us with one, of which its launch and three
// dependent reads are 5).
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ float peer_load(uint32_t addr, uint32_t rank) {
    float v;
    asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\tld.shared::cluster.f32 %0, [a];\n\t}"
                 : "=f"(v) : "r"(addr), "r"(rank) : "memory");
    return v;
}
// This block's slice as a share of its own, and an empty state to start from.
template <int D, int GH>
__device__ __forceinline__ void take_slice(Work& w, Item& it, int C, float* fin) {
    for (int i = threadIdx.x; i < GH * (D + 2); i += ATT_NT) fin[i] = i % (D + 2) == D ? -INFINITY : 0.f;
    it.start = 0;
    it.id = blockIdx.x / C;
    it.n = w.rows_of(it.id);
    const int per = ((it.n + C - 1) / C + 15) & ~15, off = min(it.n, (int)(blockIdx.x % C) * per);
    w.q = 1;
    w.f = off;
    w.f_end = min(it.n, off + per);
    __syncthreads();
}
// Joins the cluster's states (fin, [head][D + 2]) in order of rank; every block stores a part of the item's heads.
template <int D>
__device__ __forceinline__ void join_cluster(const float* fin, int item, int HG, int GH, int G, int C, float* out) {
    cluster_barrier();
    const int u = item / HG, h0 = (item % HG) * GH, heads = min(G - h0, GH);
    const uint32_t base = smem_u32(fin);
    for (int i = (int)(blockIdx.x % C) * ATT_NT + threadIdx.x; i < heads * D; i += C * ATT_NT) {
        const uint32_t at = base + (uint32_t)(i / D) * (D + 2) * 4u;
        float M = -INFINITY, L = 0.f, o = 0.f;
        for (int s = 0; s < C; ++s) {
            const float ms = peer_load(at + D * 4u, s), ls = peer_load(at + (D + 1) * 4u, s), os = peer_load(at + (i % D) * 4u, s);
            const float mn = fmaxf(M, ms), a = rescale(M, mn), c = rescale(ms, mn);
            L = fmaf(ls, c, L * a);
            o = fmaf(os, c, o * a);
            M = mn;
        }
        out[((size_t)u * G + h0 + i / D) * D + i % D] = L > 0.f || L != L || o != o ? o / L : 0.f;   // (an empty cache attends to nothing)
    }
    cluster_barrier();          // (shared memory stays until every peer has read it)
}

// part: per item and piece, for each of the GH heads D weighted sums, the maximum and the sum (log2 units); pieces:
// per item, how many there are.
template <typename T, int D, int GH, bool CL>
__global__ void __launch_bounds__(ATT_NT, 1)
attend_partial_fma_kernel(const T* __restrict__ q, const T* __restrict__ K, const T* __restrict__ V,
                      const int32_t* __restrict__ len, float* __restrict__ part, int32_t* __restrict__ pieces, int rows, int G,
                      int U, int max_pieces, float scale_log2e, int C, float* __restrict__ out) {
    constexpr int N = Vec<T>::N, LPR = D / N, GPW = 32 / LPR;      // elements per 16 bytes, lanes per row, groups per warp
    constexpr int SROWS = ATT_STAGE_BYTES / (D * (int)sizeof(T));  // rows per stage
    static_assert(SROWS == ATT_WARPS * GPW * RPI, "a stage is one round of every group");
    constexpr int NV = RPI * GH, CNT = NV > LPR ? NV / LPR : 1;    // products per lane, and how many it keeps
    constexpr int REP = NV < LPR ? LPR / NV : 1, RL = RPI / CNT;   // lanes holding the same product; lanes per head's rows
    static_assert(CNT <= RPI, "a lane's products belong to one head");
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t* ring = smem;                                          // [stage][K | V][SROWS][D]
    float* sm_acc = reinterpret_cast<float*>(smem + ATT_STAGES * 2 * ATT_STAGE_BYTES);   // [warp][GH][D]
    float* fin = sm_acc + ATT_WARPS * GH * D;                      // [GH][D + 2]: this block's state (clusters)
    __shared__ __align__(8) uint64_t full[ATT_STAGES], empty[ATT_STAGES];
    __shared__ float sm_m[ATT_WARPS][GH], sm_l[ATT_WARPS][GH];
    __shared__ ShareSmem sh;
    __shared__ volatile int s_bad;

    const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
    Work w;
    w.len = len; w.rows = rows; w.HG = (G + GH - 1) / GH; w.items = U * w.HG; w.pad = CL ? 0 : item_rows(D, sizeof(T));
    if (threadIdx.x == 0) {
        for (int i = 0; i < ATT_STAGES; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], ATT_WARPS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_bad = 0;
    }
    grid_dependency_wait();
    Item it;
    if (CL) take_slice<D, GH>(w, it, C, fin);
    else if (!take_share(w, it, sh)) return;
    const int item = it.id;

    if (warp == ATT_WARPS) {
        // ---- copies
        if (wl == 0) {
            uint32_t k = 0;
            bool ok = true;
            while (ok && w.settle(it)) {
                const size_t r0 = (size_t)(it.id / w.HG) * rows + it.off;
                for (int r = 0; r < it.cnt; r += SROWS, ++k) {
                    const int s = k % ATT_STAGES;
                    ok = mbar_wait(&empty[s], ((k / ATT_STAGES) & 1) ^ 1, &s_bad);
                    if (!ok) break;
#ifdef KVM_TEST_DROP_ATTEND_STAGE
                    if (blockIdx.x == KVM_TEST_DROP_CTA && k == (uint32_t)(KVM_TEST_DROP_ATTEND_STAGE)) continue;   // test build only: this stage never arrives
#endif
                    const uint32_t bytes = (uint32_t)min(SROWS, it.cnt - r) * D * sizeof(T);
                    const uint32_t dst = smem_u32(ring + s * 2 * ATT_STAGE_BYTES), bar = smem_u32(&full[s]);
                    mbar_expect_tx(&full[s], 2 * bytes);
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(dst), "l"(K + (r0 + r) * D), "r"(bytes), "r"(bar) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(dst + ATT_STAGE_BYTES), "l"(V + (r0 + r) * D), "r"(bytes), "r"(bar) : "memory");
                }
                w.f += it.cnt;
            }
            drain(full, k);
        }
        if (!CL) return;
        __syncwarp();
    }
    // ---- arithmetic
    const int lane = wl % LPR, g = wl / LPR;                       // lane within the row, group within the warp
    const int head = lane / (RL * REP);                            // the head whose products this lane finishes
    const int rl = (lane / REP) % RL;                              // ... for rows rl * CNT .. + CNT of the group's four
    const int lb = g * LPR;                                        // the group's first lane
    uint32_t k = 0;
    while (warp != ATT_WARPS && w.settle(it)) {
        const int u = it.id / w.HG, h0 = (it.id % w.HG) * GH;
        uint64_t qp[GH][N / 2], acc[GH][N / 2];
#pragma unroll
        for (int h = 0; h < GH; ++h) {
            float f[N];
            Vec<T>::unpack(ldg16(q + ((size_t)u * G + min(h0 + h, G - 1)) * D + lane * N), f);
#pragma unroll
            for (int e = 0; e < N / 2; ++e) { qp[h][e] = pack2(f[2 * e], f[2 * e + 1]); acc[h][e] = 0ull; }
        }
        float m = -INFINITY, l = 0.f;                              // of this lane's head (l: of this lane's rows)
        for (int r = 0; r < it.cnt; r += SROWS, ++k) {
            const int s = k % ATT_STAGES;
            // (the block's own copies always complete; a wait that ran out all the same makes the outputs NaN)
            if (!__all_sync(0xffffffffu, mbar_wait(&full[s], (k / ATT_STAGES) & 1, &s_bad))) break;
            const int row = (warp * GPW + g) * RPI, live = it.cnt - r - row;      // rows of the group that exist
            const uint4* sk = reinterpret_cast<const uint4*>(ring + s * 2 * ATT_STAGE_BYTES) + row * LPR + lane;
            const uint4* sv = reinterpret_cast<const uint4*>(ring + s * 2 * ATT_STAGE_BYTES + ATT_STAGE_BYTES) + row * LPR + lane;
            float v[NV];                                           // product of head h, row i: v[h * RPI + i]
#pragma unroll
            for (int i = 0; i < RPI; ++i) {
                float f[N];
                Vec<T>::unpack(sk[i * LPR], f);
#pragma unroll
                for (int h = 0; h < GH; ++h) {
                    uint64_t a = 0ull;
#pragma unroll
                    for (int e = 0; e < N / 2; ++e) a = ffma2(qp[h][e], pack2(f[2 * e], f[2 * e + 1]), a);
                    float lo, hi;
                    unpack2(a, lo, hi);
                    v[h * RPI + i] = lo + hi;
                }
            }
#pragma unroll
            for (int o = LPR / 2, c = NV; o > 0; o >>= 1) {
                if (c > 1) {
                    c >>= 1;
                    const bool up = (lane & o) != 0;
#pragma unroll
                    for (int i = 0; i < NV / 2; ++i) {
                        if (i >= c) break;
                        const float keep = up ? v[i + c] : v[i], give = up ? v[i] : v[i + c];
                        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                    }
                } else {
                    v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
                }
            }
            float p[CNT], mx = -INFINITY;
#pragma unroll
            for (int i = 0; i < CNT; ++i) {
                p[i] = rl * CNT + i < live ? v[i] * scale_log2e : -INFINITY;
                mx = fmaxf(mx, p[i]);
            }
#pragma unroll
            for (int o = REP; o < REP * RL; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const bool grow = mx > m;
            if (__any_sync(0xffffffffu, grow)) {
                const float mn = grow ? mx + REF_STEP : m, alpha = grow ? exp2f(m - mn) : 1.f;
                m = mn;
                l *= alpha;
#pragma unroll
                for (int h = 0; h < GH; ++h) {
                    const float a = __shfl_sync(0xffffffffu, alpha, lb + h * RL * REP);
                    const uint64_t a2 = pack2(a, a);
#pragma unroll
                    for (int e = 0; e < N / 2; ++e) acc[h][e] = ffma2(acc[h][e], a2, 0ull);
                }
            }
#pragma unroll
            for (int i = 0; i < CNT; ++i) {
                p[i] = p[i] == -INFINITY ? 0.f : exp2f(p[i] - m);
                l += p[i];
            }
#pragma unroll
            for (int i = 0; i < RPI; ++i) {
                uint4 raw = sv[i * LPR];
                if (i >= live) raw = make_uint4(0, 0, 0, 0);       // (a stage's unwritten rows may hold anything)
                float f[N];
                Vec<T>::unpack(raw, f);
#pragma unroll
                for (int h = 0; h < GH; ++h) {
                    const float a = __shfl_sync(0xffffffffu, p[i % CNT], lb + (h * RL + i / CNT) * REP);
                    const uint64_t a2 = pack2(a, a);
#pragma unroll
                    for (int e = 0; e < N / 2; ++e) acc[h][e] = ffma2(a2, pack2(f[2 * e], f[2 * e + 1]), acc[h][e]);
                }
            }
            __syncwarp();
            if (wl == 0) mbar_arrive(&empty[s]);
        }
        // ---- piece end: the warp's groups, then the warps, in a fixed order
#pragma unroll
        for (int o = REP; o < REP * RL; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        float M = m;
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        const float wgt = rescale(m, M);
        l *= wgt;
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (g == 0 && lane == head * RL * REP) { sm_m[warp][head] = M; sm_l[warp][head] = l; }
#pragma unroll
        for (int h = 0; h < GH; ++h) {
            const float a = __shfl_sync(0xffffffffu, wgt, lb + h * RL * REP);
#pragma unroll
            for (int e = 0; e < N / 2; ++e) {
                float x[2];
                unpack2(acc[h][e], x[0], x[1]);
#pragma unroll
                for (int z = 0; z < 2; ++z) {
                    x[z] *= a;
#pragma unroll
                    for (int o = LPR; o < 32; o <<= 1) x[z] += __shfl_xor_sync(0xffffffffu, x[z], o);
                }
                if (g == 0) *reinterpret_cast<float2*>(sm_acc + (warp * GH + h) * D + lane * N + 2 * e) = make_float2(x[0], x[1]);
            }
        }
        named_bar(1, ATT_WARPS * 32);
        store_piece<D, GH>(sm_m, sm_l, sm_acc, s_bad != 0, CL ? fin : piece_slot(w, it, part, pieces, max_pieces, GH * (D + 2)), GH);
        named_bar(1, ATT_WARPS * 32);
        w.f += it.cnt;
    }
    if (CL) join_cluster<D>(fin, item, w.HG, GH, G, C, out);
}

// ------------------------------------------------------------------ bf16 caches: the same on warp-level matrix products
// With bf16 rows the FMA kernel spends 420 instructions per warp and stage on unpacking, multiplying and shuffling; the
// matrix instructions take a fifth of that, and up to eight query heads for the price of one.  (The work is a stream of
// K and V past a handful of queries: bandwidth-bound, so the warp-level instructions' rate is no limit, and their
// operands need neither tensor memory nor a barrier between the two products.)
//   S = K q^T   16 rows x 8 heads per product chain (K rows as they lie, q as the constant operand)
//   O^T += V^T P  16 channels x 8 heads per product; P enters as three bf16 terms (24 bits, exact), V is bf16 already,
//               and every 16 rows' products start from zero and are added in fp32, so that nothing is rounded earlier
//               than in fp32 arithmetic.  The terms are all positive, so that an infinite V times any weight is infinite
//               as in fp32 arithmetic (a term that is zero or negative would make it NaN)
// Rows come by TMA with the 128-byte swizzle (ldmatrix without bank conflicts).
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t transpose8x8(uint32_t x) {
    uint32_t r;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(x));
    return r;
}

// Takes the largest bf16 number below x out of x (8 bits; what is left is exact), but at least `least`.  Three of these
// use up a positive fp32 number without ever leaving zero: 1 = 255/256 + 255/65536 + 1/65536.  (x = 0 with least = 0: 0.)
__device__ __forceinline__ uint32_t take_bf16(float& x, float least) {
    const float t = fmaxf(__uint_as_float((__float_as_uint(x) - 1u) & 0xffff0000u), least);
    x -= t;
    return __float_as_uint(t);
}

constexpr int MMA_GH = 8;                   // query heads of a product

template <int D, bool CL>
__global__ void __launch_bounds__(ATT_NT, 1)
attend_partial_mma_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                          const __nv_bfloat16* __restrict__ q, const int32_t* __restrict__ len, float* __restrict__ part,
                          int32_t* __restrict__ pieces, int rows, int G, int U, int max_pieces, float scale_log2e, int C, float* __restrict__ out) {
    constexpr int KCH = D / 64;                                    // 64-channel (128-byte) column chunks
    constexpr int SROWS = ATT_STAGE_BYTES / (D * 2);               // rows per stage (64 or 128)
    constexpr int CHUNK = SROWS * 128;                             // bytes of a column chunk of a stage
    constexpr int NB = SROWS / 16;                                 // 16-row blocks per stage, one per warp
    static_assert(ATT_WARPS % NB == 0, "stages are dealt to whole sets of NB warps");
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* ring = smem_raw + (base - smem_u32(smem_raw));        // [stage][K | V][KCH][SROWS][128 B]
    float* sm_acc = reinterpret_cast<float*>(ring + ATT_STAGES * 2 * ATT_STAGE_BYTES);   // [warp][MMA_GH][D]
    float* fin = sm_acc + ATT_WARPS * MMA_GH * D;                  // [MMA_GH][D + 2]: this block's state (clusters)
    __shared__ __align__(8) uint64_t full[ATT_STAGES], empty[ATT_STAGES];
    __shared__ float sm_m[ATT_WARPS][MMA_GH], sm_l[ATT_WARPS][MMA_GH];
    __shared__ ShareSmem sh;
    __shared__ volatile int s_bad;

    const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
    const int stride = min(G, MMA_GH);                             // heads a piece's state is laid out for
    Work w;
    w.len = len; w.rows = rows; w.HG = (G + MMA_GH - 1) / MMA_GH; w.items = U * w.HG; w.pad = CL ? 0 : item_rows(D, 2);
    if (threadIdx.x == 0) {
        for (int i = 0; i < ATT_STAGES; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], NB);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_bad = 0;
    }
    grid_dependency_wait();
    Item it;
    if (CL) take_slice<D, MMA_GH>(w, it, C, fin);
    else if (!take_share(w, it, sh)) return;
    const int item = it.id;

    if (warp == ATT_WARPS) {
        // ---- copies (a stage's rows past the piece are rows of the next pieces, or zeros past the tensor: masked)
        if (wl == 0) {
            uint32_t k = 0;
            bool ok = true;
            while (ok && w.settle(it)) {
                const int r0 = it.off, u = it.id / w.HG;
                for (int r = 0; r < it.cnt; r += SROWS, ++k) {
                    const int s = k % ATT_STAGES;
                    ok = mbar_wait(&empty[s], ((k / ATT_STAGES) & 1) ^ 1, &s_bad);
                    if (!ok) break;
#ifdef KVM_TEST_DROP_ATTEND_STAGE
                    if (blockIdx.x == KVM_TEST_DROP_CTA && k == (uint32_t)(KVM_TEST_DROP_ATTEND_STAGE)) continue;   // test build only: this stage never arrives
#endif
                    mbar_expect_tx(&full[s], 2 * ATT_STAGE_BYTES);
                    uint8_t* st = ring + s * 2 * ATT_STAGE_BYTES;
#pragma unroll
                    for (int c = 0; c < KCH; ++c) {
                        tma_load_3d(st + c * CHUNK, &map_k, &full[s], c * 64, r0 + r, u);
                        tma_load_3d(st + ATT_STAGE_BYTES + c * CHUNK, &map_v, &full[s], c * 64, r0 + r, u);
                    }
                }
                w.f += it.cnt;
            }
            drain(full, k);
        }
        if (!CL) return;
        __syncwarp();
    }
    // ---- arithmetic.  gid, tig: row and column pair of this lane in the 8x8 fragments
    const int gid = wl >> 2, tig = wl & 3, blk = warp % NB;
    const int sset = warp / NB;                                    // takes the stages k with k % (ATT_WARPS / NB) == sset
    // ldmatrix addresses: K rows 0..15 x two 16-byte pieces; V (transposed) rows 0..7, 8..15 x two pieces
    const int krow = blk * 16 + (wl & 15), kpc = wl >> 4;
    const int vrow = blk * 16 + (wl & 7) + ((wl >> 4) << 3), vpc = (wl >> 3) & 1;
    uint32_t k = 0;
    while (warp != ATT_WARPS && w.settle(it)) {
        const int u = it.id / w.HG, h0 = (it.id % w.HG) * MMA_GH, heads = min(G - h0, MMA_GH);
        uint32_t qf[D / 16][2];                                    // q^T as B fragments: channels 2 tig.. (+8), head gid
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
#pragma unroll
            for (int x = 0; x < 2; ++x)
                qf[ks][x] = gid < heads ? __ldg(reinterpret_cast<const uint32_t*>(q + ((size_t)u * G + h0 + gid) * D + ks * 16 + x * 8) + tig) : 0u;
        float o[D / 16][4];                                        // channel dt * 16 + gid (+8), heads 2 tig, 2 tig + 1
#pragma unroll
        for (int dt = 0; dt < D / 16; ++dt)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[dt][e] = 0.f;
        float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};    // of heads 2 tig, 2 tig + 1 (l: of this lane's rows)
        for (int r = 0; r < it.cnt; r += SROWS, ++k) {
            if ((int)(k % (ATT_WARPS / NB)) != sset) continue;
            const int s = k % ATT_STAGES;
            // (the block's own copies always complete; a wait that ran out all the same makes the outputs NaN)
            if (!__all_sync(0xffffffffu, mbar_wait(&full[s], (k / ATT_STAGES) & 1, &s_bad))) break;
            const int live = it.cnt - r - blk * 16;                // rows of the block that exist
            if (live > 0) {
                const uint32_t kb = base + s * 2 * ATT_STAGE_BYTES, vb = kb + ATT_STAGE_BYTES;
                float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    uint32_t a[4];
                    ldsm4(a, kb + (ks / 4) * CHUNK + krow * 128 + ((((ks % 4) * 2 + kpc) ^ (krow & 7)) << 4));
                    mma16816(ks & 1 ? c1 : c0, a, qf[ks][0], qf[ks][1]);
                }
                float x[4];                                        // rows gid, gid + 8 x heads 2 tig, 2 tig + 1
#pragma unroll
                for (int e = 0; e < 4; ++e) x[e] = gid + (e >> 1) * 8 < live ? (c0[e] + c1[e]) * scale_log2e : -INFINITY;
                const float mx[2] = {fmaxf(x[0], x[2]), fmaxf(x[1], x[3])};
                if (__any_sync(0xffffffffu, mx[0] > m[0] || mx[1] > m[1])) {
                    float alpha[2];
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        float t = mx[y];
#pragma unroll
                        for (int z = 4; z < 32; z <<= 1) t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, z));
                        const float mn = t > m[y] ? t + REF_STEP : m[y];
                        alpha[y] = rescale(m[y], mn);
                        m[y] = mn;
                        l[y] *= alpha[y];
                    }
#pragma unroll
                    for (int dt = 0; dt < D / 16; ++dt)
#pragma unroll
                        for (int e = 0; e < 4; ++e) o[dt][e] *= alpha[e & 1];
                }
                // weights, as three bf16 terms each, in the B operand's layout (rows 2 tig.. of head gid)
                float p[4], least[4];                              // (least: the smallest bf16 number, 0 for a weight of 0)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    p[e] = rescale(x[e], m[e & 1]);
                    l[e & 1] += p[e];
                    least[e] = p[e] > 0.f ? __uint_as_float(0x00010000u) : 0.f;
                }
                uint32_t pb[3][2];
#pragma unroll
                for (int t = 0; t < 3; ++t)
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        const uint32_t lo = take_bf16(p[2 * y], least[2 * y]), hi = take_bf16(p[2 * y + 1], least[2 * y + 1]);
                        pb[t][y] = transpose8x8(__byte_perm(lo, hi, 0x7632));
                    }
                // rows that do not exist may hold anything: their V becomes zero (masks of the operand's rows 2 tig.. + 8)
                uint32_t mask[2] = {0xffffffffu, 0xffffffffu};
                if (live < 16)
#pragma unroll
                    for (int y = 0; y < 2; ++y)
                        mask[y] = (2 * tig + y * 8 < live ? 0xffffu : 0u) | (2 * tig + 1 + y * 8 < live ? 0xffff0000u : 0u);
#pragma unroll
                for (int dt = 0; dt < D / 16; ++dt) {
                    uint32_t a[4];
                    ldsm4_t(a, vb + (dt / 4) * CHUNK + vrow * 128 + ((((dt % 4) * 2 + vpc) ^ (vrow & 7)) << 4));
                    if (live < 16) { a[0] &= mask[0]; a[1] &= mask[0]; a[2] &= mask[1]; a[3] &= mask[1]; }
                    float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int t = 2; t >= 0; --t) mma16816(c, a, pb[t][0], pb[t][1]);
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[dt][e] += c[e];
                }
            }
            __syncwarp();
            if (wl == 0) mbar_arrive(&empty[s]);
        }
#pragma unroll
        for (int y = 0; y < 2; ++y)
#pragma unroll
            for (int z = 4; z < 32; z <<= 1) l[y] += __shfl_xor_sync(0xffffffffu, l[y], z);
        if (gid == 0) {
            sm_m[warp][2 * tig] = m[0]; sm_m[warp][2 * tig + 1] = m[1];
            sm_l[warp][2 * tig] = l[0]; sm_l[warp][2 * tig + 1] = l[1];
        }
#pragma unroll
        for (int dt = 0; dt < D / 16; ++dt)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (2 * tig + (e & 1) < heads) sm_acc[(warp * MMA_GH + 2 * tig + (e & 1)) * D + dt * 16 + gid + (e >> 1) * 8] = o[dt][e];
        named_bar(1, ATT_WARPS * 32);
        store_piece<D, MMA_GH>(sm_m, sm_l, sm_acc, s_bad != 0,
                               CL ? fin : piece_slot(w, it, part, pieces, max_pieces, stride * (D + 2)), heads);
        named_bar(1, ATT_WARPS * 32);
        w.f += it.cnt;
    }
    if (CL) join_cluster<D>(fin, item, w.HG, MMA_GH, G, C, out);
}

// ------------------------------------------------------------------ short units in numbers: small blocks, several per SM
// An item costs a persistent block about 3 us beside its rows (lengths, queries, the joining of its warps, one after the
// other), which nothing hides where the items are short and many.  Here every (query head, chunk of rows) is a block of its
// own, four to an SM: a group of LPR lanes takes four rows at a time from memory straight into registers.  The query heads
// of a KV head read its rows one by one (through L2), which is why this form is for few of them.
constexpr int ROW_NT = 256, ROW_BLOCKS_PER_SM = 4;
constexpr int ROW_MIN_CHUNK = 64;           // fewest rows of a chunk (bounds the number of pieces)
template <typename T, int D>
__global__ void __launch_bounds__(ROW_NT) attend_partial_rows_kernel(const T* __restrict__ q, const T* __restrict__ K,
                                                                     const T* __restrict__ V, const int32_t* __restrict__ len,
                                                                     float* __restrict__ part, int32_t* __restrict__ pieces,
                                                                     int rows, int chunk, int G, float scale_log2e) {
    constexpr int N = Vec<T>::N, LPR = D / N, NGRP = ROW_NT / LPR;
    __shared__ float sm_m[NGRP], sm_l[NGRP];
    __shared__ __align__(16) float sm_acc[NGRP][D];
    const int split = blockIdx.x, bh = blockIdx.y, u = bh / G;     // b * Hq + h = unit * G + head of the group
    grid_dependency_wait();
    const int n = len ? max(0, min(len[u], rows)) : rows;
    const int r0 = split * chunk, r1 = min(r0 + chunk, n);
    const int grp = threadIdx.x / LPR, lane = threadIdx.x % LPR;
    const unsigned gmask = (LPR == 32) ? 0xffffffffu : (((1u << LPR) - 1u) << ((threadIdx.x % 32) / LPR * LPR));
    const T* Ku = K + (size_t)u * rows * D;
    const T* Vu = V + (size_t)u * rows * D;
    float qf[N];
    Vec<T>::unpack(ldg16(q + (size_t)bh * D + lane * N), qf);
    float m = -INFINITY, l = 0.f, acc[N];
#pragma unroll
    for (int e = 0; e < N; ++e) acc[e] = 0.f;
    for (int r = r0 + grp * RPI; r < r1; r += NGRP * RPI) {
        uint4 kraw[RPI], vraw[RPI];
#pragma unroll
        for (int i = 0; i < RPI; ++i) {
            const int ri = min(r + i, r1 - 1);                     // clamped rows are loaded but given no weight
            kraw[i] = ldg16(Ku + (size_t)ri * D + lane * N);
            vraw[i] = ldg16(Vu + (size_t)ri * D + lane * N);
        }
        float s[RPI];
#pragma unroll
        for (int i = 0; i < RPI; ++i) {
            float kf[N];
            Vec<T>::unpack(kraw[i], kf);
            s[i] = 0.f;
#pragma unroll
            for (int e = 0; e < N; ++e) s[i] = fmaf(qf[e], kf[e], s[i]);
        }
#pragma unroll
        for (int off = 1; off < LPR; off <<= 1)
#pragma unroll
            for (int i = 0; i < RPI; ++i) s[i] += __shfl_xor_sync(gmask, s[i], off);
        float mn = m;
#pragma unroll
        for (int i = 0; i < RPI; ++i) {
            s[i] = r + i < r1 ? s[i] * scale_log2e : -INFINITY;
            mn = fmaxf(mn, s[i]);
        }
        const float corr = rescale(m, mn);
        l *= corr;
#pragma unroll
        for (int e = 0; e < N; ++e) acc[e] *= corr;
#pragma unroll
        for (int i = 0; i < RPI; ++i) {
            const float p = rescale(s[i], mn);                     // 0 for a clamped row
            float vf[N];
            if (r + i >= r1) vraw[i] = make_uint4(0, 0, 0, 0);
            Vec<T>::unpack(vraw[i], vf);
            l += p;
#pragma unroll
            for (int e = 0; e < N; ++e) acc[e] = fmaf(p, vf[e], acc[e]);
        }
        m = mn;
    }
    if (lane == 0) { sm_m[grp] = m; sm_l[grp] = l; }
#pragma unroll
    for (int e = 0; e < N; ++e) sm_acc[grp][lane * N + e] = acc[e];
    __syncthreads();
    if (threadIdx.x < D) {
        float M = -INFINITY, L = 0.f, o = 0.f;
#pragma unroll
        for (int g = 0; g < NGRP; ++g) M = fmaxf(M, sm_m[g]);
#pragma unroll
        for (int g = 0; g < NGRP; ++g) {
            const float w = rescale(sm_m[g], M);
            L = fmaf(sm_l[g], w, L);
            o = fmaf(sm_acc[g][threadIdx.x], w, o);
        }
        float* dst = part + ((size_t)bh * gridDim.x + split) * (D + 2);
        dst[threadIdx.x] = o;
        if (threadIdx.x == 0) {
            dst[D] = M; dst[D + 1] = L;
            if (split == 0) pieces[bh] = gridDim.x;
        }
    }
}

// One block per query head: its pieces' states in order.
template <int D>
__global__ void __launch_bounds__(D) attend_combine_kernel(const float* __restrict__ part, const int32_t* __restrict__ pieces,
                                                           const int32_t* __restrict__ len, float* __restrict__ out, int rows,
                                                           int G, int gh, int max_pieces) {
    const int u = blockIdx.x / G, h = blockIdx.x % G;              // b * Hq + h = unit * G + head of the group
    const int item = u * ((G + gh - 1) / gh) + h / gh;
    grid_dependency_wait();     // the partial states come from the kernel before this one
    const int n = len ? min(__ldg(len + u), rows) : rows;
    float o = 0.f, L = 0.f;
    if (n > 0) {                                                   // an empty cache attends to nothing
        const int np = __ldcg(pieces + item);
        const float* p = part + ((size_t)item * max_pieces * gh + h % gh) * (D + 2);
        float M = -INFINITY;
        // the next `count` pieces: their loads leave together
        auto join = [&](auto count, int s0) {
            constexpr int NB = decltype(count)::value;
            float ms[NB], ls[NB], os[NB], mn = M;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const float* ps = p + (size_t)(s0 + i) * gh * (D + 2);
                const bool in = s0 + i < np;
                ms[i] = in ? __ldcg(ps + D) : -INFINITY;
                ls[i] = in ? __ldcg(ps + D + 1) : 0.f;
                os[i] = in ? __ldcg(ps + threadIdx.x) : 0.f;
                mn = fmaxf(mn, ms[i]);
            }
            const float a = rescale(M, mn);
            L *= a;
            o *= a;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const float c = rescale(ms[i], mn);
                L = fmaf(ls[i], c, L);
                o = fmaf(os[i], c, o);
            }
            M = mn;
        };
        // (one unit of 8192 rows is cut into 128 pieces: four at a time they took 27 us to join; where there are many units
        // of one or two pieces sixteen at a time cost 6 us more on 2560 heads)
        if (np <= 2) join(std::integral_constant<int, 2>{}, 0);
        else
            for (int s0 = 0; s0 < np; s0 += 16) join(std::integral_constant<int, 16>{}, s0);
    }
    out[(size_t)blockIdx.x * D + threadIdx.x] = L > 0.f || L != L || o != o ? o / L : 0.f;   // (o alone is NaN where every piece gave up)
}

// err = |O - O*|_2 and ref = |O|_2 per (batch, query head).
template <int D>
__global__ void __launch_bounds__(D) perturbation_kernel(const float* __restrict__ O, const float* __restrict__ Os,
                                                         float* __restrict__ err, float* __restrict__ ref) {
    __shared__ float se[D / 32], sr[D / 32];
    grid_dependency_wait();     // both attention outputs come from the kernels before this one
    const int bh = blockIdx.x;
    const float a = O[(size_t)bh * D + threadIdx.x], c = Os[(size_t)bh * D + threadIdx.x];
    float e = (a - c) * (a - c), r = a * a;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        e += __shfl_xor_sync(0xffffffffu, e, off);
        r += __shfl_xor_sync(0xffffffffu, r, off);
    }
    if ((threadIdx.x & 31) == 0) { se[threadIdx.x >> 5] = e; sr[threadIdx.x >> 5] = r; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float te = 0.f, tr = 0.f;
#pragma unroll
        for (int w = 0; w < D / 32; ++w) { te += se[w]; tr += sr[w]; }
        err[bh] = sqrtf(te);
        ref[bh] = sqrtf(tr);
    }
}

// Query heads that share a pass over the rows.
inline int head_group(const Dims& d) {
    if (d.dtype == KVM_BF16) return d.G < MMA_GH ? d.G : MMA_GH;
    return d.G >= 5 ? 8 : (d.G >= 3 ? 4 : d.G);
}
// Pieces an item can fall into: shares are at least ATT_MIN_SHARE rows.
inline int most_pieces(int rows) { return (rows + ATT_MIN_SHARE - 2) / ATT_MIN_SHARE + 1; }

// What the current device holds of a kernel's two forms at a time: SMs, and clusters of 1, 2, 4 and 8 blocks (a cluster
// lies within a GPC, whose SMs eight rarely divides: 15 clusters of eight, 33 of four on 148 SMs).
struct Room {
    int sms = 0, clusters[4] = {};
};
// Finds it out once per device, together with the shared-memory opt-in.
template <typename KC, typename KS>
cudaError_t prepare_forms(KC clustered, KS shares, int smem, Room (&room_of)[KVM_MAX_DEVICES], std::mutex& mu, Room& room) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= KVM_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!room_of[dev].sms) {
        Room r;
        if ((e = cudaFuncSetAttribute(shares, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
        if ((e = cudaFuncSetAttribute(clustered, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&r.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        for (int i = 0; i < 4; ++i) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(r.sms << i));
            cfg.blockDim = dim3(ATT_NT);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 1u << i;
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if ((e = cudaOccupancyMaxActiveClusters(&r.clusters[i], clustered, &cfg)) != cudaSuccess) return e;
        }
        room_of[dev] = r;
    }
    room = room_of[dev];
    return cudaSuccess;
}

// The small blocks: as many chunks per query head as keep every SM's blocks busy in one wave.
template <typename T, int D>
cudaError_t launch_rows(const Dims& d, const void* q, const void* K, const void* V, int rows, const int32_t* len, float* out,
                        float* part, int sms, cudaStream_t st) {
    const int heads = d.B * d.Hq, most = (rows + ROW_MIN_CHUNK - 1) / ROW_MIN_CHUNK;
    int want = ROW_BLOCKS_PER_SM * sms / heads;
    want = want < 1 ? 1 : want > most ? most : want;
    const int chunk = (rows + want - 1) / want, n = (rows + chunk - 1) / chunk;
    int32_t* pieces = reinterpret_cast<int32_t*>(part);
    float* states = part + (heads + 3) / 4 * 4;
    const cudaError_t e = launch_dependent(attend_partial_rows_kernel<T, D>, dim3(n, heads), dim3(ROW_NT), 0, st, (const T*)q,
                                           (const T*)K, (const T*)V, len, states, pieces, rows, chunk, d.G, d.scale * LOG2E);
    if (e != cudaSuccess) return e;
    return launch_dependent(attend_combine_kernel<D>, dim3(heads), dim3(D), 0, st, (const float*)states, (const int32_t*)pieces,
                            len, out, rows, d.G, 1, n);
}

// How a call is dealt: clusters of `cluster` blocks per item, small blocks per query head and chunk (`rows`), or, with
// neither, equal shares.
struct Form {
    int cluster = 0;
    bool rows = false;
};

struct Scratch {
    int items, gh, mp;
    float* part;            // the scratch; laid out for the two large forms:
    int32_t* pieces;
    float *states, *out;
    unsigned grid(int sms, int rows, int row_bytes) const {
        const long long most = ((long long)items * (rows + ATT_ITEM_BYTES / row_bytes) + ATT_MIN_SHARE - 1) / ATT_MIN_SHARE;
        return (unsigned)(most < sms ? most : sms);
    }
    // The form that is fastest for full units (lengths are on the device), shares where it is close: they follow the lengths.
    // Measured in us, bf16, D = 128 unless said otherwise; clusters / shares / small blocks.
    //   No more items than blocks: by estimates (`block`: bytes/ns that a block of the two large forms gets through, 6.5 TB/s
    // together): a slice of an item, all clusters being at work at the same time; all rows, a second kernel and the pieces
    // of an item; every query head's rows through L2, a second kernel and the pieces of a head.  1 unit x 8192 rows 11.6 /
    // 14.6 / 13.1, 1 x 32768 32 / 20 / 44, 16 x 8192 20.3 (clusters of four) and 25.9 (of eight, of which 15 fit) / 19.0 / 21,
    // 32 x 2048 10.5 / 12.2 / 11.6, 64 x 16384 half full 72 / 65 / -, one unit of eight fp32 heads x 8192 32 / 18 / 16.
    //   More items: small blocks while what they save, the items' cost, exceeds their way through L2 per query head.  One
    // head: - / 107 / 77 (4096 x 200), 50.5 / 49.0 (1024 x 512), 33 / 34 (320 x 1024), 57 / 61 (320 x 2048); in fp32 42 / 41
    // (1024 x 200), 85 / 93 (1024 x 512).  Two heads: 35.5 / 34.5 (1024 x 200), 54 / 64 (1024 x 512).  Four: 10.1 / 8.2 (160 x
    // 48), 12.1 / 15.2 (160 x 200), 107 / 110 (4096 x 48).
    Form choose(const Room& room, const Dims& d, int rows, int row_bytes, double block) const {
        Form f;
        const int heads = d.B * d.Hq, sms = room.sms;
        const double unit = rows * (double)row_bytes;
        if (items > sms) {
            f.rows = (d.G * unit <= 208.0 * 1024 && (d.G <= 2 || heads <= 9 * sms)) ||
                     (d.dtype == KVM_BF16 && d.G == 1 && unit <= 512.0 * 1024);
            return f;
        }
        const double most = (rows + ATT_MIN_SHARE - 1) / ATT_MIN_SHARE;
        auto pieces = [&](double n) { return n < most ? n : most; };
        const double all = sms * block < 6500.0 ? sms * block : 6500.0, l2 = d.G == 1 ? 5800.0 : d.G == 2 ? 7700.0 : 9000.0;
        const double shares = 7.0 + items * unit / 1e3 / all + 0.055 * pieces((double)sms / items);
        const double small = 6.8 + heads * unit / 1e3 / l2 + 0.06 * pieces((double)ROW_BLOCKS_PER_SM * sms / heads);
        int i = 3;
        while (i > 0 && items > room.clusters[i]) --i;
        const int C = 1 << i;
        const double part = 6500.0 / (items * C);
        const double cluster = 4.8 + (rows + C - 1) / C * (double)row_bytes / 1e3 / (part < block ? part : block);
        if (cluster * 1.06 < shares && cluster < small) f.cluster = C;
        else f.rows = small < shares;
        return f;
    }
};

// One of a kernel's two forms on the stream.
template <int D, typename KC, typename KS, typename... Args>
cudaError_t launch_form(KC clustered, KS shares, const Dims& d, const Scratch& sc, const Room& room, const Form& f, int smem, int rows,
                        int row_bytes, const int32_t* len, cudaStream_t st, Args... args) {
    if (f.cluster)
        return launch_dependent_cluster(clustered, dim3(sc.items * f.cluster), dim3(ATT_NT), smem, f.cluster, st, args..., f.cluster, sc.out);
    const cudaError_t e = launch_dependent(shares, dim3(sc.grid(room.sms, rows, row_bytes)), dim3(ATT_NT), smem, st, args..., 0, sc.out);
    if (e != cudaSuccess) return e;
    return launch_dependent(attend_combine_kernel<D>, dim3(d.B * d.Hq), dim3(D), 0, st, (const float*)sc.states,
                            (const int32_t*)sc.pieces, len, sc.out, rows, d.G, sc.gh, sc.mp);
}

template <typename T, int D, int GH>
cudaError_t launch_fma(const Dims& d, const void* q, const void* K, const void* V, int rows, const int32_t* len,
                       const Scratch& sc, cudaStream_t st) {
    constexpr int smem = ATT_STAGES * 2 * ATT_STAGE_BYTES + (ATT_WARPS * D + D + 2) * GH * (int)sizeof(float);
    constexpr int row_bytes = 2 * D * (int)sizeof(T);
    constexpr double block = GH == 1 ? 80.0 : GH == 2 ? 72.0 : GH == 4 ? 56.0 : 40.0;
    const auto clustered = attend_partial_fma_kernel<T, D, GH, true>;
    const auto shares = attend_partial_fma_kernel<T, D, GH, false>;
    static std::mutex mu;
    static Room room_of[KVM_MAX_DEVICES];
    Room room;
    const cudaError_t e = prepare_forms(clustered, shares, smem, room_of, mu, room);
    if (e != cudaSuccess) return e;
    const Form f = sc.choose(room, d, rows, row_bytes, block);
    if (f.rows) return launch_rows<T, D>(d, q, K, V, rows, len, sc.out, sc.part, room.sms, st);
    return launch_form<D>(clustered, shares, d, sc, room, f, smem, rows, row_bytes, len, st, (const T*)q, (const T*)K, (const T*)V,
                          len, sc.states, sc.pieces, rows, d.G, d.U, sc.mp, d.scale * LOG2E);
}
template <int D>
cudaError_t launch_mma(const Dims& d, const void* q, const void* K, const void* V, int rows, const int32_t* len,
                       const Scratch& sc, cudaStream_t st) {
    constexpr int smem = 1024 + ATT_STAGES * 2 * ATT_STAGE_BYTES + (ATT_WARPS * D + D + 2) * MMA_GH * (int)sizeof(float);
    constexpr int row_bytes = 4 * D;
    constexpr double block = D == 128 ? 72.0 : 56.0;
    const auto clustered = attend_partial_mma_kernel<D, true>;
    const auto shares = attend_partial_mma_kernel<D, false>;
    static std::mutex mu;
    static Room room_of[KVM_MAX_DEVICES];
    Room room;
    const cudaError_t e = prepare_forms(clustered, shares, smem, room_of, mu, room);
    if (e != cudaSuccess) return e;
    const Form f = sc.choose(room, d, rows, row_bytes, block);
    if (f.rows) return launch_rows<__nv_bfloat16, D>(d, q, K, V, rows, len, sc.out, sc.part, room.sms, st);
    CUtensorMap mk, mv;
    if (!make_map(&mk, K, d.U, rows, D, ATT_STAGE_BYTES / (2 * D)) || !make_map(&mv, V, d.U, rows, D, ATT_STAGE_BYTES / (2 * D)))
        return cudaErrorNotSupported;
    return launch_form<D>(clustered, shares, d, sc, room, f, smem, rows, row_bytes, len, st, mk, mv, (const __nv_bfloat16*)q, len,
                          sc.states, sc.pieces, rows, d.G, d.U, sc.mp, d.scale * LOG2E);
}

template <int D>
cudaError_t launch_t(const Dims& d, const void* q, const void* K, const void* V, int rows, const int32_t* len, float* out,
                     float* part, cudaStream_t st) {
    Scratch sc;
    sc.gh = head_group(d);
    sc.items = d.U * ((d.G + sc.gh - 1) / sc.gh);
    sc.mp = most_pieces(rows);
    sc.part = part;
    sc.pieces = reinterpret_cast<int32_t*>(part);
    sc.states = part + (sc.items + 3) / 4 * 4;
    sc.out = out;
    auto fn = d.dtype == KVM_BF16 ? launch_mma<D>
              : sc.gh == 1        ? launch_fma<float, D, 1>
              : sc.gh == 2        ? launch_fma<float, D, 2>
              : sc.gh == 4        ? launch_fma<float, D, 4>
                                  : launch_fma<float, D, 8>;
    return fn(d, q, K, V, rows, len, sc, st);
}

}  // namespace

// The pieces' states and their counts, in the form that needs more.
size_t attend_scratch_floats(const Dims& d) {
    const int gh = head_group(d);
    const size_t items = (size_t)d.U * ((d.G + gh - 1) / gh);
    const size_t shares = (items + 3) / 4 * 4 + items * most_pieces(d.S) * gh * (d.D + 2), heads = (size_t)d.B * d.Hq;
    const size_t small = (heads + 3) / 4 * 4 + heads * ((d.S + ROW_MIN_CHUNK - 1) / ROW_MIN_CHUNK) * (d.D + 2);
    return shares > small ? shares : small;
}

cudaError_t launch_attend(const Dims& d, const void* q, const void* K, const void* V, int rows, const int32_t* len,
                          float* out, float* part, cudaStream_t st) {
    return d.D == 128 ? launch_t<128>(d, q, K, V, rows, len, out, part, st) : launch_t<64>(d, q, K, V, rows, len, out, part, st);
}

cudaError_t launch_perturbation(const Dims& d, const float* O, const float* Os, float* err, float* ref,
                                cudaStream_t st) {
    if (d.D == 128) return launch_dependent(perturbation_kernel<128>, dim3(d.B * d.Hq), dim3(128), 0, st, O, Os, err, ref);
    return launch_dependent(perturbation_kernel<64>, dim3(d.B * d.Hq), dim3(64), 0, st, O, Os, err, ref);
}

}  // namespace kvm
