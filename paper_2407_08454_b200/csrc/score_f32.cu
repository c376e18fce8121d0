// Aggregated attention scores of fp32 tensors on the tensor cores, without giving up fp32 inputs:
//   pass 1 (row pass)     lse_i = ln sum_{j<=i} exp(c q_i.k_j)                       Eq. 1, causal
//   pass 2 (column pass)  a_j   = (1/G) sum_g sum_{i>=j} exp(c q^g_i.k_j - lse^g_i)  Algorithm 2 / Eq. 6, Section 5.2
//
// What bounds it: the tensor pipe, by six bf16 products per logit.  An fp32 number is the exact sum of three bf16
// numbers, x = h + m + l (8 significant bits each, every residual is exact), so q.k is nine bf16 products; the three
// smallest (m.l, l.m, l.l: together below 2^-26 of |q||k|) are left out.  h.h goes into one TMEM accumulator (D / 16
// additions), the five smaller products into a second one, and the epilogue adds the two: the large accumulator is
// rounded no more often than a plain fp32 loop's would be, and the small one's rounding is 2^-8 of that.  Against fp64
// (random Gaussian rows, D = 128) the logits' error is that of the FMA loop this kernel replaces: the test compares.
//
// One CTA per SM, persistent, warp-specialised:
//   warps 0-7   epilogue: two groups of four (one warp per TMEM lane quarter) take alternate steps
//   warps 8-14  converters: read fp32 rows (L2 for all but the first touch), split them and write the three planes
//               in the layout the tensor core reads (128-byte rows, 128-byte swizzle); no split copy of Q or K ever
//               exists in global memory, so the pass needs no workspace for it and moves no extra bytes
//   warp  15    MMA issue: the warp walks and waits together, one elected lane issues; owns tensor memory
// As in the bf16 kernel a work item is a 128-row A tile (queries in pass 1, keys in pass 2) with all the B tiles it
// meets under the causal mask, A rows are TMEM lanes, and a thread owns a row (pass 1) or column (pass 2) of the map.
//
// Split of the work: a step (one 128 x 128 logit tile) costs ~24 D clocks and there are few of them in the sizes
// fp32 layers come in (40 for 4 heads x 512 tokens, 4800 for 16 x 2999), so items are not dealt whole: the steps of all
// items form one list and every CTA takes q = ceil(steps / 148) consecutive ones, which is balanced to one step.  An
// item that is cut leaves one partial state per piece: (max, sum) per query row, joined by a kernel between the passes or, where
// those are few, by the steps that read them (join_between below), or a partial column sum per key, added in piece order
// by combine_kernel (or by the segment kernel that follows in a compress call).  Where the pieces' states would not fit
// 4 MiB (large problems, where whole items balance well anyway) items stay whole and the states are final.  The rule
// depends on the shape only: results are reproducible.
//
// Measured on a B200 (us, row / column pass; FMA tiles before): 16 / 8 heads x 2999 tokens x 128 1300 / 1890 -> 105 / 107;
// 32 heads x 4096 x 128 351 / 377; 4 heads x 512 x 64 100 / 74 -> 9 / 9.  What bounds a step now is its 48 products: 3,340 of
// 3,960 clocks, at the clock that so busy a tensor pipe is left by the power limit.  Before, the epilogue did (two steps in
// 10,900 clocks, 5,000 of a step's 10,000 spent on joining the row pass's states): now those are joined by a kernel between
// the passes where a step would read many, asked for a step ahead, and the exponentials are single instructions.
// Tried without gain: eleven converter warps, a barrier per plane, planes split beforehand and fetched by TMA (the extra pass
// costs what the conversion costs here).
//
// Every wait on an mbarrier is bounded (see tc_common.cuh); a wait that runs out raises a flag, every role leaves its
// loops, outputs are NaN and kvm_stats.status is set when given.
#include <stddef.h>

#include <mutex>

#include "score_plan.cuh"
#include "similarity_core.cuh"
#include "tc_common.cuh"

namespace kvm {
namespace {

using namespace tc;
using plan::Plan;
using plan::Walk;
using plan::add_state;

constexpr int TILE = plan::TILE;
constexpr int KCHUNK = 64;                         // channels per 128-byte swizzled bf16 row
constexpr int NPLANE = 3;
constexpr uint32_t PLANE_BYTES = TILE * 128;       // [128 rows x 64 bf16]
constexpr uint32_t CHUNK_BYTES = NPLANE * PLANE_BYTES;
constexpr int NSTAGE = 2;                          // ring of B chunks (three planes each)
constexpr int NACC = 2;                            // accumulator pairs: 2 x (128 + 128) columns = all of TMEM
constexpr int NEPI = 8, NCONV = 7;                // warps; with the MMA warp sixteen, i.e. 128 registers a thread
constexpr int NTHREADS = (NEPI + NCONV + 1) * 32;
constexpr int SIM_RUN = 8;                         // consecutive tokens per lane group (similarities)
constexpr int NSLOT = 8;                           // piece-end buffers in rotation
// The row pass's states are joined by a kernel between the passes where an epilogue group would read this many of them one after
// the other (steps of a CTA / 2, by the pieces of a row): the launch takes 1.2 us, a state 0.2-0.4 us of every step, of which the
// step's own products hide a part (twice the channels, or a second step under way, hide more).  us a kvm_score call, read by the
// steps / joined between; D = 64: 1 head x 256 tokens (2 states) 16.2 / 17.5, 16 / 8 x 512 (3, two steps) 21.3 / 22.5, 8 / 4 x 1024 (5,
// two steps) 24.0 / 24.6, 32 x 512 (4, three steps) 28.3 / 27.6, 4 x 512 (4) 19.7 / 19.1, 1 x 700 (6) 21.7 / 19.5; D = 128: 4 x 512 (4)
// 21.5 / 22.5, 32 x 512 (4, three steps) 35.9 / 37.0, 8 / 4 x 1024 (5, two steps) 28.9 / 30.4, 16 / 8 x 700 (6) 34.6 / 34.7, 32 x 700 (6)
// 50.0 / 49.2, 4 x 2048 (10) 45.2 / 43.0, 16 / 8 x 2999 (34) 212.9 / 200.8.
bool join_between(const Plan& p, int D) {
    return (p.q + 1) / 2 * (unsigned)p.pr >= (D == 64 && p.q != 2 ? 4u : 6u);
}
constexpr size_t SPLIT_BYTES_MAX = (size_t)KVM_STATIC_SCORE_ROWS * sizeof(float);
constexpr float LOG2E = 1.4426950408889634f, LN2 = 0.6931471805599453f;

// Items are cut where the pieces' results fit 4 MiB (large problems balance well with whole ones); one rule for both passes.
size_t split_bytes(const Dims& d, const Plan& p) {
    return (size_t)p.NH * d.S * p.pieces(p.T) * sizeof(float2) + (size_t)p.U * d.S * p.pieces(p.G * p.T) * sizeof(float);
}
bool make_plan(const Dims& d, Plan& p) {
    if (!plan::make(d, p)) return false;
    if (split_bytes(d, p) <= SPLIT_BYTES_MAX) {
        p.split_row = p.split_col = 1;
        p.pr = p.pieces(p.T);
        p.pc = p.pieces(p.G * p.T);
    }
    return true;
}

struct alignas(16) Shared {
    uint64_t full_a[2], empty_a, full_b[NSTAGE], empty_b[NSTAGE], acc_full[NACC], acc_empty[NACC];
    uint32_t tmem_base;
    int abort_flag;
    int arrived[NSLOT][4];
    float part_m[NSLOT][2][TILE], part_l[NSLOT][2][TILE];
    alignas(16) float nl[NEPI][TILE];   // per epilogue warp: minus the log-sum-exp (log2 units) of the step's queries
};

static_assert(offsetof(Shared, nl) % 16 == 0, "read two at a time, in 8 bytes");

// A 128-row x 64-channel chunk of a [S, D] fp32 matrix on its way to three bf16 planes, in units of eight channels:
// unit u = t + k * (converter threads) is the eight channels u % 8 of row u / 8.
constexpr int NU = TILE * 8, UNITS = (NU + NCONV * 32 - 1) / (NCONV * 32);   // units, units per thread
struct Chunk { const float* src; int row0; };      // first channel of row 0 of the matrix; the chunk's first row
template <int D>
__device__ __forceinline__ void load_unit(float4 (&v)[2], const Chunk& c, int u, int S) {
    const int row = c.row0 + (u >> 3);
    const float4* p = reinterpret_cast<const float4*>(c.src + (size_t)row * D + (u & 7) * 8);
    const bool in = row < S && u < NU;
    v[0] = in ? __ldg(p) : make_float4(0.f, 0.f, 0.f, 0.f);
    v[1] = in ? __ldg(p + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
}
// Eight numbers rounded to bf16, those that would round to infinity to the largest finite number (the residual of fp32's
// lowest value, say, is then a number).
__device__ __forceinline__ uint32_t pack2_finite(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint4 pack_finite(const float* f) {
    return make_uint4(pack2_finite(f[0], f[1]), pack2_finite(f[2], f[3]), pack2_finite(f[4], f[5]), pack2_finite(f[6], f[7]));
}
__device__ __forceinline__ void split_unit(const float4 (&v)[2], uint8_t* dst, int u) {
    const int r = u >> 3, piece = u & 7;
    float x[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
    uint8_t* at = dst + r * 128 + ((piece ^ (r & 7)) << 4);
#pragma unroll
    for (int pl = 0; pl < NPLANE; ++pl) {
        const uint4 w = pl == 0 ? pack_finite(x) : Vec<__nv_bfloat16>::pack(x);
        *reinterpret_cast<uint4*>(at + (NPLANE - 1 - pl) * PLANE_BYTES) = w;
        if (pl + 1 < NPLANE) {
            float y[8];
            Vec<__nv_bfloat16>::unpack(w, y);
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] -= y[e];        // exact
        }
    }
}

// The converters' chunks in order: of every piece the first chunks of its B tiles that fill the ring, then the A tile,
// then the rest of the B tiles.  (The ring's stages come free while the last piece's products drain, the A tile's space
// only once they have all retired.)
template <int KCH, int PASS>
struct Feed {
    static constexpr int D = KCH * KCHUNK;
    Walk<PASS> w;
    const float *A, *B;                         // the piece's A matrix, and its (first head's) B matrix
    int n, c, a, chunks, lead, g, bt;           // piece, next B chunk, next A chunk, B chunks and lead, cursor of B
    uint32_t bcnt;                              // B chunks so far
    __device__ __forceinline__ void piece(const Plan& p, const float* Q, const float* K, int Hq, int Hkv, int S) {
        if (!w.valid()) return;
        const int b = w.head / (PASS == 1 ? Hq : Hkv), hh = w.head % (PASS == 1 ? Hq : Hkv), per = p.T - w.tile;
        A = (PASS == 1 ? Q : K) + (size_t)w.head * S * D;
        B = PASS == 1 ? K + ((size_t)b * Hkv + hh / p.G) * S * D : Q + ((size_t)b * Hq + (size_t)hh * p.G) * S * D;
        g = PASS == 1 ? 0 : w.i0 / per;
        bt = PASS == 1 ? w.i0 : w.tile + w.i0 % per;
        chunks = w.n * KCH;
        lead = min(chunks, NSTAGE);
        c = a = 0;
    }
    __device__ __forceinline__ bool is_a() const { return c == lead && a < KCH; }
    __device__ __forceinline__ Chunk chunk(int S) const {
        if (is_a()) return {A + a * KCHUNK, w.tile * TILE};
        return {B + (size_t)g * S * D + (c % KCH) * KCHUNK, bt * TILE};
    }
    __device__ __forceinline__ void next(const Plan& p, const float* Q, const float* K, int Hq, int Hkv, int S) {
        if (is_a()) ++a;
        else {
            if (c % KCH == KCH - 1 && ++bt == p.T && PASS == 2) { bt = w.tile; ++g; }
            ++c; ++bcnt;
        }
        if (c == chunks && a == KCH) { w.next(p); ++n; piece(p, Q, K, Hq, Hkv, S); }
    }
};

// flat (nullable): the rows' log-sum-exp, times flat_mul in log2 units; else states hold it (join_states_kernel) or, with JOIN, the
// row pass's states are joined here (a kernel of its own: 0.4 % of the others' time).
template <int KCH, int PASS, bool JOIN = false>
__global__ void __launch_bounds__(NTHREADS, 1)
score_f32_kernel(const float* __restrict__ Q, const float* __restrict__ K, float2* __restrict__ states,
                 const float* __restrict__ flat, float flat_mul, float* __restrict__ out, kvm_stats* stats,
                 const Plan plan, int Hq, int Hkv, int S, float scale2, float* __restrict__ sim_out) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sA = smem_raw + (base - smem_u32(smem_raw));     // [KCH][plane][128 rows][128 B]
    uint8_t* sB = sA + KCH * CHUNK_BYTES;                     // [NSTAGE][plane][128 rows][128 B]
    Shared& sh = *reinterpret_cast<Shared*>(sB + NSTAGE * CHUNK_BYTES);
    volatile int* abort_flag = &sh.abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) mbar_init(&sh.full_a[i], NCONV);
        mbar_init(&sh.empty_a, 1);
        for (int i = 0; i < NSTAGE; ++i) { mbar_init(&sh.full_b[i], NCONV); mbar_init(&sh.empty_b[i], 1); }
        for (int i = 0; i < NACC; ++i) { mbar_init(&sh.acc_full[i], 1); mbar_init(&sh.acc_empty[i], 4); }
        sh.abort_flag = 0;
        for (int i = 0; i < NSLOT * 4; ++i) (&sh.arrived[0][0])[i] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == NEPI + NCONV) tmem_alloc(&sh.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh.tmem_base;
    grid_dependency_wait();     // (the set-up above runs beside the end of the kernel before this one)

    bool ok = true;
    Walk<PASS> w;
    w.init(plan);
    if (warp >= NEPI && warp < NEPI + NCONV) {
        // ============================== converters ==============================
        // A thread's units of the next chunk are requested as those of this one leave its registers, so that a chunk's
        // way from L2 runs under the work on the chunk before it.
        const int t = threadIdx.x - NEPI * 32;
        Feed<KCH, PASS> f;
        f.w = w; f.n = 0; f.bcnt = 0;
        f.piece(plan, Q, K, Hq, Hkv, S);
        float4 v[UNITS][2];
        bool more = f.w.valid();
        if (more) {
            const Chunk ch = f.chunk(S);
#pragma unroll
            for (int k = 0; k < UNITS; ++k) load_unit<KCH * KCHUNK>(v[k], ch, t + k * NCONV * 32, S);
        }
        while (more) {
            const bool fa = f.is_a();
            const int ac = f.a;
            const uint32_t bc = f.bcnt;
            const int s = bc % NSTAGE;
            if (fa) {
                if (ac == 0) ok = mbar_wait(&sh.empty_a, (f.n & 1) ^ 1, abort_flag);
            } else {
                ok = mbar_wait(&sh.empty_b[s], ((bc / NSTAGE) & 1) ^ 1, abort_flag);
            }
            if (!__all_sync(0xffffffffu, ok)) break;
            uint8_t* dst = fa ? sA + ac * CHUNK_BYTES : sB + s * CHUNK_BYTES;
            f.next(plan, Q, K, Hq, Hkv, S);
            more = f.w.valid();
            const Chunk ch = more ? f.chunk(S) : Chunk{Q, S};             // (row S and beyond: nothing is read)
#pragma unroll
            for (int k = 0; k < UNITS; ++k) {
                const int u = t + k * NCONV * 32;
                if (u < NU) split_unit(v[k], dst, u);
                load_unit<KCH * KCHUNK>(v[k], ch, u, S);
            }
            fence_proxy_async();
            __syncwarp();
#ifdef KVM_TEST_DROP_SCORE_STEP
            if (blockIdx.x == KVM_TEST_DROP_CTA && !fa && bc == (uint32_t)(KVM_TEST_DROP_SCORE_STEP)) continue;   // test build only (see the bf16 kernel)
#endif
            if (lane == 0) mbar_arrive(fa ? &sh.full_a[ac] : &sh.full_b[s]);
        }
        // The neighbour similarities (Eq. 2, which need K alone), while the last products and exponentials drain: the key
        // rows are dealt to the converter warps of all CTAs in runs of SIM_RUN tokens.
        if (PASS == 2 && sim_out) {
            constexpr int D = KCH * KCHUNK, LPR = D / Vec<float>::N, GPW = 32 / LPR;
            const unsigned runs = (unsigned)(S + SIM_RUN - 1) / SIM_RUN, n_runs = (unsigned)plan.U * runs;
            const int gl = lane % LPR, gbase = lane / LPR * LPR;
            const unsigned gmask = LPR == 32 ? 0xffffffffu : (((1u << LPR) - 1u) << gbase);
            for (unsigned g = (blockIdx.x * NCONV + (warp - NEPI)) * GPW + lane / LPR; g < n_runs; g += gridDim.x * NCONV * GPW) {
                const unsigned u = g / runs;
                const int j0 = (int)(g - u * runs) * SIM_RUN;
                simcore::run<float, D, SIM_RUN>(K + (size_t)u * S * D, sim_out + (size_t)u * S, j0, min(j0 + SIM_RUN, S), gl, gbase, gmask);
            }
        }
    } else if (warp == NEPI + NCONV) {
        // ============================== MMA issue ==============================
        {
            // (The whole warp walks and waits, one elected lane issues: descriptors stay in uniform registers.  250 -> 244 us on
            // 16 / 8 heads x 2999 x 128.)
            constexpr uint32_t IDESC = idesc_bf16(TILE);
            // (planes lie in the order l, m, h)
            const uint32_t da0 = (uint32_t)smem_desc(base), db0 = (uint32_t)smem_desc(base + KCH * CHUNK_BYTES);
            const uint32_t dhi = (uint32_t)(smem_desc(base) >> 32);
            uint32_t bcnt = 0, cnt = 0;
            for (int n = 0; ok && w.valid(); ++n, w.next(plan)) {
                for (int i = 0; ok && i < w.n; ++i, ++cnt) {
                    const int as = cnt & 1;
                    ok = mbar_wait_warp(&sh.acc_empty[as], ((cnt >> 1) & 1) ^ 1, abort_flag);
                    const uint32_t d_hi = tmem_base + as * (2 * TILE), d_lo = d_hi + TILE;
#pragma unroll
                    for (int kc = 0; kc < KCH; ++kc, ++bcnt) {
                        const int s = bcnt % NSTAGE;
                        if (i == 0) ok = ok && mbar_wait_warp(&sh.full_a[kc], n & 1, abort_flag);
                        ok = ok && mbar_wait_warp(&sh.full_b[s], (bcnt / NSTAGE) & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        if (elect_one()) {
                            const uint32_t da = da0 + ((kc * CHUNK_BYTES) >> 4), db = db0 + s * (CHUNK_BYTES >> 4);
#pragma unroll
                            for (int ks = 0; ks < KCHUNK / 16; ++ks)
#pragma unroll
                                for (int z = 0; z < 6; ++z) {
                                    constexpr int PX[6] = {2, 1, 2, 0, 1, 2}, PY[6] = {0, 1, 1, 2, 2, 2};
                                    umma_bf16_lo(z == 5 ? d_hi : d_lo, da + ((PX[z] * PLANE_BYTES + ks * 32) >> 4), dhi,
                                                 db + ((PY[z] * PLANE_BYTES + ks * 32) >> 4), dhi, IDESC,
                                                 z == 5 ? (kc | ks) != 0 : (kc | ks | z) != 0);
                                }
                            umma_commit(&sh.empty_b[s]);
                        }
                    }
                    if (ok && elect_one()) umma_commit(&sh.acc_full[as]);
                }
                if (ok && elect_one()) umma_commit(&sh.empty_a);
            }
        }
    } else {
        // ============================== epilogue ==============================
        const int lq = warp & 3, grp = warp >> 2, row = lq * 32 + lane;
        const uint32_t t_lane = tmem_base + ((uint32_t)(lq * 32) << 16) + grp * (2 * TILE);
        float* nl = sh.nl[warp];
        const uint64_t sc2 = pack2(scale2, scale2);
        uint32_t cnt = 0, own = 0;
        const size_t rows = (size_t)plan.NH * S;
        // The log-sum-exp (log2 units) of four of the 128 queries of tile t of the group's query head h: the caller's or the row
        // pass's, what join_states_kernel left, or made of the row pass's states here.  Queries past the end weigh nothing.
        auto ask = [&](float (&v)[4], int h, int t) {
            const int qh = (w.head / Hkv) * Hq + (w.head % Hkv) * plan.G + h;
            const size_t r = (size_t)qh * S + t * TILE + lane;
            const int left = S - t * TILE - lane;
            if (!JOIN && flat) {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = e * 32 < left ? flat[r + e * 32] * flat_mul : INFINITY;
            } else if (!JOIN) {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = e * 32 < left ? __ldcg(&states[r + e * 32].x) : INFINITY;
            } else {
                const int np = plan.row_pieces(qh, t);
                float M[4], L[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) { M[e] = -INFINITY; L[e] = 0.f; }
#pragma unroll 1
                for (int x = 0; x < np; ++x) {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (e * 32 < left) add_state(M[e], L[e], __ldcg(states + (size_t)x * rows + r + e * 32));
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = e * 32 < left ? M[e] + log2f(L[e]) : INFINITY;
            }
        };
        float ahead[4] = {0.f, 0.f, 0.f, 0.f};
        for (int n = 0; w.valid(); ++n, w.next(plan)) {
            float m = -INFINITY;
            uint64_t l2[2] = {0ull, 0ull};                   // four sums, of every fourth column
            const int per = plan.T - w.tile;
            bool asked = false;
            int g = PASS == 1 ? 0 : w.i0 / per, bt = PASS == 1 ? w.i0 : w.tile + w.i0 % per;
            for (int i = 0; i < w.n; ++i, ++cnt) {
                const int cur = bt, cg = g;
                if (++bt == plan.T && PASS == 2) { bt = w.tile; ++g; }
                if ((int)(cnt & 1) != grp) continue;
                if (PASS == 2) {
                    // minus the log-sum-exp of the step's 128 queries, four per lane (asked for during this group's step
                    // before where that belongs to the same piece)
                    float v[4];
                    if (!asked) ask(v, cg, cur);
                    else
#pragma unroll
                        for (int e = 0; e < 4; ++e) v[e] = ahead[e];
                    __syncwarp();                                   // the last step's values have been read
#pragma unroll
                    for (int e = 0; e < 4; ++e) nl[e * 32 + lane] = v[e] > -INFINITY || v[e] != v[e] ? -v[e] : -INFINITY;   // (a query with no key to see weighs nothing)
                    __syncwarp();
                }
                ok = mbar_wait(&sh.acc_full[grp], own & 1, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                ++own;
                if (ok) tc_fence_after();
                if (PASS == 2) {
                    asked = !JOIN && i + 2 < w.n;
                    if (asked) {
                        const int bn = bt + 1 == plan.T ? w.tile : bt + 1, gn = bt + 1 == plan.T ? g + 1 : g;
                        ask(ahead, gn, bn);
                    }
                }
                const bool diag = cur == w.tile;
                // (rolled up: with every role's loops unrolled the instruction cache is what the kernel waits for)
#pragma unroll 1
                for (int cq = 0; cq < 4; ++cq) {
                    // on the diagonal tile whole 32-column quarters are masked (skipped) or valid
                    const bool skip = !ok || (diag && (PASS == 1 ? cq > lq : cq < lq));
                    const bool mask = diag && cq == lq;
                    uint32_t hi[32], lo[32];
                    if (!skip) {
                        tmem_ld32_issue(t_lane + cq * 32, hi);
                        tmem_ld32_issue(t_lane + TILE + cq * 32, lo);
                        tmem_ld_wait();
                    }
                    if (cq == 3) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sh.acc_empty[grp]);
                    }
                    if (skip) continue;
                    tmem_ld_fence(hi);
                    tmem_ld_fence(lo);
                    float v[32];
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        uint64_t x = fadd2(pack2(__uint_as_float(hi[c]), __uint_as_float(hi[c + 1])),
                                           pack2(__uint_as_float(lo[c]), __uint_as_float(lo[c + 1])));
                        if (PASS == 2) x = ffma2(x, sc2, *reinterpret_cast<const uint64_t*>(nl + cq * 32 + c));
                        unpack2(x, v[c], v[c + 1]);
                    }
                    if (mask) {
#pragma unroll
                        for (int c = 0; c < 32; ++c)
                            if (PASS == 1 ? c > lane : c < lane) v[c] = -INFINITY;   // key after query
                    }
                    if (PASS == 1) {
                        float mx = v[0];
#pragma unroll
                        for (int c = 1; c + 1 < 32; c += 2) mx = fmax3(mx, v[c], v[c + 1]);
                        const float mn = fmaxf(m, fmaxf(mx, v[31]) * scale2), ref = mn == -INFINITY ? 0.f : mn;
                        // (what is flushed to zero below 2^-126 would not change a sum that holds the maximum's 1)
                        const float f = ex2(m - ref);
                        const uint64_t f2 = pack2(f, f), nref2 = pack2(-ref, -ref);
#pragma unroll
                        for (int e = 0; e < 2; ++e) l2[e] = fmul2(l2[e], f2);
#pragma unroll
                        for (int c = 0; c < 32; c += 2) {
                            float x0, x1;
                            unpack2(ffma2(pack2(v[c], v[c + 1]), sc2, nref2), x0, x1);
                            l2[(c >> 1) & 1] = fadd2(l2[(c >> 1) & 1], pack2(ex2(x0), ex2(x1)));
                        }
                        m = mn;
                    } else {
                        // A key whose every weight is below 2^-126 keeps a score: the slow exponential, which does not flush,
                        // where one could be (four instructions for one).
                        float low = v[0];
#pragma unroll
                        for (int c = 1; c + 1 < 32; c += 2) low = fmin3(low, v[c], v[c + 1]);
                        if (__any_sync(0xffffffffu, !(fminf(low, v[31]) >= -126.f))) {
#pragma unroll
                            for (int c = 0; c < 32; c += 2) l2[(c >> 1) & 1] = fadd2(l2[(c >> 1) & 1], pack2(exp2f(v[c]), exp2f(v[c + 1])));
                        } else {
#pragma unroll
                            for (int c = 0; c < 32; c += 2) l2[(c >> 1) & 1] = fadd2(l2[(c >> 1) & 1], pack2(ex2(v[c]), ex2(v[c + 1])));
                        }
                    }
                }
            }
            float l[4];
            unpack2(l2[0], l[0], l[1]);
            unpack2(l2[1], l[2], l[3]);
            // ---- piece end: the two warps that own a row leave their sums in shared memory; whichever comes
            // last adds them in a fixed order and stores.  Nobody waits.  (Buffers: when a warp finishes step k the MMA
            // thread has issued step k - 1, so the other group has handed step k - 3 back but may not have delivered it.
            // With one-step pieces the warp then delivers piece k, and piece k + 1 in which it has no step: five
            // pieces are open at most.)
            const int slot = n % NSLOT;
            // (After a give-up nothing keeps the groups within a few steps of one another, and a piece's buffer could be
            // taken for a later one's: every warp marks the rows of its pieces by itself then.)
            bool bad = __any_sync(0xffffffffu, *abort_flag != 0);
            int before = 1;
            if (!bad) {
                sh.part_m[slot][grp][row] = m;
                sh.part_l[slot][grp][row] = (l[0] + l[1]) + (l[2] + l[3]);
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    before = atomicAdd(&sh.arrived[slot][lq], 1);
                }
                before = __shfl_sync(0xffffffffu, before, 0);
            }
            if (before == 1) {
                __threadfence_block();
                if (!bad && lane == 0) sh.arrived[slot][lq] = 0;
                bad = bad || *abort_flag != 0;   // (read again: the other group may have given up before it came here)
                const int gi = w.tile * TILE + row;
                const float m0 = sh.part_m[slot][0][row], m1 = sh.part_m[slot][1][row];
                const float l0 = sh.part_l[slot][0][row], l1 = sh.part_l[slot][1][row];
                if (gi < S) {
                    const size_t at = (size_t)w.head * S + gi;
                    if (PASS == 1) {
                        const float M = bad ? 0.f : fmaxf(m0, m1);
                        const float L = bad ? NAN : (m0 > -INFINITY ? l0 * exp2f(m0 - M) : 0.f) + (m1 > -INFINITY ? l1 * exp2f(m1 - M) : 0.f);
                        if (plan.split_row) {
                            states[(size_t)w.piece(plan) * rows + at] = make_float2(M, L);
                        } else {
                            out[at] = M + log2f(L);
                        }
                    } else {
                        const float a = bad ? NAN : l0 + l1;
                        if (plan.split_col) {
                            out[(size_t)w.piece(plan) * plan.U * S + at] = a;
                        } else {
                            out[at] = a / (float)plan.G;
                        }
                    }
                }
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh.abort_flag && stats) stats->status = KVM_E_DEVICE_TIMEOUT;
    if (warp == NEPI + NCONV) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// The row pass's states (or final log2-unit values, when items were whole) as the natural-log lse the caller asked for.
__global__ void __launch_bounds__(256) row_lse_kernel(const float2* __restrict__ states, const float* __restrict__ flat,
                                                      float* __restrict__ lse, const Plan plan, int S) {
    grid_dependency_wait();
    const size_t rows = (size_t)plan.NH * S, r = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    if (flat) { lse[r] = __ldcg(flat + r) * LN2; return; }
    const int head = (int)(r / S), np = plan.row_pieces(head, (int)(r - (size_t)head * S) / TILE);
    float M = -INFINITY, L = 0.f;
    for (int x = 0; x < np; ++x) {
        const float2 st = __ldcg(states + (size_t)x * rows + r);
        add_state(M, L, st);
    }
    lse[r] = (M + log2f(L)) * LN2;
}

// Partial column sums -> scores.
__global__ void __launch_bounds__(256) combine_kernel(const float* __restrict__ part, float* __restrict__ scores,
                                                      const Plan plan, int S) {
    grid_dependency_wait();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < S) scores[(size_t)blockIdx.y * S + j] = plan::column_sum(part, plan, S, blockIdx.y, j);
}
// The row pass's states of cut items -> the rows' log-sum-exp (log2 units), in the place of their first states.
__global__ void __launch_bounds__(256) join_states_kernel(float2* __restrict__ states, const Plan plan, int S) {
    grid_dependency_wait();
    const size_t rows = (size_t)plan.NH * S, r = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    const int head = (int)(r / S), np = plan.row_pieces(head, (int)(r - (size_t)head * S) / TILE);
    float M = -INFINITY, L = 0.f;
#pragma unroll 2
    for (int x = 0; x < np; ++x) add_state(M, L, __ldcg(states + (size_t)x * rows + r));
    states[r].x = M + log2f(L);
}
// Bytes of the two passes' states and sums.
size_t state_bytes(const Dims& d, const Plan& p) {
    const size_t rows = (size_t)p.NH * d.S;
    return p.split_row ? split_bytes(d, p) : rows * sizeof(float);
}
template <int KCH>
cudaError_t launch_t(const Dims& d, const Plan& plan, const float* Q, const float* K, const float* lse_in, void* scratch,
                     float* scores, kvm_stats* stats, cudaStream_t st, float* sim_out, float* lse_out, ScorePart* parts) {
    const size_t smem = 1024 + (size_t)(KCH + NSTAGE) * CHUNK_BYTES + sizeof(Shared);
    static std::mutex mu;
    static bool done[KVM_MAX_DEVICES] = {};
    cudaError_t e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if (dev < 0 || dev >= KVM_MAX_DEVICES) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!done[dev]) {
            e = cudaFuncSetAttribute(score_f32_kernel<KCH, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            e = cudaFuncSetAttribute(score_f32_kernel<KCH, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            e = cudaFuncSetAttribute(score_f32_kernel<KCH, 2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            done[dev] = true;
        }
    }
    const long long items = (long long)plan.NH * plan.T, citems = (long long)plan.U * plan.T;
    const dim3 block(NTHREADS), rgrid(plan.split_row ? plan.grid_split() : (unsigned)(items < plan::CTAS ? items : plan::CTAS)),
        cgrid(plan.split_col ? plan.grid_split() : (unsigned)(citems < plan::CTAS ? citems : plan::CTAS));
    const size_t rows = (size_t)plan.NH * d.S;
    float2* states = plan.split_row ? (float2*)scratch : nullptr;
    float* flat = plan.split_row ? nullptr : (float*)scratch;            // log2 units
    float* part = plan.split_row ? (float*)((float2*)scratch + rows * plan.pr) : nullptr;
    const float scale2 = d.scale * LOG2E;
    if (!lse_in) {
        e = launch_dependent(score_f32_kernel<KCH, 1>, rgrid, block, smem, st, Q, K, states, (const float*)nullptr,
                             1.f, flat, stats, plan, d.Hq, d.Hkv, d.S, scale2, (float*)nullptr);
        if (e != cudaSuccess) return e;
    }
    if (lse_out) {
        e = launch_dependent(row_lse_kernel, dim3((unsigned)((rows + 255) / 256)), dim3(256), 0, st, (const float2*)states,
                             (const float*)flat, lse_out, plan, d.S);
        if (e != cudaSuccess) return e;
    }
    if (!scores) return cudaSuccess;
    const bool states_in = !lse_in && plan.split_row, between = states_in && join_between(plan, d.D);
    if (between) {
        e = launch_dependent(join_states_kernel, dim3((unsigned)((rows + 255) / 256)), dim3(256), 0, st, states, plan, d.S);
        if (e != cudaSuccess) return e;
    }
    const auto columns = states_in && !between ? score_f32_kernel<KCH, 2, true> : score_f32_kernel<KCH, 2>;
    e = launch_dependent(columns, cgrid, block, smem, st, Q, K, states,
                         lse_in ? lse_in : (const float*)flat, lse_in ? LOG2E : 1.f, plan.split_col ? part : scores, stats, plan,
                         d.Hq, d.Hkv, d.S, scale2, sim_out);
    if (e != cudaSuccess || !plan.split_col) return e;
    if (parts) {                                      // the caller's next kernel adds the pieces up
        parts->part = part;
        parts->plan = plan;
        return cudaSuccess;
    }
    return launch_dependent(combine_kernel, dim3((d.S + 255) / 256, d.U), dim3(256), 0, st, (const float*)part, scores, plan, d.S);
}

}  // namespace

// Scratch of both passes: the pieces' row states and partial column sums, or one float per query row.
size_t score_f32_scratch_bytes(const Dims& d) {
    Plan p;
    if (!make_plan(d, p)) return 0;                                  // (launching this shape is refused)
    return state_bytes(d, p);
}

// lse_in (nullable): natural-log row log-sum-exp, skips the row pass.  scores may be NULL (row pass only); lse_out
// (nullable) receives the natural-log row log-sum-exp; sim_out (nullable, with scores) the neighbour similarities [U,S];
// parts (nullable): lets the column pass leave partial sums (parts->part set) for the caller's next kernel to add.
cudaError_t launch_score_f32(const Dims& d, const void* Q, const void* K, const float* lse_in, void* scratch,
                             float* scores, kvm_stats* stats, cudaStream_t st, float* sim_out, float* lse_out,
                             ScorePart* parts) {
    Plan plan;
    if (!make_plan(d, plan)) return cudaErrorInvalidValue;
    auto fn = d.D == 128 ? launch_t<2> : launch_t<1>;
    return fn(d, plan, (const float*)Q, (const float*)K, lse_in, scratch, scores, stats, st, sim_out, lse_out, parts);
}

}  // namespace kvm
