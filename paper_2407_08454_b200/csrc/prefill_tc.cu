// Causal attention over the whole prompt on the 5th-generation tensor cores (bf16 inputs):
//   O_i = sum_{j<=i} softmax_j(c q_i.k_j) v_j,   lse_i = ln sum_{j<=i} exp(c q_i.k_j)          Eq. 1
// This is the attention a prefill runs anyway; its row log-sum-exp is exactly what the score step's row pass
// computes, so a caller that runs this kernel hands `lse` to kvm_compress_with_lse and pays for no row pass.
//
// A work item is one 128-row query tile of one query head with the key/value tiles 0..it it attends to.  Per
// key tile ("step") two tcgen05.mma chains run: S = Q K^T into a 128-column TMEM accumulator, and O += P V into
// another, with P = exp(S - reference) written to shared memory as bf16 by the softmax warps in the layout the
// tensor core reads (128-byte rows, 128-byte swizzle) and V read with its head dimension contiguous (the layout
// it has in memory).  Two groups of four softmax warps take alternate steps, each with its own S accumulator, P
// tile, O accumulator, reference maximum and row sum, so that one group's exponentials run under the other
// group's products; the two partial results of a row are joined when the item ends, by the group that took the
// item's first step (groups swap from item to item: step j of item n belongs to group (j + n) & 1), which reads
// the other group's accumulator first and hands it back at once, so that the other group's first step of the next
// item runs beside the join.  The logits stay two steps ahead of the P V products across item boundaries (the Q
// tile is released when the item's last Q K^T has been issued).  A softmax thread owns one
// query row = one TMEM lane: it holds the 128 logits of a step in registers (the accumulator is handed back at
// once), and multiplies its row of O by exp(old - new reference) only when the maximum has grown by more than
// 8 (log2 units) since the reference was set, so that most steps touch O not at all.
//
// One CTA per SM, persistent:  warps 0-7 softmax (group = warp / 4),  warp 8 producer of the Q and K tiles (TMA,
// 128-byte swizzle; K and V tiles in rings of two),  warp 9 one thread issues the Q K^T MMAs and owns tensor memory,  warp 10 one
// thread issues the P V MMAs (two issuing threads: neither product's waits hold the other's issue up),  warp 11
// producer of the V tiles (the third warpgroup gives registers up to the softmax warpgroups).  Items are dealt
// longest first, boustrophedon.  Every wait on an mbarrier is bounded; a wait that runs out raises a flag, every
// role leaves its loops, the rows in hand are written as NaN, kvm_stats.status is set when given, tensor memory
// is freed.  (The test build of the library, never shipped, shortens the limit and makes the producer leave out one
// V tile, so that this path can be exercised: KVM_TEST_WAIT_LIMIT_CLOCKS, KVM_TEST_DROP_B_STAGE.)
#include <mutex>

#include "tc_common.cuh"

namespace kvm {
namespace {

using namespace tc;

constexpr int TILE = 128;
constexpr int KCHUNK = 64;
constexpr int NKV = 2;                  // ring depth of the K tiles and of the V tiles
constexpr int NGRP = 2;                 // softmax groups taking alternate steps
constexpr int NSOFT = 4 * NGRP;         // softmax warps: one per TMEM lane quarter and group
constexpr int NTHREADS = (NSOFT + 4) * 32;   // three warpgroups: two of softmax warps, one with producer, MMA issue and two idle warps
// Registers: the launch gives every thread 168 (65536 / 384); the softmax warpgroups then take 208 each and the
// third warpgroup keeps 56 (2 x 128 x 208 + 128 x 56 = 60416 <= 384 x 168 = 64512).
constexpr int REGS_SOFTMAX = 208, REGS_OTHER = 56;
constexpr uint32_t CHUNK_BYTES = TILE * 128;            // [128 rows x 64 bf16]
constexpr float LOG2E = 1.4426950408889634f, LN2 = 0.6931471805599453f;
constexpr float RESCALE_STEP = 8.f;     // the reference maximum follows the running maximum in steps of at least this: a
                                        // weight is at most 2^RESCALE_STEP (values up to 2^-8 of the largest bf16 stay finite)
constexpr uint32_t S_COLS = TILE, O_COL0 = NGRP * S_COLS;  // TMEM columns: S of group 0 | S of group 1 | O 0 | O 1

struct __align__(8) Bars {
    uint64_t q_full, q_empty;
    uint64_t k_full[NKV], k_empty[NKV], v_full[NKV], v_empty[NKV];
    uint64_t s_full[NGRP], s_empty[NGRP];
    uint64_t p_full[NGRP][2], pv_half[NGRP], pv_done[NGRP], o_empty[NGRP];   // P by halves of the key tile
    uint64_t part_full, part_empty;     // the handing group's row state at item end: written / read
};
struct alignas(16) Shared {
    Bars bar;
    uint32_t tmem_base;
    int abort_flag;
    float part_m[TILE], part_l[TILE];   // the handing group's row state at item end (through part_full / part_empty)
};

struct Sched {
    int P, c, NH, T;
    // (32-bit arithmetic: the launcher refuses shapes whose item count does not fit; a 64-bit division here costs
    // every role several hundred clocks at every item boundary)
    __device__ __forceinline__ bool item(int n, int& head, int& tile) const {
        const unsigned k = (unsigned)n * (unsigned)P + (unsigned)((n & 1) ? (P - 1 - c) : c);
        if (k >= (unsigned)NH * (unsigned)T) return false;
        const unsigned r = k / (unsigned)NH;
        head = (int)(k - r * (unsigned)NH);
        tile = T - 1 - (int)r;
        return true;
    }
};

template <int KCH>
__global__ void __launch_bounds__(NTHREADS, 1)
prefill_attend_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                      const __grid_constant__ CUtensorMap map_v, __nv_bfloat16* __restrict__ O,
                      float* __restrict__ lse, kvm_stats* stats, int B, int Hq, int Hkv, int S, float scale2) {
    constexpr int D = KCH * KCHUNK;
    constexpr uint32_t TILE_BYTES = KCH * CHUNK_BYTES;     // a Q, K or V tile
    constexpr uint32_t P_BYTES = 2 * CHUNK_BYTES;          // P: [2 key chunks][128 rows][128 B]
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* aligned = smem_raw + (base - smem_u32(smem_raw));
    uint8_t* sQ = aligned;
    uint8_t* sK = sQ + TILE_BYTES;
    uint8_t* sV = sK + NKV * TILE_BYTES;
    uint8_t* sP = sV + NKV * TILE_BYTES;                   // one P tile per group
    Shared& sh = *reinterpret_cast<Shared*>(sP + NGRP * P_BYTES);
    volatile int* abort_flag = &sh.abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = Hq / Hkv;
    const int T = (S + TILE - 1) / TILE;
    const Sched sc{(int)gridDim.x, (int)blockIdx.x, B * Hq, T};

    if (threadIdx.x == 0) {
        mbar_init(&sh.bar.q_full, 1); mbar_init(&sh.bar.q_empty, 1);
        for (int i = 0; i < NKV; ++i) {
            mbar_init(&sh.bar.k_full[i], 1); mbar_init(&sh.bar.k_empty[i], 1);
            mbar_init(&sh.bar.v_full[i], 1); mbar_init(&sh.bar.v_empty[i], 1);
        }
        for (int i = 0; i < NGRP; ++i) {
            mbar_init(&sh.bar.s_full[i], 1); mbar_init(&sh.bar.s_empty[i], 4);
            for (int h = 0; h < 2; ++h) mbar_init(&sh.bar.p_full[i][h], 4);
            mbar_init(&sh.bar.pv_half[i], 1); mbar_init(&sh.bar.pv_done[i], 1);
        }
        for (int i = 0; i < NGRP; ++i) mbar_init(&sh.bar.o_empty[i], 4);
        mbar_init(&sh.bar.part_full, 4); mbar_init(&sh.bar.part_empty, 4);
        sh.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == NSOFT + 1) tmem_alloc(&sh.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh.tmem_base;
    grid_dependency_wait();

    if (warp >= NSOFT) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_OTHER));
      if (warp == NSOFT) {
        // ============================== producer of the Q and K tiles ==============================
        // (The V tiles have a producer of their own: a V tile's slot comes free a step or two after the K tile's
        // of the same step, and one thread loading both in turn would hold the next K tile back behind that wait.)
        if (lane == 0) {
            uint32_t kv = 0;                                  // K tiles loaded so far
            bool ok = true;
            int head, tile;
            for (int n = 0; ok && sc.item(n, head, tile); ++n) {
                ok = mbar_wait(&sh.bar.q_empty, (n & 1) ^ 1, abort_flag);
                if (!ok) break;
                mbar_expect_tx(&sh.bar.q_full, TILE_BYTES);
#pragma unroll
                for (int kc = 0; kc < KCH; ++kc)
                    tma_load_3d(sQ + kc * CHUNK_BYTES, &map_q, &sh.bar.q_full, kc * KCHUNK, tile * TILE, head);
                const int kvhead = (head / Hq) * Hkv + (head % Hq) / G;
                for (int j = 0; j <= tile; ++j, ++kv) {
                    const int s = kv % NKV;
                    ok = mbar_wait(&sh.bar.k_empty[s], ((kv / NKV) & 1) ^ 1, abort_flag);
                    if (!ok) break;
                    mbar_expect_tx(&sh.bar.k_full[s], TILE_BYTES);
#pragma unroll
                    for (int kc = 0; kc < KCH; ++kc)
                        tma_load_3d(sK + s * TILE_BYTES + kc * CHUNK_BYTES, &map_k, &sh.bar.k_full[s], kc * KCHUNK,
                                    j * TILE, kvhead);
                }
            }
            // Copies already issued complete on their own; before shared memory is given back, let them land
            // (bounded: each try_wait suspends for a while by itself).
            if (*abort_flag)
                for (uint32_t it = 0; it < (1u << 14); ++it) mbar_try(&sh.bar.q_full, 0);
        }
      } else if (warp == NSOFT + 3) {
        // ============================== producer of the V tiles ==============================
        if (lane == 0) {
            uint32_t kv = 0;                                  // V tiles loaded so far
            bool ok = true;
            int head, tile;
            for (int n = 0; ok && sc.item(n, head, tile); ++n) {
                const int kvhead = (head / Hq) * Hkv + (head % Hq) / G;
                for (int j = 0; j <= tile; ++j, ++kv) {
#ifdef KVM_TEST_DROP_B_STAGE
                    if (kv == (uint32_t)(KVM_TEST_DROP_B_STAGE)) continue;   // test build only: this V tile never arrives
#endif
                    const int s = kv % NKV;
                    ok = mbar_wait(&sh.bar.v_empty[s], ((kv / NKV) & 1) ^ 1, abort_flag);
                    if (!ok) break;
                    mbar_expect_tx(&sh.bar.v_full[s], TILE_BYTES);
#pragma unroll
                    for (int kc = 0; kc < KCH; ++kc)
                        tma_load_3d(sV + s * TILE_BYTES + kc * CHUNK_BYTES, &map_v, &sh.bar.v_full[s], kc * KCHUNK,
                                    j * TILE, kvhead);
                }
            }
            if (*abort_flag)
                for (uint32_t it = 0; it < (1u << 14); ++it) mbar_try(&sh.bar.v_full[0], 0);
        }
      } else if (warp == NSOFT + 1) {
        // ============================== MMA issue: S = Q K^T ==============================
        // Step j of item n belongs to group (j + n) & 1.  This thread runs ahead of the P V products as far as the
        // two S accumulators allow (a group's next S is issued as soon as the group has taken the last one into
        // registers), across item boundaries too: Q is released as soon as the item's last Q K^T has been issued,
        // so the next Q tile and the next item's first S tiles arrive while the last products drain.  (Its
        // commits cover its own MMAs only: the two products are issued by two threads.)
        if (lane == 0) {
            constexpr uint32_t IDESC_S = idesc_bf16(TILE);
            const uint64_t desc_q = smem_desc(base);
            const uint64_t desc_k0 = smem_desc(base + TILE_BYTES);
            uint32_t ks_cnt = 0;                             // K tiles consumed so far
            uint32_t s_ph = 0;                               // bit g: parity of the S tiles produced for group g
            bool ok = true;
            int head, tile;
            for (int n = 0; ok && sc.item(n, head, tile); ++n) {
                ok = mbar_wait(&sh.bar.q_full, n & 1, abort_flag);
                for (int j = 0; ok && j <= tile; ++j) {
                    const int g = (j + n) & 1;
                    const int s = ks_cnt % NKV;
                    ok = mbar_wait(&sh.bar.k_full[s], (ks_cnt / NKV) & 1, abort_flag) &&
                         mbar_wait(&sh.bar.s_empty[g], ((s_ph >> g) & 1) ^ 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t dk = (uint32_t)desc_k0 + s * (TILE_BYTES >> 4);
#pragma unroll
                    for (int kc = 0; kc < KCH; ++kc)
#pragma unroll
                        for (int ks = 0; ks < KCHUNK / 16; ++ks)
                            umma_bf16_lo(tmem_base + g * S_COLS, (uint32_t)desc_q + ((kc * CHUNK_BYTES + ks * 32) >> 4),
                                         (uint32_t)(desc_q >> 32), dk + ((kc * CHUNK_BYTES + ks * 32) >> 4),
                                         (uint32_t)(desc_k0 >> 32), IDESC_S, (kc | ks) ? 1u : 0u);
                    umma_commit(&sh.bar.k_empty[s]);
                    umma_commit(&sh.bar.s_full[g]);
                    ++ks_cnt; s_ph ^= 1u << g;
                }
                if (ok) umma_commit(&sh.bar.q_empty);        // every product that reads this Q tile has been issued
            }
        }
      } else if (warp == NSOFT + 2) {
        // ============================== MMA issue: O += P V ==============================
        if (lane == 0) {
            constexpr uint32_t IDESC_O = idesc_bf16(D, true);
            const uint32_t v_addr0 = base + TILE_BYTES + NKV * TILE_BYTES;
            const uint64_t desc_p0 = smem_desc(v_addr0 + NKV * TILE_BYTES);
            const uint64_t desc_v0 = smem_desc_mn(v_addr0, CHUNK_BYTES);
            const uint32_t dv_base = (uint32_t)desc_v0, v_hi = (uint32_t)(desc_v0 >> 32), p_hi = (uint32_t)(desc_p0 >> 32);
            uint32_t vs_cnt = 0;                             // V tiles consumed so far
            uint32_t pv_ph = 0;                              // bit g: parity of the P V products issued for group g
            bool ok = true;
            int head, tile;
            for (int n = 0; ok && sc.item(n, head, tile); ++n) {
                for (int j = 0; ok && j <= tile; ++j) {
                    const int g = (j + n) & 1;
                    if (j < 2) ok = mbar_wait(&sh.bar.o_empty[g], (n & 1) ^ 1, abort_flag);   // the last item's O of this group has been read
                    const int s = vs_cnt % NKV;
                    ok = ok && mbar_wait(&sh.bar.v_full[s], (vs_cnt / NKV) & 1, abort_flag);
                    const uint32_t dv0 = dv_base + s * (TILE_BYTES >> 4);                          // 16 keys further: + 2 KB
                    const uint32_t dp = (uint32_t)desc_p0 + g * (P_BYTES >> 4);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {                   // the first half's products run while the second is made
                        ok = ok && mbar_wait(&sh.bar.p_full[g][h], (pv_ph >> g) & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4) {            // 16 keys per MMA
                            const int kk = h * 4 + k4;
                            umma_bf16_lo(tmem_base + O_COL0 + g * S_COLS, dp + ((h * CHUNK_BYTES + k4 * 32) >> 4), p_hi,
                                         dv0 + ((kk * 16 * 128) >> 4), v_hi, IDESC_O, ((j >> 1) | kk) ? 1u : 0u);
                        }
                        if (h == 0) umma_commit(&sh.bar.pv_half[g]);
                    }
                    if (!ok) break;
                    umma_commit(&sh.bar.v_empty[s]);
                    umma_commit(&sh.bar.pv_done[g]);         // the group's P may be overwritten, its O read or rescaled
                    ++vs_cnt; pv_ph ^= 1u << g;
                }
            }
        }
      }
    } else {
        // ============================== softmax ==============================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SOFTMAX));
        const int grp = warp >> 2, lq = warp & 3;
        const int row = lq * 32 + lane;                      // query row of the tile = TMEM lane
        const uint32_t t_lane = tmem_base + ((uint32_t)(lq * 32) << 16);
        const uint32_t t_s = t_lane + grp * S_COLS, t_o = t_lane + O_COL0 + grp * S_COLS;
        uint8_t* prow = sP + grp * P_BYTES + row * 128;
        uint32_t s_cnt = 0, pv_cnt = 0;                      // this group's steps so far
        uint32_t pv_other = 0;                               // the other group's (the joining group reads both results)
        bool ok = true;
        int head, tile;
        for (int n = 0; ok && sc.item(n, head, tile); ++n) {
            float m = -INFINITY, l = 0.f;                    // reference maximum (log2 units) and sum relative to it
            const int j_first = (grp + n) & 1;               // this group's first step of the item
            for (int j = j_first; j <= tile; j += NGRP) {
                ok = mbar_wait(&sh.bar.s_full[grp], s_cnt & 1, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                uint32_t vr[TILE];
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_ld32_issue(t_s + q * 32, vr + q * 32);
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.bar.s_empty[grp]);   // the accumulator goes back at once
                ++s_cnt;
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_ld_fence(vr + q * 32);
                float v[TILE];
#pragma unroll
                for (int c = 0; c < TILE; ++c) v[c] = __uint_as_float(vr[c]);
                if (j == tile) {                             // diagonal tile: keys after the query do not exist for it
#pragma unroll
                    for (int c = 0; c < TILE; ++c)
                        if (c > row) v[c] = -INFINITY;
                }
                float mx = v[0];
#pragma unroll
                for (int c = 1; c + 1 < TILE; c += 2) mx = fmax3(mx, v[c], v[c + 1]);
                mx = fmaxf(mx, v[TILE - 1]) * scale2;
                // the reference moves only when the maximum has outgrown it by RESCALE_STEP: exp2(x - m) stays
                // below 2^RESCALE_STEP, and O is rescaled rarely
                float alpha = 1.f;
                const bool first = j == j_first;             // the group's first step of the item
                const bool grow = mx > m + RESCALE_STEP;
                if (first) m = mx;
                else if (grow) { alpha = ex2(m - mx); m = mx; }
                const bool rescale = !first && __any_sync(0xffffffffu, grow);
                if (rescale) {
                    // (the group's previous P V has to be done before its O is touched)
                    ok = mbar_wait(&sh.bar.pv_done[grp], (pv_cnt & 1) ^ 1, abort_flag);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int q = 0; q < D / 32; ++q) {
                        uint32_t orr[32];
                        tmem_ld32_issue(t_o + q * 32, orr);
                        tmem_ld_wait();
                        tmem_ld_fence(orr);
#pragma unroll
                        for (int c = 0; c < 32; ++c) orr[c] = __float_as_uint(__uint_as_float(orr[c]) * alpha);
                        tmem_st32(t_o + q * 32, orr);
                    }
                    tmem_st_wait();
                }
                // p = 2^(x - m), summed in fp32, rounded to bf16 for the tensor core, in two halves of 64 keys: the
                // products with the first half run while the second is computed, and a half of the P tile may be
                // overwritten as soon as the last step's products with that half are done
                const uint64_t sc2 = pack2(scale2, scale2), nm2 = pack2(-m, -m);
                float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t pk[TILE / 4];
#pragma unroll
                    for (int c = 0; c < TILE / 2; c += 2) {
                        float x0, x1;
                        unpack2(ffma2(pack2(v[h * 64 + c], v[h * 64 + c + 1]), sc2, nm2), x0, x1);
                        const float e0 = ex2(x0), e1 = ex2(x1);
                        sum[(c >> 1) & 3] += e0 + e1;
                        pk[c >> 1] = Vec<__nv_bfloat16>::pack2(e0, e1);
                    }
                    ok = mbar_wait(h ? &sh.bar.pv_done[grp] : &sh.bar.pv_half[grp], (pv_cnt & 1) ^ 1, abort_flag);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    // P row: 16-byte piece c of key chunk h sits at piece c ^ (row & 7) of the row's 128 bytes
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        *reinterpret_cast<uint4*>(prow + h * CHUNK_BYTES + ((c ^ (row & 7)) << 4)) =
                            make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
                    fence_proxy_async();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh.bar.p_full[grp][h]);
                }
                if (!ok) break;
                l = l * alpha + ((sum[0] + sum[1]) + (sum[2] + sum[3]));
                ++pv_cnt;
            }
            const int n_own = tile >= j_first ? (tile - j_first) / 2 + 1 : 0;
            const int n_other = tile + 1 - n_own;            // steps the other group takes in this item
            pv_other += n_other;
            // ---- item end: one group hands its row state to the other, which joins the two partial results:
            //      O = (O_a 2^(m_a - M) + O_b 2^(m_b - M)) / (l_a 2^(m_a - M) + l_b 2^(m_b - M)),  M = max(m_a, m_b)
            // The joining group is the one that took the item's first step (group n & 1), so the other one is
            // free for the next item's first step while the join runs.
            if (grp != (n & 1)) {
                // (every item, also one in which this group had no step: the two groups count items alike)
                ok = ok && mbar_wait(&sh.bar.part_empty, (n & 1) ^ 1, abort_flag);   // the last item's has been read
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                sh.part_m[row] = m;
                sh.part_l[row] = l;
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.bar.part_full);
                continue;
            }
            if (ok) {
                ok = mbar_wait(&sh.bar.part_full, n & 1, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
            }
            const float m1 = ok ? sh.part_m[row] : -INFINITY, l1 = ok ? sh.part_l[row] : 0.f;
            __syncwarp();
            if (ok && lane == 0) mbar_arrive(&sh.bar.part_empty);
            const int gi = tile * TILE + row;
            if (ok) {
                ok = mbar_wait(&sh.bar.pv_done[grp], (pv_cnt & 1) ^ 1, abort_flag);
                if (ok && n_other > 0) ok = mbar_wait(&sh.bar.pv_done[grp ^ 1], (pv_other & 1) ^ 1, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
            }
            ok = ok && (*abort_flag == 0);
            __nv_bfloat16* orow = O + ((size_t)head * S + gi) * D;
            if (ok) {
                tc_fence_after();
                const float M = fmaxf(m, m1);
                const float w0 = n_own > 0 ? ex2(m - M) : 0.f, w1 = n_other > 0 ? ex2(m1 - M) : 0.f;
                const float L = l * w0 + l1 * w1;
                const float f0 = w0 / L, f1 = w1 / L;
                // the other group's accumulator first, whole, so that it goes back at once: that group is
                // already at work on the next item
                // (a group without a step in this item has a stale accumulator: it is read all the same, so that
                // the registers are not conditional, and replaced by zeros)
                uint32_t o1[D];
#pragma unroll
                for (int q = 0; q < D / 32; ++q) tmem_ld32_issue(t_lane + O_COL0 + (grp ^ 1) * S_COLS + q * 32, o1 + q * 32);
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.bar.o_empty[grp ^ 1]);
#pragma unroll
                for (int q = 0; q < D / 32; ++q) tmem_ld_fence(o1 + q * 32);
                const bool has0 = n_own > 0, has1 = n_other > 0;
#pragma unroll
                for (int q = 0; q < D / 32; ++q) {
                    uint32_t o0[32];
                    tmem_ld32_issue(t_o + q * 32, o0);
                    tmem_ld_wait();
                    tmem_ld_fence(o0);
                    if (gi < S) {
#pragma unroll
                        for (int c = 0; c < 32; c += 8) {
                            float f[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const float a0 = has0 ? __uint_as_float(o0[c + e]) : 0.f;
                                const float a1 = has1 ? __uint_as_float(o1[q * 32 + c + e]) : 0.f;
                                f[e] = fmaf(a1, f1, a0 * f0);
                            }
                            *reinterpret_cast<uint4*>(orow + q * 32 + c) = Vec<__nv_bfloat16>::pack(f);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.bar.o_empty[grp]);
                if (gi < S) lse[(size_t)head * S + gi] = (M + log2f(L)) * LN2;
            } else if (gi < S) {
                // a wait gave up: what this row would have received is marked, not made up
                for (int c = 0; c < D; c += 8)
                    *reinterpret_cast<uint4*>(orow + c) = make_uint4(0x7FC07FC0u, 0x7FC07FC0u, 0x7FC07FC0u, 0x7FC07FC0u);
                lse[(size_t)head * S + gi] = NAN;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh.abort_flag && stats) stats->status = KVM_E_DEVICE_TIMEOUT;
    if (warp == NSOFT + 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------ two query tiles per CTA
// The same attention with two query tiles in hand that read the same keys and values: two query heads of a group with one
// tile each, or (one head per group, or an odd number) two neighbouring tiles of a head.  Softmax group g owns tile g:
//   S_g = Q_g K_j^T  ->  P_g = exp(S_g - reference), written over S_g in tensor memory  ->  O_g += P_g V_j,
// and while one tile's products run the other's exponentials do.  What bounds the kernel above is shared memory: a step of
// 128 x 128 x 128 reads two operands for each product (128 KB), writes P (32 KB) and receives K and V (64 KB), 1,750 clocks at
// 128 bytes a clock.  Here P is read from tensor memory and K and V serve two tiles: 64 + 32 + 32 KB.  Two steps, one of each
// tile, take 2,950 clocks (head dimension 64: 2,680): 1,720 of a tile's softmax (1,024 of them exponentials at the unit's full
// rate), the rest until its next logits are there; the tensor pipe is busy 2,180 (1,300) of them.
// O is divided by the sum of the rounded weights, so that what rounding them did to a row's largest weight cancels (the
// kernel above has two references a row, whose weights are exactly 1), and a reference is its row's maximum again whenever
// any row of the warp has outgrown its own by RESCALE_STEP: O is multiplied for all 32 rows then anyway, and the largest
// weight is exactly 1 more often.  Error of O against 64 bits, kernel above / this one / this one with only the outgrown row's
// reference moved, by 12 (x 1e-3; rounding O alone 1.64-1.66): 32 heads x 4096 x 128 1.996 / 1.924 / 1.970 (146 / 130.4 / 129.2 us),
// 32 / 8 x 10007 x 64 2.052 / 1.978 / 2.024 (695 / 572 / 574), 256 / 128 x 300 x 64 1.879 / 1.873 / 1.887, 240 / 30 x 461 x 64
// 1.897 / 1.888 / 1.913.
// A tile's products are issued in the order P V (j), Q K^T (j + 1) by one thread.  An S that is there says that the last P V is
// done (a commit covers all that its thread issued before): O may be rescaled, and P written, without another barrier.  That Q K^T
// may take the place of the P that P V reads, with no wait between them, rests on a CTA's products passing its tensor pipe in the
// order of their issue.  PTX promises this for products of one accumulator and shape only; here the accumulators differ (and with
// 64 channels the shape).  Published attention kernels for this architecture rely on it likewise, and the tests compare the bits
// of many runs.
constexpr int NST = 2;                  // iterations in the rings of K and V tiles
constexpr int REGS_PAIR_OTHER = 88;     // (2 x 128 x 208 + 128 x 88 = 384 x 168, what the block is launched with)
constexpr int P_FIRST = 96;             // keys of a step whose P is handed over first

struct __align__(8) PairBars {
    uint64_t q_full[2], q_empty[2], k0_full, k0_done;   // an item's Q tiles; its first K tile, loaded and used
    uint64_t kv_full[NST], kv_empty[NST];   // iteration j: V tile j and K tile j + 1
    uint64_t s_full[2], p_full[2][2], o_full[2];
};
struct alignas(16) PairShared {
    PairBars bar;
    uint32_t tmem_base;
    int abort_flag;
};

// Item i of a CTA: tile[g] of query head[g] (n[g] key tiles; 0: none), longest first, boustrophedon.  Of an odd number of tiles
// it is the first, shortest one that stays alone.
struct PairSched {
    int P, c, NH, T, by_head;
    __device__ __forceinline__ bool item(int i, int (&head)[2], int (&tile)[2], int (&n)[2]) const {
        const unsigned k = (unsigned)i * (unsigned)P + (unsigned)((i & 1) ? (P - 1 - c) : c);
        const unsigned per = (unsigned)(by_head ? NH / 2 : NH), rows = (unsigned)(by_head ? T : (T + 1) / 2);
        if (k >= per * rows) return false;
        const unsigned r = k / per, h = k - r * per, t = rows - 1 - r;
        for (int g = 0; g < 2; ++g) {
            head[g] = (int)(by_head ? 2 * h + g : h);
            tile[g] = by_head ? (int)t : 2 * (int)t + g - (T & 1);
            n[g] = tile[g] + 1;
        }
        return true;
    }
};

template <int KCH>
__global__ void __launch_bounds__(NTHREADS, 1)
prefill_pair_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                    const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o, __nv_bfloat16* __restrict__ O,
                    float* __restrict__ lse, kvm_stats* stats, int NH, int G, int S, float scale2) {
    constexpr int D = KCH * KCHUNK;
    constexpr uint32_t TILE_BYTES = KCH * CHUNK_BYTES;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sQ = smem_raw + (base - smem_u32(smem_raw));  // two Q tiles
    uint8_t* sK = sQ + 2 * TILE_BYTES;
    uint8_t* sV = sK + NST * TILE_BYTES;
    uint8_t* sO = sV + NST * TILE_BYTES;                   // 32 rows of 64 channels per softmax warp
    PairShared& sh = *reinterpret_cast<PairShared*>(sO + NSOFT * 4096);
    volatile int* abort_flag = &sh.abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int T = (S + TILE - 1) / TILE;
    const PairSched sc{(int)gridDim.x, (int)blockIdx.x, NH, T, G % 2 == 0};
    int head[2], tile[2], n[2];

    if (threadIdx.x == 0) {
        mbar_init(&sh.bar.k0_full, 1); mbar_init(&sh.bar.k0_done, 1);
        for (int i = 0; i < NST; ++i) { mbar_init(&sh.bar.kv_full[i], 1); mbar_init(&sh.bar.kv_empty[i], 1); }
        for (int g = 0; g < 2; ++g) {
            mbar_init(&sh.bar.q_full[g], 1); mbar_init(&sh.bar.q_empty[g], 1);
            mbar_init(&sh.bar.s_full[g], 1); mbar_init(&sh.bar.o_full[g], 1);
            for (int h = 0; h < 2; ++h) mbar_init(&sh.bar.p_full[g][h], 4);
        }
        sh.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == NSOFT + 1) tmem_alloc(&sh.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh.tmem_base;
    grid_dependency_wait();

    if (warp >= NSOFT) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_PAIR_OTHER));
      if (warp == NSOFT) {
        // ============================== producer ==============================
        if (lane == 0) {
            uint32_t kv = 0;                                  // K tiles (= V tiles = iterations) before this item
            uint32_t q_ph = 0;                                // bit g: phase of Q tile g
            bool ok = true;
            auto load = [&](uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int t, int h) {
#pragma unroll
                for (int kc = 0; kc < KCH; ++kc) tma_load_3d(dst + kc * CHUNK_BYTES, map, bar, kc * KCHUNK, t * TILE, h);
            };
            for (int i = 0; ok && sc.item(i, head, tile, n); ++i) {
                const int kvhead = head[0] / G, len = max(n[0], n[1]);
                // The first K tile's place is free (the last item's third iteration from the end has been waited for, or it was
                // that item's first tile), and a Q tile's as soon as its own last Q K^T is done.
                if (i > 0) ok = mbar_wait(&sh.bar.k0_done, (i & 1) ^ 1, abort_flag);
                if (!ok) break;
                mbar_expect_tx(&sh.bar.k0_full, TILE_BYTES);
                load(sK + (kv % NST) * TILE_BYTES, &map_k, &sh.bar.k0_full, 0, kvhead);
                for (int g = 0; ok && g < 2; ++g) {
                    if (n[g] == 0) continue;
                    ok = mbar_wait(&sh.bar.q_empty[g], ((q_ph >> g) & 1) ^ 1, abort_flag);
                    if (!ok) break;
                    q_ph ^= 1u << g;
                    mbar_expect_tx(&sh.bar.q_full[g], TILE_BYTES);
                    load(sQ + g * TILE_BYTES, &map_q, &sh.bar.q_full[g], tile[g], head[g]);
                }
                for (int j = 0; ok && j < len; ++j) {
                    const uint32_t x = kv + (uint32_t)j, s = x % NST;
                    ok = mbar_wait(&sh.bar.kv_empty[s], ((x / NST) & 1) ^ 1, abort_flag);
                    if (j == 1) ok = ok && mbar_wait(&sh.bar.k0_done, i & 1, abort_flag);   // K tile 2 takes the first one's place
                    if (!ok) break;
#ifdef KVM_TEST_DROP_B_STAGE
                    if (x == (uint32_t)(KVM_TEST_DROP_B_STAGE)) continue;   // test build only: these tiles never arrive
#endif
                    mbar_expect_tx(&sh.bar.kv_full[s], TILE_BYTES * (1u + (j + 1 < len)));
                    if (j + 1 < len) load(sK + ((x + 1) % NST) * TILE_BYTES, &map_k, &sh.bar.kv_full[s], j + 1, kvhead);
                    load(sV + s * TILE_BYTES, &map_v, &sh.bar.kv_full[s], j, kvhead);
                }
                kv += (uint32_t)len;
            }
            if (*abort_flag)                                  // copies already issued land (bounded)
                for (uint32_t it = 0; it < (1u << 14); ++it) mbar_try(&sh.bar.k0_full, 0);
        }
      } else if (warp == NSOFT + 1) {
        // ============================== MMA issue ==============================
        // (One warp for both tiles, a tile's two products together: issued by two threads they share the tensor pipe evenly, both
        // tiles' logits arrive at the same time, and the exponentials of both run together and wait together: 4,280 clocks for
        // two steps against 3,070.)
        constexpr uint32_t IDESC_S = idesc_bf16(TILE), IDESC_O = idesc_bf16(D, true);
        const uint64_t dq = smem_desc(base), dk = smem_desc(base + 2 * TILE_BYTES);
        const uint64_t dv = smem_desc_mn(base + (2 + NST) * TILE_BYTES, CHUNK_BYTES);
        const uint32_t q_lo = (uint32_t)dq, k_lo = (uint32_t)dk, hi = (uint32_t)(dk >> 32), v_lo = (uint32_t)dv, v_hi = (uint32_t)(dv >> 32);
        uint32_t kv = 0, p_ph = 0, q_ph = 0;                 // iterations before this item; phases of P and Q (bit g)
        bool ok = true;
        auto logits = [&](int g, uint32_t x, bool last) {    // S_g = Q_g K^T with K tile number x; the item's last one
            if (elect_one()) {
#pragma unroll
                for (int kc = 0; kc < KCH; ++kc)
#pragma unroll
                    for (int ks = 0; ks < KCHUNK / 16; ++ks)
                        umma_bf16_lo(tmem_base + g * S_COLS, q_lo + ((g * TILE_BYTES + kc * CHUNK_BYTES + ks * 32) >> 4), hi,
                                     k_lo + (x % NST) * (TILE_BYTES >> 4) + ((kc * CHUNK_BYTES + ks * 32) >> 4), hi, IDESC_S, (kc | ks) ? 1u : 0u);
                umma_commit(&sh.bar.s_full[g]);
                if (last) umma_commit(&sh.bar.q_empty[g]);
            }
        };
        // An item's first logits of a tile come right after the tile's last P V of the item before.
        int nn[2] = {0, 0};
        auto first_logits = [&](int g, int i, uint32_t x) {
            if (nn[g] == 0) return;
            ok = ok && mbar_wait_warp(&sh.bar.k0_full, i & 1, abort_flag) && mbar_wait_warp(&sh.bar.q_full[g], (q_ph >> g) & 1, abort_flag);
            if (!ok) return;
            q_ph ^= 1u << g;
            tc_fence_after();
            logits(g, x, nn[g] == 1);
        };
        bool valid = sc.item(0, head, tile, nn);
        for (int i = 0; ok && valid; ++i) {
            n[0] = nn[0]; n[1] = nn[1];
            const int len = max(n[0], n[1]);
            if (i == 0) {
#pragma unroll
                for (int g = 0; g < 2; ++g) first_logits(g, 0, 0u);
                if (ok && elect_one()) umma_commit(&sh.bar.k0_done);
            }
            valid = sc.item(i + 1, head, tile, nn);
            for (int j = 0; ok && j < len; ++j) {
                const uint32_t x = kv + (uint32_t)j, s = x % NST;
                ok = mbar_wait_warp(&sh.bar.kv_full[s], (x / NST) & 1, abort_flag);
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    if (!ok || j >= n[g]) continue;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {            // the first keys' products run while the last ones' P is made
                        ok = ok && mbar_wait_warp(&sh.bar.p_full[g][h], (p_ph >> g) & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        if (elect_one()) {
#pragma unroll
                            for (int kk = h ? P_FIRST / 16 : 0; kk < (h ? TILE / 16 : P_FIRST / 16); ++kk)   // 16 keys per MMA: 8 columns of P, 2 KB of V
                                umma_bf16_ts(tmem_base + O_COL0 + g * D, tmem_base + g * S_COLS + kk * 8,
                                             v_lo + s * (TILE_BYTES >> 4) + ((kk * 16 * 128) >> 4), v_hi, IDESC_O, (j | kk) ? 1u : 0u);
                            if (h && j == n[g] - 1) umma_commit(&sh.bar.o_full[g]);
                        }
                    }
                    if (!ok) break;
                    p_ph ^= 1u << g;
                    if (j + 1 < n[g]) logits(g, x + 1, j + 2 == n[g]);
                    else if (valid) first_logits(g, i + 1, kv + (uint32_t)len);
                }
                if (ok && elect_one()) umma_commit(&sh.bar.kv_empty[s]);
            }
#pragma unroll
            for (int g = 0; g < 2; ++g)
                if (ok && valid && n[g] == 0) first_logits(g, i + 1, kv + (uint32_t)len);
            if (ok && valid && elect_one()) umma_commit(&sh.bar.k0_done);
            kv += (uint32_t)len;
        }
      }
    } else {
        // ============================== softmax of tile g ==============================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SOFTMAX));
        const int g = warp >> 2, lq = warp & 3;
        const int row = lq * 32 + lane;                      // query row of the tile = TMEM lane
        const uint32_t t_lane = tmem_base + ((uint32_t)(lq * 32) << 16);
        const uint32_t t_s = t_lane + g * S_COLS, t_o = t_lane + O_COL0 + g * D;
        const uint64_t sc2 = pack2(scale2, scale2);
        uint32_t s_ph = 0, o_ph = 0;
        bool ok = true;
        for (int i = 0; sc.item(i, head, tile, n); ++i) {
            const int mine = g ? n[1] : n[0], my_tile = g ? tile[1] : tile[0], my_head = g ? head[1] : head[0];
            if (mine == 0) continue;
            float m = -INFINITY, l = 0.f, lr = 0.f;          // reference maximum (log2 units); sums relative to it: exact, of the rounded weights
#pragma unroll 1
            for (int j = 0; j < mine; ++j) {
                ok = ok && mbar_wait(&sh.bar.s_full[g], s_ph, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                s_ph ^= 1;
                tc_fence_after();
                uint32_t vr[TILE];
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_ld32_issue(t_s + q * 32, vr + q * 32);
                tmem_ld_wait();
#pragma unroll
                for (int q = 0; q < 4; ++q) tmem_ld_fence(vr + q * 32);
                float v[TILE];
#pragma unroll
                for (int c = 0; c < TILE; ++c) v[c] = __uint_as_float(vr[c]);
                if (j == my_tile) {                          // diagonal tile: keys after the query do not exist for it
#pragma unroll
                    for (int c = 0; c < TILE; ++c)
                        if (c > row) v[c] = -INFINITY;
                }
                // p = 2^(x - m), summed in fp32, rounded to bf16 for the tensor core.  The first 32 keys are tried with the
                // reference as it is, beside the search for the step's maximum (which alone takes 300 of 1,700 clocks): the
                // warp's references move only when a row's maximum has outgrown its own by RESCALE_STEP, seldom after the first step.
                uint64_t sum[2] = {0ull, 0ull};
                float rsum[4] = {0.f, 0.f, 0.f, 0.f};
                float pk[16];                                // (two bf16 each)
                auto exponentials = [&](int q) {
                    const uint64_t nm2 = pack2(-m, -m);
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        float x0, x1;
                        unpack2(ffma2(pack2(v[q * 32 + c], v[q * 32 + c + 1]), sc2, nm2), x0, x1);
                        const float e0 = ex2(x0), e1 = ex2(x1);
                        sum[(c >> 1) & 1] = fadd2(sum[(c >> 1) & 1], pack2(e0, e1));
                        const uint32_t r = Vec<__nv_bfloat16>::pack2(e0, e1);
                        add_bf16x2(rsum[c & 2], rsum[(c & 2) + 1], r);
                        pk[c >> 1] = __uint_as_float(r);
                    }
                };
                exponentials(0);
                float mx4[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
                for (int c = 4; c + 7 < TILE; c += 8)
#pragma unroll
                    for (int e = 0; e < 4; ++e) mx4[e] = fmax3(mx4[e], v[c + e], v[c + 4 + e]);
#pragma unroll
                for (int e = 0; e < 4; ++e) mx4[e] = fmaxf(mx4[e], v[TILE - 4 + e]);
                const float mx = fmaxf(fmax3(mx4[0], mx4[1], mx4[2]), mx4[3]) * scale2;
                float alpha = 1.f;
                if (__any_sync(0xffffffffu, mx > m + RESCALE_STEP)) {
                    if (mx > m) { alpha = ex2(m - mx); m = mx; }
                    sum[0] = sum[1] = 0ull;
                    rsum[0] = rsum[1] = rsum[2] = rsum[3] = 0.f;
                    exponentials(0);
                    if (j > 0) {                             // (an S that is there says that the last P V is done)
#pragma unroll
                        for (int q = 0; q < D / 16; ++q) {
                            float o[16];
                            tmem_ld16(t_o + q * 16, o);
#pragma unroll
                            for (int c = 0; c < 16; ++c) o[c] *= alpha;
                            tmem_st16(t_o + q * 16, o);
                        }
                    }
                }
                // (96 keys are handed over first: their products run while the last ones' P is made)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q > 0) exponentials(q);
                    tmem_st16(t_s + q * 16, pk);
                    if (q == P_FIRST / 32 - 1 || q == 3) {
                        tmem_st_wait();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sh.bar.p_full[g][q == 3]);
                    }
                }
                float s0, s1;
                unpack2(fadd2(sum[0], sum[1]), s0, s1);
                l = l * alpha + (s0 + s1);
                lr = lr * alpha + ((rsum[0] + rsum[1]) + (rsum[2] + rsum[3]));
            }
            // ---- item end: O / l, 64 channels of the warp's 32 rows at a time through shared memory (stored by the threads that
            // own the rows, 16 bytes each: 3,000 clocks)
            const int gi = my_tile * TILE + row;
            ok = ok && mbar_wait(&sh.bar.o_full[g], o_ph, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
                o_ph ^= 1;
                tc_fence_after();
                const float f = 1.f / lr;
                uint8_t* buf = sO + warp * 4096;
#pragma unroll
                for (int kc = 0; kc < KCH; ++kc) {
                    uint32_t o[64];
                    tmem_ld32_issue(t_o + kc * 64, o);
                    tmem_ld32_issue(t_o + kc * 64 + 32, o + 32);
                    tmem_ld_wait();
                    tmem_ld_fence(o);
                    tmem_ld_fence(o + 32);
                    if (lane == 0) bulk_wait_read();
                    __syncwarp();
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        float y[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) y[e] = __uint_as_float(o[c * 8 + e]) * f;
                        *reinterpret_cast<uint4*>(buf + lane * 128 + ((c ^ (lane & 7)) << 4)) = Vec<__nv_bfloat16>::pack(y);
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0 && my_tile * TILE + lq * 32 < S)
                        tma_store_3d(&map_o, buf, kc * KCHUNK, my_tile * TILE + lq * 32, my_head);
                }
                tc_fence_before();                           // (the next item's first P says that O has been read)
                if (gi < S) lse[(size_t)my_head * S + gi] = (m + log2f(l)) * LN2;
            } else if (gi < S) {
                // a wait gave up: what this row, and those of the items after it, would have received is marked, not made up
                __nv_bfloat16* orow = O + ((size_t)my_head * S + gi) * D;
                for (int c = 0; c < D; c += 8)
                    *reinterpret_cast<uint4*>(orow + c) = make_uint4(0x7FC07FC0u, 0x7FC07FC0u, 0x7FC07FC0u, 0x7FC07FC0u);
                lse[(size_t)my_head * S + gi] = NAN;
            }
        }
        if (lane == 0) bulk_wait();
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh.abort_flag && stats) stats->status = KVM_E_DEVICE_TIMEOUT;
    if (warp == NSOFT + 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

template <int KCH>
cudaError_t launch_t(const Dims& d, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& mo,
                     __nv_bfloat16* O, float* lse, kvm_stats* stats, cudaStream_t st) {
    const size_t smem = 1024 + (size_t)(1 + 2 * NKV) * KCH * CHUNK_BYTES + NGRP * 2 * CHUNK_BYTES + sizeof(Shared);
    const size_t pair_smem = 1024 + (size_t)(2 + 2 * NST) * KCH * CHUNK_BYTES + NSOFT * 4096 + sizeof(PairShared);
    static std::mutex mu;
    static int sms_of[KVM_MAX_DEVICES] = {};
    cudaError_t e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if (dev < 0 || dev >= KVM_MAX_DEVICES) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!sms_of[dev]) {
            e = cudaFuncSetAttribute(prefill_attend_kernel<KCH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            e = cudaFuncSetAttribute(prefill_pair_kernel<KCH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pair_smem);
            if (e != cudaSuccess) return e;
            if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
            sms_of[dev] = sms;
        }
        sms = sms_of[dev];
    }
    const int T = (d.S + TILE - 1) / TILE;
    const long long items = (long long)d.B * d.Hq * T;
    if (items + sms >= (1ll << 31)) return cudaErrorInvalidValue;   // the schedule counts items in 32 bits
    const int G = d.Hq / d.Hkv;
    const long long heads = (long long)d.B * d.Hq, pairs = G % 2 == 0 ? items / 2 : heads * ((T + 1) / 2);
    // Two tiles at a time where the longest pair is not what a CTA's share is made of: its two tiles take turns where single ones
    // would run beside one another.  (us, single tiles / pairs, steps over T x 148 beside them; D = 128: 8 heads x 4096 tokens 0.9
    // 40.9 / 57.8, 10 heads 1.1 52.3 / 58.7, 12 heads 1.3 62.2 / 59.0, 14 heads 1.6 69.6 / 59.5, 32 heads 3.6 146 / 130; 32 x 1024 1.0
    // 24.7 / 23.4, 48 x 1024 1.5 25.8 / 19.9; D = 64: 100 x 500 1.7 16.5 / 16.2, 32 / 8 x 10007 8.6 695 / 572.)
    bool two = heads * T * (T + 1) >= 3ll * sms * T;
    // Neighbouring tiles of a head are no pair where there is one tile (D = 64: 512 heads 14.4 / 15.5, 1024 heads 23.0 / 24.2; with
    // 128 channels the output's way through shared memory is worth more: 444 heads 15.2 / 14.7, 512 17.4 / 17.6, 1024 31.3 / 28.1),
    // and single tiles are faster where a few CTAs have a second pair (2 tiles, D = 128: 148 heads 13.1 / 11.0, 157 15.2 / 16.0, 193
    // 15.7 / 17.1, 202 17.5 / 16.8; D = 64: 11.0 / 9.1, 12.4 / 13.9, 12.5 / 14.6, 14.4 / 14.7) or a short one beside the longest
    // (4 tiles, D = 64: 94 heads 16.3 / 14.9, 99 16.4 / 17.0, 109 17.0 / 18.0, 114 18.8 / 17.8; D = 128: 104 20.7 / 20.1).
    if (G % 2 != 0) {
        if (T == 1) two = two && KCH == 2;
        if (T == 2) two = two && (heads <= sms || 3 * heads > 4ll * sms);
        if (T == 4) two = two && (KCH == 2 || 3 * heads <= 2ll * sms || 4 * heads > 3ll * sms);
    }
    if (two)
        return launch_dependent(prefill_pair_kernel<KCH>, dim3((unsigned)(pairs < sms ? pairs : sms)), dim3(NTHREADS), pair_smem, st, mq, mk,
                                mv, mo, O, lse, stats, d.B * d.Hq, G, d.S, d.scale * LOG2E);
    const int grid = (int)(items < sms ? items : sms);
    return launch_dependent(prefill_attend_kernel<KCH>, dim3((unsigned)grid), dim3(NTHREADS), smem, st, mq, mk, mv, O, lse, stats, d.B,
                            d.Hq, d.Hkv, d.S, d.scale * LOG2E);
}

}  // namespace

cudaError_t launch_prefill_attend(const Dims& d, const void* Q, const void* K, const void* V, void* O, float* lse,
                                  kvm_stats* stats, cudaStream_t st) {
    CUtensorMap mq, mk, mv, mo;
    if (!make_map(&mq, Q, d.B * d.Hq, d.S, d.D) || !make_map(&mk, K, d.B * d.Hkv, d.S, d.D) ||
        !make_map(&mv, V, d.B * d.Hkv, d.S, d.D) || !make_map(&mo, O, d.B * d.Hq, d.S, d.D, 32))
        return cudaErrorNotSupported;
    __nv_bfloat16* Ob = reinterpret_cast<__nv_bfloat16*>(O);
    return d.D == 128 ? launch_t<2>(d, mq, mk, mv, mo, Ob, lse, stats, st) : launch_t<1>(d, mq, mk, mv, mo, Ob, lse, stats, st);
}

}  // namespace kvm
