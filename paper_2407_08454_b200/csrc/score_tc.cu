// Aggregated attention scores on the 5th-generation tensor cores (bf16 inputs).
//
//   pass 1 (row pass)     lse_i = ln sum_{j<=i} exp(c q_i.k_j)                     Eq. 1, causal
//   pass 2 (column pass)  a_j   = (1/G) sum_g sum_{i>=j} exp(c q^g_i.k_j - lse^g_i)  Algorithm 2 / Eq. 6, Section 5.2
//
// Both passes are the same machine.  A work item owns one 128-row "A" tile that
// stays in shared memory (a query tile in pass 1, a key tile in pass 2) and
// streams the 128-row "B" tiles it interacts with under the causal mask (key
// tiles 0..it, resp. query tiles jt..T-1 of each of the G query heads).  A
// step is one 128x128xD tcgen05.mma chain into a 128-column TMEM accumulator
// whose lanes are the A rows.  In pass 1 a thread therefore owns a
// query row and keeps its running max / sum; in pass 2 the product is computed
// transposed (A = keys), so a thread owns a key and adds up its column of the
// attention map in registers, with no cross-lane reduction.
//
// Pass 2 needs exp(c s_ij - lse_i) with lse varying along the accumulator's columns.  Instead of
// fetching lse per column in the epilogue, pass 1 stores e_i = -lse_i / c as three bf16 terms
// (hi + mid + lo, 24 significant bits) in a 16-channel side tensor, and pass 2 appends one more
// K = 16 MMA per step: A' = ones in the three channels, B' = that side tensor.  The tensor core,
// which is far from busy here, then delivers q.k - lse/c directly and the epilogue is a bare
// multiply, exponential and add per logit.
//
// One CTA per SM, persistent, warp-specialised:
//   warps 0-15 epilogue: four groups of four take the steps in turn, each with an accumulator of its
//              own; a warp reads TMEM lanes 32*(w%4).., does exp2 on the SFUs, keeps row/column state
//   warp  16   producer: TMA (cp.async.bulk.tensor, 128B swizzle) into a ring of four B tiles
//   warp  17   MMA issue: one thread issues tcgen05.mma / tcgen05.commit; owns TMEM
//   warps 18-19 the neighbour-key similarities, on the side
// How the work is dealt to the CTAs: score_plan.cuh.
//
// What bounds the passes: one exponential per logit on the special-function unit (1,024 clocks a step; 88 % of the elapsed
// cycles of a single launch on 32 / 8 heads x 32768, 75 % on 32 heads x 4096, whose CTAs have 114 steps each), at the clock
// that the 1 kW power limit leaves (1,700-1,850 of 1,965 MHz in sustained calls; 32 heads x 4096 x 128: 97 us a pass, 58 at
// full clock and 100 %).  The power goes to all of it: with the exponentials replaced by a multiply
// 92 % of the energy is left, with an eighth of the products 75 %, without the B tiles' way from L2 80-95 %.
//
// Every wait on an mbarrier is bounded.  A wait that runs out raises a flag in
// shared memory; from then on every role stops touching tensor memory and
// barriers' payloads, finishes its loops without waiting, the outputs of the
// affected items are poisoned with NaN, kvm_stats.status is set when given,
// tensor memory is freed and the kernel returns.
//
// Two compile-time switches exist for the test of that give-up path and are never set in the
// library that ships: KVM_TEST_WAIT_LIMIT_CLOCKS shortens the limit of every wait, and
// KVM_TEST_DROP_SCORE_STEP = k makes the producer of block KVM_TEST_DROP_CTA leave out its k-th B stage (barrier not
// armed, copies not issued), so that the MMA warp's wait for it runs out.
#include <cuda.h>

#include <mutex>
#include <type_traits>

#include "score_plan.cuh"
#include "similarity_core.cuh"
#include "tc_common.cuh"

namespace kvm {
namespace {

using namespace tc;
using plan::Plan;
using plan::Walk;

constexpr int TILE = plan::TILE;     // rows of an A or B tile = MMA M = MMA N
constexpr int KCHUNK = 64;           // bf16 elements per 128-byte swizzle row
constexpr int NSTAGE = 4;            // ring of B tiles
constexpr int NGRP = 4;              // epilogue groups of four warps = accumulators of 128 TMEM columns (all 512)
constexpr int NSLOT = 5;             // item-end buffers in rotation (see the item end)
constexpr int PCH = 16;              // channels of the lse side tensor (one K = 16 MMA slice; 3 are used)
constexpr uint32_t PTILE_BYTES = TILE * PCH * 2;   // 4 KB: 128 rows x 32 B
constexpr int NEPI_WARPS = 4 * NGRP;
constexpr int QCOLS = 32;               // columns of one TMEM load (a "quarter" of a tile)
constexpr int NSIM_WARPS = 2;           // neighbour-key similarities on the side (one of the two passes)
constexpr int SIM_RUN = 8;              // consecutive tokens per lane group and round trip
constexpr int NTHREADS = (NEPI_WARPS + 2 + NSIM_WARPS) * 32;
constexpr float LOG2E = 1.4426950408889634f;

constexpr uint32_t IDESC = tc::idesc_bf16(TILE);

// ------------------------------------------------------------------ per-chunk arithmetic of the two passes
// A chunk is 32 consecutive accumulator columns of this thread's row, already masked with -inf where the
// causal mask or the sequence end excludes them.  The exponentials' results are added one by one: packing them
// into pairs for a packed add costs a register move per result, which is more than the add it saves.
//
// Row pass: fold the chunk into the running maximum m and sum l (log2 units: x = v * scale2).
__device__ __forceinline__ void chunk_row_pass(const float (&v)[QCOLS], float& m, float& l, float scale2, uint64_t sc2) {
    float mx[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        mx[c] = fmax3(v[c], v[c + 4], v[c + 8]);
        mx[c] = fmax3(mx[c], v[c + 12], v[c + 16]);
        mx[c] = fmax3(mx[c], v[c + 20], v[c + 24]);
        mx[c] = fmaxf(mx[c], v[c + 28]);
    }
    const float mtile = fmaxf(fmax3(mx[0], mx[1], mx[2]), mx[3]);
    const float mnew = fmaxf(m, mtile * scale2);
    if (mnew > -INFINITY) {
        // packed multiply-add for the exponents (the accumulator registers come in adjacent pairs)
        const uint64_t nm2 = pack2(-mnew, -mnew);
        float sum[8] = {l * ex2(m - mnew), 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < QCOLS; c += 2) {
            float x0, x1;
            unpack2(ffma2(pack2(v[c], v[c + 1]), sc2, nm2), x0, x1);
            sum[c & 7] += ex2(x0);
            sum[(c + 1) & 7] += ex2(x1);
        }
        l = ((sum[0] + sum[1]) + (sum[2] + sum[3])) + ((sum[4] + sum[5]) + (sum[6] + sum[7]));
        m = mnew;
    }
}
// Column pass: the accumulator already holds q.k - lse/c; scale, exponentiate, add to eight partial sums.
__device__ __forceinline__ void chunk_col_pass(const float (&v)[QCOLS], float (&acc)[8], uint64_t sc2) {
#pragma unroll
    for (int c = 0; c < QCOLS; c += 2) {
        float x0, x1;
        unpack2(fmul2(pack2(v[c], v[c + 1]), sc2), x0, x1);
        acc[c & 7] += ex2(x0);
        acc[(c + 1) & 7] += ex2(x1);
    }
}

struct __align__(8) Barriers {
    uint64_t full_a[2], empty_a[2];
    uint64_t full_b[NSTAGE], empty_b[NSTAGE];
    uint64_t acc_full[NGRP], acc_empty[NGRP];
};

struct alignas(16) Shared {
    Barriers bar;
    uint32_t tmem_base;
    int abort_flag;
    // Partial sums of the epilogue groups at item end, in NSLOT buffers used in rotation, and how many of the four warps
    // that own a lane quarter's rows have delivered theirs.  (The row pass also needs the partial maxima and keeps both
    // arrays where the column pass keeps its side tiles and ones, which the row pass does not have.)
    float part_l[NSLOT][NGRP][TILE];
    int arrived[NSLOT][4];
};

// e = -lse / c in the accumulator's units as hi + mid + lo, the side tensor's three channels.
__device__ __forceinline__ void store_side(__nv_bfloat16* dst_row, float e) {
    const __nv_bfloat16 eh = __float2bfloat16_rn(e);
    const float r1 = e - __bfloat162float(eh);
    const __nv_bfloat16 em = __float2bfloat16_rn(r1);
    const __nv_bfloat16 el = __float2bfloat16_rn(r1 - __bfloat162float(em));
    uint4* dst = reinterpret_cast<uint4*>(dst_row);
    dst[0] = make_uint4((uint32_t)__bfloat16_as_ushort(eh) | ((uint32_t)__bfloat16_as_ushort(em) << 16),
                        (uint32_t)__bfloat16_as_ushort(el), 0u, 0u);
    dst[1] = make_uint4(0u, 0u, 0u, 0u);
}

// Tensor maps of the layers' queries and keys, the keys themselves, and the map of the side tensor (which lies in the
// workspace: one for all layers); units and query heads of a layer.
template <int NL> struct Maps {
    CUtensorMap q[NL], k[NL], side;
    const __nv_bfloat16* keys[NL];
    int U, H;
};

// out: the column pass's scores [U,S], or its partial sums [piece][U,S] when items are cut; states: the row pass's
// partial (maximum, sum) per piece and row when items are cut, else it writes the side tensor.
template <int KCH, int PASS, int NL>
__global__ void __launch_bounds__(NTHREADS, 1)
score_tc_kernel(const __grid_constant__ Maps<NL> maps, __nv_bfloat16* __restrict__ lsep_out, float2* __restrict__ states,
                float* __restrict__ out, kvm_stats* stats, const Plan plan, int Hq, int Hkv, int S, float scale2,
                float* __restrict__ sim_out) {
    constexpr int pass = PASS;
    extern __shared__ uint8_t smem_raw[];
    constexpr uint32_t CHUNK_BYTES = TILE * 128;            // one [128 rows x 64 bf16] TMA box
    constexpr uint32_t TILE_BYTES = KCH * CHUNK_BYTES;      // a tile: [KCH][128 rows][128 B]
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* aligned = smem_raw + (base - smem_u32(smem_raw));
    uint8_t* sA = aligned;                                  // 2 A tiles
    uint8_t* sB = aligned + 2 * TILE_BYTES;                 // NSTAGE B tiles
    uint8_t* sP = sB + NSTAGE * TILE_BYTES;                 // NSTAGE lse side tiles (pass 2)
    uint8_t* sOnes = sP + NSTAGE * PTILE_BYTES;             // constant A' tile: ones in the used channels
    Shared& sh = *reinterpret_cast<Shared*>(sOnes + PTILE_BYTES);
    volatile int* abort_flag = &sh.abort_flag;
    static_assert(2 * NSLOT * NGRP * TILE * sizeof(float) <= (NSTAGE + 1) * PTILE_BYTES, "the row pass's item-end buffers fit the side tiles' space");
    float* part_m = reinterpret_cast<float*>(sP);                                   // [NSLOT][NGRP][TILE], row pass only
    float* part_l = (pass == 1) ? part_m + NSLOT * NGRP * TILE : &sh.part_l[0][0][0];   // [NSLOT][NGRP][TILE]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = plan.G, T = plan.T;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) { mbar_init(&sh.bar.full_a[i], 1); mbar_init(&sh.bar.empty_a[i], 1); }
        for (int i = 0; i < NSTAGE; ++i) { mbar_init(&sh.bar.full_b[i], 1); mbar_init(&sh.bar.empty_b[i], 1); }
        for (int i = 0; i < NGRP; ++i) { mbar_init(&sh.bar.acc_full[i], 1); mbar_init(&sh.bar.acc_empty[i], 4); }
        sh.abort_flag = 0;
        for (int i = 0; i < NSLOT * 4; ++i) (&sh.arrived[0][0])[i] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (pass == 2 && threadIdx.x < PTILE_BYTES / 16) {
        // every 16-byte chunk of every row = bf16 {1, 1, 1, 0, 0, 0, 0, 0}: the same under any swizzle; the B'
        // side tensor is zero outside channels 0..2, so the ones of the second chunk multiply zeros
        reinterpret_cast<uint4*>(sOnes)[threadIdx.x] = make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor core's reads
    }
    if (warp == NEPI_WARPS + 1) tmem_alloc(&sh.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh.tmem_base;
    // (the set-up above runs beside the end of the kernel before this one; the column pass reads what that wrote)
    grid_dependency_wait();
    Walk<PASS> w;
    w.init(plan);

    // `cnt` counts steps of this CTA across items; step cnt goes to B stage cnt % NSTAGE and epilogue group cnt % NGRP.
    if (warp == NEPI_WARPS) {
        // ============================== producer ==============================
        if (lane == 0) {
            uint32_t cnt = 0;
            bool ok = true;
            int last_a[2] = {-1, -1}, last_b[NSTAGE];      // parity of the last load issued per buffer (-1: none)
            for (int s = 0; s < NSTAGE; ++s) last_b[s] = -1;
            for (int n = 0; ok && w.valid(); ++n, w.next(plan)) {
                const int ab = n & 1;
                ok = mbar_wait(&sh.bar.empty_a[ab], ((n >> 1) & 1) ^ 1, abort_flag);
                if (!ok) break;
                last_a[ab] = (n >> 1) & 1;
                const int per_layer = (pass == 1) ? maps.H : maps.U, layer = NL > 1 ? w.head / per_layer : 0;
                const int head = w.head - layer * per_layer;             // within its layer
                const CUtensorMap* mapA = (pass == 1) ? &maps.q[layer] : &maps.k[layer];
                const CUtensorMap* mapB = (pass == 1) ? &maps.k[layer] : &maps.q[layer];
                mbar_expect_tx(&sh.bar.full_a[ab], TILE_BYTES);
#pragma unroll
                for (int kc = 0; kc < KCH; ++kc)
                    tma_load_3d(sA + ab * TILE_BYTES + kc * CHUNK_BYTES, mapA, &sh.bar.full_a[ab], kc * KCHUNK,
                                w.tile * TILE, head);
                const int b = head / (pass == 1 ? Hq : Hkv), hh = head % (pass == 1 ? Hq : Hkv), per = T - w.tile;
                int bhead = (pass == 1) ? b * Hkv + hh / G : b * Hq + hh * G + w.i0 / per;   // B tile cursor, advanced incrementally
                int btile = (pass == 1) ? w.i0 : w.tile + w.i0 % per;
                for (int t = 0; t < w.n; ++t, ++cnt) {
                    const int s = cnt % NSTAGE;
                    ok = mbar_wait(&sh.bar.empty_b[s], ((cnt / NSTAGE) & 1) ^ 1, abort_flag);
                    if (!ok) break;
#ifdef KVM_TEST_DROP_SCORE_STEP
                    if (blockIdx.x == KVM_TEST_DROP_CTA && cnt == (uint32_t)(KVM_TEST_DROP_SCORE_STEP)) continue;   // test build only: this stage never arrives
#endif
                    last_b[s] = (cnt / NSTAGE) & 1;
                    mbar_expect_tx(&sh.bar.full_b[s], TILE_BYTES + (pass == 2 ? PTILE_BYTES : 0u));
#pragma unroll
                    for (int kc = 0; kc < KCH; ++kc)
                        tma_load_3d(sB + s * TILE_BYTES + kc * CHUNK_BYTES, mapB, &sh.bar.full_b[s], kc * KCHUNK, btile * TILE, bhead);
                    if (pass == 2) tma_load_3d(sP + s * PTILE_BYTES, &maps.side, &sh.bar.full_b[s], 0, btile * TILE, layer * maps.H + bhead);
                    if (++btile == T && pass == 2) { btile = w.tile; ++bhead; }   // next query head of the group
                }
            }
            // Copies already issued complete on their own; before shared memory is given
            // back, wait (bounded) for the ones nobody consumed.
            if (*abort_flag) {
                for (int s = 0; s < NSTAGE; ++s)
                    for (uint32_t it = 0; last_b[s] >= 0 && it < (1u << 16); ++it)
                        if (mbar_try(&sh.bar.full_b[s], (uint32_t)last_b[s])) break;
                for (int s = 0; s < 2; ++s)
                    for (uint32_t it = 0; last_a[s] >= 0 && it < (1u << 16); ++it)
                        if (mbar_try(&sh.bar.full_a[s], (uint32_t)last_a[s])) break;
            }
        }
    } else if (warp == NEPI_WARPS + 1) {
        // ============================== MMA issue ==============================
        if (lane == 0) {
            uint32_t cnt = 0;
            bool ok = true;
            // descriptors of one layout differ in the low half only (the 16-byte-unit start address)
            const uint64_t d0 = smem_desc(base), p0 = smem_desc_sw32(base + (2 + NSTAGE) * TILE_BYTES);
            const uint32_t dhi = (uint32_t)(d0 >> 32), phi = (uint32_t)(p0 >> 32);
            const uint32_t desc_a0 = (uint32_t)d0, desc_b0 = desc_a0 + ((2 * TILE_BYTES) >> 4);
            const uint32_t desc_p0 = (uint32_t)p0, desc_ones = desc_p0 + ((NSTAGE * PTILE_BYTES) >> 4);
            for (int n = 0; ok && w.valid(); ++n, w.next(plan)) {
                const int ab = n & 1;
                ok = mbar_wait(&sh.bar.full_a[ab], (n >> 1) & 1, abort_flag);
                if (!ok) break;
                for (int t = 0; t < w.n; ++t, ++cnt) {
                    const int s = cnt % NSTAGE, as = cnt % NGRP;
                    ok = mbar_wait(&sh.bar.full_b[s], (cnt / NSTAGE) & 1, abort_flag) &&
                         mbar_wait(&sh.bar.acc_empty[as], ((cnt / NGRP) & 1) ^ 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t da = desc_a0 + ab * (TILE_BYTES >> 4), db = desc_b0 + s * (TILE_BYTES >> 4);
                    const uint32_t d = tmem_base + as * TILE;
#pragma unroll
                    for (int kc = 0; kc < KCH; ++kc)
#pragma unroll
                        for (int ks = 0; ks < KCHUNK / 16; ++ks)
                            umma_bf16_lo(d, da + ((kc * CHUNK_BYTES + ks * 32) >> 4), dhi, db + ((kc * CHUNK_BYTES + ks * 32) >> 4),
                                         dhi, IDESC, (kc | ks) ? 1u : 0u);
                    if (pass == 2)                         // + ones x (-lse/c): one more K = 16 slice
                        umma_bf16_lo(d, desc_ones, phi, desc_p0 + s * (PTILE_BYTES >> 4), phi, IDESC, 1u);
                    umma_commit(&sh.bar.empty_b[s]);       // B stage reusable once these MMAs retire
                    umma_commit(&sh.bar.acc_full[as]);     // accumulator ready for the epilogue
                }
                if (ok) umma_commit(&sh.bar.empty_a[ab]);  // A tile reusable
            }
        }
    } else if (warp >= NEPI_WARPS + 2) {
        // ============================== similarity on the side ==============================
        // Eq. 2 needs nothing but K, and the epilogue warps leave issue slots and memory bandwidth unused:
        // the key rows are dealt to these warps of all CTAs in runs of SIM_RUN tokens.
        if (sim_out) {
            constexpr int D = KCH * KCHUNK, LPR = D / 8, GPW = 32 / LPR;
            const int runs = (S + SIM_RUN - 1) / SIM_RUN;
            // (32-bit arithmetic: U * runs is far below 2^31 for tensors that fit a GPU — the launcher
            // checks it — and a 64-bit division per run would cost a third of the run's own work)
            const unsigned n_runs = (unsigned)plan.U * (unsigned)runs;
            const int gl = lane % LPR, gbase = lane / LPR * LPR;
            const unsigned gmask = (LPR == 32) ? 0xffffffffu : (((1u << LPR) - 1u) << gbase);
            const unsigned stride = gridDim.x * NSIM_WARPS * GPW;
            for (unsigned g = (blockIdx.x * NSIM_WARPS + (warp - NEPI_WARPS - 2)) * GPW + lane / LPR;
                 g < n_runs; g += stride) {
                const unsigned u = g / (unsigned)runs, layer = NL > 1 ? u / (unsigned)maps.U : 0u;
                const int j0 = (int)(g - u * (unsigned)runs) * SIM_RUN;
                simcore::run<__nv_bfloat16, D, SIM_RUN>(maps.keys[layer] + (size_t)(u - layer * maps.U) * S * D, sim_out + (size_t)u * S, j0,
                                                        min(j0 + SIM_RUN, S), gl, gbase, gmask);
            }
        }
    } else {
        // ============================== epilogue ==============================
        // Four groups of four warps take the steps in turn, each with an accumulator of its own, so that one group's
        // waits, TMEM loads and bookkeeping run beside the other three groups' exponentials.  Within a group a warp
        // owns a TMEM lane quarter and takes the step's 128 columns 32 at a time; the accumulator is handed back as
        // soon as the last load has landed.  The loops are kept short: unrolled whole, with a copy for each mask, they leave
        // the instruction cache (see the fp32 kernel).
        const int lq = warp & 3, grp = warp >> 2;
        const int row = lq * 32 + lane;                      // A row = TMEM lane
        const uint32_t t_lane = tmem_base + ((uint32_t)(lq * 32) << 16) + grp * TILE;
        const uint64_t sc2 = pack2(scale2, scale2);
        bool ok = true;
        uint32_t cnt = 0, own = 0;                           // steps of the CTA before this item; this group's steps
        uint32_t multi = 0;                                  // items of several steps so far (they rotate the buffers)
        for (; w.valid(); w.next(plan)) {
            float m = -INFINITY, l = 0.f;                    // pass 1 state
            float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // pass 2 state: eight partial sums
            const int first = (grp - (int)cnt) & (NGRP - 1); // this group's first step of the item
            const int per = T - w.tile;
            int bt = 0;                                      // pass 2: offset of the step's query tile from the item's key tile
            if (pass == 2) bt = (w.i0 + first) % per;
            for (int t = first; t < w.n; t += NGRP, ++own) {
                ok = mbar_wait(&sh.bar.acc_full[grp], own & 1, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (ok) tc_fence_after();
                const bool diag = (pass == 1) ? w.i0 + t == w.tile : bt == 0;
                const int left = (pass == 2) ? S - (w.tile + bt) * TILE : TILE;      // live columns (queries < S)
                // 32 columns; the last ones of the accumulator release it once they have landed
                auto quarter = [&](int cq, bool last, auto masked) {
                    uint32_t vr[QCOLS];
                    tmem_ld32_issue(t_lane + cq * QCOLS, vr);
                    tmem_ld_wait();
                    if (last) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sh.bar.acc_empty[grp]);
                    }
                    tmem_ld_fence(vr);
                    float v[QCOLS];
#pragma unroll
                    for (int c = 0; c < QCOLS; ++c) v[c] = __uint_as_float(vr[c]);
                    const int ncol = left - cq * QCOLS;
                    if (decltype(masked)::value && ((diag && cq == lq) || ncol < QCOLS)) {
                        const int lo = (pass == 2 && diag && cq == lq) ? lane : 0;                 // query before key
                        const int hi = (pass == 1) ? lane + 1 : ncol;                              // key after query; past the end
#pragma unroll
                        for (int c = 0; c < QCOLS; ++c)
                            if (c < lo || c >= hi) v[c] = -INFINITY;
                    }
                    if (pass == 1) chunk_row_pass(v, m, l, scale2, sc2);
                    else chunk_col_pass(v, acc, sc2);
                };
                if (ok && !diag && left >= TILE) {
                    // (two quarters per round: 1 % less time than one on 32768 tokens, four the same)
#pragma unroll 2
                    for (int cq = 0; cq < 4; ++cq) quarter(cq, cq == 3, std::false_type{});
                } else {
                    // On the diagonal tile whole 32-column quarters are masked (left out) or valid, one is mixed.
                    const int q0 = (pass == 2 && diag) ? lq : 0, q1 = (pass == 1 && diag) ? lq + 1 : 4;
#pragma unroll 1
                    for (int cq = q0; ok && cq < q1; ++cq) quarter(cq, cq == q1 - 1, std::true_type{});
                }
                if (pass == 2) { bt += NGRP; while (bt >= per) bt -= per; }
            }
            cnt += (uint32_t)w.n;
            // ---- item end.  The groups that had a step leave their partial states in shared memory; of the warps that
            // own a row whichever comes last combines them in a fixed order (so the result does not depend on who does
            // it) and stores.  Nobody waits: a group goes straight on to the next item.  A group without a step has
            // nothing to say, and the only group of a one-step item keeps its state to itself.
            // (Buffers: when a warp has finished step k the MMA thread has issued steps k - 3 .. k, so the other
            // groups have handed steps up to k - 5 .. k - 7 back but may not have delivered them.  Items of several
            // steps rotate the buffers; when the one five such items on is delivered, at least 9 steps have passed.)
            const int nstep = min(w.n, NGRP);
            if (first >= nstep) { multi += w.n > 1; continue; }
            const int gi = w.tile * TILE + row;
            const float mine = (pass == 1) ? l : ((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7]));
            float M = m, L = mine;
            // (After a give-up nothing keeps the groups within a few steps of one another, and an item's buffer could be
            // taken for a later one's: every warp marks the rows of its items by itself then.)
            bool bad = __any_sync(0xffffffffu, *abort_flag != 0);
            if (w.n > 1) {
                const int slot = multi % NSLOT;
                ++multi;
                if (!bad) {
                    float* pm = part_m + slot * NGRP * TILE + row;       // + q * TILE: the group with the item's step q
                    float* pl = part_l + slot * NGRP * TILE + row;
                    if (pass == 1) pm[first * TILE] = m;
                    pl[first * TILE] = mine;
                    __syncwarp();
                    int before = 0;
                    if (lane == 0) {
                        __threadfence_block();
                        before = atomicAdd(&sh.arrived[slot][lq], 1);
                    }
                    before = __shfl_sync(0xffffffffu, before, 0);
                    if (before != nstep - 1) continue;
                    __threadfence_block();
                    if (lane == 0) sh.arrived[slot][lq] = 0;
                    L = 0.f;
                    if (pass == 1) {
                        M = pm[0];
                        for (int q = 1; q < nstep; ++q) M = fmaxf(M, pm[q * TILE]);
                        for (int q = 0; q < nstep; ++q) L += pl[q * TILE] * ex2(pm[q * TILE] - M);
                    } else {
                        for (int q = 0; q < nstep; ++q) L += pl[q * TILE];
                    }
                    bad = *abort_flag != 0;      // (read again: another group may have given up before it came here)
                }
            }
            if (bad) { M = 0.f; L = NAN; }
            if (gi < S) {
                const size_t at = (size_t)w.head * S + gi;
                if (pass == 1) {
                    // lse in log2 units is M + log2 L
                    if (plan.split_row) states[(size_t)w.piece(plan) * plan.NH * S + at] = make_float2(M, L);
                    else store_side(lsep_out + at * PCH, -(M + log2f(L)) / scale2);
                } else {
                    if (plan.split_col) out[(size_t)w.piece(plan) * plan.U * S + at] = L;
                    else out[at] = L / (float)G;
                }
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh.abort_flag && stats) stats->status = KVM_E_DEVICE_TIMEOUT;
    if (warp == NEPI_WARPS + 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------ host side
// [heads, S, 16] bf16 side tensor of pass 2: boxes of [1, 128 rows, 16 channels] (32-byte rows), 32-byte swizzle.
bool make_map_side(CUtensorMap* map, const void* ptr, int heads, int S) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)PCH, (cuuint64_t)S, (cuuint64_t)heads};
    cuuint64_t strides[2] = {(cuuint64_t)PCH * 2, (cuuint64_t)S * PCH * 2};
    cuuint32_t box[3] = {PCH, TILE, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Caller-supplied natural-log lse -> the side tensor pass 2 multiplies in (e = -lse * log2(e) / scale2 as hi+mid+lo).
__global__ void __launch_bounds__(256) lse_split_kernel(const float* __restrict__ lse, __nv_bfloat16* __restrict__ side,
                                                        long long rows, float neg_log2e_over_scale2) {
    grid_dependency_wait();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < rows) store_side(side + (size_t)i * PCH, __ldcg(lse + i) * neg_log2e_over_scale2);
}

// The row pass's states of cut items -> the side tensor, and the natural-log lse when asked for.
__global__ void __launch_bounds__(256) join_rows_kernel(const float2* __restrict__ states, __nv_bfloat16* __restrict__ side,
                                                        float* __restrict__ lse_out, const Plan plan, int S, float scale2) {
    grid_dependency_wait();
    const size_t rows = (size_t)plan.NH * S, r = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    const int head = (int)(r / S), np = plan.row_pieces(head, (int)(r - (size_t)head * S) / TILE);
    float M = -INFINITY, L = 0.f;
#pragma unroll 4
    for (int x = 0; x < np; ++x) plan::add_state(M, L, __ldcg(states + (size_t)x * rows + r));
    const float lse2 = M + log2f(L);
    store_side(side + r * PCH, -lse2 / scale2);
    if (lse_out) lse_out[r] = lse2 * 0.6931471805599453f;
}

// The row pass's side tensor back to a natural-log lse per query row: lse = -(hi + mid + lo) * scale2 * ln 2.
__global__ void __launch_bounds__(256) side_to_lse_kernel(const __nv_bfloat16* __restrict__ side, float* __restrict__ lse,
                                                          long long rows, float neg_scale2_ln2) {
    grid_dependency_wait();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows) return;
    const uint2 raw = __ldcg(reinterpret_cast<const uint2*>(side + (size_t)i * PCH));
    const float hi = __uint_as_float(raw.x << 16), mid = __uint_as_float(raw.x & 0xffff0000u);
    const float lo = __uint_as_float(raw.y << 16);
    lse[i] = ((hi + mid) + lo) * neg_scale2_ln2;
}

// Partial column sums -> scores.
__global__ void __launch_bounds__(256) combine_kernel(const float* __restrict__ part, float* __restrict__ scores,
                                                      const Plan plan, int S) {
    grid_dependency_wait();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < S) scores[(size_t)blockIdx.y * S + j] = plan::column_sum(part, plan, S, blockIdx.y, j);
}

// How the passes are dealt: items are cut where the longest one exceeds a CTA's equal share by more than cutting costs.
// Rows: a launch (join_rows_kernel, about as long as four steps).  Columns: the additions in the kernel that reads the
// scores, about as long as three (32 heads x 389 tokens, 3 steps per CTA and items of up to 4: cut 30.0 us a call,
// whole 29.2; 32 query / 8 KV heads x 2048 tokens, 30 and up to 64: column pass 28.3 us cut, 49.9 whole).
bool make_plan(const Dims& d, Plan& p) {
    if (!plan::make(d, p)) return false;
    if ((long long)d.B * d.Hkv * ((d.S + SIM_RUN - 1) / SIM_RUN) + plan::CTAS * 64 >= (1ll << 31)) return false;   // (the similarity warps' runs)
    p.split_row = p.T > (int)p.q + 4;
    p.split_col = p.G * p.T > (int)p.q + 3;
    if (p.split_row) p.pr = p.pieces(p.T);
    if (p.split_col) p.pc = p.pieces(p.G * p.T);
    return true;
}
struct Scratch {
    size_t states, part, bytes;      // offsets: the side tensor comes first
};
Scratch layout(const Dims& d, const Plan& p) {
    auto up = [](size_t n) { return (n + 255) / 256 * 256; };
    Scratch s;
    const size_t rows = (size_t)p.NH * d.S;
    s.states = up(rows * PCH * 2);
    s.part = s.states + (p.split_row ? up(rows * p.pr * sizeof(float2)) : 0);
    s.bytes = s.part + (p.split_col ? (size_t)p.U * d.S * p.pc * sizeof(float) : 0);
    return s;
}

template <int KCH, int NL>
cudaError_t launch_t(const Dims& d, const Plan& plan, const Maps<NL>& maps, const float* lse_in, char* scratch, float* scores,
                     kvm_stats* stats, cudaStream_t st, float* sim_out, float* lse_out, ScorePart* parts) {
    const size_t smem = 1024 + (size_t)(2 + NSTAGE) * KCH * TILE * 128 + (size_t)(NSTAGE + 1) * PTILE_BYTES + sizeof(Shared);
    // the shared-memory opt-in is made once per device and kernel instantiation
    static std::mutex mu;
    static bool done[KVM_MAX_DEVICES] = {};
    cudaError_t e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if (dev < 0 || dev >= KVM_MAX_DEVICES) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!done[dev]) {
            e = cudaFuncSetAttribute(score_tc_kernel<KCH, 1, NL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            e = cudaFuncSetAttribute(score_tc_kernel<KCH, 2, NL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            done[dev] = true;
        }
    }
    const Scratch sc = layout(d, plan);
    __nv_bfloat16* side = reinterpret_cast<__nv_bfloat16*>(scratch);
    float2* states = reinterpret_cast<float2*>(scratch + sc.states);
    float* part = reinterpret_cast<float*>(scratch + sc.part);
    const float scale2 = d.scale * LOG2E;
    const long long rows = (long long)plan.NH * d.S;
    const dim3 row_blocks((unsigned)((rows + 255) / 256));
    auto grid = [&](int split, int heads) {
        const long long items = (long long)heads * plan.T;
        return dim3(split ? plan.grid_split() : (unsigned)(items < plan::CTAS ? items : plan::CTAS));
    };
    if (!lse_in) {
        // (the kernels wait for what precedes them by themselves, so each is scheduled while that drains)
        e = launch_dependent(score_tc_kernel<KCH, 1, NL>, grid(plan.split_row, plan.NH), dim3(NTHREADS), smem, st, maps, side,
                             states, (float*)nullptr, stats, plan, d.Hq, d.Hkv, d.S, scale2,
                             scores ? (float*)nullptr : sim_out);
        if (e == cudaSuccess && plan.split_row)
            e = launch_dependent(join_rows_kernel, row_blocks, dim3(256), 0, st, (const float2*)states, side, lse_out, plan, d.S, scale2);
        else if (e == cudaSuccess && lse_out)
            e = launch_dependent(side_to_lse_kernel, row_blocks, dim3(256), 0, st, (const __nv_bfloat16*)side, lse_out, rows,
                                 -scale2 * 0.6931471805599453f);
    } else {
        e = launch_dependent(lse_split_kernel, row_blocks, dim3(256), 0, st, lse_in, side, rows, -LOG2E / scale2);
    }
    if (e != cudaSuccess || !scores) return e;        // (row pass only)
    e = launch_dependent(score_tc_kernel<KCH, 2, NL>, grid(plan.split_col, plan.U), dim3(NTHREADS), smem, st, maps,
                         (__nv_bfloat16*)nullptr, (float2*)nullptr, plan.split_col ? part : scores, stats, plan, d.Hq, d.Hkv,
                         d.S, scale2, sim_out);
    if (e != cudaSuccess || !plan.split_col) return e;
    if (parts) {                                      // the caller's next kernel adds the pieces up
        parts->part = part;
        parts->plan = plan;
        return cudaSuccess;
    }
    return launch_dependent(combine_kernel, dim3((d.S + 255) / 256, d.U), dim3(256), 0, st, (const float*)part, scores, plan, d.S);
}

}  // namespace

// Bytes of scratch: the lse side tensor, and what cut items leave.
size_t score_tc_scratch_bytes(const Dims& d) {
    Plan p;
    return make_plan(d, p) ? layout(d, p).bytes : 0;      // (launching a shape without a plan is refused)
}

// sim_out (nullable): when given, the spare warps of the column pass (of the row pass when scores is NULL and
// the column pass does not run) also write the neighbour-key similarities [U,S] there, so the caller needs no
// similarity kernel.  (Measured on a 32-head, 4096-token layer: 0.9 us less per call beside the column pass
// than beside the row pass; the spare warps share two of the four schedulers with the epilogue warps of two
// TMEM lane quarters, which then lag the others, and an accumulator goes back when its slowest warp is done.)
// scores may be NULL (row pass only); lse_out (nullable) receives the natural-log row log-sum-exp [B,Hq,S].
// parts (nullable): lets the column pass leave partial sums (parts->part set) for the caller's next kernel to add.
template <int NL>
static cudaError_t launch_score_n(const Dims& d, const Layers& L, const float* lse_in, void* scratch, float* scores,
                                  kvm_stats* stats, cudaStream_t st, float* sim_out, float* lse_out, ScorePart* parts) {
    Maps<NL> maps;
    Plan plan;
    if (!make_plan(d, plan)) return cudaErrorInvalidValue;
    maps.U = L.U; maps.H = L.H;
    for (int l = 0; l < L.n; ++l) {
        if (!make_map(&maps.q[l], L.Q[l], L.H, d.S, d.D) || !make_map(&maps.k[l], L.K[l], L.U, d.S, d.D)) return cudaErrorNotSupported;
        maps.keys[l] = reinterpret_cast<const __nv_bfloat16*>(L.K[l]);
    }
    if (!make_map_side(&maps.side, scratch, d.B * d.Hq, d.S)) return cudaErrorNotSupported;
    auto fn = d.D == 128 ? launch_t<2, NL> : launch_t<1, NL>;
    return fn(d, plan, maps, lse_in, (char*)scratch, scores, stats, st, sim_out, lse_out, parts);
}
// d: the layers together (a batch of n times a layer's).
cudaError_t launch_score_tc(const Dims& d, const Layers& L, const float* lse_in, void* scratch, float* scores, kvm_stats* stats,
                            cudaStream_t st, float* sim_out, float* lse_out, ScorePart* parts) {
    auto fn = L.n == 1 ? launch_score_n<1> : launch_score_n<MAX_LAYERS>;
    return fn(d, L, lse_in, scratch, scores, stats, st, sim_out, lse_out, parts);
}

}  // namespace kvm
