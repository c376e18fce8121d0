// How the score passes' work is dealt to the CTAs, for both storage types.
//
// A step is one 128 x 128 tile of the causal map.  A row-pass item is a query tile with the key tiles before and at it,
// a column-pass item a key tile with the query tiles at and after it of each of the G query heads.  Both passes have
// the same number of steps.  Two ways to deal them:
//   whole   items sorted by length, dealt boustrophedon: within 2 % of a greedy schedule when a CTA gets several items,
//           and every item's result is final.  The heads are taken in groups whose streamed tiles fit L2 together: the
//           CTAs at work at one time stream the tiles of every head of the group, over and over (128 heads x 4096 x 128
//           without groups: 134 MB of them from HBM 16 times a pass, 430 us at the clock that the power left; 370 with);
//   split   all steps form one list and CTA c takes q = ceil(steps / 148) consecutive ones from c q: balanced to one
//           step whatever the shape (few heads, or few KV heads with long items), but an item that is cut leaves one
//           partial result per piece.
#pragma once
#include "common.cuh"

namespace kvm {
namespace plan {

constexpr int TILE = 128;
constexpr long long GROUP_BYTES = 40ll << 20;
constexpr int MIN_ROUNDS = 6;
constexpr int CTAS = 148;       // (the split is a function of the shape alone, that of all layers that go together, so that results are)

struct Plan {
    int NH, U, G, T;            // query heads and units in total, query heads per unit, tiles per head
    unsigned steps, q;          // steps of a pass, steps per CTA when split
    int split_row, split_col;
    int pr, pc;                 // most pieces of an item (1 when whole)
    int hg_row, hg_col;         // heads (units) of a group when whole
    int rounds_row, rounds_col; // ... and items per CTA and group
    __host__ __device__ unsigned tri() const { return (unsigned)T * (unsigned)(T + 1) / 2; }
    // first step of an item, and how many CTAs share it
    __host__ __device__ unsigned row_start(int head, int tile) const { return (unsigned)head * tri() + (unsigned)tile * (unsigned)(tile + 1) / 2; }
    __host__ __device__ unsigned col_start(int u, int tile) const {
        const unsigned jr = (unsigned)(T - 1 - tile);
        return (unsigned)G * ((unsigned)u * tri() + jr * (jr + 1) / 2);
    }
    __host__ __device__ int row_pieces(int head, int tile) const {
        const unsigned f = row_start(head, tile);
        return (int)((f + (unsigned)tile) / q - f / q) + 1;
    }
    __host__ __device__ int col_pieces(int u, int tile) const {
        const unsigned f = col_start(u, tile);
        return (int)((f + (unsigned)(G * (T - tile)) - 1) / q - f / q) + 1;
    }
    int pieces(int len) const {
        const int n = (len - 1 + (int)q - 1) / (int)q + 1;
        return n < len ? n : len;
    }
    unsigned grid_split() const { return (steps + q - 1) / q; }
};

// Everything but the choice of how to deal (false: more steps than any tensors that fit a GPU have).
inline bool make(const Dims& d, Plan& p) {
    p.NH = d.B * d.Hq; p.U = d.U; p.G = d.G; p.T = (d.S + TILE - 1) / TILE;
    const long long steps = (long long)p.NH * p.T * (p.T + 1) / 2;
    if (steps + (long long)p.NH + CTAS >= (1ll << 31)) return false;
    p.steps = (unsigned)steps;
    p.q = (p.steps + CTAS - 1) / CTAS;
    p.split_row = p.split_col = 0;
    p.pr = p.pc = 1;
    // Every group is dealt in whole rounds of the grid: of the group sizes in the upper half of what L2 takes the one
    // whose last round is fullest, and no groups where one would be dealt in few rounds (a CTA's shares then differ by
    // several percent: 8 units x 32768 tokens, whose CTAs walk the same tiles side by side anyway).
    auto group = [&](int heads, long long bytes_per_head, int& hg, int& rounds) {
        const long long items = (long long)heads * p.T, grid = items < CTAS ? items : CTAS;
        const int most = (int)(GROUP_BYTES / bytes_per_head);
        hg = heads;
        double best = -1.0;
        for (int h = most / 2 + 1; heads > most && h <= most; ++h) {
            const long long r = ((long long)h * p.T + grid - 1) / grid;
            const double full = (double)((long long)h * p.T) / (double)(r * grid);
            if (r >= MIN_ROUNDS && full > best) { best = full; hg = h; }
        }
        rounds = (int)(((long long)hg * p.T + grid - 1) / grid);
    };
    const long long head_bytes = (long long)d.S * d.D * (d.dtype == KVM_BF16 ? 2 : 4);
    group(p.NH, (head_bytes + p.G - 1) / p.G, p.hg_row, p.rounds_row);     // a unit's G heads stream the same keys
    group(p.U, head_bytes * p.G, p.hg_col, p.rounds_col);
    return true;
}

__device__ __forceinline__ unsigned tri_root(unsigned x) {       // largest t with t (t + 1) / 2 <= x
    unsigned t = (unsigned)((sqrtf(8.f * (float)x + 1.f) - 1.f) * 0.5f);
    while (t * (t + 1) / 2 > x) --t;
    while ((t + 1) * (t + 2) / 2 <= x) ++t;
    return t;
}

// A CTA's pieces, one after the other.  head: query head (pass 1) or unit (pass 2); tile: the A tile; the piece is
// steps [i0, i0 + n) of the item; B tile of step i: key tile i (pass 1), query tile tile + i % (T - tile) of query head
// i / (T - tile) of the group (pass 2).  (32-bit arithmetic: a 64-bit division costs every role several hundred clocks
// at every piece.)
template <int PASS>
struct Walk {
    unsigned f, f_end;          // next step and end of the share (split); item number of this CTA (whole)
    int head, tile, i0, n;
    bool ok;
    __device__ __forceinline__ bool split(const Plan& p) const { return PASS == 1 ? p.split_row : p.split_col; }
    __device__ __forceinline__ int len(const Plan& p) const { return PASS == 1 ? tile + 1 : p.G * (p.T - tile); }
    __device__ __forceinline__ void item(const Plan& p) {
        const unsigned P = gridDim.x;
        const unsigned heads = PASS == 1 ? p.NH : p.U, hg = PASS == 1 ? p.hg_row : p.hg_col;
        const unsigned rounds = PASS == 1 ? p.rounds_row : p.rounds_col;
        for (;; ++f) {
            const unsigned g = f / rounds, h0 = g * hg;
            ok = h0 < heads;
            if (!ok) return;
            const unsigned n_h = min(hg, heads - h0), k = (f - g * rounds) * P + ((f & 1) ? P - 1 - blockIdx.x : blockIdx.x);
            if (k >= n_h * (unsigned)p.T) continue;        // (the last round of a group; the next one may have an item)
            const unsigned r = k / n_h;
            head = (int)(h0 + k - r * n_h);
            tile = PASS == 1 ? p.T - 1 - (int)r : (int)r;
            break;
        }
        i0 = 0;
        n = len(p);
    }
    __device__ __forceinline__ void init(const Plan& p) {
        if (!split(p)) { f = 0; item(p); return; }
        f = min(blockIdx.x * p.q, p.steps);
        f_end = min(f + p.q, p.steps);
        ok = f < f_end;
        if (!ok) return;
        if (PASS == 1) {
            head = (int)(f / p.tri());
            const unsigned r = f - (unsigned)head * p.tri();
            tile = (int)tri_root(r);
            i0 = (int)(r - (unsigned)tile * (unsigned)(tile + 1) / 2);
        } else {
            const unsigned gt = (unsigned)p.G * p.tri();
            head = (int)(f / gt);
            const unsigned r = f - (unsigned)head * gt, jr = tri_root(r / (unsigned)p.G);
            tile = p.T - 1 - (int)jr;
            i0 = (int)(r - (unsigned)p.G * (jr * (jr + 1) / 2));
        }
        n = (int)min((unsigned)(len(p) - i0), f_end - f);
    }
    __device__ __forceinline__ bool valid() const { return ok; }
    __device__ __forceinline__ void next(const Plan& p) {
        if (!split(p)) { ++f; item(p); return; }
        f += (unsigned)n;
        ok = f < f_end;
        if (PASS == 1) { if (++tile == p.T) { tile = 0; ++head; } }
        else { if (--tile < 0) { tile = p.T - 1; ++head; } }
        i0 = 0;
        n = (int)min((unsigned)len(p), f_end - f);
    }
    // which of the item's pieces this is (split only)
    __device__ __forceinline__ unsigned piece(const Plan& p) const {
        return blockIdx.x - (PASS == 1 ? p.row_start(head, tile) : p.col_start(head, tile)) / p.q;
    }
};

// Folds a partial (maximum, sum) of a query row into (M, L); log2 units.  (A piece whose wait ran out leaves the state
// (0, NaN), whatever maximum it had by then: with -inf the sum would be passed over here.)
__device__ __forceinline__ void add_state(float& M, float& L, float2 st) {
    const float mn = fmaxf(M, st.x);
    if (mn > -INFINITY) L = L * exp2f(M - mn) + st.y * exp2f(st.x - mn);
    M = mn;
}

// Partial column sums [piece][U, S] -> the score of key j of unit u, in piece order.
__device__ __forceinline__ float column_sum(const float* __restrict__ part, const Plan& p, int S, int u, int j) {
    const size_t keys = (size_t)p.U * S, k = (size_t)u * S + j;
    const int np = p.col_pieces(u, j / TILE);
    float a = 0.f;
    for (int x = 0; x < np; ++x) a += __ldcg(part + (size_t)x * keys + k);
    return a / (float)p.G;
}

}  // namespace plan

// The column pass's partial sums when items were cut and their sum is left to the kernel that reads the scores
// (part = nullptr: the scores are final).
struct ScorePart {
    const float* part = nullptr;
    plan::Plan plan = {};
};

}  // namespace kvm
