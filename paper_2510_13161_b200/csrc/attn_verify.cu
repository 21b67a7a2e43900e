// Branch-tree attention of the verify step: every tree node (kappa x gamma draft tokens + the root)
// attends to the paged KV cache of the verified prefix and to the tree's own K/V under the branch-causal mask (node i
// sees tree token j iff j is i or an ancestor of i), for all layers.
//
// Work decomposition.  The rows that share one head's K/V stream are the G = Hq/Hkv query heads of all n tree nodes;
// they are cut in row tiles of at most 128 (whole nodes).  A CTA works on TWO streams at a time, each (KV head, row
// tile), because one stream alone is a chain (Q K^T -> softmax -> P V) that leaves the tensor cores idle for as long as
// its softmax takes:
//   one row tile per head     both streams are that tile, on alternate KV tiles (merged when the part ends)   "split"
//   an even number            two row tiles of the same head, over the same KV tiles in shared memory         "shared"
//   an odd number             units of two neighbouring heads, which have the same length: pairs of tiles of either
//                             head as above, and one CTA with the two tiles left over, one of each head       "mixed"
// A unit is (layer, request, one or two heads).  Its keys are cut in 16-token slots (one KV page, or 16 tree tokens),
// eight to a 128-token tile.  The tiles of all units form one sequence that is split evenly over groups of CTAs (the
// CTAs of a group walk the same tiles at the same time, so that K/V leave HBM once); a unit that a boundary cuts leaves
// one (max, sum, accumulator) record per side and row tile, and attn_merge_kernel combines them in group order.
//
// Per CTA, 12 warps:
//   warps 0, 3  stage K and V tiles into one ring (32 KB a stage at d = 128): a TMA box per page and per 8 tree tokens,
//               128-byte swizzle (a slot is [token / 8][64-column half][token % 8][128 B]: an evenly strided K-major
//               operand over the whole tile and an MN-major one per slot).  The V warp stages Q too (boxes of whole nodes)
//   warps 1, 2  issue, each for one stream and in turns, P V of one tile and Q K^T of the stream's next tile.  The
//               tcgen05.mma of a thread execute in order, so a Q K^T may overwrite the S / P columns that the P V ahead
//               of it reads without waiting for its completion.  Warp 1 owns TMEM
//   warps 4..7, 8..11  softmax of stream 0 and of stream 1, one thread per row (TMEM lane): P = exp2(s * c - offset)
//               over the first half of S's columns as bf16.  The row's offset is the maximum of the first tile in which
//               it sees anything; it moves only when a half tile's sum of P passes 2^14 (that half is then redone from
//               S, which is still there), and is carried exactly through the sum and the division.
// e4m3 cache (d = 128; F8): Q K^T multiplies codes (kind::f8f6f4, Q divided by its scale and rounded when it is staged), but P V
// does not: four more warps (12..15) widen each V tile to f16, exactly, and P is f16.  In an 8-bit P V, P as e4m3 costs 2.6% of
// the output (root mean square) and its own conversions; the tensor cores have the time, the softmax sets the pace.  K and
// V then have rings of their own, and the widening warps stage the next unit's Q in passing, eight rows per V tile.
// TMEM: S0 | S1 (128 columns each) | O0 | O1 (d columns each) = 512 columns at d = 128.
// Every mbarrier wait is bounded; on expiry the kernel records MIRROR_DEV_TIMEOUT and unwinds.
//
// What bounds it.  Per 256 rows x 128 tokens at d = 128 the tensor cores need 2048 cycles (64 per tcgen05.mma of
// N = 128, measured) and the special-function units 2048 (16 exponentials per cycle and SM; measured 2300 with the loads,
// conversions and stores around them), of ~3700 that such a step takes; under the 1 kW limit the clock falls to ~1.6 GHz.
// (128 rows and 64-token tiles per CTA, alternating two softmax groups, took 4360 cycles for the same work.)  What the
// twelve warps execute per tile has to stay in the SM's instruction cache: loops are kept rolled and rare paths out of
// line on purpose; unrolled, the same step took 4900 cycles, most of them in instruction fetch.  Tried and neutral: a
// third of the exponentials as polynomials on the FMA pipe, and Q K^T by halves of a tile behind the same half's P V (no
// wait for scores, but 96 instead of 64 cycles of tensor core per 128 tokens: the same time at the power limit).
// Measured (bf16, d = 128, tiles of 16-token pages): 80 layers x 16 requests x 520 rows 25.0 -> 20.5 ms at the same
// power; 64 layers x 32768 tokens x 264 rows 4.0 -> 3.4 ms; e4m3 cache, 64 layers x 4 x 4096..16384 tokens x 136 rows (64-token
// tiles with e4m3 P before): 2.25 -> 1.85 ms.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "attn_common.h"

namespace {

using attn::pack_bf16;
using attn::slot_mask;

constexpr int kThreads = 384;
constexpr int kConvWarps = 4;                       // (e4m3 cache) warps 12..15
constexpr int kWideStages = 2;                      // (e4m3 cache) V tiles widened to f16
constexpr int kSlotTok = kAttnSlotTok;
constexpr int kTileSlots = 8;
constexpr int kTileTok = kSlotTok * kTileSlots;     // 128
constexpr int kRows = 128;                          // UMMA M: rows of a stream
constexpr int kMaxStages = 10;
// A half tile whose sum of P stays below this is as it should be: no P of it overflows f16 (e4m3 cache), and sums of P V stay in
// fp32's range for values up to 2^113 (bf16 P would allow more, but values of 1e25 under P of 2^43 already overflow).
constexpr float kSumLimit = 16384.f;
constexpr int kTmemCols = 512;
constexpr int kTmemO = 2 * kTileTok;
constexpr int kCtrlBytes = 528;
constexpr size_t kSmemLimit = 232448;               // 227 KB

enum { kSplit = 0, kPaired = 1 };

struct AttnParams {
    int L, B, n, Hq, Hkv, G;
    int mode;                             // kSplit: one row tile, streams on alternate KV tiles; kPaired: two row tiles
    int heads_per_unit;                   // 1, or 2 when the row tiles of a head are odd in number
    int n_cta;                            // CTAs of a group
    int gs;                               // query heads of a row tile (G, or a share of a large G)
    int node_tiles, nodes_tile;           // row tiles along the nodes and nodes in each
    int n_rt;                             // row tiles of one KV head
    int n_groups;                         // CTA groups (grid = n_groups * n_cta)
    int snap_cap;                         // boundaries move to a unit boundary that is at most this many tiles away
    int units;                            // layers x requests x heads (or pairs of heads)
    int whole_groups;                     // group count that divides the units evenly (attn::whole_unit_groups), 0: none
    int unit_cuts;                        // fewer units than groups: groups per unit, rounded down; 0 otherwise
    int cut_tiles;                        // tiles that a group may take longer for it
    int never_cut;                        // 1: units are so short that they are dealt out whole whatever their lengths
    float lm_ns;                          // > 0: time of the weight stream that is launched behind and runs beside this (see share_choice)
    int deal;                             // 1: where SMs are left to it, whole units are dealt out
    int group_chunk;                      // groups that fill whole TPCs (pairs of SMs)
    int late_merge;                       // 1: the merge runs behind a launch that waited for this one
    int max_pages, num_pages, layer_pages;
    int tree_slots;
    float scale_log2e;
    const int32_t* page_table;
    const int32_t* prefix_len;
    const __nv_bfloat16* v_pool;
    // e4m3 cache: pools, k_new and v_new hold e4m3 codes; a code times its (layer, KV head) scale is the value.  Q stays bf16
    // in memory; its operand is e4m3(q / q_scale), rounded when it is staged.
    const __nv_bfloat16* q;
    const float* k_scale;                 // [L, Hkv]
    const float* v_scale;                 // [L, Hkv]
    float q_scale;
    __nv_bfloat16* out;
    float* lse_out;
    float* partial;                       // [grid][2 slots][2 streams][D + 4][128]
    attn::GroupBegin* begins;             // [n_groups]
    int* status;
    long long wait_limit;                 // SM cycles after which a wait gives up
    int stall_after;                      // test aid: the K producer stops after this many stages (-1: never)
    int stall_merge;                      // test aid: 1: the merge's first wait runs out
};

struct Maps {
    CUtensorMap k, v, kn, vn, q;
};

__device__ __forceinline__ void dev_check(const AttnParams& p, int detail) {
    if (atomicCAS(p.status, 0, MIRROR_DEV_CHECK) == 0) atomicExch(p.status + 1, detail);
}

// ---- the tile sequence ---------------------------------------------------------------------------------------
// Units in the order (layer, request, head or pair of heads); cumT[b] = KV tiles of one unit of the requests before b.
__device__ __forceinline__ int tiles_of(int len, int tree_slots) {
    return ((len + kSlotTok - 1) / kSlotTok + tree_slots + kTileSlots - 1) / kTileSlots;
}

// The tiles of one unit that this CTA works on.
struct Segment {
    int layer, b, g;
    int t_first, t_last, tiles;           // tiles [t_first, t_last) of the unit's `tiles`
    int len, pages_full, pages_all, slots_all;
};
__device__ __forceinline__ void fill_segment(Segment& s, int left, const AttnParams& p, const int* s_len) {
    s.len = s_len[s.b];
    s.pages_full = s.len / kSlotTok;
    s.pages_all = (s.len + kSlotTok - 1) / kSlotTok;
    s.slots_all = s.pages_all + p.tree_slots;
    s.tiles = tiles_of(s.len, p.tree_slots);
    s.t_last = min(s.tiles, s.t_first + left);
}
// (out of line: code that runs once)
__device__ __noinline__ void first_segment(Segment& s, int left, const AttnParams& p, const int* s_len) { fill_segment(s, left, p, s_len); }
// the unit behind s (a segment that is followed by another one ends with its unit)
__device__ __noinline__ Segment next_segment(const Segment& s, int left, const AttnParams& p, const int* s_len) {
    Segment t;
    t.layer = s.layer; t.b = s.b; t.g = s.g + 1; t.t_first = 0;
    if (t.g == p.Hkv / p.heads_per_unit) {
        t.g = 0;
        if (++t.b == p.B) { t.b = 0; ++t.layer; }
    }
    fill_segment(t, left, p, s_len);
    return t;
}

// ---- barriers ------------------------------------------------------------------------------------------------
struct Ctrl {
    uint64_t full[kMaxStages], empty[kMaxStages];       // K/V ring (e4m3: the first half K, the second V, rings of their own)
    uint64_t wide_full[kWideStages], wide_empty[kWideStages];       // e4m3: V tiles widened to f16
    uint64_t q_full[4], q_empty[4];                     // (as many as Q buffers)
    uint64_t s_full[2], p_full[2][2], o_full[2];        // per stream (P: per half of the tile)
    uint64_t pv_half[2];                                // P V of a tile's first half is through
    uint64_t turn[2];                                   // the issuing warps take turns
    uint64_t exp_turn[2][4];                            // the two softmax warps of a scheduler take turns
    uint64_t pair[4];                                   // split: the two softmax warps of a TMEM quarter meet
    Segment first;                                      // where this CTA's range begins
    int n_tiles;
    int place;                                          // this CTA's among the records: by its group, not by its block
    int* status;
    long long wait_limit;
    uint32_t tmem_base;
    volatile int abort;
};
static_assert(sizeof(Ctrl) <= kCtrlBytes, "control block");

// How the tile sequence is cut into one range per CTA group.  (This runs in front of every launch's first copy, by one
// warp and from a cold instruction cache: few divisions, and those of 32 bits.)
struct Partition {
    int tiles_per_layer, total_tiles;     // (total_tiles -1: the sequence does not fit 31 bits)
    bool whole;                           // units are dealt out whole, by number
    int n_groups, snap_tol;
    int share, rest;                      // total_tiles = n_groups * share + rest
};
// Does a group take at most `more` tiles longer when each unit of `tiles` has `cuts` groups to itself than in an even split over
// `groups`?
__host__ __device__ inline bool cuts_pay(int tiles, int units, int groups, int cuts, int more) {
    return (long long)tiles * groups - (long long)tiles * units * cuts <= (long long)more * cuts * groups;
}
// How many groups to use when a weight stream that does not depend on this launch follows it (lmhead_pair_free_kernel): it takes
// whatever SMs are left.  Attention is bound by its exponentials and uses a quarter to two thirds of HBM, the stream uses nothing
// else, so side by side they take less than one after the other.  A choice (0: all groups, up to 31) is weighed by the time at
// which both are through: attention at kStepNs per step and kUnitSteps more per unit, the stream at the rate of the SMs that it has
// meanwhile (kFullSms keep HBM busy) and of the bandwidth that is left to it, then alone; it has to gain 3%.  (48 layers x 2048
// tokens x 285 rows before 1.56 GB of weights: 28 of 49 groups, 469 -> 433 us; unshared 447.)
constexpr float kStepNs = 2100.f, kUnitSteps = 4.5f, kFullSms = 85.f, kHbmBytesNs = 6500.f, kShareGain = 0.97f;
struct Share {
    int g;
    float total;                          // ns
};
__host__ __device__ inline float quick_quotient(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fdividef(a, b);
#else
    return a / b;
#endif
}
__host__ __device__ inline Share share_choice(const AttnParams& p, float total_tiles, int most, int sms, float step_bytes, int choice) {
    const float units = (float)p.units, steps = p.mode == kSplit ? 0.5f * (total_tiles + units) : total_tiles;
    const float work = steps + kUnitSteps * units;
    float g = fmaxf((float)(most - ((most * choice * 1639) >> 16)), 1.f), t;         // (a fortieth of the groups less from choice to choice)
    if (p.deal) {                                                     // (whole units; a quotient's last bit does not matter)
        const float k = ceilf(quick_quotient(units, g) - 1e-3f);
        g = ceilf(quick_quotient(units, k) - 1e-3f);
        t = k * quick_quotient(work, units);
    } else {
        t = quick_quotient(work, g) + kUnitSteps;
    }
    t *= kStepNs;
    const float hbm = 1.f - quick_quotient(g * step_bytes * steps, work * (kStepNs * kHbmBytesNs));
    const float rate = fminf(((float)sms - g * (float)p.n_cta) * (1.f / kFullSms), fmaxf(hbm, 0.1f));
    return {(int)g, t + fmaxf(0.f, p.lm_ns - t * rate)};
}
__device__ __noinline__ int share_groups(const AttnParams& p, int total_tiles, int most, int sms, float step_bytes) {
    const int lane = threadIdx.x & 31;
    const Share s = share_choice(p, (float)total_tiles, most, sms, step_bytes, lane);
    // the least total time, and of equals the most groups
    const uint32_t key = (__float_as_uint(s.total) & ~31u) | (uint32_t)lane;
    const uint32_t best = __reduce_min_sync(0xffffffffu, key);
    const bool gains = __uint_as_float(best) < kShareGain * __shfl_sync(0xffffffffu, s.total, 0);
    const int g = __shfl_sync(0xffffffffu, s.g, best & 31u);
    return gains ? g : most;
}
__device__ __forceinline__ Partition make_partition(const AttnParams& p, const int* cumT, float step_bytes) {
    Partition q;
    const long long per = (long long)(p.Hkv / p.heads_per_unit) * cumT[p.B], total = per * p.L;
    q.tiles_per_layer = (int)per;
    q.total_tiles = total < (1ll << 31) ? (int)total : -1;
    q.n_groups = min(p.n_groups, p.units);
    q.snap_tol = q.share = q.rest = 0;
    q.whole = p.never_cut != 0;
    if (p.lm_ns > 0.f && q.total_tiles > 0 && q.n_groups > 1) {
        const int most = min(p.n_groups, p.never_cut ? p.units : q.total_tiles), g = share_groups(p, q.total_tiles, most, gridDim.x, step_bytes);
        if (g < most) {
            q.n_groups = g;
            q.whole |= p.deal != 0;
            q.share = (int)((uint32_t)q.total_tiles / (uint32_t)g);
            q.rest = q.total_tiles - q.share * g;
            q.snap_tol = min(p.snap_cap, q.share >> 2);
            return q;
        }
    }
    if (p.never_cut) return q;                                        // (group_begin counts units; short launches fetch no more code)
    // Units of equal length (every request has the same number of tiles): a group count that divides the units, if one
    // exists within 15% of the CTA groups there are, gives every group the same number of WHOLE units: no unit is cut,
    // nothing is left to merge and all groups end together, which is worth more than the few SMs left idle.
    bool equal_units = true;
    for (int b = 1; b < p.B; ++b) equal_units &= (cumT[b + 1] - cumT[b]) == cumT[1];
    // Else every group gets at least one tile, or two where its streams take alternate tiles (one alone would leave a stream
    // without work and the merge with twice the records).
    const int split = p.mode == kSplit ? 1 : 0, most = min(p.n_groups, max(1, q.total_tiles >> split));
    q.n_groups = p.whole_groups > 0 && equal_units ? p.whole_groups : most;
    // Fewer units than groups, all of one length: the same number of groups for every unit, where that costs a group few tiles.
    // (An even split over all groups makes most of them work on two units: a second Q, which an e4m3 cache converts, a second
    // epilogue and record; whole units also need no merge.  64 units of 9 tiles over 74 groups, bf16 / e4m3: 53 -> 30 / 68 -> 36 us;
    // 16 units over 37 groups, two each: 39 -> 33 / 54 -> 40.  But 16 units of 157 tiles over 74 groups, four each, bf16, which is
    // 5 tiles longer: 95 -> 104.)
    if (p.unit_cuts > 0 && equal_units) {
        const int cuts = min(p.unit_cuts, max(1, cumT[1] >> split));
        if (cuts_pay(cumT[1], p.units, most, cuts, p.cut_tiles)) q.n_groups = p.units * cuts;
    }
    q.share = (int)((uint32_t)q.total_tiles / (uint32_t)q.n_groups);
    q.rest = q.total_tiles - q.share * q.n_groups;
    // A boundary that falls within snap_tol tiles of a unit boundary moves there (a cut costs about as much as a tile).
    // snap_tol is at most a quarter of the smallest even share, so boundaries stay strictly increasing.
    q.snap_tol = min(p.snap_cap, q.share >> 2);
    return q;
}
// Where group g's range begins: tile x of the sequence, tile t of unit (layer, b, g).  (Position and unit in one go: found again
// from the position, and with the divisions of a fully rounded quotient in share_choice, this took 3500 to 8500 cycles of a launch.)
struct Begin {
    int x, layer, b, g, t;
};
__device__ __noinline__ Begin group_begin(const Partition& q, int g, const AttnParams& p, const int* cumT) {
    Begin u = {g <= 0 ? 0 : q.total_tiles, 0, 0, 0, 0};
    if (g <= 0 || g >= q.n_groups) return u;
    const int hu = p.Hkv / p.heads_per_unit;
    if (q.whole) {                                                    // first tile of unit number units * g / n_groups
        const uint32_t n = (uint32_t)q.n_groups, us = (uint32_t)p.units / n, rest = (uint32_t)p.units - us * n;
        const uint32_t unit = us * g + (rest ? rest * g / n : 0), per = (uint32_t)(p.B * hu);
        u.layer = (int)(unit / per);
        u.g = (int)(unit - u.layer * per);
        if (p.B > 1) {
            u.b = (int)((uint32_t)u.g / (uint32_t)hu);
            u.g -= u.b * hu;
        }
        u.x = u.layer * q.tiles_per_layer + hu * cumT[u.b] + u.g * (cumT[u.b + 1] - cumT[u.b]);
        return u;
    }
    u.x = q.share * g + (q.rest ? (int)((uint32_t)(q.rest * g) / (uint32_t)q.n_groups) : 0);       // total_tiles * g / n_groups
    u.layer = (int)((uint32_t)u.x / (uint32_t)q.tiles_per_layer);     // (the tile count fits 31 bits: checked in the prologue)
    int rem = u.x - u.layer * q.tiles_per_layer;
    while (u.b + 1 < p.B && hu * cumT[u.b + 1] <= rem) ++u.b;
    rem -= hu * cumT[u.b];
    const int Tb = cumT[u.b + 1] - cumT[u.b];
    u.g = (int)((uint32_t)rem / (uint32_t)Tb);
    u.t = rem - u.g * Tb;
    if (u.t <= Tb - u.t) {                                            // to the unit boundary close by
        if (u.t <= q.snap_tol) { u.x -= u.t; u.t = 0; }
    } else if (Tb - u.t <= q.snap_tol) {
        u.x += Tb - u.t;
        u.t = 0;
        if (++u.g == hu) {
            u.g = 0;
            if (++u.b == p.B) { u.b = 0; ++u.layer; }
        }
    }
    return u;
}

// A launch that leaves SMs to another one leaves whole TPCs (the other's CTAs come in pairs), spread over the chip as blocks are
// over its GPCs: of every `chunk` groups all work or none.  Which one group number `g` stands for, of `most`, `used` of them at work.
__host__ __device__ inline int spread_group(int g, int most, int used, int chunk) {
    const int chunks = most / chunk, n = (used + chunk - 1) / chunk, c = g / chunk;
    if (used >= most || n >= chunks || c >= chunks) return g;
    const int r0 = c * n / chunks, r1 = (c + 1) * n / chunks;
    return (r1 > r0 ? r0 : n + c - r0) * chunk + (g - c * chunk);
}

// Prefix lengths (clamped to the page table) and the tile counts they give, by one warp.
__device__ __forceinline__ void load_lengths(const AttnParams& p, int* cumT, int* s_len, bool report) {
    const int lane = threadIdx.x & 31;
    int acc = 0;
    if (lane == 0) cumT[0] = 0;
#pragma unroll 1
    for (int b0 = 0; b0 < p.B; b0 += 32) {
        const int b = b0 + lane;
        int len = b < p.B ? p.prefix_len[b] : 0;
        if (len < 0 || len > p.max_pages * kSlotTok) {
            if (report) dev_check(p, 300 + b);
            len = len < 0 ? 0 : p.max_pages * kSlotTok;
        }
        int sum = b < p.B ? tiles_of(len, p.tree_slots) : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += v;
        }
        if (b < p.B) { s_len[b] = len; cumT[b + 1] = acc + sum; }
        acc += __shfl_sync(0xffffffffu, sum, 31);
    }
    __syncwarp();
}

// Which (head of the unit, row tile) stream `grp` of CTA `rb` of a group is, and whether both streams share K/V tiles.
struct StreamId {
    int head_off, rt;
    bool exists, shared_kv;
};
__device__ __forceinline__ StreamId stream_of(const AttnParams& p, int rb, int grp) {
    StreamId s;
    s.head_off = 0; s.rt = 0; s.exists = true; s.shared_kv = false;
    if (p.mode == kSplit) return s;
    s.shared_kv = true;
    if (p.heads_per_unit == 1) {
        s.rt = 2 * rb + grp;
        if (s.rt >= p.n_rt) { s.rt = p.n_rt - 1; s.exists = false; }      // (an odd tile count and an odd head count)
        return s;
    }
    const int h2 = (p.n_rt - 1) / 2;
    if (rb == p.n_cta - 1) { s.head_off = grp; s.rt = p.n_rt - 1; s.shared_kv = false; return s; }
    s.head_off = rb / h2;
    s.rt = 2 * (rb % h2) + grp;
    return s;
}

// ---- packed fp32 pairs, tensor memory ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ void tmem_st_32x32b_x32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
          "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
          "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st_32x32b_x16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Wait for this thread's tcgen05.ld, naming the registers it filled: without the dependence the compiler may move
// arithmetic on them ahead of the wait.
__device__ __forceinline__ void tmem_ld_wait32(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]),
                   "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]),
                   "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]),
                   "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :: "memory");
}
__device__ __forceinline__ void tmem_ld_wait16(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]),
                   "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :: "memory");
}

// 32 scores of a row -> 16 words of bf16 (F8: f16) P = exp2(s * c - offset); the fp32 values are added to four running sums
// (two packed pairs).
template <bool F8>
__device__ __forceinline__ void exp_chunk(const uint32_t (&r)[32], uint64_t sc2, uint64_t neg_off2, uint32_t* pk, uint64_t& s0, uint64_t& s1) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        float a, b;
        unpack2(fma2(pack2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1])), sc2, neg_off2), a, b);
        a = ptx::ex2_approx(a);
        b = ptx::ex2_approx(b);
        if (j & 1) s1 = add2(s1, pack2(a, b));
        else s0 = add2(s0, pack2(a, b));
        if (F8) asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(pk[j]) : "f"(b), "f"(a));
        else asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[j]) : "f"(b), "f"(a));
    }
}

template <int D, bool F8>
struct Cfg {
    static_assert(!F8 || D == 128, "an e4m3 row must fill a 128-byte swizzle row");
    static constexpr int kThreads = ::kThreads + (F8 ? 32 * kConvWarps : 0);
    static constexpr int kRowBytes = D * (F8 ? 1 : 2);             // one token's K (or V) row of one head
    static constexpr int kHalves = kRowBytes / 128;
    static constexpr int kSlotBytes = kHalves * kSlotTok * 128;    // one slot of K or V = one TMA box
    static constexpr int kGroupStride = kHalves * 1024;            // between the 8-token groups of one half
    static constexpr int kStageBytes = kTileSlots * kSlotBytes;    // one K or V tile
    static constexpr int kQHalfBytes = kRows * 128;                // one 64-column half of a Q buffer
    static constexpr int kQBytes = kHalves * kQHalfBytes;
    static constexpr int kVHalves = D * 2 / 128;                   // V as P V reads it: 16 bits per element
    static constexpr int kVSlotBytes = kVHalves * kSlotTok * 128;
    static constexpr int kWideBytes = F8 ? kTileSlots * kVSlotBytes : 0;        // one V tile widened to f16
    static constexpr size_t kFixedBytes = kWideStages * kWideBytes + kCtrlBytes;           // of shared memory, beside Q buffers and ring
};

// Scores of tokens that the row does not see become -inf, in TMEM: a pass of its own over a unit's last tiles, so that the
// loop over all the others carries no mask code.
__device__ __noinline__ void mask_tile(uint32_t s_addr, int slot0, const Segment& sg, unsigned long long anc0, unsigned long long anc1) {
#pragma unroll 1
    for (int c = 0; c < kTileSlots; ++c) {
        const uint32_t cm = slot_mask(slot0 + c, sg.pages_full, sg.pages_all, sg.slots_all, sg.len, anc0, anc1);
        if (__all_sync(0xffffffffu, cm == 0xffffu)) continue;
        uint32_t r[16];
        ptx::tmem_ld_32x32b_x16(s_addr + (uint32_t)(c * 16), r);
        tmem_ld_wait16(r);
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (!((cm >> j) & 1u)) r[j] = 0xff800000u;
        tmem_st_32x32b_x16(s_addr + (uint32_t)(c * 16), r);
    }
    tmem_st_wait();
}
// Row maximum over chunks of 32 scores (a unit's first tile, and what is redone).
__device__ __noinline__ float tile_max(uint32_t s_addr, int chunks) {
    float m = -INFINITY;
#pragma unroll 1
    for (int c = 0; c < chunks; ++c) {
        uint32_t r[32];
        ptx::tmem_ld_32x32b_x32(s_addr + (uint32_t)(c * 32), r);
        tmem_ld_wait32(r);
#pragma unroll
        for (int j = 0; j < 32; j += 2)          // (three operands: one instruction for two scores)
            asm("max.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(__uint_as_float(r[j])), "f"(__uint_as_float(r[j + 1])));
    }
    return m;
}
// A new offset for the rows whose sum over the 64 scores at s_addr outgrew the limit (`grow`): the maximum of those scores.
// The row's accumulator (o_cols columns, 0: none yet) is rescaled to it.  Returns (offset, factor).
__device__ __noinline__ float2 move_offset(uint32_t s_addr, uint32_t o_addr, int o_cols, bool grow, float off, float sc) {
    const float mx = tile_max(s_addr, 2);
    const float next = grow ? mx * sc : off, alpha = grow ? exp2f(off - next) : 1.f;
#pragma unroll 1
    for (int c = 0; c < o_cols; c += 16) {
        uint32_t r[16];
        ptx::tmem_ld_32x32b_x16(o_addr + (uint32_t)c, r);
        tmem_ld_wait16(r);
#pragma unroll
        for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) * alpha);
        tmem_st_32x32b_x16(o_addr + (uint32_t)c, r);
    }
    tmem_st_wait();
    return make_float2(next, alpha);
}

// Q as e4m3 codes: those of the correctly rounded quotients x / q_scale.
__device__ __noinline__ uint32_t unusual_codes(uint2 v, float s) {
    return pack_e4m3x4(__fdiv_rn(__uint_as_float(v.x << 16), s), __fdiv_rn(__uint_as_float(v.x & 0xffff0000u), s),
                             __fdiv_rn(__uint_as_float(v.y << 16), s), __fdiv_rn(__uint_as_float(v.y & 0xffff0000u), s));
}
// One row, four elements per lane, into the K-major operand tile `q` ([row][128 B], 128-byte swizzle).
__device__ __forceinline__ void store_q_row(uint8_t* q, int row, uint2 v, const E4m3Scale& qs) {
    const int lane = threadIdx.x & 31;
    uint32_t code;
    if (qs.usual)
        code = pack_e4m3x4(qs.quotient(__uint_as_float(v.x << 16)), qs.quotient(__uint_as_float(v.x & 0xffff0000u)),
                                 qs.quotient(__uint_as_float(v.y << 16)), qs.quotient(__uint_as_float(v.y & 0xffff0000u)));
    else
        code = unusual_codes(v, qs.s);
    *reinterpret_cast<uint32_t*>(q + row * 128 + (((lane >> 2) ^ (row & 7)) << 4) + (lane & 3) * 4) = code;
}
__device__ __forceinline__ const __nv_bfloat16* row_of_lane(const __nv_bfloat16* qrow, int r) {
    return (const __nv_bfloat16*)__shfl_sync(0xffffffffu, (unsigned long long)qrow, r);
}
// Four e4m3 codes as four f16 (exact).
__device__ __forceinline__ uint2 widen4(uint32_t w) {
    uint2 r;
    asm("{\n\t.reg .b16 lo, hi;\n\t"
        "mov.b32 {lo, hi}, %2;\n\t"
        "cvt.rn.f16x2.e4m3x2 %0, lo;\n\t"
        "cvt.rn.f16x2.e4m3x2 %1, hi;\n\t}"
        : "=r"(r.x), "=r"(r.y) : "r"(w));
    return r;
}

// kEarly: only q and the tree's K/V come from the kernel ahead (see mirror_attn_launch).  An instance of its own: long calls never
// take these branches.
template <int D, bool F8, bool kEarly>
__global__ void __launch_bounds__(Cfg<D, F8>::kThreads, 1)
attn_verify_kernel(const __grid_constant__ Maps tm, const __grid_constant__ AttnTree tree, const __grid_constant__ AttnParams p,
                   const int n_stages) {
    using C = Cfg<D, F8>;
    extern __shared__ __align__(1024) uint8_t smem[];
    // Q buffers: per stream, or (split) of alternating units; e4m3: two per stream, or (split) two
    uint8_t* sQ = smem;
    const int q_bufs = F8 && p.mode != kSplit ? 4 : 2;
    uint8_t* wide = sQ + q_bufs * C::kQBytes;                            // [2] V tiles widened to f16 (e4m3 cache)
    uint8_t* ring = wide + kWideStages * C::kWideBytes;             // [n_stages] K or V tiles
    // stages of a ring: one that K and V share, or (e4m3) two of half the stages
    const int ring_n = F8 ? n_stages >> 1 : n_stages;
    Ctrl* ctrl = (Ctrl*)(ring + (size_t)n_stages * C::kStageBytes);
    float* xch = (float*)((uint8_t*)ctrl + kCtrlBytes);             // split: [128 rows][2 streams][offset, sum]
    int* cumT = (int*)(xch + (p.mode == kSplit ? kRows * 4 : 0));   // [B+1] tiles per unit, prefix-summed over the requests
    int* s_len = cumT + (p.B + 1);                                  // [B] clamped prefix lengths

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rb = blockIdx.x % p.n_cta;
    const bool split = p.mode == kSplit;
    const bool shared_kv = stream_of(p, rb, 0).shared_kv;

    // ---- prologue (programmatic dependent launch: barriers and tensor memory are set up while the kernel ahead in the
    // stream is still running; nothing of global memory is touched before it has completed)
    if (tid == 0) {
        const uint32_t readers = shared_kv ? 2 : 1;                 // issuing warps that read a K/V stage
        for (int s = 0; s < n_stages; ++s) { ptx::mbar_init(&ctrl->full[s], 1); ptx::mbar_init(&ctrl->empty[s], F8 && s >= ring_n ? kConvWarps : readers); }
        if (F8)
            for (int s = 0; s < kWideStages; ++s) { ptx::mbar_init(&ctrl->wide_full[s], kConvWarps); ptx::mbar_init(&ctrl->wide_empty[s], readers); }
        for (int g = 0; g < 2; ++g) {
            ptx::mbar_init(&ctrl->s_full[g], 1); ptx::mbar_init(&ctrl->p_full[g][0], 4); ptx::mbar_init(&ctrl->p_full[g][1], 4);
            ptx::mbar_init(&ctrl->o_full[g], 1); ptx::mbar_init(&ctrl->turn[g], 1); ptx::mbar_init(&ctrl->pv_half[g], 1);
        }
        for (int s = 0; s < q_bufs; ++s) { ptx::mbar_init(&ctrl->q_full[s], !F8 ? 1 : split ? 8 : 4); ptx::mbar_init(&ctrl->q_empty[s], split ? 2 : 1); }
        for (int s = 0; s < 4; ++s) {
            ptx::mbar_init(&ctrl->pair[s], 2);
            ptx::mbar_init(&ctrl->exp_turn[0][s], 1); ptx::mbar_init(&ctrl->exp_turn[1][s], 1);
        }
        ctrl->abort = 0;
        ctrl->status = p.status;
        ctrl->wait_limit = p.wait_limit;
        ptx::fence_mbar_init();
        ptx::prefetch_tmap(&tm.k); ptx::prefetch_tmap(&tm.v); ptx::prefetch_tmap(&tm.kn); ptx::prefetch_tmap(&tm.vn);
        if (!F8) ptx::prefetch_tmap(&tm.q);
    }
    // Rows that the Q copies do not fill are zeros: the tensor cores multiply 128 rows whatever the tile holds, and under the
    // power limit zeros are cheaper than whatever lies there.
    const int pad = kRows - p.gs * p.nodes_tile;
    for (int i = tid; i < q_bufs * C::kHalves * pad * 8; i += C::kThreads) {
        const int half = i / (pad * 8), c = i - half * pad * 8;
        *reinterpret_cast<uint4*>(sQ + half * C::kQHalfBytes + p.gs * p.nodes_tile * 128 + c * 16) = make_uint4(0, 0, 0, 0);
    }
    ptx::fence_proxy_async();
    if (warp == 1) {
        ptx::tmem_alloc(&ctrl->tmem_base, kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    // (kEarly: the K producer waits in front of the tree's rows, the V producer in front of Q)
    if (!kEarly) {
        ptx::grid_dep_wait();
        ptx::grid_dep_launch();             // the kernel behind may be scheduled as soon as SMs free up
    }
    if (warp == 0) {
        load_lengths(p, cumT, s_len, true);
        const Partition part = make_partition(p, cumT, (float)(C::kStageBytes * (split ? 4 : 2)));
        const int block_group = blockIdx.x / p.n_cta, group = p.lm_ns > 0.f ? spread_group(block_group, p.n_groups, part.n_groups, p.group_chunk) : block_group;
        const bool fits = part.total_tiles >= 0 && (ptx::smem_u32(smem) & 1023) == 0;
        if (!fits && lane == 0) dev_check(p, 600);
        Begin u = {};
        if (fits && group < part.n_groups && lane < 2) u = group_begin(part, group + lane, p, cumT);
        const int x1 = __shfl_sync(0xffffffffu, u.x, 1);
        if (lane == 0) {
            ctrl->n_tiles = x1 - u.x;
            ctrl->place = group * p.n_cta + rb;
            Segment& s = ctrl->first;
            s.layer = u.layer; s.b = u.b; s.g = u.g; s.t_first = u.t;
            if (u.x < x1) first_segment(s, x1 - u.x, p, s_len);
            if (rb == 0 && group < p.n_groups) p.begins[group] = {u.x < x1 && u.t > 0 ? 1 : 0, u.layer, u.b, u.g};
        }
    }
    __syncthreads();
    const uint32_t tmem_base = ctrl->tmem_base;
    const int n_tiles = ctrl->n_tiles;               // tiles of this CTA's range

    if (warp < 4) {
        if (n_tiles > 0 && (warp == 0 || warp == 3)) {
            // ======================================================================= K and V producers
            // Ring order (first use by the issuing warps): K of step 0, then per step V, next K -- of stream 0 and, when the
            // streams have K/V tiles of their own, of stream 1.  Both warps walk that order; each fills its own stages.
            // (one copy of the code for both.  e4m3: V has a ring of its own, in front of the warps that widen it.)
            {
                const bool V = warp == 3;
                const CUtensorMap* const map = V ? &tm.v : &tm.k;
                Segment sg = ctrl->first;                          // of the step that is filled next
                int t = sg.t_first, left = n_tiles;                // its tile; tiles from it to the end of the range
                uint32_t st = 0, ph = 1;
                int filled = 0;
                bool ok = true, stop = false;
                auto skip = [&](int n) {
                    st += (uint32_t)n;
                    if (st >= (uint32_t)ring_n) { st -= (uint32_t)ring_n; ph ^= 1; }
                };
                auto pass = [&](int n) {                           // stages that the other producer fills
                    if (!F8) skip(n);
                };
                const int st0 = F8 && V ? ring_n : 0;              // the ring's first stage
                // page ids of a tile, one per lane (0..7), fetched a tile ahead
                int pg = 0, pg_t = -1, pg_next = 0;
                auto fetch = [&](int tt) -> int {
                    const int sl = tt * kTileSlots + lane;
                    return (lane < kTileSlots && sl < sg.pages_all) ? p.page_table[(size_t)sg.b * p.max_pages + sl] : 0;
                };
                auto emit = [&](int tt, int g) {
                    if (p.stall_after >= 0 && !V && filled >= p.stall_after) { ok = false; stop = true; return; }     // (test aid: see AttnParams)
                    if (tt != pg_t) {
                        pg = (pg_t >= 0 && tt == pg_t + 1) ? pg_next : fetch(tt);
                        pg_next = fetch(tt + 1);
                        pg_t = tt;
                    }
                    if (!ptx::warp_wait(ctrl, &ctrl->empty[st0 + st], ph, 10)) { ok = false; return; }
                    uint8_t* const dst = ring + (size_t)(st0 + st) * C::kStageBytes;
                    uint64_t* const bar = &ctrl->full[st0 + st];
                    const int head = sg.g * p.heads_per_unit + stream_of(p, rb, g).head_off;
                    const int sl0 = tt * kTileSlots, n_sl = min(kTileSlots, sg.slots_all - sl0);
                    if (pg < 0 || pg >= p.num_pages) { dev_check(p, 400); pg = 0; }
                    const int row0 = sg.layer * p.layer_pages;
                    int ragged = -1;                               // V: slot of a partial page in this tile
                    if (V && sg.pages_all > sg.pages_full && sg.pages_full >= sl0 && sg.pages_full < sl0 + kTileSlots) {
                        // V rows beyond the prefix must be zeros (P is 0 there, but 0 x NaN is not): 16-byte copies with zero fill
                        ragged = sg.pages_full - sl0;
                        const int rp = __shfl_sync(0xffffffffu, pg, ragged), valid = sg.len - sg.pages_full * kSlotTok;
                        const uint8_t* src = (const uint8_t*)p.v_pool + ((size_t)(row0 + rp) * p.Hkv + head) * (size_t)(kSlotTok * C::kRowBytes);
                        constexpr int kRowChunks = C::kRowBytes / 16;
#pragma unroll 1
                        for (int c = lane; c < kSlotTok * kRowChunks; c += 32) {
                            const int tr = c / kRowChunks, cc = c % kRowChunks;
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                                         ::"r"(ptx::smem_u32(dst + ragged * C::kSlotBytes + attn::kv_slot_off<C::kHalves>(tr, cc))),
                                           "l"(src + c * 16), "r"(tr < valid ? 16u : 0u) : "memory");
                        }
                        asm volatile("cp.async.wait_all;" ::: "memory");
                        ptx::fence_proxy_async();
                        __syncwarp();
                    }
                    // One elected lane issues all boxes from uniform registers, without a loop: 8 boxes take ~300 cycles; a lane per
                    // box, or a loop, 700.
                    // (the barrier's one arrival is its arming, so copies that land before it cannot complete the phase)
                    if (sl0 + kTileSlots <= sg.pages_full) {
                        int row[kTileSlots];
#pragma unroll
                        for (int k = 0; k < kTileSlots; ++k) row[k] = (row0 + __shfl_sync(0xffffffffu, pg, k)) * p.Hkv + head;
                        if (ptx::elect_one()) {
                            ptx::mbar_arrive_expect_tx(bar, (uint32_t)C::kStageBytes);
#pragma unroll
                            for (int k = 0; k < kTileSlots; ++k) ptx::tma_load_5d(dst + k * C::kSlotBytes, map, bar, 0, 0, 0, 0, row[k]);
                        }
                    } else {
                        if (kEarly && sl0 + n_sl > sg.pages_all) ptx::grid_dep_wait();
                        const bool leader = ptx::elect_one();
                        if (leader) ptx::mbar_arrive_expect_tx(bar, (uint32_t)((n_sl - (ragged >= 0)) * C::kSlotBytes));
#pragma unroll 1
                        for (int k = 0; k < n_sl; ++k) {
                            const int page = __shfl_sync(0xffffffffu, pg, k), sl = sl0 + k;
                            uint8_t* const d = dst + k * C::kSlotBytes;
                            if (sl < sg.pages_all) {
                                if (leader && k != ragged) ptx::tma_load_5d(d, map, bar, 0, 0, 0, 0, (row0 + page) * p.Hkv + head);
                            } else if (leader) {                   // tree tokens, eight to a box (tokens that do not exist arrive as zeros)
#pragma unroll 1
                                for (int sub = 0; sub < 2; ++sub)
                                    ptx::tma_load_5d(d + sub * C::kGroupStride, V ? &tm.vn : &tm.kn, bar, 0, (sl - sg.pages_all) * kSlotTok + sub * 8, 0,
                                                     head, sg.layer * p.B + sg.b);
                            }
                        }
                    }
                    __syncwarp();
                    ++filled;
                    skip(1);
                };
                // Q of a segment, once the buffers' last Q K^T is through.  (The V warp is ahead of the issuing warps; waiting here,
                // behind V of the segment before, holds nothing up that is needed soon.)
                auto load_q = [&](const Segment& s, uint32_t n_seg) {
                    for (int k = 0; k < (split ? 1 : 2); ++k) {
                        const int buf = split ? (int)(n_seg & 1) : k;
                        const uint32_t use = split ? n_seg >> 1 : n_seg;          // how often this buffer has been filled
                        if (!ptx::warp_wait(ctrl, &ctrl->q_empty[buf], (use & 1) ^ 1, 11)) { ok = false; break; }
                        if (lane == 0) {
                            const StreamId id = stream_of(p, rb, k);
                            const int head = (s.g * p.heads_per_unit + id.head_off) * p.G + (id.rt / p.node_tiles) * p.gs;
                            ptx::mbar_arrive_expect_tx(&ctrl->q_full[buf], (uint32_t)(p.gs * p.nodes_tile * 128 * C::kHalves));
                            for (int h = 0; h < C::kHalves; ++h)
                                ptx::tma_load_5d(sQ + buf * C::kQBytes + h * C::kQHalfBytes, &tm.q, &ctrl->q_full[buf], 0, head,
                                                 (id.rt % p.node_tiles) * p.nodes_tile, h, s.layer * p.B + s.b);
                        }
                        __syncwarp();
                    }
                };
                auto prefetch_ragged = [&](const Segment& s) {     // (that page is copied by this warp itself: let it not wait for HBM)
                    if (s.pages_all == s.pages_full || s.t_last < s.tiles) return;
                    const int page = p.page_table[(size_t)s.b * p.max_pages + s.pages_full];
                    if (page < 0 || page >= p.num_pages) return;
                    const uint8_t* src = (const uint8_t*)p.v_pool + ((size_t)(s.layer * p.layer_pages + page) * p.Hkv + s.g * p.heads_per_unit) * (size_t)(kSlotTok * C::kRowBytes);
                    for (int c = lane; c < p.heads_per_unit * kSlotTok * C::kRowBytes / 128; c += 32) ptx::prefetch_l2(src + c * 128);
                };
                if (V) {
                    if (kEarly) {
                        ptx::grid_dep_wait();
                        ptx::grid_dep_launch();
                    }
                    if (!F8) load_q(sg, 0);
                    prefetch_ragged(sg);
                }
                uint32_t n_seg = 0;
                int prev = 0;                                      // K: stages of the step before (0, 1 or, with K/V of their own, 2)
                // tiles of the step at t: 1, or (split) up to 2
                auto width = [&](const Segment& s, int tt) { return split ? min(2, s.t_last - tt) : 1; };
#pragma unroll 1
                while (left > 0 && ok) {
                    const int w = width(sg, t);
                    const bool two = !shared_kv && (!split || w > 1);           // stream 1 has a stage of its own in this step
                    if (V) {
                        // what follows this step decides how many K stages lie between
                        const bool seg_end = t + w >= sg.t_last, more = left > w;
                        Segment nx = sg;
                        if (seg_end && more) nx = next_segment(sg, left - w, p, s_len);
                        const bool next_two = more && !shared_kv && (!split || nx.t_last - (seg_end ? 0 : t + w) > 1);
                        if (prev == 0) { pass(1 + (two ? 1 : 0)); prev = 1; }   // K of the first step
#pragma unroll 1
                        for (int g = 0; g < (two ? 2 : 1) && ok; ++g) {
                            emit(split ? t + g : t, g);
                            if (g == 0) pass(more ? 1 : 0);
                        }
                        if (!ok) break;
                        pass(next_two ? 1 : 0);
                        if (seg_end && more) {
                            if (!F8) load_q(nx, ++n_seg);
                            prefetch_ragged(nx);
                            sg = nx;
                            pg_t = -1;
                            t = 0;
                        } else {
                            t += w;
                        }
                    } else {
#pragma unroll 1
                        for (int g = 0; g < 2 && ok; ++g) {
                            pass(prev > g ? 1 : 0);                // V of the step before
                            if (g == 0 || two) emit(split ? t + g : t, g);
                        }
                        if (!ok) break;
                        prev = two ? 2 : 1;
                        t += w;
                        if (t >= sg.t_last && left > w) {
                            sg = next_segment(sg, left - w, p, s_len);
                            pg_t = -1;
                            t = 0;
                        }
                    }
                    left -= w;
                }
                if (!ok && !stop) {
                    // let copies already in flight land before the CTA's shared memory goes away (every stage's last fill)
                    for (int s = 0; s < ring_n; ++s) ptx::mbar_wait(&ctrl->full[st0 + s], (s < (int)st ? ph : ph ^ 1) ^ 1, 20000000ll);
                }
            }
        } else if (n_tiles > 0) {
            // ======================================================================= tensor-core issuers
            // One warp per stream: what a warp executes between two chains (waits, ring bookkeeping, ~800 cycles) is more than the
            // tensor cores' queue covers, so one warp for both left them idle a third of the time.  They take turns issuing: left
            // to themselves the two streams fall into step, both in their softmax and then both waiting.  (The turns also keep an
            // issuer that has no tile in a step, or skips the other's stages, within one round of the ring: further ahead, a
            // stage's parity would pass for that of the round before.)  The whole warp walks the schedule and one elected lane
            // issues, which keeps descriptors in uniform registers.
            const uint32_t hi_q = ptx::umma_desc_hi_sw128(1024), hi_k = ptx::umma_desc_hi_sw128(C::kGroupStride),
                           hi_v = ptx::umma_desc_hi_sw128(C::kVHalves * 1024);
            const uint32_t q_lo = ptx::umma_desc_lo(ptx::smem_u32(sQ), 16);
            const uint32_t k_lo = ptx::umma_desc_lo(ptx::smem_u32(ring), 16);
            const uint32_t v_lo = ptx::umma_desc_lo(ptx::smem_u32(F8 ? wide : ring), 1024);                    // MN-major: LBO = next 64-column atom
            const uint32_t idesc_pv = (F8 ? attn::umma_idesc_plain(kRows, D) : ptx::umma_idesc_bf16(kRows, D)) | (1u << 16);      // B operand MN-major
            const uint32_t q_half = (uint32_t)(C::kQHalfBytes >> 4), q_buf = (uint32_t)(C::kQBytes >> 4);
            bool ok = true;
            uint32_t st = 0, ph = 0;                 // next ring stage
            uint32_t p_par = 0;                      // parity of the next P
            uint32_t wst = 0, wph = 0;               // e4m3: next widened V tile
            auto skip_k = [&](int n) {               // stages that only the other issuer reads
                st += (uint32_t)n;
                if (st >= (uint32_t)ring_n) { st -= (uint32_t)ring_n; ph ^= 1; }
            };
            auto skip_v = [&](int n) {
                if (!F8) return skip_k(n);
                wst += (uint32_t)n;
                if (wst >= kWideStages) { wst -= kWideStages; wph ^= 1; }
            };
            auto wait = [&](uint64_t* bar, uint32_t parity, int where) { ok = ok && ptx::warp_wait(ctrl, bar, parity, where); };
            auto take_k = [&]() -> uint32_t {        // wait for the next stage of the ring
                const uint32_t s = st;
                wait(&ctrl->full[s], ph, 21);
                skip_k(1);
                return s;
            };
            auto take_v = [&]() -> uint32_t {
                if (!F8) return take_k();
                const uint32_t s = wst;
                wait(&ctrl->wide_full[s], wph, 25);
                skip_v(1);
                return s;
            };
            uint64_t* const v_empty = F8 ? ctrl->wide_empty : ctrl->empty;
            // A cursor over the steps of a segment: tiles and slots from the step's first tile to the segment's (unit's) end.
            struct Cursor {
                int tiles, slots;
                bool first;
            };
            const int step = split ? 2 : 1, sp = split ? 1 : 0, g = warp - 1, own = g & sp;
            auto slots_of = [&](const Cursor& c) { return min(kTileSlots, c.slots - kTileSlots * own); };
            const uint32_t s_d = tmem_base + (uint32_t)(g * kTileTok), o_d = tmem_base + kTmemO + (uint32_t)(g * D);
            // per turn: P V of one step, Q K^T of the next (the first turn only scores)
            Segment sg = ctrl->first;
            Cursor nx = {sg.t_last - sg.t_first, sg.slots_all - sg.t_first * kTileSlots, true}, cur = {0, 0, false};
            int left = n_tiles - nx.tiles;           // tiles behind the segment of nx
            uint32_t seg = 0, turn_par = g == 0 ? 1 : 0;
#pragma unroll 1
            while (ok) {
                // (tiles of its own: the ring holds, per step, V of stream 0, the next K of stream 0, V and next K of stream 1)
                if (!shared_kv && g == 1) { skip_v(cur.tiles > 0); skip_k(nx.tiles > 0); }
                const bool do_pv = cur.tiles > own, do_qk = nx.tiles > own;
                const int buf = split ? (int)(seg & 1) : F8 ? g * 2 + (int)(seg & 1) : g;
                uint32_t vst = 0, kst = 0;
                if (do_pv) vst = take_v();
                if (do_qk) {
                    kst = take_k();
                    if (nx.first) wait(&ctrl->q_full[buf], (split || F8 ? seg >> 1 : seg) & 1, 20);
                }
                const int pv_sl = do_pv ? slots_of(cur) : 0;
                const uint32_t vb = v_lo + vst * (uint32_t)((F8 ? C::kWideBytes : C::kStageBytes) >> 4);
                // O_g (+)= P V: one 16-token step per slot, 8 columns of P
                auto pv = [&](int k0, int k1) {
#pragma unroll 1
                    for (int k = k0; k < k1; ++k)
                        ptx::umma_f16_tmem_a(o_d, s_d + (uint32_t)(k * 8), vb + (uint32_t)(k * (C::kVSlotBytes / 16)), hi_v, idesc_pv, k > 0 || !cur.first);
                };
                if (do_pv) {
                    // the first half of P is multiplied while the softmax is at the second
                    wait(&ctrl->p_full[g][0], p_par, 23);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (ptx::elect_one()) {
                        pv(0, min(pv_sl, kTileSlots / 2));
                        ptx::umma_commit(&ctrl->pv_half[g]);
                    }
                    __syncwarp();
                    wait(&ctrl->p_full[g][1], p_par, 24);
                    p_par ^= 1;
                }
                wait(&ctrl->turn[g], turn_par, 22);
                turn_par ^= 1;
                if (!ok) break;
                ptx::tc_fence_after();
                const uint32_t n_qk = slots_of(nx) * kSlotTok, idesc_qk = F8 ? attn::umma_idesc_plain(kRows, n_qk) : ptx::umma_idesc_bf16(kRows, n_qk);
                const uint32_t kb = k_lo + kst * (uint32_t)(C::kStageBytes >> 4);
                const uint32_t qa = q_lo + (uint32_t)buf * q_buf;
                if (ptx::elect_one()) {
                    if (do_pv) {
                        pv(kTileSlots / 2, pv_sl);
                        ptx::umma_commit(&v_empty[vst]);
                        if (cur.tiles <= step + own) ptx::umma_commit(&ctrl->o_full[g]);      // the accumulator of this segment is complete
                    }
                    if (do_qk) {
                        // S_g = Q K^T: 32 bytes of every row per instruction
#pragma unroll 1
                        for (int kk = 0; kk < C::kRowBytes / 32; ++kk) {
                            const uint32_t a = qa + (kk >> 2) * q_half + (uint32_t)((kk & 3) * 2), b = kb + (uint32_t)((kk >> 2) * 64 + (kk & 3) * 2);
                            if (F8) attn::umma_e4m3_lohi(s_d, a, hi_q, b, hi_k, idesc_qk, kk != 0);
                            else ptx::umma_f16_lohi(s_d, a, hi_q, b, hi_k, idesc_qk, kk != 0);
                        }
                        ptx::umma_commit(&ctrl->s_full[g]);
                        ptx::umma_commit(&ctrl->empty[kst]);
                    }
                    ptx::mbar_arrive(&ctrl->turn[g ^ 1]);
                    // the segment's last Q K^T (split: of either stream, or it has no tile for this one)
                    if (nx.tiles > 0 && nx.tiles <= step + own && (do_qk || nx.first)) ptx::umma_commit(&ctrl->q_empty[buf]);
                }
                __syncwarp();
                if (!shared_kv && g == 0) { skip_v(cur.tiles > sp); skip_k(nx.tiles > sp); }
                if (nx.tiles <= 0) break;
                cur = nx;
                nx.tiles -= step;
                nx.slots -= step * kTileSlots;
                nx.first = false;
                if (nx.tiles <= 0 && left > 0) {
                    sg = next_segment(sg, left, p, s_len);
                    nx.tiles = sg.t_last;
                    nx.slots = sg.slots_all;
                    nx.first = true;
                    left -= nx.tiles;
                    ++seg;
                }
            }
        }
    } else if (F8 && warp >= 12) {
        // =========================================================================== V from e4m3 to f16
        // (Exact.  P stays f16: rounded to e4m3, as an 8-bit P V would need it, each weight is off by up to 6%.)
        const int c_tid = tid - 32 * 12, cw = warp - 12;
        // A thread has the same place in every slot.  Eight neighbouring lanes take four chunks of 16 codes of rows r and r ^ 5:
        // with the swizzle neither their loads nor their stores meet in a bank.
        const int tok = (c_tid >> 6) * 8 + (((c_tid >> 4) & 3) ^ (((c_tid >> 2) & 1) * 5)), chunk = ((c_tid >> 3) & 1) * 4 + (c_tid & 3);
        const uint32_t src_off = attn::kv_slot_off<1>(tok, chunk), dst_off0 = attn::kv_slot_off<2>(tok, 2 * chunk), dst_off1 = attn::kv_slot_off<2>(tok, 2 * chunk + 1);
        // These warps also stage the next unit's Q while they are at this one's V: eight rows per V tile, loaded a tile ahead (a
        // load takes ~3000 cycles here).  split: all four share the one operand; else two per stream.
        const int q_all = p.gs * p.nodes_tile, q_grp = split ? 0 : cw >> 1, q_share = ((split ? (q_all + 3) >> 2 : (q_all + 1) >> 1) + 7) & ~7;
        const int q_row0 = (split ? cw : cw & 1) * q_share, q_rows = min(q_share, q_all - q_row0);
        const StreamId id = stream_of(p, rb, q_grp);
        const E4m3Scale qs(p.q_scale);
        uint2 qv[8];
        int left = n_tiles;
        uint32_t n_seg = 0, st = 0, ph = 0, wst = 0, wph = 1;
        bool ok = true;
        Segment sg = ctrl->first, nx = sg;
        // (the first segment's Q is converted out of the buffers that these warps are about to fill)
        if (left > 0) ok = ptx::warp_wait(ctrl, &ctrl->q_full[0], 0, 28) && (split || ptx::warp_wait(ctrl, &ctrl->q_full[2], 0, 28));
#pragma unroll 1
        while (left > 0 && ok) {
            const int seg_tiles = sg.t_last - sg.t_first;
            left -= seg_tiles;
            int q_at = 0, q_loaded = 0, q_end = 0;                 // next Q: rows stored, loaded, and in all
            if (left > 0) {
                nx = next_segment(sg, left, p, s_len);
                q_end = max(q_rows, 0);
            }
            ++n_seg;
            const int q_buf = split ? (int)(n_seg & 1) : q_grp * 2 + (int)(n_seg & 1);
            auto q_step = [&]() {                                  // store the rows that were loaded, load the next ones
                if (q_at < q_loaded) {
                    if (q_at == 0 && !ptx::warp_wait(ctrl, &ctrl->q_empty[q_buf], ((n_seg >> 1) & 1) ^ 1, 11)) { ok = false; return; }
#pragma unroll 1
                    for (; q_at < q_loaded; ++q_at) {
                        store_q_row(sQ + q_buf * C::kQBytes, q_row0 + q_at, qv[0], qs);
#pragma unroll
                        for (int k = 0; k < 7; ++k) qv[k] = qv[k + 1];         // (rotated: registers take no index)
                    }
                }
                if (q_loaded < q_end) {
                    const int r = q_row0 + q_loaded + lane;        // (eight of the lanes count)
                    const int hl = (id.rt / p.node_tiles) * p.gs + r % p.gs, node = (id.rt % p.node_tiles) * p.nodes_tile + r / p.gs;
                    const uint32_t real = __ballot_sync(0xffffffffu, id.exists && r < p.gs * p.nodes_tile && hl < p.G && node < p.n);
                    const __nv_bfloat16* row = p.q + (((size_t)(nx.layer * p.B + nx.b) * p.n + node) * (size_t)p.Hq + (nx.g * p.heads_per_unit + id.head_off) * p.G + hl) * D;
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const __nv_bfloat16* src = row_of_lane(row, k);
                        qv[k] = make_uint2(0, 0);
                        if (real >> k & 1u) qv[k] = *reinterpret_cast<const uint2*>(src + lane * 4);
                    }
                    q_loaded += 8;
                }
            };
            const int n_v = seg_tiles * (split || shared_kv ? 1 : 2);          // V tiles of this segment
#pragma unroll 1
            for (int i = 0; i < n_v || q_at < q_end; ++i) {
            if (i >= n_v) {                                        // (a short segment: the rest of Q by itself)
                q_step();
                if (!ok) break;
                continue;
            }
            if (!ptx::warp_wait(ctrl, &ctrl->full[ring_n + st], ph, 26) || !ptx::warp_wait(ctrl, &ctrl->wide_empty[wst], wph, 27)) { ok = false; break; }
            const uint8_t* const src = ring + (size_t)(ring_n + st) * C::kStageBytes + src_off;
            uint8_t* const dst = wide + (size_t)wst * C::kWideBytes;
#pragma unroll 1
            for (int k = 0; k < kTileSlots; k += 4) {
                uint4 v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] = *reinterpret_cast<const uint4*>(src + (k + j) * C::kSlotBytes);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint2 a = widen4(v[j].x), b = widen4(v[j].y), c = widen4(v[j].z), e = widen4(v[j].w);
                    *reinterpret_cast<uint4*>(dst + (k + j) * C::kVSlotBytes + dst_off0) = make_uint4(a.x, a.y, b.x, b.y);
                    *reinterpret_cast<uint4*>(dst + (k + j) * C::kVSlotBytes + dst_off1) = make_uint4(c.x, c.y, e.x, e.y);
                }
            }
            ptx::fence_proxy_async();                              // (read by the tensor cores)
            __syncwarp();
            if (lane == 0) { ptx::mbar_arrive(&ctrl->wide_full[wst]); ptx::mbar_arrive(&ctrl->empty[ring_n + st]); }
            if (++st == (uint32_t)ring_n) { st = 0; ph ^= 1; }
            if (++wst == kWideStages) { wst = 0; wph ^= 1; }
            q_step();
            if (!ok) break;
            }
            if (left > 0 && ok && q_end == 0) ok = ptx::warp_wait(ctrl, &ctrl->q_empty[q_buf], ((n_seg >> 1) & 1) ^ 1, 11);      // (no arrival ahead of its phase)
            if (left > 0 && ok) {
                ptx::fence_proxy_async();
                __syncwarp();
                if (lane < 2) ptx::mbar_arrive(&ctrl->q_full[q_buf]);          // (twice: the first segment's Q comes from twice the warps)
            }
            sg = nx;
        }
    } else {
        // =========================================================================== softmax / epilogue
        const int w4 = warp & 3;                                   // TMEM lane quarter of this warp
        const int grp = (warp >> 2) - 1;                           // stream
        const StreamId id = stream_of(p, rb, grp);
        const int row = w4 * 32 + lane;
        const int hl = (id.rt / p.node_tiles) * p.gs + row % p.gs;                   // query head within the KV head's G
        const int node = (id.rt % p.node_tiles) * p.nodes_tile + row / p.gs;
        const bool row_ok = id.exists && row < p.gs * p.nodes_tile && hl < p.G && node < p.n;
        const bool warp_has_rows = __any_sync(0xffffffffu, row_ok);
        const unsigned long long anc0 = tree.anc[row_ok ? node : 0][0], anc1 = tree.anc[row_ok ? node : 0][1];
        const uint32_t lane_base = tmem_base + ((uint32_t)(w4 * 32) << 16);
        const uint32_t s_addr = lane_base + (uint32_t)(grp * kTileTok), o_addr = lane_base + kTmemO + (uint32_t)(grp * D);
        constexpr int kRowW = D + 4;                               // record: D accumulator columns, then (max, sum)
        float sc = p.scale_log2e;                                  // scores -> log2 units (e4m3: times the unit's Q and K scales)
        uint32_t xph = 0;                                          // parity of the split pair's exchange barrier
        auto pair_sync = [&]() -> bool {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&ctrl->pair[w4]);
            const bool r = ptx::warp_wait(ctrl, &ctrl->pair[w4], xph, 35);
            xph ^= 1;
            return r;
        };
        // The two softmax warps of a scheduler, one of either stream, take turns at a tile's exponentials: left to themselves the
        // streams fall into step, both at the special-function unit and then both waiting for their scores.  Not over an e4m3
        // cache: its Q K^T is over so soon that the turns cost more than the step (2.16 -> 2.35 ms).
        uint32_t t_par = grp == 0 ? 1 : 0;
        auto take_turn = [&]() -> bool {
            if (F8) return true;
            const bool r = ptx::warp_wait(ctrl, &ctrl->exp_turn[grp][w4], t_par, 36);
            t_par ^= 1;
            return r;
        };
        auto pass_turn = [&]() {
            if (F8) return;
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&ctrl->exp_turn[grp ^ 1][w4]);
        };
        uint32_t s_par = 0, o_par = 0;
        bool ok = true;
        int left = n_tiles;                                        // tiles from the segment's first to the range's end
        Segment sg = ctrl->first;
        if (F8 && left > 0) {
            // e4m3: the first segment's Q (the ones behind it are staged by the warps that widen V), each warp its rows, or (split)
            // half of them
            const int r0 = split ? grp * 16 : 0, r1 = split ? r0 + 16 : 32, buf = split ? 0 : grp * 2;
            const E4m3Scale qs(p.q_scale);
            const __nv_bfloat16* qrow = p.q + (((size_t)(sg.layer * p.B + sg.b) * p.n + node) * (size_t)p.Hq + (sg.g * p.heads_per_unit + id.head_off) * p.G + hl) * D;
            const uint32_t real = __ballot_sync(0xffffffffu, row_ok);
            // All rows are requested first, into the buffers of widened V, which are not in use yet.  (What this costs is mostly
            // the fetch of code that runs once, at some 600 cycles per 128 bytes: the loops are as short as they can be.)
            uint8_t* const raw = wide + (split ? 0 : grp * C::kWideBytes) + w4 * 32 * 256;
            const int r_end = min(r1, 32 - __clz(real));
#pragma unroll 1
            for (int r = r0 + (lane >> 4); r < r1; r += 2) {
                const __nv_bfloat16* src = row_of_lane(qrow, r);
                if (real >> r & 1u)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ptx::smem_u32(raw + r * 256 + (lane & 15) * 16)), "l"(src + (lane & 15) * 8) : "memory");
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
#pragma unroll 1
            for (int r = r0; r < r_end; ++r)
                store_q_row(sQ + buf * C::kQBytes, w4 * 32 + r, real >> r & 1u ? *reinterpret_cast<const uint2*>(raw + r * 256 + lane * 8) : make_uint2(0, 0), qs);
            ptx::fence_proxy_async();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&ctrl->q_full[buf]);
        }
#pragma unroll 1
        while (left > 0 && ok) {
            float vsc = 1.f;                                       // e4m3: the V scale
            if (F8) {
                const int h = sg.layer * p.Hkv + sg.g * p.heads_per_unit + id.head_off;
                sc = p.scale_log2e * p.q_scale * __ldg(p.k_scale + h);
                vsc = __ldg(p.v_scale + h);
            }
            const uint64_t sc2 = pack2(sc, sc);
            // this row's offset (log2 units) and running sum (rows that do not exist: one that makes every P 0)
            float off = row_ok ? -INFINITY : 1e30f, l_run = 0.f;
            bool redone = false;
            const int mine = split ? (sg.t_last - sg.t_first + 1 - grp) >> 1 : sg.t_last - sg.t_first;     // tiles of this stream
            for (int i = 0; i < mine; ++i) {
                const int t = split ? sg.t_first + 2 * i + grp : sg.t_first + i;
                if (!ptx::warp_wait(ctrl, &ctrl->s_full[grp], s_par, 30)) { ok = false; break; }
                s_par ^= 1;
                ptx::tc_fence_after();
                if (warp_has_rows) {
                    if ((t + 1) * kTileSlots > sg.pages_full) mask_tile(s_addr, t * kTileSlots, sg, anc0, anc1);
                    // The offset is set by the first tile in which the row sees anything (before that every P was 0).
                    if (__any_sync(0xffffffffu, off == -INFINITY)) {
                        const float mx = tile_max(s_addr, 4);
                        if (off == -INFINITY) off = mx * sc;       // (-inf when nothing is visible yet)
                    }
                    // Two halves of 64 scores, one copy of the code.  P of a half goes over S columns that have been read.
                    float sum = 0.f;
                    uint32_t ra[32];
                    ptx::tmem_ld_32x32b_x32(s_addr, ra);
                    if (!take_turn()) { ok = false; break; }
#pragma unroll 1
                    for (int h = 0; h < 2;) {
                        uint32_t pk[32], rb_[32];
                        const float o = (off == -INFINITY) ? 0.f : -off;
                        const uint64_t no2 = pack2(o, o);
                        uint64_t s0 = 0, s1 = 0;                   // (two zeros each)
                        tmem_ld_wait32(ra);
                        ptx::tmem_ld_32x32b_x32(s_addr + (uint32_t)(h * 64 + 32), rb_);
                        exp_chunk<F8>(ra, sc2, no2, pk, s0, s1);
                        tmem_ld_wait32(rb_);
                        ptx::tmem_ld_32x32b_x32(s_addr + 64, ra);  // (of no use to the second half)
                        exp_chunk<F8>(rb_, sc2, no2, pk + 16, s0, s1);
                        float a, b;
                        unpack2(add2(s0, s1), a, b);
                        const float half_sum = a + b;
                        // The offset moves when the sum outgrows the limit (an overflow makes it infinite, which counts): rare, and
                        // then this half is redone.  (The accumulator may be touched: the tile before was multiplied before this
                        // tile was scored, and for this tile's first half there is a barrier.)
                        if (h == 1 && !redone) pass_turn();
                        const bool grow = half_sum > kSumLimit && !redone;
                        if (__any_sync(0xffffffffu, grow)) {
                            tmem_ld_wait32(ra);
                            if (h == 1) {
                                if (!ptx::warp_wait(ctrl, &ctrl->pv_half[grp], s_par ^ 1, 33)) { ok = false; break; }
                                ptx::tc_fence_after();
                            }
                            const float2 m = move_offset(s_addr + (uint32_t)(h * 64), o_addr, i + h > 0 ? D : 0, grow, off, sc);
                            off = m.x;
                            l_run *= m.y;
                            sum *= m.y;
                            redone = true;
                            ptx::tmem_ld_32x32b_x32(s_addr + (uint32_t)(h * 64), ra);
                            continue;
                        }
                        redone = false;
                        sum += half_sum;
                        tmem_st_32x32b_x32(s_addr + (uint32_t)(h * 32), pk);
                        tmem_st_wait();
                        ptx::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(&ctrl->p_full[grp][h]);
                        ++h;
                    }
                    if (!ok) break;
                    tmem_ld_wait32(ra);
                    l_run += sum;
                } else {
                    if (!take_turn()) { ok = false; break; }
                    pass_turn();
                    if (lane == 0) { ptx::mbar_arrive(&ctrl->p_full[grp][0]); ptx::mbar_arrive(&ctrl->p_full[grp][1]); }
                }
            }
            if (ok && split && grp == 1 && ((sg.t_last - sg.t_first) & 1)) {       // (stream 0 has one tile more)
                ok = take_turn();
                pass_turn();
            }
            if (!ok) break;
            // ---- end of this CTA's part of the unit
            const bool whole = sg.t_first == 0 && sg.t_last == sg.tiles;
            const int head = (sg.g * p.heads_per_unit + id.head_off) * p.G + hl;
            const size_t lb = (size_t)sg.layer * p.B + sg.b;
            __nv_bfloat16* orow = p.out + ((lb * p.n + node) * (size_t)p.Hq + head) * D;
            float* lse_ptr = p.lse_out ? p.lse_out + (lb * p.Hq + head) * p.n + node : nullptr;
            const int slot = (sg.t_first > 0) ? 0 : 1;             // a unit that began before this CTA's range uses slot 0
            // record layout [column][row]: a warp's store of one column is one contiguous 128-byte line
            float* rec = p.partial + (((size_t)ctrl->place * 2 + slot) * 2 + (split ? 0 : grp)) * kRowW * kRows + row;
            left -= sg.t_last - sg.t_first;
            Segment nx = sg;
            if (left > 0) nx = next_segment(sg, left, p, s_len);
            if (split) {
                float* xc = xch + (size_t)row * 4;                 // [row][stream][offset, sum]
                xc[grp * 2] = off;
                xc[grp * 2 + 1] = l_run;
            }
            if (mine > 0) {
                if (!ptx::warp_wait(ctrl, &ctrl->o_full[grp], o_par, 32)) { ok = false; break; }
                o_par ^= 1;
            }
            float M = off, Lsum = l_run;
            float w0 = 1.f, w1 = 0.f;
            if (split) {
                ptx::tc_fence_before();
                if (!pair_sync()) { ok = false; break; }
                const float* xc = xch + (size_t)row * 4;
                const float m_a = xc[0], l_a = xc[1], m_b = xc[2], l_b = xc[3];       // (a stream without tiles: -inf, 0)
                M = fmaxf(m_a, m_b);
                w0 = m_a != -INFINITY ? exp2f(m_a - M) : 0.f;
                w1 = m_b != -INFINITY ? exp2f(m_b - M) : 0.f;
                Lsum = w0 * l_a + w1 * l_b;
            }
            ptx::tc_fence_after();
            if (warp_has_rows) {
                const float inv = 1.f / Lsum;                      // (e4m3: V codes times the unit's V scale)
                // split: this warp combines its half of the columns of both accumulators; otherwise all columns of its own.
                // (16 columns at a time: this runs once per unit, and what it costs is mostly the instruction fetch)
                const int c_lo = split ? grp * (D / 2) : 0, c_hi = split ? c_lo + D / 2 : D;
                const uint32_t o_first = split ? lane_base + kTmemO : o_addr;
                if (!split) w0 = M != -INFINITY ? 1.f : 0.f;
                if (whole) { w0 *= inv; w1 *= inv; }
                if (F8) { w0 *= vsc; w1 *= vsc; }
#pragma unroll 1
                for (int c = c_lo; c < c_hi; c += 16) {
                    uint32_t r[16];
                    float acc[16];
                    ptx::tmem_ld_32x32b_x16(o_first + (uint32_t)c, r);
                    tmem_ld_wait16(r);
                    // (an accumulator that no P V wrote may hold anything: a weight of 0 does not read it)
#pragma unroll
                    for (int j = 0; j < 16; ++j) acc[j] = w0 != 0.f ? w0 * __uint_as_float(r[j]) : 0.f;
                    if (split) {
                        ptx::tmem_ld_32x32b_x16(o_first + (uint32_t)(D + c), r);
                        tmem_ld_wait16(r);
#pragma unroll
                        for (int j = 0; j < 16; ++j) acc[j] = w1 != 0.f ? fmaf(w1, __uint_as_float(r[j]), acc[j]) : acc[j];
                    }
                    if (!whole) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) rec[(size_t)(c + j) * kRows] = acc[j];
                    } else if (row_ok) {
                        *reinterpret_cast<uint4*>(orow + c) = make_uint4(pack_bf16(acc[0], acc[1]), pack_bf16(acc[2], acc[3]), pack_bf16(acc[4], acc[5]), pack_bf16(acc[6], acc[7]));
                        *reinterpret_cast<uint4*>(orow + c + 8) = make_uint4(pack_bf16(acc[8], acc[9]), pack_bf16(acc[10], acc[11]), pack_bf16(acc[12], acc[13]), pack_bf16(acc[14], acc[15]));
                    }
                }
                if (!split || grp == 0) {
                    if (!whole) {
                        rec[(size_t)D * kRows] = M;
                        rec[(size_t)(D + 1) * kRows] = Lsum;
                    } else if (lse_ptr && row_ok) {
                        *lse_ptr = M * kAttnLn2 + logf(Lsum);
                    }
                }
            }
            // (split: the exchange words are rewritten and the accumulators overwritten in the next part: both warps must
            // have read them.  Otherwise a stream's next P V waits for a P that its own warps write after this.)
            ptx::tc_fence_before();
            if (split && !pair_sync()) { ok = false; break; }
            sg = nx;
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

// Merge of the units that the partition cut: one block per (inner boundary, row tile of the group).
template <int D>
__global__ void __launch_bounds__(attn::kMergeThreads) attn_merge_kernel(const __grid_constant__ AttnParams p) {
    const int n_str = p.mode == kSplit ? 1 : 2;
    const int rb = blockIdx.y / n_str, grp = blockIdx.y % n_str;
    const StreamId id = stream_of(p, rb, grp);
    // (behind a launch that itself has waited for the attention, its records are complete: only this launch's end has to wait)
    ptx::grid_dep_launch();                       // (the kernel behind only sets itself up before this one has completed)
    if (!p.late_merge) ptx::grid_dep_wait();
    attn::merge_boundary<D>(
        p.begins, p.n_groups, p.n, p.Hq, p.B, p.out, p.lse_out, p.status, p.wait_limit, p.stall_merge,
        [&](int row, const attn::GroupBegin& u, int& node, int& head) {
            const int hl = (id.rt / p.node_tiles) * p.gs + row % p.gs;
            node = (id.rt % p.node_tiles) * p.nodes_tile + row / p.gs;
            head = (u.g * p.heads_per_unit + id.head_off) * p.G + hl;
            return id.exists && row < p.gs * p.nodes_tile && hl < p.G && node < p.n;
        },
        [&](int group, int slot) { return p.partial + (((size_t)(group * p.n_cta + rb) * 2 + slot) * 2 + grp) * (D + 4) * kRows; });
    if (p.late_merge) ptx::grid_dep_wait();
}

mirror_status merge_launch(mirror_ctx* ctx, const AttnParams& p, cudaStream_t stream) {
    auto merge = ctx->desc.head_dim == 128 ? attn_merge_kernel<128> : attn_merge_kernel<64>;
    const dim3 grid((unsigned)(p.n_groups - 1), (unsigned)(p.n_cta * (p.mode == kSplit ? 1 : 2)));
    MIRROR_CUDA_OK(cudaFuncSetAttribute(merge, cudaFuncAttributeMaxDynamicSharedMemorySize, attn::kMergeSmem));
    MIRROR_CUDA_OK(mirror_launch_pdl(merge, grid, dim3(attn::kMergeThreads), attn::kMergeSmem, stream, p));
    ctx->launches += 1;
    MIRROR_CUDA_OK(cudaGetLastError());
    return MIRROR_OK;
}

}  // namespace

mirror_status mirror_attn_launch(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree, const MirrorTreeInfo& ti,
                                 const void* q, const void* k_new, const void* v_new, void* out, float* lse_out,
                                 float* partial_ws, cudaStream_t stream, const MirrorAttnFp8* f8, bool keep_rounding,
                                 MirrorAttnBeside* beside, bool early) {
    if (keep_rounding && !f8) return mirror_attn_tile64_launch(ctx, kv, tree, ti, q, k_new, v_new, out, lse_out, partial_ws, stream, early);
    const int D = ctx->desc.head_dim, Hkv = ctx->desc.n_kv_heads, Hq = ctx->desc.n_q_heads;
    AttnParams p;
    p.L = kv->num_layers; p.B = tree->batch; p.n = ti.n; p.Hq = Hq; p.Hkv = Hkv; p.G = Hq / Hkv;
    if (p.B > kAttnMaxBatch) return MIRROR_ERR_SHAPE;
    // Row tiles of whole nodes: the G heads of a KV head, or (large G) an even share of them, times as many nodes as 128
    // rows hold; the share that needs the fewest tiles, the nodes spread evenly over them.
    p.n_rt = 0;
    for (int hc = (p.G + kRows - 1) / kRows; hc <= p.G && hc <= 8 + (p.G + kRows - 1) / kRows; ++hc) {
        const int gs = (p.G + hc - 1) / hc, node_tiles = (p.n + kRows / gs - 1) / (kRows / gs), shares = (p.G + gs - 1) / gs;
        if (p.n_rt == 0 || shares * node_tiles < p.n_rt) {
            p.n_rt = shares * node_tiles;
            p.gs = gs;
            p.node_tiles = node_tiles;
            p.nodes_tile = (p.n + node_tiles - 1) / node_tiles;
        }
    }
    p.mode = p.n_rt == 1 ? kSplit : kPaired;
    // (a group of two heads needs a CTA per row tile: not with more row tiles than SMs, where a head alone still fits)
    p.heads_per_unit = (p.n_rt > 1 && p.n_rt % 2 == 1 && Hkv % 2 == 0 && p.n_rt <= ctx->num_sms) ? 2 : 1;
    p.n_cta = p.heads_per_unit == 2 ? p.n_rt : (p.n_rt + 1) / 2;
    p.n_groups = ctx->num_sms / p.n_cta;
    if (ctx->tune.attn_groups >= 1 && ctx->tune.attn_groups <= p.n_groups) p.n_groups = ctx->tune.attn_groups;
    if (p.n_groups < 1 || p.n_groups * sizeof(attn::GroupBegin) > kWsNotesBytes) return MIRROR_ERR_SHAPE;
    p.snap_cap = (ctx->tune.attn_snap + 1) / 2;              // (given in tiles of 64 tokens)
    // Units of at most six tiles (the page table says how long a prefix can be) take a CTA less time whole than the merge
    // kernel behind a cut would: a launch and a pass over the records, ~6 us.
    const bool whole = ctx->tune.attn_whole_units != 0;
    const int64_t units = (int64_t)p.L * p.B * (Hkv / p.heads_per_unit);
    if (units > 0x7fffffff) return MIRROR_ERR_SHAPE;        // (a unit has a tile at least: the tiles are counted in 31 bits)
    p.units = (int)units;
    p.whole_groups = whole && units >= p.n_groups ? attn::whole_unit_groups(p.n_groups, units) : 0;
    p.unit_cuts = whole && units < p.n_groups ? p.n_groups / (int)units : 0;
    p.cut_tiles = f8 || p.unit_cuts == 1 ? 8 : 2;
    const int most_tiles = (kv->max_pages_per_req + (p.n + kSlotTok - 1) / kSlotTok + kTileSlots - 1) / kTileSlots;      // of a unit
    p.never_cut = whole && most_tiles <= 6;
    // Beside a weight stream: whole units, where one request's are short (a cut costs about as much as two tiles, a launch behind it not counted).
    p.lm_ns = 0.f;
    p.deal = p.never_cut || (whole && p.B == 1 && units >= 2 * p.n_groups && most_tiles <= 64);
    p.group_chunk = p.n_cta % 2 ? 2 : 1;
    // One request: all units have the same length whatever it is, so the host can tell when the partition gives every
    // group whole units (each unit holds at least one tile): nothing is cut and the merge kernel has nothing to do.
    bool no_cuts = p.n_groups == 1 || p.never_cut || (p.B == 1 && (p.whole_groups > 0 || (p.unit_cuts == 1 && cuts_pay(most_tiles, p.units, p.n_groups, 1, p.cut_tiles))));
    p.late_merge = 0;
    if (beside) {
        // Is the launch behind to run beside this one?  Its merge then comes last (~10 us): yes where there is none, where a shared
        // chip is the faster one if prefixes are as long as the page table allows (the device, which knows them, decides), and
        // unless this one takes so much longer that nothing is gained; with many rows, where what it fills in, the time
        // between the first CTA's end and the last one's, is longer than the merge.
        // SMs are left to it only if it comes in more units than fit the chip at a time: of a single wave those that find no SM take as
        // long behind this launch as all of them would.  (32 layers of 1500 tokens before 32000 ids of 4096, SMs left / not: 17 nodes 111 /
        // 97 us, 57 nodes 170 / 152; 42 layers of 106 tokens before 12480 ids of 7680: 66 / 60.)
        // How good the choices are, over 90 drawn steps of up to 128 rows: 4.4% shorter than in sequence by the geometric mean, at worst 2.4%
        // longer; the best of eight fixed shares, another one each time, is 4% below them, and more than 12% for a tenth of the steps.
        const float tiles = (float)most_tiles * (float)p.units, step_bytes = (float)(kTileTok * 2 * D * (f8 ? 1 : 2) * (p.mode == kSplit ? 2 : 1));
        const int most = std::min(p.n_groups, p.units), sms = ctx->num_sms;
        p.lm_ns = beside->work_ns;
        const Share all = share_choice(p, tiles, most, sms, step_bytes, 0);
        bool share = false;
        if (beside->stream && beside->in_parts && beside->work_ns > 2e4f && 3 * most * p.n_cta > sms && p.n_groups > 1)
            for (int c = 1; c < 32; ++c) share |= share_choice(p, tiles, most, sms, step_bytes, c).total < kShareGain * all.total;
        const float attn_ns = all.total - p.lm_ns;
        beside->granted = no_cuts || share || (beside->stream ? attn_ns < 8.f * beside->work_ns : attn_ns > 3e5f && beside->work_ns > 0.25f * attn_ns);
        if (!share) p.lm_ns = 0.f;
        else no_cuts = no_cuts && p.deal;
        p.late_merge = beside->granted;
    }
    p.wait_limit = ctx->tune.wait_limit_cycles;
    p.stall_after = (ctx->tune.test_stall_after >= 0 && ctx->tune.test_stall_attn_left-- > 0) ? ctx->tune.test_stall_after : -1;
    p.stall_merge = ctx->tune.test_stall_merges > 0 && ctx->tune.test_stall_merges-- > 0;
    p.max_pages = kv->max_pages_per_req; p.num_pages = kv->num_pages;
    const int64_t page_elems = (int64_t)Hkv * kSlotTok * D;
    if (kv->layer_stride % page_elems != 0) return MIRROR_ERR_UNSUPPORTED;
    p.layer_pages = (int)(kv->layer_stride / page_elems);
    p.tree_slots = (p.n + kSlotTok - 1) / kSlotTok;
    p.scale_log2e = ctx->scale * 1.4426950408889634f;
    p.page_table = kv->page_table; p.prefix_len = kv->prefix_len;
    if (f8 && (!f8->k_scale || !f8->v_scale || !(f8->q_scale > 0.f))) return D != 128 ? MIRROR_ERR_UNSUPPORTED : MIRROR_ERR_ARG;
    if (f8 && D != 128) return MIRROR_ERR_UNSUPPORTED;
    p.q = (const __nv_bfloat16*)q;
    p.k_scale = f8 ? f8->k_scale : nullptr; p.v_scale = f8 ? f8->v_scale : nullptr; p.q_scale = f8 ? f8->q_scale : 1.f;
    p.v_pool = (const __nv_bfloat16*)kv->v_pool;
    p.out = (__nv_bfloat16*)out; p.lse_out = lse_out;
    p.partial = partial_ws; p.begins = (attn::GroupBegin*)((uint8_t*)partial_ws - kWsNotesBytes); p.status = ctx->d_status;

    AttnTree at;
    memcpy(at.anc, ti.anc, sizeof at.anc);
    Maps tm;
    {
        // pool as (64 columns, 8 tokens, D/64 halves, 2 token groups, (layer*page)*head): one box is one page of one head,
        // landing as [token / 8][half][token % 8][128 B] (e4m3 pools through the same 16-bit map: 64 "columns" are a row's 128 bytes)
        const uint64_t total_pages = (uint64_t)(p.L - 1) * p.layer_pages + p.num_pages, row = (uint64_t)D * (f8 ? 1 : 2);
        const uint64_t dims[5] = {64, 8, row / 128, 2, total_pages * (uint64_t)Hkv};
        const uint64_t strides[4] = {row, 128, 8 * row, kSlotTok * row};
        const uint32_t box[5] = {64, 8, (uint32_t)(row / 128), 2, 1};
        mirror_status st = mirror_make_tmap(ctx, &tm.k, kv->k_pool, 5, dims, strides, box);
        if (st == MIRROR_OK) st = mirror_make_tmap(ctx, &tm.v, kv->v_pool, 5, dims, strides, box);
        if (st != MIRROR_OK) return st;
        // the tree's K/V as (64 columns, n tokens, D/64 halves, heads, layer*request): one box is eight tokens of one head
        const uint64_t lb = (uint64_t)p.L * p.B;
        const uint64_t ndims[5] = {64, (uint64_t)p.n, row / 128, (uint64_t)Hkv, lb};
        const uint64_t nstrides[4] = {Hkv * row, 128, row, (uint64_t)p.n * Hkv * row};
        const uint32_t nbox[5] = {64, 8, (uint32_t)(row / 128), 1, 1};
        st = mirror_make_tmap(ctx, &tm.kn, k_new, 5, ndims, nstrides, nbox);
        if (st == MIRROR_OK) st = mirror_make_tmap(ctx, &tm.vn, v_new, 5, ndims, nstrides, nbox);
        if (st != MIRROR_OK) return st;
        if (!f8) {
        // Q as (64 columns, heads, n nodes, D/64 halves, layer*request): one box is one half of a row tile
        const uint64_t qdims[5] = {64, (uint64_t)Hq, (uint64_t)p.n, row / 128, lb};
        const uint64_t qstrides[4] = {row, Hq * row, 128, (uint64_t)p.n * Hq * row};
        const uint32_t qbox[5] = {64, (uint32_t)p.gs, (uint32_t)p.nodes_tile, 1, 1};
        st = mirror_make_tmap(ctx, &tm.q, q, 5, qdims, qstrides, qbox);
        if (st != MIRROR_OK) return st;
        }
    }
    auto launch = [&](auto cfg, auto kern) -> mirror_status {
        using C = decltype(cfg);
        const size_t fixed = (f8 && p.mode != kSplit ? 4 : 2) * (size_t)C::kQBytes + C::kFixedBytes + (p.mode == kSplit ? kRows * 16 : 0) + (2 * (size_t)p.B + 1) * 4;
        int stages = (int)((kSmemLimit - fixed) / C::kStageBytes);
        if (stages > kMaxStages) stages = kMaxStages;
        if (f8) stages &= ~1;                               // (K and V have half each)
        if (stages < 4) return MIRROR_ERR_UNSUPPORTED;
        const size_t smem = fixed + (size_t)stages * C::kStageBytes;
        MIRROR_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit));
        cudaLaunchConfig_t cfg_l = {};
        cfg_l.gridDim = dim3((unsigned)(p.lm_ns > 0.f ? align_up((size_t)p.n_groups * p.n_cta, 2) : (size_t)p.n_groups * p.n_cta));
        cfg_l.blockDim = dim3(C::kThreads);
        cfg_l.dynamicSmemBytes = smem;
        cfg_l.stream = stream;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;       // (neighbouring blocks on the SMs of a TPC: see spread_group)
        attr[1].val.clusterDim.x = 2;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
        cfg_l.attrs = attr;
        cfg_l.numAttrs = p.lm_ns > 0.f ? 2 : 1;
        MIRROR_CUDA_OK(cudaLaunchKernelEx(&cfg_l, kern, tm, at, p, stages));
        ctx->launches += 1;
        MIRROR_CUDA_OK(cudaGetLastError());
        if (no_cuts) return MIRROR_OK;
        if (p.late_merge) {
            static_assert(sizeof(AttnParams) <= sizeof beside->merge, "room for the launch's parameters");
            beside->merge_needed = true;
            memcpy(beside->merge, &p, sizeof p);
            return MIRROR_OK;
        }
        // which units the partition cut is only known on the device (it depends on the prefix lengths)
        return merge_launch(ctx, p, stream);
    };
    if (f8) return launch(Cfg<128, true>{}, attn_verify_kernel<128, true, false>);        // (its softmax warps read q themselves)
    if (D == 128) return launch(Cfg<128, false>{}, early ? attn_verify_kernel<128, false, true> : attn_verify_kernel<128, false, false>);
    return launch(Cfg<64, false>{}, early ? attn_verify_kernel<64, false, true> : attn_verify_kernel<64, false, false>);
}

mirror_status mirror_attn_late_merge(mirror_ctx* ctx, const MirrorAttnBeside& beside, cudaStream_t stream) {
    if (!beside.merge_needed) return MIRROR_OK;
    AttnParams p;
    memcpy(&p, beside.merge, sizeof p);
    return merge_launch(ctx, p, stream);
}
