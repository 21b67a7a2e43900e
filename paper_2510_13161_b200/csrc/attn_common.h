// Definitions shared by the two attention kernels (attn_verify.cu, attn_tile64.cu).
#pragma once
#include "mirror_internal.h"

// Token tree as the kernels read it: bit j of anc[i] says that node j is node i or an ancestor of it.
struct AttnTree {
    unsigned long long anc[MIRROR_MAX_NODES][2];
};

constexpr int kAttnSlotTok = 16;                    // keys are cut in 16-token slots: one KV page, or 16 tree tokens
constexpr int kAttnMaxBatch = 1024;
constexpr float kAttnLn2 = 0.6931471805599453f;

#ifdef __CUDACC__
namespace attn {

// Group count that gives every group the same number of whole units, if one exists within 15% of n_groups; else 0.
// (Host and device: the host uses it to tell whether a launch can cut a unit at all.)
__host__ __device__ inline int whole_unit_groups(int n_groups, long long units) {
    for (int g = n_groups; g >= 1 && g * 100 >= n_groups * 85; --g)
        if (units % g == 0) return g;
    return 0;
}

// Shared-memory placement of a K/V slot (16 tokens of one head): [token / 8][64-column half][token % 8][128 B], so the
// 8-token groups of one half are 1024 * (d / 64) bytes apart, uniformly across the slots of a ring: that is the
// 8-row-group stride (SBO) of the K-major Q K^T operand and, with the halves 1024 B apart (LBO), the MN-major P V operand.
template <int HALVES>
__device__ __forceinline__ uint32_t kv_slot_off(int tok, int chunk) {                 // chunk: 16-byte column chunk
    return (uint32_t)((tok >> 3) * HALVES * 1024 + (chunk >> 3) * 1024 + (tok & 7) * 128 + (((chunk & 7) ^ (tok & 7)) << 4));
}

// Visibility of the 16 score columns of slot `sl` for a row whose visible tree tokens are the bits of (anc0, anc1).
__device__ __forceinline__ uint32_t slot_mask(int sl, int pages_full, int pages_all, int slots_all, int len, unsigned long long anc0,
                                              unsigned long long anc1) {
    if (sl < pages_full) return 0xffffu;
    if (sl < pages_all) return (1u << (len - sl * kAttnSlotTok)) - 1u;                 // ragged page: 1..15 valid tokens
    if (sl >= slots_all) return 0;
    const int ts = sl - pages_all;                                                      // tree tokens 16*ts .. 16*ts+15
    return (uint32_t)(((ts < 4) ? anc0 : anc1) >> ((ts & 3) * 16)) & 0xffffu;           // ancestors-or-self (all < n)
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// ---- merge of the units that the partition cut across CTA groups ------------------------------------------------
// What a CTA group leaves for the merge: the unit that its range begins inside of (part == 0: it begins with a unit).
struct GroupBegin {
    int part, layer, b, g;
};
constexpr int kMergeThreads = 512;        // 128 rows x 4 column quarters
constexpr int kMergeBatch = 32;           // parts whose (max, sum) are in shared memory at a time

// A block per (inner boundary, row tile) and blockIdx.z.  A unit cut by k boundaries left k + 1 (max, sum, accumulator)
// records, like split-KV partials; the blocks of those boundaries share its merge by output columns (8-column chunks
// dealt round-robin), each combining all parts of its columns in group order, so a unit that many CTAs shared (few units
// per launch, long contexts) is not merged by one block alone.  Which unit a boundary cuts is read from the groups' own
// notes (finding it again from the lengths cost more than the merge).  What bounds it is the chain of loads and the
// fetch of code that runs once, so the code is small: the parts' (max, sum) come side by side into shared memory and
// become weights there, and the loop over the parts is two loads and three multiply-adds.
// map(row, GroupBegin) -> false, or the row's node and query head; record(group, slot) -> its record in slot 0 (of the unit
// that began before the group's range) or 1, [column][128 rows], D accumulator columns, then (max, sum).
template <int D, class Map, class Record>
__device__ __forceinline__ void merge_boundary(const GroupBegin* table, int n_groups, int n, int Hq, int B, __nv_bfloat16* out, float* lse_out,
                                               Map map, Record record) {
    __shared__ GroupBegin s_begin[512];
    __shared__ float s_w[kMergeBatch][128], s_l[kMergeBatch][128];              // max, then weight; sum
    const int tid = threadIdx.x, g = blockIdx.x + 1;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    for (int i = tid; i < n_groups; i += kMergeThreads) s_begin[i] = table[i];
    __syncthreads();
    const GroupBegin u = s_begin[g];
    if (!u.part) return;                                                        // the boundary is a unit boundary (or beyond the last group)
    // the groups ga..gb hold this unit's parts; the blocks of the boundaries ga+1..gb share the merge by columns
    auto same = [&](int i) { const GroupBegin& v = s_begin[i]; return v.part && v.layer == u.layer && v.b == u.b && v.g == u.g; };
    int ga = g - 1, gb = g;
    while (ga > 0 && same(ga)) --ga;
    while (gb + 1 < n_groups && same(gb + 1)) ++gb;
    const int parts = gb - ga + 1;
    const int n_blocks = (parts - 1) * gridDim.z, j_blk = (g - (ga + 1)) * gridDim.z + blockIdx.z;

    constexpr int kChunks = D / 8;                                              // 8 output columns, 2 of them a thread quarter's
    const int row = tid & 127, cq = tid >> 7;
    int node = 0, head = 0;
    const bool has_row = map(row, u, node, head);
    const size_t lb = (size_t)u.layer * B + u.b;
    // group ga holds the unit's first tile (its record is in slot 1), the later groups began inside the unit (slot 0)
    const float* const first = record(ga, 1) + row;
    const float* const second = record(ga + 1, 0) + row;
    const size_t stride = record(1, 0) - record(0, 0);
    auto part_of = [&](int k) -> const float* { return k == 0 ? first : second + (size_t)(k - 1) * stride; };
    auto load_batch = [&](int k0) {                                             // (max, sum) of the parts from k0 on
        const int nk = has_row ? min(kMergeBatch, parts - k0) : 0;
#pragma unroll 4
        for (int k = cq; k < nk; k += 4) {
            const float* src = part_of(k0 + k) + (size_t)D * 128;
            s_w[k][row] = __ldcg(src);
            s_l[k][row] = __ldcg(src + 128);
        }
        __syncthreads();
        return nk;
    };
    auto weigh = [&](int nk, float M) {
        __syncthreads();                                                        // (all maxima of the batch have been read)
        for (int k = cq; k < nk; k += 4) s_w[k][row] = s_w[k][row] == -INFINITY ? 0.f : exp2f(s_w[k][row] - M);
        __syncthreads();
    };
    float Mm = -INFINITY;
    int nk = 0;
#pragma unroll 1
    for (int k0 = 0; k0 < parts; k0 += kMergeBatch) {
        if (k0 > 0) __syncthreads();
        nk = load_batch(k0);
        for (int k = 0; k < nk; ++k) Mm = fmaxf(Mm, s_w[k][row]);
    }
    const bool one_batch = parts <= kMergeBatch;
    if (one_batch) weigh(nk, Mm);
    const bool writes_lse = lse_out && j_blk == 0;
#pragma unroll 1
    for (int chunk = j_blk; chunk < kChunks; chunk += n_blocks) {
        float Lm = 0.f, a0 = 0.f, a1 = 0.f;
        const size_t col = (size_t)(chunk * 8 + cq * 2) * 128;
#pragma unroll 1
        for (int k0 = 0; k0 < parts; k0 += kMergeBatch) {
            if (!one_batch) {
                __syncthreads();
                nk = load_batch(k0);
                weigh(nk, Mm);
            }
#pragma unroll 8
            for (int k = 0; k < nk; ++k) {
                const float* src = part_of(k0 + k) + col;
                const float wgt = s_w[k][row];
                Lm = fmaf(wgt, s_l[k][row], Lm);
                a0 = fmaf(wgt, __ldcg(src), a0);
                a1 = fmaf(wgt, __ldcg(src + 128), a1);
            }
        }
        if (!has_row) continue;
        const float inv = 1.f / Lm;
        *reinterpret_cast<uint32_t*>(out + ((lb * n + node) * (size_t)Hq + head) * D + chunk * 8 + cq * 2) = pack_bf16(a0 * inv, a1 * inv);
        if (writes_lse && chunk == 0 && cq == 0) lse_out[(lb * Hq + head) * n + node] = Mm * kAttnLn2 + logf(Lm);
    }
}

}  // namespace attn
#endif
