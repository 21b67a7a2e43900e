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

// Instruction descriptor with format codes 0: e4m3 x e4m3 (kind::f8f6f4) or f16 x f16 (kind::f16) -> fp32, tile M x N.
__device__ __forceinline__ uint32_t umma_idesc_plain(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// D (+)= A B^T with both operands e4m3 in shared memory (descriptor halves), 32 columns.
__device__ __forceinline__ void umma_e4m3_lohi(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                               uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// ---- merge of the units that the partition cut across CTA groups ------------------------------------------------
// What a CTA group leaves for the merge: the unit that its range begins inside of (part == 0: it begins with a unit).
struct GroupBegin {
    int part, layer, b, g;
};
constexpr int kMergeThreads = 512;        // 128 rows x 4 column quarters
constexpr int kMergeSlots = 32;           // (part, 8-column chunk) pairs in shared memory at a time
constexpr int kMergeSmem = kMergeSlots * 10 * 128 * 4;      // their columns, then the parts' (max, sum)

// A block per (inner boundary, row tile).  A unit cut by k boundaries left k + 1 (max, sum, accumulator) records, like
// split-KV partials; the k blocks of those boundaries share its merge by output columns (8-column chunks dealt
// round-robin), each combining all parts of its columns in group order, so a unit that many CTAs shared (few units per
// launch, long contexts) is not merged by one block alone.  Which unit a boundary cuts is read from the groups' own notes
// (finding it again from the lengths cost more than the merge).  What bounds it is the chain of loads and the fetch of
// code that runs once: a chunk of a record is 4 KB in one piece, so bulk copies bring everything a block needs at once,
// and the arithmetic runs out of shared memory (17 parts of 85 rows: 15 us with loads in the loop over the parts, 8 with
// eight parts' loads in flight).
// The caller has waited for the records, and lets the kernel behind be launched.
// map(row, GroupBegin) -> false, or the row's node and query head; record(group, slot) -> its record in slot 0 (of the unit
// that began before the group's range) or 1, [column][128 rows], D accumulator columns, then (max, sum).  wait_limit: SM cycles
// after which a wait gives up; stall: test aid, 1 makes the first wait run out (it expects bytes that nobody copies).
template <int D, class Map, class Record>
__device__ __forceinline__ void merge_boundary(const GroupBegin* table, int n_groups, int n, int Hq, int B, __nv_bfloat16* out, float* lse_out,
                                               int* status, long long wait_limit, int stall, Map map, Record record) {
    extern __shared__ __align__(128) float s_cols[];                            // [slot][8 columns][128 rows]
    float(*const s_ml)[2][128] = (float(*)[2][128])(s_cols + kMergeSlots * 8 * 128);     // [part][max, then weight | sum][128 rows]
    __shared__ GroupBegin s_begin[512];
    __shared__ uint64_t s_bar;
    const int tid = threadIdx.x, warp = tid >> 5, g = blockIdx.x + 1;
    if (tid == 0) { ptx::mbar_init(&s_bar, 1); ptx::fence_mbar_init(); }
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
    const int n_blocks = parts - 1, j_blk = g - (ga + 1);
    constexpr int kChunks = D / 8;                                              // 8 output columns, 2 of them a thread quarter's
    const int row = tid & 127, cq = tid >> 7;
    int node = 0, head = 0;
    const bool has_row = map(row, u, node, head);
    const size_t lb = (size_t)u.layer * B + u.b;
    // group ga holds the unit's first tile (its record is in slot 1), the later groups began inside the unit (slot 0)
    const float* const first = record(ga, 1);
    const float* const second = record(ga + 1, 0);
    const size_t stride = record(1, 0) - record(0, 0);
    uint32_t phase = 0;
    // One load: n_ch chunks (c0, c0 + n_blocks, ...) of the parts [k0, k0 + nk), with the parts' (max, sum) unless n_ch < 0 (then
    // only those).  false: the copies did not arrive (reported).
    auto fetch = [&](int k0, int nk, int c0, int n_ch, bool ml) -> bool {
        ptx::fence_proxy_async();          // (the weights that weigh() stored where the copies land)
        __syncthreads();
        if (tid == 0) ptx::mbar_arrive_expect_tx(&s_bar, (uint32_t)(nk * (n_ch * 4096 + (ml ? 1024 : 0)) + 16 * stall));
        __syncthreads();
        for (int i = warp; i < nk * (n_ch + 1); i += kMergeThreads / 32) {
            const int c = i / nk, k = i - c * nk;
            const float* src = k0 + k == 0 ? first : second + (size_t)(k0 + k - 1) * stride;
            if (c == n_ch && !ml) continue;
            src += c == n_ch ? (size_t)D * 128 : (size_t)(c0 + c * n_blocks) * 8 * 128;
            float* const dst = c == n_ch ? &s_ml[k][0][0] : s_cols + (size_t)i * 8 * 128;
            if ((tid & 31) == 0)
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(c == n_ch ? 1024u : 4096u), "r"(ptx::smem_u32(&s_bar)) : "memory");
        }
        const bool ok = ptx::mbar_wait(&s_bar, phase, wait_limit);
        if (!ok) {
            if (atomicCAS(status, 0, MIRROR_DEV_TIMEOUT) == 0) atomicExch(status + 1, 38);
            ptx::mbar_wait(&s_bar, phase, 20000000ll);       // (the block's shared memory is not given back under copies in flight)
        }
        phase ^= 1;
        return __syncthreads_and(ok);
    };
    auto weigh = [&](int nk, float M) {                                         // maxima -> weights
        __syncthreads();
        for (int k = cq; k < nk; k += 4) s_ml[k][0][row] = s_ml[k][0][row] == -INFINITY ? 0.f : exp2f(s_ml[k][0][row] - M);
        __syncthreads();
    };
    const bool one_batch = parts <= kMergeSlots;
    const int n_ch = max(1, kMergeSlots / parts);                               // chunks side by side when the parts are few
    float Mm = -INFINITY;
    if (!one_batch)
        for (int k0 = 0; k0 < parts; k0 += kMergeSlots) {
            const int nk = min(kMergeSlots, parts - k0);
            if (!fetch(k0, nk, 0, 0, true)) return;
            for (int k = 0; k < nk; ++k) Mm = fmaxf(Mm, s_ml[k][0][row]);
        }
#pragma unroll 1
    for (int c0 = j_blk; c0 < kChunks; c0 += n_ch * n_blocks) {
        const int nc = min(n_ch, (kChunks - c0 + n_blocks - 1) / n_blocks);
        float Lm = 0.f, a0 = 0.f, a1 = 0.f;
        if (one_batch) {
            if (!fetch(0, parts, c0, nc, c0 == j_blk)) return;
            if (c0 == j_blk) {
                for (int k = 0; k < parts; ++k) Mm = fmaxf(Mm, s_ml[k][0][row]);
                weigh(parts, Mm);
            }
        }
#pragma unroll 1
        for (int c = 0; c < nc; ++c) {
            Lm = a0 = a1 = 0.f;
#pragma unroll 1
            for (int k0 = 0; k0 < parts; k0 += kMergeSlots) {
                const int nk = min(kMergeSlots, parts - k0);
                if (!one_batch) {
                    if (!fetch(k0, nk, c0, 1, true)) return;
                    weigh(nk, Mm);
                }
                const float* col = s_cols + (size_t)(c * nk * 8 + cq * 2) * 128 + row;
#pragma unroll 4
                for (int k = 0; k < nk; ++k) {
                    const float wgt = s_ml[k][0][row];
                    Lm = fmaf(wgt, s_ml[k][1][row], Lm);
                    a0 = fmaf(wgt, col[k * 1024], a0);
                    a1 = fmaf(wgt, col[k * 1024 + 128], a1);
                }
            }
            const int chunk = c0 + c * n_blocks;
            if (!has_row) continue;
            const float inv = 1.f / Lm;
            *reinterpret_cast<uint32_t*>(out + ((lb * n + node) * (size_t)Hq + head) * D + chunk * 8 + cq * 2) = pack_bf16(a0 * inv, a1 * inv);
            if (lse_out && chunk == 0 && cq == 0) lse_out[(lb * Hq + head) * n + node] = Mm * kAttnLn2 + logf(Lm);
        }
    }
}

}  // namespace attn
#endif
