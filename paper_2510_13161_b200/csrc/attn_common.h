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

}  // namespace attn
#endif
