// LM head for many hidden rows (Eq. 1 over the B * (1 + kappa*gamma) rows of a batched verify step): the same fused
// GEMM + row reductions as lmhead_kernel, issued on CTA PAIRS (tcgen05 cta_group::2).
//
// Why a second kernel: with M >= ~200 rows the LM head stops being a weight stream and becomes a GEMM, and a
// single-CTA 128 x N tile asks the L2 for more bytes per flop than it delivers.  A pair of CTAs (the two SMs of a
// TPC) runs one UMMA of 256 vocabulary rows x N hidden rows per K step: each CTA stages its own 128 weight rows and
// only HALF of the hidden rows, and the tensor cores of both SMs read both halves.  Per K block of 64 a CTA loads
// 16 KB + N/2 * 128 B for 128 * N * 64 * 2 flop: 131 flop/B at N = 256 against 79 flop/B before.
//
// Work unit = (256-row vocabulary tile, row chunk of N <= 256 hidden rows).  Units are dealt to the pairs round-robin
// in the order (tile major, chunk minor), so that at any time the pairs work on a handful of neighbouring tiles and
// the chunks of one tile run on different pairs at the same moment: every weight tile leaves HBM once and the other
// chunks hit it in L2.  Each unit leaves one partial (max, argmax, sum-exp) per hidden row and 128-row half tile;
// lmhead_merge_kernel folds them in a fixed order, so the result does not depend on which pair ran which unit (and a launch that
// runs beside an attention launch hands them out by a counter: kFree).
//
// Per CTA, 6 warps as in lmhead_kernel: warp 0 TMA producer (own W rows + own half of the hidden chunk), warp 1
// TMEM owner; in the pair's leader (cluster rank 0) its elected lane issues the UMMAs for both CTAs; warps 2..5
// epilogue over the CTA's own 128 accumulator lanes.
// Barriers that the other CTA signals: the copies of BOTH CTAs complete their bytes on the leader's `full` barrier
// (the peer's TMA names the leader's barrier; no thread sits in between), the UMMA completion is committed with a
// multicast arrive to `empty` / `acc_full` of both CTAs, and the peer's epilogue warps arrive remotely on the leader's
// `acc_empty`.  Every wait is bounded; both CTAs meet at a cluster barrier before the TMEM is released.
#include <math.h>
#include <stdlib.h>

#include <algorithm>

#include "mirror_internal.h"

namespace {

constexpr int kThreads = 192;
constexpr int kBK = 64;
constexpr int kTileV = 128;                 // vocabulary rows per CTA and unit
constexpr int kPairV = 2 * kTileV;          // per pair
constexpr int kMaxStages = 8;
constexpr int kAcc = 2;
constexpr int kMaxChunkRows = 256;
constexpr int kSmemBudget = 232448;
constexpr int kUnitRing = 16;               // units named ahead (kFree); the producer is at most stages + 3 units ahead of the epilogue
constexpr int kCtrlBytes = 1024 + 4 * kMaxChunkRows * 12;
constexpr int kTopkBytes = 5 * kMaxChunkRows * 4;      // Top-kappa: each epilogue warp's row maxima of one unit, and the rows' bars

struct PairParams {
    int M, V, H;
    int n_chunks, chunk_rows, half_rows;
    int acc_stride, tmem_cols;
    int stages, stage_bytes;
    int rows_cta, a_bytes;                  // vocabulary rows a CTA loads per unit (<= 128, a multiple of 8) and their bytes per stage
    int ctas_per_sm;                        // 2 when few rows leave room for two CTAs' pipelines on an SM
    int k_slices, kb_per_slice;             // split-K (plain GEMM mode only): K blocks of 64 per unit
    int n_units;
    int w_keep;                             // 1: weight tiles are re-read by other chunks, keep them in L2
    float inv_T, inv_T_log2e;
    float* logits_out;                      // reduce mode: nullable [M, V]; plain GEMM mode: [k_slices][M, V] partial sums
    float* part_max;                        // [partials][M]
    int* part_idx;
    float* part_sum;
    int* status;
    int topk;                               // > 0: the epilogue collects candidates for each row's topk best (logit, id) pairs
    float* part_topv;                       // [4 * CTA + warp][M][topk]: sorted lists
    int* part_topi;
    uint32_t* topk_bar;                     // largest logit seen in each of topk shares of the vocabulary (bar_word; order_key, 0: none, 1: none finite)
    int fp8;                                // 1: W and the hidden rows are e4m3 bytes (K counted in 128-byte blocks all the same)
    const float* w_scale;                   // fp8: [V] scale of each weight row
    const float* h_scale;                   // fp8: [M] scale of each hidden row
    long long wait_limit;                   // SM cycles after which a wait gives up
    int stall_after;                        // test aid: the producers stop after this many stages (-1: never)
    int w_early;                            // 1: W is older than the kernel ahead: the first stages' weights are requested before the wait
    __nv_bfloat16* act;                     // kGated: [M, V / 2]
    int sums;                               // 0: the partials' sums are not read
    int running;                            // 1: a CTA keeps its rows' state over its units and leaves one partial; 0: a partial per unit
    uint32_t* unit_ctr;                     // kFree: {next unit, pairs that are through}; both zero between launches
    int n_own;                              // kFree: the first units, one per pair, that are not handed out by the counter (0 or the pairs)
};

struct Ctrl {
    uint64_t full[kMaxStages];              // leader only: the stage has landed in both CTAs (transaction bytes of both)
    uint64_t empty[kMaxStages];             // UMMAs that read the stage have completed (multicast commit)
    uint64_t acc_full[kAcc];                // accumulator complete (multicast commit)
    uint64_t acc_empty[kAcc];               // leader only: 4 + 4 epilogue warps have drained the accumulator
    uint64_t unit_full[kUnitRing];          // kFree: the leader has named this CTA's unit
    int unit[kUnitRing];
    alignas(16) float bcast[4][32];         // per epilogue warp: a value per column, for all lanes
    int* status;
    long long wait_limit;
    uint32_t tmem_base;
    volatile int abort;
};
static_assert(sizeof(Ctrl) <= 1024, "control block");

__device__ __forceinline__ void fail(const PairParams& p, Ctrl* c, int where) {
    c->abort = 1;
    if (atomicCAS(p.status, 0, MIRROR_DEV_TIMEOUT) == 0) atomicExch(p.status + 1, where);
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {      // every thread of both CTAs
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of the same shared-memory object in the CTA of rank `rank`
__device__ __forceinline__ uint32_t map_to_rank(const void* smem_ptr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(ptx::smem_u32(smem_ptr)), "r"(rank));
    return r;
}
// (Without a scope, that is a release within the CTA, although the waiter acquires at cluster scope: what it hands over is tensor memory,
// whose reads tcgen05.wait::ld and, towards the waiter's UMMAs, tcgen05.fence::before_thread_sync have ordered; no memory that the arriving
// thread wrote goes with it.  A release at cluster scope would hold a unit's end up behind its spilled logits and state; 132 rows x
// 137273 x 768: 82.7 us, without 80.1.)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// a word into the shared memory of a CTA of the pair, counted on a barrier there
__device__ __forceinline__ void st_async(uint32_t cluster_addr, int v, uint32_t bar_cluster_addr) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(cluster_addr), "r"(v), "r"(bar_cluster_addr) : "memory");
}
// Has the phase completed?  (Does not block; try_wait may, for as long as the hardware likes: asked that way for the K block behind the
// one at hand, the issuer held that one back until the other had arrived, and short launches took up to half as long again.)
__device__ __forceinline__ bool poll(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(ptx::smem_u32(bar)), "r"(parity)
        : "memory");
    return __all_sync(0xffffffffu, ok != 0);
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_result, uint32_t ncols) {    // one warp of EACH CTA
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ptx::smem_u32(smem_result)), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {         // one warp of EACH CTA
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// TMA load into this CTA's shared memory whose bytes are counted on a barrier of the pair's leader (cluster address)
__device__ __forceinline__ void tma_load_2d_pair(void* smem_dst, const void* map, uint32_t bar_cluster_addr, int x, int y,
                                                 uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(ptx::smem_u32(smem_dst)), "l"(map), "r"(bar_cluster_addr), "r"(x), "r"(y), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d_pair(void* smem_dst, const void* map, uint32_t bar_cluster_addr, int x, int y, int z, int w, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
        ::"r"(ptx::smem_u32(smem_dst)), "l"(map), "r"(bar_cluster_addr), "r"(x), "r"(y), "r"(z), "r"(w), "l"(policy)
        : "memory");
}
// D[tmem of both CTAs] (+)= A (128 rows from each CTA's shared memory) * B (N/2 rows from each CTA's shared memory); the low words of
// the two descriptors, which share the high one
__device__ __forceinline__ void umma_pair_f16(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
// the same for e4m3 operands (32 elements of K per instruction: the same 32 bytes of a 128-byte swizzled row)
__device__ __forceinline__ void umma_pair_f8(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], da, db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
// instruction descriptor for e4m3 x e4m3 -> fp32, both operands K-major
__host__ __device__ __forceinline__ uint32_t umma_idesc_e4m3(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// arrive on the barrier at this shared-memory offset in BOTH CTAs once all UMMAs issued so far have completed
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(ptx::smem_u32(bar)), "h"((uint16_t)3)
                 : "memory");
}

// Fused Top-kappa (Eq. 6).  Every epilogue warp has, for every hidden row, a sorted list of K (logit, id) pairs in global
// memory (order: logit descending, id ascending); lmhead_topk_merge_kernel merges the lists of a row.  A list alone would
// be a poor filter (a warp meets only ~150 of a row's logits), so the CTAs share a bar: the vocabulary falls into K shares
// by the CTA that meets it, the largest logit met so far in each share is kept in global memory (atomicMax, one per CTA
// and row and only when it grows: one per warp and unit on neighbouring words queued for 50 us), and the smallest of those
// K maxima is at most the row's K-th best logit, since K different ids attain it.  A row whose maximum in a unit -- which
// the reduction has anyway -- is below the bar is done with one comparison; after the first unit that is nearly every
// row.  (What a list holds depends on timing, which candidates are best does not.)
__device__ __forceinline__ size_t bar_word(int share, int row) { return ((size_t)share * kMaxChunkRows + row) * 8; }    // (a sector each)
// Insertion by a whole warp: lane i has the list's i-th pair.
__device__ __forceinline__ void topk_list_insert(float* lv, int* li, int K, float x, int xi) {
    const int lane = threadIdx.x & 31;
    const float v = lane < K ? __ldcg(lv + lane) : INFINITY;
    const int i = lane < K ? __ldcg(li + lane) : -1;
    const unsigned behind = __ballot_sync(0xffffffffu, lane < K && (x > v || (x == v && xi < i)));   // pairs that x goes in front of
    const float pv = __shfl_up_sync(0xffffffffu, v, 1);
    const int pi = __shfl_up_sync(0xffffffffu, i, 1);
    if ((behind >> lane) & 1u) {
        const bool first = lane == __ffs(behind) - 1;
        __stcg(lv + lane, first ? x : pv);
        __stcg(li + lane, first ? xi : pi);
    }
    __syncwarp();
}

// The 32 pairs of a warp, one per lane, best first (bitonic network; `merge`: the input is bitonic already).
__device__ __forceinline__ void warp_sort_pairs(float& v, int& i, bool merge = false) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
        if (merge && k < 32) continue;
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, v, j);
            const int oi = __shfl_xor_sync(0xffffffffu, i, j);
            const bool mine_better = v > ov || (v == ov && i < oi);
            const bool keep_better = ((lane & j) == 0) == ((lane & k) == 0);
            if (mine_better != keep_better) { v = ov; i = oi; }
        }
    }
}
// A list and up to 32 candidates (lane: x, xi; -inf for none) at once: what the first units bring, before there is a bar.
// empty: the list holds nothing yet.
__device__ __noinline__ void topk_list_merge(float* lv, int* li, int K, float x, int xi, bool empty) {
    const int lane = threadIdx.x & 31;
    warp_sort_pairs(x, xi);
    if (!empty) {
        const float rv = __shfl_sync(0xffffffffu, x, 31 - lane);
        const int ri = __shfl_sync(0xffffffffu, xi, 31 - lane);
        x = lane < K ? __ldcg(lv + lane) : -INFINITY;
        xi = lane < K ? __ldcg(li + lane) : 0x7fffffff;
        if (rv > x || (rv == x && ri < xi)) { x = rv; xi = ri; }          // best 32 of both, as a bitonic sequence
        warp_sort_pairs(x, xi, true);
    }
    if (lane < K) { __stcg(lv + lane, x); __stcg(li + lane, xi); }
    __syncwarp();
}

// The reduction of column j over the 32 lanes, for all columns at once, into lane j: at every step a lane gives away the half of its
// columns that its partner keeps.  The tree is that of a butterfly per column, with a fifth of its shuffles.
template <class Op>
__device__ __forceinline__ float reduce_columns(float (&v)[32], Op op) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const float keep = up ? v[k + o] : v[k], give = up ? v[k] : v[k + o];
            v[k] = op(keep, __shfl_xor_sync(0xffffffffu, give, o));
        }
    }
    return v[0];
}
// f(j, lane j's x) for all j
template <class F>
__device__ __forceinline__ void for_lanes(float* bcast, float x, F f) {
    __syncwarp();                                             // (the words' last readers)
    bcast[threadIdx.x & 31] = x;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        const float4 b = *reinterpret_cast<const float4*>(bcast + j);
        f(j, b.x); f(j + 1, b.y); f(j + 2, b.z); f(j + 3, b.w);
    }
}

// kReduce: LM head (row reductions in the epilogue, optional spill).  !kReduce: plain GEMM C = W h^T for the layer
// projections, split along K when there are fewer tiles than CTA pairs; the epilogue only stores fp32 partial sums.
// kFp8 / kTopk: e4m3 operands with per-row scales / Top-kappa lists in the epilogue, as separate instantiations so that
// the plain bf16 head carries none of their registers and branches.
// kEarly: a kernel of its own, since the few instructions that it adds in front of the wait cost the others up to 6%.
// kFree: nothing that this launch reads is written by the kernel ahead (an attention launch, which has waited for all before it), so
// its CTAs begin as SMs come free, and only their end waits.  They begin at very different times, so the pairs take units from
// a counter: the leader's producer names them to both CTAs.  Results do not depend on who takes what: argmax does not, and
// where sums are asked for every unit leaves partials of its own.
// kGated: plain GEMM of a gate and an up projection (the rows [0, I) and [I, 2I) of W) whose epilogue leaves bf16(silu(gate) * up).  A
// warp's 32 accumulator lanes are 16 gate rows and the 16 up rows that go with them (a fourth dimension of W's tensor map deals
// them so), and lanes 16 apart exchange half of their columns.
template <bool kReduce, bool kFp8, bool kTopk, bool kEarly, bool kFree, bool kGated>
__device__ __forceinline__ void pair_gemm_body(const CUtensorMap& tm_w, const CUtensorMap& tm_h, const PairParams& p) {
    extern __shared__ uint8_t smem_raw[];
    // (the dynamic shared window starts at the same offset in both CTAs, so the aligned layout is the same too)
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* stage_base = smem;
    Ctrl* ctrl = (Ctrl*)(smem + (size_t)p.stages * p.stage_bytes);
    float* st_max = (float*)((uint8_t*)ctrl + 1024);          // [4][kMaxChunkRows]
    int* st_idx = (int*)(st_max + 4 * kMaxChunkRows);
    float* st_sum = (float*)(st_idx + 4 * kMaxChunkRows);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const int n_kb = p.H / kBK;
    // unit -> (vocabulary tile, K slice, row chunk); chunk fastest, so the chunks of a tile run side by side
    auto decode = [&](int u, int& tile, int& slice, int& chunk) {
        chunk = u % p.n_chunks;
        const int t2 = u / p.n_chunks;
        slice = t2 % p.k_slices;
        tile = t2 / p.k_slices;
    };

    auto load_w = [&](uint8_t* dst, uint32_t bar, int kb, int tile, uint64_t policy) {
        if (kGated) tma_load_4d_pair(dst, &tm_w, bar, kb * kBK, 0, 0, (tile * 2 + (int)rank) * (kTileV / 32), policy);
        else tma_load_2d_pair(dst, &tm_w, bar, kb * kBK, (tile * 2 + (int)rank) * p.rows_cta, policy);
    };

    if (tid == 0) {
        for (int s = 0; s < p.stages; ++s) {
            ptx::mbar_init(&ctrl->full[s], 1);
            ptx::mbar_init(&ctrl->empty[s], 1);
        }
        for (int a = 0; a < kAcc; ++a) { ptx::mbar_init(&ctrl->acc_full[a], 1); ptx::mbar_init(&ctrl->acc_empty[a], 8); }
        if (kFree)
            for (int i = 0; i < kUnitRing; ++i) ptx::mbar_init(&ctrl->unit_full[i], 1);
        ctrl->abort = 0;
        ctrl->status = p.status;
        ctrl->wait_limit = p.wait_limit;
        ptx::fence_mbar_init();
        ptx::prefetch_tmap(&tm_w);
        ptx::prefetch_tmap(&tm_h);
    }
    if (warp == 1) {
        tmem_alloc_pair(&ctrl->tmem_base, (uint32_t)p.tmem_cols);
        tmem_relinquish_pair();
    }
    ptx::tc_fence_before();
    __syncthreads();
    cluster_sync_all();                 // the other CTA's barriers exist before anything arrives on them
    ptx::tc_fence_after();
    const uint32_t tmem_base = ctrl->tmem_base;
    // The weights of the first stages, while the kernel ahead is still at work (their rows of x follow behind the wait).
    int n_early = 0;
    if (kEarly && p.w_early && warp == 0 && pair < p.n_units) {
        int tile, slice, chunk;
        decode(pair, tile, slice, chunk);
        const int kb0 = slice * p.kb_per_slice;
        n_early = min(p.stages, min(n_kb, kb0 + p.kb_per_slice) - kb0);
        const uint64_t pol_w = p.w_keep ? ptx::policy_evict_normal() : ptx::policy_evict_first();
        for (int s = 0; s < n_early && lane == 0; ++s) {
            if (rank == 0) ptx::mbar_arrive_expect_tx(&ctrl->full[s], 2u * (uint32_t)p.stage_bytes);
            load_w(stage_base + s * p.stage_bytes, map_to_rank(&ctrl->full[s], 0), kb0 + s, tile, pol_w);
        }
    }
    if (!kFree) ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    // kFree: unit number j of this pair, or (no more, or a failure) one past the last; whole warps
    auto named_unit = [&](uint32_t j) -> int {
        const uint32_t e = j % kUnitRing;
        if (!ptx::warp_wait<true>(ctrl, &ctrl->unit_full[e], (j / kUnitRing) & 1, 17)) return p.n_units;
        return *(volatile int*)&ctrl->unit[e];
    };

    // Producer and issuer: the whole warp walks the schedule and one elected lane issues, which keeps addresses and descriptors in
    // uniform registers; the next K block's barrier is polled ahead of the instructions that hold the lane up.  What the issuer spends
    // on a K block is the pace of a pair that its memory could feed faster, and of the tensor cores: with all of it in one lane 600 cycles
    // (four UMMAs 280, a wait that need not wait 114, the commit 58), whatever the rows.  16 pairs alone, 2 x 64 rows each of 10 KB: 52 ->
    // 108 GB/s per SM; LM head of 152064 x 5120 at 196 / 392 / 520 rows 334 / 594 / 849 -> 289 / 511 / 669 us.
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        const uint64_t pol_w = p.w_keep ? ptx::policy_evict_normal() : ptx::policy_evict_first();
        const uint64_t pol_h = ptx::policy_evict_last();
        const uint32_t full0 = map_to_rank(&ctrl->full[0], 0);
        int s = 0, n_issued = 0;
        uint32_t ph = 0;
        bool ok = true;
        // the rows of x that belong to the weights requested early.  (A loop of its own: a test per K block in the main loop
        // made 275 rows x 42306 x 2304 take 110 instead of 102 us.)
        for (; kEarly && n_issued < n_early && ok; ++n_issued) {
            if (p.stall_after >= 0 && n_issued >= p.stall_after) { ok = false; break; }           // (test aid, as below)
            int tile, slice, chunk;
            decode(pair, tile, slice, chunk);
            if (ptx::elect_one())
                tma_load_2d_pair(stage_base + s * p.stage_bytes + p.a_bytes, &tm_h, full0 + s * 8, (slice * p.kb_per_slice + n_issued) * kBK,
                                 chunk * p.chunk_rows + (int)rank * p.half_rows, pol_h);
            if (++s == p.stages) { s = 0; ph ^= 1; }
        }
        int kb_skip = n_issued;
        auto name_unit = [&](uint32_t j) {                         // (the leader's)
            if (ptx::elect_one()) {
                int u = p.n_units;                                 // (as many pairs as units: no need to ask)
                if (j == 0 && p.n_own > 0) u = pair;
                else if (p.n_own < p.n_units) u = (int)min(p.n_own + atomicAdd(p.unit_ctr, 1u), (uint32_t)p.n_units);
                for (uint32_t r = 0; r < 2; ++r) st_async(map_to_rank(&ctrl->unit[j % kUnitRing], r), u, map_to_rank(&ctrl->unit_full[j % kUnitRing], r));
            }
            __syncwarp();
        };
        auto take_unit = [&](uint32_t j) {
            if (ptx::elect_one()) ptx::mbar_arrive_expect_tx(&ctrl->unit_full[j % kUnitRing], 4);
            __syncwarp();
            return named_unit(j);
        };
        uint32_t j = 0;
        if (kFree && rank == 0) name_unit(0);
        for (int u = kFree ? take_unit(0) : pair; u < p.n_units && ok; u = kFree ? take_unit(++j) : u + n_pairs) {
            int tile, slice, chunk;
            decode(u, tile, slice, chunk);
            const int h_row = chunk * p.chunk_rows + (int)rank * p.half_rows;
            const int kb_end = min(n_kb, (slice + 1) * p.kb_per_slice);
            int kb = slice * p.kb_per_slice + kb_skip;
            kb_skip = 0;
            const int kb_name = min(kb + p.stages, kb_end) - 1;    // (the counter's answer takes ~1 us: asked for with all stages in flight)
#pragma unroll 1
            for (; kb < kb_end; ++kb) {
                if (p.stall_after >= 0 && n_issued >= p.stall_after) { ok = false; break; }       // (test aid: neither arms nor copies)
                if (!ptx::warp_wait(ctrl, &ctrl->empty[s], ph ^ 1, 11)) { ok = false; break; }
                if (ptx::elect_one()) {
                    if (rank == 0) ptx::mbar_arrive_expect_tx(&ctrl->full[s], 2u * (uint32_t)p.stage_bytes);
                    uint8_t* dst = stage_base + s * p.stage_bytes;
                    load_w(dst, full0 + s * 8, kb, tile, pol_w);
                    tma_load_2d_pair(dst + p.a_bytes, &tm_h, full0 + s * 8, kb * kBK, h_row, pol_h);
                }
                __syncwarp();
                ++n_issued;
                if (++s == p.stages) { s = 0; ph ^= 1; }
                if (kFree && rank == 0 && kb == kb_name) name_unit(j + 1);
            }
        }
        // (copies still in flight after a failure: the leader's issuer or its 2 s limit outlasts them, and both CTAs
        // meet at the cluster barrier below before either one's shared memory goes away)
    } else if (warp == 1) {
        if (rank == 0) {
            // -------------------------------------------------------------- UMMA issuer (leader)
            const uint32_t idesc = kFp8 ? umma_idesc_e4m3(kPairV, p.chunk_rows) : ptx::umma_idesc_bf16(kPairV, p.chunk_rows);
            const uint32_t hi = ptx::umma_desc_hi_sw128(1024), lo0 = ptx::umma_desc_lo(ptx::smem_u32(stage_base), 16);
            const uint32_t stage_lo = (uint32_t)p.stage_bytes >> 4, a_lo = (uint32_t)p.a_bytes >> 4;
            int s = 0, ab = 0;
            uint32_t ph = 0, aph = 0, lo = lo0;
            bool ok = true;
            uint32_t j = 0;
            for (int u = kFree ? named_unit(0) : pair; u < p.n_units && ok; u = kFree ? named_unit(++j) : u + n_pairs) {
                if (!ptx::warp_wait<true>(ctrl, &ctrl->acc_empty[ab], aph ^ 1, 12)) { ok = false; break; }
                const uint32_t d_tmem = tmem_base + (uint32_t)(ab * p.acc_stride);
                int tile, slice, chunk;
                decode(u, tile, slice, chunk);
                const int nk = min(n_kb, (slice + 1) * p.kb_per_slice) - slice * p.kb_per_slice;
                bool ready = poll(&ctrl->full[s], ph);
#pragma unroll 1
                for (int kb = 0; kb < nk; ++kb) {
                    if (!ready && !ptx::warp_wait_slow<false>(ctrl, &ctrl->full[s], ph, 13)) { ok = false; break; }
                    ptx::tc_fence_after();
                    uint64_t* const done = &ctrl->empty[s];
                    const uint32_t a = lo;
                    lo += stage_lo;
                    if (++s == p.stages) { s = 0; ph ^= 1; lo = lo0; }
                    ready = poll(&ctrl->full[s], ph);              // (the next K block's; of no use behind the last one of all)
                    if (ptx::elect_one()) {
#pragma unroll
                        for (int k4 = 0; k4 < kBK / 16; ++k4) {
                            if (kFp8) umma_pair_f8(d_tmem, a + k4 * 2, a + a_lo + k4 * 2, hi, idesc, (kb | k4) != 0);
                            else umma_pair_f16(d_tmem, a + k4 * 2, a + a_lo + k4 * 2, hi, idesc, (kb | k4) != 0);
                        }
                        umma_commit_pair(done);
                        if (kb + 1 == nk) umma_commit_pair(&ctrl->acc_full[ab]);
                    }
                    __syncwarp();
                }
                if (++ab == kAcc) { ab = 0; aph ^= 1; }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (both CTAs, own 128 lanes)
        const int q = warp & 3;
        float* my_max = st_max + q * kMaxChunkRows;
        int* my_idx = st_idx + q * kMaxChunkRows;
        float* my_sum = st_sum + q * kMaxChunkRows;
        float* const unit_max = kTopk ? (float*)((uint8_t*)ctrl + kCtrlBytes) + q * kMaxChunkRows : nullptr;    // this unit's maxima
        const int n_cg = (p.chunk_rows + 31) / 32;
        // the four warps hold disjoint vocabulary rows: one partial per hidden row out of their four states
        auto flush = [&](size_t pbase, int rbase) {
            for (int c = (warp - 2) * 32 + lane; c < p.chunk_rows; c += 128) {
                const int row = rbase + c;
                if (row >= p.M) continue;
                float m = -INFINITY, s = 0.f;
                int idx = 0x7fffffff;
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const float pm = st_max[w * kMaxChunkRows + c], ps = st_sum[w * kMaxChunkRows + c];
                    const int pi = st_idx[w * kMaxChunkRows + c];
                    if (pm == -INFINITY) continue;
                    if (pm > m || (pm == m && pi < idx)) {
                        s = ps + (m == -INFINITY ? 0.f : s * exp2f((m - pm) * p.inv_T_log2e));
                        m = pm; idx = pi;
                    } else {
                        s += ps * exp2f((pm - m) * p.inv_T_log2e);
                    }
                }
                p.part_max[pbase + row] = m;
                p.part_idx[pbase + row] = idx;
                p.part_sum[pbase + row] = s;
            }
        };
        // this warp's Top-kappa lists: [M][topk] (one row chunk, so the CTA meets all rows in every unit)
        float* const my_tv = kTopk ? p.part_topv + ((size_t)blockIdx.x * 4 + q) * p.M * p.topk : nullptr;
        int* const my_ti = kTopk ? p.part_topi + ((size_t)blockIdx.x * 4 + q) * p.M * p.topk : nullptr;
        int ab = 0;
        uint32_t aph = 0;
        bool ok = true;
        // One row chunk: a CTA meets the same hidden rows in every unit and keeps a running state per row, flushed once
        // (one partial per CTA).  Several chunks: every unit flushes its own partial (one per 128-row vocabulary tile).
        const bool running = kFree ? p.running != 0 : p.n_chunks == 1;
        if (kReduce && running) {
            for (int c = lane; c < kMaxChunkRows; c += 32) { my_max[c] = -INFINITY; my_idx[c] = 0x7fffffff; my_sum[c] = 0.f; }
            __syncwarp();
        }
        if constexpr (kReduce && kTopk) {
            for (int i = lane; i < p.M * p.topk; i += 32) { __stcg(my_tv + i, -INFINITY); __stcg(my_ti + i, 0x7fffffff); }      // empty
            __syncwarp();
        }
        uint32_t j = 0;
        // (a partial per unit: the four warps meet at barriers, so all of them go on or none)
        auto next_unit = [&](uint32_t i) -> int {
            const int u = ctrl->abort ? p.n_units : named_unit(i);
            if (running) return u;
            uint32_t go;
            asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                         : "=r"(go) : "r"((uint32_t)(u < p.n_units)) : "memory");
            return go ? u : p.n_units;
        };
        for (int u = kFree ? next_unit(0) : pair; u < p.n_units; u = kFree ? next_unit(++j) : u + n_pairs) {
            int tile, slice, chunk;
            decode(u, tile, slice, chunk);
            const int rbase = chunk * p.chunk_rows;
            const int vt = tile * 2 + (int)rank;                 // 128-row vocabulary tile of this CTA
            if (ok && (ctrl->abort || !ptx::mbar_wait(&ctrl->acc_full[ab], aph, p.wait_limit))) { fail(p, ctrl, 16); ok = false; }
            if (ok) {
                ptx::tc_fence_after();
                // (a unit of fewer than 128 rows per CTA leaves stale shared memory in the accumulator lanes beyond them)
                const int vid = vt * p.rows_cta + q * 32 + lane;
                const bool valid = q * 32 + lane < p.rows_cta && vid < p.V;
                const bool any_valid = __ballot_sync(0xffffffffu, valid) != 0;          // warp-uniform
                const int n_rows = min(p.chunk_rows, p.M - rbase);                       // hidden rows of this chunk
                const float sw = (kFp8 && valid) ? p.w_scale[vid] : 1.f;                 // fp8: this lane's weight-row scale
                for (int cg = 0; cg < n_cg; ++cg) {
                    uint32_t r[32];
                    ptx::tmem_ld_32x32b_x32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * p.acc_stride + cg * 32), r);
                    ptx::tmem_ld_wait();
                    float upd_m = -INFINITY, upd_s = 0.f;
                    int upd_i = 0x7fffffff;
                    const int ncol = n_rows - cg * 32;       // columns of this group that are hidden rows (the rest hold zeros)
                    if constexpr (kGated) {
                        const bool lo = lane < 16;
                        const int I = p.V >> 1, col = (vt * 4 + q) * 16 + (lane & 15), c0 = cg * 32 + (lo ? 0 : 16);
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const float mine = __uint_as_float(lo ? r[k] : r[k + 16]), other = __shfl_xor_sync(0xffffffffu, __uint_as_float(lo ? r[k + 16] : r[k]), 16);
                            const float gate = 0.f + (lo ? mine : other), up = 0.f + (lo ? other : mine);       // (the sum of one slice)
                            if (c0 + k < n_rows && col < I) p.act[(size_t)(rbase + c0 + k) * I + col] = __float2bfloat16_rn(gate / (1.0f + expf(-gate)) * up);
                        }
                    } else if (any_valid && ncol > 0) {
                        // The 32 columns go through the reductions side by side; lane j ends with the result of column j.  (A butterfly per
                        // column set the pace of short rows: 320 shuffles per warp and 32 columns, now 62 and two passes through shared memory.)
                        float v[32];
                        if constexpr (kFp8) {
                            // logit = (sum of e4m3 products) * weight-row scale * hidden-row scale; lane j fetches column j's scale
                            const int cr = rbase + cg * 32 + lane;
                            for_lanes(ctrl->bcast[q], cr < p.M ? p.h_scale[cr] : 0.f, [&](int j, float sh) { r[j] = __float_as_uint(__uint_as_float(r[j]) * (sw * sh)); });
                        }
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = valid ? __uint_as_float(r[j]) : -INFINITY;
                        if (p.logits_out && valid) {
                            float* dst = p.logits_out + ((size_t)slice * p.M + rbase + cg * 32) * p.V + vid;
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (j < ncol) dst[(size_t)j * p.V] = v[j];
                        }
                        if (kReduce) {
                            float t[32];
#pragma unroll
                            for (int j = 0; j < 32; ++j) t[j] = v[j];
                            upd_m = reduce_columns(t, [](float a, float b) { return fmaxf(a, b); });
                            unsigned at_max = 0;
                            for_lanes(ctrl->bcast[q], upd_m, [&](int j, float m) {
                                const unsigned eq = __ballot_sync(0xffffffffu, v[j] == m);
                                if (lane == j) at_max = eq;
                                v[j] -= m;
                            });
                            upd_i = vid - lane + (__ffs(at_max) - 1);
                            if (p.sums) {
#pragma unroll
                                for (int j = 0; j < 32; ++j) v[j] = ptx::ex2_approx(v[j] * p.inv_T_log2e);      // (below 2^-126: 0 beside the maximum's 1)
                                upd_s = reduce_columns(v, [](float a, float b) { return a + b; });
                            }
                        }
                    }
                    const int c = cg * 32 + lane;          // lane j holds column cg*32+j of this unit
                    if constexpr (kTopk) unit_max[c] = upd_m;
                    if (!kReduce) {
                    } else if (!running) {
                        my_max[c] = upd_m; my_idx[c] = upd_i; my_sum[c] = upd_s;
                    } else if (upd_m != -INFINITY) {
                        const float om = my_max[c], os = my_sum[c];
                        if (upd_m > om) {           // ids only grow along a CTA's units: equality keeps the older, lower id
                            my_sum[c] = upd_s + (om == -INFINITY ? 0.f : os * exp2f((om - upd_m) * p.inv_T_log2e));
                            my_max[c] = upd_m;
                            my_idx[c] = upd_i;
                        } else {
                            my_sum[c] = os + upd_s * exp2f((upd_m - om) * p.inv_T_log2e);
                        }
                    }
                }
                if constexpr (!kTopk) {
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(map_to_rank(&ctrl->acc_empty[ab], 0));
                }
            }
            if constexpr (kReduce && kTopk) {
                // (all four warps meet here whatever happened to one of them)
                const int K = p.topk, n_rows = min(p.chunk_rows, p.M - rbase);
                float* const all_max = (float*)((uint8_t*)ctrl + kCtrlBytes);
                uint32_t* const bars = (uint32_t*)(all_max + 4 * kMaxChunkRows);
                asm volatile("bar.sync 1, 128;" ::: "memory");
                // (a row without a finite logit, an input's NaN, counts as met at the lowest key; a CTA beyond the vocabulary has met nothing)
                const int share = (int)(blockIdx.x % (uint32_t)K);
                const uint32_t seen = vt * p.rows_cta < p.V ? 1u : 0u;
                for (int c = (warp - 2) * 32 + lane; ok && c < n_rows; c += 128) {
                    uint32_t key = seen;
                    for (int w = 0; w < 4; ++w) {
                        const float m = all_max[w * kMaxChunkRows + c];
                        if (m > -INFINITY) key = max(key, mirror_order_key(m));
                    }
                    if (key > __ldcg(p.topk_bar + bar_word(share, c))) atomicMax(p.topk_bar + bar_word(share, c), key);
                }
                // The first unit's logits would all pass a bar that does not exist yet, and cost their warps a sort per row (1.2 us a row in
                // all).  The other CTAs are at their first unit too: until each share has a word it is worth waiting, for as long as
                // those sorts would take at most (no one has to arrive: a share that stays empty lets everything pass), if there is
                // a CTA with vocabulary for each share.
                const bool first = u == pair && min((int)gridDim.x, (p.V + p.rows_cta - 1) / p.rows_cta) >= K;
                const long long t0 = clock64(), limit = 2000ll * n_rows;
                for (int c = (warp - 2) * 32 + lane; c < n_rows; c += 128) {
                    uint32_t bar;
                    do {
                        bar = 0xffffffffu;
#pragma unroll 4
                        for (int k = 0; k < K; ++k) bar = min(bar, __ldcg(p.topk_bar + bar_word(k, c)));
                    } while (bar == 0 && first && clock64() - t0 < limit);
                    bars[c] = bar;
                }
                asm volatile("bar.sync 1, 128;" ::: "memory");
                const int vid = vt * p.rows_cta + q * 32 + lane;
                const bool valid = q * 32 + lane < p.rows_cta && vid < p.V;
                for (int cg = 0; ok && cg < n_cg; ++cg) {
                    const int c = cg * 32 + lane;
                    unsigned cols = __ballot_sync(0xffffffffu, c < n_rows && unit_max[c] > -INFINITY && mirror_order_key(unit_max[c]) >= bars[c]);
                    while (cols) {
                        const int j = __ffs(cols) - 1;
                        cols &= cols - 1;
                        uint32_t w;
                        asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(w)
                                     : "r"(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * p.acc_stride + cg * 32 + j)) : "memory");
                        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(w) :: "memory");
                        const float x = valid ? __uint_as_float(w) : -INFINITY;
                        unsigned hit = __ballot_sync(0xffffffffu, x > -INFINITY && mirror_order_key(x) >= bars[cg * 32 + j]);
                        float* const lv = my_tv + (size_t)(cg * 32 + j) * K;
                        int* const li = my_ti + (size_t)(cg * 32 + j) * K;
                        if (__popc(hit) > 2) {
                            const bool in = (hit >> lane) & 1u;
                            topk_list_merge(lv, li, K, in ? x : -INFINITY, in ? vid : 0x7fffffff, u == pair);
                            continue;
                        }
                        while (hit) {
                            const int src = __ffs(hit) - 1;
                            hit &= hit - 1;
                            topk_list_insert(lv, li, K, __shfl_sync(0xffffffffu, x, src), vid - lane + src);
                        }
                    }
                }
            }
            if (kTopk && ok) {
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_rank(&ctrl->acc_empty[ab], 0));
            }
            if (++ab == kAcc) { ab = 0; aph ^= 1; }
            if (kReduce && !running) {
                // fold the four warps' results (disjoint vocabulary rows) into one partial per hidden row
                asm volatile("bar.sync 1, 128;" ::: "memory");
                if (ok && !ctrl->abort) flush((size_t)vt * p.M, rbase);
                asm volatile("bar.sync 1, 128;" ::: "memory");
            }
        }
        if (kReduce && running) {
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (ok && !ctrl->abort) flush((size_t)blockIdx.x * p.M, 0);
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    cluster_sync_all();                 // no remote arrive or multicast commit is in flight towards a CTA that has left
    if (warp == 1) {
        ptx::tc_fence_after();
        tmem_dealloc_pair(tmem_base, (uint32_t)p.tmem_cols);
    }
    if (kFree) {
        if (p.n_own < p.n_units && rank == 0 && tid == 0) {        // the last pair leaves the counter as it found it
            __threadfence();
            if (atomicAdd(p.unit_ctr + 1, 1u) + 1 == (uint32_t)n_pairs) p.unit_ctr[0] = p.unit_ctr[1] = 0;
        }
        ptx::grid_dep_wait();               // (whatever waits for this launch waits for the one ahead, too)
    }
}

__global__ void __launch_bounds__(kThreads, 2)
lmhead_pair_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_h, const PairParams p) {
    pair_gemm_body<true, false, false, false, false, false>(tm_w, tm_h, p);
}
__global__ void __launch_bounds__(kThreads, 2)
lmhead_pair_early_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_h, const PairParams p) {
    pair_gemm_body<true, false, false, true, false, false>(tm_w, tm_h, p);
}
__global__ void __launch_bounds__(kThreads, 2)
lmhead_pair_free_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_h, const PairParams p) {
    pair_gemm_body<true, false, false, false, true, false>(tm_w, tm_h, p);
}
__global__ void __launch_bounds__(kThreads, 2)
lmhead_pair_topk_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_h, const PairParams p) {
    pair_gemm_body<true, false, true, false, false, false>(tm_w, tm_h, p);
}
__global__ void __launch_bounds__(kThreads, 2)
lmhead_pair_fp8_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_h, const PairParams p) {
    pair_gemm_body<true, true, false, false, false, false>(tm_w, tm_h, p);
}
__global__ void __launch_bounds__(kThreads, 2)
linear_pair_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_h, const PairParams p) {
    pair_gemm_body<false, false, false, true, false, false>(tm_w, tm_h, p);
}

__global__ void __launch_bounds__(kThreads, 2)
linear_gated_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_h, const PairParams p) {
    pair_gemm_body<false, false, false, true, false, true>(tm_w, tm_h, p);
}

int next_pow2(int x) {
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

int ctas_per_sm_for(const MirrorTuning& tune, int M) {
    const int max_rows = tune.lm_pair2_max_rows;      // up to this many rows two CTAs share an SM (<= 256 TMEM columns and >= 4 stages each)
    int c = M <= max_rows ? 2 : 1;
    if (tune.lm_ctas_per_sm == 1 || (tune.lm_ctas_per_sm == 2 && M <= max_rows)) c = tune.lm_ctas_per_sm;
    return c;
}

// shapes shared by both modes: row chunks, accumulator layout, pipeline depth
mirror_status pair_shape(const MirrorTuning& tune, int M, int V, int H, PairParams* p, int rows_cta = kTileV, int topk = 0) {
    if (M <= 0 || V <= 0 || H <= 0 || H % kBK != 0) return MIRROR_ERR_SHAPE;
    p->M = M; p->V = V; p->H = H;
    p->n_chunks = (M + kMaxChunkRows - 1) / kMaxChunkRows;
    p->chunk_rows = (int)align_up((size_t)((M + p->n_chunks - 1) / p->n_chunks), 16);
    p->half_rows = p->chunk_rows / 2;
    p->acc_stride = next_pow2(p->chunk_rows < 32 ? 32 : p->chunk_rows);
    p->tmem_cols = kAcc * p->acc_stride;
    p->rows_cta = rows_cta;
    p->a_bytes = rows_cta * kBK * 2;
    p->stage_bytes = p->a_bytes + p->half_rows * kBK * 2;
    // Few rows (a weight stream): two CTAs per SM with five or six stages each keep more bytes in flight than one CTA with
    // eight, deal the units to twice as many pairs, and let the CTAs of the next kernel move in one by one.
    p->ctas_per_sm = ctas_per_sm_for(tune, M);
    p->topk = topk;
    p->part_topv = nullptr; p->part_topi = nullptr; p->topk_bar = nullptr;
    p->stages = (kSmemBudget / p->ctas_per_sm - kCtrlBytes - 2048 - (topk > 0 ? kTopkBytes : 0)) / p->stage_bytes;
    if (p->stages > kMaxStages) p->stages = kMaxStages;
    if (tune.lm_stages >= 2 && tune.lm_stages < p->stages) p->stages = tune.lm_stages;
    p->wait_limit = tune.wait_limit_cycles;
    p->stall_after = -1;
    p->w_early = 0;
    p->running = p->n_chunks == 1;
    p->sums = 1;
    p->unit_ctr = nullptr;
    p->n_own = 0;
    p->act = nullptr;
    if (p->stages < 2) return MIRROR_ERR_SHAPE;
    p->k_slices = 1;
    p->kb_per_slice = H / kBK;
    p->inv_T = p->inv_T_log2e = 1.f;
    p->logits_out = nullptr;
    p->fp8 = 0; p->w_scale = nullptr; p->h_scale = nullptr;
    p->part_max = nullptr; p->part_idx = nullptr; p->part_sum = nullptr;
    return MIRROR_OK;
}

mirror_status pair_launch(mirror_ctx* ctx, bool reduce, const void* x, const void* W, PairParams& p, int n_pairs, cudaStream_t stream) {
    CUtensorMap tm_w, tm_h;
    {
        const uint64_t dims[2] = {(uint64_t)p.H, (uint64_t)p.V};
        const uint64_t strides[1] = {(uint64_t)p.H * 2};
        const uint32_t box_w[2] = {kBK, (uint32_t)p.rows_cta};
        // gate and up rows: (H columns, 16 rows, gate or up, groups of 16 rows)
        const uint64_t half = (uint64_t)p.V / 2, gdims[4] = {(uint64_t)p.H, 16, 2, half / 16};
        const uint64_t gstrides[3] = {(uint64_t)p.H * 2, half * p.H * 2, 16 * (uint64_t)p.H * 2};
        const uint32_t gbox[4] = {kBK, 16, 2, kTileV / 32};
        mirror_status st = p.act ? mirror_make_tmap(ctx, &tm_w, W, 4, gdims, gstrides, gbox) : mirror_make_tmap(ctx, &tm_w, W, 2, dims, strides, box_w);
        if (st != MIRROR_OK) return st;
        const uint64_t hdims[2] = {(uint64_t)p.H, (uint64_t)p.M};
        const uint32_t box_h[2] = {kBK, (uint32_t)p.half_rows};
        st = mirror_make_tmap(ctx, &tm_h, x, 2, hdims, strides, box_h);
        if (st != MIRROR_OK) return st;
    }
    const size_t smem = (size_t)p.stages * p.stage_bytes + kCtrlBytes + (p.topk > 0 ? kTopkBytes : 0) + 1024;
    if (!ctx->lm_pair_attr_set) {
        MIRROR_CUDA_OK(cudaFuncSetAttribute(lmhead_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget));
        MIRROR_CUDA_OK(cudaFuncSetAttribute(lmhead_pair_early_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget));
        MIRROR_CUDA_OK(cudaFuncSetAttribute(lmhead_pair_free_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget));
        MIRROR_CUDA_OK(cudaFuncSetAttribute(lmhead_pair_topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget));
        MIRROR_CUDA_OK(cudaFuncSetAttribute(lmhead_pair_fp8_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget));
        MIRROR_CUDA_OK(cudaFuncSetAttribute(linear_gated_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget));
        MIRROR_CUDA_OK(cudaFuncSetAttribute(linear_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget));
        ctx->lm_pair_attr_set = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_pairs * 2);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (p.fp8 && (p.topk > 0 || !reduce)) return MIRROR_ERR_UNSUPPORTED;
    auto kern = !reduce ? (p.act ? linear_gated_kernel : linear_pair_kernel) : p.fp8 ? lmhead_pair_fp8_kernel : p.topk > 0 ? lmhead_pair_topk_kernel : p.unit_ctr ? lmhead_pair_free_kernel : p.w_early ? lmhead_pair_early_kernel : lmhead_pair_kernel;
    MIRROR_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, tm_w, tm_h, p));
    ctx->launches += 1;
    MIRROR_CUDA_OK(cudaGetLastError());
    return MIRROR_OK;
}

}  // namespace

int mirror_lmhead_pair_partials(int V) { return 2 * ((V + kPairV - 1) / kPairV); }

bool mirror_lmhead_topk_fusable(const mirror_ctx* ctx, int M, int topk) {
    return topk > 0 && M <= kMaxChunkRows && M >= ctx->tune.lm_pair_min_rows && 8 * ctx->num_sms <= kMirrorTopkMaxLists;      // (4 per CTA, 2 CTAs per SM)
}

// Of a small vocabulary hardly more is met than the bar needs to become good, so many candidates go into the lists, and these
// cost a row what its kappa and the CTAs are; a selection from spilled logits costs kappa passes over a row's V logits, 148
// rows at a time.  The line, between the two over H of 1024 and 5120, V of 1024..60000, kappa of 1..32 and up to 256 rows
// (us at H = 1024, selected in the epilogue / spilled): 256 rows x 1024 ids, kappa 32: 436 / 70; 100 x 4096, 8: 48 / 33; 180 x 8192, 8:
// 47 / 48; 256 x 8192, 8: 61 / 54; 100 x 16000, 8: 50 / 54; 256 x 16000, 8: 57 / 78; 256 x 30370, 32: 131 / 353.
bool mirror_lmhead_topk_spills(const mirror_ctx* ctx, int M, int topk) {
    const long long V = ctx->desc.vocab;
    return V <= 65536 && V * (topk + 4) <= std::min(2000ll * (M - 8), 5200ll * (M - 16));
}

mirror_status mirror_lmhead_pair_launch(mirror_ctx* ctx, const void* hidden, int M, const void* W, float* logits_out,
                                        void* partial_ws, size_t partial_bytes, cudaStream_t stream, int* n_partials,
                                        const float* w_scale, const float* h_scale, int topk, void* topk_ws, size_t topk_ws_bytes,
                                        MirrorLmStart start, bool sums) {
    const bool fp8 = w_scale != nullptr;
    if (fp8 && (!h_scale || ctx->desc.hidden % 128 != 0)) return MIRROR_ERR_SHAPE;
    // (e4m3 rows are staged exactly like bf16 rows of half as many elements: the same bytes, boxes and swizzle)
    const int V = ctx->desc.vocab, H = fp8 ? ctx->desc.hidden / 2 : ctx->desc.hidden;
    // A weight stream (two CTAs per SM) is as long as its busiest pair: the rows a CTA takes per unit are chosen so that
    // the units come out in whole waves over the pairs (152064 rows over 148 pairs: five units of 2 x 104 rows each
    // instead of four or five of 2 x 128).
    int rows_cta = kTileV;
    const bool free_start = start == MIRROR_LM_AT_ONCE && !fp8 && topk == 0 && ctx->d_unit_ctr;
    const bool stream_mode = ctas_per_sm_for(ctx->tune, M) == 2;
    if (stream_mode) {
        // A partial per unit: as many units as the workspace has room for, 2 x 128 rows each for a large vocabulary.  (Dealt out by the
        // counter these are the better ones: with room for balanced units of 2 x 104, the sampled step of 57 rows and 48 layers took
        // 470 instead of 460 us, over a prefix of 256 tokens 336 instead of 321, and that of 99 rows 587 instead of 558.)
        const size_t most = free_start && sums ? partial_bytes / ((size_t)M * 24) : SIZE_MAX;
        const int pairs = ctx->num_sms;
        long long best = -1;
        for (int r = kTileV; r >= 64; r -= 8) {
            const long long units = (V + 2 * r - 1) / (2 * r), waves = (units + pairs - 1) / pairs;
            if ((best < 0 || waves * r < best) && (size_t)units <= most) { best = waves * r; rows_cta = r; }
        }
        const int set = ctx->tune.lm_rows;
        if (set >= 8 && set <= kTileV && set % 8 == 0 && (size_t)((V + 2 * set - 1) / (2 * set)) <= most) rows_cta = set;
    }
    const int n_tiles = (V + 2 * rows_cta - 1) / (2 * rows_cta);
    PairParams p;
    mirror_status st = pair_shape(ctx->tune, M, V, H, &p, rows_cta, topk);
    if (st != MIRROR_OK) return st;
    p.n_units = n_tiles * p.n_chunks;
    int n_pairs = ctx->num_sms / 2 * p.ctas_per_sm;
    if (n_pairs > p.n_units) n_pairs = p.n_units;
    if (n_pairs < 1) return MIRROR_ERR_UNSUPPORTED;
    // partials: one per CTA (single row chunk: running state) or one per 128-row vocabulary tile
    p.sums = sums;
    if (free_start) {
        p.running = p.n_chunks == 1 && !sums;
        p.unit_ctr = ctx->d_unit_ctr;
        // Few units to a pair: one each, in the order in which the pairs begin, and only the rest as they come.  (A unit takes as long as
        // its chain of K blocks, however few pairs are at work: a pair that began early and took a second one would end last.
        // 24 layers x 2 x 4807..18176 tokens before 18841 ids of 7424: 170 us in one wave, 190 by the counter.)
        p.n_own = p.n_units <= 2 * n_pairs ? n_pairs : 0;
    }
    const size_t P = p.running ? (size_t)2 * n_pairs : (size_t)2 * n_tiles;
    if (partial_bytes < P * M * 12) return MIRROR_ERR_WORKSPACE;
    p.w_keep = p.n_chunks > 1;
    p.w_early = start == MIRROR_LM_WEIGHTS_EARLY && stream_mode;       // (a weight stream; with more rows the tensor cores set the pace)
    if (ctx->tune.test_stall_after >= 0 && ctx->tune.test_stall_lm_left-- > 0) p.stall_after = ctx->tune.test_stall_after;
    p.inv_T = 1.0f / ctx->temperature;
    p.inv_T_log2e = p.inv_T * 1.4426950408889634f;
    p.logits_out = logits_out;
    p.part_max = (float*)partial_ws;
    p.part_idx = (int*)(p.part_max + P * M);
    p.part_sum = (float*)(p.part_idx + P * M);
    p.status = ctx->d_status;
    if (topk > 0) {
        if (p.n_chunks != 1 || !ctx->d_topk_bar) return MIRROR_ERR_UNSUPPORTED;      // (one row chunk: a list lives as long as its CTA)
        if (!topk_ws || topk_ws_bytes < 4 * P * M * (size_t)topk * 8) return MIRROR_ERR_WORKSPACE;
        p.part_topv = (float*)topk_ws;
        p.part_topi = (int*)(p.part_topv + 4 * P * M * (size_t)topk);
        p.topk_bar = ctx->d_topk_bar;
    }
    p.fp8 = fp8 ? 1 : 0;
    p.w_scale = w_scale;
    p.h_scale = h_scale;
    st = pair_launch(ctx, true, hidden, W, p, n_pairs, stream);
    if (st != MIRROR_OK) return st;
    *n_partials = (int)P;
    return MIRROR_OK;
}

// Split of the K axis for a plain GEMM with few output tiles: the slice count that fills the CTA pairs best (whole
// waves of units), slices of at least 512 K elements.
int mirror_linear_slices(const mirror_ctx* ctx, int M, int N, int K) {
    const int n_tiles = (N + kPairV - 1) / kPairV, n_chunks = (M + kMaxChunkRows - 1) / kMaxChunkRows;
    const int n_kb = K / kBK, n_pairs = ctx->num_sms / 2 > 0 ? ctx->num_sms / 2 * ctas_per_sm_for(ctx->tune, M) : 1;
    int best = 1;
    double best_eff = 0.0;
    for (int s = 1; s <= 16; ++s) {
        const int per = (n_kb + s - 1) / s;
        if (s > 1 && per < 8) break;
        const int eff_s = (n_kb + per - 1) / per;
        const long long units = (long long)n_tiles * n_chunks * eff_s;
        const long long waves = (units + n_pairs - 1) / n_pairs;
        const double eff = (double)units / (double)(waves * n_pairs);
        if (eff > best_eff + 0.02) { best_eff = eff; best = eff_s; }
    }
    return best;
}

// partial[s][M][N] (fp32) = sum over K slice s of x[M, K] * W[N, K]^T; the caller sums the slices in order.
mirror_status mirror_linear_partial_launch(mirror_ctx* ctx, const void* x, int M, const void* W, int N, int K, float* partial,
                                           size_t partial_bytes, cudaStream_t stream, int* k_slices, bool w_early) {
    PairParams p;
    mirror_status st = pair_shape(ctx->tune, M, N, K, &p);
    if (st != MIRROR_OK) return st;
    const int n_tiles = (N + kPairV - 1) / kPairV, n_kb = K / kBK;
    const int s = mirror_linear_slices(ctx, M, N, K);
    p.kb_per_slice = (n_kb + s - 1) / s;
    p.k_slices = (n_kb + p.kb_per_slice - 1) / p.kb_per_slice;
    if (partial_bytes < (size_t)p.k_slices * M * N * sizeof(float)) return MIRROR_ERR_WORKSPACE;
    p.n_units = n_tiles * p.n_chunks * p.k_slices;
    int n_pairs = ctx->num_sms / 2 * p.ctas_per_sm;
    if (n_pairs > p.n_units) n_pairs = p.n_units;
    if (n_pairs < 1) return MIRROR_ERR_UNSUPPORTED;
    p.w_keep = p.n_chunks > 1;
    p.w_early = w_early;
    p.logits_out = partial;
    p.status = ctx->d_status;
    st = pair_launch(ctx, false, x, W, p, n_pairs, stream);
    if (st != MIRROR_OK) return st;
    *k_slices = p.k_slices;
    return MIRROR_OK;
}

// act[M, I] (bf16) = silu(x W_gate^T) * (x W_up^T), W = [gate rows; up rows], in one kernel (I a multiple of 16).
mirror_status mirror_linear_gated_launch(mirror_ctx* ctx, const void* x, int M, const void* W, int I, int K, void* act, cudaStream_t stream) {
    PairParams p;
    mirror_status st = pair_shape(ctx->tune, M, 2 * I, K, &p);
    if (st != MIRROR_OK) return st;
    if (I % 16 != 0) return MIRROR_ERR_SHAPE;
    p.n_units = (2 * I + kPairV - 1) / kPairV * p.n_chunks;
    int n_pairs = ctx->num_sms / 2 * p.ctas_per_sm;
    if (n_pairs > p.n_units) n_pairs = p.n_units;
    if (n_pairs < 1) return MIRROR_ERR_UNSUPPORTED;
    p.w_keep = p.n_chunks > 1;
    p.w_early = 1;
    p.act = (__nv_bfloat16*)act;
    p.status = ctx->d_status;
    return pair_launch(ctx, false, x, W, p, n_pairs, stream);
}
