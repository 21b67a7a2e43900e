// Acceptance, branch selection, emitted tokens and reuse lookup (Sec. 3.1; Eq. 3 / Eq. 10).
//
// Greedy: one thread block per request.  Warps take branches round-robin; lane j of a warp tests the node at depth j+1 of
// its branch, a ballot gives the number of leading passes (the acceptance operator of Eq. 3 applied to that branch).
// Thread 0 then picks the longest branch (lowest index on ties) and the deciding row R, and emits argmax[R].
//
// Speculative sampling and the rule over the tree draw a token by inverse CDF over the vocabulary, in fp64.  What bounds
// them is the fp64 exponentials (150 k per pass: 30 us on one SM), so a CLUSTER of up to 16 CTAs per request shares the
// vocabulary (cluster_shape): each warp has one contiguous chunk that it reads coalesced.  The chunks' sums go to every CTA
// through distributed shared memory; all of them scan the same numbers and take the same decisions, one cluster barrier
// per pass, nothing spins.  The chunk that holds the crossing is then summed again in a part per warp and the part searched, so
// the search is three short steps.  (One block per request with a contiguous segment per thread: 97-117 us for 8 and 16
// requests x 128-152 k ids.)
#include <string.h>

#include <algorithm>

#include "mirror_internal.h"

namespace {

constexpr int kGreedyThreads = 256;
constexpr int kFoldThreads = 1024;                    // of a greedy block that folds the LM head's partials itself
constexpr int kSpecThreads = 512;                     // of a CTA of the chain rule's clusters
constexpr int kMaxWarps = 32;                         // of a CTA of the clusters: 16 or 32
constexpr int kMaxChunks = 256;                       // warps of a cluster: up to 16 CTAs (above 8: opt-in) of 16 warps, or 8 of 32

struct AcceptTreeParams {
    int n, n_branches, gamma;
    unsigned char parent[MIRROR_MAX_NODES];
    unsigned char path[MIRROR_MAX_BRANCHES][MIRROR_MAX_DEPTH];
    unsigned char path_len[MIRROR_MAX_BRANCHES];
};

struct AcceptArgs {
    int mode, emit_bonus, V, n_cand;
    double inv_T;
    const int32_t* tokens;
    const int32_t* target_argmax;
    const float* logits;
    const float* lse;
    const float* q_probs;
    const float* u_accept;
    const float* u_resample;
    const int32_t* cand_ids;
    mirror_accept_out out;
    double* tree_scratch;          // nullable fp64 [B, 2, V]: running distribution of the tree rule
    int* status;
};

__device__ __forceinline__ double warp_excl_scan(double v, int lane, double* total) {
    double inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        double t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    *total = __shfl_sync(0xffffffffu, inc, 31);
    return inc - v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// What a branch test says about node c (token x, parent row r): the target's probability and the draft's, its uniform.
struct NodeTest {
    double p, q, u;
};
__device__ __forceinline__ void bad_token(const AcceptArgs& a, int c) {      // (first error wins)
    if (atomicCAS(a.status, 0, MIRROR_DEV_CHECK) == 0) atomicExch(a.status + 1, 100 + c);
}
// ok: the token is in the vocabulary (a node without one is rejected, and reported by whoever comes to it).
__device__ __forceinline__ NodeTest node_test(const AcceptTreeParams& tp, const AcceptArgs& a, int b, int c, bool& ok) {
    NodeTest t = {0.0, 0.0, 0.0};
    const int x = a.tokens[(size_t)b * tp.n + c];
    ok = x >= 0 && x < a.V;
    if (!ok) return t;
    const size_t row = (size_t)b * tp.n + tp.parent[c];
    t.u = (double)a.u_accept[(size_t)b * tp.n + c];
    t.q = (double)a.q_probs[((size_t)b * (tp.n - 1) + (c - 1)) * a.V + x];
    t.p = exp((double)a.logits[row * a.V + x] * a.inv_T - (double)a.lse[row]);
    return t;
}

// The decision's outputs, by the first threads of one block.
__device__ __forceinline__ void write_out(const AcceptTreeParams& tp, const AcceptArgs& a, int b, int A, int best, int R, bool have_extra, int extra,
                                          const unsigned char* path) {
    const int tid = threadIdx.x, gamma = tp.gamma, n = tp.n;
    const int32_t* tok = a.tokens + (size_t)b * n;
    if (tid <= gamma) {
        int e = -1;
        if (tid < A) e = tok[path[tid]];
        else if (tid == A && have_extra) e = extra;
        a.out.emitted[(size_t)b * (gamma + 1) + tid] = e;
        if (tid < gamma) a.out.accepted_nodes[(size_t)b * gamma + tid] = (tid < A) ? (int)path[tid] : -1;
    }
    if (tid == 0) {
        a.out.n_accepted[b] = A;
        a.out.best_branch[b] = best;
        a.out.decide_row[b] = R;
        a.out.n_emitted[b] = A + (have_extra ? 1 : 0);
        int slot = -1;
        if (have_extra && a.cand_ids)
            for (int k = 0; k < a.n_cand; ++k)
                if (a.cand_ids[((size_t)b * n + R) * a.n_cand + k] == extra) { slot = k; break; }
        a.out.reuse_slot[b] = slot;
    }
}

// Longest branch out of the branches' leading accepts (lowest index on ties), by one thread.
struct Choice {
    int A, best, R, rej_node;
};
__device__ __forceinline__ Choice choose(const AcceptTreeParams& tp, const int* len) {
    Choice c = {0, 0, 0, -1};
    for (int i = 0; i < tp.n_branches; ++i)
        if (len[i] > c.A) { c.A = len[i]; c.best = i; }
    if (c.A > 0) c.R = tp.path[c.best][c.A - 1];
    if (tp.n_branches > 0 && c.A < tp.path_len[c.best]) c.rej_node = tp.path[c.best][c.A];
    return c;
}

// FOLD: the rows' argmax comes out of the LM head's row partials, in the block that needs it: a launch less (the merge kernel
// in front and this one took 5.5 us of a toy model's step of 22).  Lanes are rows, warps share the partials.
template <bool FOLD>
__global__ void __launch_bounds__(FOLD ? kFoldThreads : kGreedyThreads)
accept_greedy_kernel(const __grid_constant__ AcceptTreeParams tp, const AcceptArgs a, const MirrorLmPartials parts, int32_t* argmax_out) {
    constexpr int kBlockWarps = (FOLD ? kFoldThreads : kGreedyThreads) / 32;
    __shared__ int s_len[MIRROR_MAX_BRANCHES];
    __shared__ Choice s_choice;
    __shared__ float s_max[FOLD ? kBlockWarps : 1][33];
    __shared__ int s_idx[FOLD ? kBlockWarps : 1][33];
    __shared__ int32_t s_argmax[FOLD ? MIRROR_MAX_NODES : 1];
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = tp.n;
    const int32_t* tok = a.tokens + (size_t)b * n;
    const int32_t* am = FOLD ? s_argmax : a.target_argmax + (size_t)b * n;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (FOLD) {
        const size_t M = (size_t)gridDim.x * n;
        // the comparator (logit descending, id ascending) makes the result independent of the order
        auto fold = [](float& m, int& i, float om, int oi) {
            if (om > m || (om == m && om != -INFINITY && oi < i)) { m = om; i = oi; }
        };
#pragma unroll 1
        for (int r0 = 0; r0 < n; r0 += 32) {
            float m = -INFINITY;
            int i = 0x7fffffff;
            if (r0 + lane < n) {
                const size_t at = (size_t)b * n + r0 + lane;
#pragma unroll 4
                for (int k = warp; k < parts.count; k += kBlockWarps) fold(m, i, parts.max[k * M + at], parts.idx[k * M + at]);
            }
            s_max[warp][lane] = m;
            s_idx[warp][lane] = i;
            __syncthreads();
            if (r0 + warp < n) {                                   // (as many warps as lanes)
                m = s_max[lane][warp];
                i = s_idx[lane][warp];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) fold(m, i, __shfl_xor_sync(0xffffffffu, m, o), __shfl_xor_sync(0xffffffffu, i, o));
                if (lane == 0) {
                    s_argmax[r0 + warp] = i;
                    argmax_out[(size_t)b * n + r0 + warp] = i;
                }
            }
            __syncthreads();
        }
    }
    for (int br = warp; br < tp.n_branches; br += kBlockWarps) {
        const int len = tp.path_len[br];
        bool pass = true;
        if (lane < len) {
            const int c = tp.path[br][lane];
            pass = tok[c] == am[tp.parent[c]];
        }
        const unsigned fail = __ballot_sync(0xffffffffu, lane < len && !pass);
        if (lane == 0) s_len[br] = fail ? (__ffs(fail) - 1) : len;
    }
    __syncthreads();
    if (tid == 0) s_choice = choose(tp, s_len);
    __syncthreads();
    const Choice c = s_choice;
    const bool have_extra = (c.rej_node >= 0) || tp.n_branches == 0 || a.emit_bonus != 0;
    write_out(tp, a, b, c.A, c.best, c.R, have_extra, have_extra ? am[c.R] : -1, tp.path[c.best]);
}

// ---- the cluster's view of the vocabulary --------------------------------------------------------------------------
__device__ __forceinline__ void cluster_barrier() {       // release / acquire: also of what the CTAs wrote to global memory
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t remote(const void* smem, uint32_t rank) {      // the same object in CTA `rank`
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(ptx::smem_u32(smem)), "r"(rank));
    return r;
}

struct DrawShared {
    double sum[2][2][kMaxChunks];                         // [pass parity][which sum][chunk]: the same in every CTA after a pass
    double sub[kMaxWarps];
    int token;                                            // CTA 0's: the drawn token (-1: none yet)
    int last;                                             // CTA 0's: last id with positive mass
};
template <int kWarps>
struct Draw {
    DrawShared& s;
    int V, rank, n_cta, chunk_len, lo, hi;                // [lo, hi): this warp's chunk
    uint32_t pass = 0;
    static constexpr int kAhead = kWarps == 32 ? 4 : 8;   // ids a thread loads before it works on the first (as registers allow)
    __device__ Draw(DrawShared& sh, int vocab) : s(sh), V(vocab) {
        uint32_t r, n;
        asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
        asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
        rank = (int)r;
        n_cta = (int)n;
        const int chunks = n_cta * kWarps;
        chunk_len = ((V + chunks - 1) / chunks + 31) & ~31;
        lo = min((rank * kWarps + (int)(threadIdx.x >> 5)) * chunk_len, V);
        hi = min(lo + chunk_len, V);
        cluster_barrier();                                // (every CTA of the cluster has started: its shared memory may be written to)
    }
    // One pass over the vocabulary: load(v) fetches what id v's masses need, add(v, loaded, x0, x1) adds them to x0 and x1;
    // kAhead loads are in flight per thread.  Returns this warp's chunk sums to all CTAs (kTwo: both, else the first).
    template <bool kTwo, class L, class F>
    __device__ __forceinline__ void sums(L load, F add) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        double x = 0.0, y = 0.0;
#pragma unroll 1
        for (int v0 = lo + lane; v0 < hi; v0 += 32 * kAhead) {
            decltype(load(0)) in[kAhead];
#pragma unroll
            for (int k = 0; k < kAhead; ++k)
                if (v0 + 32 * k < hi) in[k] = load(v0 + 32 * k);
#pragma unroll
            for (int k = 0; k < kAhead; ++k)
                if (v0 + 32 * k < hi) add(v0 + 32 * k, in[k], x, y);
        }
        const double sx = warp_sum(x), sy = kTwo ? warp_sum(y) : 0.0;
        const uint32_t par = pass & 1;
        if (lane < n_cta) {
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote(&s.sum[par][0][rank * kWarps + warp], lane)), "d"(sx) : "memory");
            if (kTwo) asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote(&s.sum[par][1][rank * kWarps + warp], lane)), "d"(sy) : "memory");
        }
        cluster_barrier();        // (the words of this parity are written again two passes later, behind another barrier)
        ++pass;
    }
    // After sums(): total of one of the two, the same number in every thread of every CTA; *excl: of the chunks before this lane's.
    __device__ __forceinline__ double total(int which, double* excl = nullptr) const {
        const int lane = threadIdx.x & 31, per = n_cta * kWarps / 32;
        const double* c = s.sum[(pass - 1) & 1][which] + lane * per;
        double mine = 0.0, tot;
        for (int k = 0; k < per; ++k) mine += c[k];
        const double e = warp_excl_scan(mine, lane, &tot);
        if (excl) *excl = e;
        return tot;
    }
    // After sums(): min{v : sum_{w <= v} mass(w) > u * total}, searched in the chunk that holds the crossing; the last id with
    // positive mass if rounding leaves none.  Collective; the token is valid in CTA 0.
    template <class F>
    __device__ __forceinline__ int pick(int which, double u, F mass) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, per = n_cta * kWarps / 32;
        double excl;
        const double thr = u * total(which, &excl);
        const double* c = s.sum[(pass - 1) & 1][which] + lane * per;
        int found = -1;
        double found_excl = 0.0;
        for (int k = 0; k < per; ++k) {
            if (found < 0 && excl + c[k] > thr) { found = lane * per + k; found_excl = excl; }
            excl += c[k];
        }
        const unsigned any = __ballot_sync(0xffffffffu, found >= 0);
        if (threadIdx.x == 0 && rank == 0) s.token = s.last = -1;
        if (any) {
            const int src = __ffs(any) - 1;
            found = __shfl_sync(0xffffffffu, found, src);
            found_excl = __shfl_sync(0xffffffffu, found_excl, src);
        }
        cluster_barrier();
        if (any && found / kWarps == rank) {
            // the chunk in as many parts as the CTA has warps, then the part with the crossing id by id
            const int c_lo = min(found * chunk_len, V), c_hi = min(c_lo + chunk_len, V);
            const int part = (((chunk_len >> 5) + kWarps - 1) / kWarps) << 5;
            auto part_lo = [&](int w) { return min(c_lo + w * part, c_hi); };
            double x = 0.0;
            for (int v = part_lo(warp) + lane; v < part_lo(warp + 1); v += 32) x += mass(v);
            x = warp_sum(x);
            if (lane == 0) s.sub[warp] = x;
            __syncthreads();
            double tot;
            const double mine = lane < kWarps ? s.sub[lane] : 0.0;
            const double before = found_excl + warp_excl_scan(mine, lane, &tot);
            const unsigned over = __ballot_sync(0xffffffffu, lane < kWarps && before + mine > thr);
            const unsigned some = __ballot_sync(0xffffffffu, mine > 0.0);
            // (the parts' sums may round below the chunk's: then the last part with any mass)
            const int w = over ? __ffs(over) - 1 : some ? 31 - __clz(some) : 0;
            if (warp == w) {
                double run = __shfl_sync(0xffffffffu, before, w);
                int tok = -1, last = part_lo(w);
                for (int v0 = part_lo(w); v0 < part_lo(w + 1) && tok < 0; v0 += 32) {
                    const int v = v0 + lane;
                    const double m = v < part_lo(w + 1) ? mass(v) : 0.0;
                    double step;
                    const double e = run + warp_excl_scan(m, lane, &step);
                    const unsigned hit = __ballot_sync(0xffffffffu, m > 0.0 && e + m > thr);
                    const unsigned pos = __ballot_sync(0xffffffffu, m > 0.0);
                    if (hit) tok = v0 + __ffs(hit) - 1;
                    if (pos) last = v0 + 31 - __clz(pos);
                    run += step;
                }
                if (lane == 0) asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(remote(&s.token, 0)), "r"(tok >= 0 ? tok : last) : "memory");
            }
        } else if (!any) {
            // rounding left the threshold above every cumulative sum (the same in every CTA): the last id with positive mass
            int last = -1;
            for (int v = lo + lane; v < hi; v += 32)
                if (mass(v) > 0.0) last = v;
            if (last >= 0) asm volatile("red.shared::cluster.max.s32 [%0], %1;" ::"r"(remote(&s.last, 0)), "r"(last) : "memory");
        }
        cluster_barrier();
        return s.token >= 0 ? s.token : s.last;
    }
};

__global__ void __launch_bounds__(kSpecThreads, 1)
accept_spec_kernel(const __grid_constant__ AcceptTreeParams tp, const AcceptArgs a) {
    __shared__ DrawShared s_draw;
    __shared__ int s_len[MIRROR_MAX_BRANCHES];
    __shared__ unsigned char s_pass[MIRROR_MAX_NODES];
    __shared__ Choice s_choice;
    Draw<kSpecThreads / 32> draw(s_draw, a.V);
    const int b = blockIdx.x / draw.n_cta, tid = threadIdx.x, n = tp.n, V = a.V;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    // every CTA evaluates the tests itself, from numbers that are identical in all of them
    if (tid > 0 && tid < n) {
        bool ok;
        const NodeTest t = node_test(tp, a, b, tid, ok);
        if (!ok) bad_token(a, tid);
        s_pass[tid] = ok && t.u * t.q <= t.p;
    }
    __syncthreads();
    for (int br = tid; br < tp.n_branches; br += kSpecThreads) {
        int k = 0;
        while (k < tp.path_len[br] && s_pass[tp.path[br][k]]) ++k;
        s_len[br] = k;
    }
    __syncthreads();
    if (tid == 0) s_choice = choose(tp, s_len);
    __syncthreads();
    const Choice c = s_choice;
    const bool have_extra = (c.rej_node >= 0) || tp.n_branches == 0 || a.emit_bonus != 0;
    int extra = -1;
    if (have_extra) {
        // inverse-CDF draw from max(0, p - q') (rejection) or p (bonus, or a residual without mass)
        const size_t row = (size_t)b * n + c.R;
        const float* lr = a.logits + row * V;
        const double lse = (double)a.lse[row];
        const float* qc = c.rej_node >= 0 ? a.q_probs + ((size_t)b * (n - 1) + (c.rej_node - 1)) * V : nullptr;
        draw.template sums<true>([&](int v) { return make_float2(lr[v], qc ? qc[v] : 0.f); },
                  [&](int, float2 in, double& sp, double& sr) {
                      const double p = exp((double)in.x * a.inv_T - lse);
                      sp += p;
                      sr += fmax(p - (double)in.y, 0.0);        // (without q: not looked at)
                  });
        const bool use_res = qc && draw.total(1) > 0.0;
        extra = draw.pick(use_res ? 1 : 0, (double)a.u_resample[row], [&](int v) {
            const double p = exp((double)lr[v] * a.inv_T - lse);
            return use_res ? fmax(p - (double)qc[v], 0.0) : p;
        });
    }
    if (draw.rank == 0) write_out(tp, a, b, c.A, c.best, c.R, have_extra, extra, tp.path[c.best]);
    cluster_barrier();                                    // no CTA may leave while a peer can still write to its shared memory
}

// ---------------------------------------------------------------------------------------------------
// Lossless acceptance over a token tree: sequential multi-round rejection over the siblings of each accepted
// row (the speculative-sampling rule of Sec. 3.1 applied to sibling sets, for tree drafts).  The walk goes down from the
// root: at row r the current distribution m starts as the target's p_r; the children of r are tested in node order
// against m: child c (token x, draft distribution q_c) passes iff u_accept[c] * q_c[x] <= m[x] and the walk moves to
// c; a child that fails turns m into the normalised residual max(0, m - q_c).  m[v] is either re-evaluated from the
// logits, the rejected siblings' q rows and their normalisers Z_i, or -- when the caller's workspace has room --
// kept in fp64 scratch memory (two buffers, so that a residual without mass can be dropped); both follow the
// definition's operation order per element.  A rejection costs one pass over the vocabulary for Z, the final draw one
// more.  What the tests read of p and q themselves is fetched for all nodes at once in front of the walk.
// ---------------------------------------------------------------------------------------------------
constexpr int kMaxRejected = MIRROR_MAX_BRANCHES;     // siblings rejected at one row
struct Loaded {
    double m;
    float q;
};

template <int kThreads>
__global__ void __launch_bounds__(kThreads, 1)
accept_tree_kernel(const __grid_constant__ AcceptTreeParams tp, const AcceptArgs a) {
    __shared__ DrawShared s_draw;
    __shared__ NodeTest s_test[MIRROR_MAX_NODES];
    __shared__ bool s_ok[MIRROR_MAX_NODES];
    __shared__ double s_Z[kMaxRejected];
    __shared__ int s_rej[kMaxRejected];
    __shared__ unsigned char s_path[MIRROR_MAX_DEPTH];
    Draw<kThreads / 32> draw(s_draw, a.V);
    const int b = blockIdx.x / draw.n_cta, tid = threadIdx.x, n = tp.n, V = a.V;
    const int32_t* tok = a.tokens + (size_t)b * n;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (tid > 0 && tid < n) s_test[tid] = node_test(tp, a, b, tid, s_ok[tid]);
    __syncthreads();

    int r = 0, A = 0, n_rej = 0, n_children = 0;
    double* const buf0 = a.tree_scratch ? a.tree_scratch + (size_t)b * 2 * V : nullptr;
    double* const buf1 = buf0 ? buf0 + V : nullptr;
    // Buffer that holds the current residual (when n_rej > 0).  Residuals go to the two buffers in turn for the whole walk, never
    // back to buf0 at a new row: a slower CTA may still be at the test that led there, which reads m[token] from `cur`.  What was
    // last read from the other buffer lies behind the barrier of the pass that made `cur` the current one.
    int cur = 0;
    double inv_Z = 1.0;                            // 1 / Z of the last effective rejection
    // m[v] at row r after the rejections recorded so far, from the logit or (kept) the unnormalised residual
    auto source = [&](const float* lr, int v) -> double { return buf0 && n_rej > 0 ? (cur ? buf1 : buf0)[v] : (double)lr[v]; };
    auto raw = [&](double src, double lse_r, int v) -> double {             // before the division by the last Z
        if (buf0 && n_rej > 0) return src;
        double m = exp(src * a.inv_T - lse_r);
        for (int i = 0; i < n_rej; ++i) {
            if (i > 0) m /= s_Z[i - 1];
            m = fmax(m - (double)a.q_probs[((size_t)b * (n - 1) + (s_rej[i] - 1)) * V + v], 0.0);
        }
        return m;
    };
    auto mass = [&](double src, double lse_r, int v) -> double {            // (times 1/Z: one rounding away from the quotient)
        const double m = raw(src, lse_r, v);
        return n_rej == 0 ? m : buf0 ? m * inv_Z : m / s_Z[n_rej - 1];
    };
    bool summed = false;                           // the last pass's sums are those of the current m, times Z
    // (the whole walk is the same in every thread of every CTA)
    for (;;) {
        const size_t row = (size_t)b * n + r;
        const float* lr = a.logits + row * V;
        const double lse_r = (double)a.lse[row];
        n_rej = 0;
        n_children = 0;
        summed = false;
        int next = -1;
        for (int c = r + 1; c < n; ++c) {
            if (tp.parent[c] != r) continue;
            ++n_children;
            if (s_ok[c]) {
                const NodeTest t = s_test[c];
                if (t.u * t.q <= (n_rej == 0 ? t.p : mass(source(lr, tok[c]), lse_r, tok[c]))) { next = c; break; }
            } else if (tid == 0) {
                bad_token(a, c);
            }
            // rejected: normaliser of the residual (a residual without mass leaves m as it is)
            const float* qc = a.q_probs + ((size_t)b * (n - 1) + (c - 1)) * V;
            double* const nxt = !buf0 ? nullptr : (cur ? buf0 : buf1);
            draw.template sums<false>([&](int v) { return Loaded{source(lr, v), qc[v]}; },
                      [&](int v, const Loaded& in, double& x, double&) {
                          const double res = fmax(mass(in.m, lse_r, v) - (double)in.q, 0.0);
                          if (nxt) nxt[v] = res;
                          x += res;
                      });
            const double Z = draw.total(0);
            summed = Z > 0.0 && n_rej < kMaxRejected;
            if (summed) {
                if (tid == 0) { s_rej[n_rej] = c; s_Z[n_rej] = Z; }
                if (nxt) cur = (nxt == buf1) ? 1 : 0;
                inv_Z = 1.0 / Z;
                ++n_rej;
            }
            __syncthreads();
        }
        if (next < 0) break;
        if (tid == 0 && A < MIRROR_MAX_DEPTH) s_path[A] = (unsigned char)next;
        ++A;
        r = next;
        __syncthreads();
        if (A >= MIRROR_MAX_DEPTH) { n_children = 0; n_rej = 0; summed = false; break; }      // (cannot happen: depth <= gamma <= 32)
    }
    const bool have_extra = (n_children > 0) || a.emit_bonus != 0;
    int extra = -1;
    if (have_extra) {
        const size_t row = (size_t)b * n + r;
        const float* lr = a.logits + row * V;
        const double lse_r = (double)a.lse[row];
        // (a rejection has just added the same masses up: the draw needs them only up to a factor)
        if (!summed) draw.template sums<false>([&](int v) { return source(lr, v); }, [&](int v, double in, double& x, double&) { x += raw(in, lse_r, v); });
        extra = draw.pick(0, (double)a.u_resample[row], [&](int v) { return raw(source(lr, v), lse_r, v); });
    }
    if (draw.rank == 0) {
        // the lowest-index branch that contains the accepted path
        int best = 0;
        for (int i = 0; i < tp.n_branches; ++i) {
            bool same = tp.path_len[i] >= A;
            for (int k = 0; k < A && same; ++k) same = (tp.path[i][k] == s_path[k]);
            if (same) { best = i; break; }
        }
        write_out(tp, a, b, A, best, r, have_extra, extra, s_path);
    }
    cluster_barrier();                                    // no CTA may leave while a peer can still write to its shared memory
}

// CTAs and threads per request.
//   - Chain rule: enough CTAs that a warp's chunk is a few steps, no more (a pass ends with a barrier of the cluster); 16 only
//     for few requests: a cluster lives in one GPC, and eight of 16 CTAs do not all fit at once (B = 8: 20.7 us against 16.9 with
//     8 CTAs).
//   - Tree rule: without scratch memory a pass costs an exponential and a chain of up to `siblings` subtractions and divisions
//     per id: from four siblings on as many threads as there are ids, up to 8192, in 1024-thread CTAs where 16 CTAs do not fit (8
//     siblings, 16 requests: 32000 ids 150 -> 84 us, 8192 ids 181 -> 94; a walk without rejections takes 4 us longer in
//     1024-thread CTAs).  Else as the chain rule, but the walk has many passes: 8 CTAs from 16 k ids while they all fit (8 siblings,
//     8 requests x 32000 ids: 42 -> 32 us; 16 requests, one branch: 15 -> 21).
struct ClusterShape {
    int n_cta, threads;
};
ClusterShape cluster_shape(const mirror_ctx* ctx, int batch, bool tree, bool scratch, int siblings) {
    const int V = ctx->desc.vocab;
    const bool chains = tree && !scratch && siblings >= 4, few = batch * 32 <= ctx->num_sms;
    if (few && V > (chains ? 4096 : 65536)) return {16, 512};
    if (chains) return V > 4096 ? ClusterShape{8, 1024} : ClusterShape{V > 2048 ? 8 : V > 1024 ? 4 : 2, 512};
    return {V > (tree && batch * 16 <= ctx->num_sms ? 16384 : 32768) ? 8 : V > 8192 ? 4 : 2, 512};
}

}  // namespace

mirror_status mirror_accept_launch(mirror_ctx* ctx, const mirror_tree* tree, const MirrorTreeInfo& ti,
                                   const mirror_accept_in* in, const mirror_accept_out* out, cudaStream_t stream,
                                   double* tree_scratch, const MirrorLmPartials* partials, int32_t* argmax_out) {
    AcceptTreeParams tp;
    tp.n = ti.n;
    tp.n_branches = ti.n_branches;
    tp.gamma = tree->gamma;
    for (int i = 0; i < MIRROR_MAX_NODES; ++i) tp.parent[i] = (i < ti.n && ti.parent[i] >= 0) ? (unsigned char)ti.parent[i] : 255;
    memcpy(tp.path, ti.path, sizeof tp.path);
    memcpy(tp.path_len, ti.path_len, sizeof tp.path_len);
    AcceptArgs a;
    a.mode = in->mode;
    a.emit_bonus = in->emit_bonus;
    a.V = ctx->desc.vocab;
    a.n_cand = in->cand_ids ? in->n_cand : 0;
    a.inv_T = 1.0 / (double)ctx->temperature;
    a.tokens = tree->tokens;
    a.target_argmax = in->target_argmax;
    a.logits = in->logits;
    a.lse = in->lse;
    a.q_probs = in->q_probs;
    a.u_accept = in->u_accept;
    a.u_resample = in->u_resample;
    a.cand_ids = in->cand_ids;
    a.out = *out;
    a.tree_scratch = tree_scratch;
    a.status = ctx->d_status;
    if (in->mode == MIRROR_ACCEPT_GREEDY) {
        const MirrorLmPartials none = {0, nullptr, nullptr};
        if (partials) MIRROR_CUDA_OK(mirror_launch_pdl(accept_greedy_kernel<true>, dim3(tree->batch), dim3(kFoldThreads), 0, stream, tp, a, *partials, argmax_out));
        else MIRROR_CUDA_OK(mirror_launch_pdl(accept_greedy_kernel<false>, dim3(tree->batch), dim3(kGreedyThreads), 0, stream, tp, a, none, argmax_out));
    } else {
        const bool by_tree = in->mode == MIRROR_ACCEPT_SPEC_TREE;
        int siblings = 0, children[MIRROR_MAX_NODES] = {};
        for (int i = 1; i < ti.n; ++i) siblings = std::max(siblings, ++children[ti.parent[i]]);
        const ClusterShape shape = cluster_shape(ctx, tree->batch, by_tree, tree_scratch != nullptr, siblings);
        auto kern = !by_tree ? accept_spec_kernel : shape.threads == 1024 ? accept_tree_kernel<1024> : accept_tree_kernel<512>;
        const unsigned n_cta = (unsigned)shape.n_cta;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)tree->batch * n_cta);
        cfg.blockDim = dim3(shape.threads);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = stream;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = n_cta;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        if (n_cta > 8) MIRROR_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        MIRROR_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, tp, a));
    }
    ctx->launches += 1;
    MIRROR_CUDA_OK(cudaGetLastError());
    return MIRROR_OK;
}

extern "C" mirror_status mirror_accept_select(mirror_ctx* ctx, const mirror_tree* tree, const mirror_accept_in* in,
                                              const mirror_accept_out* out, void* stream) {
    if (!ctx || !tree || !in || !out || !tree->tokens) return MIRROR_ERR_ARG;
    if (!out->n_accepted || !out->best_branch || !out->n_emitted || !out->emitted || !out->accepted_nodes ||
        !out->decide_row || !out->reuse_slot)
        return MIRROR_ERR_ARG;
    if (in->mode == MIRROR_ACCEPT_GREEDY) {
        if (!in->target_argmax) return MIRROR_ERR_ARG;
    } else if (in->mode == MIRROR_ACCEPT_SPEC_SAMPLING || in->mode == MIRROR_ACCEPT_SPEC_TREE) {
        if (!in->logits || !in->lse || !in->u_accept || !in->u_resample) return MIRROR_ERR_ARG;
        if (tree->n_nodes > 1 && !in->q_probs) return MIRROR_ERR_ARG;
    } else {
        return MIRROR_ERR_ARG;
    }
    if (in->cand_ids && in->n_cand < 0) return MIRROR_ERR_ARG;
    MirrorTreeInfo ti;
    mirror_status st = mirror_build_tree(tree, &ti);
    if (st != MIRROR_OK) return st;
    MIRROR_CUDA_OK(cudaSetDevice(ctx->device));
    double* tree_scratch = nullptr;
    if (in->mode == MIRROR_ACCEPT_SPEC_TREE && ctx->ws) {
        MirrorWsLayout L;
        mirror_ws_layout(ctx, (size_t)tree->batch * tree->n_nodes, &L, (size_t)tree->batch);
        if (ctx->ws_bytes >= L.end_accept) tree_scratch = (double*)((uint8_t*)ctx->ws + L.accept_scratch);
    }
    return mirror_accept_launch(ctx, tree, ti, in, out, (cudaStream_t)stream, tree_scratch);
}
