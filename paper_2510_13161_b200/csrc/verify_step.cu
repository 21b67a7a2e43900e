// Public entry points for attention and for the fused verify step (attention over all layers ->
// LM head with fused reductions -> acceptance), all enqueued on one stream.
#include <algorithm>

#include "mirror_internal.h"

namespace {

mirror_status check_kv(const mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree) {
    if (!kv->k_pool || !kv->v_pool || !kv->page_table || !kv->prefix_len) return MIRROR_ERR_ARG;
    if (kv->num_layers <= 0 || kv->num_pages <= 0 || kv->max_pages_per_req <= 0) return MIRROR_ERR_ARG;
    if (((uintptr_t)kv->k_pool & 15) || ((uintptr_t)kv->v_pool & 15)) return MIRROR_ERR_ARG;
    const int64_t page_elems = (int64_t)ctx->desc.n_kv_heads * ctx->desc.page_size * ctx->desc.head_dim;
    if (kv->num_layers > 1 && (kv->layer_stride < (int64_t)kv->num_pages * page_elems)) return MIRROR_ERR_SHAPE;
    if (kv->layer_stride % page_elems != 0) return MIRROR_ERR_UNSUPPORTED;
    (void)tree;
    return MIRROR_OK;
}

// Do two ranges of device memory have no byte in common?
bool apart(const void* a, size_t a_bytes, const void* b, size_t b_bytes) {
    return (uintptr_t)a + a_bytes <= (uintptr_t)b || (uintptr_t)b + b_bytes <= (uintptr_t)a;
}

}  // namespace

extern "C" mirror_status mirror_attn_verify(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree,
                                            const void* q, const void* k_new, const void* v_new, void* out,
                                            float* lse_out, void* stream) {
    if (!ctx || !kv || !tree || !q || !k_new || !v_new || !out) return MIRROR_ERR_ARG;
    mirror_status st = check_kv(ctx, kv, tree);
    if (st != MIRROR_OK) return st;
    if (((uintptr_t)q & 15) || ((uintptr_t)k_new & 15) || ((uintptr_t)v_new & 15) || ((uintptr_t)out & 15)) return MIRROR_ERR_ARG;
    MirrorTreeInfo ti;
    st = mirror_build_tree(tree, &ti);
    if (st != MIRROR_OK) return st;
    MirrorWsLayout L;
    mirror_ws_layout(ctx, (size_t)tree->batch * tree->n_nodes, &L);
    if (!ctx->ws || ctx->ws_bytes < L.end_attn) return MIRROR_ERR_WORKSPACE;
    MIRROR_CUDA_OK(cudaSetDevice(ctx->device));
    uint8_t* ws = (uint8_t*)ctx->ws;
    return mirror_attn_launch(ctx, kv, tree, ti, q, k_new, v_new, out, lse_out, (float*)(ws + L.attn_partial), (cudaStream_t)stream);
}

extern "C" mirror_status mirror_attn_verify_fp8(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree, const void* q,
                                                const void* k_new_fp8, const void* v_new_fp8, const float* k_scale,
                                                const float* v_scale, float q_scale, void* out, float* lse_out, void* stream) {
    if (!ctx || !kv || !tree || !q || !k_new_fp8 || !v_new_fp8 || !k_scale || !v_scale || !out || !(q_scale > 0.f)) return MIRROR_ERR_ARG;
    if (ctx->desc.head_dim != 128) return MIRROR_ERR_UNSUPPORTED;
    mirror_status st = check_kv(ctx, kv, tree);
    if (st != MIRROR_OK) return st;
    if (((uintptr_t)q & 15) || ((uintptr_t)k_new_fp8 & 15) || ((uintptr_t)v_new_fp8 & 15) || ((uintptr_t)out & 15)) return MIRROR_ERR_ARG;
    MirrorTreeInfo ti;
    st = mirror_build_tree(tree, &ti);
    if (st != MIRROR_OK) return st;
    MirrorWsLayout L;
    mirror_ws_layout(ctx, (size_t)tree->batch * tree->n_nodes, &L);
    if (!ctx->ws || ctx->ws_bytes < L.end_attn) return MIRROR_ERR_WORKSPACE;
    MIRROR_CUDA_OK(cudaSetDevice(ctx->device));
    uint8_t* ws = (uint8_t*)ctx->ws;
    const MirrorAttnFp8 f8 = {k_scale, v_scale, q_scale};
    return mirror_attn_launch(ctx, kv, tree, ti, q, k_new_fp8, v_new_fp8, out, lse_out, (float*)(ws + L.attn_partial),
                              (cudaStream_t)stream, &f8);
}

namespace {

struct HostIO {                       // host-buffer variant: pinned host inputs / outputs of one step
    const void* h_q;
    const void* h_k_new;
    const void* h_v_new;
    const int32_t* h_tokens;
    const mirror_accept_host_out* h_out;
};

constexpr int kHostChunks = kMirrorHostChunks;
enum { kEvTokens = kHostChunks, kEvBegin, kEvDecided, kEvSent };       // events behind the pieces' own

mirror_status ensure_copy_stream(mirror_ctx* ctx) {
    if (ctx->copy_stream) return MIRROR_OK;
    MIRROR_CUDA_OK(cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking));
    MIRROR_CUDA_OK(cudaStreamCreateWithFlags(&ctx->back_stream, cudaStreamNonBlocking));
    for (cudaEvent_t& e : ctx->copy_ev) MIRROR_CUDA_OK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return MIRROR_OK;
}

// Pieces of a host-buffer step: layers [l0[c], l1[c]) are copied together and attended to in one launch, in this order.
//   - Without explicit hidden rows the LM head needs the last layer's output: that layer is a piece of its own, the first.
//   - What arrives while the LM head streams its weights (its time from the bytes and operations it moves; copies at 50 GB/s,
//     PCIe as measured) is one piece: it is attended to after the decision anyway, and one launch over 47 layers takes 94 us
//     where eleven launches took 300.
//   - The rest is attended to as it arrives.  A piece costs its three copies ~11 us of the link whatever their size and its
//     launch ~27 us of the GPU, so pieces start at 3 MB (the GPU has work 60 us later) and double up to 24 MB: 87 MB for 41
//     layers' short contexts took 1938 us in 28 pieces of 3 MB, and takes 1700.
struct HostPieces {
    int n = 0, l0[kHostChunks], l1[kHostChunks];
    void add(int a, int b) { if (b > a) { l0[n] = a; l1[n] = b; ++n; } }
};
HostPieces plan_pieces(int layers, bool last_first, double layer_bytes, double lm_bytes, double lm_flops) {
    constexpr double kCopyRate = 50e9, kPiece = 3e6;
    const double lm_s = lm_bytes / 6.4e12 > lm_flops / 1.2e15 ? lm_bytes / 6.4e12 : lm_flops / 1.2e15;
    HostPieces h;
    const int rest = last_first ? layers - 1 : layers;
    if (last_first) h.add(layers - 1, layers);
    int bulk = (int)(lm_s * kCopyRate / layer_bytes);
    if (bulk > rest || (rest - bulk) * layer_bytes < kPiece) bulk = rest;
    h.add(0, bulk);
    const double cap = std::max(8 * kPiece, (rest - bulk) * layer_bytes / (kHostChunks - 8));      // (there are only so many events)
    double size = kPiece;
    for (int at = bulk; at < rest;) {
        int take = std::max(1, (int)(size / layer_bytes));
        if ((rest - at - take) * layer_bytes < kPiece || h.n == kHostChunks - 1) take = rest - at;      // (no crumb at the end)
        h.add(at, at + take);
        at += take;
        size = std::min(2 * size, cap);
    }
    return h;
}

mirror_status verify_step_impl(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree, const void* q, const void* k_new,
                               const void* v_new, const void* hidden, const void* W, const mirror_accept_in* acc,
                               const mirror_accept_out* out, void* attn_out, int32_t* argmax_out, void* stream, const HostIO* io,
                               const MirrorAttnFp8* f8 = nullptr) {
    if (f8 && io) return MIRROR_ERR_UNSUPPORTED;          // (the host-buffer step takes the bf16 cache)
    if (!ctx || !kv || !tree || !q || !k_new || !v_new || !W || !acc || !out || !attn_out || !tree->tokens) return MIRROR_ERR_ARG;
    if (!out->n_accepted || !out->best_branch || !out->n_emitted || !out->emitted || !out->accepted_nodes ||
        !out->decide_row || !out->reuse_slot)
        return MIRROR_ERR_ARG;
    mirror_status st = check_kv(ctx, kv, tree);
    if (st != MIRROR_OK) return st;
    const bool spec = acc->mode == MIRROR_ACCEPT_SPEC_SAMPLING || acc->mode == MIRROR_ACCEPT_SPEC_TREE;
    if (!spec && acc->mode != MIRROR_ACCEPT_GREEDY) return MIRROR_ERR_ARG;
    if (spec && (!acc->u_accept || !acc->u_resample || (tree->n_nodes > 1 && !acc->q_probs))) return MIRROR_ERR_ARG;
    if (!hidden && ctx->desc.n_q_heads * ctx->desc.head_dim != ctx->desc.hidden) return MIRROR_ERR_SHAPE;
    MirrorTreeInfo ti;
    st = mirror_build_tree(tree, &ti);
    if (st != MIRROR_OK) return st;
    const size_t M = (size_t)tree->batch * tree->n_nodes;
    MirrorWsLayout L;
    mirror_ws_layout(ctx, M, &L, (size_t)tree->batch);
    if (!ctx->ws || ctx->ws_bytes < (spec ? L.end_logits : L.end_lmhead)) return MIRROR_ERR_WORKSPACE;
    MIRROR_CUDA_OK(cudaSetDevice(ctx->device));
    uint8_t* ws = (uint8_t*)ctx->ws;
    cudaStream_t s = (cudaStream_t)stream;

    // (host-buffer variant) pieces of layers, copied on the second stream and attended to in that order
    HostPieces pieces;
    const size_t q_layer = M * (size_t)ctx->desc.n_q_heads * ctx->desc.head_dim * 2;        // bytes per layer
    const size_t kv_layer = M * (size_t)ctx->desc.n_kv_heads * ctx->desc.head_dim * 2;
    auto attend_piece = [&](int c) -> mirror_status {
        MIRROR_CUDA_OK(cudaStreamWaitEvent(s, ctx->copy_ev[c], 0));
        const int l0 = pieces.l0[c], l1 = pieces.l1[c];
        mirror_kv kv_c = *kv;
        kv_c.k_pool = (const __nv_bfloat16*)kv->k_pool + (size_t)l0 * kv->layer_stride;
        kv_c.v_pool = (const __nv_bfloat16*)kv->v_pool + (size_t)l0 * kv->layer_stride;
        kv_c.num_layers = l1 - l0;
        return mirror_attn_launch(ctx, &kv_c, tree, ti, (const uint8_t*)q + l0 * q_layer, (const uint8_t*)k_new + l0 * kv_layer,
                                  (const uint8_t*)v_new + l0 * kv_layer, (uint8_t*)attn_out + l0 * q_layer, nullptr,
                                  (float*)(ws + L.attn_partial), s);
    };
    const bool ev = ctx->stage_ev_on && !io;
    if (ev) MIRROR_CUDA_OK(cudaEventRecord(ctx->stage_ev[0], s));
    // Hidden rows of the caller's own do not depend on the attention: the LM head is launched beside it (see lmhead_pair.cu), on the
    // SMs that the attention leaves or has done with.  The attention's merge then comes behind the LM head's: behind the decision where that
    // folds the row partials itself, else in front of the decision, which waits for it.
    const size_t attn_bytes = (size_t)kv->num_layers * q_layer;
    const bool w_apart = apart(W, (size_t)ctx->desc.vocab * ctx->desc.hidden * 2, attn_out, attn_bytes);
    const bool at_once = hidden && !io && !ev && (int)M >= ctx->tune.lm_pair_min_rows && w_apart &&
                         apart(hidden, M * (size_t)ctx->desc.hidden * 2, attn_out, attn_bytes);
    MirrorAttnBeside beside;
    if (at_once) {
        const double bytes_ns = 2.0 * ctx->desc.vocab * ctx->desc.hidden / 6400.0, flops_ns = bytes_ns * M * 6400.0 / 1.2e6;
        beside.work_ns = (float)std::max(bytes_ns, flops_ns);
        beside.stream = M <= 128;                            // (more rows: the tensor cores set the LM head's pace, too)
        beside.in_parts = ctx->desc.vocab > ctx->num_sms * 256;      // (a CTA pair per SM, units of up to 2 x 128 ids)
        st = mirror_attn_launch(ctx, kv, tree, ti, q, k_new, v_new, attn_out, nullptr, (float*)(ws + L.attn_partial), s, f8, false, &beside);
        if (st != MIRROR_OK) return st;
    } else if (!io) {
        st = mirror_attn_launch(ctx, kv, tree, ti, q, k_new, v_new, attn_out, nullptr, (float*)(ws + L.attn_partial), s, f8);
        if (st != MIRROR_OK) return st;
    } else {
        // Host inputs.  The layers' attention problems are independent of one another and the LM head reads only the last
        // layer's output (or rows of its own), so the decision comes first and the layers it does not need are copied on a
        // second stream meanwhile.  The copies start only after everything already queued on `stream` (the previous step may
        // still read the staging buffers).
        st = ensure_copy_stream(ctx);
        if (st != MIRROR_OK) return st;
        cudaStream_t cs = ctx->copy_stream;
        MIRROR_CUDA_OK(cudaEventRecord(ctx->copy_ev[kEvBegin], s));
        MIRROR_CUDA_OK(cudaStreamWaitEvent(cs, ctx->copy_ev[kEvBegin], 0));
        MIRROR_CUDA_OK(cudaMemcpyAsync((void*)tree->tokens, io->h_tokens, M * sizeof(int32_t), cudaMemcpyHostToDevice, cs));
        MIRROR_CUDA_OK(cudaEventRecord(ctx->copy_ev[kEvTokens], cs));
        pieces = plan_pieces(kv->num_layers, hidden == nullptr, (double)(q_layer + 2 * kv_layer), 2.0 * ctx->desc.vocab * ctx->desc.hidden,
                             2.0 * M * ctx->desc.vocab * ctx->desc.hidden);
        for (int c = 0; c < pieces.n; ++c) {
            const size_t l0 = (size_t)pieces.l0[c], nl = (size_t)(pieces.l1[c] - pieces.l0[c]);
            MIRROR_CUDA_OK(cudaMemcpyAsync((uint8_t*)q + l0 * q_layer, (const uint8_t*)io->h_q + l0 * q_layer, nl * q_layer,
                                           cudaMemcpyHostToDevice, cs));
            MIRROR_CUDA_OK(cudaMemcpyAsync((uint8_t*)k_new + l0 * kv_layer, (const uint8_t*)io->h_k_new + l0 * kv_layer, nl * kv_layer,
                                           cudaMemcpyHostToDevice, cs));
            MIRROR_CUDA_OK(cudaMemcpyAsync((uint8_t*)v_new + l0 * kv_layer, (const uint8_t*)io->h_v_new + l0 * kv_layer, nl * kv_layer,
                                           cudaMemcpyHostToDevice, cs));
            MIRROR_CUDA_OK(cudaEventRecord(ctx->copy_ev[c], cs));
        }
        if (!hidden) {
            st = attend_piece(0);
            if (st != MIRROR_OK) return st;
        }
    }
    if (ev) MIRROR_CUDA_OK(cudaEventRecord(ctx->stage_ev[1], s));

    // (Its weights may be requested early: behind an attention launch, which waits for all before it, nothing of the caller's can
    // still be writing them; nor does the attention, unless they lie in its output.)
    // LM-head rows: the given hidden states, else the last layer's attention output ([B*n, Hq*d] == [M, H])
    const void* rows = hidden;
    if (!rows) {
        const size_t layer_elems = M * (size_t)ctx->desc.n_q_heads * ctx->desc.head_dim;
        rows = (const __nv_bfloat16*)attn_out + (size_t)(kv->num_layers - 1) * layer_elems;
    }
    int32_t* d_argmax = argmax_out ? argmax_out : (int32_t*)(ws + L.argmax);
    float* d_lse = (float*)(ws + L.lse);
    float* d_logits = spec ? (float*)(ws + L.logits) : nullptr;
    // greedy: the acceptance kernel folds the GEMM's row partials itself, a block per request.  (Up to 256 rows the GEMM leaves
    // a partial per CTA, ~10 loads per lane; beyond, one per 128 vocabulary ids, and a block per row is worth its launch.)
    MirrorLmPartials partials;
    const bool defer = !spec && M <= 256;
    st = mirror_lmhead_launch(ctx, rows, (int)M, W, 0, nullptr, nullptr, 0, d_argmax, nullptr, spec ? d_lse : nullptr, nullptr,
                              nullptr, nullptr, d_logits, ws + L.lm_partial, L.lm_partial_bytes, d_lse, s,
                              ev ? ctx->stage_ev[2] : nullptr, nullptr, nullptr, 0, defer ? &partials : nullptr,
                              beside.granted ? MIRROR_LM_AT_ONCE : io || !w_apart ? MIRROR_LM_AFTER : MIRROR_LM_WEIGHTS_EARLY);
    if (st != MIRROR_OK) return st;

    // The attention's merge, beside the kernel that folds the row partials, or (below) beside the acceptance that folds them itself.
    // (The draws of the other acceptance kernels leave it no registers: behind them it took 15 us more.)
    if (!defer) st = mirror_attn_late_merge(ctx, beside, s);
    if (st != MIRROR_OK) return st;

    if (io) MIRROR_CUDA_OK(cudaStreamWaitEvent(s, ctx->copy_ev[kEvTokens], 0));
    mirror_accept_in in = *acc;
    in.target_argmax = d_argmax;
    in.logits = d_logits;
    in.lse = d_lse;
    // the tree rule keeps its running distribution in the workspace when the caller sized it for that
    double* tree_scratch = (acc->mode == MIRROR_ACCEPT_SPEC_TREE && ctx->ws_bytes >= L.end_accept) ? (double*)(ws + L.accept_scratch) : nullptr;
    st = mirror_accept_launch(ctx, tree, ti, &in, out, s, tree_scratch, defer ? &partials : nullptr, d_argmax);
    if (st != MIRROR_OK) return st;
    if (defer) st = mirror_attn_late_merge(ctx, beside, s);
    if (st != MIRROR_OK) return st;
    if (ev) MIRROR_CUDA_OK(cudaEventRecord(ctx->stage_ev[3], s));
    const mirror_accept_host_out* h = io ? io->h_out : nullptr;
    if (h) {
        // the decision goes back on a stream of its own: four short copies would hold the attention up by ~10 us
        const size_t B = (size_t)tree->batch;
        cudaStream_t bs = ctx->back_stream;
        MIRROR_CUDA_OK(cudaEventRecord(ctx->copy_ev[kEvDecided], s));
        MIRROR_CUDA_OK(cudaStreamWaitEvent(bs, ctx->copy_ev[kEvDecided], 0));
        if (h->n_accepted) MIRROR_CUDA_OK(cudaMemcpyAsync(h->n_accepted, out->n_accepted, B * 4, cudaMemcpyDeviceToHost, bs));
        if (h->best_branch) MIRROR_CUDA_OK(cudaMemcpyAsync(h->best_branch, out->best_branch, B * 4, cudaMemcpyDeviceToHost, bs));
        if (h->n_emitted) MIRROR_CUDA_OK(cudaMemcpyAsync(h->n_emitted, out->n_emitted, B * 4, cudaMemcpyDeviceToHost, bs));
        if (h->emitted) MIRROR_CUDA_OK(cudaMemcpyAsync(h->emitted, out->emitted, B * (size_t)(tree->gamma + 1) * 4, cudaMemcpyDeviceToHost, bs));
        MIRROR_CUDA_OK(cudaEventRecord(ctx->copy_ev[kEvSent], bs));
    }
    for (int c = hidden ? 0 : 1; c < pieces.n; ++c) {
        st = attend_piece(c);
        if (st != MIRROR_OK) return st;
    }
    if (h) MIRROR_CUDA_OK(cudaStreamWaitEvent(s, ctx->copy_ev[kEvSent], 0));
    return MIRROR_OK;
}

}  // namespace

extern "C" mirror_status mirror_verify_step(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree,
                                            const void* q, const void* k_new, const void* v_new, const void* hidden,
                                            const void* W, const mirror_accept_in* acc, const mirror_accept_out* out,
                                            void* attn_out, int32_t* argmax_out, void* stream) {
    return verify_step_impl(ctx, kv, tree, q, k_new, v_new, hidden, W, acc, out, attn_out, argmax_out, stream, nullptr);
}

extern "C" mirror_status mirror_verify_step_fp8(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree, const void* q,
                                                const void* k_new_fp8, const void* v_new_fp8, const float* k_scale,
                                                const float* v_scale, float q_scale, const void* hidden, const void* W,
                                                const mirror_accept_in* acc, const mirror_accept_out* out, void* attn_out,
                                                int32_t* argmax_out, void* stream) {
    if (!k_scale || !v_scale || !(q_scale > 0.f)) return MIRROR_ERR_ARG;
    if (ctx && ctx->desc.head_dim != 128) return MIRROR_ERR_UNSUPPORTED;
    const MirrorAttnFp8 f8 = {k_scale, v_scale, q_scale};
    return verify_step_impl(ctx, kv, tree, q, k_new_fp8, v_new_fp8, hidden, W, acc, out, attn_out, argmax_out, stream, nullptr, &f8);
}

extern "C" mirror_status mirror_verify_step_host(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree, const void* h_q,
                                                 const void* h_k_new, const void* h_v_new, const int32_t* h_tokens, void* d_q,
                                                 void* d_k_new, void* d_v_new, const void* hidden, const void* W,
                                                 const mirror_accept_in* acc, const mirror_accept_out* out,
                                                 const mirror_accept_host_out* h_out, void* attn_out, void* stream) {
    if (!h_q || !h_k_new || !h_v_new || !h_tokens) return MIRROR_ERR_ARG;
    HostIO io{h_q, h_k_new, h_v_new, h_tokens, h_out};
    return verify_step_impl(ctx, kv, tree, d_q, d_k_new, d_v_new, hidden, W, acc, out, attn_out, nullptr, stream, &io);
}

extern "C" mirror_status mirror_set_stage_events(mirror_ctx* ctx, void* const* events4) {
    if (!ctx) return MIRROR_ERR_ARG;
    ctx->stage_ev_on = false;
    if (!events4) return MIRROR_OK;
    for (int i = 0; i < 4; ++i) {
        if (!events4[i]) return MIRROR_ERR_ARG;
        ctx->stage_ev[i] = (cudaEvent_t)events4[i];
    }
    ctx->stage_ev_on = true;
    return MIRROR_OK;
}
