// Roll-forward of the paged KV cache after a verify step (Sec. 3.1: the target commits the accepted prefix of the
// window and rolls its state forward): the K/V rows of the root and of the accepted nodes of the chosen branch, in
// path order, become tokens prefix_len .. prefix_len + A of every layer and KV head, and the prefix grows by A + 1.
// Pure data movement: 2 * L * (A + 1) * Hkv * d bf16 values per request.
#include "mirror_internal.h"

namespace {

struct CommitParams {
    int L, B, n, Hkv, d, gamma, max_pages, num_pages;
    int advance;                          // 1: a block has all layers of its request, and moves the prefix itself
    long long layer_stride;               // elements between the layers' pools
    __nv_bfloat16* k_pool;
    __nv_bfloat16* v_pool;
    const __nv_bfloat16* k_new;           // [L, B, n, Hkv, d]
    const __nv_bfloat16* v_new;
    const int32_t* page_table;
    int32_t* prefix_len;
    const int32_t* accepted_nodes;        // [B, gamma]
    const int32_t* n_accepted;            // [B]
    int* status;
};

// grid (L, B), or (1, B) when a request has so little to copy (16-byte accesses) that one block does it in a few steps: then the
// prefix can be moved here as well, which saves the second launch (a third of the time for a toy model).
__global__ void __launch_bounds__(256) kv_commit_kernel(const CommitParams p) {
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    const int b = blockIdx.y;
    int A = p.n_accepted[b];
    if (A < 0 || A > p.gamma) { if (threadIdx.x == 0 && atomicCAS(p.status, 0, MIRROR_DEV_CHECK) == 0) atomicExch(p.status + 1, 800); A = 0; }
    const int len = p.prefix_len[b];
    const int chunks_per_row = p.d / 8;                       // 16-byte chunks of one (token, head) row
    const int per_layer = (A + 1) * p.Hkv * chunks_per_row, total = p.advance ? p.L * per_layer : per_layer;
    for (int k = threadIdx.x; k < total; k += blockDim.x) {
        const int layer = blockIdx.x + k / per_layer, i = k % per_layer;
        const int cc = i % chunks_per_row, h = (i / chunks_per_row) % p.Hkv, j = i / (chunks_per_row * p.Hkv);
        const int node = (j == 0) ? 0 : p.accepted_nodes[(size_t)b * p.gamma + j - 1];
        const int pos = len + j;
        bool ok = len >= 0 && node >= 0 && node < p.n && pos < p.max_pages * 16;
        int page = ok ? p.page_table[(size_t)b * p.max_pages + pos / 16] : -1;
        ok = ok && page >= 0 && page < p.num_pages;
        if (!ok) {                                            // reported, not written
            if (atomicCAS(p.status, 0, MIRROR_DEV_CHECK) == 0) atomicExch(p.status + 1, 801);
            continue;
        }
        const size_t src = ((((size_t)layer * p.B + b) * p.n + node) * p.Hkv + h) * p.d + cc * 8;
        const size_t dst = (size_t)layer * p.layer_stride + (((size_t)page * p.Hkv + h) * 16 + pos % 16) * p.d + cc * 8;
        *reinterpret_cast<uint4*>(p.k_pool + dst) = *reinterpret_cast<const uint4*>(p.k_new + src);
        *reinterpret_cast<uint4*>(p.v_pool + dst) = *reinterpret_cast<const uint4*>(p.v_new + src);
    }
    if (p.advance) {
        __syncthreads();                                      // (every thread has read the old length)
        if (threadIdx.x == 0) p.prefix_len[b] = len + A + 1;
    }
}

// after every layer has read the old lengths
__global__ void kv_advance_kernel(int B, int gamma, const int32_t* n_accepted, int32_t* prefix_len) {
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const int A = n_accepted[b];
    prefix_len[b] += ((A < 0 || A > gamma) ? 0 : A) + 1;
}

}  // namespace

// elem_bytes 2: bf16 cache.  1: e4m3 codes; a row of d codes is moved as d / 2 16-bit units, the layout is the same.
static mirror_status kv_commit_impl(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree, const void* k_new,
                                    const void* v_new, const int32_t* accepted_nodes, const int32_t* n_accepted,
                                    int32_t* prefix_len, void* stream, int elem_bytes) {
    if (!ctx || !kv || !tree || !k_new || !v_new || !accepted_nodes || !n_accepted || !prefix_len) return MIRROR_ERR_ARG;
    if (!kv->k_pool || !kv->v_pool || !kv->page_table) return MIRROR_ERR_ARG;
    if (tree->batch <= 0 || tree->n_nodes <= 0 || tree->n_nodes > MIRROR_MAX_NODES || tree->gamma < 0 || tree->gamma > MIRROR_MAX_DEPTH)
        return MIRROR_ERR_SHAPE;
    if (kv->num_layers <= 0 || kv->num_pages <= 0 || kv->max_pages_per_req <= 0) return MIRROR_ERR_ARG;
    if (((uintptr_t)k_new & 15) || ((uintptr_t)v_new & 15) || ((uintptr_t)kv->k_pool & 15) || ((uintptr_t)kv->v_pool & 15)) return MIRROR_ERR_ARG;
    MIRROR_CUDA_OK(cudaSetDevice(ctx->device));
    CommitParams p;
    p.L = kv->num_layers; p.B = tree->batch; p.n = tree->n_nodes; p.Hkv = ctx->desc.n_kv_heads;
    p.d = ctx->desc.head_dim * elem_bytes / 2;
    if (kv->layer_stride * elem_bytes % 2 != 0) return MIRROR_ERR_SHAPE;
    p.gamma = tree->gamma; p.max_pages = kv->max_pages_per_req; p.num_pages = kv->num_pages;
    p.layer_stride = kv->layer_stride * elem_bytes / 2;
    p.k_pool = (__nv_bfloat16*)const_cast<void*>(kv->k_pool);
    p.v_pool = (__nv_bfloat16*)const_cast<void*>(kv->v_pool);
    p.k_new = (const __nv_bfloat16*)k_new; p.v_new = (const __nv_bfloat16*)v_new;
    p.page_table = kv->page_table; p.prefix_len = prefix_len;
    p.accepted_nodes = accepted_nodes; p.n_accepted = n_accepted;
    p.status = ctx->d_status;
    cudaStream_t s = (cudaStream_t)stream;
    p.advance = (long long)p.L * (p.gamma + 1) * p.Hkv * (p.d / 8) <= 4 * 256;
    MIRROR_CUDA_OK(mirror_launch_pdl(kv_commit_kernel, dim3(p.advance ? 1u : (unsigned)p.L, (unsigned)p.B), dim3(256), 0, s, p));
    ctx->launches += 1;
    if (!p.advance) MIRROR_CUDA_OK(mirror_launch_pdl(kv_advance_kernel, dim3((unsigned)((p.B + 127) / 128)), dim3(128), 0, s, p.B, p.gamma, n_accepted, prefix_len));
    if (!p.advance) ctx->launches += 1;
    MIRROR_CUDA_OK(cudaGetLastError());
    return MIRROR_OK;
}

extern "C" mirror_status mirror_kv_commit(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree, const void* k_new,
                                          const void* v_new, const int32_t* accepted_nodes, const int32_t* n_accepted,
                                          int32_t* prefix_len, void* stream) {
    return kv_commit_impl(ctx, kv, tree, k_new, v_new, accepted_nodes, n_accepted, prefix_len, stream, 2);
}

extern "C" mirror_status mirror_kv_commit_fp8(mirror_ctx* ctx, const mirror_kv* kv, const mirror_tree* tree, const void* k_new_fp8,
                                              const void* v_new_fp8, const int32_t* accepted_nodes, const int32_t* n_accepted,
                                              int32_t* prefix_len, void* stream) {
    return kv_commit_impl(ctx, kv, tree, k_new_fp8, v_new_fp8, accepted_nodes, n_accepted, prefix_len, stream, 1);
}
