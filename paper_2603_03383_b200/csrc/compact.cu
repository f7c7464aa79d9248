// In-place KV compaction of the accepted path (Section 3.2, "Zero-Copy Retrieval",
// applied to the K/V rows): row seq_len + acc_nodes[j] -> row seq_len + j for
// j = 1..accept_len, every layer and KV head, then seq_len += accept_len + 1.
#include "common.cuh"

namespace mtv {

// grid = (Hkv, B, n_layers).  A source row of step j may be the destination of a later
// step j' (acc_nodes = [0,2,..]: j=1 reads slot 2, j=2 writes slot 2), so the block
// stages every source row in shared memory before it writes anything.
__global__ void __launch_bounds__(256)
kv_compact_kernel(int T, int K, int D, int Lcap, __nv_bfloat16 *const *__restrict__ k_caches,
                  __nv_bfloat16 *const *__restrict__ v_caches, int64_t sb, int64_t sh, int64_t st,
                  const int32_t *__restrict__ seq_lens, const int32_t *__restrict__ accept_len,
                  const int32_t *__restrict__ acc_nodes, int32_t *__restrict__ dev_error) {
    __shared__ uint4 stage[2 * MTV_MAX_K * 16];  // [k|v][j][D/8 <= 16]
    const int g = blockIdx.x, b = blockIdx.y, layer = blockIdx.z;
    let_next_start();
    previous_done();
    const int L = seq_lens[b];
    const int n = accept_len[b];
    if (L + T > Lcap || n <= 0) return;
    if (!MTV_INDEX_OK(n, K + 1, dev_error)) return;      // accept_len comes from the caller's device memory
    const int vec = D / 8;
    __nv_bfloat16 *kc = k_caches[layer] + b * sb + g * sh;
    __nv_bfloat16 *vc = v_caches[layer] + b * sb + g * sh;
    const int total = 2 * n * vec;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int which = e / (n * vec), j = (e / vec) % n, c = e % vec;
        const int node = acc_nodes[(size_t)b * (K + 1) + j + 1];
        const int src = L + node;
        const __nv_bfloat16 *base = which ? vc : kc;
        stage[e] = MTV_INDEX_OK(node, T, dev_error) ? *reinterpret_cast<const uint4 *>(base + (int64_t)src * st + c * 8)
                                                    : make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int which = e / (n * vec), j = (e / vec) % n, c = e % vec;
        __nv_bfloat16 *base = which ? vc : kc;
        if (!MTV_INDEX_OK(acc_nodes[(size_t)b * (K + 1) + j + 1], T, dev_error)) continue;   // a row that was not read is not written
        *reinterpret_cast<uint4 *>(base + (int64_t)(L + j + 1) * st + c * 8) = stage[e];
    }
}

// Acceptance, compaction and the advance of seq_lens of a whole step in one launch: three launches of 1 to 3 us each, one
// waiting for the other, were 8 us of every step.  grid = (Hkv, B, layer groups); every block works the acceptance of its
// sequence out for itself (T nodes' keys from L2, the paths' scores), the first one writes it down, and the last block of
// a sequence to have read its length (ticket, nobody waits) advances it.
__global__ void __launch_bounds__(256)
accept_compact_kernel(int T, int K, int P, int ns, int D, int Lcap, int n_layers, int layers_per_block,
                      const unsigned long long *__restrict__ part, const int32_t *__restrict__ tree_tok,
                      const int32_t *__restrict__ ri, __nv_bfloat16 *const *__restrict__ k_caches,
                      __nv_bfloat16 *const *__restrict__ v_caches, int64_t sb, int64_t sh, int64_t st, int32_t *seq_lens,
                      int32_t *__restrict__ accept_len, int32_t *__restrict__ best_path, int32_t *__restrict__ acc_nodes,
                      int32_t *__restrict__ acc_tok, int32_t *__restrict__ next_root, int32_t *__restrict__ status,
                      int32_t *tickets, int32_t *gate, int32_t *__restrict__ dev_error) {
    __shared__ int32_t am[MTV_MAX_T], tok[MTV_MAX_T], node_of[MTV_MAX_K + 1];
    __shared__ unsigned int best_key;
    __shared__ uint4 stage[2 * MTV_MAX_K * 16];  // [k|v][j][D/8 <= 16]
    let_next_start();
    const int g = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
    if (tid == 0) best_key = 0;
    previous_done();
    if (tid == 0 && g == 0 && b == 0 && blockIdx.z == 0) *gate = 0;      // every kernel that waits at it is complete
    const int L = seq_lens[b];
    // two threads per node take turns over its keys
    const int i = tid >> 1;
    unsigned long long best = 0;
    if (i < T) {
        const unsigned long long *x = part + ((size_t)b * T + i) * ns;
#pragma unroll 4
        for (int s = tid & 1; s < ns; s += 2) best = x[s] > best ? x[s] : best;
    }
    const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, 1);
    if (i < T && (tid & 1) == 0) {
        best = other > best ? other : best;
        am[i] = (int32_t)(0xffffffffu - (uint32_t)(best & 0xffffffffu));
        tok[i] = tree_tok[(size_t)b * T + i];
    }
    __syncthreads();
    // key = len * 256 + (255 - p): max() picks the longest match, then the lowest path
    for (int p = tid; p < P; p += blockDim.x) {
        const int32_t *path = ri + (size_t)p * (K + 1);
        int len = 0;
        for (int j = 1; j <= K; ++j) {
            const int node = path[j];
            if (node < 0) break;
            if (!MTV_INDEX_OK(node, T, dev_error) || !MTV_INDEX_OK(path[j - 1], T, dev_error)) break;
            if (tok[node] != am[path[j - 1]]) break;
            len = j;
        }
        atomicMax(&best_key, (unsigned)len * 256u + (255u - (unsigned)p));
    }
    __syncthreads();
    const int n = best_key / 256, bp = 255 - (int)(best_key % 256);
    if (tid <= K) {
        int node = tid <= n ? ri[(size_t)bp * (K + 1) + tid] : -1;
        if (node >= 0 && !MTV_INDEX_OK(node, T, dev_error)) node = -1;
        node_of[tid] = node;
        if (g == 0 && blockIdx.z == 0) {
            acc_nodes[(size_t)b * (K + 1) + tid] = node;
            acc_tok[(size_t)b * (K + 1) + tid] = node >= 0 ? tok[node] : -1;
            if (tid == n && node >= 0) next_root[b] = am[node];
            if (tid == 0) { accept_len[b] = n; best_path[b] = bp; }
        }
    }
    __syncthreads();
    const bool fits = L + T <= Lcap;
    const int vec = D / 8, total = fits ? 2 * n * vec : 0, l0 = (int)blockIdx.z * layers_per_block;
    for (int layer = l0; layer < min(n_layers, l0 + layers_per_block) && total > 0; ++layer) {
        __nv_bfloat16 *kc = k_caches[layer] + b * sb + g * sh, *vc = v_caches[layer] + b * sb + g * sh;
        for (int e = tid; e < total; e += blockDim.x) {         // all sources before any row is written
            const int which = e / (n * vec), j = (e / vec) % n, c = e % vec, node = node_of[j + 1];
            if (node >= 0) stage[e] = *reinterpret_cast<const uint4 *>((which ? vc : kc) + (int64_t)(L + node) * st + c * 8);
        }
        __syncthreads();
        for (int e = tid; e < total; e += blockDim.x) {
            const int which = e / (n * vec), j = (e / vec) % n, c = e % vec;
            if (node_of[j + 1] >= 0) *reinterpret_cast<uint4 *>((which ? vc : kc) + (int64_t)(L + j + 1) * st + c * 8) = stage[e];
        }
        __syncthreads();
    }
    if (tid != 0) return;
    __threadfence();             // this block has read the length: before its ticket says so
    if (atomicAdd(&tickets[b], 1) == (int)(gridDim.x * gridDim.z) - 1) {
        __threadfence();
        if (status) status[b] = fits ? MTV_OK : MTV_ERR_CAPACITY;
        if (fits) seq_lens[b] = L + n + 1;
    }
}

int accept_compact(const mtv_tree *tree, const mtv_step_args *a, int ns, const unsigned long long *part, int32_t *tickets,
                   const Gate &gate, cudaStream_t stream) {
    if (!a->tree_tok || !a->accept_len || !a->best_path || !a->acc_nodes || !a->acc_tok || !a->next_root || !a->k_caches || !a->v_caches ||
        !a->seq_lens || a->B < 1 || a->Hkv < 1 || a->n_layers < 1 || a->Lcap < 1)
        return MTV_ERR_INVALID_ARG;
    if (tree->P > 255 || (a->D != 64 && a->D != 128) || a->B > 65535 || a->n_layers > 65535) return MTV_ERR_UNSUPPORTED_SHAPE;
    if (a->stride_t % 8 || a->stride_h % 8 || a->stride_b % 8) return MTV_ERR_INVALID_ARG;
    // as many layers per block as leave about eight blocks per SM: each repeats the acceptance
    int per = (int)((long)a->Hkv * a->B * a->n_layers / (8L * sm_count()));
    per = per < 1 ? 1 : per > a->n_layers ? a->n_layers : per;
    TapScope tap(MTV_KERNEL_KV_COMPACT, stream);
    MTV_CUDA_CHECK(launch_dependent(accept_compact_kernel, dim3(a->Hkv, a->B, (a->n_layers + per - 1) / per), 256, 0, stream, tree->T,
                                    tree->K, tree->P, ns, a->D, a->Lcap, a->n_layers, per, part, a->tree_tok, tree->d_retrieve,
                                    reinterpret_cast<__nv_bfloat16 *const *>(a->k_caches),
                                    reinterpret_cast<__nv_bfloat16 *const *>(a->v_caches), a->stride_b, a->stride_h, a->stride_t,
                                    a->seq_lens, a->accept_len, a->best_path, a->acc_nodes, a->acc_tok, a->next_root, a->status,
                                    tickets, gate.word, tree->d_error));
    return MTV_OK;
}

// Runs after every compaction block has read seq_lens (next kernel on the stream).
__global__ void seq_lens_advance_kernel(int B, int T, int Lcap, int32_t *seq_lens, const int32_t *accept_len,
                                        int32_t *status, int K, int32_t *dev_error) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    let_next_start();
    previous_done();
    if (b >= B) return;
    const int L = seq_lens[b];
    if (L + T > Lcap) {
        if (status) status[b] = MTV_ERR_CAPACITY;
        return;
    }
    if (status) status[b] = MTV_OK;
    if (!MTV_INDEX_OK(accept_len[b], K + 1, dev_error)) return;
    seq_lens[b] = L + accept_len[b] + 1;
}

}  // namespace mtv

extern "C" int kv_compact_accepted(const mtv_tree_t *tree, int B, int Hkv, int D, int n_layers,
                                   mtv_bf16 *const *k_caches, mtv_bf16 *const *v_caches,
                                   int64_t stride_b, int64_t stride_h, int64_t stride_t, int Lcap,
                                   int32_t *seq_lens, const int32_t *accept_len, const int32_t *acc_nodes,
                                   int32_t *status, void *stream) {
    using namespace mtv;
    MTV_RANGE("kv_compact_accepted");
    if (!tree || !k_caches || !v_caches || !seq_lens || !accept_len || !acc_nodes || B < 1 || Hkv < 1 ||
        n_layers < 1 || Lcap < 1)
        return MTV_ERR_INVALID_ARG;
    if (D != 64 && D != 128) return MTV_ERR_UNSUPPORTED_SHAPE;
    if (stride_t % 8 || stride_h % 8 || stride_b % 8) return MTV_ERR_INVALID_ARG;
    if (B > 65535 || n_layers > 65535) return MTV_ERR_UNSUPPORTED_SHAPE;
    cudaStream_t st = (cudaStream_t)stream;
    {
        TapScope tap(MTV_KERNEL_KV_COMPACT, st);
        MTV_CUDA_CHECK(launch_dependent(kv_compact_kernel, dim3(Hkv, B, n_layers), 256, 0, st, tree->T, tree->K, D, Lcap,
                                        reinterpret_cast<__nv_bfloat16 *const *>(k_caches),
                                        reinterpret_cast<__nv_bfloat16 *const *>(v_caches), stride_b, stride_h, stride_t, seq_lens,
                                        accept_len, acc_nodes, tree->d_error));
    }
    TapScope tap(MTV_KERNEL_SEQ_ADVANCE, st);
    MTV_CUDA_CHECK(launch_dependent(seq_lens_advance_kernel, dim3((B + 127) / 128), 128, 0, st, B, tree->T, Lcap, seq_lens, accept_len,
                                    status, tree->K, tree->d_error));
    MTV_CUDA_CHECK(cudaGetLastError());
    return MTV_OK;
}
