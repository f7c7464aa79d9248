// Tree K/V append with rotary embedding — the step just before the tree attention
// (Section 3.2: tree_indices maps the flattened tree nodes to their positions).  Node i of
// sequence b sits at position seq_lens[b] + depth[i]; its rotated K row and its V row go to cache
// row seq_lens[b] + i, its query is rotated in place.
//
// Bound by memory: per node and layer Hq rows are read and written, 2 Hkv rows read and 2 Hkv written.  What kept it from
// that was the double-precision sine and cosine (positions reach tens of thousands of radians), computed anew for every
// layer, and 2-byte accesses.  A block now takes one node of one sequence for several layers, so that its angles are
// computed once, and moves 16-byte chunks: 32 layers of two sequences with 28 / 4 heads (75 MB) took 28 us
// and take 15.7 (4.8 TB/s).
#include "common.cuh"

namespace mtv {

constexpr int ROPE_THREADS = 256;

__device__ __forceinline__ void rope_rotate8(uint4 &a, uint4 &b, const float *cs, const float *sn) {
    uint32_t *wa = reinterpret_cast<uint32_t *>(&a), *wb = reinterpret_cast<uint32_t *>(&b);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const __nv_bfloat162 x = *reinterpret_cast<__nv_bfloat162 *>(&wa[k]), y = *reinterpret_cast<__nv_bfloat162 *>(&wb[k]);
        const float2 x1 = __bfloat1622float2(x), x2 = __bfloat1622float2(y);
        const float2 c = *reinterpret_cast<const float2 *>(cs + 2 * k), s = *reinterpret_cast<const float2 *>(sn + 2 * k);
        const __nv_bfloat162 o1 = __floats2bfloat162_rn(x1.x * c.x - x2.x * s.x, x1.y * c.y - x2.y * s.y);
        const __nv_bfloat162 o2 = __floats2bfloat162_rn(x2.x * c.x + x1.x * s.x, x2.y * c.y + x1.y * s.y);
        wa[k] = *reinterpret_cast<const uint32_t *>(&o1);
        wb[k] = *reinterpret_cast<const uint32_t *>(&o2);
    }
}

// grid = (T, B, layer groups).  One layer (caches given directly) or all layers of a step in one launch (caches through
// the device pointer arrays of kv_compact_accepted; q, k_new, v_new then hold the layers back to back).
__global__ void __launch_bounds__(ROPE_THREADS)
tree_kv_append_rope_kernel(int T, int Hq, int Hkv, int D, int Lcap, int n_layers, int layers_per_block, __nv_bfloat16 *__restrict__ q,
                           const __nv_bfloat16 *__restrict__ k_new, const __nv_bfloat16 *__restrict__ v_new,
                           __nv_bfloat16 *__restrict__ k_cache, __nv_bfloat16 *__restrict__ v_cache,
                           __nv_bfloat16 *const *__restrict__ k_caches, __nv_bfloat16 *const *__restrict__ v_caches,
                           int64_t sb, int64_t sh, int64_t st, const int32_t *__restrict__ seq_lens,
                           const int32_t *__restrict__ depth, double log2_theta, int32_t *__restrict__ status) {
    __shared__ __align__(16) float cs[64], sn[64];   // D / 2 <= 64
    const int i = blockIdx.x, b = blockIdx.y, B = gridDim.y;
    previous_done();
    let_next_start();
    const int L = seq_lens[b];
    if (L + T > Lcap) {
        if (status && i == 0 && threadIdx.x == 0) status[b] = MTV_ERR_CAPACITY;
        return;
    }
    if (status && i == 0 && threadIdx.x == 0) status[b] = MTV_OK;
    const int half = D / 2;
    if ((int)threadIdx.x < half) {
        const double pos = (double)L + (double)depth[i];
        const double ang = pos * exp2(-2.0 * threadIdx.x / D * log2_theta);
        double s, c;
        sincos(ang, &s, &c);
        cs[threadIdx.x] = (float)c;
        sn[threadIdx.x] = (float)s;
    }
    __syncthreads();
    // A thread takes two chunks of 8 columns of a row, half a row apart: D / 16 threads per row, rows of a layer in the
    // order queries, keys, values.
    const int per_row = D / 16, shift = D == 128 ? 3 : 2;
    const int c = threadIdx.x & (per_row - 1), rows = Hq + 2 * Hkv;
    const int l_end = min(n_layers, ((int)blockIdx.z + 1) * layers_per_block);
    const int n_rows = (l_end - (int)blockIdx.z * layers_per_block) * rows;
    for (int e = threadIdx.x >> shift; e < n_rows; e += ROPE_THREADS >> shift) {
        const int layer = (int)blockIdx.z * layers_per_block + e / rows, h = e % rows;
        const size_t node = ((size_t)layer * B + b) * T + i;
        const __nv_bfloat16 *src;
        __nv_bfloat16 *dst;
        if (h < Hq) {
            dst = q + (node * Hq + h) * D;
            src = dst;
        } else {
            const bool is_v = h >= Hq + Hkv;
            const int g = h - Hq - (is_v ? Hkv : 0);
            src = (is_v ? v_new : k_new) + (node * Hkv + g) * D;
            dst = k_caches ? (is_v ? v_caches : k_caches)[layer] : (is_v ? v_cache : k_cache);
            dst += b * sb + g * sh + (int64_t)(L + i) * st;
        }
        const bool aligned = (((uintptr_t)src | (uintptr_t)dst) & 15) == 0;   // else element by element
        uint4 x1, x2;
        if (aligned) {
            x1 = *reinterpret_cast<const uint4 *>(src + c * 8);
            x2 = *reinterpret_cast<const uint4 *>(src + half + c * 8);
        } else {
            for (int k = 0; k < 8; ++k) {
                reinterpret_cast<__nv_bfloat16 *>(&x1)[k] = src[c * 8 + k];
                reinterpret_cast<__nv_bfloat16 *>(&x2)[k] = src[half + c * 8 + k];
            }
        }
        if (h < Hq + Hkv) rope_rotate8(x1, x2, cs + c * 8, sn + c * 8);
        if (aligned) {
            *reinterpret_cast<uint4 *>(dst + c * 8) = x1;
            *reinterpret_cast<uint4 *>(dst + half + c * 8) = x2;
        } else {
            for (int k = 0; k < 8; ++k) {
                dst[c * 8 + k] = reinterpret_cast<const __nv_bfloat16 *>(&x1)[k];
                dst[half + c * 8 + k] = reinterpret_cast<const __nv_bfloat16 *>(&x2)[k];
            }
        }
    }
}

// Enough blocks to fill the device a few times over, as many layers per block as that leaves.
static dim3 rope_grid(int T, int B, int n_layers, int *layers_per_block) {
    const long blocks = (long)T * B * n_layers;
    long per = blocks / (6L * sm_count());
    per = per < 1 ? 1 : per > n_layers ? n_layers : per;
    *layers_per_block = (int)per;
    return dim3(T, B, (n_layers + per - 1) / per);
}

}  // namespace mtv

extern "C" int tree_kv_append_rope(const mtv_tree_t *tree, int B, int Hq, int Hkv, int D, mtv_bf16 *q,
                                   const mtv_bf16 *k_new, const mtv_bf16 *v_new, mtv_bf16 *k_cache, mtv_bf16 *v_cache,
                                   int64_t stride_b, int64_t stride_h, int64_t stride_t, int Lcap,
                                   const int32_t *seq_lens, float rope_theta, int32_t *status, void *stream) {
    using namespace mtv;
    MTV_RANGE("tree_kv_append_rope");
    if (!tree || !tree->on_device || !q || !k_new || !v_new || !k_cache || !v_cache || !seq_lens) return MTV_ERR_INVALID_ARG;
    if (B < 1 || Hq < 1 || Hkv < 1 || Lcap < tree->T || rope_theta < 0.f) return MTV_ERR_INVALID_ARG;
    if ((D != 64 && D != 128) || B > 65535) return MTV_ERR_UNSUPPORTED_SHAPE;
    const double theta = rope_theta == 0.f ? 10000.0 : (double)rope_theta;
    int per = 1;
    const dim3 grid = rope_grid(tree->T, B, 1, &per);
    MTV_CUDA_CHECK(launch_dependent(
        tree_kv_append_rope_kernel, grid, ROPE_THREADS, 0, (cudaStream_t)stream, tree->T, Hq, Hkv, D, Lcap, 1, per, reinterpret_cast<__nv_bfloat16 *>(q), reinterpret_cast<const __nv_bfloat16 *>(k_new),
        reinterpret_cast<const __nv_bfloat16 *>(v_new), reinterpret_cast<__nv_bfloat16 *>(k_cache),
        reinterpret_cast<__nv_bfloat16 *>(v_cache), nullptr, nullptr, stride_b, stride_h, stride_t, seq_lens,
        tree->d_depth, log2(theta), status));
    MTV_CUDA_CHECK(cudaGetLastError());
    return MTV_OK;
}

extern "C" int tree_kv_append_rope_layers(const mtv_tree_t *tree, int B, int Hq, int Hkv, int D, int n_layers,
                                          mtv_bf16 *q_layers, const mtv_bf16 *k_new_layers, const mtv_bf16 *v_new_layers,
                                          mtv_bf16 *const *k_caches, mtv_bf16 *const *v_caches, int64_t stride_b,
                                          int64_t stride_h, int64_t stride_t, int Lcap, const int32_t *seq_lens,
                                          float rope_theta, int32_t *status, void *stream) {
    using namespace mtv;
    MTV_RANGE("tree_kv_append_rope_layers");
    if (!tree || !tree->on_device || !q_layers || !k_new_layers || !v_new_layers || !k_caches || !v_caches || !seq_lens)
        return MTV_ERR_INVALID_ARG;
    if (B < 1 || Hq < 1 || Hkv < 1 || n_layers < 1 || Lcap < tree->T || rope_theta < 0.f) return MTV_ERR_INVALID_ARG;
    if ((D != 64 && D != 128) || B > 65535 || n_layers > 65535) return MTV_ERR_UNSUPPORTED_SHAPE;
    const double theta = rope_theta == 0.f ? 10000.0 : (double)rope_theta;
    int per = 1;
    const dim3 grid = rope_grid(tree->T, B, n_layers, &per);
    MTV_CUDA_CHECK(launch_dependent(
        tree_kv_append_rope_kernel, grid, ROPE_THREADS, 0, (cudaStream_t)stream, tree->T, Hq, Hkv, D, Lcap, n_layers, per, reinterpret_cast<__nv_bfloat16 *>(q_layers),
        reinterpret_cast<const __nv_bfloat16 *>(k_new_layers), reinterpret_cast<const __nv_bfloat16 *>(v_new_layers),
        nullptr, nullptr, reinterpret_cast<__nv_bfloat16 *const *>(k_caches),
        reinterpret_cast<__nv_bfloat16 *const *>(v_caches), stride_b, stride_h, stride_t, seq_lens, tree->d_depth,
        log2(theta), status));
    MTV_CUDA_CHECK(cudaGetLastError());
    return MTV_OK;
}
