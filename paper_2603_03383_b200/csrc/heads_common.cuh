// Pieces shared by the two vocabulary-projection kernels of the Medusa heads (Section 3.1): the
// parameter block, the ordering of candidates, and everything that follows the projection itself —
// merging the warps' candidate lists per CTA, the merge across the CTAs of a head by the last one to
// finish (atomic ticket, nobody waits), and the expansion into tree tokens by the last head (Section 3.2).
#pragma once
#include "common.cuh"

namespace mtv {

constexpr int HT_NB = 16;   // batch rows one pass of the tensor-core projection serves

// (value, id) ordering of the candidate lists: larger value first, equal values by smaller id.
__device__ __forceinline__ bool cand_before(float va, int ia, float vb, int ib) {
    return va > vb || (va == vb && ia < ib);
}

// A sorted list of candidates held by a warp: lane s has entry s.  Insertion of one candidate (the same in all lanes) into a
// list of kd entries: the entries ahead of it stay, the others move down by one.
__device__ __forceinline__ void list_insert(float &ev, int &ei, float z, int v, int kd, int lane) {
    const int pos = __popc(__ballot_sync(0xffffffffu, lane < kd && cand_before(ev, ei, z, v)));
    const float uv = __shfl_up_sync(0xffffffffu, ev, 1);
    const int ui = __shfl_up_sync(0xffffffffu, ei, 1);
    if (lane < kd && lane > pos) { ev = uv; ei = ui; }
    if (lane == pos && pos < kd) { ev = z; ei = v; }
}
// lanes l and l ^ o: the better one goes to the lower lane if `down`, else to the upper
__device__ __forceinline__ void cand_exchange(float &v, int &i, int o, bool down, int lane) {
    const float ov = __shfl_xor_sync(0xffffffffu, v, o);
    const int oi = __shfl_xor_sync(0xffffffffu, i, o);
    const bool lower = (lane & o) == 0, mine_better = cand_before(v, i, ov, oi);
    if ((lower == down) != mine_better) { v = ov; i = oi; }
}
// One candidate per lane (cand: it has one) against a list of kd <= 16 entries in shared memory.  A few are inserted one
// after the other (about 100 cycles each); many, as when a list is still empty, are sorted over the lanes and merged (about
// 900 cycles).  s_thr: the best kd-th entry of any list of this batch row in the CTA, as an order-preserving integer.
static __device__ __noinline__ void list_update(float z, int v, bool cand, float *lv, int32_t *li, int kd, int *s_thr, int lane) {
    unsigned m = __ballot_sync(0xffffffffu, cand);
    float ev = lane < kd ? lv[lane] : -INFINITY;
    int ei = lane < kd ? li[lane] : 0x7fffffff;
    if (__popc(m) < 8) {
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            list_insert(ev, ei, __shfl_sync(0xffffffffu, z, src), __shfl_sync(0xffffffffu, v, src), kd, lane);
        }
    } else {
        float x = cand ? z : -INFINITY;
        int xi = cand ? v : 0x7fffffff;
#pragma unroll 1
        for (int k = 2; k <= 32; k <<= 1)          // bitonic sort, best first
#pragma unroll 1
            for (int o = k >> 1; o > 0; o >>= 1) cand_exchange(x, xi, o, (lane & k) == 0, lane);
        // the better of entry s and candidate 15 - s: the sixteen best of both, bitonic
        const float rv = __shfl_sync(0xffffffffu, x, 15 - (lane & 15));
        const int ri = __shfl_sync(0xffffffffu, xi, 15 - (lane & 15));
        if (!cand_before(ev, ei, rv, ri)) { ev = rv; ei = ri; }
#pragma unroll 1
        for (int o = 8; o > 0; o >>= 1) cand_exchange(ev, ei, o, true, lane);
    }
    if (lane < kd) { lv[lane] = ev; li[lane] = ei; }
    if (lane == kd - 1) {
        const int bits = __float_as_int(ev);
        atomicMax(s_thr, bits ^ ((bits >> 31) & 0x7fffffff));
    }
    __syncwarp();
}
__device__ __forceinline__ float thr_value(int ord) { return __int_as_float(ord ^ ((ord >> 31) & 0x7fffffff)); }

struct VocabParams {
    int B, H, V, K, T, C;
    const __nv_bfloat16 *W2;
    const float *hprime;
    const int32_t *kd_arr, *off_arr, *tree_indices, *root_tok;
    float *part_val;
    int32_t *part_idx;
    int32_t *counters;   // [btiles][K + 1], zeroed by the residual-block kernel
    int32_t *cand;
    float *cand_logit;
    int32_t *tree_tok;
    int32_t *dev_error;
    Gate gate;           // the weights are complete behind it (no word: behind the previous kernel)
    int gate_clear;      // the last CTA of all clears it
    int expand;          // the last head to finish expands all heads' candidates into the tree tokens
    int tile_rows;       // (tensor cores) vocabulary rows per tile
    int x_rows;          // (tensor cores) rows of the activation operand
    int rows_per_stage, n_stages, n_it;
    uint32_t stage_bytes, xs_off, lists_off, zbuf_off, bars_off;
};

// lval / lidx: [n_warps][NB][MTV_MAX_TOPK] sorted candidate lists in shared memory (unused slots hold
// (-inf, 0x7fffffff)); smem / scratch_bytes: shared memory free for the cross-CTA merge (at least
// per * MTV_MAX_TOPK * 8 bytes: one warp's staging area; more lets more warps merge batch rows side by side).
// Every thread of the CTA calls this.
__device__ __forceinline__ void vocab_tail(const VocabParams &p, const int NB, const int n_warps, const float *lval,
                                           const int32_t *lidx, unsigned char *smem, const int k, const int bz,
                                           const int b0, const int per, const int kd, const uint32_t scratch_bytes) {
    __shared__ int s_flag;
    // ---- merge the warps' lists: rank each entry among all CONS_WARPS*kd entries of its batch row
    for (int e = threadIdx.x; e < NB * n_warps * MTV_MAX_TOPK; e += (int)blockDim.x) {
        const int b = e / (n_warps * MTV_MAX_TOPK);
        const int w = (e / MTV_MAX_TOPK) % n_warps, sl = e % MTV_MAX_TOPK;
        if (sl >= kd || b0 + b >= p.B) continue;
        const float zz = lval[(w * NB + b) * MTV_MAX_TOPK + sl];
        const int id = lidx[(w * NB + b) * MTV_MAX_TOPK + sl];
        int rank = 0;
        for (int w2 = 0; w2 < n_warps; ++w2)
            for (int s2 = 0; s2 < kd; ++s2) {
                const float z2 = lval[(w2 * NB + b) * MTV_MAX_TOPK + s2];
                const int id2 = lidx[(w2 * NB + b) * MTV_MAX_TOPK + s2];
                // unused slots all carry the same sentinel: order them by position
                if (cand_before(z2, id2, zz, id) || (z2 == zz && id2 == id && (w2 * MTV_MAX_TOPK + s2) < (w * MTV_MAX_TOPK + sl)))
                    ++rank;
            }
        if (rank < kd) {
            const size_t o = (((size_t)k * p.B + b0 + b) * per + blockIdx.x) * MTV_MAX_TOPK + rank;
            p.part_val[o] = zz;
            p.part_idx[o] = id;
        }
    }
    // ---- last CTA of this head merges the CTAs' lists (ticket: nobody waits)
    int32_t *counters = p.counters + (size_t)bz * (p.K + 1);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_flag = atomicAdd(&counters[k], 1) == per - 1;
    __syncthreads();
    if (!s_flag) return;
    __threadfence();
    {
        // The CTAs' lists are sorted, so the best kd of all of them come out of a kd-round tournament over
        // the lists' heads.  Each warp takes one batch row at a time: it stages the row's lists in shared
        // memory, lane l plays for lists l, l + 32, ...
        const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
        const int off = p.off_arr[k];
        const uint32_t per_warp = (uint32_t)per * MTV_MAX_TOPK * 8;
        int n_w = (int)(scratch_bytes / per_warp);
        if (n_w > (int)blockDim.x / 32) n_w = (int)blockDim.x / 32;
        constexpr int MAXL = 8;                               // lists per lane: up to 256 CTAs per head
        if (warp < n_w) {
            float *mval = reinterpret_cast<float *>(smem + (size_t)warp * per_warp);   // [per][MTV_MAX_TOPK]
            int32_t *midx = reinterpret_cast<int32_t *>(mval + per * MTV_MAX_TOPK);
            for (int b = warp; b < NB && b0 + b < p.B; b += n_w) {
                const size_t base = ((size_t)k * p.B + b0 + b) * per * MTV_MAX_TOPK;
                __syncwarp();
                // the kd entries of each list, many loads in flight (all sixteen slots of every list, one round trip to L2
                // at a time, took 8 us at the end of every call)
                const unsigned n_e = (unsigned)(per * kd), inv = (1u << 20) / (unsigned)kd + 1u;   // e / kd for e < 4096
#pragma unroll 1
                for (unsigned e0 = lane; e0 < n_e; e0 += 32 * 8) {
                    float v[8];
                    int id[8];
                    unsigned at[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const unsigned e = min(e0 + 32 * q, n_e - 1), c = (e * inv) >> 20;
                        at[q] = c * MTV_MAX_TOPK + (e - c * (unsigned)kd);
                        v[q] = __ldcg(p.part_val + base + at[q]);
                        id[q] = __ldcg(p.part_idx + base + at[q]);
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q) { mval[at[q]] = v[q]; midx[at[q]] = id[q]; }
                }
                __syncwarp();
                int head[MAXL];
#pragma unroll
                for (int q = 0; q < MAXL; ++q) head[q] = 0;
                for (int r = 0; r < kd; ++r) {
                    // this lane's best head
                    float bv = -INFINITY;
                    int bi = 0x7fffffff, bq = -1;
#pragma unroll
                    for (int q = 0; q < MAXL; ++q) {
                        const int c = lane + 32 * q;
                        if (c < per && head[q] < kd) {
                            const float v = mval[c * MTV_MAX_TOPK + head[q]];
                            const int id = midx[c * MTV_MAX_TOPK + head[q]];
                            if (bq < 0 || cand_before(v, id, bv, bi)) { bv = v; bi = id; bq = q; }
                        }
                    }
                    // the warp's best: value first, then id, then lane (equal sentinels)
                    float wv = bv;
                    int wi = bi, wl = bq < 0 ? 64 : lane;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const float ov = __shfl_xor_sync(0xffffffffu, wv, o);
                        const int oi = __shfl_xor_sync(0xffffffffu, wi, o);
                        const int ol = __shfl_xor_sync(0xffffffffu, wl, o);
                        const bool other = ol < 64 && (wl >= 64 || cand_before(ov, oi, wv, wi) || (ov == wv && oi == wi && ol < wl));
                        if (other) { wv = ov; wi = oi; wl = ol; }
                    }
                    if (lane == 0) {
                        p.cand[(size_t)(b0 + b) * p.C + off + r] = wi;
                        if (p.cand_logit) p.cand_logit[(size_t)(b0 + b) * (p.C - 1) + off - 1 + r] = wv;
                    }
                    if (lane == wl) {
#pragma unroll
                        for (int q = 0; q < MAXL; ++q)
                            if (q == bq) ++head[q];
                    }
                }
            }
        }
    }
    // ---- last head of this batch tile expands the candidates into the tree tokens
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_flag = atomicAdd(&counters[p.K], 1) == p.K - 1;
        if (s_flag && p.gate_clear) *p.gate.word = 0;
    }
    __syncthreads();
    if (!s_flag || !p.expand) return;
    __threadfence();
    for (int e = threadIdx.x; e < NB * p.T; e += (int)blockDim.x) {
        const int b = b0 + e / p.T, i = e % p.T;
        if (b >= p.B) break;
        const int slot = p.tree_indices[i];
        if (!MTV_INDEX_OK(slot, p.C, p.dev_error)) continue;
        const int32_t root = p.root_tok[b];
        if (i == 0) p.cand[(size_t)b * p.C] = root;
        p.tree_tok[(size_t)b * p.T + i] = slot == 0 ? root : __ldcg(p.cand + (size_t)b * p.C + slot);
    }
}

}  // namespace mtv
