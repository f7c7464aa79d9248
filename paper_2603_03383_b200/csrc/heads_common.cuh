// Pieces shared by the two vocabulary-projection kernels of the Medusa heads (Section 3.1): the
// parameter block, the ordering of candidates, and everything that follows the projection itself —
// merging the warps' candidate lists per CTA, the merge across the CTAs of a head by the last one to
// finish (atomic ticket, nobody waits), and the expansion of the head's candidates into tree tokens (Section 3.2).
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
// Two sorted lists of sixteen, a half warp each has one of either: the sixteen best of both, sorted.  (The better of entry s and the
// other list's entry 15 - s are those sixteen, as a bitonic sequence.)  About 200 cycles.
__device__ __forceinline__ void list_merge(float &v, int &i, float ov, int oi, int lane) {
    const int src = (lane & 16) | (15 - (lane & 15));
    const float rv = __shfl_sync(0xffffffffu, ov, src);
    const int ri = __shfl_sync(0xffffffffu, oi, src);
    if (cand_before(rv, ri, v, i)) { v = rv; i = ri; }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) cand_exchange(v, i, o, true, lane);
}
// One candidate per lane (cand: it has one; their ids ascend with the lanes) against a list of kd <= 16 entries in shared memory.  A
// few are inserted one after the other (about 100 cycles each); many, as when a list is still empty, are ranked, each lane counting
// those before its own, and merged: a quarter of the time that sorting them over the lanes took, and the first tile of a
// CTA has all lists of up to sixteen batch rows to fill.  s_thr: the best kd-th entry of any list of this batch row in the CTA, as an
// order-preserving integer.  ranked: sixteen places of this warp.
static __device__ __noinline__ void list_update(float z, int v, bool cand, float *lv, int32_t *li, int kd, int *s_thr, int lane, float2 *ranked) {
    unsigned m = __ballot_sync(0xffffffffu, cand);
    float ev = lane < kd ? lv[lane] : -INFINITY;
    int ei = lane < kd ? li[lane] : 0x7fffffff;
    if (__popc(m) < 6) {
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            list_insert(ev, ei, __shfl_sync(0xffffffffu, z, src), __shfl_sync(0xffffffffu, v, src), kd, lane);
        }
    } else {
        const int bits = __float_as_int(z + 0.f);              // (-0.0 and 0.0 are equal)
        const int key = cand ? bits ^ ((bits >> 31) & 0x7fffffff) : (int)0x80000000;      // (no number has this key)
        int before = 0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const int other = __shfl_sync(0xffffffffu, key, j);
            before += (other > key) | ((other == key) & (j < lane));
        }
        if (before < 16) ranked[before] = make_float2(cand ? z : -INFINITY, __int_as_float(cand ? v : 0x7fffffff));
        __syncwarp();
        const float2 c = ranked[lane & 15];
        list_merge(ev, ei, c.x, __float_as_int(c.y), lane);
        __syncwarp();
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
    int tile_rows;       // (tensor cores) vocabulary rows per tile
    int x_rows;          // (tensor cores) rows of the activation operand
    int rows_per_stage, n_stages, n_it;
    uint32_t stage_bytes, xs_off, lists_off, zbuf_off, bars_off;
};

// One pass over n sorted lists of sixteen of each of `rows` rows, by all warps of the CTA: `parts` units per row, each of which leaves the
// best sixteen of its share.  The two half warps of a unit merge every other list of it, with the next lists on their way; a warp has
// R units side by side, whose chains of shuffles overlap.  src(row, list, slot, v, i) reads an entry, dst(row, part, slot, v, i) takes one.
template <int R, typename Src, typename Dst>
__device__ __forceinline__ void merge_pass(int rows, int n, int parts, const Src &src, const Dst &dst) {
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, half = lane >> 4, s = lane & 15, n_warps = (int)blockDim.x / 32;
    const int units = rows * parts, turns = (n + 2 * parts - 1) / (2 * parts);
#pragma unroll 1
    for (int unit0 = warp; unit0 < units; unit0 += R * n_warps) {
        float v[R], v0[R], v1[R];
        int i[R], i0[R], i1[R], row[R], list[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int unit = min(unit0 + r * n_warps, units - 1);      // (past the end: once more, and not kept)
            row[r] = unit / parts;
            list[r] = (unit - row[r] * parts) * 2 + half;
        }
        auto load = [&](int t, float (&lv)[R], int (&li)[R]) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int at = list[r] + t * 2 * parts;
                lv[r] = -INFINITY;
                li[r] = 0x7fffffff;
                if (at < n) src(row[r], at, s, lv[r], li[r]);
            }
        };
        load(0, v, i);
        load(1, v0, i0);
        load(2, v1, i1);
#pragma unroll 1
        for (int t = 1; t < turns; ++t) {      // (rolled: this code is met cold)
            float v2[R];
            int i2[R];
            load(t + 2, v2, i2);
#pragma unroll
            for (int r = 0; r < R; ++r) list_merge(v[r], i[r], v0[r], i0[r], lane);
#pragma unroll
            for (int r = 0; r < R; ++r) { v0[r] = v1[r]; i0[r] = i1[r]; v1[r] = v2[r]; i1[r] = i2[r]; }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            list_merge(v[r], i[r], __shfl_xor_sync(0xffffffffu, v[r], 16), __shfl_xor_sync(0xffffffffu, i[r], 16), lane);
            const int unit = unit0 + r * n_warps;
            if (half == 0 && unit < units) dst(row[r], list[r] / 2, s, v[r], i[r]);
        }
    }
}
// The same for many lists of which few can matter: the kd-th largest of the lists' first entries bounds what is looked for, so that only
// lists that begin at or above it are merged (kd of them, more where first entries are equal).  A warp per row; lists [row][n][16] in
// global memory, n <= 160.  (Apart: few calls come here, and the others' code is better off without it.)
static __device__ __noinline__ void merge_leading(int rows, int n, int kd, const float *part_val, const int32_t *part_idx, float2 (*result)[16]) {
    constexpr int Q = 5;
    const auto src = [&](int row, int l, int s, float &v, int &i) {
        v = __ldcg(part_val + (row * n + l) * 16 + s);
        i = __ldcg(part_idx + (row * n + l) * 16 + s);
    };
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, half = lane >> 4, s = lane & 15, n_warps = (int)blockDim.x / 32;
#pragma unroll 1
    for (int row = warp; row < rows; row += n_warps) {
        int key[Q], rest[Q];               // order-preserving images of the first entries
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float v = -INFINITY;
            int i;
            if (lane + 32 * q < n) src(row, lane + 32 * q, 0, v, i);
            const int bits = __float_as_int(v + 0.f);          // (-0.0 and 0.0 are equal)
            rest[q] = key[q] = lane + 32 * q < n ? bits ^ ((bits >> 31) & 0x7fffffff) : (int)0x80000000;
        }
        int bound = (int)0x80000000;
#pragma unroll 1
        for (int r = 0; r < kd; ++r) {
            int best = rest[0];
#pragma unroll
            for (int q = 1; q < Q; ++q) best = max(best, rest[q]);
            bound = __reduce_max_sync(0xffffffffu, best);
            bool take = lane == __ffs(__ballot_sync(0xffffffffu, best == bound)) - 1;          // one of them
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if (take && rest[q] == bound) { rest[q] = (int)0x80000000; take = false; }
        }
        unsigned in[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) in[q] = __ballot_sync(0xffffffffu, lane + 32 * q < n && key[q] >= bound);
        auto pop = [&]() {                 // the next list, or n
            int c = n;
#pragma unroll
            for (int q = Q - 1; q >= 0; --q)
                if (in[q]) c = 32 * q + __ffs(in[q]) - 1;
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if (c >> 5 == q && c < n) in[q] &= in[q] - 1;
            return c;
        };
        auto load = [&](float &v, int &i) {          // a list for each half warp; false: there was none for either
            const int c0 = pop(), c1 = pop(), c = half ? c1 : c0;
            v = -INFINITY;
            i = 0x7fffffff;
            if (c < n) src(row, c, s, v, i);
            return c0 < n;
        };
        float v, nv;
        int i, ni;
        load(v, i);
        bool more = load(nv, ni);
#pragma unroll 1
        while (more) {
            const float ov = nv;
            const int oi = ni;
            more = load(nv, ni);
            list_merge(v, i, ov, oi, lane);
        }
        list_merge(v, i, __shfl_xor_sync(0xffffffffu, v, 16), __shfl_xor_sync(0xffffffffu, i, 16), lane);
        if (half == 0) result[row][s] = make_float2(v, __int_as_float(i));
    }
    __syncthreads();
}
// The best sixteen of n sorted lists for each row: passes that take about four lists into one, the last one up to eight, until one is left.  (A tournament of
// kd rounds over the lists' heads, a warp per row, took 26 us for 16 rows of 37 lists at the end of a call, 9 us for two rows.)
struct MergeSmem {
    float2 a[52][16], b[26][16];      // what passes leave
    int32_t tok[16][16];              // candidates of a head
};
template <typename Src, typename Dst>
__device__ __forceinline__ void merge_lists(int rows, int n, MergeSmem *sm, const Src &src, const Dst &dst) {
    constexpr int R = 3;
    const int n_warps = (int)blockDim.x / 32;
    int parts = max(1, min((n + 3) / 4, R * n_warps / rows));
    if (rows * parts > n_warps && rows * parts < 2 * n_warps) parts = max(1, n_warps / rows);     // (a unit per warp, rather than two for some)
    if (parts == 1) {
        const auto to = [&](int row, int, int s, float v, int i) { dst(row, s, v, i); };
        if (rows <= n_warps) merge_pass<1>(rows, n, 1, src, to);
        else merge_pass<R>(rows, n, 1, src, to);
        return;
    }
    float2 (*from)[16] = sm->a, (*to)[16] = sm->b;
    {
        const auto leave = [&](int row, int part, int s, float v, int i) { from[row * parts + part][s] = make_float2(v, __int_as_float(i)); };
        if (rows * parts <= n_warps) merge_pass<1>(rows, n, parts, src, leave);
        else merge_pass<R>(rows, n, parts, src, leave);
    }
#pragma unroll 1
    do {
        __syncthreads();
        n = parts;
        parts = n <= 8 ? 1 : max(1, min((n + 3) / 4, n_warps / rows));
        merge_pass<1>(
            rows, n, parts,
            [&](int row, int l, int s, float &v, int &i) {
                const float2 e = from[row * n + l][s];
                v = e.x;
                i = __float_as_int(e.y);
            },
            [&](int row, int part, int s, float v, int i) {
                if (parts == 1) dst(row, s, v, i);
                else to[row * parts + part][s] = make_float2(v, __int_as_float(i));
            });
        float2 (*const t)[16] = from;
        from = to;
        to = t;
    } while (parts > 1);
}

// One or two candidates of n <= 160 sorted lists for each row: a warp per row has the first kd entries of all lists in registers and takes
// the best of them kd times: one round trip to L2 and no barrier, where merging lists of sixteen costs the same whatever is wanted.  us a call
// of one row and one / two candidates a head (H = 512, V = 16000), merged -> so: one head (148 lists) 19.4 -> 14.4 / 19.4 -> 14.8, four heads
// (37) 22.6 -> 19.6 / 22.7 -> 20.3; 16 rows, one candidate 33.9 -> 31.4 and 47.2 -> 42.1.  From three candidates on merging is faster than
// what went before it (one row of 148 lists 20.6 -> 19.5), with one it was not (16.2 -> 19.4).
constexpr int FEW = 2, FEW_LISTS = 160;
template <typename Src, typename Dst>
__device__ __forceinline__ void best_few(int rows, int n, int kd, const Src &src, const Dst &dst) {
    constexpr int Q = FEW_LISTS / 32;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, n_warps = (int)blockDim.x / 32;
#pragma unroll 1
    for (int row = warp; row < rows; row += n_warps) {
        float v[Q][FEW];
        int i[Q][FEW];
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int s = 0; s < FEW; ++s) {
                v[q][s] = -INFINITY;
                i[q][s] = 0x7fffffff;
                if (lane + 32 * q < n && s < kd) src(row, lane + 32 * q, s, v[q][s], i[q][s]);
            }
#pragma unroll 1
        for (int r = 0; r < kd; ++r) {
            float bv = v[0][0];
            int bi = i[0][0];
#pragma unroll
            for (int q = 1; q < Q; ++q)
                if (cand_before(v[q][0], i[q][0], bv, bi)) { bv = v[q][0]; bi = i[q][0]; }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (cand_before(ov, oi, bv, bi)) { bv = ov; bi = oi; }
            }
            if (lane == 0) dst(row, r, bv, bi);
#pragma unroll
            for (int q = 0; q < Q; ++q)        // the list that it came from goes on (those that have ended all begin alike)
                if (i[q][0] == bi) { v[q][0] = v[q][1]; i[q][0] = i[q][1]; }
        }
    }
}

// lval / lidx: [n_warps][NB][MTV_MAX_TOPK] sorted candidate lists in shared memory (unused slots hold
// (-inf, 0x7fffffff)); smem: sizeof(MergeSmem), free by now.  Every thread of the CTA calls this.
__device__ __forceinline__ void vocab_tail(const VocabParams &p, const int NB, const int n_warps, const float *lval,
                                           const int32_t *lidx, unsigned char *smem, const int k, const int bz,
                                           const int b0, const int per, const int kd) {
    __shared__ int s_flag;
    MergeSmem *sm = reinterpret_cast<MergeSmem *>(smem);
    const int rows = min(NB, p.B - b0);
    const size_t list0 = ((size_t)k * p.B + b0) * per;        // lists of all CTAs: [head][batch row][CTA][16]
    // ---- the warps' lists
    const bool few = kd <= FEW && per <= FEW_LISTS;       // (the other entries of the CTAs' lists are then neither written nor read)
    const auto of_warp = [&](int b, int w, int s, float &v, int &i) {
        v = lval[(w * NB + b) * MTV_MAX_TOPK + s];
        i = lidx[(w * NB + b) * MTV_MAX_TOPK + s];
    };
    const auto leave = [&](int b, int s, float v, int i) {
        const size_t o = (list0 + (size_t)b * per + blockIdx.x) * MTV_MAX_TOPK + s;
        p.part_val[o] = v;
        p.part_idx[o] = i;
    };
    if (few) best_few(rows, n_warps, kd, of_warp, leave);
    else merge_lists(rows, n_warps, sm, of_warp, leave);
    // ---- last CTA of this head merges the CTAs' lists (ticket: nobody waits)
    int32_t *counters = p.counters + (size_t)bz * (p.K + 1);
    __syncthreads();
    if (threadIdx.x == 0) {            // (one fence for the CTA: the barriers order the others' accesses against it)
        __threadfence();
        s_flag = atomicAdd(&counters[k], 1) == per - 1;
        __threadfence();
    }
    __syncthreads();
    if (!s_flag) return;
    static_assert(MTV_MAX_T <= 192, "a thread per tree node");
    const int off = p.off_arr[k], node = threadIdx.x, slot = node < p.T ? p.tree_indices[node] : -1;
    const auto take = [&](int b, int s, float v, int i) {
        sm->tok[b][s] = i;
        if (s >= kd) return;
        p.cand[(size_t)(b0 + b) * p.C + off + s] = i;
        if (p.cand_logit) p.cand_logit[(size_t)(b0 + b) * (p.C - 1) + off - 1 + s] = v;
    };
    // Rough cycles of either way: 500 for a turn of merges, 1500 for the passes behind the first; 3500 and 350 per candidate for a row by its
    // leading lists.  (13 rows of 148 lists with three candidates wanted: 58 -> 40 us a call; 16 rows of 29 lists are faster by merging all.)
    const int warps = (int)blockDim.x / 32, parts = max(1, min((per + 3) / 4, 3 * warps / rows));
    const int all = (rows * parts + 3 * warps - 1) / (3 * warps) * ((per + 2 * parts - 1) / (2 * parts)) * 500 + (parts > 1 ? 1500 : 0);
    const auto of_cta = [&](int b, int c, int s, float &v, int &i) {
        const size_t o = (list0 + (size_t)b * per + c) * MTV_MAX_TOPK + s;
        v = __ldcg(p.part_val + o);
        i = __ldcg(p.part_idx + o);
    };
    if (few) {
        best_few(rows, per, kd, of_cta, take);
    } else if (per <= 160 && (rows + warps - 1) / warps * (3500 + 350 * kd) < all) {
        merge_leading(rows, per, kd, p.part_val + list0 * MTV_MAX_TOPK, p.part_idx + list0 * MTV_MAX_TOPK, sm->a);
        for (int e = threadIdx.x; e < rows * 16; e += (int)blockDim.x) take(e / 16, e % 16, sm->a[e / 16][e % 16].x, __float_as_int(sm->a[e / 16][e % 16].y));
    } else {
        merge_lists(rows, per, sm, of_cta, take);
    }
    __syncthreads();
    // ---- the tokens of the tree nodes that are this head's candidates (the first head: and the root's)
    if (slot >= off && slot < off + kd)
        for (int b = 0; b < rows; ++b) p.tree_tok[(size_t)(b0 + b) * p.T + node] = sm->tok[b][slot - off];
    if (off == 1) {
        if (node < p.T && MTV_INDEX_OK(slot, p.C, p.dev_error) && slot == 0)
            for (int b = 0; b < rows; ++b) p.tree_tok[(size_t)(b0 + b) * p.T + node] = p.root_tok[b0 + b];
        if ((int)threadIdx.x < rows) p.cand[(size_t)(b0 + threadIdx.x) * p.C] = p.root_tok[b0 + threadIdx.x];     // (more rows than nodes, maybe)
    }
    if (p.gate_clear && threadIdx.x == 0 && atomicAdd(&counters[p.K], 1) == p.K - 1) *p.gate.word = 0;     // (all have read it)
}

}  // namespace mtv
