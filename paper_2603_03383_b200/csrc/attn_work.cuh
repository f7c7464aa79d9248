// How the tree attention divides the key groups of all items among teams of CTAs, the exponentials of a tile, the workspace of
// partial results and their merge (attention.cu).
#pragma once
#include "attn_common.cuh"

namespace mtv {

constexpr int AT_BN = 128;            // keys per group
constexpr int AT_THREADS = 640;
constexpr int AT_SOFTMAX_WARPS = 16;
constexpr int AT_PIECES = 4;          // piece descriptors in flight
// How long a CTA waits for the others of an item, in cycles.  In the bounds-checking build it looks once: nearly all slices
// are then left to the last one.
#ifdef MTV_DEBUG_BOUNDS
constexpr long long AT_MERGE_WAIT = 0;
#else
constexpr long long AT_MERGE_WAIT = 2000000;
#endif
constexpr int AT_MAX_CTAS = MERGE_COUNTERS;   // a pair of merge counters per CTA (the first of a team's, for the item it begins)
constexpr int AT_DEPART = 16;         // ints from a CTA's first counter to its second
constexpr int AT_MAX_LAYERS = 64;     // layers per launch (two tensor maps each in the kernel's parameters)
// registers per thread: 96 at launch, moved from the four auxiliary warps to the sixteen softmax warps
constexpr int AT_LAUNCH_REGS = 96, AT_SOFTMAX_REGS = 104, AT_AUX_REGS = 64;
static_assert(512 * AT_SOFTMAX_REGS + 128 * AT_AUX_REGS <= AT_THREADS * AT_LAUNCH_REGS, "register split");
constexpr float AT_SUM_LIMIT = 4294967296.f;   // 2^32: a thread's sum of P over a group beyond it moves the reference

struct AttnPiece {      // 32 bytes
    int layer, b, head, gb, cnt, L, flags, first;   // key groups [gb, gb + cnt); cnt = 0: no more pieces;
                                                    // first: first team that contributes to the item
};
// flags: not a whole item; starts at the item's first group; from this bit on, how many groups have their weights in two terms
constexpr int PIECE_PARTIAL = 1, PIECE_HEAD = 2, PIECE_TWO_SHIFT = 8;
struct AttnMerge {      // a partial piece of this CTA, for the merge at the end
    int first, n, layer, b, head, pad;             // first contributing team, number of them
};

template <int ML>
struct __align__(64) AttnMaps {
    CUtensorMap q, k[ML], v[ML];
};

// Where a (layer, sequence, head) is in the one tensor map of all layers: dimension 3 at head + head_b * sequence, dimension 4 at
// b * sequence + layer * layer.
struct CacheFold {
    int head_b, b, layer;
};
struct AttnParams {
    const int32_t *seq_lens;
    const uint64_t *anc;     // [T][2]
    __nv_bfloat16 *out;      // [layers][B][T][Hq][D]
    uint4 *ws_o;             // [CTA][2 slabs][D / 4 chunks][128 rows] 16-byte chunks of O / l, fp32
    float2 *ws_ml;           // [CTA][2 slabs][128 rows] (m, l)
    int32_t *left;           // [CTA][2 slabs] 1: the CTA's slice of the item is left to the last one
    int32_t *counters;       // merge counters, zero between calls; the second one counts slices left in its upper half
    int32_t *status;         // [B] or null
    int32_t *dev_error;
    float scale_log2;
    int B, T, G, Hq, Hkv, Lcap, n_layers;
    int npc, R;              // tree nodes per tile (128 / G) and the rows they fill
    unsigned inv_g;          // 65536 / G rounded up: row r of a tile is node (r * inv_g) >> 16 (exact for r < 256, G <= 8)
    int n_blk, teams;        // CTAs of a team, teams
    int n_tiles, two_cuts;   // row tiles of an item; see two_term_groups
    CacheFold fold;
    int out32;               // out begins at a multiple of 32 bytes
    Gate gate;               // with a word: the inputs are complete behind it, the previous kernel is waited for at the end
};

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
// P = 2^(scale S - m) of 32 scores (two values per instruction where the instruction set has packed forms) and its
// contribution to the row sum.  pk: bf16 pairs; TWO: rest has what their rounding left, as bf16 pairs.  All exponentials are the
// special-function unit's: it needs 1024 cycles for a tile of scores, what the tensor core needs, and with a quarter of them as
// polynomials on the FMA pipes a step of 4 x 32768 keys takes 4 % longer (867 -> 902 us for four layers), since the board's power
// limit, not a pipe, sets the pace there.
template <bool TWO>
__device__ __forceinline__ void exp_quarter(const uint32_t (&s)[32], float2 sc2, float2 nm2, float2 &la, float2 &lb, uint32_t *pk, uint32_t *rest) {
#pragma unroll
    for (int e = 0; e < 16; e += 2) {
        const float2 x01 = __ffma2_rn(make_float2(__uint_as_float(s[2 * e]), __uint_as_float(s[2 * e + 1])), sc2, nm2);
        const float2 x23 = __ffma2_rn(make_float2(__uint_as_float(s[2 * e + 2]), __uint_as_float(s[2 * e + 3])), sc2, nm2);
        const float2 p01 = make_float2(ex2(x01.x), ex2(x01.y)), p23 = make_float2(ex2(x23.x), ex2(x23.y));
        la = __fadd2_rn(la, p01);
        lb = __fadd2_rn(lb, p23);
        pk[e] = pack2_bf16(p01.x, p01.y);
        pk[e + 1] = pack2_bf16(p23.x, p23.y);
        if (TWO) {
            const float2 r01 = __fadd2_rn(p01, make_float2(-bf16_lo(pk[e]), -bf16_hi(pk[e])));
            const float2 r23 = __fadd2_rn(p23, make_float2(-bf16_lo(pk[e + 1]), -bf16_hi(pk[e + 1])));
            rest[e] = pack2_bf16(r01.x, r01.y);
            rest[e + 1] = pack2_bf16(r23.x, r23.y);
        }
    }
}
// the largest scale * s of 32 scores; NEG: the scale is negative
template <bool NEG>
__device__ __forceinline__ float max_quarter(const uint32_t (&s)[32], float scale) {
    constexpr uint32_t sign = NEG ? 0x80000000u : 0u;
    float a = -INFINITY, b = -INFINITY;
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
        a = ptx::fmax3(a, __uint_as_float(s[e] ^ sign), __uint_as_float(s[e + 1] ^ sign));
        b = ptx::fmax3(b, __uint_as_float(s[e + 2] ^ sign), __uint_as_float(s[e + 3] ^ sign));
    }
    return fmaxf(a, b) * fabsf(scale);
}
// Output row of row r of a CTA's tile (in units of D elements from the item's first row), or -1 if it belongs to nobody: CTA blk of
// a team has row tile blk.  With a group size that does not divide 128 the last 128 - R rows of a tile do (whatever the tile's
// shared memory held is computed and never written out).
__device__ __forceinline__ int node_in_tile(const AttnParams &p, int r) { return (int)(((unsigned)r * p.inv_g) >> 16); }
__device__ __forceinline__ int out_row(const AttnParams &p, int blk, int r) {
    const int n = node_in_tile(p, r), node = blk * p.npc + n;
    return r < p.R && node < p.T ? node * p.Hq + (r - n * p.G) : -1;
}
template <int D>
__device__ __forceinline__ uint4 *item_out(const AttnParams &p, int layer, int b, int hd) {      // first row of an item's output
    return reinterpret_cast<uint4 *>(p.out + (((size_t)layer * p.B + b) * p.T * p.Hq + hd * p.G) * D);
}
// slabs of the workspace: 16-byte chunk c (4 columns) of row r; the row's (m, l)
template <int D>
__device__ __forceinline__ uint4 *slab_o(const AttnParams &p, int cta, int slab, int r, int c) {
    return p.ws_o + (((unsigned)cta * 2 + slab) * (D / 4) + c) * 128 + r;
}
__device__ __forceinline__ float2 *slab_ml(const AttnParams &p, int cta, int slab, int r) {
    return p.ws_ml + ((unsigned)cta * 2 + slab) * 128 + r;
}

// The counters that the contributors of an item meet at: of its first contributor, for row tile blk.
__device__ __forceinline__ int32_t *merge_counter(const AttnParams &p, int first, int blk) {
    return p.counters + (first * p.n_blk + blk) * MERGE_STRIDE;
}
// Rows of a tile that is shared between CTAs: contributor c0 combines its share of them, a thread per VC 16-byte chunks of a row, with
// the loads of NS contributors in flight.  All CTAs do this at the same time, and L2 gives some 20 bytes per cycle and SM then, so the
// bytes count more than the round trips: with five contributors or a single chunk at a time (its (m, l) are a third of the
// bytes) eight one-layer calls on ragged lengths take 306 and 343 us instead of 285.
template <int D>
struct MergeSlice {
    static constexpr int VC = 2, NS = 3, NT = D / 4 / VC;    // (VC = 2: 16 bytes of output)
    int r_begin, n_my;
    unsigned inv_n;                                      // e / n_my = (e * inv_n) >> 20 for e < 2048, n_my <= 64
    __device__ __forceinline__ MergeSlice(const AttnParams &p, const AttnMerge &m, int c0) {
        const int per = (p.R + m.n - 1) / m.n;           // (m.n >= 2)
        r_begin = c0 * per;
        n_my = max(0, min(p.R, r_begin + per) - r_begin);
        inv_n = n_my > 0 ? ((1u << 20) + n_my - 1) / n_my : 0;
    }
    __device__ __forceinline__ void run(const AttnParams &p, const AttnMerge &m, int thread, int blk) const {
        uint4 *dst = item_out<D>(p, m.layer, m.b, m.head);
#pragma unroll 1
        for (int e = thread; e < n_my * NT; e += AT_SOFTMAX_WARPS * 32) {
            const int c = (int)(((unsigned)e * inv_n) >> 20), r = r_begin + e - c * n_my;
            float acc[4 * VC], mm = -INFINITY, wsum = 0.f;
#pragma unroll
            for (int k = 0; k < 4 * VC; ++k) acc[k] = 0.f;
#pragma unroll 1
            for (int s0 = 0; s0 < m.n; s0 += NS) {
                float2 ml[NS];
                uint4 v[NS][VC];
#pragma unroll
                for (int k = 0; k < NS; ++k) {
                    const int s = s0 + k, cta = (m.first + s) * p.n_blk + blk;
                    const int sl = s == 0 ? 1 : 0;       // the first contributor's piece begins the item
                    ml[k] = make_float2(-INFINITY, 0.f);
#pragma unroll
                    for (int q = 0; q < VC; ++q) v[k][q] = make_uint4(0u, 0u, 0u, 0u);
                    if (s < m.n) {
                        ml[k] = __ldcg(slab_ml(p, cta, sl, r));
#pragma unroll
                        for (int q = 0; q < VC; ++q) v[k][q] = __ldcg(slab_o<D>(p, cta, sl, r, c * VC + q));
                    }
                }
                float mc = mm;
#pragma unroll
                for (int k = 0; k < NS; ++k) mc = fmaxf(mc, ml[k].x);
                const float resc = mm == -INFINITY ? 0.f : ex2(mm - mc);
                mm = mc;
                wsum *= resc;
#pragma unroll
                for (int k = 0; k < 4 * VC; ++k) acc[k] *= resc;
#pragma unroll
                for (int k = 0; k < NS; ++k) {
                    const float wt = ml[k].x == -INFINITY ? 0.f : ex2(ml[k].x - mc) * ml[k].y;
                    wsum += wt;
#pragma unroll
                    for (int q = 0; q < VC; ++q) {
                        const uint32_t vw[4] = {v[k][q].x, v[k][q].y, v[k][q].z, v[k][q].w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) acc[4 * q + i] = fmaf(wt, __uint_as_float(vw[i]), acc[4 * q + i]);
                    }
                }
            }
            const float inv = wsum == 0.f ? 0.f : 1.f / wsum;
            const int o = out_row(p, blk, r);
            if (o >= 0)
                dst[o * (D / 8) + c] =
                    make_uint4(pack2_bf16(acc[0] * inv, acc[1] * inv), pack2_bf16(acc[2] * inv, acc[3] * inv),
                               pack2_bf16(acc[4] * inv, acc[5] * inv), pack2_bf16(acc[6] * inv, acc[7] * inv));
        }
    }
};
// The same for many contributors, whose slices have few rows: `split` lanes of a warp share the contributors of a chunk, that many fewer
// round trips to L2.  (One sequence of 9284 keys and a single head, cut into 73 pieces: 30 -> 17 us a call.  Apart from run(), whose code is
// slower for being both: ragged calls 256 -> 272 us; and for fewer contributors the way here costs more than it saves: head size
// 64 with four 158 -> 166 us.)
constexpr int MERGE_MANY = 24;
template <int D>
__device__ __forceinline__ void few_rows(const AttnParams &p, const AttnMerge &m, int r_begin, int n_my, int thread, int blk) {
    constexpr int VC = 2, NS = 3, NT = D / 4 / VC;
    // (more than 24 contributors: at most six rows each, 96 chunks)
    static_assert((128 / (MERGE_MANY + 1) + 1) * NT * 4 <= AT_SOFTMAX_WARPS * 32, "a thread per chunk and share");
    const int all = n_my * NT, split = all * 8 <= AT_SOFTMAX_WARPS * 32 ? 8 : 4, each = 32 / split, sub = (thread & 31) / each;
    const int e = (thread >> 5) * each + (thread & 31) % each, e_in = min(e, all - 1), c = e_in / n_my, r = r_begin + e_in - c * n_my;
    float acc[4 * VC], mm = -INFINITY, wsum = 0.f;
#pragma unroll
    for (int k = 0; k < 4 * VC; ++k) acc[k] = 0.f;
    auto join = [&](float mc) {                      // another reference
        const float resc = mm == -INFINITY ? 0.f : ex2(mm - mc);
        mm = mc;
        wsum *= resc;
#pragma unroll
        for (int k = 0; k < 4 * VC; ++k) acc[k] *= resc;
    };
#pragma unroll 1
    for (int s0 = sub; s0 < m.n; s0 += split * NS) {
        float2 ml[NS];
        uint4 v[NS][VC];
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const int s = s0 + k * split, cta = (m.first + s) * p.n_blk + blk;
            const int sl = s == 0 ? 1 : 0;
            ml[k] = make_float2(-INFINITY, 0.f);
#pragma unroll
            for (int q = 0; q < VC; ++q) v[k][q] = make_uint4(0u, 0u, 0u, 0u);
            if (s < m.n) {
                ml[k] = __ldcg(slab_ml(p, cta, sl, r));
#pragma unroll
                for (int q = 0; q < VC; ++q) v[k][q] = __ldcg(slab_o<D>(p, cta, sl, r, c * VC + q));
            }
        }
        float mc = mm;
#pragma unroll
        for (int k = 0; k < NS; ++k) mc = fmaxf(mc, ml[k].x);
        join(mc);
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const float wt = ml[k].x == -INFINITY ? 0.f : ex2(ml[k].x - mc) * ml[k].y;
            wsum += wt;
#pragma unroll
            for (int q = 0; q < VC; ++q) {
                const uint32_t vw[4] = {v[k][q].x, v[k][q].y, v[k][q].z, v[k][q].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[4 * q + i] = fmaf(wt, __uint_as_float(vw[i]), acc[4 * q + i]);
            }
        }
    }
#pragma unroll 1
    for (int o = each; o < 32; o <<= 1) {
        join(fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, o)));
        wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
#pragma unroll
        for (int k = 0; k < 4 * VC; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    }
    const float inv = wsum == 0.f ? 0.f : 1.f / wsum;
    const int o = out_row(p, blk, r);
    if (o >= 0 && sub == 0 && e < all)
        item_out<D>(p, m.layer, m.b, m.head)[o * (D / 8) + c] =
            make_uint4(pack2_bf16(acc[0] * inv, acc[1] * inv), pack2_bf16(acc[2] * inv, acc[3] * inv),
                       pack2_bf16(acc[4] * inv, acc[5] * inv), pack2_bf16(acc[6] * inv, acc[7] * inv));
}
template <int D>
static __device__ __noinline__ void merge_few_rows(const AttnParams &p, const AttnMerge &m, int r_begin, int n_my, int thread, int blk) {
    few_rows<D>(p, m, r_begin, n_my, thread, blk);
}
// The slices that CTAs left, of one item, by the softmax warps of the CTA that was the last to leave it: summed as their own CTAs would
// have, since bits must not depend on who is late.  (Out of the way of the usual case, whose registers it must not touch, and calling nothing:
// with calls of merge_few_rows from here, or a choice between the two in the kernel, the compiler's registers for the kernel change, and eight
// one-layer calls with twenty contributors take 136 to 139 us instead of 124, or at ragged lengths 269 instead of 256.)
template <int D>
static __device__ __noinline__ void merge_left(const AttnParams &p, const AttnMerge &m, int blk, int thread) {
#pragma unroll 1
    for (int c = 0; c < m.n; ++c) {
        if (!__ldcg(p.left + ((m.first + c) * p.n_blk + blk) * 2 + (c == 0 ? 1 : 0))) continue;
        const MergeSlice<D> slice(p, m, c);
        if (m.n <= MERGE_MANY) slice.run(p, m, thread, blk);
        else if (slice.n_my > 0) few_rows<D>(p, m, slice.r_begin, slice.n_my, thread, blk);
    }
}

// a / b, b > 0.  A quotient of small numbers is at most one off when it is formed in fp32, and its remainder says which way; the
// chain of these that a launch starts with takes a third of the time that integer divisions take.
__device__ __forceinline__ unsigned quotient(unsigned a, unsigned b) {
    if (a >= 1u << 22) return a / b;
    unsigned q = (unsigned)__fdividef((float)a, (float)b);
    const int r = (int)(a - q * b);
    if (r < 0) --q;
    else if ((unsigned)r >= b) ++q;
    return q;
}
// Runs that whole items or whole pieces make longer by more than this have more second terms, see two_term_groups.
constexpr int WHOLE_EXACT = 5, PAD_EXACT = 2;
// The pieces of one team's run, derived by one warp from the lengths on the device (see attention.cu).  COST: what an item costs
// beside its key groups, in groups; WHOLE, PAD: how much longer a run may be made for whole items, and for one piece to a run.
template <int COST, int WHOLE, int PAD>
struct PieceWalk {
    const AttnParams &p;
    const int lane;
    const unsigned LH, teams, team;
    const bool lone;                      // one row tile, or the last of an odd number of them
    float two_rate = 0.f;                 // see two_term_groups
    int chunk = 0, len = 0, g = 0;        // lengths and group counts of sequences chunk .. chunk + 31, one per lane
    bool pad = false;
    unsigned u = 1, pos = 0, hi = 0, off = 0;
    int layer = 0, b = 0, head = 0, n_part = 0;

    __device__ __forceinline__ PieceWalk(const AttnParams &p_, int team_, int lane_, bool lone_)
        : p(p_), lane(lane_), LH((unsigned)p_.n_layers * (unsigned)p_.Hkv), teams((unsigned)p_.teams), team((unsigned)team_), lone(lone_) {}
    // (the lengths may be looked at before the kernel that writes them is complete, and again behind it)
    __device__ __forceinline__ int length(int at) const { return at < p.B ? ld_relaxed(p.seq_lens + at) : 0; }
    // Key groups of a sequence.  0: it has no room for the tree's rows, or no rows at all (nothing here may wrap or become
    // negative: the sums below are other sequences' positions); it is passed over, which report() says.
    __device__ __forceinline__ int groups(int l) const { return l > -p.T && l <= p.Lcap - p.T ? (l + p.T + AT_BN - 1) / AT_BN : 0; }
    __device__ __forceinline__ void load_chunk(int b0) {
        chunk = b0;
        len = length(b0 + lane);
        g = b0 + lane < p.B ? groups(len) : 0;
    }
    // May the work be divided by lengths that may still change?  (More than 32 are read more than once, which must agree.)
    __device__ __forceinline__ bool early() const { return p.B <= 32; }
    // Were they the ones that are there now?
    __device__ __forceinline__ bool still_so() const { return __all_sync(0xffffffffu, length(lane) == len); }
    __device__ __forceinline__ void report() const {
        if (blockIdx.x == 0 && p.status)
            for (int b = lane; b < p.B; b += 32) p.status[b] = groups(length(b)) > 0 ? MTV_OK : MTV_ERR_CAPACITY;
    }
    __device__ __forceinline__ unsigned padded(unsigned gg) const { return gg == 0 ? 0u : pad ? quotient(gg + u - 1, u) * u : gg + COST; }
    __device__ __forceinline__ void divide() {
        layer = b = head = n_part = 0;
        off = 0;
        unsigned sum = 0, nz = 0, g_max = 0, g_min = 0xffffffffu;
        for (int b0 = 0; b0 < p.B; b0 += 32) {
            load_chunk(b0);
            sum += __reduce_add_sync(0xffffffffu, (unsigned)g);
            nz += __popc(__ballot_sync(0xffffffffu, g > 0));
            g_max = max(g_max, __reduce_max_sync(0xffffffffu, (unsigned)g));
            g_min = min(g_min, __reduce_min_sync(0xffffffffu, g > 0 ? (unsigned)g : 0xffffffffu));
        }
        // Piece length u of either way to divide.  Padding to whole pieces wastes the teams it leaves idle, cutting anywhere gives most
        // teams a second piece, and so a second partial result: whichever is shorter.  (Eight one-layer calls, cutting where
        // padding makes a piece longer by more than 5 / 7 groups: 4 x 8000 keys, T = 128, 531 / 491 us; seven ragged sequences
        // 281 / 272.)
        const unsigned u_cut = max(1u, quotient(LH * (sum + nz * COST) + teams - 1, teams));
        pad = LH * nz <= teams;
        u = pad ? max(1u, quotient(LH * sum + teams - 1, teams)) : u_cut;
        // Whole items, if that makes no run longer than the division above by more than a merge takes: no team shares one.
        const unsigned whole = pad ? g_max : quotient(LH * nz + teams - 1, teams) * (g_max + COST);
        unsigned v_head;                      // length of one head's row of all sequences in the CTAs' common address space
        const unsigned u_even = u;
        bool longer = false;
        if ((pad || g_min == g_max) && whole <= u + WHOLE) {
            longer = whole > u + WHOLE_EXACT;
            u = max(1u, whole);
            v_head = pad ? nz * u : sum + nz * COST;
        } else if (pad) {
            // the smallest u for which the pieces fit the teams: sixteen candidates at once, two lanes each
            const unsigned mine = u + (lane & 15);
            unsigned n = 0;
            for (int b0 = 0; b0 < p.B; b0 += 32) {
                if (b0 != chunk) load_chunk(b0);
                for (int i = lane >> 4, e = min(32, p.B - b0); i < (e + 1) / 2 * 2; i += 2) {
                    const unsigned gi = (unsigned)__shfl_sync(0xffffffffu, g, i & 31);
                    n += quotient(gi + mine - 1, mine);
                }
            }
            n += __shfl_xor_sync(0xffffffffu, n, 16);
            const unsigned fit = __ballot_sync(0xffffffffu, LH * n <= teams && mine <= u_cut + PAD) & 0xffffu;
            if (fit) {
                u = __shfl_sync(0xffffffffu, mine, __ffs(fit) - 1);
                longer = u > u_cut + PAD_EXACT;
                v_head = u * __shfl_sync(0xffffffffu, n, __ffs(fit) - 1);
            } else {
                pad = false;
                u = u_cut;
                v_head = sum + nz * COST;
            }
        } else {
            v_head = sum + nz * COST;
        }
        two_rate = __fdividef((float)p.two_cuts, (float)max(1u, LH * (LH * nz > (unsigned)p.two_cuts ? sum + nz : sum)));
        if (longer) two_rate += __fdividef(1.f, (float)u_even);
        const unsigned v_layer = v_head * (unsigned)p.Hkv;
        pos = team * u;
        hi = min(pos + u, v_layer * (unsigned)p.n_layers);
        // where the run begins
        if (pos < hi) {
            layer = p.n_layers == 1 ? 0 : (int)quotient(pos, v_layer);
            unsigned rem = pos - (unsigned)layer * v_layer;
            for (int b0 = 0;; b0 += 32) {
                if (b0 != chunk) load_chunk(b0);
                const unsigned mine = padded((unsigned)g) * (unsigned)p.Hkv;
                unsigned incl = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                const unsigned m = __ballot_sync(0xffffffffu, rem < incl);
                if (m) {
                    const int at = __ffs(m) - 1;
                    b = b0 + at;
                    rem -= __shfl_sync(0xffffffffu, incl - mine, at);
                    break;
                }
                rem -= __shfl_sync(0xffffffffu, incl, 31);
            }
            const unsigned gp = padded((unsigned)__shfl_sync(0xffffffffu, g, b - chunk));
            head = (int)quotient(rem, gp);
            off = rem - (unsigned)head * gp;
        }
    }
    // How many of a piece's groups have their weights in two terms at head size 128.  The error is that of the output's rounding
    // and, independent of it and as large, that of the weights' rounding in the groups with one term: .00166 sqrt(1 + their
    // share).  A division among all SMs, two row tiles to an SM, has more and shorter pieces than one among pairs, or one that
    // leaves items whole, and has two terms in the first group of each of them (in two groups where an SM has a single row tile):
    // the error must not show which of the two it is.  So a piece has one such group for each piece that two_cuts teams would
    // begin in it, where those cut anywhere an item counting its groups and one; parts of one are spread evenly over the items
    // (golden ratio), and a tenth of one is added for what the spread misses.  (4208 drawn problems replayed: nowhere an error
    // larger than the finer division's by more than 0.05 %, 2.3 % less on average.)  Rel. error against 64 bits with the finer
    // division / one group of every piece / as it is, 32 / 8 heads: L = 512, 4 layers .00203 / .00219 / .00166, 32 layers .00215 /
    // .00220 / .00212, 8 layers of a single row tile .00185 / .00203 / .00166; L = 8192, 32 layers .00234 / .00234 / .00234.  Such a
    // group costs .8 k cycles more than another: eight ragged one-layer calls take 293 us, with none but the first of every piece
    // 288; the attention of 28 layers of 28 / 4 heads at 1500 and 2800 keys 162.2 and 161.4.
    // Where runs are longer by more than WHOLE_EXACT and PAD_EXACT, pieces shorter than those of two_cuts teams have been joined, that
    // had such a group each: one more for every u_even groups, which is at least as many as there were.  (9000 drawn problems replayed: no
    // share of two-term groups falls below that of a division with those limits; without this 255 did, by up to .23.  11 layers of two
    // sequences of eleven groups, a single row tile: an error of .00183 without.  46 steps of 4 to 29 layers that are divided so: errors up
    // to 7 % smaller than without, times the same on average and up to 5 % longer.)
    __device__ __forceinline__ int two_term_groups(int cnt, bool head, unsigned item) const {
        const float part = (float)((item * 2654435769u) >> 8) * (1.f / 16777216.f) + 0.1f;
        const int n = max(1, (int)(pad || head ? (float)(cnt - 1) * two_rate + part + 1.f : (float)cnt * two_rate + part));
        return min(lone ? 2 * n : n, cnt);
    }
    // The next piece of the run (all lanes agree); false at its end.  A piece that is not a whole item goes down in merges, too.
    __device__ __forceinline__ bool next(AttnPiece &d, AttnMerge *merges, volatile int *n_merge) {
        while (pos < hi) {
            const unsigned gg = (unsigned)__shfl_sync(0xffffffffu, g, b - chunk), gp = padded(gg);
            const int L = __shfl_sync(0xffffffffu, len, b - chunk);
            const unsigned end = min(gp, off + (hi - pos)), a = pos - off;
            const unsigned r0 = min(off, gg), r1 = min(end, gg);
            d.layer = layer; d.b = b; d.head = head; d.gb = (int)r0; d.cnt = (int)(r1 - r0); d.L = L;
            const bool part = r1 - r0 < gg;
            d.flags = (part ? PIECE_PARTIAL : 0) | (r0 == 0 ? PIECE_HEAD : 0) |
                      two_term_groups(d.cnt, r0 == 0, ((unsigned)layer * (unsigned)p.B + (unsigned)b) * (unsigned)p.Hkv + (unsigned)head) << PIECE_TWO_SHIFT;
            d.first = (int)quotient(a, u);
            if (r1 > r0 && part && n_part < 2) {
                if (lane == 0) {
                    AttnMerge m;
                    m.first = d.first; m.n = (int)quotient(a + gg - 1, u) - m.first + 1;
                    m.layer = layer; m.b = b; m.head = head; m.pad = 0;
                    merges[n_part] = m;
                    *n_merge = n_part + 1;
                }
                ++n_part;
            }
            pos += end - off;
            off = 0;
            if (++head == p.Hkv) {        // the next sequence that fits, in this layer or the next
                head = 0;
                unsigned m = __ballot_sync(0xffffffffu, g > 0) & ~(0xffffffffu >> (31 - (b - chunk)));
                while (!m && pos < hi) {
                    int b0 = chunk + 32;
                    if (b0 >= p.B) { b0 = 0; ++layer; }
                    if (b0 != chunk) load_chunk(b0);
                    m = __ballot_sync(0xffffffffu, g > 0);
                }
                b = chunk + (m ? __ffs(m) - 1 : 0);
            }
            if (r1 > r0) return true;
        }
        d.cnt = 0;
        return false;
    }
};

}  // namespace mtv
