// Tree attention (Section 3.2 / Fig. 2(b)) on the 5th-generation tensor cores, head sizes 64 and 128: all T tree nodes
// attend to the prefix and to their ancestors-or-self among the tree rows of the KV cache, for one layer or for all
// layers of a step in one launch.
//
// Work.  An ITEM is one (layer, sequence, KV head, row block): up to two tiles of 128 query rows — 128 / G whole tree
// nodes times the G query heads that share the KV head — against all 128-key groups of the sequence.  The grid is
// persistent, one CTA per SM; the key groups of all items, laid end to end, are divided evenly among the CTAs whatever
// the sequences' lengths, so that a CTA works on a run of consecutive PIECES: the end of one item, whole items, the
// beginning of another.  Items with several row blocks go to teams of CTAs that walk the same keys at the same time (the
// second read of a key group finds it in L2).  Every CTA derives its run from the lengths on the device.
//   * More items than teams: an item counts its groups plus AT_ITEM_COST (what starting and ending an item costs beside
//     its groups) and the cuts fall anywhere.
//   * Fewer: no CTA gets two pieces; the piece length is the smallest for which the pieces of all items fit the teams.
// Pieces that are not whole items leave O / l (fp32: where an item is cut must not show in its precision) and (m, l) in the
// workspace; at the end of the launch the CTAs that share an item meet at a counter and each combines a slice of its rows.
// They all do so when the device is this launch's alone (the grid never exceeds one CTA per SM), but nothing depends on it:
// a warp that has waited for a millisecond leaves its slice to the last one to leave and makes room.
//
// One piece.  Two STREAMS of 128 query rows by 128 keys share the tensor core: with two row tiles stream t owns tile t and
// both see every key group; with one row tile both use it and take alternate groups (merged at the end).  A stream runs
//     S(0) | PV(0) S(1) | PV(1) S(2) | ...
// with S of the next group issued right behind O += P V of this one, so that the softmax of one stream runs under the
// MMAs of the other.  P (bf16) overwrites the scores it came from in tensor memory; the tensor core executes one thread's
// MMAs in issue order, which is what lets S(j + 1) follow the PV(j) that reads P(j) under it.  Each stream has an issuing
// warp of its own and they take turns: an issue blocks until the tensor core has nearly caught up and a barrier test costs
// about a hundred cycles, so with one warp for both the tensor core idled through every test; without turns the streams
// fall into step and compute their softmax at the same time, with the tensor core idle (4.4 k cycles per pair of ticks
// against 3.6 k with one warp).
//   warps 0-7 / 8-15  softmax of stream 0 / 1: two threads own a query row, 64 columns each
//   warps 16 / 18     issue the MMAs of stream 0 / 1
//   warp 17           derives the CTA's pieces and requests K and V tiles (TMA) through a ring
//   warp 19           requests the query tiles (TMA) and clears the V rows past the last key (their P is 0, but 0 * NaN
//                     would poison O)
// Tensor memory: S of stream 0 and 1 (128 columns each), O of stream 0 and 1.
//
// What bounds it: per tile pair and key group the tensor core needs 2048 cycles at D = 128 and the special-function unit
// 1536 (a quarter of the exponentials run as polynomials on the FMA pipes); the dependent chain of one stream, scores
// visible -> exponentials -> P visible -> PV -> S, sets what is reached of it.  Four softmax warps per scheduler rather than
// two shorten that chain: a warp's exponentials take 1.2 k cycles for 128 columns, most of it latency.
//
// The reference of a row's exponentials is the maximum of its first group, rounded up to a whole number; it moves only when
// the sum of a thread's P in some later group exceeds 2^32, or one of its exponents 32 where a polynomial would not show it in
// the sum (from 128 on its result is meaningless).  P and O are floating-point numbers, so a reference that is not the maximum
// costs range, and the exactness of the largest weights, which a second term of P makes up for (see two_terms); in return no
// maximum is formed and nothing is exchanged between the two threads of a row in an ordinary group.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "attn_common.cuh"

namespace mtv {

// attention_pair.cu
bool attn_pair_eligible(int D, int G);
int attn_pair_plan(int T, int G, int B, int Hkv, int Lcap, int *n_blk_out);
int launch_tree_attn_pair(const mtv_tree *tree, int B, int Hq, int Hkv, const __nv_bfloat16 *q, const __nv_bfloat16 *k,
                          const __nv_bfloat16 *v, int64_t sb, int64_t sh, int64_t st, int Lcap, const int32_t *seq_lens,
                          float scale_log2, __nv_bfloat16 *out, int32_t *status, void *ws_o, float *ws_ml, int32_t *ws_order,
                          cudaStream_t stream);

constexpr int AT_BN = 128;            // keys per group
constexpr int AT_THREADS = 640;
constexpr int AT_SOFTMAX_WARPS = 16;
constexpr int AT_MMA_WARP = 16, AT_TMA_WARP = 17, AT_Q_WARP = 19;   // warp 18: MMAs of stream 1
constexpr int AT_PIECES = 4;          // piece descriptors in flight
constexpr int AT_ITEM_COST = 1;       // what an item costs beside its key groups, in groups
// How long a warp waits for the others of an item, in cycles.  In the bounds-checking build it looks once: nearly all slices
// are then left to the last warp.
#ifdef MTV_DEBUG_BOUNDS
constexpr long long AT_MERGE_WAIT = 0;
#else
constexpr long long AT_MERGE_WAIT = 2000000;
#endif
constexpr int AT_MAX_CTAS = 256;      // merge counters in the tree object: one pair per CTA
constexpr int AT_MAX_LAYERS = 64;     // layers per launch (two tensor maps each in the kernel's parameters)
// registers per thread: 96 at launch, moved from the four auxiliary warps to the sixteen softmax warps
constexpr int AT_LAUNCH_REGS = 96, AT_SOFTMAX_REGS = 104, AT_AUX_REGS = 64;
static_assert(512 * AT_SOFTMAX_REGS + 128 * AT_AUX_REGS <= AT_THREADS * AT_LAUNCH_REGS, "register split");
// P goes to the tensor core as bf16, whose rounding is the largest error beside the output's own.  Where a reference that
// follows the row's maximum made the largest weights exact (they were 1), a fixed reference does not: P then has a second bf16
// term, what the rounding of the first left.  At head size 64 in every group (O += P V is short there); at 128 in a piece's
// first group, whose maximum alone used to be the reference.  Rel. error against 64 bits with one term / two / the kernels that
// this one replaced: D = 64, L = 128: .00235 / .00166 / .00214, L <= 5003: .00233 / .00166 / .00210; D = 128, L = 512:
// .00235 / .00204 / .00268.  Cost: eight one-layer calls at head size 64 171 -> 198 us, steps at 128 1 to 2 %.
template <int D>
__host__ __device__ constexpr bool two_terms(int group) { return D == 64 || group == 0; }   // of the stream's groups of a piece
constexpr float AT_SUM_LIMIT = 4294967296.f;   // 2^32: a thread's sum of P over a group beyond it moves the reference
constexpr float LOG2E = 1.4426950408889634f;

// tensor-memory columns: S of stream t at 128 t, O at 256 + 128 t.  P lies over S, each half of the keys over its own scores:
// keys 0-63 at columns 0-31, keys 64-127 at 64-95; in two terms each quarter over its own: keys 0-31 at columns 0-15, their
// second terms at 16-31, and so on.
constexpr uint32_t TM_S = 0, TM_O = 256;

// Shared memory: two query tiles, the K/V ring, the (m, l) exchange of the two streams, barriers, descriptors.
template <int D>
struct AttnSmem {
    static constexpr uint32_t TILE = 128 * D * 2;          // 128 rows as D / 64 halves of 128-byte rows (128-byte swizzle)
    static constexpr uint32_t HALF = 128 * 128;
    static constexpr int STAGES = D == 128 ? 5 : 10;
    static constexpr uint32_t OFF_RING = 2 * TILE;
    static constexpr uint32_t OFF_ML = OFF_RING + STAGES * TILE;
    static constexpr uint32_t OFF_BAR = OFF_ML + 4 * 128 * 4;
    static constexpr int BAR_KV_FULL = 0;
    static constexpr int BAR_KV_EMPTY = STAGES;
    static constexpr int BAR_TAIL = 2 * STAGES;             // a V tile whose last rows must be cleared lands here first
    static constexpr int BAR_Q_FULL = 3 * STAGES;           // [2 tiles]
    static constexpr int BAR_Q_EMPTY = BAR_Q_FULL + 2;
    static constexpr int BAR_S = BAR_Q_EMPTY + 2;           // [2 streams] scores of a tick complete
    static constexpr int BAR_P = BAR_S + 2;                 // [2] P of a group written
    static constexpr int BAR_O = BAR_P + 2;                 // [2] the stream's O of the piece complete
    static constexpr int BAR_PC_FULL = BAR_O + 2;           // [AT_PIECES]
    static constexpr int BAR_PC_EMPTY = BAR_PC_FULL + AT_PIECES;
    static constexpr int BAR_XM = BAR_PC_EMPTY + AT_PIECES;    // [2 streams][4] the two warps of a row quarter, references
    static constexpr int BAR_XO = BAR_XM + 8;                  // [2][4] the two (one row tile: [4], the four) warps, results
    static constexpr int BAR_STAGED = BAR_XO + 8;              // [STAGES] the output rows staged in a slot have left it
    static constexpr int BAR_DRAIN = BAR_STAGED + STAGES;
    static constexpr int BAR_TURN = BAR_DRAIN + 2;          // [2] the stream's turn to issue
    static constexpr int BAR_COUNT = BAR_TURN + 2;
    static constexpr uint32_t OFF_DESC = OFF_BAR + (BAR_COUNT * 8 + 15) / 16 * 16;
    static constexpr uint32_t OFF_MISC = OFF_DESC + AT_PIECES * 32;
    static constexpr uint32_t TOTAL = OFF_MISC + 112;
    static_assert(TOTAL <= 227 * 1024, "shared memory");
};

struct AttnPiece {      // 32 bytes
    int layer, b, head, gb, cnt, L, flags, first;   // key groups [gb, gb + cnt); cnt = 0: no more pieces;
                                                    // first: first team that contributes to the item
};
constexpr int PIECE_PARTIAL = 1, PIECE_HEAD = 2;   // not a whole item; starts at the item's first group
struct AttnMerge {      // a partial piece of this CTA, for the merge at the end
    int first, n, layer, b, head, pad;             // first contributing team, number of them
};

template <int ML>
struct __align__(64) AttnMaps {
    CUtensorMap q, k[ML], v[ML];
};

struct AttnParams {
    const int32_t *seq_lens;
    const uint64_t *anc;     // [T][2]
    __nv_bfloat16 *out;      // [layers][B][T][Hq][D]
    uint4 *ws_o;             // [CTA][2 slabs][2 tiles][D / 4 chunks][128 rows] 16-byte chunks of O / l, fp32
    float2 *ws_ml;           // [CTA][2 slabs][2 tiles][128 rows] (m, l)
    int32_t *left;           // [CTA][2 slabs][16 warps] 1: the warp's slice of the item is left to the last one
    int32_t *arrive, *depart;   // [CTA] merge counters, zero between calls; depart counts slices left in its upper half
    int32_t *status;         // [B] or null
    int32_t *dev_error;
    float scale_log2;
    int B, T, G, Hq, Hkv, Lcap, n_layers;
    int npc, R;              // tree nodes per tile (128 / G) and the rows they fill
    unsigned inv_g;          // 65536 / G rounded up: row r of a tile is node (r * inv_g) >> 16 (exact for r < 256, G <= 8)
    int n_tiles, n_blk, teams;
    Gate gate;               // with a word: the inputs are complete behind it, the previous kernel is waited for at the end
};

// Operands: queries and keys K-major; V N-major, its next 64 columns one half tile further.
// bf16 x bf16 -> fp32, M = 128
constexpr uint32_t AT_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);
constexpr uint32_t AT_B_NMAJOR = 1u << 16;

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ float trunc_bf16(float x) { return bf16_hi(__float_as_uint(x)); }
// P = 2^(scale S - m) of 32 scores (two values per instruction where the instruction set has packed forms) and its
// contribution to the row sum.  Every fourth quadruple runs on the FMA pipes: the special-function unit is the bottleneck of
// a group.  pk: bf16 pairs; TWO: rest has what their rounding left, as bf16 pairs.  top: the largest exponent among those of
// the polynomials, which go wrong silently where ex2 gives +inf or NaN.
template <int DEGREE, bool TWO>
__device__ __forceinline__ void exp_quarter(const uint32_t (&s)[32], float2 sc2, float2 nm2, float2 &la, float2 &lb, uint32_t *pk, uint32_t *rest,
                                            float &top) {
#pragma unroll
    for (int e = 0; e < 16; e += 2) {
        const float2 x01 = __ffma2_rn(make_float2(__uint_as_float(s[2 * e]), __uint_as_float(s[2 * e + 1])), sc2, nm2);
        const float2 x23 = __ffma2_rn(make_float2(__uint_as_float(s[2 * e + 2]), __uint_as_float(s[2 * e + 3])), sc2, nm2);
        float2 p01, p23;
        if (e % 8 == 6) {
            top = ptx::fmax3_nan(top, x01.x, x01.y);
            top = ptx::fmax3_nan(top, x23.x, x23.y);
            p01 = exp2_poly2<DEGREE>(x01);
            p23 = exp2_poly2<DEGREE>(x23);
        } else {
            p01 = make_float2(ex2(x01.x), ex2(x01.y));
            p23 = make_float2(ex2(x23.x), ex2(x23.y));
        }
        la = __fadd2_rn(la, p01);
        lb = __fadd2_rn(lb, p23);
        if (TWO) {
            pk[e] = pack2_bf16(p01.x, p01.y);
            pk[e + 1] = pack2_bf16(p23.x, p23.y);
            const float2 r01 = __fadd2_rn(p01, make_float2(-bf16_lo(pk[e]), -bf16_hi(pk[e])));
            const float2 r23 = __fadd2_rn(p23, make_float2(-bf16_lo(pk[e + 1]), -bf16_hi(pk[e + 1])));
            rest[e] = pack2_bf16(r01.x, r01.y);
            rest[e + 1] = pack2_bf16(r23.x, r23.y);
        } else {
            pk[e] = pack2_bf16(p01.x, p01.y);
            pk[e + 1] = pack2_bf16(p23.x, p23.y);
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
// Build option -DMTV_TRACE: cycle stamps of one CTA's phases into a buffer given by mtv_trace_set (development aid).
#ifdef MTV_TRACE
__device__ long long *g_trace = nullptr;   // [ctas][8 rows][512]
#define TRACE_INIT(row, cond)                                                                          \
    int trace_n = 0;                                                                                   \
    long long *trace_row = g_trace && (cond) ? g_trace + ((size_t)blockIdx.x * 8 + (row)) * 512 : nullptr
#define TRACE()                                                          \
    do {                                                                 \
        if (trace_row && trace_n < 512) trace_row[trace_n++] = clock64(); \
    } while (0)
#else
#define TRACE_INIT(row, cond)
#define TRACE()
#endif

// Position of tiles in the order in which a piece of cnt groups consumes them, and back.
//   two row tiles: K0 V0 K1 V1 ...        one row tile: K0 K1 V0 K2 V1 K3 ... V(cnt-1)
// Behind them a piece that is a whole item takes a ring slot per row tile to stage its output rows in.
__device__ __forceinline__ int k_pos(bool one, int i) { return one ? (i == 0 ? 0 : 2 * i - 1) : 2 * i; }
__device__ __forceinline__ int v_pos(bool one, int i, int cnt) { return one ? min(2 * i + 2, 2 * cnt - 1) : 2 * i + 1; }
__device__ __forceinline__ void tile_at(bool one, int pos, int cnt, bool &is_v, int &idx) {
    if (!one) { is_v = pos & 1; idx = pos >> 1; return; }
    if (pos == 0) { is_v = false; idx = 0; return; }
    if (pos & 1) { idx = (pos + 1) >> 1; is_v = idx >= cnt; if (is_v) idx = cnt - 1; return; }
    is_v = true; idx = (pos - 2) >> 1;
}

__device__ __forceinline__ int ring_slots(const AttnPiece &d, bool one) {
    return 2 * d.cnt + (d.flags & PIECE_PARTIAL ? 0 : one ? 1 : 2);
}

// Output row of row r of tile t of a row block (in units of D elements from the item's first row), or -1 if it belongs to nobody.
// With a group size that does not divide 128 the last 128 - R rows of a tile do (whatever the tile's shared memory held is
// computed and never written out).
__device__ __forceinline__ int node_in_tile(const AttnParams &p, int r) { return (int)(((unsigned)r * p.inv_g) >> 16); }
__device__ __forceinline__ int out_row(const AttnParams &p, int blk, int t, int r) {
    const int n = node_in_tile(p, r), node = (blk * 2 + t) * p.npc + n;
    return r < p.R && node < p.T ? node * p.Hq + (r - n * p.G) : -1;
}
template <int D>
__device__ __forceinline__ uint4 *item_out(const AttnParams &p, int layer, int b, int hd) {      // first row of an item's output
    return reinterpret_cast<uint4 *>(p.out + (((size_t)layer * p.B + b) * p.T * p.Hq + hd * p.G) * D);
}
// slabs of the workspace: 16-byte chunk c (4 columns) of row r of tile t; the row's (m, l)
template <int D>
__device__ __forceinline__ uint4 *slab_o(const AttnParams &p, int cta, int slab, int t, int r, int c) {
    return p.ws_o + ((((unsigned)cta * 2 + slab) * 2 + t) * (D / 4) + c) * 128 + r;
}
__device__ __forceinline__ float2 *slab_ml(const AttnParams &p, int cta, int slab, int t, int r) {
    return p.ws_ml + (((unsigned)cta * 2 + slab) * 2 + t) * 128 + r;
}

// Rows of an item that is shared between CTAs: tile 0's, then tile 1's; contributor c0 combines its share of them, a thread per
// 16-byte chunk of the output, with the loads of several contributors in flight.  This is warp w's part of it.
template <int D>
__device__ __forceinline__ void merge_slice(const AttnParams &p, const AttnMerge &m, int c0, int w, int blk, bool one, int lane) {
    constexpr int VC = 2, NS = 3;                        // chunks per thread and contributor; contributors at a time
    const int rows = one ? p.R : 2 * p.R;
    const int per = (rows + m.n - 1) / m.n, r_begin = c0 * per;
    const int n_my = max(0, min(rows, r_begin + per) - r_begin);
    const unsigned inv_n = n_my > 0 ? ((1u << 20) + n_my - 1) / n_my : 0;    // e / n_my for e < 4096, n_my <= 256
    uint4 *dst = item_out<D>(p, m.layer, m.b, m.head);
#pragma unroll 1
    for (int e = w * 32 + lane; e < n_my * (D / 8); e += AT_SOFTMAX_WARPS * 32) {
        const int c = (int)(((unsigned)e * inv_n) >> 20), rr = r_begin + e - c * n_my;
        const int t = rr >= p.R, r = rr - t * p.R;
        float acc[8], mm = -INFINITY, wsum = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] = 0.f;
#pragma unroll 1
        for (int s0 = 0; s0 < m.n; s0 += NS) {
            float2 ml[NS];
            uint4 v[NS][VC];
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                const int s = min(s0 + k, m.n - 1), cta = (m.first + s) * p.n_blk + blk;
                const int sl = s == 0 ? 1 : 0;       // the first contributor's piece begins the item
                ml[k] = __ldcg(slab_ml(p, cta, sl, t, r));
#pragma unroll
                for (int q = 0; q < VC; ++q) v[k][q] = __ldcg(slab_o<D>(p, cta, sl, t, r, c * VC + q));
                if (s0 + k >= m.n) ml[k] = make_float2(-INFINITY, 0.f);
            }
            float mc = mm;
#pragma unroll
            for (int k = 0; k < NS; ++k) mc = fmaxf(mc, ml[k].x);
            const float resc = mm == -INFINITY ? 0.f : ex2(mm - mc);
            mm = mc;
            wsum *= resc;
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] *= resc;
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
        const int o = out_row(p, blk, t, r);
        if (o >= 0)
            dst[o * (D / 8) + c] =
                make_uint4(pack2_bf16(acc[0] * inv, acc[1] * inv), pack2_bf16(acc[2] * inv, acc[3] * inv),
                           pack2_bf16(acc[4] * inv, acc[5] * inv), pack2_bf16(acc[6] * inv, acc[7] * inv));
    }
}
// The slices that warps left, of one item, by the softmax warps of the CTA whose warp was the last to leave it.  (Out of the way of the
// usual case: as part of the merge below it cost the softmax loop, of all things, 4 %.)
template <int D>
static __device__ __noinline__ void merge_left(const AttnParams &p, const AttnMerge &m, int blk, bool one, int warp, int lane) {
    for (int u = warp; u < m.n * AT_SOFTMAX_WARPS; u += AT_SOFTMAX_WARPS) {
        const int c = u / AT_SOFTMAX_WARPS, w = u % AT_SOFTMAX_WARPS, cta = (m.first + c) * p.n_blk + blk;
        if (__ldcg(p.left + ((unsigned)cta * 2 + (c == 0 ? 1 : 0)) * AT_SOFTMAX_WARPS + w)) merge_slice<D>(p, m, c, w, blk, one, lane);
    }
}

// NEG: the scale is negative (only taken at head size 64, and kept apart so that the usual case pays nothing for it)
template <int D, int ML, bool NEG>
__global__ void __launch_bounds__(AT_THREADS, 1)
tree_attn_kernel(const __grid_constant__ AttnMaps<ML> maps, const __grid_constant__ AttnParams p) {
    using SM = AttnSmem<D>;
    constexpr int ST = SM::STAGES;
    extern __shared__ __align__(1024) unsigned char smem[];
    // Programmatic dependent launch: let the next kernel of the stream be set up while this one runs.
    let_next_start();
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t sbase = ptx::smem_u32(smem);
    auto bar = [&](int i) { return sbase + SM::OFF_BAR + (uint32_t)i * 8u; };
    AttnPiece *desc = reinterpret_cast<AttnPiece *>(smem + SM::OFF_DESC);
    AttnMerge *merges = reinterpret_cast<AttnMerge *>(smem + SM::OFF_MISC);                 // [2]
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + SM::OFF_MISC + 64);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + SM::OFF_MISC + 68);
    volatile int *n_merge = reinterpret_cast<volatile int *>(smem + SM::OFF_MISC + 72);     // partial pieces of this CTA
    int *left_items = reinterpret_cast<int *>(smem + SM::OFF_MISC + 108);                   // of this CTA's: bit i, merges[i]
    volatile int *beyond = reinterpret_cast<volatile int *>(smem + SM::OFF_MISC + 76);      // [2 streams][4] a sum beyond AT_SUM_LIMIT

    const int team = (int)blockIdx.x / p.n_blk, blk = (int)blockIdx.x % p.n_blk;
    const bool one = blk * 2 + 1 >= p.n_tiles;      // this CTA's row block has a single row tile

    if (warp == AT_Q_WARP && lane == 0) {
        ptx::prefetch_tensormap(&maps.q);
        if (ML == 1) { ptx::prefetch_tensormap(&maps.k[0]); ptx::prefetch_tensormap(&maps.v[0]); }
        for (int s = 0; s < ST; ++s) {
            ptx::mbar_init(bar(SM::BAR_KV_FULL + s), 1);
            ptx::mbar_init(bar(SM::BAR_KV_EMPTY + s), one ? 1 : 2);      // the streams that use the tile
            ptx::mbar_init(bar(SM::BAR_TAIL + s), 1);
            ptx::mbar_init(bar(SM::BAR_STAGED + s), one ? 16 : 8);       // the softmax warps of the row tile
        }
        for (int t = 0; t < 2; ++t) {
            ptx::mbar_init(bar(SM::BAR_Q_FULL + t), 1);
            ptx::mbar_init(bar(SM::BAR_Q_EMPTY + t), one ? 2 : 1);
            ptx::mbar_init(bar(SM::BAR_S + t), 1);
            ptx::mbar_init(bar(SM::BAR_P + t), 8);
            ptx::mbar_init(bar(SM::BAR_O + t), 1);
        }
        for (int i = 0; i < AT_PIECES; ++i) {
            ptx::mbar_init(bar(SM::BAR_PC_FULL + i), 1);
            ptx::mbar_init(bar(SM::BAR_PC_EMPTY + i), AT_SOFTMAX_WARPS + 3);   // + issuing and query warps
        }
        for (int i = 0; i < 8; ++i) {
            ptx::mbar_init(bar(SM::BAR_XM + i), 2);
            ptx::mbar_init(bar(SM::BAR_XO + i), one ? 4 : 2);
            beyond[i] = 0;
        }
        for (int t = 0; t < 2; ++t) {
            ptx::mbar_init(bar(SM::BAR_DRAIN + t), 1);
            ptx::mbar_init(bar(SM::BAR_TURN + t), 1);
        }
        ptx::fence_mbar_init();
        *abort_flag = 0;
        *n_merge = 0;
        *left_items = 0;
    }
    if (warp == AT_MMA_WARP) {
        ptx::tmem_alloc(ptx::smem_u32(const_cast<uint32_t *>(tmem_slot)), 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    // Ends the set-up; nothing in front of it touches global memory.  Behind it the previous kernel of the stream is
    // complete (its outputs may be this kernel's inputs, and it may share the workspace and counters), or what this kernel reads
    // was written before the gate's call.
    auto begin = [&]() -> uint32_t {
        if (p.gate.word && threadIdx.x == 0) wait_gate(p.gate);
        asm volatile("bar.sync 0, %0;" ::"n"(AT_THREADS) : "memory");
        ptx::tc_fence_after();
        if (p.gate.word) ptx::fence_proxy_async_global();      // (for the TMA loads that follow)
        else previous_done();
        return *tmem_slot;                    // tensor-memory base
    };

    // A wait that ran out: everybody stops at the next chance, the sticky error is raised.
    auto give_up = [&]() {
        *abort_flag = 1;
        atomicExch(p.dev_error, MTV_ERR_TIMEOUT);
    };
    // The pieces in order, for the warps that follow them (whole warp or one thread).
    auto read_piece = [&](int pi, AttnPiece &d) -> bool {
        if (!ptx::mbar_wait(bar(SM::BAR_PC_FULL + pi % AT_PIECES), (pi / AT_PIECES) & 1)) { give_up(); return false; }
        d = desc[pi % AT_PIECES];
        return !*abort_flag;
    };
    auto free_piece = [&](int pi) { ptx::mbar_arrive(bar(SM::BAR_PC_EMPTY + pi % AT_PIECES)); };

    if (warp >= AT_SOFTMAX_WARPS) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(AT_AUX_REGS));
    if (warp == AT_TMA_WARP) {
        // ------------------------------------------------------------ this CTA's pieces; K and V tiles
        const unsigned LH = (unsigned)p.n_layers * (unsigned)p.Hkv, teams = (unsigned)p.teams;
        int chunk = 0, len = 0, g = 0;        // lengths and group counts of sequences chunk .. chunk + 31, one per lane
        bool pad = false;
        unsigned u = 1, pos = 0, hi = 0, off = 0;
        int layer = 0, b = 0, head = 0;
        bool real = false;
        auto load_chunk = [&](int b0) {
            chunk = b0;
            const int at = b0 + lane;
            len = at < p.B && real ? p.seq_lens[at] : 0;
            g = at < p.B && len + p.T <= p.Lcap ? (len + p.T + AT_BN - 1) / AT_BN : 0;   // 0: does not fit, reported below
        };
        auto padded = [&](unsigned gg) { return gg == 0 ? 0u : pad ? (gg + u - 1) / u * u : gg + AT_ITEM_COST; };
        // The instructions of a launch come from L2 anew; this stretch runs once without lengths while the set-up goes on.
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            if (pass == 1) { (void)begin(); real = true; }
            unsigned sum = 0, nz = 0;
            for (int b0 = 0; b0 < p.B; b0 += 32) {
                load_chunk(b0);
                sum += __reduce_add_sync(0xffffffffu, (unsigned)g);
                nz += __popc(__ballot_sync(0xffffffffu, g > 0));
                if (real && blockIdx.x == 0 && p.status && b0 + lane < p.B) p.status[b0 + lane] = g > 0 ? MTV_OK : MTV_ERR_CAPACITY;
            }
            // Piece length u of either way to divide.  Padding to whole pieces wastes the teams it leaves idle, cutting
            // anywhere gives most teams two pieces, that is about two groups' worth of extra start and end: whichever is
            // shorter.
            const unsigned u_cut = max(1u, (LH * (sum + nz * AT_ITEM_COST) + teams - 1) / teams);
            unsigned v_head = 0;                  // length of one head's row of all sequences in the CTAs' common address space
            pad = LH * nz <= teams;
            u = pad ? max(1u, (LH * sum + teams - 1) / teams) : u_cut;
            for (;;) {
                v_head = 0;
                for (int b0 = 0; b0 < p.B; b0 += 32) {
                    if (b0 != chunk) load_chunk(b0);
                    v_head += __reduce_add_sync(0xffffffffu, padded((unsigned)g));
                }
                if (!pad || LH * (v_head / u) <= teams) break;
                if (++u > u_cut + 2) { pad = false; u = u_cut; }
            }
            const unsigned v_layer = v_head * (unsigned)p.Hkv;
            pos = (unsigned)team * u;
            hi = min(pos + u, v_layer * (unsigned)p.n_layers);
            // where the run begins
            if (pos < hi) {
                layer = (int)(pos / v_layer);
                unsigned rem = pos % v_layer;
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
                head = (int)(rem / gp);
                off = rem % gp;
            }
        }
        int n_part = 0;
        // the next piece of the run (all lanes agree); false at its end
        auto next_piece = [&](AttnPiece &d) -> bool {
            while (pos < hi) {
                const unsigned gg = (unsigned)__shfl_sync(0xffffffffu, g, b - chunk), gp = padded(gg);
                const int L = __shfl_sync(0xffffffffu, len, b - chunk);
                const unsigned end = min(gp, off + (hi - pos)), a = pos - off;
                const unsigned r0 = min(off, gg), r1 = min(end, gg);
                d.layer = layer; d.b = b; d.head = head; d.gb = (int)r0; d.cnt = (int)(r1 - r0); d.L = L;
                const bool part = r1 - r0 < gg;
                d.flags = (part ? PIECE_PARTIAL : 0) | (r0 == 0 ? PIECE_HEAD : 0);
                d.first = (int)(a / u);
                if (r1 > r0 && part && n_part < 2) {
                    if (lane == 0) {
                        AttnMerge m;
                        m.first = d.first; m.n = (int)((a + gg - 1) / u) - m.first + 1;
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
        };
        int n_pub = 0;
        bool ok = true;
        auto publish = [&](const AttnPiece &d) {
            if (n_pub >= AT_PIECES && !ptx::mbar_wait(bar(SM::BAR_PC_EMPTY + n_pub % AT_PIECES), (n_pub / AT_PIECES - 1) & 1)) ok = false;
            if (lane == 0) {
                desc[n_pub % AT_PIECES] = d;
                ptx::mbar_arrive(bar(SM::BAR_PC_FULL + n_pub % AT_PIECES));
            }
            __syncwarp();
            ++n_pub;
        };
        uint32_t seq = 0;                     // ring slots handed out so far: slot seq % ST
        uint32_t empty_ph = 0, staged_ph = 0, staging = 0;   // bit s: phase of either barrier of slot s; it stages output rows
        // slots [from, to) of a piece, in the order of their use
        auto request = [&](const AttnPiece &d, int from, int to) {
            const int n_keys = d.L + p.T, groups = (n_keys + AT_BN - 1) / AT_BN;
            for (int pos_t = from; pos_t < to && ok && !*abort_flag; ++pos_t, ++seq) {
                const uint32_t s = seq % ST;
                if (seq >= (uint32_t)ST) {
                    if ((staging >> s) & 1) {
                        ok = ptx::mbar_wait(bar(SM::BAR_STAGED + s), (staged_ph >> s) & 1);
                        staged_ph ^= 1u << s;
                    } else {
                        ok = ptx::mbar_wait(bar(SM::BAR_KV_EMPTY + s), (empty_ph >> s) & 1);
                        empty_ph ^= 1u << s;
                    }
                    if (!ok) break;
                }
                const bool stage = pos_t >= 2 * d.cnt;
                staging = (staging & ~(1u << s)) | (stage ? 1u << s : 0u);
                if (lane == 0) {
                    if (stage) {
                        ptx::mbar_arrive(bar(SM::BAR_KV_FULL + s));        // the slot is the softmax warps'
                    } else {
                        bool is_v;
                        int idx;
                        tile_at(one, pos_t, d.cnt, is_v, idx);
                        const bool tail = is_v && d.gb + idx == groups - 1 && (n_keys & 15) != 0;
                        const uint32_t fb = bar((tail ? SM::BAR_TAIL : SM::BAR_KV_FULL) + s);
                        ptx::mbar_arrive_expect_tx(fb, SM::TILE);
                        ptx::tma_load_5d(sbase + SM::OFF_RING + s * SM::TILE, is_v ? &maps.v[ML == 1 ? 0 : d.layer] : &maps.k[ML == 1 ? 0 : d.layer],
                                         fb, 0, (d.gb + idx) * AT_BN, 0, d.head, d.b);
                    }
                }
                __syncwarp();
            }
        };
        // A piece is published before the ring can block on the tiles of the one before it: the query warp looks ahead.
        AttnPiece cur, nxt;
        bool have = next_piece(cur);
        publish(cur);
        int done = 0;
        if (have) { done = min(ring_slots(cur, one), ST); request(cur, 0, done); }
        while (have && ok && !*abort_flag) {
            const bool more = next_piece(nxt);
            publish(nxt);
            request(cur, done, ring_slots(cur, one));
            done = 0;
            cur = nxt;
            have = more;
        }
        if (!ok && lane == 0) give_up();
        if (*abort_flag && lane == 0) {
            // copies still in flight get a bounded chance to land before the shared memory goes away
            for (uint32_t t = seq > (uint32_t)ST ? seq - ST : 0; t < seq; ++t)
                if (!ptx::mbar_wait(bar(SM::BAR_KV_FULL + t % ST), (t / ST) & 1)) break;
        }
    } else if (warp == AT_Q_WARP) {
        // ------------------------------------------------------------ query tiles; V rows past the last key
        const int n_q = one ? 1 : 2;
        (void)begin();
        uint32_t uses = 0, seq = 0, parity = 0;       // parity: bit s = phase of tail barrier s
        AttnPiece d;
        bool ok = true;
        auto request_q = [&]() {
            for (int t = 0; t < n_q && ok; ++t) {
                ok = uses == 0 || ptx::mbar_wait(bar(SM::BAR_Q_EMPTY + t), (uses - 1) & 1);
                if (ok && lane == 0) {
                    ptx::mbar_arrive_expect_tx(bar(SM::BAR_Q_FULL + t), (uint32_t)(p.R * D * 2));
                    for (int h = 0; h < D / 64; ++h)
                        ptx::tma_load_5d(sbase + t * SM::TILE + h * SM::HALF, &maps.q, bar(SM::BAR_Q_FULL + t), 0, d.head * p.G,
                                         (blk * 2 + t) * p.npc, h, d.layer * p.B + d.b);
                }
                __syncwarp();
            }
            ++uses;
        };
        for (int pi = 0; ok && read_piece(pi, d); ++pi) {
            __syncwarp();
            if (lane == 0) free_piece(pi);
            if (d.cnt == 0) break;
            request_q();                              // as soon as the piece before no longer needs the tiles
            const int n_keys = d.L + p.T, groups = (n_keys + AT_BN - 1) / AT_BN;
            if (ok && d.gb + d.cnt == groups && (n_keys & 15) != 0) {
                const uint32_t s = (seq + (uint32_t)v_pos(one, d.cnt - 1, d.cnt)) % ST;
                ok = ptx::mbar_wait(bar(SM::BAR_TAIL + s), (parity >> s) & 1);
                if (!ok) break;
                parity ^= 1u << s;
                // only the rows up to the next multiple of 16 take part in O += P V
                const int v0 = n_keys - (groups - 1) * AT_BN, v1 = (v0 + 15) / 16 * 16;
                unsigned char *vt = smem + SM::OFF_RING + s * SM::TILE;
                for (int e = v0 * 8 + lane; e < v1 * 8; e += 32)
#pragma unroll
                    for (int h = 0; h < D / 64; ++h)
                        *reinterpret_cast<uint4 *>(vt + h * SM::HALF + e * 16) = make_uint4(0u, 0u, 0u, 0u);
                ptx::fence_proxy_async();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(SM::BAR_KV_FULL + s));
            }
            seq += (uint32_t)ring_slots(d, one);
        }
        if (!ok && lane == 0) give_up();
        __syncwarp();
        if (*abort_flag && uses > 0)
            for (int t = 0; t < n_q; ++t) ptx::mbar_wait(bar(SM::BAR_Q_FULL + t), (uses - 1) & 1);
    } else {
        // ------------------------------------------------------------ MMA issuer of one stream
        // The whole warp walks the loop, so that descriptors and addresses stay in uniform registers; one elected lane
        // issues.  (A lane of a divergent warp has to move every operand of every MMA into uniform registers first:
        // 85-130 cycles an MMA, more than the 64 it takes.)
        const bool leader = ptx::elect_one();
        const int st = warp == AT_MMA_WARP ? 0 : 1, qt = one ? 0 : st;
        const int first = one ? st : 0, step = one ? 2 : 1;
        const uint32_t ring_lo = ptx::desc_lo(sbase + SM::OFF_RING, 16), ring_v_lo = ptx::desc_lo(sbase + SM::OFF_RING, SM::HALF);
        const uint32_t dq = ptx::desc_lo(sbase + qt * SM::TILE, 16);
        const uint32_t tmem = begin();
        const uint32_t t_s = tmem + TM_S + st * 128, t_o = tmem + TM_O + st * 128;
        AttnPiece d;
        uint32_t slot0 = 0, phase0 = 0;       // ring slot and phase of the piece's first tile
        uint32_t q_ph = 0, p_ph = 0, turn_ph = st == 0 ? 1 : 0;   // stream 0 begins: a wait for the phase before the first passes
        bool ok = true;
        TRACE_INIT(0 + 3 * st, lane == 0);
        for (int pi = 0; ok && read_piece(pi, d); ++pi) {
            __syncwarp();
            if (lane == 0) free_piece(pi);
            const int cnt = __shfl_sync(0xffffffffu, d.cnt, 0);
            if (cnt == 0) break;
            const int last_valid = d.L + p.T - (d.gb + cnt - 1) * AT_BN;       // keys of the piece's last group (or more than 128)
            const int last_steps = __shfl_sync(0xffffffffu, min(8, (last_valid + 15) / 16), 0);
            // ring slot and phase of the tile at a position of the piece
            auto tile = [&](int pos, uint32_t &s, uint32_t &ph) {
                const uint32_t t = slot0 + (uint32_t)pos;
                s = t % ST;
                ph = (phase0 + t / ST) & 1;
            };
            auto my_turn = [&]() { ok = ok && ptx::mbar_wait(bar(SM::BAR_TURN + st), turn_ph); turn_ph ^= 1; };
            auto pass_turn = [&]() { if (leader) ptx::mbar_arrive(bar(SM::BAR_TURN + (st ^ 1))); };
            auto wait_k = [&](int j, uint32_t &s) {
                uint32_t ph;
                tile(k_pos(one, j), s, ph);
                ok = ok && ptx::mbar_wait(bar(SM::BAR_KV_FULL + s), ph);
                ptx::tc_fence_after();
            };
            // S of group j (its K tile, in slot s, has landed).  The other stream is told shortly before the end: its
            // first MMA then follows without a gap.
            auto issue_s = [&](int j, uint32_t s) {
                const uint32_t dk = ring_lo + s * (SM::TILE >> 4);
                const uint32_t idesc = AT_IDESC | ((uint32_t)(2 * (j == cnt - 1 ? last_steps : 8)) << 17);   // N = keys rounded up to 16
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    constexpr uint32_t half = SM::HALF >> 4;
                    const uint32_t o = (kk / 4) * half + (kk % 4) * 2;
                    ptx::mma_ss_elect(t_s, dq + o, dk + o, ptx::DESC_HI, idesc, kk > 0, leader);
                    if (kk == D / 16 - 3) pass_turn();
                }
                ptx::tc_commit_elect(bar(SM::BAR_S + st), leader);
            };
            uint32_t ks = 0;
            ok = ptx::mbar_wait(bar(SM::BAR_Q_FULL + qt), q_ph);
            q_ph ^= 1;
            // Both streams take cnt / step + 1 turns (rounded up), whether they have something to issue or not.
            const int turns = (cnt + step - 1) / step + 1;
            if (first < cnt) wait_k(first, ks);
            my_turn();
            if (ok && first < cnt) issue_s(first, ks);
            else pass_turn();
            for (int i = 1; i < turns && ok && !*abort_flag; ++i) {
                const int j = first + (i - 1) * step;
                if (j >= cnt) { my_turn(); pass_turn(); continue; }
                const bool more = j + step < cnt;
                uint32_t s, ph;
                tile(v_pos(one, j, cnt), s, ph);
                TRACE();
                if (more) wait_k(j + step, ks);
                ok = ok && ptx::mbar_wait(bar(SM::BAR_KV_FULL + s), ph);
                TRACE();
                ok = ok && ptx::mbar_wait(bar(SM::BAR_P + st), p_ph);
                TRACE();
                my_turn();
                if (!ok) break;
                TRACE();
                ptx::tc_fence_after();
                const uint32_t dv = ring_v_lo + s * (SM::TILE >> 4);
                constexpr uint32_t idesc = AT_IDESC | AT_B_NMAJOR | ((uint32_t)(D / 8) << 17);
                const int steps = j == cnt - 1 ? last_steps : 8;
                // the A operand of sixteen keys: where P lies (see TM_S)
                auto issue_pv = [&](int kk, uint32_t col, bool accumulate) {
                    ptx::mma_ts_elect(t_o, t_s + (kk / 4) * 64 + col, dv + kk * 128, ptx::DESC_HI, idesc, accumulate, leader);
                };
                if (two_terms<D>(i - 1)) {
                    if (steps == 8 && D == 64) {
#pragma unroll
                        for (int kk = 0; kk < 16; ++kk)
                            issue_pv(kk & 7, kk / 2 % 2 * 32 + kk % 2 * 8 + kk / 8 * 16, j > first || kk > 0);
                    } else {
#pragma unroll 1
                        for (int kk = 0; kk < 2 * steps; ++kk) {
                            const int k = kk >> 1;
                            issue_pv(k, k / 2 % 2 * 32 + k % 2 * 8 + kk % 2 * 16, j > first || kk > 0);
                        }
                    }
                } else if (steps == 8) {
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) issue_pv(kk, kk % 4 * 8, true);
                } else {
#pragma unroll 1
                    for (int kk = 0; kk < steps; ++kk) issue_pv(kk, kk % 4 * 8, true);
                }
                p_ph ^= 1;
                TRACE();
                if (more) {
                    issue_s(j + step, ks);
                } else {
                    pass_turn();
                    ptx::tc_commit_elect(bar(SM::BAR_O + st), leader);
                }
            }
            const uint32_t t = slot0 + (uint32_t)__shfl_sync(0xffffffffu, ring_slots(d, one), 0);
            phase0 += t / ST;
            slot0 = t % ST;
        }
        if (!ok && lane == 0) give_up();
        __syncwarp();
        if (*abort_flag) {                // let what was issued finish
            ptx::tc_commit_elect(bar(SM::BAR_DRAIN + st), leader);
            ptx::mbar_wait(bar(SM::BAR_DRAIN + st), 0);
        }
        __syncwarp();
    }
    } else {
        // ------------------------------------------------------------ softmax warps
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(AT_SOFTMAX_REGS));
        // Thread (row, hf) of stream st: query row `row`, columns [64 hf, 64 hf + 64) of every group of the stream.
        const int qd = warp & 3, hf = (warp >> 2) & 1, st = warp >> 3;
        const int row = qd * 32 + lane;
        const int tile = one ? 0 : st;
        const int step = one ? 2 : 1, first = one ? st : 0;
        // 128 bits: the row's node sees tree row i
        const uint32_t *anc = reinterpret_cast<const uint32_t *>(p.anc + ((blk * 2 + tile) * p.npc + node_in_tile(p, row)) * 2);
        const bool mine = out_row(p, blk, tile, row) >= 0;
        auto anc_word = [&](int w) -> uint32_t {
            if (w < 0) return 0xffffffffu;     // prefix rows are visible to every node
            return w < 4 && mine ? anc[w] : 0u;    // past the tree rows: nothing
        };
        const uint32_t tmem = begin();
        const uint32_t lane_base = tmem + ((uint32_t)(qd * 32) << 16);
        const uint32_t t_s = lane_base + TM_S + st * 128 + hf * 64, t_o = lane_base + TM_O + st * 128;
        // (addresses in 32 bits and formed where they are used, phases in one word: the loop below has no register to spare)
        auto bar_s = [&]() { return bar(SM::BAR_S + st); };
        auto x_at = [&](int s, int h) { return sbase + SM::OFF_ML + (uint32_t)((s * 2 + h) * 128 + row) * 4u; };   // [stream][half][row]
        const uint32_t beyond_at = sbase + SM::OFF_MISC + 76u + (uint32_t)(st * 4 + qd) * 4u;
        if (lane < 2) p.left[((unsigned)blockIdx.x * 2 + lane) * AT_SOFTMAX_WARPS + warp] = 0;      // (released with the arrivals)
        constexpr uint32_t hidden = NEG ? 0x7f800000u : 0xff800000u;   // times the scale: -inf
        uint32_t phases = 0, seq = 0;             // bit 0: scores, 1: O, 2 and 3: the two exchanges
        auto phase = [&](int i) { return (phases >> i) & 1u; };
        bool ok = true;
        TRACE_INIT(1 + st, qd == 0 && hf == 0 && lane == 0);
        float m_used = -INFINITY, l = 0.f;
        bool begun = false;                    // the stream's O holds something of this piece
        auto meet = [&]() {                    // the two warps of these rows
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(SM::BAR_XM + st * 4 + qd));
            if (!ptx::mbar_wait(bar(SM::BAR_XM + st * 4 + qd), phase(2))) ok = false;
            phases ^= 4;
        };
        // The reference becomes max(both halves' mx) where `is_first` or that exceeds it; O and l (and P, if already written
        // against the old one) follow.  The two warps of the rows do this together.
        auto move_reference = [&](float mx, bool is_first, bool p_written) {
            ptx::sts_f32(x_at(st, hf), mx);
            meet();
            const float both = ceilf(fmaxf(mx, ptx::lds_f32(x_at(st, hf ^ 1))));
            const float m_new = is_first ? both : fmaxf(m_used, both);
            const bool need = !is_first && m_new != m_used && m_used != -INFINITY;
            if (__any_sync(0xffffffffu, need)) {
                const float alpha = need ? ex2(m_used - m_new) : 1.f;
                uint32_t x[16];
#pragma unroll 1
                for (int c = 0; p_written && c < 4; ++c) {       // both terms (a power of two: exact)
                    ptx::tmem_ld16(t_s + c * 16, x);
                    ptx::tmem_ld_wait_for16(x);
#pragma unroll
                    for (int e = 0; e < 16; ++e) x[e] = pack2_bf16(bf16_lo(x[e]) * alpha, bf16_hi(x[e]) * alpha);
                    ptx::tmem_st16(t_s + c * 16, x);
                }
#pragma unroll 1
                for (int c = 0; begun && c < D / 32; ++c) {      // this half's columns of O; the stream's earlier MMAs are complete
                    ptx::tmem_ld16(t_o + hf * (D / 2) + c * 16, x);
                    ptx::tmem_ld_wait_for16(x);
#pragma unroll
                    for (int e = 0; e < 16; ++e) x[e] = __float_as_uint(__uint_as_float(x[e]) * alpha);
                    ptx::tmem_st16(t_o + hf * (D / 2) + c * 16, x);
                }
                ptx::tmem_st_wait();
                l *= alpha;
            }
            m_used = m_new;
            if (is_first) return;                  // (the values exchanged are not written again before both warps' P is used)
            if (lane == 0) ptx::sts_u32(beyond_at, 0u);
            ptx::tc_fence_before();
            meet();
            ptx::tc_fence_after();
        };
        // Waits for the tensor core; meanwhile the other warp of these rows may ask to move the reference.  If it asks for the
        // very group that is waited for (complete between the two tests), this warp's P of that group does not exist yet: the
        // barrier, tested again behind the flag, then says so, the group is taken first, and the question is met at the next
        // wait.  Otherwise the asked-for group is the one whose P this warp has written, and the barrier cannot complete
        // before they have met.
        auto wait_tc = [&](uint32_t b, uint32_t parity) {
            const long long t0 = clock64();
            while (!ptx::mbar_try_wait(b, parity)) {
                if (ptx::lds_u32(beyond_at)) {
                    if (!ptx::mbar_try_wait(b, parity)) move_reference(-INFINITY, false, true);
                    continue;
                }
                if (clock64() - t0 > ptx::WAIT_CYCLE_LIMIT) { ok = false; return; }
            }
        };
        for (int pi = 0; ok; ++pi) {
            if (!ptx::mbar_wait(bar(SM::BAR_PC_FULL + pi % AT_PIECES), (pi / AT_PIECES) & 1)) { ok = false; break; }
            const volatile AttnPiece &d = desc[pi % AT_PIECES];    // (freed at the end of the piece)
            const int cnt = d.cnt;
            if (cnt == 0 || *abort_flag) break;
            const int a_first = d.gb * AT_BN + hf * 64 - d.L;      // tree row of this half's first column in the first group
            m_used = -INFINITY;
            l = 0.f;
            begun = false;
            const bool releases = qd == 0 && hf == 0 && lane == 0;
            if (first >= cnt && releases) ptx::mbar_arrive(bar(SM::BAR_Q_EMPTY + tile));
            // These scores are complete: this stream is done with their K tile and, the MMAs before them being complete too, with
            // the V tile of its previous group.
            auto scores_done = [&](int j) {
                phases ^= 1;
                TRACE();
                ptx::tc_fence_after();
                if (releases) {
                    ptx::mbar_arrive(bar(SM::BAR_KV_EMPTY + (seq + (uint32_t)k_pos(one, j)) % ST));
                    if (j >= step) ptx::mbar_arrive(bar(SM::BAR_KV_EMPTY + (seq + (uint32_t)v_pos(one, j - step, cnt)) % ST));
                    if (j + step >= cnt) ptx::mbar_arrive(bar(SM::BAR_Q_EMPTY + tile));
                }
            };
            auto p_done = [&]() {
                ptx::tmem_st_wait();
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(SM::BAR_P + st));
                begun = true;
                TRACE();
            };
            constexpr int DEGREE = D == 128 ? 3 : 4;
            const float2 sc2 = make_float2(p.scale_log2, p.scale_log2);
            // ---- the first group: its maximum, then its P in two terms, a quarter at a time (the scores are loaded twice, which
            //      costs less than the registers of all of them in two terms)
            if (first < cnt) {
                if (!ptx::mbar_wait(bar_s(), phase(0))) { ok = false; break; }
                scores_done(first);
                const int a0 = a_first + first * AT_BN;      // tree row of this half's first column
                auto quarter = [&](uint32_t (&q)[32], int c) {
                    ptx::tmem_ld32(t_s + 32 * c, q);
                    ptx::tmem_ld_wait_for(q);
                    if (a0 + 64 > 0) {       // bit e of vis is column e (see below)
                        const uint32_t vis = __funnelshift_r(anc_word((a0 >> 5) + c), anc_word((a0 >> 5) + c + 1), a0 & 31);
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (!((vis >> e) & 1u)) q[e] = hidden;
                    }
                };
                uint32_t q[32], pk[16], rest[16];
                float mx = -INFINITY;
#pragma unroll 1
                for (int c = 0; c < 2; ++c) {
                    quarter(q, c);
                    mx = fmaxf(mx, max_quarter<NEG>(q, p.scale_log2));
                }
                move_reference(mx, true, false);
                if (!ok) break;
                const float m_eff = m_used == -INFINITY ? 0.f : m_used;
                float2 la = make_float2(0.f, 0.f), lb = make_float2(0.f, 0.f);
                float top = -INFINITY;
#pragma unroll 1
                for (int c = 0; c < 2; ++c) {
                    quarter(q, c);
                    exp_quarter<DEGREE, true>(q, sc2, make_float2(-m_eff, -m_eff), la, lb, pk, rest, top);
                    ptx::tmem_st16(t_s + 32 * c, pk);
                    ptx::tmem_st16(t_s + 32 * c + 16, rest);
                }
                l = top != top ? top : (la.x + la.y) + (lb.x + lb.y);      // (no exponent is above 0 here)
                p_done();
            }
            for (int j = first + step; j < cnt; j += step) {
                float sum;
                bool asked = false;
#pragma unroll 1
                for (;;) {
                    if (!asked) {
                        wait_tc(bar_s(), phase(0));
                        if (!ok) break;
                        scores_done(j);
                    }
                    uint32_t qa[32], qb[32];
                    ptx::tmem_ld32(t_s, qa);
                    ptx::tmem_ld32(t_s + 32, qb);
                    ptx::tmem_ld_wait_for(qa);
                    ptx::tmem_ld_wait_for(qb);
                    const int a0 = a_first + j * AT_BN;      // tree row of this half's first column
                    if (a0 + 64 > 0) {
                        // the half overlaps the tree rows or the end of the cache: bit e of vis is column e of a quarter
                        const int w = a0 >> 5, sh = a0 & 31;     // floor division
                        const uint32_t w1 = anc_word(w + 1);
                        const uint32_t va = __funnelshift_r(anc_word(w), w1, sh), vb = __funnelshift_r(w1, anc_word(w + 2), sh);
#pragma unroll
                        for (int e = 0; e < 32; ++e) {
                            if (!((va >> e) & 1u)) qa[e] = hidden;
                            if (!((vb >> e) & 1u)) qb[e] = hidden;
                        }
                    }
                    if (asked) {      // (by a NaN, too, which the row's sum then has to show)
                        const float mx = fmaxf(max_quarter<NEG>(qa, p.scale_log2), max_quarter<NEG>(qb, p.scale_log2));
                        move_reference(mx > m_used + 16.f ? mx : -INFINITY, false, false);
                    }
                    const float m_eff = m_used == -INFINITY ? 0.f : m_used;
                    const float2 nm2 = make_float2(-m_eff, -m_eff);
                    float2 la = make_float2(0.f, 0.f), lb = make_float2(0.f, 0.f);
                    float top = -INFINITY;
                    // (rows that belong to nobody may hold anything)
                    auto fits = [&]() {
                        sum = (la.x + la.y) + (lb.x + lb.y);
                        if (asked && top != top) sum = top;
                        return asked || !__any_sync(0xffffffffu, mine && (sum > AT_SUM_LIMIT || !(top <= 32.f)));
                    };
                    if constexpr (two_terms<D>(1)) {
                        uint32_t pa[16], pb[16], ra[16], rb[16];
                        exp_quarter<DEGREE, true>(qa, sc2, nm2, la, lb, pa, ra, top);
                        exp_quarter<DEGREE, true>(qb, sc2, nm2, la, lb, pb, rb, top);
                        if (fits()) {
                            ptx::tmem_st16(t_s, pa);
                            ptx::tmem_st16(t_s + 16, ra);
                            ptx::tmem_st16(t_s + 32, pb);
                            ptx::tmem_st16(t_s + 48, rb);
                            break;
                        }
                    } else {
                        uint32_t pk[32];
                        exp_quarter<DEGREE, false>(qa, sc2, nm2, la, lb, pk, nullptr, top);
                        exp_quarter<DEGREE, false>(qb, sc2, nm2, la, lb, pk + 16, nullptr, top);
                        if (fits()) {
                            ptx::tmem_st32(t_s, pk);
                            break;
                        }
                    }
                    // rare: ask the other warp of these rows to come and move the reference, start over
                    asked = true;
                    if (lane == 0) ptx::sts_u32(beyond_at, 1u);
                }
                if (!ok) break;
                l += sum;
                p_done();
            }
            // ---- the stream's O of this piece
            const bool ran = first < cnt;       // (a one-tile piece of a single group has no second stream)
            if (ok && ran) {
                wait_tc(bar(SM::BAR_O + st), phase(1));
                phases ^= 2;
                if (releases) {
                    const int jl = one ? cnt - 1 - ((cnt - 1 - st) & 1) : cnt - 1;    // the stream's last group
                    ptx::mbar_arrive(bar(SM::BAR_KV_EMPTY + (seq + (uint32_t)v_pos(one, jl, cnt)) % ST));
                }
                ptx::tc_fence_after();
            }
            if (!ok) break;
            const bool partial = d.flags & PIECE_PARTIAL;
            const int slab = d.flags & PIECE_HEAD ? 1 : 0;
            // ---- the sums of a row's threads: l of the two halves and, in a one-tile piece, of the two streams:
            //      O = (w0 O0 + w1 O1) / (w0 l0 + w1 l1) with w_t = exp2(m_t - m)
            auto gather = [&]() {
                ptx::tc_fence_before();
                __syncwarp();
                const uint32_t bar_xo = bar(SM::BAR_XO + (one ? qd : st * 4 + qd));
                if (lane == 0) ptx::mbar_arrive(bar_xo);
                if (!ptx::mbar_wait(bar_xo, phase(3))) ok = false;
                phases ^= 8;
                ptx::tc_fence_after();
            };
            volatile float *x_m = reinterpret_cast<volatile float *>(smem + SM::TILE);   // [stream][row]: the unused query tile
            ptx::sts_f32(x_at(st, hf), l);
            if (one && hf == 0) x_m[st * 128 + row] = m_used;
            gather();
            float l_all = l + ptx::lds_f32(x_at(st, hf ^ 1)), m_all = m_used, w_own = 1.f, w_oth = 0.f;
            if (one) {
                const float l_oth = ptx::lds_f32(x_at(st ^ 1, 0)) + ptx::lds_f32(x_at(st ^ 1, 1));
                const float m_oth = x_m[(st ^ 1) * 128 + row];
                m_all = fmaxf(m_used, m_oth);
                w_own = m_used == -INFINITY ? 0.f : ex2(m_used - m_all);
                w_oth = m_oth == -INFINITY ? 0.f : ex2(m_oth - m_all);
                l_all = w_own * l_all + w_oth * l_oth;
            }
            if (!ok) break;
            const float inv_l = l_all == 0.f ? 0.f : 1.f / l_all;     // (NaN stays NaN)
            w_own *= inv_l;
            w_oth *= inv_l;
            // this thread's columns: a half of them, a quarter in a one-tile piece.  Partial results go to the workspace, whose
            // layout suits them; output rows are staged in a ring slot (each warp for itself, 16-byte chunks swizzled)
            // and leave as runs of 64 or 128 bytes: a thread storing its own row straight to memory took 6 k cycles.
            const bool other_ran = one && (st == 1 || cnt > 1);
            const int n_col = one ? D / 4 : D / 2, c_begin = one ? (st * 2 + hf) * n_col : hf * n_col;
            const uint32_t sq = seq + 2u * (uint32_t)cnt + (one ? 0 : st), slot = sq % ST;
            const uint32_t n_ch = (uint32_t)n_col / 8, rowb = n_ch * 16;          // chunks and bytes of a row's part
            unsigned char *stage = smem + SM::OFF_RING + slot * SM::TILE + (uint32_t)(one ? warp : warp & 7) * 32u * rowb;
            if (!partial && !ptx::mbar_wait(bar(SM::BAR_KV_FULL + slot), (sq / ST) & 1)) { ok = false; break; }
#pragma unroll 1
            for (int c0 = 0; c0 < n_col; c0 += 16) {
                uint32_t o[16];
                float v[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] = 0.f;
                if (ran) {
                    ptx::tmem_ld16(t_o + c_begin + c0, o);
                    ptx::tmem_ld_wait_for16(o);
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = __uint_as_float(o[e]) * w_own;
                }
                if (other_ran) {
                    ptx::tmem_ld16(lane_base + TM_O + (st ^ 1) * 128 + c_begin + c0, o);
                    ptx::tmem_ld_wait_for16(o);
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] = fmaf(__uint_as_float(o[e]), w_oth, v[e]);
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const uint32_t ch = (uint32_t)c0 / 8 + e;
                    if (!partial) {
                        *reinterpret_cast<uint4 *>(stage + lane * rowb + ((ch ^ (lane & (n_ch - 1))) << 4)) =
                            make_uint4(pack2_bf16(v[8 * e], v[8 * e + 1]), pack2_bf16(v[8 * e + 2], v[8 * e + 3]),
                                       pack2_bf16(v[8 * e + 4], v[8 * e + 5]), pack2_bf16(v[8 * e + 6], v[8 * e + 7]));
                    } else if (mine) {
#pragma unroll
                        for (int q = 0; q < 2; ++q)
                            *slab_o<D>(p, blockIdx.x, slab, tile, row, c_begin / 4 + 2 * ch + q) =
                                make_uint4(__float_as_uint(v[8 * e + 4 * q]), __float_as_uint(v[8 * e + 4 * q + 1]),
                                           __float_as_uint(v[8 * e + 4 * q + 2]), __float_as_uint(v[8 * e + 4 * q + 3]));
                    }
                }
            }
            if (!partial) {
                __syncwarp();
                const uint32_t sh = n_ch == 8 ? 3 : n_ch == 4 ? 2 : 1, ch = lane & (n_ch - 1);     // n_ch lanes store a row's part
                uint4 *dst = item_out<D>(p, d.layer, d.b, d.head) + c_begin / 8 + ch;
#pragma unroll 2
                for (uint32_t r = lane >> sh; r < 32; r += 32u >> sh) {
                    const uint4 x = *reinterpret_cast<const uint4 *>(stage + r * rowb + ((ch ^ (r & (n_ch - 1))) << 4));
                    const int o = out_row(p, blk, tile, qd * 32 + r);
                    if (o >= 0) dst[o * (D / 8)] = x;
                }
                ptx::fence_proxy_async();         // (the next tile comes into the slot through the async proxy)
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(SM::BAR_STAGED + slot));
            }
            if (partial) {
                if (mine && hf == 0 && (!one || st == 0)) *slab_ml(p, blockIdx.x, slab, tile, row) = make_float2(m_all, l_all);
                // this warp's part is written: tell those that share the item (each warp counts for itself)
                __syncwarp();
                if (lane == 0) {
                    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p.arrive + d.first * p.n_blk + blk) : "memory");
                }
            }
            seq += 2u * (uint32_t)cnt + (partial ? 0u : one ? 1u : 2u);
            __syncwarp();
            if (lane == 0) free_piece(pi);
            gather();                             // O and the exchanged values have been read: the next piece may overwrite them
        }
        if (!ok && lane == 0) give_up();
        // ---- merge of the items this CTA shares with others.  Every warp comes here when its own pieces are done.
        const int n_m = *n_merge;
#pragma unroll 1
        for (int i = 0; i < n_m; ++i) {
            const AttnMerge m = merges[i];
            const int ctr = m.first * p.n_blk + blk, all = m.n * AT_SOFTMAX_WARPS, c0 = team - m.first;
            int departed = 0, full = 0;
            if (lane == 0) {
                // relaxed polls (a round trip to L2 each), one acquire when the counter is full
                int32_t *c = p.arrive + ctr;
                const long long t0 = clock64();
                while (!(full = *reinterpret_cast<volatile int32_t *>(c) >= all))
                    if (clock64() - t0 > AT_MERGE_WAIT) break;
                if (full) {
                    (void)ld_acquire(c);
                    departed = atomicAdd(p.depart + ctr, 1);         // (its round trip overlaps the merge)
                } else {
                    p.left[((unsigned)blockIdx.x * 2 + (c0 == 0 ? 1 : 0)) * AT_SOFTMAX_WARPS + warp] = 1;
                    __threadfence();
                    departed = atomicAdd(p.depart + ctr, 0x10001) + 0x10000;
                }
            }
            if (__shfl_sync(0xffffffffu, full, 0)) merge_slice<D>(p, m, c0, warp, blk, one, lane);
            // The last warp to leave: its CTA does what others left, all parts and all marks being complete, and the counters go
            // back to zero (nobody polls them any more; the next call cannot start before this kernel has ended).
            if (lane == 0 && (departed & 0xffff) == all - 1) {
                if (departed >> 16) {
                    (void)ld_acquire(p.arrive + ctr);
                    (void)ld_acquire(p.depart + ctr);
                    atomicOr(left_items, 1 << i);
                }
                p.arrive[ctr] = 0;
                p.depart[ctr] = 0;
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == AT_MMA_WARP) ptx::tmem_dealloc(*tmem_slot, 512);
    if (warp < AT_SOFTMAX_WARPS && *left_items)       // (the other warps have too few registers for it)
        for (int i = 0; i < 2; ++i)
            if ((*left_items >> i) & 1) merge_left<D>(p, merges[i], blk, one, warp, lane);
    if (p.gate.word) previous_done();
}

// ---------------------------------------------------------------------------------------- host
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

// Encoding a map costs the host a microsecond or two and a step over 32 layers needs 65, so encoded maps are kept in a
// direct-mapped table keyed by everything that goes into them (a decode loop passes the same caches and strides step
// after step).
namespace {
struct MapKey {
    const void *base;
    cuuint64_t dims[5], strides[4];
    cuuint32_t box[5];
    int rank, device;
};
struct MapSlot {
    MapKey key;
    CUtensorMap map;
    bool valid = false;
};
constexpr int MAP_SLOTS = 2048;
MapSlot g_map_slots[MAP_SLOTS];
std::mutex g_map_mutex;
}  // namespace

bool tensor_map_bf16(CUtensorMap *map, const void *base, int rank, const cuuint64_t *dims, const cuuint64_t *strides_bytes,
                     const cuuint32_t *box) {
    MapKey key;
    memset(&key, 0, sizeof key);
    key.base = base;
    key.rank = rank;
    for (int i = 0; i < rank; ++i) { key.dims[i] = dims[i]; key.box[i] = box[i]; }
    for (int i = 0; i + 1 < rank; ++i) key.strides[i] = strides_bytes[i];
    if (cudaGetDevice(&key.device) != cudaSuccess) key.device = -1;
    const uint64_t h = ((uint64_t)(uintptr_t)base >> 8) * 0x9E3779B97F4A7C15ull + dims[1] * 0xC2B2AE3D27D4EB4Full +
                       box[1] * 0x165667B19E3779F9ull + (uint64_t)rank * 0x27D4EB2F165667C5ull;
    MapSlot &slot = g_map_slots[(h >> 40) % MAP_SLOTS];
    std::lock_guard<std::mutex> lock(g_map_mutex);
    if (slot.valid && memcmp(&slot.key, &key, sizeof key) == 0) {
        *map = slot.map;
        return true;
    }
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint32_t ones[5] = {1, 1, 1, 1, 1};
    if (fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(base), key.dims, key.strides, key.box, ones,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    slot.key = key;
    slot.map = *map;
    slot.valid = true;
    return true;
}

namespace {
// Row blocks of a problem and the CTAs that work on it.
struct AttnPlan {
    int npc, n_tiles, n_blk, teams;
};
AttnPlan attn_plan(int T, int G) {
    AttnPlan a;
    a.npc = 128 / G;                                 // tree nodes per tile
    a.n_tiles = (T + a.npc - 1) / a.npc;
    a.n_blk = (a.n_tiles + 1) / 2;
    const int sms = sm_count() < AT_MAX_CTAS ? sm_count() : AT_MAX_CTAS;
    a.teams = sms / a.n_blk;
    return a;
}
}  // namespace

// Workspace: two slabs (a CTA has at most two pieces that are not whole items) of two tiles for every CTA; the kernel on CTA
// pairs keeps a slab per key split of a query block and the order of the sequences.
AttnWs attn_ws_layout(const mtv_tree *t, int B, int Hq, int Hkv, int D, int Lcap) {
    AttnWs w;
    w.o_off = w.ml_off = w.left_off = w.total = 0;
    if (Hq / Hkv > 8) return w;          // the call itself refuses such a group; sizes are asked for before that
    const AttnPlan a = attn_plan(t->T, Hq / Hkv);
    const size_t slabs = (size_t)a.teams * a.n_blk * 2;
    w.ml_off = align_up(slabs * 2 * 128 * D * sizeof(float), 256);
    w.left_off = align_up(w.ml_off + slabs * 2 * 128 * sizeof(float2), 256);
    w.total = align_up(w.left_off + slabs * AT_SOFTMAX_WARPS * sizeof(int32_t), 256);
    if (attn_pair_eligible(D, Hq / Hkv)) {
        int n_blk = 1;
        const int ns = attn_pair_plan(t->T, Hq / Hkv, B, Hkv, Lcap, &n_blk);
        const size_t pair_slabs = ns > 1 ? (size_t)B * Hkv * n_blk * ns : 0;
        w.pair_ml_off = align_up(pair_slabs * 256 * D * sizeof(__nv_bfloat16), 256);
        w.order_off = align_up(w.pair_ml_off + pair_slabs * 256 * sizeof(float2), 256);
        w.total = std::max(w.total, align_up(w.order_off + (size_t)B * sizeof(int32_t), 256) + 256);
    }
    return w;
}

// Which kernel a call for ONE layer takes at head size 128 (several layers always take the one of this file: 32 layers at
// L = 512 take 60 us instead of 320, at L = 8192 290 instead of 570).  The kernel on CTA pairs starts and ends faster but
// leaves pairs idle where blocks and splits do not fill the 74; this one divides the groups evenly.  Only the capacity is known
// here, not the lengths.  us per call, lengths uniform in [h / 4, h] with h = all, a half, a quarter, an eighth of the
// capacity (pairs / even division):
//      7 sequences, 28 / 4 heads, capacity  8112:   72 / 60    41 / 38    26 / 30    18 / 25
//     12 sequences, 16 / 4 heads, capacity  8192:   71 / 58    40 / 35    25 / 28    17 / 25
//      4 sequences, T = 128,      capacity 32896:  266 / 197  137 / 149   78 / 70    42 / 42
//      3 sequences, 16 / 4 heads, capacity 20000:   38 / 39    25 / 31    18 / 27    15 / 22
//     16 sequences, 32 / 8 heads, capacity 32768:  427 / 381  217 / 198  106 / 126   70 / 91
//     16 sequences, 32 / 8 heads, capacity  4224:   59 / 68    42 / 53    31 / 31    27 / 23
// With more blocks than pairs the pairs are all busy, longest sequence first, and what the even division gains in a full cache it
// loses in one that is a quarter full: pairs.  With fewer, the even division is taken where the estimate for a full cache (us
// per group on a pair and on an SM, start and end) is better by a tenth; such a call on a nearly empty cache pays 7 us.
static bool pair_kernel_is_better(int T, int G, int B, int Hkv, int Lcap) {
    int n_blk = 1;
    const int ns = attn_pair_plan(T, G, B, Hkv, Lcap, &n_blk);
    const double blocks = (double)B * Hkv * n_blk, groups = (Lcap + AT_BN - 1) / AT_BN;
    if (blocks > 0.5 * sm_count()) return true;
    const double pairs = 0.97 * ceil(groups / ns) + 9.0, even = 1.55 * blocks * groups / sm_count() + 22.0;
    return pairs <= 1.1 * even;
}

template <int D, int ML, bool NEG>
static int launch_attn(const mtv_tree *tree, const AttnPlan &a, AttnParams &p, const __nv_bfloat16 *q, mtv_bf16 *const *k,
                       mtv_bf16 *const *v, int64_t sb, int64_t sh, int64_t st, cudaStream_t stream) {
    AttnMaps<ML> maps;
    {
        const cuuint64_t row = (cuuint64_t)p.Hq * D * 2;
        const cuuint64_t qd[5] = {64, (cuuint64_t)p.Hq, (cuuint64_t)p.T, D / 64, (cuuint64_t)p.B * p.n_layers};
        const cuuint64_t qs[4] = {D * 2, row, 128, row * p.T};
        const cuuint32_t qb[5] = {64, (cuuint32_t)p.G, (cuuint32_t)p.npc, 1, 1};
        const cuuint64_t cd[5] = {64, (cuuint64_t)p.Lcap, D / 64, (cuuint64_t)p.Hkv, (cuuint64_t)p.B};
        const cuuint64_t cs[4] = {(cuuint64_t)st * 2, 128, (cuuint64_t)sh * 2, (cuuint64_t)sb * 2};
        const cuuint32_t cb[5] = {64, AT_BN, D / 64, 1, 1};
        if (!tensor_map_bf16(&maps.q, q, 5, qd, qs, qb)) return MTV_ERR_CUDA;
        for (int l = 0; l < p.n_layers; ++l)
            if (!tensor_map_bf16(&maps.k[l], k[l], 5, cd, cs, cb) || !tensor_map_bf16(&maps.v[l], v[l], 5, cd, cs, cb))
                return MTV_ERR_CUDA;
    }
    static PerDeviceOnce once;
    bool *done = once.flag();
    if (!done || !*done) {
        cudaFuncAttributes fa;
        MTV_CUDA_CHECK(cudaFuncGetAttributes(&fa, tree_attn_kernel<D, ML, NEG>));
        if (fa.numRegs < AT_LAUNCH_REGS) {   // the register split would wait for registers that the launch does not own
            set_last_error_text("tree_attn_kernel: compiled with fewer registers than its split needs");
            return MTV_ERR_CUDA;
        }
        MTV_CUDA_CHECK(cudaFuncSetAttribute(tree_attn_kernel<D, ML, NEG>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnSmem<D>::TOTAL));
        if (done) *done = true;
    }
    TapScope tap(MTV_KERNEL_ATTN_PARTIAL, stream);
    MTV_CUDA_CHECK(launch_dependent(tree_attn_kernel<D, ML, NEG>, dim3(a.teams * a.n_blk), AT_THREADS, AttnSmem<D>::TOTAL, stream, maps, p));
    return MTV_OK;
}

// The attention of n_layers layers with the same lengths (q, out: layers back to back; k, v: host arrays of cache
// pointers), as few launches as the parameter space allows.  A launch of many layers divides all their work among the
// SMs at once: no layer ends with SMs that wait for its longest piece, and the start, the end and the merge of a launch
// are paid once.
int tree_attention_layers(const mtv_tree *tree, int B, int Hq, int Hkv, int D, int n_layers, const mtv_bf16 *q,
                          mtv_bf16 *const *k, mtv_bf16 *const *v, int64_t stride_b, int64_t stride_h, int64_t stride_t,
                          int Lcap, const int32_t *seq_lens, float scale, mtv_bf16 *out, int32_t *status, void *ws,
                          size_t ws_bytes, void *stream, const Gate *alongside) {
    if (!tree || !tree->on_device || !q || !k || !v || !seq_lens || !out || !ws) return MTV_ERR_INVALID_ARG;
    if (B < 1 || Hq < 1 || Hkv < 1 || n_layers < 1 || Lcap < tree->T) return MTV_ERR_INVALID_ARG;
    if ((D != 64 && D != 128) || Hq % Hkv != 0 || Hq / Hkv > 8 || B > 65535) return MTV_ERR_UNSUPPORTED_SHAPE;
    if (stride_t % 8 || stride_h % 8 || stride_b % 8 || stride_t < D) return MTV_ERR_INVALID_ARG;
    uintptr_t bits = (uintptr_t)q | (uintptr_t)out;
    for (int l = 0; l < n_layers; ++l) {
        if (!k[l] || !v[l]) return MTV_ERR_INVALID_ARG;
        bits |= (uintptr_t)k[l] | (uintptr_t)v[l];
    }
    if (bits & 15) return MTV_ERR_INVALID_ARG;
    if (D == 128 && scale < 0.f) return MTV_ERR_INVALID_ARG;
    const AttnWs Lw = attn_ws_layout(tree, B, Hq, Hkv, D, Lcap);
    if (ws_bytes < Lw.total) return MTV_ERR_WORKSPACE;
    if (n_layers == 1 && attn_pair_eligible(D, Hq / Hkv) && pair_kernel_is_better(tree->T, Hq / Hkv, B, Hkv, Lcap)) {
        TapScope tap(MTV_KERNEL_ATTN_PARTIAL, (cudaStream_t)stream);
        return launch_tree_attn_pair(tree, B, Hq, Hkv, reinterpret_cast<const __nv_bfloat16 *>(q),
                                     reinterpret_cast<const __nv_bfloat16 *>(k[0]), reinterpret_cast<const __nv_bfloat16 *>(v[0]),
                                     stride_b, stride_h, stride_t, Lcap, seq_lens,
                                     (scale == 0.f ? 1.f / sqrtf((float)D) : scale) * LOG2E, reinterpret_cast<__nv_bfloat16 *>(out),
                                     status, (char *)ws + Lw.o_off, reinterpret_cast<float *>((char *)ws + Lw.pair_ml_off),
                                     reinterpret_cast<int32_t *>((char *)ws + Lw.order_off), (cudaStream_t)stream);
    }
    const AttnPlan a = attn_plan(tree->T, Hq / Hkv);
    AttnParams p;
    p.seq_lens = seq_lens; p.anc = tree->d_anc; p.status = status; p.dev_error = tree->d_error;
    p.ws_o = reinterpret_cast<uint4 *>((char *)ws + Lw.o_off);
    p.ws_ml = reinterpret_cast<float2 *>((char *)ws + Lw.ml_off);
    p.left = reinterpret_cast<int32_t *>((char *)ws + Lw.left_off);
    p.arrive = tree->d_counters; p.depart = tree->d_counters + AT_MAX_CTAS;
    p.scale_log2 = (scale == 0.f ? 1.f / sqrtf((float)D) : scale) * LOG2E;
    p.B = B; p.T = tree->T; p.G = Hq / Hkv; p.Hq = Hq; p.Hkv = Hkv; p.Lcap = Lcap;
    p.npc = a.npc; p.R = a.npc * p.G; p.inv_g = (65536u + p.G - 1) / p.G; p.n_tiles = a.n_tiles; p.n_blk = a.n_blk; p.teams = a.teams;
    p.gate = alongside ? *alongside : Gate{};
    const size_t per_layer = (size_t)B * tree->T * Hq * D;
    cudaStream_t st = (cudaStream_t)stream;
    // positions in the common address space of a launch's groups are 32 bits wide
    const double layer_len = (double)B * Hkv * ((Lcap + AT_BN - 1) / AT_BN + 1);
    int per_launch = n_layers == 1 ? 1 : AT_MAX_LAYERS;
    while (per_launch > 1 && per_launch * layer_len > 4e9) per_launch /= 2;
    for (int l = 0; l < n_layers; l += per_launch) {
        if (l > 0) p.gate = Gate{};          // (it shares the counters and the workspace with the launch before)
        p.n_layers = n_layers - l < per_launch ? n_layers - l : per_launch;
        p.out = reinterpret_cast<__nv_bfloat16 *>(out) + l * per_layer;
        const __nv_bfloat16 *ql = reinterpret_cast<const __nv_bfloat16 *>(q) + l * per_layer;
        auto launch = p.n_layers == 1
                          ? (D == 128 ? launch_attn<128, 1, false> : scale < 0.f ? launch_attn<64, 1, true> : launch_attn<64, 1, false>)
                          : (D == 128 ? launch_attn<128, AT_MAX_LAYERS, false>
                                      : scale < 0.f ? launch_attn<64, AT_MAX_LAYERS, true> : launch_attn<64, AT_MAX_LAYERS, false>);
        const int rc = launch(tree, a, p, ql, k + l, v + l, stride_b, stride_h, stride_t, st);
        if (rc != MTV_OK) return rc;
    }
    MTV_CUDA_CHECK(cudaGetLastError());
    return MTV_OK;
}

}  // namespace mtv

extern "C" int tree_verify_attention(const mtv_tree_t *tree, int B, int Hq, int Hkv, int D,
                                     const mtv_bf16 *q, const mtv_bf16 *k_cache, const mtv_bf16 *v_cache,
                                     int64_t stride_b, int64_t stride_h, int64_t stride_t, int Lcap,
                                     const int32_t *seq_lens, float scale,
                                     mtv_bf16 *out, int32_t *status,
                                     void *ws, size_t ws_bytes, void *stream) {
    MTV_RANGE("tree_verify_attention");
    mtv_bf16 *k = const_cast<mtv_bf16 *>(k_cache), *v = const_cast<mtv_bf16 *>(v_cache);
    return mtv::tree_attention_layers(tree, B, Hq, Hkv, D, 1, q, &k, &v, stride_b, stride_h, stride_t, Lcap, seq_lens, scale,
                                      out, status, ws, ws_bytes, stream);
}

#ifdef MTV_TRACE
extern "C" int mtv_trace_set(long long *buf) {
    return cudaMemcpyToSymbol(mtv::g_trace, &buf, sizeof buf) == cudaSuccess ? 0 : -1;
}
#endif
