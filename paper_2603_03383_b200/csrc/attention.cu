// Tree attention (Section 3.2 / Fig. 2(b)) on the 5th-generation tensor cores, head sizes 64 and 128: all T tree nodes
// attend to the prefix and to their ancestors-or-self among the tree rows of the KV cache, for one layer or for all
// layers of a step in one launch.
//
// Work.  An ITEM is one (layer, sequence, KV head): the tiles of 128 query rows — 128 / G whole tree nodes times the G query
// heads that share the KV head — against all 128-key groups of the sequence.  The grid is persistent, one CTA per SM, a row
// tile per CTA; the CTAs that have the tiles of an item are a TEAM and walk the same keys at the same time.  The key groups of
// all items, laid end to end, are divided evenly among the teams whatever the sequences' lengths, so that a team works on a run
// of consecutive PIECES: the end of one item, whole items, the beginning of another.  Every CTA derives its run from the
// lengths on the device (PieceWalk):
//   * More items than teams: an item counts its groups plus ITEM_COST (what starting and ending an item costs beside
//     its groups) and the cuts fall anywhere.
//   * Fewer: no team gets two pieces; the piece length is the smallest for which the pieces of all items fit the teams.
//   * Whole items where that makes no run longer by more than WHOLE_COST.
// Pieces that are not whole items leave O / l (fp32: where an item is cut must not show in its precision) and (m, l) in the
// workspace; at the end of the launch the CTAs that share a tile meet at a counter and each combines a slice of its rows.
// They all do so when the device is this launch's alone (the grid never exceeds one CTA per SM), but nothing depends on it:
// a CTA that has waited for a millisecond leaves its slice to the last one to leave and makes room.
//
// PAIR (head size 128, more than one row tile): the CTAs of a team are cta_group::2 pairs, whose MMAs (M = 256) read half of
// a group's K and V from either CTA's shared memory, so that a tile and a group cost an SM 32 KB.  Else a CTA has K and V to
// itself: at head size 64 that is 32 KB as well, and a single row tile has nobody to share with.
//
// One tile.  A CTA keeps one accumulator O, which leaves room for THREE tiles of scores in tensor memory: S of group j + 3 is
// issued right behind O += P V of group j, over the P that this one has just read (the tensor core executes one thread's MMAs in
// issue order),
//     S(0) S(1) S(2) | PV(0) S(3) | PV(1) S(4) | ...
// so that a group's softmax has the time of two other groups' MMAs and two groups' softmax run at once.  (The kernel before this
// one had two row tiles in a CTA, with an accumulator and one tile of scores each: the chain scores -> P -> PV -> scores then took
// 1.63 k cycles per tile and group, of which the tensor core worked 1024.  Now 1.25 k in pieces of hundreds of groups, 1.4 k in those of
// sixty, 1.6 k in those of twenty; what is left of the chain is 1.6 k of softmax and 1.4 k of handing over, shared by three tiles.)  The pieces follow one another in the same way: the last PV of a piece
// has the first scores of the next one behind it, and the softmax warps take that one's first group before they read and write
// the finished O.  (With pieces one after the other eight one-layer calls on ragged lengths took 281 us, now 256; 21 layers of eight
// sequences of two or three groups 161 and 151, at head size 64 145 and 134; of one group 125 and 108.)
//   warps 0-7 / 8-15  softmax of groups 2, 4, .. / 1, 3, ..: two threads own a query row, 64 columns each; the first group is
//                     everybody's, 32 columns a thread.  (All on every group: 4 % slower at 32768 keys, as what a group costs a
//                     warp beside its exponentials is paid twice as often.)
//   warp 16           issues the MMAs (odd CTA of a pair: the slot keeper)
//   warp 17           derives the pieces and requests this CTA's part of K and V groups (TMA) through a ring
//   warp 18           the slot keeper (odd CTA: tells the even one what has landed, V rows past the last key cleared)
//   warp 19           requests the query tiles; clears the V rows past the last key (their P is 0, but 0 * NaN would poison O);
//                     meets the other contributors of an item
// The slot keeper follows the scores: it gives ring slots back as soon as the MMAs that read them are complete, and puts in its
// word for a group's PV when V, and K of the scores behind it, are there.  So the issuing warp has one barrier to test per
// group: a test costs it about a hundred cycles, and the tensor core has only some two MMAs queued.
//
// What bounds it: the tensor core needs 1024 cycles for a tile and group at D = 128 and the special-function unit as many; 8 PV
// and 8 S MMAs take 1025 with every other unit busy beside them, so the rest is the chain.  At 4 x 32768 keys, T = 128, the
// board's power limit takes the clock down to 1.1 GHz of 1.97 (at 16 x 1024 to 4096 keys, T = 64, to 1.18): 7112 groups x 1253 cycles are 8.1 ms.
//
// The reference of a row's exponentials is common to its four threads: the maximum of the piece's first group, rounded up to a
// whole number.  It moves only when the sum of a thread's P in some later group exceeds 2^32.  P and O are floating-point
// numbers, so a reference that is not the maximum costs range, and the exactness of the largest weights, which a second term of
// P makes up for (see two_terms); in return no maximum is formed and nothing is exchanged between the threads of a row in an
// ordinary group.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "attn_work.cuh"

namespace mtv {

// attention_pair.cu
bool attn_pair_eligible(int D, int G);
int attn_pair_plan(int T, int G, int B, int Hkv, int Lcap, int *n_blk_out);
int launch_tree_attn_pair(const mtv_tree *tree, int B, int Hq, int Hkv, const __nv_bfloat16 *q, const __nv_bfloat16 *k,
                          const __nv_bfloat16 *v, int64_t sb, int64_t sh, int64_t st, int Lcap, const int32_t *seq_lens,
                          float scale_log2, __nv_bfloat16 *out, int32_t *status, void *ws_o, float *ws_ml, int32_t *ws_order,
                          cudaStream_t stream);


constexpr int ITEM_COST = 2;          // what an item costs beside its key groups, in groups
// What partial results cost (written, met for, read and combined), in groups, as a limit to how much longer runs are made so that a team has
// one piece.  (5: ragged calls up to 3 % slower, four sequences of 8000 keys, T = 128, 531 us instead of 491.)
constexpr int MERGE_COST = 7;
// The same for items that stay whole, so that there are no partial results.  (5: 26 steps of 4 to 28 layers that differ in this 2.8 % slower on
// average, 86 instead of 75 us for 23 layers of 12 / 2 heads, two sequences of 1470 keys, T = 82; one-layer calls of ten to twelve groups,
// which have all their groups in two terms then, 2 to 8 % faster: 17.2 us instead of 18.0.)
constexpr int WHOLE_COST = 7;
constexpr int W_MMA = 16, W_TMA = 17, W_RELAY = 18, W_Q = 19;
constexpr int NB = 3;                 // tiles of scores
constexpr float LOG2E = 1.4426950408889634f;
// P goes to the tensor core as bf16, whose rounding is the largest error beside the output's own.  Where a reference that
// follows the row's maximum makes the largest weights exact (they are 1), a fixed reference does not: P then has a second bf16
// term, what the rounding of the first left: at head size 64 in every group (O += P V is short there), at 128 in the first
// groups of a piece, of which the first has the reference for its maximum.  How many is for PieceWalk to say (two_term_groups).
template <int D>
__device__ __forceinline__ bool two_terms(int group, int n_two) { return D == 64 || group < n_two; }
// tensor-memory columns: O, and three tiles of scores; P lies over its scores, each half of the keys over its own: keys 0-63
// at columns 0-31, keys 64-127 at 64-95; in two terms each quarter over its own: keys 0-31 at columns 0-15, their second
// terms at 16-31, and so on.
constexpr uint32_t TM_O = 0, TM_S = 128;

// PAIR: K and V are divided between the two CTAs of a pair
template <int D, bool PAIR>
struct AttnSmem {
    static constexpr uint32_t TILE = 128 * D * 2;          // a query tile: 128 rows as D / 64 halves of 128-byte rows (128-byte swizzle)
    static constexpr uint32_t HALF = 128 * 128;
    static constexpr uint32_t SLOT = TILE / (PAIR ? 2 : 1);    // this CTA's part of a K group (64 keys of a pair) or V group (64 columns)
    static constexpr uint32_t K_HALF = PAIR ? 64 * 128 : HALF; // the next 64 columns of K
    static constexpr int STAGES = 10 * 16384 / SLOT;
    // The slot keeper's word on a group's PV takes in the K of the scores behind it, three groups on, where the slot that this K
    // comes into was given back two groups ago.  With five slots it is requested only when the scores of the next group but one
    // are complete, and PV need not wait for that: the issuing warp waits for it, behind PV.
    static constexpr bool K_AHEAD = STAGES >= 2 * NB + 4;
    static constexpr uint32_t OFF_RING = 2 * TILE;         // two query tiles: this piece's and the next one's; a place is free once its last scores are complete
    static constexpr uint32_t OFF_X = OFF_RING + STAGES * SLOT;
    static constexpr uint32_t OFF_BAR = OFF_X + 4 * 128 * 4;
    static constexpr int BAR_KV_FULL = 0;                  // of the even CTA of a pair: both parts (its own copy and the odd CTA's word)
    static constexpr int BAR_KV_EMPTY = BAR_KV_FULL + STAGES;
    static constexpr int BAR_TAIL = BAR_KV_EMPTY + STAGES; // V whose last rows must be cleared lands here first (odd CTA: not used)
    static constexpr int BAR_Q_FULL = BAR_TAIL + STAGES;   // [2 tiles] of the even CTA: both CTAs' tiles
    static constexpr int BAR_Q_EMPTY = BAR_Q_FULL + 2;     // [2]
    static constexpr int BAR_S = BAR_Q_EMPTY + 2;          // [3] scores of a group complete, and the PV in front of them
    static constexpr int BAR_P = BAR_S + NB;               // [3] even CTA: what PV of a group and the scores behind it wait for
    static constexpr int BAR_PV = BAR_P + NB;              // [2] PV of a piece's last group but two / but one, where no scores follow it
    static constexpr int BAR_O = BAR_PV + 2;               // O of a piece complete
    static constexpr int BAR_O_FREE = BAR_O + 1;           // even CTA: O of a piece read
    static constexpr int BAR_PC_FULL = BAR_O_FREE + 1;     // [AT_PIECES]
    static constexpr int BAR_PC_EMPTY = BAR_PC_FULL + AT_PIECES;
    static constexpr int BAR_XM = BAR_PC_EMPTY + AT_PIECES;    // [4] the four warps of a row quarter: meet
    static constexpr int BAR_XO = BAR_XM + 4;                  // [4] have read what they exchanged
    static constexpr int BAR_XG = BAR_XO + 4;                  // [4] have written all P of a piece
    static constexpr int BAR_OUT = BAR_XG + 4;                 // a partial result is written by the sixteen warps
    static constexpr int BAR_GO = BAR_OUT + 1;                 // [2] all partial results of an item are there (or the slice is left)
    static constexpr int BAR_DRAIN = BAR_GO + 2;
    static constexpr int BAR_COUNT = BAR_DRAIN + 1;
    static constexpr uint32_t OFF_DESC = OFF_BAR + (BAR_COUNT * 8 + 15) / 16 * 16;
    static constexpr uint32_t OFF_MISC = OFF_DESC + AT_PIECES * 32;
    static constexpr uint32_t OFF_ASK = OFF_MISC + 64;     // [4] a row quarter is asked to move its reference
    static constexpr uint32_t OFF_AT = OFF_ASK + 16;       // [4][4] the group that a warp of the quarter is at
    static constexpr uint32_t TOTAL = OFF_AT + 64;
    static_assert(TOTAL <= 227 * 1024, "shared memory");
    // bf16 x bf16 -> fp32, M = 256 over a pair, 128 in a CTA; N = 128 keys or D columns; V N-major
    static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((PAIR ? 256u : 128u) >> 4) << 24;
    static constexpr uint32_t IDESC_QK = IDESC | (128u >> 3) << 17, IDESC_PV = IDESC | (uint32_t)(D >> 3) << 17 | 1u << 16;
};

// The half groups of all pieces of a CTA, in the order in which the tensor core takes them and the ring has them: K of three groups, then
// V(0) K(3) V(1) K(4) ..; groups count on from piece to piece, but K runs ahead into the next piece only, whose query tile is there.
// K of group k, `before` being the first group of the piece before its own:
__device__ __forceinline__ int k_pos(int k, int before) { return k + max(k - (NB - 1), before); }
// V of group j of a piece that begins with group `first` and has cnt groups, nxt in the next one:
__device__ __forceinline__ int v_pos(int first, int j, int cnt, int nxt) { return 2 * (first + j) + min(NB, cnt + nxt - j); }

// V rows from the last key on, up to the next multiple of 16: only they take part in O += P V
template <int HALVES>
__device__ __forceinline__ void clear_tail(unsigned char *v, int valid, int lane) {
    for (int e = valid * 8 + lane; e < (valid + 15) / 16 * 16 * 8; e += 32)
#pragma unroll
        for (int h = 0; h < HALVES; ++h) *reinterpret_cast<uint4 *>(v + h * 16384 + e * 16) = make_uint4(0u, 0u, 0u, 0u);
    ptx::fence_proxy_async();
}

// PAIR: launched in clusters of two.  NEG: the scale is negative (only taken at head size 64, and kept apart so that the usual case
// pays nothing for it)
// ML: tensor maps per cache kind: one (a layer, or layers in one map), or one for each of up to ML layers
template <int D, bool PAIR, int ML, bool NEG>
__global__ void __launch_bounds__(AT_THREADS, 1)
tree_attn_kernel(const __grid_constant__ AttnMaps<ML> maps, const __grid_constant__ AttnParams p) {
    using SM = AttnSmem<D, PAIR>;
    constexpr int STAGES = SM::STAGES;
    extern __shared__ __align__(1024) unsigned char smem[];
    let_next_start();
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t rank = PAIR ? ptx::cluster_ctarank() : 0;
    const uint32_t sbase = ptx::smem_u32(smem);
    auto bar = [&](int i) { return sbase + SM::OFF_BAR + (uint32_t)i * 8u; };
    // the same barrier in the even CTA of a pair
    auto arrive_lead = [&](int i, uint32_t count = 1) {
        if (PAIR) ptx::mbar_arrive_remote(ptx::mapa(bar(i), 0), count);
        else ptx::mbar_arrive(bar(i), count);
    };
    AttnPiece *desc = reinterpret_cast<AttnPiece *>(smem + SM::OFF_DESC);
    AttnMerge *merges = reinterpret_cast<AttnMerge *>(smem + SM::OFF_MISC);                  // [2], 48 bytes
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + SM::OFF_MISC + 48);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + SM::OFF_MISC + 52);
    volatile int *n_merge = reinterpret_cast<volatile int *>(smem + SM::OFF_MISC + 56);      // partial pieces of this CTA
    volatile int *left_items = reinterpret_cast<volatile int *>(smem + SM::OFF_MISC + 60);   // of this CTA's: bit i, merges[i]; bit 2 + i: slice left

    // CTA blk of the team has row tile blk (blk = 2 block + rank)
    const int team = (int)blockIdx.x / p.n_blk, blk = (int)blockIdx.x % p.n_blk;

    if (warp == W_Q && lane == 0) {
        ptx::prefetch_tensormap(&maps.q);
        if (ML == 1) { ptx::prefetch_tensormap(&maps.k[0]); ptx::prefetch_tensormap(&maps.v[0]); }
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(bar(SM::BAR_KV_FULL + s), PAIR && rank == 0 ? 2 : 1);
            ptx::mbar_init(bar(SM::BAR_KV_EMPTY + s), 1);
            ptx::mbar_init(bar(SM::BAR_TAIL + s), 1);
        }
        for (int t = 0; t < 2; ++t) {
            ptx::mbar_init(bar(SM::BAR_Q_FULL + t), PAIR && rank == 0 ? 2 : 1);
            ptx::mbar_init(bar(SM::BAR_Q_EMPTY + t), 1);
            ptx::mbar_init(bar(SM::BAR_PV + t), 1);
        }
        for (int b = 0; b < NB; ++b) {
            ptx::mbar_init(bar(SM::BAR_S + b), 1);
            ptx::mbar_init(bar(SM::BAR_P + b), (PAIR ? 2 : 1) * (16 + 1));      // softmax warps (eight, counted twice, or all) and slot keeper of each CTA
        }
        ptx::mbar_init(bar(SM::BAR_O), 1);
        ptx::mbar_init(bar(SM::BAR_O_FREE), (PAIR ? 2 : 1) * AT_SOFTMAX_WARPS);
        for (int i = 0; i < AT_PIECES; ++i) {
            ptx::mbar_init(bar(SM::BAR_PC_FULL + i), 1);
            ptx::mbar_init(bar(SM::BAR_PC_EMPTY + i), AT_SOFTMAX_WARPS + 3);   // + warps 16, 18 and 19
        }
        for (int i = 0; i < 4; ++i) {
            ptx::mbar_init(bar(SM::BAR_XM + i), 4);
            ptx::mbar_init(bar(SM::BAR_XO + i), 4);
            ptx::mbar_init(bar(SM::BAR_XG + i), 4);
            ptx::sts_u32(sbase + SM::OFF_ASK + i * 4, 0u);
        }
        ptx::mbar_init(bar(SM::BAR_OUT), AT_SOFTMAX_WARPS);
        for (int i = 0; i < 2; ++i) ptx::mbar_init(bar(SM::BAR_GO + i), 1);
        ptx::mbar_init(bar(SM::BAR_DRAIN), 1);
        ptx::fence_mbar_init();
        *abort_flag = 0;
        *left_items = 0;
    }
    if (warp == W_MMA) {
        const uint32_t at = ptx::smem_u32(const_cast<uint32_t *>(tmem_slot));
        if (PAIR) { ptx::tmem_alloc_pair(at, 512); ptx::tmem_relinquish_pair(); }
        else { ptx::tmem_alloc(at, 512); ptx::tmem_relinquish(); }
    }
    // Ends the set-up (of both CTAs: nothing goes to the peer before); nothing in front of it touches global memory.  Behind it
    // the previous kernel of the stream is complete (its outputs may be this kernel's inputs, and it may share the workspace and
    // counters), or what this kernel reads was written before the gate's call.
    auto begin = [&]() -> uint32_t {
        if (p.gate.word && threadIdx.x == 0) wait_gate(p.gate);
        __syncwarp();
        ptx::tc_fence_before();
        if (PAIR) { ptx::cluster_arrive(); ptx::cluster_wait(); }
        else asm volatile("bar.sync 0, %0;" ::"n"(AT_THREADS) : "memory");
        ptx::tc_fence_after();
        if (p.gate.word) ptx::fence_proxy_async_global();      // (for the TMA loads that follow)
        else previous_done();
        return *tmem_slot;                    // tensor-memory base
    };
    // A wait that ran out: both CTAs stop at the next chance, the sticky error is raised.
    auto give_up = [&]() {
        *abort_flag = 1;
        if (PAIR) ptx::st_cluster_u32(ptx::mapa(ptx::smem_u32(const_cast<int *>(abort_flag)), rank ^ 1), 1u);
        atomicExch(p.dev_error, MTV_ERR_TIMEOUT);
    };
    // The pieces in order, for the warps that follow them.
    auto read_piece = [&](int pi, AttnPiece &d) -> bool {
        if (!ptx::mbar_wait(bar(SM::BAR_PC_FULL + pi % AT_PIECES), (pi / AT_PIECES) & 1)) { give_up(); return false; }
        d = desc[pi % AT_PIECES];
        return !*abort_flag;
    };
    auto free_piece = [&](int pi) { ptx::mbar_arrive(bar(SM::BAR_PC_EMPTY + pi % AT_PIECES)); };

    if (warp >= AT_SOFTMAX_WARPS) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(AT_AUX_REGS));
    if (warp == W_TMA) {
        // ------------------------------------------------------------ the pair's pieces; this CTA's halves of K and V
        // (the pair, or CTA, that has the last tile of an odd number of them)
        PieceWalk<ITEM_COST, WHOLE_COST, MERGE_COST> walk(p, team, lane, (blk | 1) >= p.n_tiles);
        // The work is divided while the kernel before this one ends, by the lengths that are there (a call that follows another has
        // nothing that changes them in between), and looked at again behind it: eight one-layer calls on ragged lengths take 291 us
        // instead of 314, at head size 64 164 instead of 172.
        AttnPiece cur, nxt;
        bool have = false;
        const bool early = walk.early();
        if (lane == 0) *n_merge = 0;
        __syncwarp();
        if (early) {
            walk.divide();
            have = walk.next(cur, merges, n_merge);
        }
        (void)begin();
        if (!early || !walk.still_so()) {
            if (lane == 0) *n_merge = 0;
            __syncwarp();
            walk.divide();
            have = walk.next(cur, merges, n_merge);
        }
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
        uint32_t slot = 0, use = 0;           // the next ring slot, and how often all have been handed out
        // a half of group j of a piece
        auto request = [&](const AttnPiece &d, bool is_v, int j) {
            if (use > 0 && !ptx::mbar_wait(bar(SM::BAR_KV_EMPTY + slot), (use - 1) & 1)) { ok = false; return; }
            if (lane == 0) {
                const int n_keys = d.L + p.T, key = (d.gb + j) * AT_BN, l = ML == 1 ? 0 : d.layer;
                const int c3 = ML == 1 ? d.head + p.fold.head_b * d.b : d.head, c4 = ML == 1 ? p.fold.b * d.b + p.fold.layer * d.layer : d.b;
                const bool tail = rank == 0 && is_v && key + AT_BN >= n_keys && (n_keys & 15) != 0;
                const uint32_t fb = bar((tail ? SM::BAR_TAIL : SM::BAR_KV_FULL) + slot), dst = sbase + SM::OFF_RING + slot * SM::SLOT;
                ptx::mbar_arrive_expect_tx(fb, SM::SLOT);
                if (is_v) ptx::tma_load_5d(dst, &maps.v[l], fb, 0, key, (int)rank, c3, c4);      // (one CTA: all columns)
                else ptx::tma_load_5d(dst, &maps.k[l], fb, 0, key + (int)rank * 64, 0, c3, c4);
            }
            __syncwarp();
            if (++slot == STAGES) { slot = 0; ++use; }
        };
        // A piece is published when the one before it begins; the first copies do not wait for that.
        publish(cur);
        int a = 0;                            // groups whose K is requested ahead of V
        if (have)
            for (; a < min(NB - 1, cur.cnt); ++a) request(cur, false, a);
        while (have && ok && !*abort_flag) {
            const bool more = walk.next(nxt, merges, n_merge);
            publish(nxt);
            for (int j = 0; j < cur.cnt && ok && !*abort_flag;) {
                const int g = j + a;
                if (a < NB && g < cur.cnt + nxt.cnt) {
                    const bool n = g >= cur.cnt;
                    AttnPiece d;
                    d.layer = n ? nxt.layer : cur.layer; d.b = n ? nxt.b : cur.b; d.head = n ? nxt.head : cur.head;
                    d.gb = n ? nxt.gb : cur.gb; d.L = n ? nxt.L : cur.L;
                    request(d, false, n ? g - cur.cnt : g);
                    ++a;
                } else {
                    request(cur, true, j);
                    ++j;
                    --a;
                }
            }
            cur = nxt;
            have = more;
        }
        walk.report();
        if (!ok && lane == 0) give_up();
        if (*abort_flag) {
            // copies still in flight land before the shared memory goes away (their barriers may wait for the peer as well, so
            // this takes the time that a copy cannot take)
            const long long t0 = clock64();
            while (clock64() - t0 < 4000000ll) {}
        }
    } else if (warp == W_Q) {
        // ------------------------------------------------------------ query tiles; even CTA: V rows past the last key
        (void)begin();
        uint32_t parity = 0;                  // bit s: phase of tail barrier s
        int first = 0, n_out = 0;             // groups of the pieces before; partial results
        if (lane < 2) p.left[blockIdx.x * 2 + lane] = 0;     // (released with the first of them)
        AttnPiece d, e;
        bool ok = true;
        auto request_q = [&](int pi, const AttnPiece &x) {
            const uint32_t t = pi & 1;
            ok = pi < 2 || ptx::mbar_wait(bar(SM::BAR_Q_EMPTY + t), (pi / 2 - 1) & 1);
            if (ok && lane == 0) {
                ptx::mbar_arrive_expect_tx(bar(SM::BAR_Q_FULL + t), (uint32_t)(p.R * D * 2));
                for (int h = 0; h < D / 64; ++h)
                    ptx::tma_load_5d(sbase + t * SM::TILE + h * SM::HALF, &maps.q, bar(SM::BAR_Q_FULL + t), 0, x.head * p.G, blk * p.npc, h,
                                     x.layer * p.B + x.b);
            }
            __syncwarp();
        };
        // the odd CTA's tile has landed: tell the even one
        auto tell_q = [&](int pi) {
            if (!PAIR || rank == 0) return;
            ok = ok && ptx::mbar_wait(bar(SM::BAR_Q_FULL + (pi & 1)), (pi / 2) & 1);
            if (ok && lane == 0) arrive_lead(SM::BAR_Q_FULL + (pi & 1));
            __syncwarp();
        };
        bool have = read_piece(0, d) && d.cnt > 0;
        __syncwarp();
        if (lane == 0) free_piece(0);
        if (have) { request_q(0, d); tell_q(0); }
        for (int pi = 0; have && ok; ++pi) {
            // the next piece's tile goes to the other place, as soon as the scores of the piece before this one are complete
            if (!read_piece(pi + 1, e)) break;
            __syncwarp();
            if (lane == 0) free_piece(pi + 1);
            have = e.cnt > 0;
            if (have) { request_q(pi + 1, e); if (!ok) break; tell_q(pi + 1); if (!ok) break; }
            const int n_keys = d.L + p.T, groups = (n_keys + AT_BN - 1) / AT_BN;
            if (rank == 0 && d.gb + d.cnt == groups && (n_keys & 15) != 0) {
                const uint32_t s = (uint32_t)v_pos(first, d.cnt - 1, d.cnt, e.cnt) % STAGES;
                ok = ptx::mbar_wait(bar(SM::BAR_TAIL + s), (parity >> s) & 1);
                if (!ok) break;
                parity ^= 1u << s;
                clear_tail<PAIR ? 1 : D / 64>(smem + SM::OFF_RING + s * SM::SLOT, n_keys - (groups - 1) * AT_BN, lane);
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(SM::BAR_KV_FULL + s));
            }
            if (d.flags & PIECE_PARTIAL) {
                // The softmax warps have written their parts: one fence and one word for all of them.  (A release by every
                // warp: 16 fences one after the other, and 16 times the polls and additions at the counters.)
                ok = ptx::mbar_wait(bar(SM::BAR_OUT), n_out & 1);
                if (!ok) break;
                ++n_out;
                if (lane == 0) {
                    __threadfence();
                    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(merge_counter(p, d.first, blk)) : "memory");
                }
            }
            first += d.cnt;
            d = e;
        }
        // The items that this CTA shares with others: a look at the counter until all parts are there, then the softmax warps
        // combine this CTA's slice.
        if (ok && !*abort_flag && lane == 0) {
            const int n_m = *n_merge;
            for (int i = 0; i < n_m; ++i) {
                const int n = merges[i].n, first = merges[i].first;
                int32_t *c = merge_counter(p, first, blk);
                const long long t0 = clock64();
                bool full;
                while (!(full = ld_acquire(c) >= n))
                    if (clock64() - t0 > AT_MERGE_WAIT) break;
                if (!full) {
                    p.left[blockIdx.x * 2 + (team == first ? 1 : 0)] = 1;
                    *left_items |= 4 << i;
                    __threadfence();
                }
                ptx::mbar_arrive(bar(SM::BAR_GO + i));
                const int before = atomicAdd(c + AT_DEPART, full ? 1 : 0x10001), marked = (before >> 16) + (full ? 0 : 1);
                // The last one to leave: its CTA does what others left, all parts and all marks being complete, and the counters go
                // back to zero (nobody looks at them any more; the next call cannot start before this kernel has ended).
                if ((before & 0xffff) == n - 1) {
                    if (marked) {
                        (void)ld_acquire(c);
                        (void)ld_acquire(c + AT_DEPART);
                        *left_items |= 1 << i;
                    }
                    c[0] = 0;
                    c[AT_DEPART] = 0;
                }
            }
        }
        __syncwarp();
        if (!ok && lane == 0) give_up();
    } else if (PAIR && warp == W_RELAY && rank == 1) {
        // ------------------------------------------------------------ odd CTA: what has landed, V rows past the last key cleared
        (void)begin();
        int at = 0, first = 0;
        AttnPiece d, e;
        bool ok = true;
        auto pass = [&](int until, bool tail, int n_keys) {       // tail: the last of them has rows to clear
            for (; ok && at < until && !*abort_flag; ++at) {
                const uint32_t s = (uint32_t)at % STAGES;
                ok = ptx::mbar_wait(bar(SM::BAR_KV_FULL + s), ((uint32_t)at / STAGES) & 1);
                if (!ok) break;
                if (tail && at == until - 1) {
                    clear_tail<PAIR ? 1 : D / 64>(smem + SM::OFF_RING + s * SM::SLOT, n_keys - (n_keys - 1) / AT_BN * AT_BN, lane);
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive_remote_release(ptx::mapa(bar(SM::BAR_KV_FULL + s), 0));
                } else if (lane == 0) {
                    arrive_lead(SM::BAR_KV_FULL + s);
                }
                __syncwarp();
            }
        };
        bool have = read_piece(0, d) && d.cnt > 0;
        __syncwarp();
        if (lane == 0) free_piece(0);
        if (have) pass(min(NB, d.cnt), false, 0);     // (whatever the next piece has)
        for (int pi = 0; have && ok; ++pi) {
            if (!read_piece(pi + 1, e)) break;
            __syncwarp();
            if (lane == 0) free_piece(pi + 1);
            const int n_keys = d.L + p.T;
            pass(v_pos(first, d.cnt - 1, d.cnt, e.cnt) + 1, (d.gb + d.cnt) * AT_BN >= n_keys && (n_keys & 15) != 0, n_keys);
            first += d.cnt;
            d = e;
            have = d.cnt > 0;
        }
        if (!ok && lane == 0) give_up();
    } else if (warp == W_RELAY || (PAIR && rank == 1)) {
        // ------------------------------------------------------------ slot keeper
        // Two things go their own ways here, so it looks at their barriers in turns: slots whose scores (and PV in front of them) are
        // complete, and groups whose V, and K of the scores behind it, are there.  (With a wait for either in order a slot of K
        // came back three half groups late: 32 layers of a single row tile, with its five slots, took 169 us instead of 148 at 4096
        // keys, 130 instead of 110 at 8192 of four heads.)  Its word on every group goes into BAR_P, behind its scores, so that it is
        // never more than a phase behind them.  When scores are complete, everything in front of them in the ring is done with.
        (void)begin();
        if (lane == 0) {
            int pi = 0, before = 0, first = 0;            // first groups of the piece before and of the piece of the next word
            int cnt = 0, nxt = 0, scored = 0, told = 0;   // their groups; scores complete and words given, from `first` on
            uint32_t freed = 0;                           // half groups given back
            AttnPiece d;
            bool known = false;                           // nxt
            if (read_piece(0, d)) cnt = d.cnt;
            auto there = [&](int at) { return ptx::mbar_test(bar(SM::BAR_KV_FULL + (uint32_t)at % STAGES), ((uint32_t)at / STAGES) & 1); };
            long long t0 = clock64();
            while (cnt > 0 && !*abort_flag) {
                if (!known && ptx::mbar_test(bar(SM::BAR_PC_FULL + (pi + 1) % AT_PIECES), ((pi + 1) / AT_PIECES) & 1)) {
                    nxt = reinterpret_cast<const volatile AttnPiece *>(desc)[(pi + 1) % AT_PIECES].cnt;
                    known = true;
                }
                const uint32_t k = (uint32_t)(first + scored);
                if (scored < cnt + nxt && ptx::mbar_test(bar(SM::BAR_S + k % NB), (k / NB) & 1)) {
                    for (const uint32_t to = (uint32_t)k_pos((int)k, scored < cnt ? before : first); freed <= to; ++freed)
                        ptx::mbar_arrive(bar(SM::BAR_KV_EMPTY + freed % STAGES));
                    ++scored;
                    if (scored == cnt) ptx::mbar_arrive(bar(SM::BAR_Q_EMPTY + (pi & 1)));
                    else if (scored == cnt + nxt) ptx::mbar_arrive(bar(SM::BAR_Q_EMPTY + ((pi + 1) & 1)));
                    t0 = clock64();
                }
                if (known && told < scored) {
                    const int at = v_pos(first, told, cnt, nxt);
                    if (rank == 1 || (there(at) && (!SM::K_AHEAD || told + NB >= cnt + nxt || there(at + 1)))) {
                        arrive_lead(SM::BAR_P + (first + told) % NB);
                        if (++told == cnt) {
                            free_piece(pi++);
                            before = first;
                            first += cnt;
                            scored -= cnt;
                            told = 0;
                            cnt = nxt;
                            nxt = 0;
                            known = false;
                        }
                        t0 = clock64();
                    }
                }
                if (clock64() - t0 > ptx::WAIT_CYCLE_LIMIT) { give_up(); break; }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ even CTA: MMA issuer
        // The whole warp walks the loop, so that descriptors and addresses stay in uniform registers; one elected lane
        // issues.  Barriers are tested while the tensor core still has MMAs queued.
        const bool leader = ptx::elect_one();
        const uint32_t ring_lo = ptx::desc_lo(sbase + SM::OFF_RING, 16), ring_v_lo = ptx::desc_lo(sbase + SM::OFF_RING, SM::HALF);
        const uint32_t tmem = begin();
        // what it has to know of a piece: groups, how many of them in two terms, steps of sixteen keys of the last
        struct Part { int cnt, n_two, last_steps; };
        bool ok = true;
        auto look = [&](int pi) {
            Part x = {0, 0, 0};
            AttnPiece d;
            if (!read_piece(pi, d)) { ok = false; return x; }
            const int last_valid = d.L + p.T - (d.gb + d.cnt - 1) * AT_BN;         // keys of the piece's last group (or more than 128)
            x.cnt = __shfl_sync(0xffffffffu, d.cnt, 0);
            x.n_two = __shfl_sync(0xffffffffu, d.flags >> PIECE_TWO_SHIFT, 0);
            x.last_steps = __shfl_sync(0xffffffffu, min(8, (last_valid + 15) / 16), 0);
            return x;
        };
        auto commit = [&](int i) {
            if (PAIR) ptx::tc_commit_pair_mask_elect(bar(i), 3, leader);
            else ptx::tc_commit_elect(bar(i), leader);
        };
        uint32_t s = 0, ph_kv = 0;                // ring slot and its phase
        auto next_slot = [&]() { if (++s == STAGES) { s = 0; ph_kv ^= 1; } };
        auto next_group = [](int t) { return t == 2 * NB - 1 ? 0 : t + 1; };
        // t_s, t_v: the next scores and the next PV as group number modulo 6: tile of scores, and from 3 on its barriers' odd phases
        int pi = 0, j = 0, ahead = 0, t_s = 0, t_v = 0, q_there = -1;      // next PV: group j of piece pi; groups that scores are ahead
        bool known = false, go = false, k_there = false;      // the next piece is; all that PV waits for, K of the scores behind it are there
        Part cur = look(0), nxt = {0, 0, 0};
        while (ok && cur.cnt > 0) {
            // scores as far ahead as there are tiles for them, into the next piece at most
            while (ahead < NB && j + ahead < cur.cnt + nxt.cnt) {
                const int q = j + ahead < cur.cnt ? pi : pi + 1;
                if (q != q_there) {
                    ok = ptx::mbar_wait(bar(SM::BAR_Q_FULL + (q & 1)), (q / 2) & 1);
                    q_there = q;
                }
                if (!k_there) ok = ok && ptx::mbar_wait(bar(SM::BAR_KV_FULL + s), ph_kv);
                if (!ok) break;
                ptx::tc_fence_after();
                const int b = t_s >= NB ? t_s - NB : t_s;
                const uint32_t dq = ptx::desc_lo(sbase + (q & 1) * SM::TILE, 16), t_d = tmem + TM_S + b * 128, dk = ring_lo + s * (SM::SLOT >> 4);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t oq = (kk / 4) * (SM::HALF >> 4) + (kk % 4) * 2, o_k = (kk / 4) * (SM::K_HALF >> 4) + (kk % 4) * 2;
                    if (PAIR) ptx::mma_pair_ss_elect(t_d, dq + oq, dk + o_k, ptx::DESC_HI, SM::IDESC_QK, kk > 0, leader);
                    else ptx::mma_ss_elect(t_d, dq + oq, dk + o_k, ptx::DESC_HI, SM::IDESC_QK, kk > 0, leader);
                    if (kk == D / 16 - 4) go = __all_sync(0xffffffffu, ptx::mbar_test(bar(SM::BAR_P + (t_v >= NB ? t_v - NB : t_v)), t_v >= NB));
                }
                commit(SM::BAR_S + b);
                next_slot();
                t_s = next_group(t_s);
                ++ahead;
                k_there = false;
            }
            if (!ok) break;
            if (j == cur.cnt) {                   // on to the next piece
                __syncwarp();
                if (lane == 0) free_piece(pi);
                ++pi;
                j = 0;
                cur = nxt;
                nxt = {0, 0, 0};
                known = false;
                continue;
            }
            if (!known) {
                nxt = look(pi + 1);
                known = true;
                continue;
            }
            if (j == 0 && pi > 0) ok = ptx::mbar_wait(bar(SM::BAR_O_FREE), (pi - 1) & 1);
            const int b = t_v >= NB ? t_v - NB : t_v;
            if (!go) ok = ok && ptx::mbar_wait(bar(SM::BAR_P + b), t_v >= NB);
            if (!ok) break;
            go = false;
            ptx::tc_fence_after();
            const uint32_t dv = ring_v_lo + s * (SM::SLOT >> 4), t_p = tmem + TM_S + b * 128;
            // the A operand of sixteen keys: where P lies (see TM_S)
            auto issue_pv = [&](int kk, uint32_t col, bool accumulate) {
                const uint32_t t_a = t_p + (kk / 4) * 64 + col;
                if (PAIR) ptx::mma_pair_ts_elect(tmem + TM_O, t_a, dv + kk * 128, ptx::DESC_HI, SM::IDESC_PV, accumulate, leader);
                else ptx::mma_ts_elect(tmem + TM_O, t_a, dv + kk * 128, ptx::DESC_HI, SM::IDESC_PV, accumulate, leader);
            };
            const int steps = j == cur.cnt - 1 ? cur.last_steps : 8;
            if (two_terms<D>(j, cur.n_two)) {
                if (D == 64 && steps == 8) {
#pragma unroll
                    for (int kk = 0; kk < 16; ++kk) issue_pv(kk & 7, kk / 2 % 2 * 32 + kk % 2 * 8 + kk / 8 * 16, j > 0 || kk > 0);
                } else {
#pragma unroll 1
                    for (int kk = 0; kk < 2 * steps; ++kk) {
                        const int k = kk >> 1;
                        issue_pv(k, k / 2 % 2 * 32 + k % 2 * 8 + kk % 2 * 16, j > 0 || kk > 0);
                    }
                }
            } else if (steps == 8) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) issue_pv(kk, kk % 4 * 8, true);
            } else {
#pragma unroll 1
                for (int kk = 0; kk < steps; ++kk) issue_pv(kk, kk % 4 * 8, true);
            }
            next_slot();
            t_v = next_group(t_v);
            const bool more = j + NB < cur.cnt + nxt.cnt;      // scores follow, and their K is there
            if (j == cur.cnt - 1) commit(SM::BAR_O);
            else if (!more) commit(SM::BAR_PV + (j == cur.cnt - 2 ? 1 : 0));
            k_there = more && SM::K_AHEAD;
            ++j;
            --ahead;
        }
        if (!ok && lane == 0) give_up();
        __syncwarp();
        if (*abort_flag) {                // let what was issued finish
            if (PAIR) ptx::tc_commit_pair_mask_elect(bar(SM::BAR_DRAIN), 1, leader);
            else ptx::tc_commit_elect(bar(SM::BAR_DRAIN), leader);
            ptx::mbar_wait(bar(SM::BAR_DRAIN), 0);
        }
        __syncwarp();
    }
    } else {
        // ------------------------------------------------------------ softmax warps
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(AT_SOFTMAX_REGS));
        // Thread (row, hf) of set e: query row `row`, columns [64 hf, 64 hf + 64) of groups 1, 3, .. (e = 1) or 2, 4, .. (e = 0).
        const int qd = warp & 3, hf = (warp >> 2) & 1, e = warp >> 3;
        const int row = qd * 32 + lane;
        // 128 bits: the row's node sees tree row i
        const uint32_t *anc = reinterpret_cast<const uint32_t *>(p.anc + (blk * p.npc + node_in_tile(p, row)) * 2);
        const bool mine = out_row(p, blk, row) >= 0;
        auto anc_word = [&](int w) -> uint32_t {
            if (w < 0) return 0xffffffffu;     // prefix rows are visible to every node
            return w < 4 && mine ? anc[w] : 0u;    // past the tree rows: nothing
        };
        const uint32_t tmem = begin();
        const uint32_t lane_base = tmem + ((uint32_t)(qd * 32) << 16);
        const uint32_t t_s0 = lane_base + TM_S + hf * 64;                 // + 128 b: this half of tile b of scores
        const uint32_t t_o = lane_base + TM_O + (e * 2 + hf) * (D / 4);        // this thread's columns of O
        auto x_at = [&](int s, int h) { return sbase + SM::OFF_X + (uint32_t)((s * 2 + h) * 128 + row) * 4u; };   // [set][half][row]
        const uint32_t ask_at = sbase + SM::OFF_ASK + (uint32_t)qd * 4u;
        constexpr uint32_t hidden = NEG ? 0x7f800000u : 0xff800000u;   // times the scale: -inf
        // Phases: bit 0: meetings, 1: what was exchanged has been read, 2: all P of a piece written, 3: BAR_PV + 1.
        uint32_t phases = 0;
        // The piece: its number, its groups, and its first group's number modulo 6 (tile of scores, and from 3 on its barriers' odd phases)
        int piece = 0, cnt = 0, t0 = 0;
        bool ok = true;
        int n_part = 0;                           // partial results written
        float m_used = -INFINITY, l = 0.f;
        auto arrive_x = [&](int i) {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(i + qd));
        };
        auto wait_x = [&](int i, uint32_t bit) {
            if (!ptx::mbar_wait(bar(i + qd), (phases >> bit) & 1)) ok = false;
            phases ^= 1u << bit;
        };
        auto meet = [&]() {                       // the four warps of these rows
            arrive_x(SM::BAR_XM);
            wait_x(SM::BAR_XM, 0);
        };
        // A warp whose exponents do not fit the reference has not written its P of group `at` yet: O += P V waits for it in all
        // groups from there on, so that all four warps come to wait for scores (or for the others' P) and meet here; next: the
        // group that this warp is to take next (a warp that asks: at).  What is there then: O with all groups before the earliest
        // one that is missing (its MMAs are waited for), and P of groups behind that one, which follow the reference like O does.
        auto move_reference = [&](float mx, int next, bool asks) {
            meet();                               // (nobody is still at what was exchanged before)
            ptx::sts_f32(x_at(e, hf), mx);
            if (lane == 0) ptx::sts_u32(sbase + SM::OFF_AT + (uint32_t)(qd * 4 + e * 2 + hf) * 4u, asks ? (uint32_t)next : 0x7fffffffu);
            meet();
            int first = 0x7fffffff;               // (not group 0, which always fits)
            float m_new = m_used;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                first = min(first, (int)ptx::lds_u32(sbase + SM::OFF_AT + (uint32_t)(qd * 4 + i) * 4u));
                m_new = fmaxf(m_new, ceilf(ptx::lds_f32(x_at(i >> 1, i & 1))));
            }
            // O += P V of the group before: told with the scores behind it, or by itself
            if (!ptx::mbar_wait(bar(SM::BAR_PC_FULL + (piece + 1) % AT_PIECES), ((piece + 1) / AT_PIECES) & 1)) ok = false;
            const int done = first - 1, nxt = ok ? reinterpret_cast<const volatile AttnPiece *>(desc)[(piece + 1) % AT_PIECES].cnt : 0;
            const uint32_t k = (uint32_t)(t0 + done + NB);
            if (done + NB < cnt + nxt) ok = ok && ptx::mbar_wait(bar(SM::BAR_S + k % NB), (k / NB) & 1);
            else if (done == cnt - 2) ok = ok && ptx::mbar_wait(bar(SM::BAR_PV + 1), (phases >> 3) & 1);
            else ok = ok && ptx::mbar_wait(bar(SM::BAR_PV), 0);      // (of the last piece only)
            ptx::tc_fence_after();
            const bool need = m_new != m_used && m_used != -INFINITY;
            if (__any_sync(0xffffffffu, need)) {
                const float alpha = need ? ex2(m_used - m_new) : 1.f;
                uint32_t x[16];
#pragma unroll 1
                for (int j = next - 4; j < next; j += 2) {    // (a power of two: exact)
                    if (j < first) continue;
                    const uint32_t t_p = t_s0 + (uint32_t)(t0 + j) % NB * 128;
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {        // (both terms)
                        ptx::tmem_ld16(t_p + c * 16, x);
                        ptx::tmem_ld_wait_for16(x);
#pragma unroll
                        for (int i = 0; i < 16; ++i) x[i] = pack2_bf16(bf16_lo(x[i]) * alpha, bf16_hi(x[i]) * alpha);
                        ptx::tmem_st16(t_p + c * 16, x);
                    }
                }
#pragma unroll 1
                for (int c = 0; c < D / 64; ++c) {
                    ptx::tmem_ld16(t_o + c * 16, x);
                    ptx::tmem_ld_wait_for16(x);
#pragma unroll
                    for (int i = 0; i < 16; ++i) x[i] = __float_as_uint(__uint_as_float(x[i]) * alpha);
                    ptx::tmem_st16(t_o + c * 16, x);
                }
                ptx::tmem_st_wait();
                l *= alpha;
            }
            m_used = m_new;
            if (lane == 0) ptx::sts_u32(ask_at, 0u);
            ptx::tc_fence_before();
            meet();
            ptx::tc_fence_after();
        };
        // Waits for the tensor core; meanwhile another warp of these rows may ask to move the reference.  What is waited for can be
        // complete all the same: the barrier, tested again behind the question, says so, and the question is met at the next
        // wait.  (The scores of the group at which a warp asks, and of all before it, are complete when it asks.)
        auto wait_tc = [&](uint32_t b, uint32_t parity, int next) {
            const long long since = clock64();
            while (!ptx::mbar_try_wait(b, parity)) {
                if (ptx::lds_u32(ask_at)) {
                    if (!ptx::mbar_try_wait(b, parity)) move_reference(-INFINITY, next, false);
                    else break;
                    continue;
                }
                if (clock64() - since > ptx::WAIT_CYCLE_LIMIT) { ok = false; return; }
            }
        };
        auto p_done = [&](int b, uint32_t count) {
            ptx::tmem_st_wait();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_lead(SM::BAR_P + b, count);
        };
        const float2 sc2 = make_float2(p.scale_log2, p.scale_log2);
        // The first group of a piece comes before the end of the piece before it: the tensor core has its PV, and the scores behind,
        // to do while O is read and written out.
        for (int pi = 0;; ++pi) {
            if (pi > 0) {                         // all P of the piece before are written: nobody asks to move its reference any more
                arrive_x(SM::BAR_XG);
                wait_tc(bar(SM::BAR_XG + qd), (phases >> 2) & 1, cnt + ((cnt ^ e) & 1));
                phases ^= 4;
            }
            ok = ok && ptx::mbar_wait(bar(SM::BAR_PC_FULL + pi % AT_PIECES), (pi / AT_PIECES) & 1);
            if (!ok || *abort_flag) break;
            const volatile AttnPiece &d = desc[pi % AT_PIECES];    // (freed at the end of the piece)
            const int cnt_new = d.cnt, a_first = d.gb * AT_BN + hf * 64 - d.L;      // tree row of this half's first column in the first group
            const int t_new = (int)((unsigned)(t0 + cnt) % (2 * NB));
            float m_new = -INFINITY, l_new = 0.f;
            if (cnt_new > 0) {
                // ---- the first group, all four threads of a row on a quarter of it each: its maximum, then its P in two terms
                const int b = t_new >= NB ? t_new - NB : t_new;
                if (!ptx::mbar_wait(bar(SM::BAR_S + b), t_new >= NB)) { ok = false; break; }
                ptx::tc_fence_after();
                const uint32_t t_q = t_s0 + (uint32_t)b * 128 + e * 32;
                const int a0 = a_first + e * 32;         // tree row of the quarter's first column
                uint32_t q[32], pk[32];
                ptx::tmem_ld32(t_q, q);
                ptx::tmem_ld_wait_for(q);
                if (a0 + 32 > 0) {                       // bit i of vis is column i (see below)
                    const uint32_t vis = __funnelshift_r(anc_word(a0 >> 5), anc_word((a0 >> 5) + 1), a0 & 31);
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (!((vis >> i) & 1u)) q[i] = hidden;
                }
                const float mx = max_quarter<NEG>(q, p.scale_log2);
                if (pi > 0) wait_x(SM::BAR_XO, 1);
                ptx::sts_f32(x_at(e, hf), mx);
                meet();
                if (!ok) break;
                m_new = ceilf(fmaxf(fmaxf(ptx::lds_f32(x_at(0, 0)), ptx::lds_f32(x_at(0, 1))), fmaxf(ptx::lds_f32(x_at(1, 0)), ptx::lds_f32(x_at(1, 1)))));
                arrive_x(SM::BAR_XO);
                const float m_eff = m_new == -INFINITY ? 0.f : m_new;
                float2 la = make_float2(0.f, 0.f), lb = make_float2(0.f, 0.f);
                exp_quarter<true>(q, sc2, make_float2(-m_eff, -m_eff), la, lb, pk, pk + 16);
                ptx::tmem_st32(t_q, pk);
                l_new = (la.x + la.y) + (lb.x + lb.y);
                p_done(b, 1);
            }
            if (pi > 0) {
                // ---- O of the piece before
                const volatile AttnPiece &o_d = desc[(pi - 1) % AT_PIECES];
                if (!ptx::mbar_wait(bar(SM::BAR_O), (pi - 1) & 1)) { ok = false; break; }
                ptx::tc_fence_after();
                // ---- the row sums of the row's four threads
                wait_x(SM::BAR_XO, 1);
                ptx::sts_f32(x_at(e, hf), l);
                arrive_x(SM::BAR_XM);
                uint32_t o[D / 4];
                if constexpr (D == 128) ptx::tmem_ld32(t_o, o);
                else ptx::tmem_ld16(t_o, o);
                wait_x(SM::BAR_XM, 0);
                if (!ok) break;
                const float l_all = (ptx::lds_f32(x_at(0, 0)) + ptx::lds_f32(x_at(0, 1))) + (ptx::lds_f32(x_at(1, 0)) + ptx::lds_f32(x_at(1, 1)));
                arrive_x(SM::BAR_XO);
                const float inv_l = l_all == 0.f ? 0.f : 1.f / l_all;     // (NaN stays NaN)
                if constexpr (D == 128) ptx::tmem_ld_wait_for(o);
                else ptx::tmem_ld_wait_for16(o);
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) arrive_lead(SM::BAR_O_FREE);
#pragma unroll
                for (int i = 0; i < D / 4; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * inv_l);
                if (o_d.flags & PIECE_PARTIAL) {
                    // to the workspace, whose layout suits a thread per row
                    const int slab = o_d.flags & PIECE_HEAD ? 1 : 0;
                    if (mine) {
#pragma unroll
                        for (int c = 0; c < D / 16; ++c)
                            *slab_o<D>(p, blockIdx.x, slab, row, (e * 2 + hf) * (D / 16) + c) = make_uint4(o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]);
                        if (hf == 0 && e == 0) *slab_ml(p, blockIdx.x, slab, row) = make_float2(m_used, l_all);
                    }
                    ++n_part;
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar(SM::BAR_OUT));
                } else if (mine) {
                    // a thread's columns are 32 or 64 bytes of its row
                    uint4 *dst = item_out<D>(p, o_d.layer, o_d.b, o_d.head) + out_row(p, blk, row) * (D / 8) + (e * 2 + hf) * (D / 32);
#pragma unroll
                    for (int c = 0; c < D / 64; ++c) {
                        uint32_t w[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) w[i] = pack2_bf16(__uint_as_float(o[16 * c + 2 * i]), __uint_as_float(o[16 * c + 2 * i + 1]));
                        if (p.out32) ptx::st_global_32(dst + 2 * c, w);
                        else {
                            dst[2 * c] = make_uint4(w[0], w[1], w[2], w[3]);
                            dst[2 * c + 1] = make_uint4(w[4], w[5], w[6], w[7]);
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) free_piece(pi - 1);
            }
            if (cnt_new <= 1 && cnt >= 2) phases ^= 8;     // (the PV of the piece's last group but one was told by itself)
            piece = pi;
            cnt = cnt_new;
            t0 = t_new;
            m_used = m_new;
            l = l_new;
            if (cnt == 0) break;
            const int n_two = d.flags >> PIECE_TWO_SHIFT;
            int t = t0 + (e == 0 ? 2 : 1);
            for (int j = e == 0 ? 2 : 1; j < cnt; j += 2, t += 2) {
                if (t >= 2 * NB) t -= 2 * NB;
                const int b = t >= NB ? t - NB : t;
                float sum;
                bool asked = false;
                const uint32_t t_s = t_s0 + (uint32_t)b * 128;
#pragma unroll 1
                for (;;) {
                    if (!asked) {
                        wait_tc(bar(SM::BAR_S + b), t >= NB, j);
                        if (!ok) break;
                        ptx::tc_fence_after();
                    }
                    uint32_t qa[32], qb[32];
                    ptx::tmem_ld32(t_s, qa);
                    ptx::tmem_ld32(t_s + 32, qb);
                    ptx::tmem_ld_wait_for(qa);
                    ptx::tmem_ld_wait_for(qb);
                    const int a0 = a_first + j * AT_BN;      // tree row of this half's first column
                    if (a0 + 64 > 0) {
                        // the half overlaps the tree rows or the end of the cache: bit i of va is column i of a quarter
                        const int w = a0 >> 5, sh = a0 & 31;     // floor division
                        const uint32_t w1 = anc_word(w + 1);
                        const uint32_t va = __funnelshift_r(anc_word(w), w1, sh), vb = __funnelshift_r(w1, anc_word(w + 2), sh);
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            if (!((va >> i) & 1u)) qa[i] = hidden;
                            if (!((vb >> i) & 1u)) qb[i] = hidden;
                        }
                    }
                    if (asked) {
                        const float mx = fmaxf(max_quarter<NEG>(qa, p.scale_log2), max_quarter<NEG>(qb, p.scale_log2));
                        move_reference(mx > m_used + 16.f ? mx : -INFINITY, j, true);
                    }
                    const float m_eff = m_used == -INFINITY ? 0.f : m_used;
                    const float2 nm2 = make_float2(-m_eff, -m_eff);
                    float2 la = make_float2(0.f, 0.f), lb = make_float2(0.f, 0.f);
                    // (rows that belong to nobody may hold anything)
                    auto fits = [&]() {
                        sum = (la.x + la.y) + (lb.x + lb.y);
                        return asked || !__any_sync(0xffffffffu, mine && sum > AT_SUM_LIMIT);
                    };
                    if (two_terms<D>(j, n_two)) {
                        uint32_t pa[16], pb[16], ra[16], rb[16];
                        exp_quarter<true>(qa, sc2, nm2, la, lb, pa, ra);
                        exp_quarter<true>(qb, sc2, nm2, la, lb, pb, rb);
                        if (fits()) {
                            ptx::tmem_st16(t_s, pa);
                            ptx::tmem_st16(t_s + 16, ra);
                            ptx::tmem_st16(t_s + 32, pb);
                            ptx::tmem_st16(t_s + 48, rb);
                            break;
                        }
                    } else {
                        uint32_t pw[32];
                        exp_quarter<false>(qa, sc2, nm2, la, lb, pw, nullptr);
                        exp_quarter<false>(qb, sc2, nm2, la, lb, pw + 16, nullptr);
                        if (fits()) {
                            ptx::tmem_st32(t_s, pw);
                            break;
                        }
                    }
                    // rare: ask the other warps of these rows to come and move the reference, start over
                    asked = true;
                    if (lane == 0) ptx::sts_u32(ask_at, 1u);
                }
                if (!ok) break;
                l += sum;
                p_done(b, 2);
            }
            if (!ok) break;
        }
        if (!ok && lane == 0) give_up();
        // ---- the items that this CTA shares with others
#pragma unroll 1
        for (int i = 0; i < n_part && ok; ++i) {
            const MergeSlice<D> slice(p, merges[i], team - merges[i].first);
            if (!ptx::mbar_wait(bar(SM::BAR_GO + i), 0)) { give_up(); break; }
            if ((*left_items >> (2 + i)) & 1) continue;
            if (merges[i].n > MERGE_MANY) {
                if (slice.n_my > 0) merge_few_rows<D>(p, merges[i], slice.r_begin, slice.n_my, warp * 32 + lane, blk);
            } else {
                slice.run(p, merges[i], warp * 32 + lane, blk);
            }
        }
    }
    __syncwarp();
    ptx::tc_fence_before();
    __syncthreads();
    // nobody leaves while the pair's MMAs may still read its shared memory or its barriers may be signalled
    if (PAIR) ptx::cluster_arrive();
    if (warp < AT_SOFTMAX_WARPS && *left_items)       // (the other warps have too few registers for it)
        for (int i = 0; i < 2; ++i)
            if ((*left_items >> i) & 1) merge_left<D>(p, merges[i], blk, warp * 32 + lane);
    __syncwarp();
    if (PAIR) ptx::cluster_wait();
    ptx::tc_fence_after();
    if (warp == W_MMA) {
        if (PAIR) ptx::tmem_dealloc_pair(*tmem_slot, 512);
        else ptx::tmem_dealloc(*tmem_slot, 512);
    }
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

// Encoding a map costs the host a microsecond or two and a step over 32 layers may need 65, so encoded maps are kept in a
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
// Layers of a launch: positions in the common address space of its groups are 32 bits wide (PieceWalk: an item counts its groups
// and ITEM_COST, or, with fewer items than teams, whole pieces; the last team's run may end a few groups behind the last item).
// A single layer is not looked at: 2^32 positions are the K and V of far more memory than a device has.
constexpr double ADDRESS_LIMIT = 4e9;
constexpr int layers_per_launch(int n_layers, double items, int groups) {
    int n = n_layers == 1 ? 1 : AT_MAX_LAYERS;
    while (n > 1 && n * items * (groups + ITEM_COST) > ADDRESS_LIMIT) n /= 2;
    return n;
}
// one group per item: every item takes 1 + ITEM_COST positions, and they stay below 2^32 whatever the number of items
static_assert(layers_per_launch(AT_MAX_LAYERS, ADDRESS_LIMIT / (AT_MAX_LAYERS * (1 + ITEM_COST)), 1) == AT_MAX_LAYERS &&
              layers_per_launch(AT_MAX_LAYERS, ADDRESS_LIMIT / (AT_MAX_LAYERS * (1 + ITEM_COST)) * 1.01, 1) == AT_MAX_LAYERS / 2, "address space");
// The two outer dimensions of a cache's tensor map: sizes, and strides in elements.
struct CacheDims {
    cuuint64_t n3, n4;
    int64_t s3, s4;
};
// Row tiles of a problem and the CTAs that work on it: at head size 128 items of more than one tile go to CTA pairs.
struct AttnPlan {
    int npc, n_tiles, n_blk, teams;      // tree nodes per tile, tiles of an item, CTAs of a team, teams
    int two_cuts;                        // see two_term_groups
    bool pair;
};
AttnPlan attn_plan(int T, int G, int D) {
    AttnPlan a;
    a.npc = 128 / G;
    a.n_tiles = (T + a.npc - 1) / a.npc;
    a.pair = D == 128 && a.n_tiles > 1;
    a.n_blk = a.pair ? (a.n_tiles + 1) / 2 * 2 : a.n_tiles;
    const int sms = sm_count() < AT_MAX_CTAS ? sm_count() : AT_MAX_CTAS;
    a.teams = (a.pair ? sms / 2 * 2 : sms) / a.n_blk;
    a.two_cuts = sms / ((a.n_tiles + 1) / 2);
    return a;
}
}  // namespace

// Workspace: two slabs (a CTA has at most two pieces that are not whole items) for every CTA; the kernel for single layers
// keeps a slab per key split of a query block and the order of the sequences.
AttnWs attn_ws_layout(const mtv_tree *t, int B, int Hq, int Hkv, int D, int Lcap) {
    AttnWs w;
    w.o_off = w.ml_off = w.left_off = w.total = 0;
    if (Hq / Hkv > 8) return w;          // the call itself refuses such a group; sizes are asked for before that
    const AttnPlan a = attn_plan(t->T, Hq / Hkv, D);
    const size_t slabs = (size_t)a.teams * a.n_blk * 2;
    w.ml_off = align_up(slabs * 128 * D * sizeof(float), 256);
    w.left_off = align_up(w.ml_off + slabs * 128 * sizeof(float2), 256);
    w.total = align_up(w.left_off + slabs * sizeof(int32_t), 256);
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
// L = 512 take 45 us instead of 320, at L = 8192 260 to 320 instead of 570).  The kernel of attention_pair.cu starts and ends
// faster but leaves pairs idle where blocks and splits do not fill them, or where a second round of blocks follows the first; this one
// divides the groups evenly.  Only the capacity is known here, not the lengths.  Estimates in us for a full cache, fitted to both
// kernels' times for 142 shapes (1 to 16 sequences, 1 to 8 heads, groups of 1 to 8, T = 16 to 128, capacities of 107 to 65536, lengths of
// 1 to 0.15 of it): the choice costs 0.8 % over the better of the two on average and 20 % at worst, where pairs alone cost 11 %,
// the even division alone 10.5 %.  us per call, pairs / even division, and what is taken:
//      1 sequence,  32 / 8 heads, capacity  8256:   18 / 23  pairs          8 sequences, 24 / 8 heads, T = 29,  3029:   35 / 28  even
//      1 sequence,   8 / 2 heads, capacity  2112:   10 / 16  pairs          4 sequences, 32 / 8 heads, T = 128, 33024: 311 / 259  even
//     16 sequences, 16 / 8 heads, T = 20,    320:   23 / 13  even          16 sequences, 32 / 8 heads, capacity 1564:   37 / 42  even
//      7 sequences, 28 / 4 heads, capacity  8176:   71 / 48  even           2 sequences, 28 / 4 heads, capacity 3064:   18 / 20  pairs
static bool pair_kernel_is_better(const AttnPlan &a, int T, int G, int B, int Hkv, int Lcap) {
    int n_blk = 1;
    const int ns = attn_pair_plan(T, G, B, Hkv, Lcap, &n_blk);
    const double items = (double)B * Hkv, groups = (Lcap + AT_BN - 1) / AT_BN;
    const double pairs = 6.19 + 0.734 * ceil(groups / ns) * std::max(1.0, items * n_blk / (sm_count() / 2)) + (ns > 1 ? 2.59 : 0.0);
    const double all = items * groups / a.teams, whole = ceil(items / a.teams) * groups;
    const double even = 7.28 + 0.607 * (whole <= all + MERGE_COST ? whole : all + 4.57 / 0.607);
    return pairs <= even;
}

// One tensor map for the caches of all layers, where they lie evenly spaced in memory and a map's five dimensions are enough: 64
// columns, rows, 64-column halves, and two for head, sequence and layer.  Of these the sequence falls away when there is one, or is
// joined with the layers (layers follow one another like sequences) or with the heads (sequences follow one another like heads).
// The launch then has 0.7 KB of parameters instead of 16.5 and three maps to look up instead of 2 n + 1: a step's call takes the host
// 17 us with 32 layers instead of 21.
static bool fold_layers(CacheFold &f, int n_layers, mtv_bf16 *const *k, mtv_bf16 *const *v, const AttnParams &p, int64_t sb, int64_t sh,
                        CacheDims &dk, CacheDims &dv) {
    if (n_layers < 2) return false;
    const int64_t gap_k = k[1] - k[0], gap_v = v[1] - v[0];
    auto fits = [](int64_t gap) { return gap > 0 && gap % 8 == 0 && gap < (int64_t)1 << 38; };      // (bytes: a multiple of 16 below 2^40)
    if (!fits(gap_k) || !fits(gap_v)) return false;
    for (int l = 2; l < n_layers; ++l)
        if (k[l] - k[0] != l * gap_k || v[l] - v[0] != l * gap_v) return false;
    const cuuint64_t H = p.Hkv, B = p.B, N = n_layers;
    if (p.B == 1) {
        f = {0, 0, 1};
        dk = {H, N, sh, gap_k};
        dv = {H, N, sh, gap_v};
    } else if (gap_k == p.B * sb && gap_v == p.B * sb) {
        f = {0, 1, p.B};
        dk = dv = {H, B * N, sh, sb};
    } else if (sb == p.Hkv * sh) {
        f = {p.Hkv, 0, 1};
        dk = {H * B, N, sh, gap_k};
        dv = {H * B, N, sh, gap_v};
    } else {
        return false;
    }
    return true;
}

template <int D, bool PAIR, int ML, bool NEG>
static int launch_attn(const mtv_tree *tree, const AttnPlan &a, AttnParams &p, const __nv_bfloat16 *q, mtv_bf16 *const *k,
                       mtv_bf16 *const *v, const CacheDims &dk, const CacheDims &dv, int64_t st, cudaStream_t stream) {
    AttnMaps<ML> maps;
    {
        const cuuint64_t row = (cuuint64_t)p.Hq * D * 2;
        const cuuint64_t qd[5] = {64, (cuuint64_t)p.Hq, (cuuint64_t)p.T, D / 64, (cuuint64_t)p.B * p.n_layers};
        const cuuint64_t qs[4] = {D * 2, row, 128, row * p.T};
        const cuuint32_t qb[5] = {64, (cuuint32_t)p.G, (cuuint32_t)p.npc, 1, 1};
        const cuuint32_t kb[5] = {64, PAIR ? AT_BN / 2 : AT_BN, D / 64, 1, 1}, vb[5] = {64, AT_BN, PAIR ? 1 : D / 64, 1, 1};
        if (!tensor_map_bf16(&maps.q, q, 5, qd, qs, qb)) return MTV_ERR_CUDA;
        auto cache_map = [&](CUtensorMap *map, const mtv_bf16 *base, const CacheDims &c, const cuuint32_t *box) {
            const cuuint64_t cd[5] = {64, (cuuint64_t)p.Lcap, D / 64, c.n3, c.n4};
            const cuuint64_t cs[4] = {(cuuint64_t)st * 2, 128, (cuuint64_t)c.s3 * 2, (cuuint64_t)c.s4 * 2};
            return tensor_map_bf16(map, base, 5, cd, cs, box);
        };
        for (int l = 0; l < (ML == 1 ? 1 : p.n_layers); ++l)
            if (!cache_map(&maps.k[l], k[l], dk, kb) || !cache_map(&maps.v[l], v[l], dv, vb)) return MTV_ERR_CUDA;
    }
    static PerDeviceOnce once;
    bool *done = once.flag();
    if (!done || !*done) {
        cudaFuncAttributes fa;
        MTV_CUDA_CHECK(cudaFuncGetAttributes(&fa, tree_attn_kernel<D, PAIR, ML, NEG>));
        if (fa.numRegs < AT_LAUNCH_REGS) {   // the register split would wait for registers that the launch does not own
            set_last_error_text("tree_attn_kernel: compiled with fewer registers than its split needs");
            return MTV_ERR_CUDA;
        }
        MTV_CUDA_CHECK(cudaFuncSetAttribute(tree_attn_kernel<D, PAIR, ML, NEG>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnSmem<D, PAIR>::TOTAL));
        if (done) *done = true;
    }
    TapScope tap(MTV_KERNEL_ATTN_PARTIAL, stream);
    MTV_CUDA_CHECK(launch_dependent_clusters(PAIR ? 2 : 1, tree_attn_kernel<D, PAIR, ML, NEG>, dim3(a.teams * a.n_blk), AT_THREADS,
                                             AttnSmem<D, PAIR>::TOTAL, stream, maps, p));
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
    if (n_layers == 1 && attn_pair_eligible(D, Hq / Hkv) && pair_kernel_is_better(attn_plan(tree->T, Hq / Hkv, D), tree->T, Hq / Hkv, B, Hkv, Lcap)) {
        TapScope tap(MTV_KERNEL_ATTN_PARTIAL, (cudaStream_t)stream);
        return launch_tree_attn_pair(tree, B, Hq, Hkv, reinterpret_cast<const __nv_bfloat16 *>(q),
                                     reinterpret_cast<const __nv_bfloat16 *>(k[0]), reinterpret_cast<const __nv_bfloat16 *>(v[0]),
                                     stride_b, stride_h, stride_t, Lcap, seq_lens,
                                     (scale == 0.f ? 1.f / sqrtf((float)D) : scale) * LOG2E, reinterpret_cast<__nv_bfloat16 *>(out),
                                     status, (char *)ws + Lw.o_off, reinterpret_cast<float *>((char *)ws + Lw.pair_ml_off),
                                     reinterpret_cast<int32_t *>((char *)ws + Lw.order_off), (cudaStream_t)stream);
    }
    const AttnPlan a = attn_plan(tree->T, Hq / Hkv, D);
    AttnParams p;
    p.seq_lens = seq_lens; p.anc = tree->d_anc; p.status = status; p.dev_error = tree->d_error;
    p.ws_o = reinterpret_cast<uint4 *>((char *)ws + Lw.o_off);
    p.ws_ml = reinterpret_cast<float2 *>((char *)ws + Lw.ml_off);
    p.left = reinterpret_cast<int32_t *>((char *)ws + Lw.left_off);
    p.counters = tree->d_counters;
    p.scale_log2 = (scale == 0.f ? 1.f / sqrtf((float)D) : scale) * LOG2E;
    p.B = B; p.T = tree->T; p.G = Hq / Hkv; p.Hq = Hq; p.Hkv = Hkv; p.Lcap = Lcap;
    p.npc = a.npc; p.R = a.npc * p.G; p.inv_g = (65536u + p.G - 1) / p.G; p.n_blk = a.n_blk; p.teams = a.teams;
    p.n_tiles = a.n_tiles; p.two_cuts = a.two_cuts;
    p.gate = alongside ? *alongside : Gate{};
    p.out32 = ((uintptr_t)out & 31) == 0;
    const size_t per_layer = (size_t)B * tree->T * Hq * D;
    cudaStream_t st = (cudaStream_t)stream;
    const int per_launch = layers_per_launch(n_layers, (double)B * Hkv, (Lcap + AT_BN - 1) / AT_BN);
    for (int l = 0; l < n_layers; l += per_launch) {
        if (l > 0) p.gate = Gate{};          // (it shares the counters and the workspace with the launch before)
        p.n_layers = n_layers - l < per_launch ? n_layers - l : per_launch;
        p.out = reinterpret_cast<__nv_bfloat16 *>(out) + l * per_layer;
        const __nv_bfloat16 *ql = reinterpret_cast<const __nv_bfloat16 *>(q) + l * per_layer;
        constexpr int ML = AT_MAX_LAYERS;
        CacheDims dk = {(cuuint64_t)Hkv, (cuuint64_t)B, stride_h, stride_b}, dv = dk;
        p.fold = {0, 1, 0};
        auto launch = p.n_layers == 1 || fold_layers(p.fold, p.n_layers, k + l, v + l, p, stride_b, stride_h, dk, dv)
                          ? (a.pair ? launch_attn<128, true, 1, false> : D == 128 ? launch_attn<128, false, 1, false>
                             : scale < 0.f ? launch_attn<64, false, 1, true> : launch_attn<64, false, 1, false>)
                          : (a.pair ? launch_attn<128, true, ML, false> : D == 128 ? launch_attn<128, false, ML, false>
                             : scale < 0.f ? launch_attn<64, false, ML, true> : launch_attn<64, false, ML, false>);
        const int rc = launch(tree, a, p, ql, k + l, v + l, dk, dv, stride_t, st);
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
