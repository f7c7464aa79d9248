// LM-head projection with the per-node argmax fused into its epilogue — the step between the
// tree attention and the acceptance (Section 3.2: acceptance needs, at every tree node, the base
// model's most likely next token).  logits[m][v] = <x[m], W[v]> for the M = B T tree nodes never go to
// memory: only argmax_v survives.
//
// A weight-streaming GEMM on the tcgen05 tensor cores.  With few nodes (M <= 128 per pass) the
// arithmetic intensity is M flop per weight byte, so HBM bounds it; the vocabulary rows are the
// MMA's M dimension, the nodes its N dimension:
//   D[128 vocabulary rows][N nodes] += W_tile[128][64 k] . X[N][64 k]^T      (both operands K-major)
// One persistent CTA per SM walks pairs of vocabulary tiles, so that a chunk of X fetched from L2
// serves two weight tiles.  A tile holds R <= 128 rows, R chosen by the host so that every CTA gets
// the same number of pairs (V = 32000 on 148 SMs: 112 rows); the MMA spans 128 rows all the same and
// the rows past R, whatever the shared memory held, are left out of the maximum.  From 129 nodes up the
// problem turns into a dense contraction, which lm_head_argmax_pair_kernel below does on CTA pairs.
// Warp roles: TMA producer (ring of stages, one stage = 64
// columns of the weight tiles and of the N node rows), MMA issuer (accumulators in tensor memory,
// double-buffered: the epilogue of one pair overlaps the MMAs of the next), four epilogue warps
// (one thread per vocabulary row: order-preserving (value, ~index) keys, maximum over the
// warp's 32 rows, shared-memory max across warps and pairs, one 64-bit atomic max per node at the end).
#include <cuda.h>

#include <climits>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tma_host.cuh"

namespace mtv {

constexpr int LM_THREADS = 192;            // warps 0-3 epilogue, warp 4 MMA issuer, warp 5 TMA producer
constexpr int LM_KC = 64;                  // columns per stage: one 128-byte swizzle span
constexpr uint32_t LM_TILE_BYTES = 128 * 128; // one weight tile of a stage: 128 rows x 64 columns
constexpr uint32_t LM_SMEM_MAX = 220 * 1024;   // dynamic part; the static part (keys, barriers) is about 1.2 KB
constexpr int LM_MAX_STAGES = 6;

constexpr uint32_t LM_IDESC_BASE = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);   // bf16 x bf16 -> fp32, M = 128

struct LmParams {
    unsigned long long *keys;   // [M] best (value, ~index) per node, zero before the launch
    int32_t *dev_error;
    int M, H, V, N;             // N = nodes per pass
    int passes;
    int R;                      // vocabulary rows per tile (<= 128, a multiple of 8), chosen so that the tiles
                                // divide evenly among the CTAs; the MMA still spans 128 rows, the rest is ignored
    int n_pairs;                // units of two weight tiles over the vocabulary
    int n_stages;
    uint32_t stage_bytes;
    Gate gate;                  // with a word: W and x are complete behind it; else behind the previous kernel
};

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void *map, uint32_t bar, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
// The weights and the nodes' states are there (a warp; TMA loads follow).
__device__ __forceinline__ void lm_inputs_there(const Gate &gate, int lane) {
    if (!gate.word) {
        previous_done();
        return;
    }
    if (lane == 0) {
        wait_gate(gate);
        ptx::fence_proxy_async_global();
    }
    __syncwarp();
}
// Best key of 32 columns over the warp's 32 rows (row of lane l: v0 + l), acc[e] = this lane's row in column e: lane l gets
// the key of column l — the order-preserving image of the value in the high word, 0xffffffff - row in the low one, so that a
// 64-bit max finds the larger value and, among equals, the lower row; 0 if no row is valid.  The images are compared as
// signed integers (-0.0 and +0.0 alike) by a warp-wide integer reduction per column: a butterfly of 64-bit keys took 1.9 k
// cycles per 32 columns and set the pace up to H = 1000 (720 nodes, H = 768, V = 84034: 106 us).
__device__ __forceinline__ unsigned long long warp_best32(const uint32_t (&acc)[32], bool valid, uint32_t v0, int lane) {
    int best = INT_MIN;
    uint32_t at = 0;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
        const int bits = __float_as_int(__uint_as_float(acc[e]) + 0.f);
        const int ord = valid ? bits ^ ((bits >> 31) & 0x7fffffff) : INT_MIN;
        const int m = __reduce_max_sync(0xffffffffu, ord);
        const uint32_t row = (uint32_t)__ffs(__ballot_sync(0xffffffffu, ord == m)) - 1u;
        if (lane == e) { best = m; at = row; }
    }
    if (best == INT_MIN) return 0ull;
    return ((unsigned long long)((uint32_t)best ^ 0x80000000u) << 32) | (0xffffffffu - (v0 + at));
}

// N nodes (64 or 128) in one pass; two weight tiles per stage, so that an X chunk serves two tiles.
template <int N>
__global__ void __launch_bounds__(LM_THREADS, 1)
lm_head_argmax_kernel(const __grid_constant__ CUtensorMap w_map, const __grid_constant__ CUtensorMap x_map,
                      const LmParams p) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned long long best[N];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag_s;
    __shared__ int issued_s;                                    // stages the producer has issued (read when giving up)
    __shared__ __align__(8) unsigned long long bar_mem[2 * LM_MAX_STAGES + 5];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t ring = raw + ((1024u - (raw & 1023u)) & 1023u);
    const uint32_t bars = ptx::smem_u32(bar_mem);
    const int NST = p.n_stages;
    auto full = [&](int s) { return bars + (uint32_t)s * 8u; };
    auto empty = [&](int s) { return bars + (uint32_t)(LM_MAX_STAGES + s) * 8u; };
    auto acc_full = [&](int u) { return bars + (uint32_t)(2 * LM_MAX_STAGES + u) * 8u; };
    auto acc_empty = [&](int u) { return bars + (uint32_t)(2 * LM_MAX_STAGES + 2 + u) * 8u; };
    const uint32_t drain_bar = bars + (uint32_t)(2 * LM_MAX_STAGES + 4) * 8u;
    volatile int *abort_flag = &abort_flag_s;
    constexpr int TILES = 2;
    constexpr uint32_t W_BYTES = TILES * LM_TILE_BYTES;
    constexpr uint32_t TMEM_COLS = 2 * TILES * N;   // 2 buffers x TILES x N columns

    let_next_start();
    for (int i = threadIdx.x; i < N; i += LM_THREADS) best[i] = 0ull;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) { ptx::mbar_init(full(s), 1); ptx::mbar_init(empty(s), 1); }
        for (int u = 0; u < 2; ++u) { ptx::mbar_init(acc_full(u), 1); ptx::mbar_init(acc_empty(u), 128); }
        ptx::mbar_init(drain_bar, 1);
        ptx::fence_mbar_init();
        abort_flag_s = 0;
        issued_s = 0;
        ptx::prefetch_tensormap(&w_map);
        ptx::prefetch_tensormap(&x_map);
    }
    if (warp == 4) {
        ptx::tmem_alloc(ptx::smem_u32(&tmem_slot), TMEM_COLS);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = tmem_slot;

    const int cta = blockIdx.x, n_cta = gridDim.x;
    const int n_pairs = p.n_pairs, R = p.R;
    const int my_pairs = cta < n_pairs ? (n_pairs - cta + n_cta - 1) / n_cta : 0;
    const int n_kc = p.H / LM_KC;
    const uint32_t x_off = W_BYTES;                      // X chunk sits after the weight chunk in a stage

    if (warp == 5) {
        // ---------------------------------------------------------------- TMA producer
        lm_inputs_there(p.gate, lane);
        int it = 0;
        for (int q = 0; q < my_pairs && !*abort_flag; ++q) {
            const int row0 = (cta + q * n_cta) * TILES * R;
            for (int kc = 0; kc < n_kc; ++kc, ++it) {
                const int s = it % NST, use = it / NST;
                if (use > 0 && !ptx::mbar_wait(empty(s), (use - 1) & 1)) { *abort_flag = 1; break; }
                if (lane == 0) {
                    const uint32_t base = ring + s * p.stage_bytes;
                    ptx::mbar_arrive_expect_tx(full(s), (uint32_t)(TILES * R + N) * 128u);
                    tma_load_2d(base, &w_map, full(s), kc * LM_KC, row0);                 // rows past V arrive as zeros
                    tma_load_2d(base + LM_TILE_BYTES, &w_map, full(s), kc * LM_KC, row0 + R);
                    tma_load_2d(base + x_off, &x_map, full(s), kc * LM_KC, 0);             // rows past M arrive as zeros
                }
                __syncwarp();
            }
        }
        if (lane == 0) issued_s = it;
    } else if (warp == 4) {
        // ---------------------------------------------------------------- MMA issuer
        constexpr uint32_t IDESC = LM_IDESC_BASE | ((uint32_t)(N >> 3) << 17);
        const bool leader = ptx::elect_one();
        int it = 0;
        bool ok = true;
        for (int q = 0; ok && q < my_pairs && !*abort_flag; ++q) {
            const int u = q & 1;
            if (q >= 2) ok = ptx::mbar_wait(acc_empty(u), ((q >> 1) - 1) & 1);   // the epilogue has read this buffer
            if (!ok) break;
            ptx::tc_fence_after();
            for (int kc = 0; kc < n_kc; ++kc, ++it) {
                const int s = it % NST;
                ok = ptx::mbar_wait(full(s), (it / NST) & 1);
                if (!ok) break;
                ptx::tc_fence_after();
                // (the whole warp, one elected lane issues: operands stay in uniform registers)
                const uint32_t w = ptx::desc_lo(ring + s * p.stage_bytes, 16);
#pragma unroll
                for (int t = 0; t < TILES; ++t)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        ptx::mma_ss_elect(tmem + (u * TILES + t) * N, w + ((t * LM_TILE_BYTES) >> 4) + kk * 2, w + (x_off >> 4) + kk * 2,
                                          ptx::DESC_HI, IDESC, kc > 0 || kk > 0, leader);
                ptx::tc_commit_elect(empty(s), leader);                         // the stage is free once these MMAs are done
                if (kc == n_kc - 1) ptx::tc_commit_elect(acc_full(u), leader);  // and so is the pair's accumulator
            }
        }
        if (!ok) *abort_flag = 1;
    } else {
        // ---------------------------------------------------------------- epilogue: thread = vocabulary row
        bool ok = true;
        for (int q = 0; q < my_pairs; ++q) {
            const int u = q & 1;
            if (*abort_flag) ok = false;
            if (ok) ok = ptx::mbar_wait(acc_full(u), (q >> 1) & 1);
            __syncwarp();
            ptx::tc_fence_after();
            const int row0 = (cta + q * n_cta) * TILES * R;
#pragma unroll 1
            for (int t = 0; t < TILES; ++t) {
                const int r = warp * 32 + lane, v0 = row0 + t * R + warp * 32;
                const bool valid = r < R && v0 + lane < p.V;           // this thread's vocabulary row (none past R)
                if (warp * 32 >= R) continue;                          // none for the whole warp
#pragma unroll 1
                for (int c = 0; c < N / 32; ++c) {
                    uint32_t acc[32];
                    ptx::tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (u * TILES + t) * N + c * 32, acc);
                    ptx::tmem_ld_wait_for(acc);
                    atomicMax(&best[c * 32 + lane], warp_best32(acc, valid, (uint32_t)v0, lane));   // node c * 32 + lane
                }
            }
            ptx::tc_fence_before();
            ptx::mbar_arrive(acc_empty(u));
        }
        if (!ok) *abort_flag = 1;
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) atomicExch(p.dev_error, MTV_ERR_TIMEOUT);
        // copies in flight and issued tensor-core work get one more bounded wait before the shared
        // and tensor memory are given back
        if (warp == 5 && lane == 0)
            for (int s = 0; s < NST; ++s) {
                const int uses = (issued_s - s + NST - 1) / NST;   // how often stage s was filled
                if (issued_s > s) ptx::mbar_wait(full(s), (uses - 1) & 1);
            }
        if (warp == 4) {
            if (lane == 0) ptx::tc_commit(drain_bar);
            __syncwarp();
            ptx::mbar_wait(drain_bar, 0);
        }
        __syncthreads();
    }
    previous_done();            // (the keys are zero)
    for (int n = threadIdx.x; n < N; n += LM_THREADS) {
        if (n < p.M && best[n] != 0ull) atomicMax(p.keys + n, best[n]);
    }
    if (warp == 4) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, TMEM_COLS);
    }
}

// ---------------------------------------------------------------------------------------- more than 128 nodes
// Bound by the tensor cores (512 MMA cycles per 64 columns of a 256 x 256 tile against 32 KB of operands per SM).  A cluster of
// two CTAs forms a tcgen05 CTA pair: D[256 vocabulary rows][N <= 256 nodes], each CTA with 128 of the rows (its operand A and its
// accumulator) and half of the nodes (operand B), so an operand byte is fetched by one SM of the pair only.  One CTA with
// 128 x 256 tiles fetched 48 KB per 512 MMA cycles, more than L2 delivers, and its issuing lane paid for moving every operand
// into uniform registers: 1029 us at 1024 nodes, V = 131072, H = 4096 (1.07 PFLOP/s).
// The (vocabulary tile, node pass) items go round the pairs, passes of a tile next to each other (its rows are then read once from
// memory); every CTA keeps the best key of all nodes in shared memory and hands them over at its end.  Per CTA: warps 0-3
// epilogue, warp 4 (even CTA) MMA issuer, warp 5 TMA producer of the CTA's own halves, warp 6 (odd CTA) relay: tells
// the issuer that the odd CTA's half of a stage has landed.
constexpr int LP_THREADS = 224;
constexpr int LP_STAGES = 6;
constexpr uint32_t LP_STAGE_BYTES = 2 * LM_TILE_BYTES;
constexpr int LP_MAX_NODES = 2048;                       // per launch: keys in shared memory
constexpr uint32_t LP_SMEM_BYTES = 1024 + LP_STAGES * LP_STAGE_BYTES + LP_MAX_NODES * 8;
static_assert(LP_SMEM_BYTES <= LM_SMEM_MAX, "shared memory");

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(LP_THREADS, 1)
lm_head_argmax_pair_kernel(const __grid_constant__ CUtensorMap w_map, const __grid_constant__ CUtensorMap x_map, const LmParams p) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag_s, issued_s;
    __shared__ __align__(8) unsigned long long bar_mem[3 * LP_STAGES + 5];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t rank = ptx::cluster_ctarank();
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw & 1023u)) & 1023u, ring = raw + pad;     // the same offset in both CTAs
    unsigned long long *best = reinterpret_cast<unsigned long long *>(smem_raw + pad + LP_STAGES * LP_STAGE_BYTES);
    const uint32_t bars = ptx::smem_u32(bar_mem);
    auto full = [&](int s) { return bars + (uint32_t)s * 8u; };
    auto empty = [&](int s) { return bars + (uint32_t)(LP_STAGES + s) * 8u; };
    auto ready = [&](int s) { return bars + (uint32_t)(2 * LP_STAGES + s) * 8u; };         // even CTA: the odd CTA's half is there
    auto acc_full = [&](int u) { return bars + (uint32_t)(3 * LP_STAGES + u) * 8u; };
    auto acc_empty = [&](int u) { return bars + (uint32_t)(3 * LP_STAGES + 2 + u) * 8u; }; // even CTA: both epilogues have read it
    const uint32_t drain_bar = bars + (uint32_t)(3 * LP_STAGES + 4) * 8u;
    volatile int *abort_flag = &abort_flag_s;
    auto give_up = [&]() {
        *abort_flag = 1;
        ptx::st_cluster_u32(ptx::mapa(ptx::smem_u32(&abort_flag_s), rank ^ 1), 1u);
    };

    let_next_start();
    for (int i = threadIdx.x; i < p.passes * p.N; i += LP_THREADS) best[i] = 0ull;
    if (threadIdx.x == 0) {
        for (int s = 0; s < LP_STAGES; ++s) { ptx::mbar_init(full(s), 1); ptx::mbar_init(empty(s), 1); ptx::mbar_init(ready(s), 1); }
        for (int u = 0; u < 2; ++u) { ptx::mbar_init(acc_full(u), 1); ptx::mbar_init(acc_empty(u), 8); }
        ptx::mbar_init(drain_bar, 1);
        ptx::fence_mbar_init();
        abort_flag_s = 0;
        issued_s = 0;
        ptx::prefetch_tensormap(&w_map);
        ptx::prefetch_tensormap(&x_map);
    }
    if (warp == 4) {
        ptx::tmem_alloc_pair(ptx::smem_u32(&tmem_slot), 512);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_arrive();
    ptx::cluster_wait();                                 // the peer's barriers and tensor memory exist
    ptx::tc_fence_after();
    const uint32_t tmem = tmem_slot;

    const int n_pairs = (int)gridDim.x >> 1, pair = (int)blockIdx.x >> 1;
    const int n_items = p.n_pairs * p.passes, half = p.N / 2;
    const int my_items = pair < n_items ? (n_items - pair + n_pairs - 1) / n_pairs : 0;
    const int n_kc = p.H / LM_KC, total = my_items * n_kc;

    if (warp == 5) {
        // ---------------------------------------------------------------- TMA producer
        lm_inputs_there(p.gate, lane);
        int it = 0;
        for (int q = 0; q < my_items && !*abort_flag; ++q) {
            const int item = pair + q * n_pairs;
            const int row0 = item / p.passes * 2 * p.R + (int)rank * p.R, node0 = item % p.passes * p.N + (int)rank * half;
            for (int kc = 0; kc < n_kc; ++kc, ++it) {
                const int s = it % LP_STAGES;
                if (it >= LP_STAGES && !ptx::mbar_wait(empty(s), (it / LP_STAGES - 1) & 1)) { give_up(); break; }
                if (lane == 0) {
                    const uint32_t base = ring + s * LP_STAGE_BYTES;
                    ptx::mbar_arrive_expect_tx(full(s), (uint32_t)(p.R + half) * 128u);
                    tma_load_2d(base, &w_map, full(s), kc * LM_KC, row0);                       // rows past V and
                    tma_load_2d(base + LM_TILE_BYTES, &x_map, full(s), kc * LM_KC, node0);      // M arrive as zeros
                }
                __syncwarp();
            }
        }
        if (lane == 0) issued_s = it;
    } else if (warp == 6) {
        // ---------------------------------------------------------------- relay (odd CTA)
        if (rank == 1)
            for (int it = 0; it < total && !*abort_flag; ++it) {
                const int s = it % LP_STAGES;
                if (!ptx::mbar_wait(full(s), (it / LP_STAGES) & 1)) { give_up(); break; }
                if (lane == 0) ptx::mbar_arrive_remote(ptx::mapa(ready(s), 0));
                __syncwarp();
            }
    } else if (warp == 4) {
        // ---------------------------------------------------------------- MMA issuer (even CTA)
        if (rank == 0) {
            const bool leader = ptx::elect_one();
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 4) << 24) | ((uint32_t)(p.N >> 3) << 17);
            int it = 0;
            bool ok = true;
            for (int q = 0; ok && q < my_items && !*abort_flag; ++q) {
                const int u = q & 1;
                if (q >= 2) ok = ptx::mbar_wait(acc_empty(u), ((q >> 1) - 1) & 1);
                if (!ok) break;
                ptx::tc_fence_after();
                for (int kc = 0; kc < n_kc; ++kc, ++it) {
                    const int s = it % LP_STAGES;
                    const uint32_t ph = (uint32_t)(it / LP_STAGES) & 1;
                    ok = ptx::mbar_wait(full(s), ph) && ptx::mbar_wait(ready(s), ph);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    const uint32_t w = ptx::desc_lo(ring + s * LP_STAGE_BYTES, 16);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        ptx::mma_pair_ss_elect(tmem + u * 256, w + kk * 2, w + (LM_TILE_BYTES >> 4) + kk * 2, ptx::DESC_HI, idesc,
                                               kc > 0 || kk > 0, leader);
                    ptx::tc_commit_pair_mask_elect(empty(s), 3, leader);                        // the stage is free in both CTAs
                    if (kc == n_kc - 1) ptx::tc_commit_pair_mask_elect(acc_full(u), 3, leader);
                }
            }
            if (!ok) give_up();
            __syncwarp();
            if (*abort_flag) {                           // issued tensor-core work gets one more bounded wait
                ptx::tc_commit_pair_mask_elect(drain_bar, 1, leader);
                ptx::mbar_wait(drain_bar, 0);
            }
        }
    } else {
        // ---------------------------------------------------------------- epilogue: thread = vocabulary row
        bool ok = true;
        for (int q = 0; q < my_items && ok; ++q) {
            const int u = q & 1, item = pair + q * n_pairs;
            ok = !*abort_flag && ptx::mbar_wait(acc_full(u), (q >> 1) & 1);
            ok = __all_sync(0xffffffffu, ok);            // (the tensor-memory loads below need the whole warp)
            if (!ok) break;
            ptx::tc_fence_after();
            const int r = warp * 32 + lane, v0 = item / p.passes * 2 * p.R + (int)rank * p.R + warp * 32;
            const bool valid = r < p.R && v0 + lane < p.V;
            unsigned long long *b = best + item % p.passes * p.N;
#pragma unroll 1
            for (int c = 0; c < (warp * 32 < p.R ? p.N / 32 : 0); ++c) {
                uint32_t acc[32];
                ptx::tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + u * 256 + c * 32, acc);
                ptx::tmem_ld_wait_for(acc);
                atomicMax(&b[c * 32 + lane], warp_best32(acc, valid, (uint32_t)v0, lane));   // node c * 32 + lane
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_remote(ptx::mapa(acc_empty(u), 0));
        }
        if (!ok) give_up();
    }
    __syncwarp();
    ptx::tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) atomicExch(p.dev_error, MTV_ERR_TIMEOUT);
        // copies in flight get one more bounded wait before the shared memory is given back
        if (warp == 5 && lane == 0)
            for (int s = 0; s < LP_STAGES; ++s) {
                const int uses = (issued_s - s + LP_STAGES - 1) / LP_STAGES;
                if (issued_s > s) ptx::mbar_wait(full(s), (uses - 1) & 1);
            }
    }
    previous_done();            // (the keys are zero)
    for (int n = threadIdx.x; n < p.passes * p.N; n += LP_THREADS)
        if (n < p.M && best[n] != 0ull) atomicMax(p.keys + n, best[n]);
    // nobody leaves while the pair's MMAs may still read its shared memory or its barriers may be signalled
    ptx::cluster_arrive();
    ptx::cluster_wait();
    ptx::tc_fence_after();
    if (warp == 4) ptx::tmem_dealloc_pair(tmem, 512);
}

static int launch_lm_head_pair(const mtv_tree_t *tree, int M, int H, int V, const mtv_bf16 *x, const mtv_bf16 *W,
                               unsigned long long *keys, const Gate &gate, cudaStream_t st) {
    for (int m0 = 0; m0 < M; m0 += LP_MAX_NODES) {
        const int m = M - m0 < LP_MAX_NODES ? M - m0 : LP_MAX_NODES;
        CUtensorMap w_map, x_map;
        LmParams p;
        p.keys = keys + m0; p.dev_error = tree->d_error; p.M = m; p.H = H; p.V = V; p.gate = gate;
        p.passes = (m + 255) / 256;
        p.N = ((m + p.passes - 1) / p.passes + 31) / 32 * 32;       // passes of equal width: no columns of an MMA for nothing
        const int pairs = sm_count() / 2;
        // as many rows per tile as make all pairs walk the same number of items
        const long rounds = ((long)((V + 255) / 256) * p.passes + pairs - 1) / pairs;
        const long tiles = rounds * pairs / p.passes;                // vocabulary tiles that fit those rounds
        p.R = (int)(((V + 2 * tiles - 1) / (2 * tiles) + 7) / 8 * 8);
        if (p.R < 32) p.R = 32;                                     // one warp's worth
        if (p.R > 128) p.R = 128;
        p.n_pairs = (V + 2 * p.R - 1) / (2 * p.R);
        p.n_stages = LP_STAGES; p.stage_bytes = LP_STAGE_BYTES;
        if (!tma_map_2d_bf16(&w_map, W, V, H, p.R) || !tma_map_2d_bf16(&x_map, x + (size_t)m0 * H, m, H, p.N / 2)) return MTV_ERR_CUDA;
        const long items = (long)p.n_pairs * p.passes;
        const int grid = 2 * (int)(items < pairs ? items : pairs);
        MTV_CUDA_CHECK(launch_dependent(lm_head_argmax_pair_kernel, dim3(grid), LP_THREADS, LP_SMEM_BYTES, st, w_map, x_map, p));
    }
    return MTV_OK;
}

__global__ void __launch_bounds__(256) lm_head_clear_kernel(int M, unsigned long long *keys) {
    let_next_start();           // (the projection starts beside this: only its last step needs the keys)
    previous_done();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < M) keys[m] = 0ull;
}
// keys -> (argmax, value)
__global__ void lm_head_finish_kernel(int M, const unsigned long long *keys, int32_t *__restrict__ am,
                                      float *__restrict__ am_val) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    let_next_start();
    previous_done();
    if (m >= M) return;
    const unsigned long long k = keys[m];
    am[m] = (int32_t)(0xffffffffu - (uint32_t)(k & 0xffffffffu));
    if (am_val) {
        const uint32_t ord = (uint32_t)(k >> 32);
        am_val[m] = __uint_as_float((ord & 0x80000000u) ? (ord & 0x7fffffffu) : ~ord);
    }
}

// The keys of all nodes.  The launches are programmatic dependents of one another: with a memset and ordinary launches the
// projection started 5 us behind whatever was in front of it.
int lm_head_keys(const mtv_tree_t *tree, int B, int H, int V, const mtv_bf16 *x, const mtv_bf16 *W, int32_t *am, float *am_val,
                 unsigned long long *keys, const Gate &gate, cudaStream_t st) {
    if (!tree || !tree->on_device || !x || !W || !keys || B < 1 || V < 1 || (am_val && !am)) return MTV_ERR_INVALID_ARG;
    if (H < 64 || H % 64 != 0) return MTV_ERR_UNSUPPORTED_SHAPE;
    if (((uintptr_t)x | (uintptr_t)W) & 15) return MTV_ERR_INVALID_ARG;
    const int M = B * tree->T;
    static PerDeviceOnce attr_once;
    bool *attr_done = attr_once.flag();
    if (!attr_done || !*attr_done) {
        MTV_CUDA_CHECK(cudaFuncSetAttribute(lm_head_argmax_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, LM_SMEM_MAX));
        MTV_CUDA_CHECK(cudaFuncSetAttribute(lm_head_argmax_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, LM_SMEM_MAX));
        MTV_CUDA_CHECK(cudaFuncSetAttribute(lm_head_argmax_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, LP_SMEM_BYTES));
        if (attr_done) *attr_done = true;
    }
    MTV_CUDA_CHECK(launch_dependent(lm_head_clear_kernel, dim3((M + 255) / 256), 256, 0, st, M, keys));
    if (M > 128) {
        const int rc = launch_lm_head_pair(tree, M, H, V, x, W, keys, gate, st);
        if (rc != MTV_OK) return rc;
    } else {
        const int N = M <= 64 ? 64 : 128;
        constexpr int tiles = 2;                             // weight tiles per stage (see the kernel)
        CUtensorMap w_map, x_map;
        LmParams p;
        p.keys = keys; p.dev_error = tree->d_error; p.M = M; p.H = H; p.V = V; p.N = N; p.passes = 1; p.gate = gate;
        p.stage_bytes = tiles * LM_TILE_BYTES + N * 128;
        p.n_stages = (int)((LM_SMEM_MAX - 1024) / p.stage_bytes);
        if (p.n_stages > LM_MAX_STAGES) p.n_stages = LM_MAX_STAGES;
        const size_t smem = 1024 + (size_t)p.n_stages * p.stage_bytes;
        int ctas = sm_count();                               // one CTA per SM
        const int min_pairs = (V + tiles * 128 - 1) / (tiles * 128);   // units of `tiles` weight tiles
        if (ctas > (V + 63) / 64) ctas = (V + 63) / 64;      // no tile below 32 rows
        if (ctas < 1) ctas = 1;
        // every CTA walks the same number of tile pairs; the tile height shrinks until they just cover V
        const int rounds = (min_pairs + ctas - 1) / ctas;
        p.n_pairs = ctas * rounds;
        p.R = ((V + tiles * p.n_pairs - 1) / (tiles * p.n_pairs) + 7) / 8 * 8;
        if (!tma_map_2d_bf16(&w_map, W, V, H, p.R) || !tma_map_2d_bf16(&x_map, x, M, H, N)) return MTV_ERR_CUDA;
        if (N == 64) MTV_CUDA_CHECK(launch_dependent(lm_head_argmax_kernel<64>, dim3(ctas), LM_THREADS, smem, st, w_map, x_map, p));
        else MTV_CUDA_CHECK(launch_dependent(lm_head_argmax_kernel<128>, dim3(ctas), LM_THREADS, smem, st, w_map, x_map, p));
    }
    if (am) MTV_CUDA_CHECK(launch_dependent(lm_head_finish_kernel, dim3((M + 127) / 128), 128, 0, st, M, keys, am, am_val));
    return MTV_OK;
}

}  // namespace mtv

extern "C" int lm_head_argmax(const mtv_tree_t *tree, int B, int H, int V, const mtv_bf16 *x, const mtv_bf16 *W,
                              int32_t *am, float *am_val, unsigned long long *keys, void *stream) {
    MTV_RANGE("lm_head_argmax");
    return mtv::lm_head_keys(tree, B, H, V, x, W, am, am_val, keys, mtv::Gate{}, (cudaStream_t)stream);
}
