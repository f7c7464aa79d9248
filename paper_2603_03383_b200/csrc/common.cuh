// Shared declarations of the CUDA library: the tree object, error plumbing and
// small device helpers.  Nothing here is used by the CPU checker.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/mtv.h"

struct mtv_tree {
    int T = 0, K = 0, P = 0, C = 0, anc_words = 0;
    int k_d[MTV_MAX_K] = {0};
    int cand_offset[MTV_MAX_K] = {0};
    std::vector<int32_t> node_ranks, parent, depth, rank, tree_indices, retrieve;
    std::vector<uint64_t> anc;
    std::vector<uint8_t> mask;
    // device copies (one allocation), valid when on_device
    bool on_device = false;
    int device = -1;
    void *d_blob = nullptr;
    const int32_t *d_tree_indices = nullptr;  // [T]
    const int32_t *d_retrieve = nullptr;      // [P][K+1]
    const uint64_t *d_anc = nullptr;          // [T][2]  (always two words per row on the device)
    const int32_t *d_kd = nullptr;            // [K]
    const int32_t *d_cand_offset = nullptr;   // [K]
    int32_t *d_error = nullptr;               // sticky device-side error word (0 = none)
    const int32_t *d_depth = nullptr;         // [T]
    int32_t *d_counters = nullptr;            // [MERGE_COUNTERS][MERGE_STRIDE] merge counters of the attention kernels, zero between calls
};

namespace mtv {

void set_last_error(const char *what, cudaError_t e);
void set_last_error_text(const char *text);

#define MTV_CUDA_CHECK(expr)                                  \
    do {                                                      \
        cudaError_t e__ = (expr);                             \
        if (e__ != cudaSuccess) {                             \
            ::mtv::set_last_error(#expr, e__);                \
            return MTV_ERR_CUDA;                              \
        }                                                     \
    } while (0)

// Merge counters of the attention kernels, in the tree object: a 128-byte line each, so that those who look at one and those who add
// to another do not queue at the same slice of L2.
constexpr int MERGE_COUNTERS = 256, MERGE_STRIDE = 32;
constexpr size_t MERGE_COUNTER_BYTES = (size_t)MERGE_COUNTERS * MERGE_STRIDE * sizeof(int32_t);

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Workspace carving shared by the entry points (all offsets 256-byte aligned).
struct HeadsWs {
    size_t hprime_off, part_val_off, part_idx_off, counters_off, tickets_off, gate_off, xsplit_off, total;
    int ctas_per_head, n_counters;
    bool use_tc;   // several batch rows: vocabulary projection on the tcgen05 tensor cores
};
HeadsWs heads_ws_layout(int K, int B, int H, int V);
// "Everything enqueued in front of the heads is complete": the word takes the call's number once that is so (see
// launch_dependent), and is cleared at the end of what may wait for it.  word null: nothing to wait for.
struct Gate {
    int32_t *word = nullptr;
    int32_t number = 0;
};
// Heads [k0, k0 + n) of a call.
// gate_stays: later kernels of the step wait at the gate, too, and the last of them clears it (null: the heads do).
struct HeadsRange {
    int k0, n;
    Gate *gate_stays = nullptr;
};
// MTV_OK, or what such a call is refused with
int heads_check(const mtv_tree *tree, int n_heads, int B, int H, int V, const mtv_bf16 *hidden, const mtv_bf16 *W1, const mtv_bf16 *W2,
                const int32_t *root_tok, const int32_t *cand, const int32_t *tree_tok, const void *ws, size_t ws_bytes);
int heads_topk_range(const mtv_tree *tree, const HeadsRange &r, int B, int H, int V, const mtv_bf16 *hidden, const mtv_bf16 *W1,
                     const mtv_bf16 *b1, const mtv_bf16 *W2, const int32_t *root_tok, int32_t *cand, float *cand_logit,
                     int32_t *tree_tok, void *ws, size_t ws_bytes, void *stream);
bool heads_tc_eligible(int B, int H);
size_t heads_tc_xsplit_bytes(int K, int H);
int launch_heads_tc(const mtv_tree *t, const HeadsRange &range, int B, int H, int V, const __nv_bfloat16 *hidden, const __nv_bfloat16 *W1,
                    const __nv_bfloat16 *b1, const __nv_bfloat16 *W2, const int32_t *root_tok, int32_t *cand,
                    float *cand_logit, int32_t *tree_tok, const HeadsWs &L, char *ws, const Gate &gate, cudaStream_t st);

struct AttnWs {
    size_t o_off, ml_off, left_off, pair_ml_off = 0, order_off = 0, total;
};
AttnWs attn_ws_layout(const mtv_tree *t, int B, int Hq, int Hkv, int D, int Lcap);
// alongside: nothing that the previous kernels in the stream back to the heads write is needed, nor their workspace touched,
// and everything before the heads is complete at this gate: the attention starts beside the previous kernel's end.
int tree_attention_layers(const mtv_tree *tree, int B, int Hq, int Hkv, int D, int n_layers, const mtv_bf16 *q,
                          mtv_bf16 *const *k, mtv_bf16 *const *v, int64_t stride_b, int64_t stride_h, int64_t stride_t,
                          int Lcap, const int32_t *seq_lens, float scale, mtv_bf16 *out, int32_t *status, void *ws,
                          size_t ws_bytes, void *stream, const Gate *alongside = nullptr);

struct AcceptWs {
    size_t part_off, total;
    int nsplit;
};
AcceptWs accept_ws_layout(const mtv_tree *t, int B, int V);
// tree_accept's scan alone: per-chunk keys into part (accept_ws_layout(...).nsplit per node); alongside: the logits are complete
// at this gate (as above).
int argmax_keys_partial(const mtv_tree *tree, int B, int V, const mtv_bf16 *logits, unsigned long long *part, const Gate &alongside,
                        cudaStream_t stream);

// lm_head_argmax; alongside: the weights and the final hidden states are complete at this gate (as above).
int lm_head_keys(const mtv_tree *tree, int B, int H, int V, const mtv_bf16 *x, const mtv_bf16 *W, int32_t *am, float *am_val,
                 unsigned long long *keys, const Gate &alongside, cudaStream_t stream);

int sm_count();   // of the current device

// Set-up that has to happen once per device (kernel attributes, symbol addresses): one flag per device ordinal.
// Two host threads that meet on first use both do the set-up; it is idempotent.
constexpr int MTV_MAX_DEVICES = 64;
struct PerDeviceOnce {
    bool done[MTV_MAX_DEVICES] = {};
    // the current device's flag, or null if the device cannot be told (the caller then does the set-up every time)
    bool *flag() {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MTV_MAX_DEVICES) return nullptr;
        return &done[dev];
    }
};

// Programmatic dependent launch: the kernel may be set up while the previous kernel of the stream runs, from the moment all
// of that kernel's blocks have executed let_next_start() or ended.  What is guaranteed is that previous_done() returns when
// the previous kernel is complete and its writes are visible.  Rules of the kernels launched so:
//   - whatever the previous kernel (or one before it) writes is touched only behind previous_done().  One exception: the tree
//     attention looks at the lengths before that, by relaxed loads, to divide its work by them; it bounds what it saw, writes
//     nothing by it, and compares it behind previous_done() (or the gate) with a second look, dividing anew where they differ;
//   - every block executes previous_done() before it ends, early or late: a kernel that is complete then implies that
//     all before it are;
//   - what was written before the heads (weights, queries, caches, lengths, logits) may be read by the heads' second kernel
//     and the kernels behind it without previous_done(), but behind a gate: the heads' first kernel executes previous_done(),
//     then stores the call's number to the gate's word with release; a reader acquires it.  (That a kernel which waited has
//     let the reader start orders nothing by itself.)  Bulk and TMA loads need the proxy fence behind the acquire.
template <typename... P, typename... A>
static inline cudaError_t launch_dependent_clusters(int cluster, void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream,
                                                    A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim = {(unsigned)cluster, 1, 1};
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <typename... P, typename... A>
static inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, A... args) {
    return launch_dependent_clusters(1, kernel, grid, threads, smem, stream, args...);
}
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void previous_done() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void open_gate(const Gate &g) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(g.word), "r"(g.number) : "memory");
}
// One thread; others read behind a barrier with it.  The word was stored before this kernel could start: a poll or two.
// (Should it not come within a millisecond, waiting for the previous kernel does as well.)
__device__ __forceinline__ void wait_gate(const Gate &g) {
    const long long t0 = clock64();
    int v;
    for (;;) {
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(g.word) : "memory");
        if (v == g.number) break;
        if (clock64() - t0 > 2000000ll) { previous_done(); break; }
    }
}

// The end of a step in one launch: acceptance from `ns` argmax keys per node (part [B][T][ns]), compaction, seq_lens.
// tickets [B]: zero before the call.  gate: the step's, cleared here.
int accept_compact(const mtv_tree *tree, const mtv_step_args *a, int ns, const unsigned long long *part, int32_t *tickets,
                   const Gate &gate, cudaStream_t stream);

// Index checks of the -DMTV_DEBUG_BOUNDS build: MTV_INDEX_OK(i, n, err) is true when 0 <= i < n; otherwise it
// records MTV_ERR_BOUNDS in the device error word and is false, and the caller skips the access.  In normal builds
// it is the constant true and the checks vanish.
#ifdef MTV_DEBUG_BOUNDS
__device__ __forceinline__ bool index_ok(long long i, long long n, int32_t *err) {
    if (i >= 0 && i < n) return true;
    if (err) atomicExch(err, MTV_ERR_BOUNDS);
    return false;
}
#define MTV_INDEX_OK(i, n, err) ::mtv::index_ok((long long)(i), (long long)(n), (err))
#else
#define MTV_INDEX_OK(i, n, err) true
#endif

// NVTX range around a C-ABI call (visible in a timeline profiler; one indirect call when no tool is attached).
// -DMTV_NO_NVTX leaves them out.
#ifndef MTV_NO_NVTX
}  // namespace mtv
#include <nvtx3/nvToolsExt.h>
namespace mtv {
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};
#define MTV_RANGE(name) ::mtv::NvtxRange mtv_nvtx_range__(name)
#else
#define MTV_RANGE(name) do { } while (0)
#endif

// Optional per-kernel event taps (see mtv_set_kernel_taps).
struct Tap {
    cudaEvent_t *start = nullptr, *stop = nullptr;
    int cap = 0, n = 0;
};
extern Tap g_taps[MTV_KERNEL_COUNT];
struct TapScope {
    Tap &t;
    cudaStream_t st;
    bool on;
    TapScope(int id, cudaStream_t s) : t(g_taps[id]), st(s), on(t.start && t.n < t.cap) {
        if (on) cudaEventRecord(t.start[t.n], st);
    }
    ~TapScope() {
        if (on) cudaEventRecord(t.stop[t.n++], st);
    }
};

}  // namespace mtv
