// Whole verification step on one stream, and its host-buffer variant.
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "sm100_ptx.cuh"

extern "C" size_t mtv_workspace_bytes(const mtv_tree_t *tree, int B, int H, int V, int Hq, int Hkv, int D, int Lcap) {
    using namespace mtv;
    if (!tree || B < 1) return 0;
    // side by side: the parts of a step overlap in time
    size_t need = 256;
    if (H > 0 && V > 0) {
        size_t heads = 0;
        for (int k = 1; k <= tree->K; ++k) heads = std::max(heads, heads_ws_layout(k, B, H, V).total);   // (a part of them at a time)
        need += heads + accept_ws_layout(tree, B, V).total;
    }
    if (Hq > 0 && Hkv > 0 && D > 0 && Lcap > 0 && Hq % Hkv == 0) need += attn_ws_layout(tree, B, Hq, Hkv, D, Lcap).total;
    return need;
}

namespace {
// The workspace of a step: heads | acceptance | attention, each with a region of its own if the buffer is large enough
// (mtv_workspace_bytes); otherwise all start at the beginning, as successive calls on one stream may, and wait for each other.
struct StepWs {
    char *accept, *attn;
    size_t accept_bytes, attn_bytes;
    bool apart;
};
StepWs step_ws(const mtv_tree_t *tree, const mtv_step_args *a) {
    StepWs w;
    char *ws = static_cast<char *>(a->ws);
    w.accept = w.attn = ws;
    w.accept_bytes = w.attn_bytes = a->ws_bytes;
    w.apart = false;
    if (!ws || a->B < 1 || a->H < 1 || a->V < 1 || a->Hq < 1 || a->Hkv < 1 || a->Hq % a->Hkv != 0 || a->D < 1 || a->Lcap < 1) return w;
    const size_t heads = mtv::heads_ws_layout(tree->K, a->B, a->H, a->V).total, accept = mtv::accept_ws_layout(tree, a->B, a->V).total;
    if (a->ws_bytes < heads + accept + mtv::attn_ws_layout(tree, a->B, a->Hq, a->Hkv, a->D, a->Lcap).total) return w;
    w.accept = ws + heads;
    w.attn = w.accept + accept;
    w.accept_bytes = accept;
    w.attn_bytes = a->ws_bytes - heads - accept;
    w.apart = true;
    return w;
}
}  // namespace

// Acceptance of a step: from stored logits, or from the fused LM head when the caller gave its operands
// (the per-node keys then sit at the start of the workspace, which no other kernel uses at that point).
static int step_accept(const mtv_tree_t *tree, const mtv_step_args *a, const StepWs &w, void *stream) {
    if (a->x_final && a->W_lm) {
        if (!a->ws || a->ws_bytes < (size_t)a->B * tree->T * sizeof(unsigned long long)) return MTV_ERR_WORKSPACE;
        unsigned long long *keys = static_cast<unsigned long long *>(a->ws);
        const int rc = lm_head_argmax(tree, a->B, a->H, a->V, a->x_final, a->W_lm, nullptr, nullptr, keys, stream);
        if (rc != MTV_OK) return rc;
        return tree_accept_keys(tree, a->B, keys, a->tree_tok, a->accept_len, a->best_path, a->acc_nodes, a->acc_tok,
                                a->next_root, stream);
    }
    return tree_accept(tree, a->B, a->V, a->logits, a->tree_tok, a->accept_len, a->best_path, a->acc_nodes, a->acc_tok,
                       a->next_root, w.accept, w.accept_bytes, stream);
}

// One step; root_tok and the optional append are given separately so that a chain of steps can feed a step's root
// from the previous step's next_root without touching the caller's structs.
static int verify_step(const mtv_tree_t *tree, const mtv_step_args *a, const int32_t *root_tok,
                       const mtv_append_args *ap, void *stream) {
    if (!tree || !a || !a->k_caches_host || !a->v_caches_host || !root_tok) return MTV_ERR_INVALID_ARG;
    // The attention needs nothing of the heads, and the scan of stored logits nothing of either: what was enqueued in front of
    // the heads is complete at the heads' gate (see launch_dependent), so each starts where SMs fall free at the end of the one
    // before.  The append, which the attention does need, goes in front of the heads.
    const StepWs w = step_ws(tree, a);
    // (in front of the append, which rotates the queries in place: a refused call can be repeated)
    int rc = mtv::heads_check(tree, tree->K, a->B, a->H, a->V, a->hidden, a->W1, a->W2, root_tok, a->cand, a->tree_tok, a->ws, a->ws_bytes);
    if (rc != MTV_OK) return rc;
    if (ap && (ap->k_new_layers || ap->v_new_layers)) {
        // the tree nodes' K/V rows of every layer, in one launch
        rc = tree_kv_append_rope_layers(tree, a->B, a->Hq, a->Hkv, a->D, a->n_layers, const_cast<mtv_bf16 *>(a->q_layers),
                                        ap->k_new_layers, ap->v_new_layers, a->k_caches, a->v_caches, a->stride_b,
                                        a->stride_h, a->stride_t, a->Lcap, a->seq_lens, ap->rope_theta, a->status, stream);
        if (rc != MTV_OK) return rc;
    }
    mtv::Gate gate;
    rc = mtv::heads_topk_range(tree, mtv::HeadsRange{0, tree->K, w.apart ? &gate : nullptr}, a->B, a->H, a->V, a->hidden, a->W1, a->b1,
                               a->W2, root_tok, a->cand, a->cand_logit, a->tree_tok, a->ws, a->ws_bytes, stream);
    if (rc != MTV_OK) return rc;
    rc = mtv::tree_attention_layers(tree, a->B, a->Hq, a->Hkv, a->D, a->n_layers, a->q_layers, a->k_caches_host, a->v_caches_host,
                                    a->stride_b, a->stride_h, a->stride_t, a->Lcap, a->seq_lens, a->scale, a->out_layers,
                                    a->status, w.attn, w.attn_bytes, stream, w.apart ? &gate : nullptr);
    if (rc != MTV_OK) return rc;
    if (w.apart) {       // acceptance and compaction in one launch behind the scan of the logits or the LM head
        unsigned long long *keys = reinterpret_cast<unsigned long long *>(w.accept);
        int ns = 1;
        if (a->x_final && a->W_lm) {
            keys = static_cast<unsigned long long *>(a->ws);     // where a caller may look for them; the heads are done, their tickets lie behind
            rc = mtv::lm_head_keys(tree, a->B, a->H, a->V, a->x_final, a->W_lm, nullptr, nullptr, keys, gate, (cudaStream_t)stream);
        } else {
            ns = mtv::accept_ws_layout(tree, a->B, a->V).nsplit;
            rc = mtv::argmax_keys_partial(tree, a->B, a->V, a->logits, keys, gate, (cudaStream_t)stream);
        }
        if (rc != MTV_OK) return rc;
        return mtv::accept_compact(tree, a, ns, keys, reinterpret_cast<int32_t *>((char *)a->ws + mtv::heads_ws_layout(tree->K, a->B, a->H, a->V).tickets_off),
                                   gate, (cudaStream_t)stream);
    }
    rc = step_accept(tree, a, w, stream);
    if (rc != MTV_OK) return rc;
    return kv_compact_accepted(tree, a->B, a->Hkv, a->D, a->n_layers, a->k_caches, a->v_caches, a->stride_b,
                               a->stride_h, a->stride_t, a->Lcap, a->seq_lens, a->accept_len, a->acc_nodes, a->status,
                               stream);
}

extern "C" int mtv_verify_step(const mtv_tree_t *tree, const mtv_step_args *a, void *stream) {
    MTV_RANGE("mtv_verify_step");
    if (!a) return MTV_ERR_INVALID_ARG;
    return verify_step(tree, a, a->root_tok, nullptr, stream);
}

// n steps back to back on one stream.  Nothing is decided on the host between them: step s + 1 takes its root token
// from step s's next_root and its prefix lengths from the seq_lens that step s's compaction advanced, both on the device.
extern "C" int mtv_verify_steps(const mtv_tree_t *tree, const mtv_step_args *steps, const mtv_append_args *appends,
                                int n_steps, void *stream) {
    MTV_RANGE("mtv_verify_steps");
    if (!tree || !steps || n_steps < 1) return MTV_ERR_INVALID_ARG;
    for (int s = 0; s < n_steps; ++s) {      // the whole chain is looked at before anything is enqueued
        if (!steps[s].root_tok && (s == 0 || !steps[s - 1].next_root)) return MTV_ERR_INVALID_ARG;
        if (!steps[s].seq_lens || steps[s].seq_lens != steps[0].seq_lens) return MTV_ERR_INVALID_ARG;   // one chain, one set of lengths
        if (!steps[s].k_caches_host || !steps[s].v_caches_host) return MTV_ERR_INVALID_ARG;
    }
    for (int s = 0; s < n_steps; ++s) {
        const mtv_step_args *a = steps + s;
        const int32_t *root = a->root_tok ? a->root_tok : steps[s - 1].next_root;
        const int rc = verify_step(tree, a, root, appends ? appends + s : nullptr, stream);
        if (rc != MTV_OK) return rc;
    }
    return MTV_OK;
}

namespace {
// Copy streams and events of the host-buffer variant, created on first use, one set per device (the variant
// synchronises anyway, so it is not one of the allocation-free hot calls).  Calls on one device take turns.
constexpr int HOST_GROUPS = 8;   // most groups of layers in which queries go up and attention outputs come down
struct HostStepAux {
    cudaStream_t up = nullptr, down = nullptr;
    cudaEvent_t start = nullptr, logits_up = nullptr, down_done = nullptr;
    cudaEvent_t q_up[HOST_GROUPS] = {}, done[HOST_GROUPS] = {};   // a group's queries are up / its attention is done
    bool ready = false;
    std::mutex busy;
};
HostStepAux g_aux_table[mtv::MTV_MAX_DEVICES];
int host_step_aux(HostStepAux **out) {
    int dev = 0;
    MTV_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= mtv::MTV_MAX_DEVICES) return MTV_ERR_UNSUPPORTED_SHAPE;
    HostStepAux &g_aux = g_aux_table[dev];
    *out = &g_aux;
    std::lock_guard<std::mutex> lock(g_aux.busy);
    if (g_aux.ready) return MTV_OK;
    MTV_CUDA_CHECK(cudaStreamCreateWithFlags(&g_aux.up, cudaStreamNonBlocking));
    MTV_CUDA_CHECK(cudaStreamCreateWithFlags(&g_aux.down, cudaStreamNonBlocking));
    for (cudaEvent_t *e : {&g_aux.start, &g_aux.logits_up, &g_aux.down_done}) MTV_CUDA_CHECK(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
    for (int i = 0; i < HOST_GROUPS; ++i) {
        MTV_CUDA_CHECK(cudaEventCreateWithFlags(&g_aux.q_up[i], cudaEventDisableTiming));
        MTV_CUDA_CHECK(cudaEventCreateWithFlags(&g_aux.done[i], cudaEventDisableTiming));
    }
    g_aux.ready = true;
    return MTV_OK;
}

// A step's small results (tokens, lengths, paths) written straight into mapped host buffers: one launch instead of a copy
// of 3 us and a gap as long for each of them.
struct HostResults {
    static constexpr int N = 7;
    const int32_t *src[N];
    int32_t *dst[N];
    int n[N];
};
__global__ void __launch_bounds__(256) host_results_kernel(const HostResults r) {
    mtv::previous_done();
#pragma unroll 1
    for (int k = 0; k < HostResults::N; ++k)
        for (int i = threadIdx.x; i < r.n[k]; i += blockDim.x) r.dst[k][i] = r.src[k][i];
}
int send_results(HostResults r, cudaStream_t st) {
    HostResults m = r;
    bool mapped = true;
    for (int k = 0; k < HostResults::N && mapped; ++k) {
        cudaPointerAttributes a;
        mapped = cudaPointerGetAttributes(&a, r.dst[k]) == cudaSuccess && a.type == cudaMemoryTypeHost && a.devicePointer;
        if (mapped) m.dst[k] = static_cast<int32_t *>(a.devicePointer);
    }
    (void)cudaGetLastError();
    if (mapped) {
        MTV_CUDA_CHECK(mtv::launch_dependent(host_results_kernel, dim3(1), 256, 0, st, m));
        return MTV_OK;
    }
    for (int k = 0; k < HostResults::N; ++k)     // pageable buffers
        MTV_CUDA_CHECK(cudaMemcpyAsync(r.dst[k], r.src[k], (size_t)r.n[k] * 4, cudaMemcpyDeviceToHost, st));
    return MTV_OK;
}
}  // namespace

// The transfers overlap the compute.  At the 7B shape with L = 8192 the queries (17 MB) take 330 us to come up, the logits as
// much again and the attention outputs to go down, against 640 us of heads and 270 us of attention.  Nothing orders the
// heads and the attention, so half of the heads run while the queries come up, then the attention in groups of layers as
// their queries arrive, its outputs leaving at once, and the other heads while the last outputs go down and the logits
// come up.  (With all heads first the outputs' way down was waited for at the end: 1173 us.)  A launch of the attention
// costs about 15 us beside its work, so there are no more groups than it takes for the first group's queries and the
// last group's outputs to hide behind half of the heads.
extern "C" int mtv_verify_step_host(const mtv_tree_t *tree, const mtv_step_args *d, const mtv_step_args *h,
                                    void *stream) {
    MTV_RANGE("mtv_verify_step_host");
    if (!tree || !d || !h || !d->k_caches_host || !d->v_caches_host) return MTV_ERR_INVALID_ARG;
    HostStepAux *aux = nullptr;
    if (host_step_aux(&aux) != MTV_OK) return MTV_ERR_CUDA;
    HostStepAux &g_aux = *aux;
    std::lock_guard<std::mutex> turn(g_aux.busy);
    cudaStream_t st = (cudaStream_t)stream, up = g_aux.up, down = g_aux.down;
    const size_t B = d->B, T = tree->T, K = tree->K;
    const size_t per_layer = B * T * d->Hq * d->D;           // elements
    const double copy_us = (double)d->n_layers * per_layer * 2 / 50e3, heads_us = 0.5 * tree->K * d->V * (double)d->H * 2 / 6.5e6;
    const int groups = std::max(1, std::min({HOST_GROUPS, d->n_layers, std::max(2, (int)(copy_us / (heads_us + 1.0)) + 1)}));
    auto first_layer = [&](int g) { return (int)((int64_t)d->n_layers * g / groups); };
    // uploads
    MTV_CUDA_CHECK(cudaEventRecord(g_aux.start, st));         // the copy streams start where the caller's stream is
    MTV_CUDA_CHECK(cudaStreamWaitEvent(up, g_aux.start, 0));
    MTV_CUDA_CHECK(cudaStreamWaitEvent(down, g_aux.start, 0));
    MTV_CUDA_CHECK(cudaMemcpyAsync((void *)d->hidden, h->hidden, B * d->H * 2, cudaMemcpyHostToDevice, st));
    MTV_CUDA_CHECK(cudaMemcpyAsync((void *)d->root_tok, h->root_tok, B * 4, cudaMemcpyHostToDevice, st));
    auto upload_q = [&](int g) {
        const size_t l0 = first_layer(g), n = first_layer(g + 1) - l0;
        MTV_CUDA_CHECK(cudaMemcpyAsync((void *)(d->q_layers + l0 * per_layer), h->q_layers + l0 * per_layer, n * per_layer * 2,
                                       cudaMemcpyHostToDevice, up));
        MTV_CUDA_CHECK(cudaEventRecord(g_aux.q_up[g], up));
        return MTV_OK;
    };
    auto heads = [&](int k0, int n) {
        return mtv::heads_topk_range(tree, mtv::HeadsRange{k0, n, nullptr}, d->B, d->H, d->V, d->hidden, d->W1, d->b1, d->W2, d->root_tok,
                                     d->cand, d->cand_logit, d->tree_tok, d->ws, d->ws_bytes, stream);
    };
    const int before = tree->K / 2;
    int rc = upload_q(0);
    if (rc == MTV_OK && before > 0) rc = heads(0, before);   // (enqueued before the other copies: each costs the host 4 us)
    for (int g = 1; g < groups && rc == MTV_OK; ++g) rc = upload_q(g);
    if (rc != MTV_OK) return rc;
    if (d->x_final && d->W_lm)
        MTV_CUDA_CHECK(cudaMemcpyAsync((void *)d->x_final, h->x_final, B * T * d->H * 2, cudaMemcpyHostToDevice, up));
    else
        MTV_CUDA_CHECK(cudaMemcpyAsync((void *)d->logits, h->logits, B * T * d->V * 2, cudaMemcpyHostToDevice, up));
    MTV_CUDA_CHECK(cudaEventRecord(g_aux.logits_up, up));
    // attention, a group of layers at a time
    for (int g = 0; g < groups; ++g) {
        const size_t l0 = first_layer(g);
        const int n = first_layer(g + 1) - (int)l0;
        MTV_CUDA_CHECK(cudaStreamWaitEvent(st, g_aux.q_up[g], 0));
        rc = mtv::tree_attention_layers(tree, d->B, d->Hq, d->Hkv, d->D, n, d->q_layers + l0 * per_layer, d->k_caches_host + l0,
                                        d->v_caches_host + l0, d->stride_b, d->stride_h, d->stride_t, d->Lcap, d->seq_lens,
                                        d->scale, d->out_layers + l0 * per_layer, d->status, d->ws, d->ws_bytes, stream);
        if (rc != MTV_OK) return rc;
        MTV_CUDA_CHECK(cudaEventRecord(g_aux.done[g], st));
        MTV_CUDA_CHECK(cudaStreamWaitEvent(down, g_aux.done[g], 0));
        MTV_CUDA_CHECK(cudaMemcpyAsync(h->out_layers + l0 * per_layer, d->out_layers + l0 * per_layer, n * per_layer * 2,
                                       cudaMemcpyDeviceToHost, down));
    }
    rc = heads(before, tree->K - before);
    if (rc != MTV_OK) return rc;
    // acceptance and compaction
    MTV_CUDA_CHECK(cudaStreamWaitEvent(st, g_aux.logits_up, 0));
    const StepWs w = step_ws(tree, d);
    rc = step_accept(tree, d, w, stream);
    if (rc != MTV_OK) return rc;
    rc = kv_compact_accepted(tree, d->B, d->Hkv, d->D, d->n_layers, d->k_caches, d->v_caches, d->stride_b, d->stride_h,
                             d->stride_t, d->Lcap, d->seq_lens, d->accept_len, d->acc_nodes, d->status, stream);
    if (rc != MTV_OK) return rc;
    rc = send_results({{d->tree_tok, d->accept_len, d->best_path, d->acc_nodes, d->acc_tok, d->next_root, d->seq_lens},
                       {h->tree_tok, h->accept_len, h->best_path, h->acc_nodes, h->acc_tok, h->next_root, h->seq_lens},
                       {(int)(B * T), (int)B, (int)B, (int)(B * (K + 1)), (int)(B * (K + 1)), (int)B, (int)B}},
                      st);
    if (rc != MTV_OK) return rc;
    MTV_CUDA_CHECK(cudaEventRecord(g_aux.down_done, down));
    MTV_CUDA_CHECK(cudaStreamWaitEvent(st, g_aux.down_done, 0));
    MTV_CUDA_CHECK(cudaStreamSynchronize(st));
    return MTV_OK;
}

// ---------------------------------------------------------------------------
// Self-test of the bounded waits: a barrier nobody arrives on.
namespace {
__global__ void selftest_wait_timeout_kernel(int32_t *dev_error) {
    __shared__ __align__(8) unsigned long long bar_mem;
    const uint32_t bar = mtv::ptx::smem_u32(&bar_mem);
    if (threadIdx.x == 0) {
        mtv::ptx::mbar_init(bar, 1);
        mtv::ptx::fence_mbar_init();
    }
    __syncwarp();
    const bool ok = mtv::ptx::mbar_wait(bar, 0);      // gives up after WAIT_CYCLE_LIMIT cycles
    if (!ok && threadIdx.x == 0) atomicExch(dev_error, MTV_ERR_TIMEOUT);
}
}  // namespace

extern "C" int mtv_debug_bounds_enabled(void) {
#ifdef MTV_DEBUG_BOUNDS
    return 1;
#else
    return 0;
#endif
}

extern "C" int mtv_selftest_wait_timeout(const mtv_tree_t *tree, void *stream) {
    if (!tree || !tree->on_device) return MTV_ERR_INVALID_ARG;
    selftest_wait_timeout_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(tree->d_error);
    MTV_CUDA_CHECK(cudaGetLastError());
    return MTV_OK;
}
