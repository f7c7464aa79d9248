"""Calls whose inputs are written by kernels enqueued directly in front of them, without a synchronisation: the early starts
inside a call must not read anything older.  The same calls with a synchronisation in between give the expected bits."""
import pytest
import torch

from paper_2603_03383_b200 import binding, synth
from tests._cases import make_tree, workspace

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,H,V", [(1, 512, 20000), (3, 512, 20000), (9, 72, 9000)])     # (9, 72): two batch tiles, no early start
@pytest.mark.parametrize("graph", [False, True])
def test_heads(B, H, V, graph):
    K = 3
    tb, tree = make_tree("cartesian", K, (4, 2, 2))
    sets = [[t.to(DEV) for t in synth.head_inputs(B, H, V, K, seed=40 + i)] for i in range(4)]
    cur = [t.clone() for t in sets[0]]
    ws = workspace(tree, B, H, V, 0, 0, 0, 0)
    cand, tt = torch.zeros(B, tree.C, dtype=torch.int32, device=DEV), torch.zeros(B, tree.T, dtype=torch.int32, device=DEV)
    call = lambda: binding.medusa_heads_topk(tree, *cur[:4], cur[4], cand, None, tt, ws)
    want = []
    for s in sets:
        for c, t in zip(cur, s):
            c.copy_(t)
        torch.cuda.synchronize()
        call()
        torch.cuda.synchronize()
        want.append((cand.clone(), tt.clone()))
    replay = call
    if graph:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            call()
        replay = g.replay
    got = []
    for i in range(12):
        for c, t in zip(cur, sets[i % 4]):
            c.copy_(t)
        replay()
        got.append((cand.clone(), tt.clone()))
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    for i, (c, t) in enumerate(got):
        assert torch.equal(c, want[i % 4][0]) and torch.equal(t, want[i % 4][1]), i


@pytest.mark.parametrize("D,B,lm_head", [(128, 1, False), (64, 2, False), (128, 2, True)])
@pytest.mark.parametrize("graph", [False, True])
def test_step(D, B, lm_head, graph):
    K, H, V, Hq, Hkv, T, L, n_layers = 4, 64, 3000, 8, 2, 64, 300, 6
    tb, tree = make_tree("rank_prior", K, (), T)
    Lcap = L + T + 40
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)

    def inputs(i):
        hidden, W1, b1, W2, root = (t.to(DEV) for t in synth.head_inputs(B, H, V, K, seed=70 + i))
        return dict(hidden=hidden, W1=W1, b1=b1, W2=W2, root_tok=root, q_layers=synth.normal_bf16(i, 1, (n_layers, B, T, Hq, D), device=DEV),
                    kc=synth.normal_bf16(i, 2, (n_layers, B, Hkv, Lcap, D), device=DEV), vc=synth.normal_bf16(i, 3, (n_layers, B, Hkv, Lcap, D), device=DEV),
                    logits=synth.normal_bf16(i, 4, (B, T, V), device=DEV), x_final=synth.normal_bf16(i, 5, (B, T, H), device=DEV),
                    W_lm=synth.normal_bf16(i, 6, (V, H), device=DEV), seq_lens=torch.full((B,), L - 17 * i, dtype=torch.int32, device=DEV))
    sets = [inputs(i) for i in range(3)]
    cur = {n: t.clone() for n, t in sets[0].items()}
    out = dict(out_layers=torch.zeros_like(cur["q_layers"]), cand=i32(B, tree.C), tree_tok=i32(B, T), accept_len=i32(B), best_path=i32(B),
               acc_nodes=i32(B, K + 1), acc_tok=i32(B, K + 1), next_root=i32(B), status=i32(B))
    ptrs = dict(k_caches=binding.cache_pointer_array(list(cur["kc"]), DEV), v_caches=binding.cache_pointer_array(list(cur["vc"]), DEV),
                k_caches_host=binding.cache_pointer_array(list(cur["kc"])), v_caches_host=binding.cache_pointer_array(list(cur["vc"])))
    ws = workspace(tree, B, H, V, Hq, Hkv, D, Lcap)
    a = binding.StepArgs()
    a.B, a.H, a.V, a.Hq, a.Hkv, a.D, a.n_layers, a.Lcap = B, H, V, Hq, Hkv, D, n_layers, Lcap
    a.stride_b, a.stride_h, a.stride_t = cur["kc"].stride()[1:4]
    for n, t in dict(cur, **out, **ptrs, ws=ws).items():
        if n not in ("kc", "vc") and (lm_head or n not in ("x_final", "W_lm")):
            setattr(a, n, t.data_ptr())
    a.ws_bytes = ws.numel()
    result = lambda: [t.clone() for t in list(out.values()) + [cur["seq_lens"], cur["kc"], cur["vc"]]]

    def load(i):
        for n, t in sets[i].items():
            cur[n].copy_(t)
    want = []
    for i in range(3):
        load(i)
        torch.cuda.synchronize()
        binding.mtv_verify_step(tree, a)
        torch.cuda.synchronize()
        want.append(result())
    replay = lambda: binding.mtv_verify_step(tree, a)
    if graph:
        load(0)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            binding.mtv_verify_step(tree, a)
        replay = g.replay
    got = []
    for i in range(9):
        load(i % 3)
        replay()
        got.append(result())
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    for i, r in enumerate(got):
        assert all(torch.equal(x, y) for x, y in zip(r, want[i % 3])), i


def test_a_refused_chain_changes_nothing():
    """Heads that are refused (here: a workspace too small for them) leave the queries unrotated and the caches as they were."""
    K, H, V, Hq, Hkv, T, L, n_layers, B, D = 4, 64, 600, 4, 1, 64, 50, 2, 1, 64
    tb, tree = make_tree("rank_prior", K, (), T)
    hidden, W1, b1, W2, root = (t.to(DEV) for t in synth.head_inputs(B, H, V, K, seed=5))
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    kc, vc = (synth.normal_bf16(1, i, (n_layers, B, Hkv, L + T, D), device=DEV) for i in (2, 3))
    q = synth.normal_bf16(1, 4, (n_layers, B, T, Hq, D), device=DEV)
    kn, vn = (synth.normal_bf16(1, i, (n_layers, B, T, Hkv, D), device=DEV) for i in (5, 6))
    d = dict(hidden=hidden, W1=W1, b1=b1, W2=W2, root_tok=root, q_layers=q, out_layers=torch.zeros_like(q), logits=synth.normal_bf16(1, 7, (B, T, V), device=DEV),
             seq_lens=torch.full((B,), L, dtype=torch.int32, device=DEV), cand=i32(B, tree.C), tree_tok=i32(B, T), accept_len=i32(B), best_path=i32(B),
             acc_nodes=i32(B, K + 1), acc_tok=i32(B, K + 1), next_root=i32(B), k_caches=binding.cache_pointer_array(list(kc), DEV),
             v_caches=binding.cache_pointer_array(list(vc), DEV), k_caches_host=binding.cache_pointer_array(list(kc)),
             v_caches_host=binding.cache_pointer_array(list(vc)), ws=workspace(tree, B, H, V, Hq, Hkv, D, L + T))
    a = binding.StepArgs()
    a.B, a.H, a.V, a.Hq, a.Hkv, a.D, a.n_layers, a.Lcap = B, H, V, Hq, Hkv, D, n_layers, L + T
    a.stride_b, a.stride_h, a.stride_t = kc.stride()[1:4]
    for n, t in d.items():
        setattr(a, n, t.data_ptr())
    a.ws_bytes = 256
    ap = binding.AppendArgs()
    ap.k_new_layers, ap.v_new_layers, ap.rope_theta = kn.data_ptr(), vn.data_ptr(), 0.0
    before = [t.clone() for t in (q, kc, vc)]
    with pytest.raises(binding.MtvError) as e:
        binding.mtv_verify_steps(tree, [a], [ap])
    torch.cuda.synchronize()
    assert e.value.code == -3
    assert all(torch.equal(x, y) for x, y in zip(before, (q, kc, vc)))
