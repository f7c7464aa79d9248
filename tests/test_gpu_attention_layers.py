"""Tree attention of several layers in one launch, the two single-layer kernels on either side of their rule, and scores whose
maximum grows along the cache (the reference of the exponentials has to move), against the fp64 checker."""

import pytest
import torch

from oracle import reference as ref
from paper_2603_03383_b200 import binding, synth
from tests._cases import assert_close, make_tree, workspace

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("T,Hq,Hkv,D,lens,n_layers", [
    (64, 8, 2, 128, [63], 2),                  # one group and the tree across a group boundary
    (64, 8, 2, 128, [64, 0, 129], 5),          # last group exactly full; an empty prefix; ragged
    (29, 4, 1, 128, [700], 3),                 # one row tile, pieces of one group
    (128, 16, 2, 128, [1000, 1], 2),           # four row blocks
    (64, 7, 1, 128, [300, 517], 9),            # rows that belong to nobody
    (65, 8, 8, 64, [127, 128], 4),
    (128, 8, 1, 64, [2500], 2),                # head size 64 with splits: fp32 partials
])
@pytest.mark.parametrize("apart", [True, False])
def test_layers_in_one_launch(T, Hq, Hkv, D, lens, n_layers, apart):
    """apart = False: a workspace too small for the parts of the step side by side, which then wait for each other."""
    K, H, V, B = 4, 64, 600, len(lens)
    tb, tree = make_tree("rank_prior", K, (), T)
    Lcap = max(lens) + T + 3
    ks = [synth.normal_bf16(T, 10 + l, (B, Hkv, Lcap, D), device=DEV) for l in range(n_layers)]
    vs = [synth.normal_bf16(T, 50 + l, (B, Hkv, Lcap, D), device=DEV) for l in range(n_layers)]
    q = synth.normal_bf16(T, 90, (n_layers, B, T, Hq, D), device=DEV)
    hidden, W1, b1, W2, root = synth.head_inputs(B, H, V, K, seed=3, device=DEV)
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    d = dict(hidden=hidden, W1=W1, b1=b1, W2=W2, root_tok=root, q_layers=q, out_layers=torch.full_like(q, 9.0),
             logits=synth.normal_bf16(T, 91, (B, T, V), device=DEV), seq_lens=torch.tensor(lens, dtype=torch.int32, device=DEV),
             cand=i32(B, tree.C), cand_logit=torch.zeros(B, tree.C - 1, device=DEV), tree_tok=i32(B, T), accept_len=i32(B),
             best_path=i32(B), acc_nodes=i32(B, K + 1), acc_tok=i32(B, K + 1), next_root=i32(B), status=i32(B),
             k_caches=binding.cache_pointer_array(ks, DEV), v_caches=binding.cache_pointer_array(vs, DEV),
             k_caches_host=binding.cache_pointer_array(ks), v_caches_host=binding.cache_pointer_array(vs),
             ws=workspace(tree, B, H, V, Hq, Hkv, D, Lcap))
    a = binding.StepArgs()
    a.B, a.H, a.V, a.Hq, a.Hkv, a.D, a.n_layers, a.Lcap = B, H, V, Hq, Hkv, D, n_layers, Lcap
    a.stride_b, a.stride_h, a.stride_t = ks[0].stride()[:3]
    for n, t in d.items():
        setattr(a, n, t.data_ptr())
    a.ws_bytes = d["ws"].numel() if apart else workspace(tree, B, 0, 0, Hq, Hkv, D, Lcap).numel()
    want = [ref.tree_attention(q[l].cpu(), ks[l].cpu(), vs[l].cpu(), torch.tensor(lens, dtype=torch.int32), tb["mask"])
            for l in range(n_layers)]
    binding.mtv_verify_step(tree, a)
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    for l in range(n_layers):
        assert_close(d["out_layers"][l], want[l], "layer %d" % l)
    acc = ref.tree_accept(ref.node_argmax(d["logits"].cpu()), d["tree_tok"].cpu(), tb)
    assert d["accept_len"].tolist() == acc["accept_len"].tolist() and d["next_root"].tolist() == acc["next_root"].tolist()
    assert d["seq_lens"].tolist() == [L + n + 1 for L, n in zip(lens, d["accept_len"].tolist())]


@pytest.mark.parametrize("T,Hq,Hkv,D,lens,Lcap", [
    (64, 8, 2, 128, [2000], 2200),             # key splits on CTA pairs
    (64, 28, 4, 128, [40, 300, 1200, 900, 64, 0, 777], 8064),   # the even division: capacity says long
    (128, 8, 4, 128, [600, 200], 33000),
    (128, 8, 2, 64, [900, 17], 1030),
])
@pytest.mark.parametrize("gain", [1.0, 40.0])
def test_single_layer_calls(T, Hq, Hkv, D, lens, Lcap, gain):
    """gain 40: the scores' spread is about 60 in log2 units, so later groups exceed the first one's maximum by far."""
    tb, tree = make_tree("rank_prior", 4, (), T)
    B = len(lens)
    q = (synth.normal_bf16(1, 1, (B, T, Hq, D), device=DEV) * gain).to(torch.bfloat16)
    k, v = (synth.normal_bf16(1, i, (B, Hkv, Lcap, D), device=DEV) for i in (2, 3))
    sl = torch.tensor(lens, dtype=torch.int32)
    top = max(lens) + T
    want = ref.tree_attention(q.cpu(), k[:, :, :top].cpu(), v[:, :, :top].cpu(), sl, tb["mask"])
    out = torch.full_like(q, 9.0)
    ws = workspace(tree, B, 0, 0, Hq, Hkv, D, Lcap)
    for _ in range(2):                          # the merge counters are back at zero after a call
        binding.tree_verify_attention(tree, q, k, v, sl.to(DEV), out, ws)
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    assert_close(out, want)


@pytest.mark.parametrize("D,n_layers", [(64, 1), (64, 4), (128, 4)])
def test_two_trees_on_two_streams(D, n_layers):
    """Launches that share the device: neither needs all its blocks resident at once."""
    T, Hq, Hkv, L = 64, 8, 2, 1500
    K, H, V, B = 4, 64, 600, 2
    sides = []
    for i in range(2):
        tb, tree = make_tree("rank_prior", K, (), T)
        Lcap = L + T
        ks, vs = ([synth.normal_bf16(i, s + l, (B, Hkv, Lcap, D), device=DEV) for l in range(n_layers)] for s in (10, 50))
        q = synth.normal_bf16(i, 90, (n_layers, B, T, Hq, D), device=DEV)
        lens = torch.tensor([L, 700 + 100 * i], dtype=torch.int32, device=DEV)
        out = torch.zeros_like(q)
        ws = workspace(tree, B, H, V, Hq, Hkv, D, Lcap)
        hidden, W1, b1, W2, root = (t.to(DEV) for t in synth.head_inputs(B, H, V, K, seed=3))
        i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
        d = dict(hidden=hidden, W1=W1, b1=b1, W2=W2, root_tok=root, q_layers=q, out_layers=out, seq_lens=lens.clone(),
                 logits=synth.normal_bf16(T, 91, (B, T, V), device=DEV), cand=i32(B, tree.C), tree_tok=i32(B, T), accept_len=i32(B),
                 best_path=i32(B), acc_nodes=i32(B, K + 1), acc_tok=i32(B, K + 1), next_root=i32(B),
                 k_caches=binding.cache_pointer_array(ks, DEV), v_caches=binding.cache_pointer_array(vs, DEV),
                 k_caches_host=binding.cache_pointer_array(ks), v_caches_host=binding.cache_pointer_array(vs), ws=ws)
        a = binding.StepArgs()
        a.B, a.H, a.V, a.Hq, a.Hkv, a.D, a.n_layers, a.Lcap = B, H, V, Hq, Hkv, D, n_layers, Lcap
        a.stride_b, a.stride_h, a.stride_t = ks[0].stride()[:3]
        for n, t in d.items():
            setattr(a, n, t.data_ptr())
        a.ws_bytes = ws.numel()
        st = torch.cuda.Stream()

        def call(tree=tree, a=a, d=d, lens=lens, q=q, ks=ks, vs=vs, out=out, ws=ws, st=st):
            with torch.cuda.stream(st):
                if n_layers == 1:
                    binding.tree_verify_attention(tree, q[0], ks[0], vs[0], lens, out[0], ws)
                else:
                    d["seq_lens"].copy_(lens)
                    binding.mtv_verify_step(tree, a)
        torch.cuda.synchronize()
        call()
        torch.cuda.synchronize()
        assert d["accept_len"].sum().item() == 0           # nothing accepted: the step moves no cache rows, calls repeat
        sides.append((tree, call, out, out.clone()))
        out.zero_()
    torch.cuda.synchronize()
    for _ in range(60):
        for _, call, _, _ in sides:
            call()
    torch.cuda.synchronize()
    for tree, _, out, want in sides:
        assert binding.mtv_device_error(tree) == 0
        assert torch.equal(out, want)


@pytest.mark.parametrize("T,Hq,Hkv,D,lens,n_layers,scale", [
    (29, 4, 1, 128, [70], 70, 0.0),                              # a second launch behind the first 64 layers
    (16, 2, 2, 64, [40, 129], 65, 0.0),
    (29, 8, 2, 128, [5 * i % 301 for i in range(70)], 2, 0.0),   # lengths in three lots of 32
    (64, 2, 1, 64, [7 * i % 401 for i in range(33)], 3, 0.0),
    (64, 8, 2, 64, [300, 0, 63], 3, -0.11),                      # a negative scale, hidden tree columns
])
@pytest.mark.parametrize("apart", [True, False])
def test_many_layers_many_sequences_negative_scale(T, Hq, Hkv, D, lens, n_layers, scale, apart):
    tb, tree = make_tree("rank_prior", 4, (), T)
    B, Lcap, H, V, K = len(lens), max(lens) + T + 3, 64, 600, 4
    ks, vs = ([synth.normal_bf16(T, s + l, (B, Hkv, Lcap, D), device=DEV) for l in range(n_layers)] for s in (100, 300))
    q = synth.normal_bf16(T, 90, (n_layers, B, T, Hq, D), device=DEV)
    sl = torch.tensor(lens, dtype=torch.int32)
    want = [ref.tree_attention(q[l].cpu(), ks[l].cpu(), vs[l].cpu(), sl, tb["mask"], scale=scale) for l in range(n_layers)]
    if B > 16:          # more sequences than the heads take: one-layer calls
        out = torch.full_like(q, 9.0)
        ws = workspace(tree, B, 0, 0, Hq, Hkv, D, Lcap)
        for l in range(n_layers):
            binding.tree_verify_attention(tree, q[l], ks[l], vs[l], sl.to(DEV), out[l], ws, scale=scale)
        torch.cuda.synchronize()
    else:
        hidden, W1, b1, W2, root = synth.head_inputs(B, H, V, K, seed=3, device=DEV)
        i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
        d = dict(hidden=hidden, W1=W1, b1=b1, W2=W2, root_tok=root, q_layers=q, out_layers=torch.full_like(q, 9.0),
                 logits=synth.normal_bf16(T, 91, (B, T, V), device=DEV), seq_lens=sl.to(DEV), cand=i32(B, tree.C), tree_tok=i32(B, T),
                 accept_len=i32(B), best_path=i32(B), acc_nodes=i32(B, K + 1), acc_tok=i32(B, K + 1), next_root=i32(B),
                 k_caches=binding.cache_pointer_array(ks, DEV), v_caches=binding.cache_pointer_array(vs, DEV),
                 k_caches_host=binding.cache_pointer_array(ks), v_caches_host=binding.cache_pointer_array(vs),
                 ws=workspace(tree, B, H, V, Hq, Hkv, D, Lcap))
        a = binding.StepArgs()
        a.B, a.H, a.V, a.Hq, a.Hkv, a.D, a.n_layers, a.Lcap = B, H, V, Hq, Hkv, D, n_layers, Lcap
        a.stride_b, a.stride_h, a.stride_t = ks[0].stride()[:3]
        a.scale = scale
        for n, t in d.items():
            setattr(a, n, t.data_ptr())
        a.ws_bytes = d["ws"].numel() if apart else workspace(tree, B, 0, 0, Hq, Hkv, D, Lcap).numel()
        binding.mtv_verify_step(tree, a)
        torch.cuda.synchronize()
        out = d["out_layers"]
    assert binding.mtv_device_error(tree) == 0
    for l in range(n_layers):
        assert_close(out[l], want[l], "layer %d" % l)
