"""Caches of all layers that one tensor map describes, against the same values in memory that no single map describes: every way in
which layers, sequences and heads may lie gives the same bits."""
import pytest
import torch

from paper_2603_03383_b200 import binding, synth
from tests._cases import make_tree, workspace

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _place(layout, x, which):
    """x [layers][B][Hkv][Lcap][D] as a list of views of that shape per layer; which: 0 K, 1 V."""
    n, B, H, L, D = x.shape
    if layout == "unevenly spaced":
        pool = torch.zeros(n * (x[0].numel() + 8 * n), dtype=x.dtype, device=DEV)
        at, out = 0, []
        for l in range(n):
            out.append(pool[at:at + x[0].numel()].view(B, H, L, D))
            at += x[0].numel() + 8 * (l + 1)
    elif layout == "one block":
        out = list(torch.zeros_like(x))
    elif layout == "gaps between layers":
        out = [row[:x[0].numel()].view(B, H, L, D) for row in torch.zeros(n, x[0].numel() + 64, dtype=x.dtype, device=DEV)]
    elif layout == "last layer first":
        out = list(torch.zeros_like(x))[::-1]
    elif layout == "rows of all heads":
        out = [t.transpose(1, 2) for t in torch.zeros(n, B, L, H, D, dtype=x.dtype, device=DEV)]
    elif layout == "rows of all heads, gaps":
        out = [row[:x[0].numel()].view(B, L, H, D).transpose(1, 2) for row in torch.zeros(n, x[0].numel() + 64, dtype=x.dtype, device=DEV)]
    else:                                        # K and V of a layer side by side: gaps that are no multiple of a sequence's
        assert layout == "K and V side by side"
        out = [t[which] for t in torch.zeros(n, 2, B, H, L, D, dtype=x.dtype, device=DEV)]
    for t, src in zip(out, x):
        t.copy_(src)
    return out


@pytest.mark.parametrize("T,Hq,Hkv,D,lens,n_layers", [
    (64, 8, 2, 128, [300, 77, 129], 3),          # pairs
    (64, 28, 4, 128, [511], 5),                  # one sequence
    (29, 4, 1, 128, [200, 130], 4),              # a single row tile, one head
    (64, 8, 4, 64, [65, 400], 3),
    (37, 3, 1, 64, [90], 2),
])
def test_layouts_of_layers(T, Hq, Hkv, D, lens, n_layers):
    K, H, V, B = 4, 64, 600, len(lens)
    tb, tree = make_tree("rank_prior", K, (), T)
    Lcap = max(lens) + T + 5
    k, v = (synth.normal_bf16(T, i, (n_layers, B, Hkv, Lcap, D), device=DEV) for i in (10, 50))
    q = synth.normal_bf16(T, 90, (n_layers, B, T, Hq, D), device=DEV)
    logits = synth.normal_bf16(T, 91, (B, T, V), device=DEV)
    hidden, W1, b1, W2, root = synth.head_inputs(B, H, V, K, seed=3, device=DEV)

    def step(layout):
        ks, vs = _place(layout, k, 0), _place(layout, v, 1)
        i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
        d = dict(hidden=hidden, W1=W1, b1=b1, W2=W2, root_tok=root, q_layers=q, out_layers=torch.full_like(q, 9.0), logits=logits,
                 seq_lens=torch.tensor(lens, dtype=torch.int32, device=DEV), cand=i32(B, tree.C), tree_tok=i32(B, T), accept_len=i32(B),
                 best_path=i32(B), acc_nodes=i32(B, K + 1), acc_tok=i32(B, K + 1), next_root=i32(B), status=i32(B),
                 k_caches=binding.cache_pointer_array(ks, DEV), v_caches=binding.cache_pointer_array(vs, DEV),
                 k_caches_host=binding.cache_pointer_array(ks), v_caches_host=binding.cache_pointer_array(vs),
                 ws=workspace(tree, B, H, V, Hq, Hkv, D, Lcap))
        a = binding.StepArgs()
        a.B, a.H, a.V, a.Hq, a.Hkv, a.D, a.n_layers, a.Lcap = B, H, V, Hq, Hkv, D, n_layers, Lcap
        a.stride_b, a.stride_h, a.stride_t = ks[0].stride()[:3]
        for name, t in d.items():
            setattr(a, name, t.data_ptr())
        a.ws_bytes = d["ws"].numel()
        binding.mtv_verify_step(tree, a)
        torch.cuda.synchronize()
        assert binding.mtv_device_error(tree) == 0
        return d["out_layers"], torch.stack(ks), torch.stack(vs), d["seq_lens"]

    want = step("unevenly spaced")
    assert (want[0] != 9.0).any(dim=-1).all()
    for layout in ("one block", "gaps between layers", "last layer first", "rows of all heads", "rows of all heads, gaps", "K and V side by side"):
        for g, w in zip(step(layout), want):
            assert torch.equal(g, w), layout
