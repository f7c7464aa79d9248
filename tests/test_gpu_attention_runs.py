"""Runs of many short items on one CTA: pieces of one to five groups follow one another, so that scores, weights and outputs of
neighbouring items are in flight together; and few long items, cut into many pieces.  Against plain PyTorch in 64 bits; the bound is that of all attention tests."""
import pytest
import torch

from paper_2603_03383_b200 import binding, synth
from tests._cases import assert_close, make_tree, workspace

pytestmark = pytest.mark.gpu
DEV = "cuda"
LENS = {"mixed": [3, 100, 192, 300, 64, 517, 0, 190], "one group": [40] * 8, "two": [130, 140, 150, 187, 128, 129, 160, 171],
        "long between short": [10, 1500, 20, 30, 700, 5, 260, 1]}


def _reference(q, k, v, lens, mask):
    """[B][T][Hq][D] in 64 bits; mask [T][T]."""
    B, T, Hq, D = q.shape
    out = torch.empty(q.shape, dtype=torch.float64, device=DEV)
    for b, L in enumerate(lens):
        n = L + T
        kk, vv = (x[b, :, :n].double().repeat_interleave(Hq // x.shape[1], dim=0) for x in (k, v))
        s = torch.einsum("thd,hnd->htn", q[b].double(), kk) / D ** 0.5
        s[:, :, L:].masked_fill_(~mask, -float("inf"))
        out[b] = torch.einsum("htn,hnd->thd", s.softmax(-1), vv)
    return out


def _check(T, Hq, Hkv, D, lens, n_layers, growing=False):
    """growing: keys of later groups are longer, so that their weights do not fit the first group's reference."""
    K, H, V, B = 4, 64, 600, len(lens)
    tb, tree = make_tree("rank_prior", K, (), T)
    mask = torch.as_tensor(tb["mask"], device=DEV).bool().view(T, T)
    Lcap = max(lens) + T + 3
    k, v = (synth.normal_bf16(T, i, (n_layers, B, Hkv, Lcap, D), device=DEV) for i in (10, 50))
    if growing:
        k *= (1 + torch.arange(Lcap, device=DEV) // 128 * 9).to(k.dtype)[:, None]
    q = synth.normal_bf16(T, 90, (n_layers, B, T, Hq, D), device=DEV)
    out = torch.full((q.numel() + 8,), 9.0, dtype=q.dtype, device=DEV)[8 if growing else 0:][:q.numel()].view(q.shape)     # at 16 or 32 bytes
    hidden, W1, b1, W2, root = synth.head_inputs(B, H, V, K, seed=3, device=DEV)
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    ks, vs = list(k), list(v)
    d = dict(hidden=hidden, W1=W1, b1=b1, W2=W2, root_tok=root, q_layers=q, out_layers=out, logits=synth.normal_bf16(T, 91, (B, T, V), device=DEV),
             seq_lens=torch.tensor(lens, dtype=torch.int32, device=DEV), cand=i32(B, tree.C), tree_tok=i32(B, T), accept_len=i32(B),
             best_path=i32(B), acc_nodes=i32(B, K + 1), acc_tok=i32(B, K + 1), next_root=i32(B), status=i32(B),
             k_caches=binding.cache_pointer_array(ks, DEV), v_caches=binding.cache_pointer_array(vs, DEV),
             k_caches_host=binding.cache_pointer_array(ks), v_caches_host=binding.cache_pointer_array(vs),
             ws=workspace(tree, B, H, V, Hq, Hkv, D, Lcap))
    a = binding.StepArgs()
    a.B, a.H, a.V, a.Hq, a.Hkv, a.D, a.n_layers, a.Lcap = B, H, V, Hq, Hkv, D, n_layers, Lcap
    a.stride_b, a.stride_h, a.stride_t = ks[0].stride()[:3]
    for n, t in d.items():
        setattr(a, n, t.data_ptr())
    a.ws_bytes = d["ws"].numel()
    want = [_reference(q[l], k[l], v[l], lens, mask) for l in range(n_layers)]
    binding.mtv_verify_step(tree, a)
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    for l in range(n_layers):
        assert_close(out[l], want[l], "layer %d" % l)


@pytest.mark.parametrize("lens", LENS)
@pytest.mark.parametrize("T,Hq,Hkv,D", [(64, 32, 8, 128), (29, 16, 8, 128), (117, 32, 8, 128), (64, 32, 8, 64), (22, 24, 8, 64)])
@pytest.mark.parametrize("growing", [False, True])
def test_runs_of_short_items(T, Hq, Hkv, D, lens, growing):
    _check(T, Hq, Hkv, D, LENS[lens], 12, growing)


@pytest.mark.parametrize("T,Hq,Hkv,D,lens,n_layers", [
    (47, 1, 1, 128, [9284], 2),        # 73 contributors with two rows each
    (100, 4, 1, 128, [4500], 1),       # pairs, 36 contributors
    (97, 4, 1, 128, [3100], 1),        # 25 contributors: the fewest that take this way
    (61, 2, 1, 64, [12000, 6000], 1),
    (128, 1, 1, 64, [18900], 1),       # 149 groups on 148 CTAs
])
@pytest.mark.parametrize("growing", [False, True])
def test_many_contributors(T, Hq, Hkv, D, lens, n_layers, growing):
    _check(T, Hq, Hkv, D, lens, n_layers, growing)
