"""How far the attention's outputs are from 64 bits, as the 2-norm of the error over the 2-norm of the result.

One rounding to bf16 with random mantissas is an error of R = 2^-8 / sqrt(3) * sqrt(E[2^2e] / E[x^2]) per element, 2^e <= |x| the
power of two below: 0.00166 for normally distributed outputs.  The weights are rounded to bf16 before they meet V: another
R, independent of it, unless the weights are carried in two terms.  Everything else is fp32 (below 1e-5)."""
import pytest
import torch

from oracle import reference as ref
from paper_2603_03383_b200 import binding, synth
from tests._cases import make_tree, workspace

pytestmark = pytest.mark.gpu
DEV = "cuda"
R = 0.00166


def _step_attention(tree, q, ks, vs, lens, Hkv, D, Lcap):
    """The attention of all layers inside mtv_verify_step (tiny heads and vocabulary beside it)."""
    n_layers, B, T, Hq, _ = q.shape
    K, H, V = tree.K, 64, 600
    hidden, W1, b1, W2, root = synth.head_inputs(B, H, V, K, seed=3, device=DEV)
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    d = dict(hidden=hidden, W1=W1, b1=b1, W2=W2, root_tok=root, q_layers=q, out_layers=torch.full_like(q, 9.0),
             logits=synth.normal_bf16(T, 91, (B, T, V), device=DEV), seq_lens=torch.tensor(lens, dtype=torch.int32, device=DEV),
             cand=i32(B, tree.C), tree_tok=i32(B, T), accept_len=i32(B), best_path=i32(B), acc_nodes=i32(B, K + 1),
             acc_tok=i32(B, K + 1), next_root=i32(B), status=i32(B),
             k_caches=binding.cache_pointer_array(ks, DEV), v_caches=binding.cache_pointer_array(vs, DEV),
             k_caches_host=binding.cache_pointer_array(ks), v_caches_host=binding.cache_pointer_array(vs),
             ws=workspace(tree, B, H, V, Hq, Hkv, D, Lcap))
    a = binding.StepArgs()
    a.B, a.H, a.V, a.Hq, a.Hkv, a.D, a.n_layers, a.Lcap = B, H, V, Hq, Hkv, D, n_layers, Lcap
    a.stride_b, a.stride_h, a.stride_t = ks[0].stride()[:3]
    for n, t in d.items():
        setattr(a, n, t.data_ptr())
    a.ws_bytes = d["ws"].numel()
    binding.mtv_verify_step(tree, a)
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    return d["out_layers"]


# bound: what the roundings of a form add up to, with 6 % for the sample (20 k to 400 k outputs) and for the outputs' distribution
@pytest.mark.parametrize("T,Hq,Hkv,D,lens,n_layers,roundings", [
    (64, 32, 8, 128, [1500] * 6, 2, 2),        # items cut anywhere: 96 of 13 groups on 148 SMs
    (64, 8, 2, 128, [3000], 4, 2),             # one item over many SMs
    (64, 8, 2, 128, [50, 64], 6, 1),           # a single group: two-term weights
    (29, 8, 2, 64, [128], 8, 1),               # head size 64: two-term weights in every group; one row tile
    (128, 16, 2, 64, [97, 2000], 2, 1),        # several row blocks, last groups of every length
    (65, 7, 1, 64, [1000], 3, 1),              # rows that belong to nobody
    # D = 128, few enough items that they stay whole or nearly so: a division among all SMs, two tiles to an SM, would make a piece of
    # every group or two, and the weights keep the second terms that its pieces would have had (one rounding and the share of keys
    # in groups with a single term; with a second term in the first group of a piece only: .0022, .0020, .0021, .0022)
    (64, 32, 8, 128, [512], 4, 1.03),           # 32 items of 5 groups on pairs
    (29, 32, 8, 128, [512], 8, 1),             # 64 items of a single row tile
    (96, 16, 4, 128, [400], 6, 1.09),           # 24 items of three row tiles
    (64, 32, 8, 128, [512], 8, 1.35),          # 64 items on 74 pairs: 65 % of the keys
])
def test_error_of_a_step(T, Hq, Hkv, D, lens, n_layers, roundings):
    tb, tree = make_tree("rank_prior", 4, (), T)
    B, Lcap = len(lens), max(lens) + T + 3
    ks, vs = ([synth.normal_bf16(T, s + l, (B, Hkv, Lcap, D), device=DEV) for l in range(n_layers)] for s in (10, 50))
    q = synth.normal_bf16(T, 90, (n_layers, B, T, Hq, D), device=DEV)
    want = [ref.tree_attention(q[l].cpu(), ks[l].cpu(), vs[l].cpu(), torch.tensor(lens, dtype=torch.int32), tb["mask"]) for l in range(n_layers)]
    out = _step_attention(tree, q, ks, vs, lens, Hkv, D, Lcap)
    want = torch.stack([w.double() for w in want])
    err = ((out.cpu().double() - want).norm() / want.norm()).item()
    assert err <= 1.06 * R * roundings ** 0.5, err
