"""Where pieces are made longer than they need be (whole items, pieces that no team begins anew within its run), weights have as many
second terms as the shorter pieces would have had: the error of the shorter ones is the bound.

R: one rounding to bf16, of the outputs; the weights' is another one in the groups with a single term."""
import pytest
import torch

from oracle import reference as ref
from paper_2603_03383_b200 import synth
from tests._cases import make_tree
from tests.test_gpu_attention_precision import DEV, R, _step_attention

pytestmark = pytest.mark.gpu


# share: of the groups of the shorter pieces that have two terms; 4 % for the sample (170 k outputs and more) and for the outputs' distribution
@pytest.mark.parametrize("T,Hq,Hkv,lens,n_layers,share", [
    (16, 4, 1, [1150] * 2, 21, 1.0),       # whole items of ten groups for pieces of four, four and two: a share of .85 by themselves
    (17, 4, 2, [1355] * 2, 11, .97),       # eleven groups: .76
    (20, 4, 1, [1265] * 3, 22, .73),       # eleven groups: .57
])
def test_longer_pieces_have_the_error_of_shorter_ones(T, Hq, Hkv, lens, n_layers, share):
    D = 128
    tb, tree = make_tree("rank_prior", 4, (), T)
    B, Lcap = len(lens), max(lens) + T + 3
    ks, vs = ([synth.normal_bf16(T, s + l, (B, Hkv, Lcap, D), device=DEV) for l in range(n_layers)] for s in (10, 50))
    q = synth.normal_bf16(T, 90, (n_layers, B, T, Hq, D), device=DEV)
    want = torch.stack([ref.tree_attention(q[l].cpu(), ks[l].cpu(), vs[l].cpu(), torch.tensor(lens, dtype=torch.int32), tb["mask"]).double()
                        for l in range(n_layers)])
    out = _step_attention(tree, q, ks, vs, lens, Hkv, D, Lcap)
    err = ((out.cpu().double() - want).norm() / want.norm()).item()
    assert err <= 1.04 * R * (2 - share) ** 0.5, err
