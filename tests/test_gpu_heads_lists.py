"""Candidate lists of the vocabulary projection where they fill, overflow and tie: slabs of one row to many tiles, top-k of 1
to 16, rising logits (every row enters the list) and falling ones (none does after the first)."""
import pytest
import torch

from oracle import reference as ref
from paper_2603_03383_b200 import binding
from tests._cases import make_tree, workspace

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B", [1, 2, 16])
@pytest.mark.parametrize("V,topk", [(17, (16,)), (149, (1, 16)), (5000, (7, 16)), (40000, (16,)), (9473, (2, 3, 1, 2, 2))])
@pytest.mark.parametrize("order", ["rising", "falling", "ties"])
def test_lists(B, V, topk, order):
    H, K = 64, len(topk)
    tb, tree = make_tree("cartesian", K, topk)
    g = torch.Generator().manual_seed(V)
    hidden = torch.zeros(B, H, dtype=torch.bfloat16)
    hidden[:, 0] = torch.arange(1, B + 1).to(torch.bfloat16)
    W1 = torch.zeros(K, H, H, dtype=torch.bfloat16)                       # h' = hidden: logits are set through W2
    W2 = torch.zeros(K, V, H, dtype=torch.bfloat16)
    steps = torch.arange(V).float()
    if order == "falling":
        steps = steps.flip(0)
    if order == "ties":
        steps = torch.randint(0, 7, (V,), generator=g).float() * 256
    W2[:, :, 0] = (steps // 256).to(torch.bfloat16)                       # exact in bf16: value = 256 hi + lo
    W2[:, :, 1] = (steps % 256).to(torch.bfloat16)
    hidden[:, 1] = hidden[:, 0] / 256
    root = torch.zeros(B, dtype=torch.int32)
    z = ref.heads_logits(hidden, W1, None, W2)
    cand_ref, _, tt_ref, _ = ref.heads_candidates(z, root, tb)
    ws = workspace(tree, B, H, V, 0, 0, 0, 0)
    cand = torch.zeros(B, tree.C, dtype=torch.int32, device=DEV)
    tt = torch.zeros(B, tree.T, dtype=torch.int32, device=DEV)
    binding.medusa_heads_topk(tree, hidden.to(DEV), W1.to(DEV), None, W2.to(DEV), root.to(DEV), cand, None, tt, ws)
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    assert torch.equal(cand.cpu(), cand_ref) and torch.equal(tt.cpu(), tt_ref)


@pytest.mark.parametrize("H,V", [(8, 3000), (1000, 700), (1024, 20000), (2040, 9000), (16384, 77)])
def test_stage_heights(H, V):
    """One batch row: stages of 32, 16, 8 rows and, for long rows, fewer rows than warps."""
    K = 2
    tb, tree = make_tree("cartesian", K, (5, 4))
    from tests._cases import oracle_heads_with_margin
    seed, inp, _, cand_ref, cl_ref, tt_ref = oracle_heads_with_margin(1, H, V, K, tb, 50 + H)
    hidden, W1, b1, W2, root = [t.to(DEV) for t in inp]
    ws = workspace(tree, 1, H, V, 0, 0, 0, 0)
    cand = torch.zeros(1, tree.C, dtype=torch.int32, device=DEV)
    cl, tt = torch.zeros(1, tree.C - 1, device=DEV), torch.zeros(1, tree.T, dtype=torch.int32, device=DEV)
    binding.medusa_heads_topk(tree, hidden, W1, b1, W2, root, cand, cl, tt, ws)
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    assert torch.equal(cand.cpu(), cand_ref) and torch.equal(tt.cpu(), tt_ref)
    assert (cl.double().cpu() - cl_ref).abs().max().item() <= 2e-5 * cl_ref.abs().max().item()


@pytest.mark.parametrize("B,H", [(1, 64), (13, 64), (16, 64), (16, 72)])
@pytest.mark.parametrize("topk", [(2,), (1, 1), (3, 2)])
def test_more_rows_than_nodes(B, H, topk):
    """The root's token in every row's candidates and tree, also where a tree has fewer nodes than there are rows."""
    V, K = 900, len(topk)
    tb, tree = make_tree("cartesian", K, topk)
    from tests._cases import oracle_heads_with_margin
    _, inp, _, cand_ref, _, tt_ref = oracle_heads_with_margin(B, H, V, K, tb, 70 + B)
    hidden, W1, b1, W2, root = [t.to(DEV) for t in inp]
    cand = torch.full((B, tree.C), -7, dtype=torch.int32, device=DEV)
    tt = torch.full((B, tree.T), -7, dtype=torch.int32, device=DEV)
    binding.medusa_heads_topk(tree, hidden, W1, b1, W2, root, cand, None, tt, workspace(tree, B, H, V, 0, 0, 0, 0))
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    assert torch.equal(cand.cpu(), cand_ref) and torch.equal(tt.cpu(), tt_ref)
