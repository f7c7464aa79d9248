"""Equal logits in the slabs of many CTAs: every weight row of a small vocabulary is there many times over, and of equal ones the lowest
id comes first, however the lists are merged (few or many candidates, one or many rows)."""
import pytest
import torch

from oracle import reference as ref
from paper_2603_03383_b200 import binding, synth
from tests._cases import MARGIN, make_tree, workspace

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,H", [(1, 64), (1, 72), (2, 72), (5, 64), (13, 64), (16, 64)])
@pytest.mark.parametrize("topk", [(1,), (2,), (3,), (16,), (1, 2), (2, 1, 3), (4, 1, 2, 1)])
def test_equal_logits(B, H, topk):
    K, V0, copies = len(topk), 61, 40
    tb, tree = make_tree("cartesian", K, topk)
    for seed in range(90, 20090, 1000):
        hidden, W1, b1, W2, root = synth.head_inputs(B, H, V0, K, seed)
        z = ref.heads_logits(hidden, W1, b1, W2).transpose(0, 1)     # [B][K][V0] in 64 bits
        best, rows = z.sort(dim=-1, descending=True)
        if (best[..., :2] - best[..., 1:3]).min() > MARGIN * z.abs().max():
            break
    want = torch.full((B, tree.C), -1, dtype=torch.int64)
    want[:, 0] = root
    for k in range(K):
        for s in range(tree.k_d[k]):                            # at most 16 <= copies: all of the best row
            want[:, tree.cand_offset[k] + s] = rows[:, k, s // copies] + s % copies * V0
    cand = torch.full((B, tree.C), -7, dtype=torch.int32, device=DEV)
    tt = torch.full((B, tree.T), -7, dtype=torch.int32, device=DEV)
    W = W2.repeat(1, copies, 1).contiguous().to(DEV)
    hidden, W1, b1, root = (t.to(DEV) for t in (hidden, W1, b1, root))
    binding.medusa_heads_topk(tree, hidden, W1, b1, W, root, cand, None, tt, workspace(tree, B, H, V0 * copies, 0, 0, 0, 0))
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    assert torch.equal(cand.long().cpu(), want)
    assert torch.equal(tt.long().cpu(), want[:, torch.tensor(tree.tree_indices)])
