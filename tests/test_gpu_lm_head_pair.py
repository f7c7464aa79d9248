"""The LM head on CTA pairs (more than 128 nodes) at the sizes where its division of the work can go wrong."""
import pytest

from paper_2603_03383_b200 import synth
from tests._cases import make_tree
from tests.test_gpu_lm_head import _check, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,V", [
    (3, 43, 64, 5),              # 129 nodes: one pass of 160; one column chunk; fewer vocabulary rows than a tile
    (4, 64, 128, 256),           # 256 nodes: one full pass, one full tile
    (1 + 256 // 43, 43, 192, 257),   # 301 nodes: two passes of 160; a tile of a single row
    (16, 128, 64, 9000),         # 2048 nodes: eight passes, the most of one launch
    (33, 64, 64, 1100),          # 2112 nodes: a second launch of 64
    (3, 100, 704, 37000),        # more items than pairs
])
def test_lm_head_pairs(B, T, H, V):
    tb, tree = make_tree("rank_prior", 4, (), T)
    x = synth.normal_bf16(21, B + H, (B, T, H))
    W = synth.normal_bf16(21, 1000 + V, (V, H))
    keys, am, val = _run(tree, x, W)
    _check(x, W, am, val)
