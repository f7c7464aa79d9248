"""Scores far above those of a piece's first group, in every part of a group's columns, and scores that are not numbers."""
import math

import pytest
import torch

from oracle import reference as ref
from paper_2603_03383_b200 import binding, synth
from tests._cases import assert_close, make_tree, workspace
from tests.test_gpu_attention_precision import _step_attention

pytestmark = pytest.mark.gpu
DEV = "cuda"
T, G = 29, 4


def _problem(D, B, Hkv, n_layers, L):
    """Queries along the first coordinate, so that a key's first element alone sets its score in every row."""
    q = torch.zeros(n_layers, B, T, Hkv * G, D, dtype=torch.bfloat16, device=DEV)
    q[..., 0] = 16.0
    ks, vs = ([synth.normal_bf16(T, s + l, (B, Hkv, L + T + 5, D), device=DEV) for l in range(n_layers)] for s in (10, 50))
    return q, ks, vs


def _run(tree, q, ks, vs, lens, Hkv, D, Lcap, step):
    if step:
        return _step_attention(tree, q, ks, vs, lens, Hkv, D, Lcap)
    out = torch.full_like(q, 9.0)
    ws = workspace(tree, len(lens), 0, 0, Hkv * G, Hkv, D, Lcap)
    sl = torch.tensor(lens, dtype=torch.int32, device=DEV)
    for l in range(q.shape[0]):
        binding.tree_verify_attention(tree, q[l], ks[l], vs[l], sl, out[l], ws)
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0
    return out


@pytest.mark.parametrize("D,step,B,Hkv,n_layers", [(64, True, 2, 8, 12), (128, True, 2, 8, 12), (64, False, 8, 16, 2), (128, False, 8, 16, 1)])
@pytest.mark.parametrize("column", [3, 12, 13, 14, 15, 31, 47, 62, 127])
def test_a_key_that_leads_by_far(D, step, B, Hkv, n_layers, column):
    """One key per item leads everything before it by 90 to 390 powers of two; the items are cut, so that most of these keys
    are not in their piece's first group."""
    tb, tree = make_tree("cartesian", 3, (4, 2, 2))
    L = 1100
    q, ks, vs = _problem(D, B, Hkv, n_layers, L)
    leads = [90.0, 120.0, 126.0] + [127.0 + 0.37 * i for i in range(9)] + [140.0, 170.0, 200.0, 255.0, 256.5, 300.0, 340.0, 383.0, 390.0]
    i = 0
    for l in range(n_layers):
        for b in range(B):
            for g in range(Hkv):
                x = leads[i % len(leads)] + 6.0            # the other scores reach about 6 above 0
                ks[l][b, g, 128 * (2 + i % 6) + column, 0] = x * math.log(2.0) * D ** 0.5 / 16.0
                i += 1
    lens = [L] * B
    want = [ref.tree_attention(q[l].cpu(), ks[l].cpu(), vs[l].cpu(), torch.tensor(lens, dtype=torch.int32), tb["mask"]) for l in range(n_layers)]
    out = _run(tree, q, ks, vs, lens, Hkv, D, L + T + 5, step)
    for l in range(n_layers):
        assert_close(out[l], want[l], "layer %d" % l)


@pytest.mark.parametrize("D,step", [(64, True), (128, True), (64, False)])
@pytest.mark.parametrize("bad", [math.nan, math.inf])
@pytest.mark.parametrize("row", [14, 128 * 5 + 3, 128 * 5 + 13])
def test_scores_that_are_not_numbers(D, step, bad, row):
    """A key of NaN, or one whose scores are +inf (inf - inf against the maximum), makes the rows that see it NaN and no others."""
    tb, tree = make_tree("cartesian", 3, (4, 2, 2))
    L, B, Hkv, n_layers = 1100, 2, 8, 6
    q, ks, vs = _problem(D, B, Hkv, n_layers, L)
    q[..., 1:] = 0.0
    ks[2][1, 3, row, 0] = bad
    out = _run(tree, q, ks, vs, [L] * B, Hkv, D, L + T + 5, step)
    hit = torch.zeros_like(out, dtype=torch.bool)
    hit[2, 1, :, 3 * G:4 * G] = True
    assert out[hit].isnan().all() and out[~hit].isfinite().all()
