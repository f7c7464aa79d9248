"""Tree attention where a piece's groups meet the three tiles of scores in every way, items of every number of row tiles, and
references that move in every group of a piece, in some rows of a tile only and in neighbouring groups at once."""
import math

import pytest
import torch

from oracle import reference as ref
from paper_2603_03383_b200 import binding, synth
from tests._cases import assert_close, make_tree, workspace
from tests.test_gpu_attention_precision import _step_attention
from tests.test_gpu_attention_range import _run

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _inputs(tb_T, n_layers, B, Hq, Hkv, D, Lcap):
    ks, vs = ([synth.normal_bf16(tb_T, s + l, (B, Hkv, Lcap, D), device=DEV) for l in range(n_layers)] for s in (10, 50))
    return synth.normal_bf16(tb_T, 90, (n_layers, B, tb_T, Hq, D), device=DEV), ks, vs


def _want(q, ks, vs, lens, tb):      # before the step: its compaction moves rows of the caches
    return [ref.tree_attention(q[l].cpu(), ks[l].cpu(), vs[l].cpu(), torch.tensor(lens, dtype=torch.int32), tb["mask"]) for l in range(q.shape[0])]


# groups per item: 1 to 8 and their last ones full, nearly empty and off the multiples of 16 keys
@pytest.mark.parametrize("T,Hq,Hkv,D", [
    (64, 8, 2, 128),     # two row tiles: one pair of CTAs
    (33, 8, 2, 128),     # the second one nearly empty
    (80, 8, 1, 128),     # five row tiles: the last pair has one
    (96, 4, 1, 128),     # three
    (128, 7, 1, 128),    # eight, of 18 nodes each
    (20, 4, 1, 128),     # one
    (128, 2, 1, 64),     # two, head size 64
    (50, 5, 1, 64),      # two of 25 nodes
])
@pytest.mark.parametrize("n_layers", [1, 9])
def test_groups_and_row_tiles(T, Hq, Hkv, D, n_layers):
    tb, tree = make_tree("rank_prior", 4, (), T)
    lens = [max(0, 128 * g - T - d) for g in range(1, 9) for d in (0, 1, 37)][n_layers % 2::3] + [0]
    q, ks, vs = _inputs(T, n_layers, len(lens), Hq, Hkv, D, max(lens) + T + 3)
    want = _want(q, ks, vs, lens, tb)
    out = _step_attention(tree, q, ks, vs, lens, Hkv, D, max(lens) + T + 3)
    for l in range(n_layers):
        assert_close(out[l], want[l], "layer %d" % l)


@pytest.mark.parametrize("T,G,D,step", [(64, 4, 128, True), (64, 4, 64, True), (29, 4, 128, True), (64, 4, 128, False), (64, 2, 64, False)])
@pytest.mark.parametrize("column", [0, 31, 32, 70, 127])
def test_references_move_in_any_group(T, G, D, step, column):
    """Every item has keys that lead all before them by 35 to 300 powers of two, in one of its groups, in the next one and, by
    more, two groups on, in other columns; only some rows see them lead."""
    tb, tree = make_tree("rank_prior", 4, (), T)
    B, Hkv, n_layers, L = 2, 8, 6 if step else 1, 1200
    q, ks, vs = _inputs(T, n_layers, B, Hkv * G, Hkv, D, L + T + 5)
    q *= 0.25
    q[..., 0] = 0.5
    q[:, :, ::5, :, 0] = 16.0
    q[:, :, 3::7, :, 0] = 16.0
    unit = math.log(2.0) * D ** 0.5 / 16.0
    i = 0
    for l in range(n_layers):
        ks[l][..., 0] *= 0.1
        for b in range(B):
            for g in range(Hkv):
                first = i % 10                       # of ten groups; the last keys may lie among the tree's rows
                for k, (lead, c) in enumerate([(35.0 + 3 * i % 90, column), (130.0 + i % 40, (column + 33) % 128), (300.0, (column + 64) % 128)]):
                    row = 128 * (first + k) + c
                    if row < L + 1:                  # (row L is the root, which every node sees)
                        ks[l][b, g, row, 0] = lead * unit
                i += 1
    want = _want(q, ks, vs, [L] * B, tb)
    out = _run(tree, q, ks, vs, [L] * B, Hkv, D, L + T + 5, step)
    for l in range(n_layers):
        assert_close(out[l], want[l], "layer %d" % l)


@pytest.mark.parametrize("D,Hkv,B", [(64, 2, 3), (128, 4, 12), (64, 1, 40)])      # (more than 32 sequences are divided in several turns)
def test_lengths_that_the_kernel_in_front_advances(D, Hkv, B):
    """A one-layer call right behind the compaction that advances the lengths, from one number of groups to another."""
    tb, tree = make_tree("rank_prior", 4, (), 64)
    T, K, Hq = 64, 4, Hkv * 4
    lens = [(128 * (2 + b % 5) - T - (b % 4)) for b in range(B)]
    alen = [b % (K + 1) for b in range(B)]
    Lcap, top = max(lens) + 8200, max(lens) + K + 1 + T      # (at head size 128 a call with room for long prefixes)
    k, v = (synth.normal_bf16(T, s, (B, Hkv, Lcap, D), device=DEV) for s in (10, 50))
    q = synth.normal_bf16(T, 90, (B, T, Hq, D), device=DEV)
    nodes = torch.tensor([[0] + [j if j <= n else -1 for j in range(1, K + 1)] for n in alen], dtype=torch.int32, device=DEV)   # (rows stay where they are)
    sl, status = torch.tensor(lens, dtype=torch.int32, device=DEV), torch.zeros(B, dtype=torch.int32, device=DEV)
    after = [L + n + 1 for L, n in zip(lens, alen)]
    want = ref.tree_attention(q.cpu(), k[:, :, :top].cpu(), v[:, :, :top].cpu(), torch.tensor(after, dtype=torch.int32), tb["mask"])
    kp, vp = binding.cache_pointer_array([k], DEV), binding.cache_pointer_array([v], DEV)
    ws, out = workspace(tree, B, 0, 0, Hq, Hkv, D, Lcap), torch.full_like(q, 9.0)
    accept = torch.tensor(alen, dtype=torch.int32, device=DEV)
    binding.kv_compact_accepted(tree, kp, vp, 1, B, Hkv, D, k.stride()[:3], Lcap, sl, accept, nodes, status=status)
    binding.tree_verify_attention(tree, q, k, v, sl, out, ws, status=status)
    torch.cuda.synchronize()
    assert binding.mtv_device_error(tree) == 0 and sl.tolist() == after and status.tolist() == [0] * B
    assert_close(out, want)


@pytest.mark.parametrize("T,bad,B", [
    (64, [2**31 - 4, -64, -65, -500, -2**31, 2**31 - 64], 10),     # sums with T that wrap, or leave no key
    (29, [-29, 3000, 2**31 - 1], 40),                            # more than 32 sequences
])
def test_lengths_that_leave_no_keys(T, bad, B):
    """Such a sequence is reported and passed over, and the others' share of the work does not depend on it."""
    tb, tree = make_tree("rank_prior", 4, (), T)
    Hq, Hkv, D, Lcap = 8, 2, 64, 1000
    lens = [17 * b + 1 for b in range(B)]
    for i, x in enumerate(bad):
        lens[(3 * i + 1) % B] = x
    good = [b for b in range(B) if 0 <= lens[b] <= Lcap - T]
    k, v = (synth.normal_bf16(T, s, (B, Hkv, Lcap, D), device=DEV) for s in (10, 50))
    q = synth.normal_bf16(T, 90, (B, T, Hq, D), device=DEV)
    want = ref.tree_attention(q[good].cpu(), k[good].cpu(), v[good].cpu(), torch.tensor([lens[b] for b in good], dtype=torch.int32), tb["mask"])
    sl, status = torch.tensor(lens, dtype=torch.int32, device=DEV), torch.full((B,), 7, dtype=torch.int32, device=DEV)
    out, ws = torch.full_like(q, 9.0), workspace(tree, B, 0, 0, Hq, Hkv, D, Lcap)
    for _ in range(2):       # (counters are back at zero behind the first call)
        binding.tree_verify_attention(tree, q, k, v, sl, out, ws, status=status)
        torch.cuda.synchronize()
        assert binding.mtv_device_error(tree) == 0
        assert status.tolist() == [0 if b in good else binding.MTV_ERR_CAPACITY for b in range(B)]
        assert_close(out[good], want)
        assert all((out[b] == 9.0).all() for b in range(B) if b not in good)
