"""Items that many CTAs share, on either side of the count from which their partial results are combined by several lanes to a chunk.

All cases have two layers: a call for one layer may take another kernel.  The bounds-checking build waits for nobody, so that there
slices are left to the last CTA of an item, which has to sum them as their own CTAs would have: the same bits in both builds."""
import hashlib
import os
import subprocess
import sys

import pytest

from paper_2603_03383_b200 import build
from tests import test_gpu_attention_runs as runs

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# (one group of 128 keys, tree rows among them, to a contributor)
CASES = [
    (64, 4, 1, 128, [3700]),      # pairs: 30 contributors, five rows each, four lanes to a chunk
    (64, 4, 1, 128, [3100]),      # 25: six rows, the most
    (64, 4, 1, 128, [3000]),      # 24: one lane to a chunk
    (47, 1, 1, 128, [3500]),      # a single row tile, 28
    (30, 4, 1, 128, [3100]),      # 25
    (30, 4, 1, 128, [3000]),      # 24
    (47, 1, 1, 128, [6900]),      # 55: three rows, eight lanes to a chunk
    (61, 2, 1, 64, [3100]),       # head size 64: 25
    (61, 2, 1, 64, [3000]),       # 24
]


@pytest.mark.parametrize("T,Hq,Hkv,D,lens", CASES)
@pytest.mark.parametrize("growing", [False, True])
def test_contributors(T, Hq, Hkv, D, lens, growing):
    runs._check(T, Hq, Hkv, D, lens, 2, growing)


def _digests():
    """Of the outputs of all cases with more than 24 contributors (assert_close is handed each layer's)."""
    seen = []
    keep, runs.assert_close = runs.assert_close, lambda got, want, what: seen.append(got.clone())
    try:
        for T, Hq, Hkv, D, lens in CASES:
            if lens[0] > 3000:
                runs._check(T, Hq, Hkv, D, lens, 2)
    finally:
        runs.assert_close = keep
    return [hashlib.sha256(t.contiguous().view(-1).view(dtype=runs.torch.uint8).cpu().numpy().tobytes()).hexdigest() for t in seen]


def test_left_slices_have_the_same_bits():
    r = subprocess.run([sys.executable, "-c", "from tests import test_gpu_attention_contributors as t; print('\\n'.join(t._digests()))"], cwd=ROOT,
                       env=dict(os.environ, MTV_LIB=build.build(variant="debug_bounds")), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    assert r.stdout.split() == _digests()
