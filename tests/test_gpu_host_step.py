"""The host-buffer step where its order of work branches: one head (none runs in front of the attention), fewer layers than
groups, more groups than two, and host buffers that are not pinned."""
import pytest
import torch

from tests.test_gpu_parity import _step_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,n_layers,B", [(1, 1, 1), (1, 3, 2), (3, 9, 1)])
@pytest.mark.parametrize("pinned", [True, False])
def test_host_step_orders(K, n_layers, B, pinned, monkeypatch):
    if not pinned:
        monkeypatch.setattr(torch.Tensor, "pin_memory", lambda self: self)
    topk = (5,) if K == 1 else (3, 2, 1)
    _step_case(B, 256, 900, 8, 2, 128, n_layers, "cartesian", K, topk, 0, [70, 131][:B], seed=9, host=True)
