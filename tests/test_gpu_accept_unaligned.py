"""Greedy acceptance over rows that start off the 16-byte grid: 16-byte units
laid over the whole block, so that a unit may hold the end of one row and the
start of the next, and the first and last unit reach past it.  Maxima, ties
and NaNs are planted at the rows' ends; bit-exact against the oracle, for
every shift of the base, through the cluster kernel and the split one."""
import numpy as np
import pytest
import torch

from tests.test_gpu_accept_ws import _run_ws
from tests.test_gpu_mask_accept import _accept_case

pytestmark = pytest.mark.gpu


def _shifted(t, shift):
    # values around the block that would win every row if they were read
    flat = torch.full((t.numel() + 8,), float("inf"), device="cuda")
    flat[4 + shift:4 + shift + t.numel()] = t.reshape(-1)
    return flat[4 + shift:4 + shift + t.numel()].view(t.shape)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("Bt,gamma,V", [(3, 2, 1), (2, 4, 2), (2, 3, 3), (5, 4, 5), (3, 7, 4099), (20, 2, 2050),
                                        (2, 8, 50001), (1, 16, 151935), (2, 3, 1024)])
def test_row_ends(Bt, gamma, V, shift):
    logits, draft = _accept_case(Bt, gamma, V, seed=V + gamma + shift)
    ends = np.random.default_rng(shift).integers(0, 6, (Bt, gamma + 1))
    for b in range(Bt):
        for r in range(gamma + 1):
            if ends[b, r] == 0:
                logits[b, r, V - 1] = 60.0
            elif ends[b, r] == 1:
                logits[b, r, 0] = 60.0
            elif ends[b, r] == 2:
                logits[b, r, 0] = logits[b, r, V - 1] = 60.0
            elif ends[b, r] == 3:
                logits[b, r, V - 1] = float("nan")
            elif ends[b, r] == 4:
                logits[b, r] = -float("inf")
    _run_ws(_shifted(logits, shift), draft)
