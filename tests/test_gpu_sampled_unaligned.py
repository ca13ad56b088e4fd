"""Stochastic acceptance over rows that start off the 16-byte grid.  Every
vocabulary remainder and base shift, with values around the rows that would
change the sums or the draw if they were read, spans on both sides of the line
between 8 and 16 scalar loads at a time; decisions and tokens by the
oracle outside the fp32 band, as in test_gpu_accept_sampled.py, through the
cluster kernel and the split one."""
import dataclasses

import pytest
import torch

from paper_2606_02544_gb300 import inputs
from tests import test_gpu_accept_sampled as base
from tests.test_gpu_accept_sampled_ws import _gpu_ws

pytestmark = pytest.mark.gpu


def _shifted(t, shift):
    flat = torch.full((t.numel() + 8,), 200.0, device="cuda")
    flat[4 + shift:4 + shift + t.numel()] = t.reshape(-1)
    return flat[4 + shift:4 + shift + t.numel()].view(t.shape)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("Bt,gamma,V", [(3, 2, 5), (2, 3, 127), (6, 4, 30001), (2, 8, 50002), (1, 16, 50003),
                                        (3, 4, 1024), (2, 1, 2), (8, 20, 50001), (24, 4, 65537)])
def test_row_ends(monkeypatch, Bt, gamma, V, shift):
    si = inputs.make_sampled_inputs(Bt, gamma, V, seed=V + shift, device="cuda")
    # heavy first and last columns: drafts and draws fall on the rows' ends
    si.target_logits[:, :, 0] += 6.0
    si.target_logits[:, :, V - 1] += 7.0
    si.draft_logits[:, :, V - 1] += 6.0
    si = dataclasses.replace(si, target_logits=_shifted(si.target_logits, shift),
                             draft_logits=_shifted(si.draft_logits, (shift + 1) % 4))
    base._compare(si)
    monkeypatch.setattr(base, "_gpu", _gpu_ws)  # (few long sequences: split over many CTAs)
    base._compare(si)
