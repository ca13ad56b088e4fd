"""Greedy acceptance around the batches at which the cluster size steps down
(a grid with fewer than two places left takes clusters one smaller): every
number of sequences from 9 to 47, bit-exact against the oracle, with row
lengths on and off the 16-byte grid."""
import pytest

from tests.test_gpu_accept_ws import _run_ws
from tests.test_gpu_mask_accept import _accept_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [64, 203])
@pytest.mark.parametrize("Bt", list(range(9, 48)))
def test_batches(Bt, V):
    logits, draft = _accept_case(Bt, 3, V, seed=Bt + V)
    _run_ws(logits, draft)
