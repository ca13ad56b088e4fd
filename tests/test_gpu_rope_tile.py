"""The RoPE prologue laid out by angle (16 threads a slot, its g query rows
and its new key together): group sizes that do not divide a warp, slot counts
that leave threads idle or go round more than once, units whose query rows
fill two row blocks only in part, and a split prefix whose later ranges hold
no new key.  Oracle, tolerance and derived bound as in test_gpu_rope.py."""
import pytest

from paper_2606_02544_gb300 import inputs
from tests.test_gpu_rope import _rope_check, _w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma,Hq,Hkv,prefix", [
    (1, 8, 8, [3, 64]),          # 2 slots, one query row each
    (32, 8, 8, [1, 700]),        # 64 slots of one row: several rounds
    (5, 24, 8, [0, 130]),        # g = 3
    (9, 7, 1, [50, 2000]),       # g = 7: 126 rows
    (31, 32, 8, [0, 100, 1500]),  # 248 rows: the second row block partly empty
    (12, 64, 8, [900, 65]),      # g = 8: 24 slots over blocks of 16
    (32, 32, 8, [4000, 3000]),   # ranges without new keys
])
def test_bf16_rope_slots(gamma, Hq, Hkv, prefix):
    w = _w(Bt=len(prefix), Hq=Hq, Hkv=Hkv, gamma=gamma, seed=gamma + Hq)
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=prefix, random_step_map=True,
                                 poison_unused_rows=True)
    _rope_check(si, 1e6)
