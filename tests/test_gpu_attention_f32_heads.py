"""fp32 attention with more KV heads than the second and third dimensions of
a grid take (65535): the call was always accepted.  Tolerance of the fp32
path as in test_gpu_attention.py."""
import pytest

from paper_2606_02544_gb300 import inputs
from tests._gpu import assert_attention_close, gpu_attention, oracle_attention
from tests.test_gpu_attention import _w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hkv", [65535, 65537])
def test_many_kv_heads(Hkv):
    w = _w("f32", Bt=2, Hq=Hkv, Hkv=Hkv, d=64, gamma=1, P=8)
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=[3, 9], random_step_map=True)
    out, word, _ = gpu_attention(si)
    ref = oracle_attention(si)
    assert word == ref.err == 0
    assert_attention_close(out, ref)
