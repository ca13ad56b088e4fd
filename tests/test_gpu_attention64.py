"""The kernel of row blocks of at most 64 query rows (two score buffers, K and
V in a ring of five, a warp without rows when there are at most 32): tile
counts around the ring and the buffers, row counts around a warp, every page
size, whole units, ranges merged in a cluster and through the workspace, with
and without rotation.  Oracle, tolerance and derived bound as in
test_gpu_attention.py."""
import pytest
import torch

from paper_2606_02544_gb300 import inputs
from tests._gpu import assert_attention_close, gpu_attention, oracle_attention
from tests.test_gpu_rope import _rope_check, _w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma,Hq,Hkv", [(1, 4, 4), (16, 8, 8), (17, 8, 8), (32, 4, 4), (8, 32, 8), (4, 8, 1),
                                          (5, 12, 2)])
@pytest.mark.parametrize("P,prefix", [(64, [0, 64, 65, 128, 190]), (16, [300, 321]), (8, [70, 1]), (192, [500, 192])])
def test_rows_and_tiles(gamma, Hq, Hkv, P, prefix):
    w = _w(Bt=len(prefix), Hq=Hq, Hkv=Hkv, gamma=gamma, P=P, seed=gamma + P)
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=prefix, random_step_map=True,
                                 poison_unused_rows=True)
    out, word, _ = gpu_attention(si)
    ref = oracle_attention(si)
    assert word == ref.err == 0
    assert_attention_close(out, ref)
    _rope_check(si, 1e6)


@pytest.mark.parametrize("Bt,gamma,hi", [(40, 3, 700), (90, 8, 400)])
def test_whole_units_in_one_and_several_waves(Bt, gamma, hi):
    g = torch.Generator().manual_seed(Bt)
    prefix = torch.randint(0, hi, (Bt,), generator=g).tolist()
    w = _w(Bt=Bt, Hq=32, Hkv=8, gamma=gamma, seed=Bt)
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=prefix, random_step_map=True,
                                 poison_unused_rows=True)
    seqs = list(range(0, Bt, 9))
    out, word, ws = gpu_attention(si)
    ref = oracle_attention(si, seqs=seqs)
    assert word == ref.err == 0 and ws == 0
    assert_attention_close(out[torch.as_tensor(seqs, device=out.device)], ref)


def test_growing_scores_across_two_buffers():
    # later keys score higher: the running maximum rises past the rescale
    # threshold many times while the next tile's scores are already there
    w = _w(Bt=1, Hq=8, Hkv=1, gamma=4, seed=2)
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=[1500])
    q = si.q[0, 0].float().mean(dim=(0, 1))
    si.q[0, 0] = q.to(si.q.dtype)
    n, P = 1500, 64
    ramp = torch.linspace(0, 900, n, device="cuda")
    for j in range(0, n, P):
        page = int(si.block_table[0, j // P])
        rows = min(P, n - j)
        si.k_cache[0, page, 0, :rows] = (ramp[j:j + rows, None] * q / q.square().sum()).to(si.q.dtype)
    out, word, _ = gpu_attention(si)
    ref = oracle_attention(si)
    assert word == ref.err == 0
    assert_attention_close(out, ref)
