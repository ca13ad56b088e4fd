"""The kernel of 65 to 128 query rows a KV head: 1, 2, 3 and more tiles a CTA
(S of the next tile is issued ahead of the commits, and the epilogue must
wait for the last PV whatever the number of tiles), whole units, ranges
through the workspace and ranges merged in a cluster, small pages, and scores
that pass the rescale threshold.  Oracle, tolerance and derived bound as in
test_gpu_attention.py; the same call again gives the same bits."""
import pytest
import torch

from paper_2606_02544_gb300 import inputs, simsd
from tests._gpu import assert_attention_close, gpu_attention, oracle_attention
from tests.test_gpu_attention import _w

pytestmark = pytest.mark.gpu

ROWS = [(16, 32, 8), (9, 32, 8), (11, 6, 2), (7, 36, 4)]  # 128, 72, 66 and 126 rows


def _check(si, seqs=None):
    plan = simsd.simsd_plan_attention(simsd.SIMSD_BF16, si.w.Bt, si.w.gamma, si.w.Hq, si.w.Hkv, si.w.d,
                                      si.block_table.shape[1], si.w.page_size, 152)
    assert plan["kernel"] == 0 and 64 < plan["rows_blk"] <= 128
    out, word, ws = gpu_attention(si)
    ref = oracle_attention(si, seqs=seqs)
    assert word == ref.err == 0
    assert_attention_close(out if seqs is None else out[torch.as_tensor(seqs, device=out.device)], ref)
    for _ in range(5):
        again, word, _ = gpu_attention(si)
        assert word == 0 and torch.equal(again, out)
    return ws


@pytest.mark.parametrize("P", [64, 16])
@pytest.mark.parametrize("gamma,Hq,Hkv", ROWS)
def test_whole_units(gamma, Hq, Hkv, P):
    w = _w(Bt=320 // Hkv, Hq=Hq, Hkv=Hkv, gamma=gamma, P=P, seed=gamma + P)
    lens = [(0, 1, 64, 65, 128, 130, 700)[i % 7] for i in range(w.Bt)]
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=lens, random_step_map=True,
                                 poison_unused_rows=True)
    assert _check(si, seqs=list(range(7))) == 0


@pytest.mark.parametrize("P", [64, 16])
@pytest.mark.parametrize("prefix,through_workspace", [([1500], True), ([3000, 70], True), ([450], False),
                                                      ([1500, 0, 64, 500, 1000], False)])
@pytest.mark.parametrize("gamma,Hq", [(16, 32), (9, 32)])
def test_ranges(gamma, Hq, prefix, through_workspace, P):
    w = _w(Bt=len(prefix), Hq=Hq, Hkv=8, gamma=gamma, P=P, seed=gamma)
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=prefix, random_step_map=True,
                                 poison_unused_rows=True)
    assert (_check(si) > 0) == through_workspace


@pytest.mark.parametrize("Bt", [1, 40])
def test_growing_scores(Bt):
    # later keys score higher: the running maximum rises past the rescale
    # threshold many times
    w = _w(Bt=Bt, Hq=32, Hkv=8, gamma=16, seed=2)
    n, P = 900, 64
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=[n] * Bt)
    ramp = torch.linspace(0, 900, n, device="cuda")
    for h in range(8):
        q = si.q[0, 0, :, 4 * h:4 * h + 4].float().mean(dim=(0, 1))
        si.q[0, 0, :, 4 * h:4 * h + 4] = q.to(si.q.dtype)
        for j in range(0, n, P):
            rows = min(P, n - j)
            si.k_cache[0, int(si.block_table[0, j // P]), h, :rows] = (
                ramp[j:j + rows, None] * q / q.square().sum()).to(si.q.dtype)
    _check(si, seqs=[0])
