"""The fp32 attention's bounded waits run out: the release of a K tile is made
to expect an arrival that never comes, as in test_gpu_wait_expiry.py (nothing
traps, faults or spins without a limit).  Whole units and ranges merged in a
cluster, one and several warps a CTA, with and without rotation (whose
consumers meet at a barrier after the wait has run out)."""
import time

import pytest
import torch

from paper_2606_02544_gb300 import inputs, simsd
from tests._gpu import assert_attention_close, gpu_attention, gpu_mask, oracle_attention
from tests.test_gpu_attention import _w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("Bt,Hq,Hkv,d,gamma,prefix", [
    (90, 16, 8, 64, 4, 200),    # whole units: one CTA each, one warp of rows
    (20, 32, 8, 128, 16, 300),  # the same, eight warps in each of two row blocks
    (1, 16, 8, 128, 4, 3000),   # 16 ranges of a cluster
    (2, 32, 8, 128, 8, 2500),   # clusters of CTAs of eight warps
])
def test_f32_wait_runs_out_and_the_context_stays_usable(Bt, Hq, Hkv, d, gamma, prefix, rope):
    w = _w("f32", Bt=Bt, Hq=Hq, Hkv=Hkv, d=d, gamma=gamma, seed=Bt)
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=[prefix - i for i in range(Bt)],
                                 random_step_map=True)
    tau, sect, pos, _, merr = gpu_mask(si, mask_bits=False)
    assert simsd.simsd_check_error(merr) == 0
    kw = dict(rope_pos=pos, rope_theta=1e6) if rope else {}
    before, word, ws = gpu_attention(si, mask=(tau, sect), **kw)
    assert word == 0 and ws == 0
    simsd.simsd_debug_expire_next_wait(simsd.DEBUG_WAIT_ATTENTION, 200)
    out = torch.full_like(si.q[0], float("nan"))
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    t0 = time.perf_counter()
    simsd.simsd_verify_attention(si.q[0], si.k_new[0], si.v_new[0], si.k_cache[0], si.v_cache[0], si.block_table,
                                 si.prefix_len, tau, sect, out, err_word=err, **kw)
    assert simsd.simsd_check_error(err) == simsd.EW_TIMEOUT
    # the drain waits for copies that were asked for, not for ones that never
    # come (each such wait would take its full limit of 1 s)
    assert time.perf_counter() - t0 < 0.9
    after, word, _ = gpu_attention(si, mask=(tau, sect), **kw)
    assert word == 0 and torch.equal(after, before)
    seqs = list(range(min(Bt, 2)))
    assert_attention_close(after[: len(seqs)], oracle_attention(si, seqs=seqs, rope_theta=kw.get("rope_theta", 0.0)))
