"""The bf16 attention's bounded waits run out (as in test_gpu_wait_expiry.py)
in the kernel of 65 to 128 query rows a KV head and in the one of up to 64:
whole units in more than one wave, ranges merged in a cluster, ranges merged
through the workspace, with and without rotation."""
import pytest
import torch

from paper_2606_02544_gb300 import inputs, simsd
from tests._gpu import assert_attention_close, gpu_attention, gpu_mask, oracle_attention
from tests.test_gpu_attention import _w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("Bt,prefix,form", [(40, 300, "whole"), (5, 1500, "cluster"), (1, 3000, "workspace")])
@pytest.mark.parametrize("gamma", [16, 9, 8, 3])
def test_attention_wait_runs_out_and_the_context_stays_usable(Bt, prefix, form, gamma, rope):
    w = _w(Bt=Bt, Hq=32, Hkv=8, gamma=gamma, seed=Bt + gamma)
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=[prefix - i for i in range(Bt)],
                                 random_step_map=True)
    plan = simsd.simsd_plan_attention(simsd.SIMSD_BF16, Bt, gamma, 32, 8, 128, si.block_table.shape[1], 64, 152)
    assert plan["kernel"] == 0 and plan["rows_blk"] == 8 * gamma
    assert form == ("whole" if plan["nsplit"] == 1 else "cluster" if plan["fuse"] else "workspace")
    tau, sect, pos, _, merr = gpu_mask(si, mask_bits=False)
    assert simsd.simsd_check_error(merr) == 0
    kw = dict(rope_pos=pos, rope_theta=1e6) if rope else {}
    before, word, ws = gpu_attention(si, mask=(tau, sect), **kw)
    assert word == 0 and (ws > 0) == (form == "workspace")
    simsd.simsd_debug_expire_next_wait(simsd.DEBUG_WAIT_ATTENTION, 200)
    out = torch.full_like(si.q[0], float("nan"))
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    work = torch.zeros(ws, dtype=torch.uint8, device="cuda") if ws else None
    simsd.simsd_verify_attention(si.q[0], si.k_new[0], si.v_new[0], si.k_cache[0], si.v_cache[0], si.block_table,
                                 si.prefix_len, tau, sect, out, workspace=work, err_word=err, **kw)
    assert simsd.simsd_check_error(err) == simsd.EW_TIMEOUT
    after, word, _ = gpu_attention(si, mask=(tau, sect), **kw)
    assert word == 0 and torch.equal(after, before)
    seqs = list(range(min(Bt, 2)))
    assert_attention_close(after[: len(seqs)], oracle_attention(si, seqs=seqs, rope_theta=kw.get("rope_theta", 0.0)))
