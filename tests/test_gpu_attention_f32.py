"""The fp32 kernel's row packing (8 rows a warp, up to 8 warps a CTA, several
row blocks), key tiles of 32 and cluster splits of up to 16 ranges, against
the fp64 oracle within the stated 1e-5 (fp32 scores of d products, sums over
at most a few thousand keys: about 1e-6).  Also: a value that is no number in
a new slot reaches only the rows that see the slot."""
import pytest
import torch

from paper_2606_02544_gb300 import inputs
from tests._gpu import assert_attention_close, gpu_attention, gpu_mask, oracle_attention

pytestmark = pytest.mark.gpu


def _w(Bt, Hq, Hkv, d, gamma, P, seed=0):
    return inputs.Workload("f32", "f32", Bt, Hq, Hkv, d, gamma, (0, 300), 1, 64, 0.5, 1.0, 1.0, seed, P)


@pytest.mark.parametrize("gamma,Hq,Hkv,d,P,prefix", [
    (1, 1, 1, 64, 64, [0]),                    # two rows, one partial tile
    (1, 8, 8, 128, 8, [33, 5, 700]),           # one warp a CTA, small pages
    (4, 2, 1, 64, 64, [128]),                  # five tiles, one range each
    (3, 6, 2, 128, 16, [0, 31, 32, 33, 500]),  # 18 rows: the last group partly empty
    (5, 24, 8, 128, 32, [29, 64, 95]),         # new slots straddle tiles
    (9, 10, 2, 64, 192, [700, 191]),           # 90 rows in two blocks, odd page size
    (16, 32, 8, 128, 64, [1000, 64]),          # two full row blocks
    (32, 32, 8, 128, 64, [100, 3]),            # four row blocks, three tiles of new slots
    (4, 16, 8, 128, 64, [4000]),               # 16 ranges of many tiles
    (2, 16, 8, 64, 16, [i % 97 for i in range(130)]),  # more units than fit at once: no split
])
def test_f32_tiles_and_splits(gamma, Hq, Hkv, d, P, prefix):
    si = inputs.make_step_inputs(_w(len(prefix), Hq, Hkv, d, gamma, P, seed=gamma + d), device="cuda",
                                 prefix_override=prefix, random_step_map=True, poison_unused_rows=True)
    seqs = None if len(prefix) < 10 else list(range(0, len(prefix), 19))
    out, word, ws = gpu_attention(si)
    ref = oracle_attention(si, seqs=seqs)
    assert word == ref.err == 0 and ws == 0
    assert_attention_close(out if seqs is None else out[seqs], ref)


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("prefix", [[40], [1500]])
def test_f32_unseen_new_value(value, prefix):
    w = _w(1, 4, 2, 128, 6, 64, seed=3)
    si = inputs.make_step_inputs(w, device="cuda", prefix_override=prefix, random_step_map=True)
    tau, sect, _, bits, _ = gpu_mask(si)
    clean, _, _ = gpu_attention(si, mask=(tau, sect))
    slot = 2
    si.v_new[0, 0, slot, :, 5] = value
    out, word, _ = gpu_attention(si, mask=(tau, sect))
    assert word == 0
    sees = ((bits[0] >> slot) & 1).bool()
    assert sees.any() and (~sees).any()
    assert torch.equal(out[0, ~sees], clean[0, ~sees])
    assert not torch.isfinite(out[0, sees][:, :, 5]).any()
