"""Stochastic acceptance of few sequences: the last CTA of a sequence reads
the span sums that other SMs have just written.  Two inputs in turn over one
workspace: a sum left from the call before would draw the other input's
token, and each call must give what it gives on a workspace of its own."""
import pytest
import torch

from paper_2606_02544_gb300 import simsd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Bt,gamma,V", [(8, 8, 151936), (1, 4, 151936), (8, 8, 50001)])
def test_calls_in_turn_over_one_workspace(Bt, gamma, V):
    nbytes = simsd.simsd_accept_sampled_workspace_bytes(Bt, gamma, V)
    assert nbytes > 0
    cases = []
    for seed in (1, 2):
        g = torch.Generator(device="cuda").manual_seed(seed)
        t = torch.randn(Bt, gamma + 1, V, generator=g, device="cuda") * 2
        d = t[:, :gamma] + torch.randn(Bt, gamma, V, generator=g, device="cuda")
        draft = torch.randint(0, V, (Bt, gamma), generator=g, device="cuda", dtype=torch.int32)
        cases.append((t, d.contiguous(), draft, torch.rand(Bt, gamma, generator=g, device="cuda"),
                      torch.rand(Bt, generator=g, device="cuda")))

    def run(case, ws):
        a = torch.full((Bt,), -9, dtype=torch.int32, device="cuda")
        tok = torch.full((Bt, gamma + 1), -9, dtype=torch.int32, device="cuda")
        simsd.simsd_accept_sampled_ws(*case, a, tok, ws)
        return a, tok

    want = []
    for case in cases:
        want.append(run(case, torch.zeros(nbytes, dtype=torch.uint8, device="cuda")))
    torch.cuda.synchronize()
    assert not torch.equal(want[0][1], want[1][1])
    ws = torch.full((nbytes,), 255, dtype=torch.uint8, device="cuda")
    got = [run(cases[i % 2], ws) for i in range(200)]
    torch.cuda.synchronize()
    for i, (a, tok) in enumerate(got):
        assert torch.equal(a, want[i % 2][0]) and torch.equal(tok, want[i % 2][1])
