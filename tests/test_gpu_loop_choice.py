"""The driver that AUTO picks on both sides of its limit of 8192 columns, and its result against a fresh fp64 solve."""
import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,driver", [(8192, "persistent"), (8193, "launches"), (20001, "launches")])
def test_auto_picks_the_chain_for_wide_results(m, driver):
    d1, k = 90, 41
    gen = torch.Generator(device="cuda").manual_seed(m)
    X = torch.randn(300, d1, generator=gen, device="cuda", dtype=torch.float64) * torch.exp(0.5 * torch.randn(d1, generator=gen, device="cuda"))
    W = torch.randn(d1, m, generator=gen, device="cuda") * torch.exp(0.5 * torch.randn(d1, 1, generator=gen, device="cuda"))
    H = (X.t() @ X).float()
    H = 0.5 * (H + H.t())
    G = (H.double() @ W.double()).float()
    solver = pkg.Solver(0)
    outs = []
    for mode in (b.LOOP_AUTO, b.LOOP_PERSISTENT, b.LOOP_LAUNCHES):
        solver.init_support(H, G, W, 1, k, b.INIT_MAGNITUDE)
        outs.append(solver.local_search(11, accept_mode=b.ACCEPT_ALWAYS, loop_mode=mode))
    solver.close()
    assert [o.loop_driver for o in outs] == [driver, "persistent", "launches"]
    I = outs[0].support.long()
    ref = torch.linalg.solve(H.double()[I][:, I], G.double()[I])
    for o in outs:
        assert torch.equal(o.swap_trace, outs[0].swap_trace)
        # 11 rank-two moves of fp32 weights, a few roundings each, cond(H_II) below 100
        assert (o.W[I].double() - ref).norm() <= 1e-5 * ref.norm()
