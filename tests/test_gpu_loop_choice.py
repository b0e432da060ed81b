"""The driver that ran, by name and under AUTO, for searches and results on both sides of its limits, and its result against a fresh fp64 solve."""
import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,swaps,driver", [(8192, 9, "persistent"), (8192, 10, "delayed"), (8193, 15, "launches"), (8193, 16, "delayed"), (20001, 11, "launches")])
def test_the_driver_that_ran_is_reported(m, swaps, driver):
    d1, k = 90, 41
    gen = torch.Generator(device="cuda").manual_seed(m)
    X = torch.randn(300, d1, generator=gen, device="cuda", dtype=torch.float64) * torch.exp(0.5 * torch.randn(d1, generator=gen, device="cuda"))
    W = torch.randn(d1, m, generator=gen, device="cuda") * torch.exp(0.5 * torch.randn(d1, 1, generator=gen, device="cuda"))
    H = (X.t() @ X).float()
    H = 0.5 * (H + H.t())
    G = (H.double() @ W.double()).float()
    solver = pkg.Solver(0)
    outs = []
    for mode in (b.LOOP_AUTO, b.LOOP_DELAYED, b.LOOP_PERSISTENT, b.LOOP_LAUNCHES):
        solver.init_support(H, G, W, 1, k, b.INIT_MAGNITUDE)
        outs.append(solver.local_search(swaps, accept_mode=b.ACCEPT_ALWAYS, loop_mode=mode))
    solver.init_support(H, G, W, 10, 4, b.INIT_MAGNITUDE)
    with pytest.raises(pkg.OsscarError, match="osscar_local_search"):
        solver.local_search(11, loop_mode=b.LOOP_DELAYED)              # single-row groups only
    solver.init_support(H, G, W, 10, 4, b.INIT_MAGNITUDE)
    assert solver.local_search(3).loop_driver == "launches"
    solver.close()
    assert [o.loop_driver for o in outs] == [driver, "delayed", "persistent", "launches"]
    assert [o.n_batches > 0 for o in outs] == [driver == "delayed", True, False, False]
    I = outs[0].support.long()
    ref = torch.linalg.solve(H.double()[I][:, I], G.double()[I])
    for o in outs:
        assert torch.equal(o.swap_trace, outs[0].swap_trace)
        # up to 16 rank-two moves of fp32 weights, a few roundings each, cond(H_II) below 100
        assert (o.W[I].double() - ref).norm() <= 1e-5 * ref.norm()
