"""The swap loop with delayed updates at the edges of its sizes, against the strict oracle and a fresh fp64 solve."""
import numpy as np
import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b
from parity import follow_trace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d1,m,k,swaps", [
    (9, 65, 2, 6),               # fewer slots than candidates of a batch, groups that return
    (9, 5, 2, 6),                # no room for the vectors of the loop: AUTO takes another one
    (33, 16, 30, 40),            # three pruned slots: the same few groups again and again
    (65, 40, 20, 33),            # two blocks; one swap more than a batch can hold
    (200, 20, 80, 150),          # terms fill their memory: matrices rewritten inside the search, groups that moved before it move again
    (513, 300, 256, 70),         # a slot more than eight blocks take
    (2400, 48, 1000, 40),        # more slots than threads of the candidate selection
])
def test_forced_swaps_follow_the_oracle(d1, m, k, swaps):
    gen = torch.Generator(device="cuda").manual_seed(d1)
    X = torch.randn(3 * d1, d1, generator=gen, device="cuda", dtype=torch.float64) * torch.exp(0.4 * torch.randn(d1, generator=gen, device="cuda"))
    W = torch.randn(d1, m, generator=gen, device="cuda") * torch.exp(0.4 * torch.randn(d1, 1, generator=gen, device="cuda"))
    H = (X.t() @ X).float()
    H = 0.5 * (H + H.t())
    G = (H.double() @ W.double()).float()
    solver = pkg.Solver(0)
    S0, _ = solver.init_support(H, G, W, 1, k, b.INIT_MAGNITUDE)
    fits = m > 5
    out = solver.local_search(swaps, accept_mode=b.ACCEPT_ALWAYS, loop_mode=b.LOOP_DELAYED if fits else b.LOOP_AUTO)
    perm = solver.debug_state(4).long()
    Hinv, V, R, c = (solver.debug_state(i).double() for i in range(4))
    solver.close()
    assert out.n_swaps == swaps and out.stop_reason == "max_swaps" and out.loop_driver == ("delayed" if fits else "persistent")
    H64, G64 = H.cpu().numpy().astype(np.float64), G.cpu().numpy().astype(np.float64)
    const = float(np.sum(W.cpu().numpy().astype(np.float64) * G64))
    trace = [tuple(int(v) for v in r) for r in out.swap_trace.cpu().numpy()]
    srch, _ = follow_trace(H64, G64, const, 1, S0.cpu().numpy(), trace, out.obj_trace.cpu().numpy(), accept="always", gpu_stop="max_swaps",
                           max_swaps=swaps, mode="lowrank", refactor_every=10)
    assert np.array_equal(out.support.cpu().numpy(), srch.result()[0])
    I, J = perm[:k], perm[k:]
    ref = torch.linalg.inv(H.double()[I][:, I])
    GI = G.double()[I]
    # fp32 entries of matrices whose condition is below 100
    assert (Hinv - ref).norm() <= 1e-5 * ref.norm()
    assert (V - ref @ GI).norm() <= 1e-5 * (ref @ GI).norm()
    HJI = H.double()[J][:, I]
    assert (R - (G.double()[J] - HJI @ ref @ GI)).norm() <= 1e-5 * R.norm()
    schur = H.double()[J, J] - ((HJI @ ref) * HJI).sum(1)
    assert torch.allclose(c.reshape(-1), schur, rtol=1e-5)
