"""How the swap loop with delayed updates ends: ties."""
import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b

pytestmark = pytest.mark.gpu


def test_ties_go_to_the_smaller_group():
    """All rows alike and most of them zero: more equal scores than a batch has candidates."""
    d1, k = 400, 190
    H = torch.eye(d1, device="cuda") * 3
    G = torch.zeros(d1, 32, device="cuda")
    G[:7] = 1.5
    S = torch.arange(5, 5 + k, dtype=torch.int32)
    solver = pkg.Solver(0)
    outs = []
    for mode in (b.LOOP_DELAYED, b.LOOP_PERSISTENT):
        solver.init_support(H, G, G / 3, 1, k, b.INIT_USER, S)
        outs.append(solver.local_search(60, accept_mode=b.ACCEPT_ALWAYS, loop_mode=mode))
    solver.close()
    assert outs[0].n_swaps == 60 and torch.equal(outs[0].swap_trace, outs[1].swap_trace)
