"""A search whose rewrite multiplies digits gives the same weights whatever the units of the inputs."""
import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b

pytestmark = pytest.mark.gpu


# 160 forced swaps leave 320 terms, and both sides have more than 2^29 multiply-adds: the rewrite takes digits.  560 swaps fill the terms
# as well: the state is rewritten inside the search, and later choices are made from it.
@pytest.mark.parametrize("spread", [0.5, 1.0])
@pytest.mark.parametrize("d1,m,k,swaps", [(2600, 1400, 1300, 160), (3500, 1000, 1700, 560)])
def test_weights_do_not_depend_on_units(d1, m, k, swaps, spread):
    gen = torch.Generator(device="cuda").manual_seed(d1)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    X = (rand(3 * d1, d1) + 0.3 * rand(3 * d1, 1)) * torch.exp(spread * rand(d1))
    W = (0.02 * rand(d1, m) * torch.exp(0.5 * rand(d1, 1))).float()
    H = (X.t() @ X).float()
    H = 0.5 * (H + H.t())
    G = (H.double() @ W.double()).float()
    del X
    solver = pkg.Solver(0)
    first = None
    for scale in (2.0 ** -8, 1.0, 2.0 ** 4, 2.0 ** 8):            # of the activations; exact in H and G
        Hs, Gs = H * scale ** 2, G * scale ** 2
        solver.init_support(Hs, Gs, W, 1, k, b.INIT_MAGNITUDE)
        out = solver.local_search(swaps, accept_mode=b.ACCEPT_ALWAYS)
        assert out.n_swaps == swaps and out.loop_driver == "delayed"
        perm = solver.debug_state(4).long()
        V, R = solver.debug_state(1).double(), solver.debug_state(2).double()
        I, J = perm[:k], perm[k:]
        ref = torch.linalg.solve(Hs.double()[I][:, I], Gs.double()[I])
        res = Gs.double()[J] - Hs.double()[J][:, I] @ ref
        assert (V - ref).norm() <= 1e-6 * ref.norm()
        assert (R - res).norm() <= 1e-6 * res.norm()
        if first is None:
            first = out
        assert torch.equal(out.swap_trace, first.swap_trace) and torch.equal(out.support, first.support)
        assert (out.W.double() - first.W.double()).norm() <= 1e-6 * first.W.double().norm()
    solver.close()
