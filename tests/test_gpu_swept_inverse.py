"""Inverses of ill-conditioned layers around the row count from which they are swept, against fp64 algebra."""
import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g,rows", [(1, 3071), (1, 3073), (8, 2304), (8, 3072), (8, 3584), (8, 4608)])
def test_inverse_of_condition_1e5(g, rows):
    nI = rows // g * g
    d1, k = (nI + 512) // g * g, nI // g
    gen = torch.Generator(device="cuda").manual_seed(rows)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    Q, U = torch.linalg.qr(rand(2 * d1, d1))[0], torch.linalg.qr(rand(d1, d1))[0]
    X = 50 * (Q * torch.logspace(0, -2.5, d1, device="cuda", dtype=torch.float64)) @ U.t()
    X *= torch.exp(0.5 * rand(d1 // g)).repeat_interleave(g)
    H = (X.t() @ X).float()
    H = 0.5 * (H + H.t())
    W = (0.05 * rand(d1, 64)).float()
    G = (H.double() @ W.double()).float()
    del X, Q, U
    solver = pkg.Solver(0)
    solver.init_support(H, G, W, g, k, b.INIT_MAGNITUDE)
    I = (solver.debug_state(4).long()[:k, None] * g + torch.arange(g, device="cuda")).reshape(-1)
    Hinv = solver.debug_state(0).double()
    solver.close()
    ref = torch.linalg.inv(H.double()[I][:, I])
    ref = 0.5 * (ref + ref.t())
    s = ref.diagonal().sqrt()
    # the rounding of an entry, and as much again for what the corrections leave of a start whose residual is 1e-2
    assert ((Hinv - ref) / (s[:, None] * s)).abs().max() <= 2.2 * 2.0 ** -24
