"""Digits of one operand that serve two products whose panels have rows of different length, against fp64 algebra."""
import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b

pytestmark = pytest.mark.gpu


# The digits of H_JI are taken for R = G_J - H_JI V and serve again for the Schur complements.  The 5040 (6996) columns of the second
# product do not fit the scratch in rows of whole cache lines, the 700 (766) of the first one do.
@pytest.mark.parametrize("d1,m,k", [(5200, 700, 5040), (11488, 766, 6996)])
def test_state_where_only_one_of_two_products_has_digit_rows_on_cache_lines(d1, m, k):
    gen = torch.Generator(device="cuda").manual_seed(d1)
    H = torch.zeros(d1, d1, device="cuda", dtype=torch.float64)
    scale = torch.exp(0.5 * torch.randn(d1, generator=gen, device="cuda"))
    for _ in range(4):
        X = torch.randn(d1, d1, generator=gen, device="cuda") * scale
        H += X.double().t() @ X.double()
    H = H.float()
    H = 0.5 * (H + H.t())
    W = torch.randn(d1, m, generator=gen, device="cuda") * 0.05
    G = (H.double() @ W.double()).float()
    solver = pkg.Solver(0)
    solver.init_support(H, G, W, 1, k, b.INIT_MAGNITUDE)
    V, R, c = (solver.debug_state(i).double() for i in (1, 2, 3))
    perm = solver.debug_state(4).long()
    solver.close()
    I, J = perm[:k], perm[k:]
    inv = torch.linalg.inv(H.double()[I][:, I])
    HJI = H.double()[J][:, I]
    P = HJI @ inv
    schur = H.double()[J, J] - (P * HJI).sum(1)
    # 39 bits of every operand; sums of up to 7000 terms beside which the result is not small
    assert torch.all((c.reshape(-1) - schur).abs() <= 2.0 ** -32 * ((P.abs() * HJI.abs()).sum(1) + H.double()[J, J]))
    Rv = G.double()[J] - HJI @ V
    assert torch.all((R - Rv).abs() <= 2.0 ** -24 * Rv.abs() + 2.0 ** -32 * (HJI.abs() @ V.abs()) + 1e-30)
