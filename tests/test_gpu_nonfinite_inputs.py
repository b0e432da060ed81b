"""Inputs with NaN and singular H end in a status or in a support that avoids them, with the context usable afterwards."""
import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b

pytestmark = pytest.mark.gpu


def _problem(d1=96, m=20):
    gen = torch.Generator().manual_seed(3)
    X, W = torch.randn(400, d1, generator=gen), torch.randn(d1, m, generator=gen)
    H = X.t() @ X
    return H.cuda(), (H @ W).cuda(), W.cuda()


@pytest.mark.parametrize("mode", [b.INIT_MAGNITUDE, b.INIT_ENERGY])
@pytest.mark.parametrize("g", [1, 4])
def test_groups_with_nan_weights_rank_last(g, mode):
    H, G, W = _problem()
    Wn = W.clone()
    Wn[[8, 40, 95]] = float("nan")
    bad = {8 // g, 40 // g, 95 // g}
    solver = pkg.Solver(0)
    solver.set_const_term(1.0)          # a trace of W^T G would be NaN
    ng = 96 // g
    for k in (1, ng // 2, ng - len(bad)):
        S = solver.init_support(H, G, Wn, g, k, mode)[0].tolist()
        assert len(set(S)) == k and not bad & set(S)
    S = solver.init_support(H, G, torch.full_like(W, float("nan")), g, ng // 2, mode)[0].tolist()
    assert S == list(range(ng // 2))
    solver.set_const_term(0.0, False)
    with pytest.raises(pkg.OsscarError, match="positive definite"):
        solver.init_support(torch.full_like(H, float("nan")), G, W, g, ng // 2, mode)
    assert len(solver.init_support(H, G, W, g, ng // 2, mode)[0]) == ng // 2
    solver.close()


@pytest.mark.parametrize("g,t_hat", [(1, 10), (1, 1), (4, 5)])
def test_nested_phase_of_a_singular_layer_is_an_error(g, t_hat):
    H, G, W = _problem()
    gen = torch.Generator().manual_seed(4)
    X = torch.randn(40, 96, generator=gen)           # fewer rows than inputs: H has rank 40
    Hs = (X.t() @ X).cuda()
    Hz = H.clone()
    Hz[:, ::3] = 0                                   # a third of the groups cannot be scored
    Hz[::3] = 0
    solver = pkg.Solver(0)
    for bad in (Hs, Hz, -H, torch.full_like(H, float("nan"))):
        with pytest.raises(pkg.OsscarError, match="positive definite"):
            solver.init_support_greedy(bad, bad @ W, W, g, 5, t_hat)
        S, drops = solver.init_support_greedy(H, G, W, g, 5, t_hat)[:2]
        assert sorted(S.tolist() + drops.tolist()) == list(range(96 // g))
    solver.close()
