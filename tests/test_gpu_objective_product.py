"""osscar_objective against fp64 at sizes around the tiles (128 rows, 256 columns, 64-wide k-blocks) and the K panels that
2 * d1 * m floats of scratch allow, down to column counts that leave no room for a panel."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d1,m", [(128, 256), (1000, 333), (129, 257), (515, 1030), (2050, 64), (700, 1), (64, 40), (1, 1), (1153, 100)])
def test_objective_matches_fp64(d1, m):
    import torch
    import paper_2403_12983_b200 as pkg
    gen = torch.Generator().manual_seed(d1 + m)
    X = torch.randn(2 * d1 + 3, d1, generator=gen)
    H = (X.double().t() @ X.double()).float()
    W, Wt = torch.randn(d1, m, generator=gen), torch.randn(d1, m, generator=gen)
    Wt[::3] = 0
    solver = pkg.Solver(0)
    got = solver.objective(H.cuda(), W.cuda(), Wt.cuda())
    solver.close()
    D = W.double() - Wt.double()
    ref = float((D * (H.double() @ D)).sum())
    # H D is summed in fp32 (chains of 128 products, at most 2^-24 sqrt(d1) relative to |H| |D| per entry), D rounded once
    bound = float((D.abs() * (H.double().abs() @ D.abs())).sum()) * 4 * 2.0 ** -24
    assert abs(got - ref) <= bound + 1e-12
