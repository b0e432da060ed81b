"""osscar_objective against fp64: below 2^29 multiply-adds and up to 384 columns on the fp32 pipes, above from digits, in slabs of the contraction that
the 2 * d1 * m floats of scratch take; sizes around the tiles (128 rows, 256 or 128 columns) and the 128-wide k-blocks."""
import pytest

pytestmark = pytest.mark.gpu


def _call(H, W, Wt):
    import paper_2403_12983_b200 as pkg
    from paper_2403_12983_b200 import binding as b
    solver = pkg.Solver(0)
    before = b.launch_count()
    got = solver.objective(H.cuda(), W.cuda(), Wt.cuda())
    launches = b.launch_count() - before
    solver.close()
    return got, launches


@pytest.mark.parametrize("d1,m", [(128, 256), (1000, 333), (129, 257), (515, 1030), (2050, 64), (700, 1), (64, 40), (1, 1), (1153, 100),
                                  (2100, 130), (1200, 384)])      # large, but too narrow for digits
def test_objective_matches_fp64(d1, m):
    import torch
    gen = torch.Generator().manual_seed(d1 + m)
    X = torch.randn(2 * d1 + 3, d1, generator=gen)
    H = (X.double().t() @ X.double()).float()
    W, Wt = torch.randn(d1, m, generator=gen), torch.randn(d1, m, generator=gen)
    Wt[::3] = 0
    got, launches = _call(H, W, Wt)
    assert launches == 5                        # status, difference, product, two-stage trace
    D = W.double() - Wt.double()
    ref = float((D * (H.double() @ D)).sum())
    # H D is summed in fp32 (at most 2^-24 sqrt(d1) relative to |H| |D| per entry), D rounded once
    bound = float((D.abs() * (H.double().abs() @ D.abs())).sum()) * 4 * 2.0 ** -24
    assert abs(got - ref) <= bound + 1e-12


@pytest.mark.parametrize("d1,m,slabs", [
    (1100, 500, 2),           # last slab of 460 rows, columns not a multiple of 128
    (1024, 513, 2),           # one column past two tiles, rows that are not 16-byte aligned
    (777, 4000, 1),           # the whole contraction at once
    (2300, 1030, 2),          # nothing divides
    (2563, 701, 3),           # last slab of 771 rows
])
@pytest.mark.parametrize("what", ["random", "refit", "outliers"])
def test_objective_from_digits_matches_fp64(d1, m, slabs, what):
    import torch
    gen = torch.Generator().manual_seed(d1 + m)
    X = torch.relu(torch.randn(2 * d1, d1, generator=gen) + 0.5 * torch.randn(2 * d1, 1, generator=gen)) * torch.exp(0.5 * torch.randn(d1, generator=gen))
    H = (X.double().t() @ X.double()).float()
    H = 0.5 * (H + H.t())
    W, Wt = torch.randn(d1, m, generator=gen), torch.randn(d1, m, generator=gen)
    Wt[::3] = 0
    if what == "refit":                         # the weights a solve returns: H D cancels in the kept rows
        G = H.double() @ W.double()
        Wt = torch.zeros(d1, m)
        Wt[::2] = torch.linalg.solve(H.double()[::2, ::2], G[::2]).float()
    if what == "outliers":
        W[torch.arange(m) % d1, torch.arange(m)] *= 1000
    got, launches = _call(H, W, Wt)
    assert launches == 2 + 6 * slabs
    D = (W - Wt).double()
    ref = float((D * (H.double() @ D)).sum())
    # entries of both operands to 2^-32 of the scale of a row or column, and the digit products left out, 3 * 2^-32 of both scales:
    # their signs are random, in the sum over rows, columns and the contraction less than one in 10^4 of that is left
    s = H.double().diagonal().sqrt()
    worst = float((D.abs() * s[:, None] * (D.abs() * s[:, None]).amax(0)).sum()) * d1 * 41 * 2.0 ** -32
    assert abs(got - ref) <= 1e-4 * worst
    assert abs(got - ref) <= 2e-8 * ref         # fp32 sums are off by 1e-9 to 4e-7 here
