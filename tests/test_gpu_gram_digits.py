"""Gram and cross term from digits at sizes around their tiles (128 rows, 256 columns, 128-wide k-blocks, 16-byte digit rows),
with chunks that accumulate, row splits for layers of few tiles, and panels cut by a small workspace; by the number of launches
each case is seen to take the path that it names."""
import pytest

pytestmark = pytest.mark.gpu


def _panels(rows, n):
    h = -(-(-(-rows // n)) // 16) * 16 if n > 1 else rows
    return [min(h, rows - i) for i in range(0, rows, h)]


@pytest.mark.parametrize("rows,d1,m,ws,panels,split", [
    ([4900, 4900], 1024, 300, None, [1, 1], True),         # 20 tiles: rows split over CTAs, second chunk added
    ([700], 1001, 70, None, [0], False),                   # nothing divides; short chunks stay on the bf16 terms
    ([300, 513], 1500, 400, None, [0, 0], False),
    ([2051], 1001, 70, None, [1], True),
    ([5003], 1152, 512, 1 << 23, [3], False),              # panels of 1680 rows, the last of 1643
    ([5003, 2048], 1152, 512, 1 << 24, [3, 2], True),      # panels whose rows are split as well
    ([2500], 1152, 512, 3499776, [0], False),              # no room for a thousand rows
    ([4096], 2600, 128, None, [1], False),                 # a tile for every SM: no split
])
def test_gram_and_cross_term_fp32(rows, d1, m, ws, panels, split):
    import torch
    import paper_2403_12983_b200 as pkg
    from paper_2403_12983_b200 import binding as b
    gen = torch.Generator().manual_seed(d1)
    scale = torch.exp(torch.randn(d1, generator=gen))
    X = [torch.relu(torch.randn(r, d1, generator=gen)) * scale for r in rows]
    W = torch.randn(d1, m, generator=gen)
    solver = pkg.Solver(0)
    if ws is None:
        solver.ensure_workspace(d1, m, 1, d1 // 2)
    else:
        solver.lend_workspace(ws)
    H = torch.empty(d1, d1, device="cuda")
    G = torch.empty(d1, m, device="cuda")
    Wd = W.cuda()
    const = None
    before = b.launch_count()
    for i, x in enumerate(X):
        solver.gram_chunk(x.cuda(), H, b.GRAM_BEGIN if i == 0 else 0)
    terms = solver._ws.numel() - 4096                                    # panels of the bf16 terms, two launches each
    rows_t = terms // (6 * ((d1 + 7) // 8 * 8))
    count = lambda n: 2 * -(-n // (n if rows_t >= n else rows_t // 64 * 64))  # noqa: E731
    launches = b.launch_count() - before
    # digits: maxima, digits, outliers, product (and its sum), and the terms that a panel with outliers takes instead
    want = sum(sum((5 if split else 4) + count(h) for h in _panels(r, n)) if n else count(r) for r, n in zip(rows, panels))
    assert launches == 1 + want
    const = solver.gram_chunk(torch.empty(0, d1, device="cuda"), H, b.GRAM_END, Wd, G, 0.0)
    solver.close()
    X64 = [x.double() for x in X]
    H64 = sum(x.t() @ x for x in X64)
    # each chunk: entries rounded to 2^-23 of their column's largest (twice that with the digit products left out), then fp32
    bound = sum(2.0 ** -22 * (torch.outer(x.abs().amax(0), x.abs().sum(0)) + torch.outer(x.abs().sum(0), x.abs().amax(0))) for x in X64)
    bound += 2.0 ** -23 * (len(X) + 1) * H64.abs()
    Hd = H.double().cpu()
    assert torch.equal(Hd, Hd.t())
    assert bool(((Hd - H64).abs() <= bound).all())
    assert float((Hd - H64).norm() / H64.norm()) < 1e-6
    G64 = Hd @ W.double()
    # G from the device's own H: 2^-30 of row and column maxima, or split bf16 terms (chains of 48 truncating additions)
    gb = 48 * 2.0 ** -24 * (Hd.abs() @ W.double().abs())
    assert bool(((G.double().cpu() - G64).abs() <= gb).all())
    assert const == pytest.approx(float((W.double() * G64).sum()), rel=1e-5)


# entries far above the rest of their column, values that repeat (their roundings do not average out), and both in one chunk
@pytest.mark.parametrize("rows,d1", [([4900, 2100], 384), ([4100], 1600), ([2500], 777)])
@pytest.mark.parametrize("kind,height", [("relu", 30), ("relu", 300), ("relu", 1000), ("relu", 1e6), ("pixels", 1), ("pixels", 8), ("constant", 6), ("constant", 40)])
def test_gram_of_columns_with_outliers(rows, d1, kind, height):
    import torch
    import paper_2403_12983_b200 as pkg
    from paper_2403_12983_b200 import binding as b
    gen = torch.Generator(device="cuda").manual_seed(d1)
    X = []
    for i, r in enumerate(rows):
        x = torch.relu(torch.randn(r, d1, generator=gen, device="cuda"))
        if kind == "pixels":
            x = torch.randint(0, 256, (r, d1), generator=gen, device="cuda").float() / 255
        if kind == "constant":
            x = (0.5 + torch.rand(1, d1, generator=gen, device="cuda")).expand(r, d1).contiguous()
        if height > 1 and i == 0:                    # the second chunk has none
            j = torch.arange(0, d1, 3, device="cuda")
            x[j * 37 % r, j] = height * x.square().mean(0).sqrt()[j]
        X.append(x)
    solver = pkg.Solver(0)
    solver.ensure_workspace(d1, 64, 1, d1 // 2)
    H, G, W = torch.empty(d1, d1, device="cuda"), torch.empty(d1, 64, device="cuda"), torch.randn(d1, 64, generator=gen, device="cuda")
    for i, x in enumerate(X):
        solver.gram_chunk(x, H, (b.GRAM_BEGIN if i == 0 else 0) | (b.GRAM_END if i == len(X) - 1 else 0), W, G, 0.0)
    solver.close()
    X = torch.cat(X).double()
    H64 = X.t() @ X                                  # no cancellation: nothing is negative
    # bf16 terms: chains of 24 truncating additions per 64 rows and one fp32 addition per drain, at most 24 x 2^-23 in all;
    # digits: 2^-19 sqrt(H_ii H_jj) at most
    assert float(((H.double() - H64).abs() / H64).max()) < 24 * 2.0 ** -23
    d = H64.diagonal().sqrt()
    assert float(((H.double() - H64).abs() / (d[:, None] * d[None, :])).max()) < 24 * 2.0 ** -23
