"""Gram and cross term from digits at sizes around their tiles (128 rows, 256 columns, 128-wide k-blocks, 16-byte digit rows),
with chunks that accumulate, row splits for layers of few tiles, and panels cut by a small workspace."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,d1,m,ws", [
    ([4900, 4900], 1024, 300, None),         # 20 tiles: rows split over CTAs, second chunk added
    ([700], 1001, 70, None),                 # nothing divides
    ([300, 513], 1500, 400, None),           # short chunks
    ([2000], 1152, 512, 1 << 23),            # panels of about two thousand rows at most
    ([4096], 2600, 128, None),               # more tiles than SMs would be: no split
])
def test_gram_and_cross_term_fp32(rows, d1, m, ws):
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
    for i, x in enumerate(X):
        flags = (b.GRAM_BEGIN if i == 0 else 0) | (b.GRAM_END if i == len(X) - 1 else 0)
        const = solver.gram_chunk(x.cuda(), H, flags, Wd, G, 0.0)
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
