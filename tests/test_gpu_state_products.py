"""State build at sizes around the tiles of the digit products (128 rows, 256 or 128 columns, 128-wide k-blocks, 16-byte
rows of digits) against plain fp64 linear algebra on the device's own H and G."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U24 = 2.0 ** -24


def _problem(d1, m, g, seed, spread):
    import torch
    gen = torch.Generator().manual_seed(seed)
    X = torch.randn(3 * d1, d1, generator=gen) + 0.3 * torch.randn(3 * d1, 1, generator=gen)
    scale = torch.exp(spread * torch.randn(d1 // g, generator=gen)).repeat_interleave(g)
    X = X * scale
    W = torch.randn(d1, m, generator=gen) * 0.05
    H = (X.double().t() @ X.double()).float()
    H = 0.5 * (H + H.t())
    return H, (H.double() @ W.double()).float(), W


# k * g rows kept: below and above whole tiles, odd column counts; the last one keeps the small products on the fp64 pipe
@pytest.mark.parametrize("d1,m,g,k,spread", [
    (2176, 512, 1, 1024, 0.5),      # whole tiles
    (2203, 517, 1, 1100, 1.5),      # nothing divides, wide spread of channel scales
    (2050, 769, 1, 1281, 0.5),      # one row past a tile, 257 columns in the last pair of tiles
    (3000, 1000, 1, 897, 0.5),      # more pruned rows than kept ones
    (1305, 4101, 1, 1290, 0.5),     # fifteen pruned rows
    (2304, 513, 9, 128, 0.5),       # groups of nine rows: fp64 panels of H_JI Hinv
    (1200, 130, 1, 500, 0.5),       # below the size at which digits pay
])
def test_state_matches_fp64_algebra(d1, m, g, k, spread):
    import torch
    import paper_2403_12983_b200 as pkg
    from paper_2403_12983_b200 import binding as b
    H, G, W = _problem(d1, m, g, 7, spread)
    solver = pkg.Solver(0)
    Hd, Gd, Wd = H.cuda(), G.cuda(), W.cuda()
    support, _ = solver.init_support(Hd, Gd, Wd, g, k, b.INIT_MAGNITUDE)
    S = support.cpu().numpy()
    Hinv, V, R, c = (solver.debug_state(i).cpu().numpy() for i in range(4))
    perm = solver.debug_state(4).cpu().numpy()
    solver.close()
    assert sorted(perm[:k].tolist()) == S.tolist()
    rows = (perm[:, None] * g + np.arange(g)).reshape(-1)
    nI = k * g
    I, J = rows[:nI], rows[nI:]
    H, G = Hd.cpu().numpy().astype(np.float64), Gd.cpu().numpy().astype(np.float64)
    HII, HJI = H[np.ix_(I, I)], H[np.ix_(J, I)]
    inv = np.linalg.inv(HII)
    inv = 0.5 * (inv + inv.T)
    s = np.sqrt(np.diag(inv))
    # stored in fp32: the rounding of the entry, and what one correction step leaves of the start's error (groups)
    assert np.max(np.abs(Hinv - inv) / (s[:, None] * s[None, :])) <= (2 if g == 1 else 8) * U24
    V64 = inv @ G[I]
    R64 = G[J] - HJI @ V64
    # V: its own fp32 rounding, and a product (four digits, fp64, or split bf16 with chains of 48 truncating additions, the
    # loosest of the three) that corrects a first V made by another one
    vb = np.abs(inv) @ (np.abs(HII) @ (np.abs(inv) @ np.abs(G[I])))
    assert np.all(np.abs(V - V64) <= 2 * U24 * np.abs(V64) + (48 * U24) ** 2 * vb + 1e-30)
    # R: the error of V carried through H_JI, and its own rounding; given the device's V, only the latter
    assert np.all(np.abs(R - R64) <= 2 * U24 * (np.abs(HJI) @ np.abs(V64) + np.abs(G[J])) + (48 * U24) ** 2 * (np.abs(HJI) @ vb) + 1e-30)
    Rv = G[J] - HJI @ V.astype(np.float64)
    assert np.all(np.abs(R - Rv) <= U24 * np.abs(Rv) + 2.0 ** -32 * (np.abs(HJI) @ np.abs(V64)) + 1e-30)
    nq = d1 // g - k
    for t in range(nq):
        r = slice(t * g, (t + 1) * g)
        h = HJI[r]
        ref = H[np.ix_(J[r], J[r])] - h @ inv @ h.T
        if g == 1 and nI >= 600:      # from the fp64 inverse
            tol = 2.0 ** -32 * (np.abs(h) @ np.abs(inv) @ np.abs(h).T + np.abs(H[np.ix_(J[r], J[r])]))
        else:                         # from the inverse rounded to fp32
            tol = 2 * U24 * (np.abs(h) @ np.abs(inv) @ np.abs(h).T)
        assert np.all(np.abs(c[t] - ref) <= tol), t
