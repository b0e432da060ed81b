"""Nested phase against fresh fp64 solves, iteration by iteration, where its kernels change hands: joint downdates too wide for
shared memory, and inverses of whole layers that are corrected in column panels from digit products (4096 rows up)."""
import pytest
import torch

import paper_2403_12983_b200 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d1,m,g,k,t_hat", [
    (640, 70, 16, 19, 10),            # 160 rows leave at once: their inverse stays in global memory
    (1000, 64, 1, 490, 255),
    (4200, 40, 1, 3700, 250),         # two column panels of the correction, the second of 1640 columns
    (4167, 20, 9, 440, 10),           # first weights too narrow for digits
    (4096, 96, 64, 62, 1),
    (26300, 24, 1, 26160, 140),       # contraction too long for five digits
])
def test_nested_phase_prunes_the_cheapest_groups(d1, m, g, k, t_hat):
    gen = torch.Generator(device="cuda").manual_seed(d1)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    ng = d1 // g
    scale = torch.exp(0.5 * rand(ng)).repeat_interleave(g)
    W = (0.05 * rand(d1, m) * torch.exp(0.5 * rand(ng)).repeat_interleave(g).unsqueeze(1)).float()
    H = torch.zeros(d1, d1, dtype=torch.float64, device="cuda")
    for _ in range(0, 3 * d1, 8192):
        X = (rand(8192, d1) + 0.3 * rand(8192, 1)) * scale
        H.addmm_(X.t(), X)
    del X
    H = H.float()
    H = 0.5 * (H + H.t())
    G = torch.cat([H[i:i + 4096].double() @ W.double() for i in range(0, d1, 4096)]).float()
    solver = pkg.Solver(0)
    support, drops, obj0, iters = solver.init_support_greedy(H, G, W, g, k, t_hat)
    solver.close()
    assert iters == -(-(ng - k) // t_hat)
    support, drops = support.tolist(), drops.tolist()
    assert sorted(support + drops) == list(range(ng))
    H, G, live, pos = H.double(), G.double(), torch.arange(ng, device="cuda"), 0
    while len(live) > k:
        rows = (live[:, None] * g + torch.arange(g, device="cuda")).reshape(-1)
        inv = torch.cholesky_inverse(torch.linalg.cholesky(H[rows][:, rows]))
        V = (inv @ G[rows]).view(len(live), g, m)
        blocks = inv.view(len(live), g, len(live), g).diagonal(dim1=0, dim2=2).permute(2, 0, 1)
        D = (V * torch.linalg.solve(blocks, V)).sum((1, 2))
        t = min(t_hat, len(live) - k)
        out = torch.tensor(drops[pos:pos + t], device="cuda")
        del inv
        left = torch.isin(live, out)
        assert int(left.sum()) == t
        # two scores may change places where they agree to the last digits of fp32 sums
        assert D[left].max() <= D[~left].min() * (1 + 1e-5)
        live, pos = live[~left], pos + t
    rows = (live[:, None] * g + torch.arange(g, device="cuda")).reshape(-1)
    const = float((W.double() * G).sum())
    obj = const - float((G[rows] * torch.linalg.solve(H[rows][:, rows], G[rows])).sum())
    # a difference of const and Tr(G_I^T V) with V rounded to fp32: 2^-24 of either at most
    assert abs(obj0 - obj) <= 1e-5 * obj + 2.0 ** -24 * const
