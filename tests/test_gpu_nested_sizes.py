"""Nested phase against fresh fp64 solves, iteration by iteration, where its kernels change hands: joint downdates too wide for
shared memory."""
import pytest
import torch

import paper_2403_12983_b200 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d1,m,g,k,t_hat", [
    (640, 70, 16, 19, 10),            # 160 rows leave at once: their inverse stays in global memory
    (1000, 64, 1, 490, 255),
])
def test_nested_phase_prunes_the_cheapest_groups(d1, m, g, k, t_hat):
    gen = torch.Generator(device="cuda").manual_seed(d1)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    ng = d1 // g
    X = rand(3 * d1, d1) + 0.3 * rand(3 * d1, 1)
    X *= torch.exp(0.5 * rand(ng)).repeat_interleave(g)
    W = (0.05 * rand(d1, m) * torch.exp(0.5 * rand(ng)).repeat_interleave(g).unsqueeze(1)).float()
    H = (X.t() @ X).float()
    H = 0.5 * (H + H.t())
    G = (H.double() @ W.double()).float()
    solver = pkg.Solver(0)
    support, drops, obj0, iters = solver.init_support_greedy(H, G, W, g, k, t_hat)
    solver.close()
    assert iters == -(-(ng - k) // t_hat)
    support, drops = support.tolist(), drops.tolist()
    assert sorted(support + drops) == list(range(ng))
    H, G, live, pos = H.double(), G.double(), torch.arange(ng, device="cuda"), 0
    while len(live) > k:
        rows = (live[:, None] * g + torch.arange(g, device="cuda")).reshape(-1)
        inv = torch.linalg.inv(H[rows][:, rows])
        V = (inv @ G[rows]).view(len(live), g, m)
        blocks = inv.view(len(live), g, len(live), g).diagonal(dim1=0, dim2=2).permute(2, 0, 1)
        D = (V * torch.linalg.solve(blocks, V)).sum((1, 2))
        t = min(t_hat, len(live) - k)
        out = torch.tensor(drops[pos:pos + t], device="cuda")
        left = torch.isin(live, out)
        assert int(left.sum()) == t
        # two scores may change places where they agree to the last digits of fp32 sums
        assert D[left].max() <= D[~left].min() * (1 + 1e-5)
        live, pos = live[~left], pos + t
    rows = (live[:, None] * g + torch.arange(g, device="cuda")).reshape(-1)
    obj = float((W.double() * G).sum() - (G[rows] * torch.linalg.solve(H[rows][:, rows], G[rows])).sum())
    assert obj0 == pytest.approx(obj, rel=1e-5)
