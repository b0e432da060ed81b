"""Products of small layers on the fp64 pipe, k-range split over the warps of a block: sizes around its tiles (32 x 32), its k pieces
(16 for each of eight warps) and the number of tiles where the larger kernel takes over."""
import pytest

from tests.test_gpu_state_products import test_state_matches_fp64_algebra as check_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d1,m", [(1, 1), (31, 33), (64, 64), (129, 257), (33, 4000), (1000, 3), (4096, 1), (2049, 2), (255, 258), (128, 1023), (300, 180)])
def test_cross_term_of_small_layers(d1, m):
    import torch
    import paper_2403_12983_b200 as pkg
    gen = torch.Generator(device="cuda").manual_seed(d1 + m)
    X = torch.randn(2 * d1 + 9, d1, generator=gen, device="cuda")
    W = torch.randn(d1, m, generator=gen, device="cuda")
    solver = pkg.Solver(0)
    solver.ensure_workspace(d1, m, 1, max(1, d1 // 2))
    H, G, const = solver.gram([X], W, 0.01)
    solver.close()
    H64, W64 = H.double(), W.double()
    ref = H64 @ W64
    # sums in fp64, one rounding of the result
    assert bool(((G.double() - ref).abs() <= 2.0 ** -24 * ref.abs() + 2.0 ** -48 * (H64.abs() @ W64.abs())).all())
    assert const == pytest.approx(float((W64 * G.double()).sum()), rel=1e-12)


@pytest.mark.parametrize("d1,m,g,k", [(40, 7, 1, 17), (70, 130, 1, 33), (144, 65, 9, 7), (400, 100, 1, 257), (700, 20, 1, 300), (640, 200, 80, 4), (1281, 65, 1, 590)])
def test_state_of_small_layers(d1, m, g, k):
    check_state(d1, m, g, k, 0.5)
