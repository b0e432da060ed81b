"""Solvers in several threads: layers of different sizes searched at the same time end as they do alone."""
import threading

import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b

pytestmark = pytest.mark.gpu


def _layer(d1, m, g, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(1024, d1, generator=gen, device="cuda") * torch.exp(0.5 * torch.randn(d1 // g, generator=gen, device="cuda")).repeat_interleave(g)
    H = X.t() @ X
    H.diagonal().add_(100.0)
    H = 0.5 * (H + H.t())
    W = torch.randn(d1, m, generator=gen, device="cuda")
    return H, H @ W, W


# shared memory of the loops: 85 KB and 118 KB (single rows), 12 KB and 216 KB (groups)
@pytest.mark.parametrize("small,large", [((64, 16, 1, 32, 12), (10240, 16, 1, 4000, 300)), ((64, 16, 8, 4, 2), (1920, 16, 96, 9, 4))])
def test_layers_of_different_sizes_at_the_same_time(small, large):
    layers = [(_layer(*cfg[:3], i), cfg) for i, cfg in enumerate((small, large))]
    alone, errors, going = [], [], threading.Event()

    def search(solver, layer, cfg):
        (H, G, W), (_, _, g, k, swaps) = layer, cfg
        solver.init_support(H, G, W, g, k, b.INIT_MAGNITUDE)
        return solver.local_search(swaps, accept_mode=b.ACCEPT_ALWAYS)

    for layer, cfg in layers:
        solver = pkg.Solver(0)
        alone.append(search(solver, layer, cfg).swap_trace.cpu())
        solver.close()

    def work(i, rounds):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                solver = pkg.Solver(0, stream)
                n = 0
                while n < rounds or (i == 0 and going.is_set()):
                    out = search(solver, *layers[i])
                    stream.synchronize()
                    assert torch.equal(out.swap_trace.cpu(), alone[i])
                    n += 1
                solver.close()
        except Exception as exc:           # noqa: BLE001
            errors.append(exc)
        if i == 1:
            going.clear()

    torch.cuda.synchronize()
    going.set()
    threads = [threading.Thread(target=work, args=(0, 1)), threading.Thread(target=work, args=(1, 6))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
