"""Timed cases of the per-layer solve: what they draw, how they call the public entry points, and their fp64 values.

Sizes are those of `workloads/` (the named layer shapes c1 to c6) plus generic ragged ones.  Activations have the
structure of those generators (rectified, correlated, unfolded patches) and, as in trained networks, channels and
neurons of very different scale (log-normal), so that the groups' impacts are well separated and a solve's choices do
not hang on the last bits of a score.  The usual start is the magnitude rule, which that spread makes worth improving.
"""
import math

import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b

ROWS = 16384                        # calibration rows of one chunk
EPS = {"ffn": 1e-7, "heads": 1e-7, "conv": 1e-5, "dense": 1e-5}
# the improving rule where the start leaves hundreds of improving swaps, the fixed number of steps of Algorithm 1 elsewhere
ACCEPT = {"ffn": b.ACCEPT_IMPROVING, "heads": b.ACCEPT_ALWAYS, "conv": b.ACCEPT_ALWAYS, "dense": b.ACCEPT_ALWAYS}
DAMP = {"ffn": 1e-2, "heads": 1e-2, "conv": 0.0, "dense": 0.0}


def _case(name, kind, n, d1, m, k, g=1, swaps=0, call="solve", init="magnitude", score="independent", block=0, t_hat=0,
          y="float32"):
    c = dict(kind=kind, n=n, d1=d1, m=m, g=g, k=k, swaps=swaps, call=call, init=init, score=score, block=block,
             t_hat=t_hat, y=y)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small dense layer, as in a sweep over many tiny layers: nothing but latency and launches
        _case("dense-64", "dense", 256, 64, 64, 32, swaps=16),
        # pointwise convolution of a mobile network, fp32 feature maps
        _case("pointwise-1024", "dense", 24500, 1024, 1024, 512, swaps=128),
        # 3 x 3 convolution, input channels as groups of nine rows
        _case("conv-512", "conv", 6272, 4608, 512, 256, g=9, swaps=24),
        # the same layer from the nested start with two channels per iteration, then swaps
        _case("conv-512-nested", "conv", 6272, 4608, 512, 256, g=9, swaps=24, t_hat=2),
        # attention heads, every pair scored exactly
        _case("heads-32x80", "heads", 262144, 2560, 2560, 16, g=80, swaps=4, score="pair_exact"),
        # a feed-forward layer of odd sizes and a ragged last chunk
        _case("ffn-ragged", "ffn", 50021, 5000, 1283, 1777, swaps=128),
        # feed-forward layer of a 1.3B-parameter block, full calibration set
        _case("ffn-8192", "ffn", 262144, 8192, 2048, 4096, swaps=256),
        # the same shape in the layer-by-layer setting: inputs of the pruned model, outputs of the dense one
        _case("ffn-8192-sequential", "ffn", 65536, 8192, 2048, 4096, swaps=24, call="cross"),
        # the error of a finished candidate on that layer
        _case("ffn-8192-objective", "ffn", 16384, 8192, 2048, 4096, call="objective"),
        # feed-forward layer of a 30B-parameter block: exchanges of 16 neurons at a time, short calibration set
        _case("ffn-28672-blocks", "ffn", 32768, 28672, 7168, 8602, swaps=48, block=16),
        # the same layer with single swaps and the full calibration set
        _case("ffn-28672", "ffn", 262144, 28672, 7168, 8602, swaps=512),
    ]


def draw(rng):
    def size(lo, hi, step=1):
        return max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step)

    def swaps(small):
        return rng.randint(4, 24) if small else rng.randint(112, 320)

    what = rng.choice(["dense", "pointwise", "conv", "nested", "heads", "ffn", "ffn", "ffn", "cross", "objective", "blocks"])
    if what in ("dense", "pointwise"):
        d1 = size(33, 400) if what == "dense" else size(256, 2048)
        return _case(None, "dense", size(2 * d1, 32768), d1, size(16, 2048), max(2, int(d1 * rng.uniform(0.3, 0.7))),
                     swaps=rng.randint(4, 24), init=rng.choice(["magnitude", "energy"]))
    if what in ("conv", "nested"):
        g = rng.choice([4, 9, 9, 25])
        ng = size(24, 4608 // g)
        return _case(None, "conv", max(2, -(-2 * g * ng // 49)) * 49, g * ng, size(16, 1024), max(2, int(ng * rng.uniform(0.3, 0.7))),
                     g=g, swaps=rng.randint(3, 16), t_hat=0 if what == "conv" else rng.choice([1, 2, 4]))
    if what == "heads":
        g, ng = rng.choice([(64, 12), (64, 32), (80, 32), (96, 16), (64, 24)])
        return _case(None, "heads", size(8192, 262144), g * ng, size(512, 4096), max(2, int(ng * rng.uniform(0.3, 0.7))),
                     g=g, swaps=rng.randint(2, 5), score=rng.choice(["pair_exact", "independent"]))
    d1 = size(768, 12288, 8)
    k = int(d1 * rng.uniform(0.25, 0.7))
    m, n = size(128, 4096), size(8192, 131072)
    if what == "cross":
        y = rng.choice(["float32", "bfloat16"])
        return _case(None, "ffn", min(n, 65536), d1, m if y == "float32" else max(8, m // 8 * 8), k, swaps=swaps(True), call="cross", y=y)
    if what == "objective":
        return _case(None, "ffn", 8192, d1, m, k, call="objective")
    if what == "blocks":
        s = rng.choice([4, 10, 16, 32])
        return _case(None, "ffn", n, d1, m, k, swaps=s * rng.randint(2, 3), block=s)
    return _case(None, "ffn", n, d1, m, k, swaps=swaps(d1 < 2048))


# ---------------------------------------------------------------------------------------------------- inputs
def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, dtype=torch.float32, device="cuda")


def _inputs(case, seed):
    """X row blocks, W and (layer-by-layer setting) Y row blocks."""
    kind, n, d1, m, g = (case[x] for x in ("kind", "n", "d1", "m", "g"))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ng = d1 // g
    scale = torch.exp(0.5 * _randn(gen, ng)).repeat_interleave(g)
    W = _randn(gen, d1, m) * (torch.exp(0.5 * _randn(gen, ng)).repeat_interleave(g) * (0.02 if kind != "dense" else d1 ** -0.5)).unsqueeze(1)
    if kind == "dense":
        A = torch.eye(d1, device="cuda") + 0.5 / math.sqrt(d1) * _randn(gen, d1, d1)
    elif kind == "ffn":
        U, Vm = _randn(gen, d1, 64), _randn(gen, 64, d1)
    rows = ROWS if kind != "dense" else 4900
    X, Y = [], []
    for r0 in range(0, n, rows):
        r = min(rows, n - r0)
        if kind == "dense":
            x = (_randn(gen, r, d1) @ A).relu_() if n >= 4096 else _randn(gen, r, d1) @ A
        elif kind == "ffn":
            x = _randn(gen, r, d1)
            x.addmm_(x @ U, Vm, alpha=1.0 / math.sqrt(64 * d1)).relu_()
        elif kind == "heads":
            x = math.sqrt(0.5) * _randn(gen, r, ng, g) + math.sqrt(0.5) * _randn(gen, r, ng, 1)
            x = x.reshape(r, d1)
        else:                                       # feature maps of 7 x 7, patches of q x q
            q = int(math.isqrt(g))
            f = _randn(gen, r // 49, ng, 7 + q - 1, 7 + q - 1).relu_()
            x = torch.nn.functional.unfold(f, (q, q)).transpose(1, 2).reshape(r, d1)
        x.mul_(scale)
        if case["call"] == "cross":
            Y.append((x @ W).to(getattr(torch, case["y"])))
            noisy = x + 0.1 * x.abs().mean() * _randn(gen, r, d1)
            x = noisy.relu_()
        X.append(x.to(torch.bfloat16 if kind in ("ffn", "heads") else torch.float32).contiguous())
    return X, W.contiguous(), Y


def prepare(case, seed):
    X, W, Y = _inputs(case, seed)
    solver = pkg.Solver(torch.cuda.current_device())
    state = {"case": case, "solver": solver, "X": X, "W": W, "Y": Y}
    if case["call"] == "objective":                 # H as a solve leaves it, and a candidate that keeps the first k rows
        H, _, _ = solver.gram(X, W, DAMP[case["kind"]])
        Wt = W + 0.01 * W.abs().mean() * _randn(torch.Generator(device="cuda").manual_seed(seed + 1), *W.shape)
        Wt[case["k"]:] = 0
        state.update(H=H, Wt=Wt, X=None)
    return state


def run(state):
    case, solver, W = state["case"], state["solver"], state["W"]
    if case["call"] == "objective":
        return {"obj": solver.objective(state["H"], W, state["Wt"])}
    kind, init = case["kind"], {"magnitude": b.INIT_MAGNITUDE, "energy": b.INIT_ENERGY}[case["init"]]
    score = b.SCORE_PAIR_EXACT if case["score"] == "pair_exact" else b.SCORE_INDEPENDENT
    if case["call"] == "cross":
        H, G, const = solver.gram_cross(state["X"], state["Y"], DAMP[kind])
        solver.init_support(H, G, W, case["g"], case["k"], init)
        out = solver.local_search(case["swaps"], score, ACCEPT[kind], accept_rel_tol=EPS[kind])
    else:
        out = pkg.solve_layer(solver, state["X"], W, case["g"], case["k"], case["swaps"], damp=DAMP[kind], init_mode=init,
                              score_mode=score, accept_mode=ACCEPT[kind], accept_rel_tol=EPS[kind], greedy_t_hat=case["t_hat"], block_pairs=case["block"])
        H, G, const = out.H, out.G, out.const_term
    return {"support": out.support, "W": out.W, "obj_trace": out.obj_trace, "swap_trace": out.swap_trace,
            "obj_init": out.obj_init, "obj_final": out.obj_final, "const": const, "H": H, "G": G}


# ---------------------------------------------------------------------------------------------------- work and tolerance
def work(case):
    n, d1, m, g, k = (case[x] for x in ("n", "d1", "m", "g", "k"))
    if case["call"] == "objective":
        return {"bytes": 4 * d1 * d1 + 8 * d1 * m, "flops": 2 * d1 * d1 * m + 2 * d1 * m}
    nI = k * g
    nJ = d1 - nI
    es = 2 if case["kind"] in ("ffn", "heads") else 4
    nbytes = n * d1 * es + 4 * d1 * d1 + 4 * d1 * m * 3
    flops = n * d1 * d1                                                    # one triangle of X^T X
    if case["call"] == "cross":
        nbytes += n * m * (4 if case["y"] == "float32" else 2)
        flops += 2 * n * d1 * m
    else:
        flops += 2 * d1 * d1 * m
    if case["t_hat"]:
        flops += d1 ** 3 + 2 * d1 * d1 * m
    flops += nI ** 3 + 2 * nI * nI * m + 2 * nJ * nI * m + nJ * nI * nI    # inverse, V, R, Schur complements
    flops += case["swaps"] * 2 * g * (nI * nI + 2 * nJ * nI + 2 * d1 * m)  # rank-2 moves of the state
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["call"] == "objective":
        return {"rel": 1e-5}
    # four times what the solves show against exact(); a block exchange keeps its whole state in fp32 between iterations.
    # Neighbouring choices of a long trace may change places where two scores agree to their last bits.
    if case["block"]:
        return {"rel": 2.5e-3, "max": 0.1, "differ": 0.01}
    return {"rel": 3e-4, "max": 5e-3, "differ": 0.01}


# ---------------------------------------------------------------------------------------------------- the same in 64 bits
def _gram64(X, d1):
    H = torch.zeros(d1, d1, dtype=torch.float64, device="cuda")
    step = max(512, -(-d1 // 8))
    for x in X:
        x = x.double()
        for j in range(0, d1, step):
            H[:min(j + step, d1), j:j + step].addmm_(x[:, :min(j + step, d1)].t(), x[:, j:j + step])
    for j in range(0, d1, step):
        H[j:, j:j + step] = H[j:j + step, j:].t().clone()
    return H


def _exchange(M, rows):
    """Principal exchange of `rows` of M = [H | G]: kept rows become pruned ones and the other way round."""
    P = torch.linalg.inv(M[rows[:, None], rows])
    panel = P @ M[rows]
    cols = M[:, rows].clone()
    cols[rows] = 0
    M.addmm_(cols, panel, alpha=-1.0)
    M[:, rows] = -cols @ P
    panel[:, rows] = P
    M[rows] = panel
    return M


def exact(case, seed):
    kind, d1, m, g, k, T = (case[x] for x in ("kind", "d1", "m", "g", "k", "swaps"))
    X, W32, Y = _inputs(case, seed)
    W, ng = W32.double(), d1 // g
    H = _gram64(X, d1)
    H.diagonal().add_(DAMP[kind] * H.diagonal().mean())
    if case["call"] == "objective":
        Wt = W32 + 0.01 * W32.abs().mean() * _randn(torch.Generator(device="cuda").manual_seed(seed + 1), *W32.shape)
        Wt[k:] = 0
        D = W - Wt.double()
        return {"obj": float((D * (H @ D)).sum())}
    if case["call"] == "cross":
        G = sum(x.double().t() @ y.double() for x, y in zip(X, Y))
        const = float(sum(y.double().square().sum() for y in Y))
    else:
        G = H @ W
        const = float((W * G).sum())
    del X, Y
    arange = torch.arange(d1, device="cuda")
    span = lambda q: (torch.as_tensor(q, device="cuda").reshape(-1, 1) * g + arange[:g]).reshape(-1)  # noqa: E731

    def gains(M, ids):
        """Tr(B^T P^-1 B) of every group in `ids`, P its diagonal block and B its rows of the right-hand side."""
        rows = span(ids)
        B = M[rows, d1:].view(len(ids), g, m)
        if g == 1:
            return B.square().sum((1, 2)) / M[rows, rows]
        rows = rows.view(-1, g)
        return (B * torch.linalg.solve(M[rows[:, :, None], rows[:, None, :]], B)).sum((1, 2))

    def sweep_in(kept):
        """[H | G] with the kept rows exchanged, and the objective there."""
        M = torch.cat([H, G], 1)
        I = span(kept)
        inv = torch.cholesky_inverse(torch.linalg.cholesky(H[I[:, None], I]))
        panel = inv @ M[I]
        cols = M[:, I].clone()
        obj = const - float((G[I] * panel[:, d1:]).sum())
        cols[I] = 0
        M.addmm_(cols, panel, alpha=-1.0)
        M[:, I] = -(cols @ inv)
        panel[:, I] = inv
        M[I] = panel
        return M, obj

    if case["t_hat"]:
        kept = torch.arange(ng, device="cuda")
        M, obj = sweep_in(kept)
        while len(kept) > k:
            take = torch.argsort(gains(M, kept), stable=True)[:min(case["t_hat"], len(kept) - k)]
            _exchange(M, span(kept[take]))
            mask = torch.ones(len(kept), dtype=torch.bool, device="cuda")
            mask[take] = False
            kept = kept[mask]
        del M
    else:
        if case["init"] == "energy":
            if g == 1:
                e = W.square().sum(1) * H.diagonal()
            else:
                rows = arange.view(ng, g)
                e = (W.view(ng, g, m) * (H[rows[:, :, None], rows[:, None, :]] @ W.view(ng, g, m))).sum((1, 2))
        else:
            e = W.view(ng, g * m).square().sum(1)
        kept = torch.argsort(-e, stable=True)[:k].sort().values
    M, obj = sweep_in(kept)
    keep = torch.zeros(ng, dtype=torch.bool, device="cuda")
    keep[kept] = True
    trace, swaps, s = [obj], [], max(1, case["block"])
    for _ in range(T // s):
        kept, pruned = keep.nonzero().flatten(), (~keep).nonzero().flatten()
        D, A = gains(M, kept), gains(M, pruned)
        if case["score"] == "pair_exact":
            best = None
            R = M[span(pruned), d1:].view(-1, g, m)
            rows = span(pruned).view(-1, g)
            for i in range(len(kept)):
                r = span(kept[i])
                left = (M[span(pruned)][:, r] @ torch.linalg.inv(M[r[:, None], r])).view(-1, g, g)
                c = M[rows[:, :, None], rows[:, None, :]] - left @ M[r][:, rows].permute(1, 0, 2)
                r1 = R - left @ M[r, d1:]
                delta = D[i] - (r1 * torch.linalg.solve(c, r1)).sum((1, 2))
                j = int(delta.argmin())
                if best is None or float(delta[j]) < best[0]:
                    best = (float(delta[j]), i, j)
            out, into = kept[best[1]:best[1] + 1], pruned[best[2]:best[2] + 1]
        else:
            out, into = kept[torch.argsort(D, stable=True)[:s]], pruned[torch.argsort(-A, stable=True)[:s]]
        B = M[span(out), d1:]
        up = float((B * torch.linalg.solve(M[span(out)[:, None], span(out)], B)).sum())
        _exchange(M, span(out))
        B = M[span(into), d1:]
        down = float((B * torch.linalg.solve(M[span(into)[:, None], span(into)], B)).sum())
        if ACCEPT[kind] == b.ACCEPT_IMPROVING and up - down > -EPS[kind] * obj:
            _exchange(M, span(out))
            break
        _exchange(M, span(into))
        obj += up - down
        keep[out], keep[into] = False, True
        trace.append(obj)
        swaps += list(zip(out.tolist(), into.tolist()))
    kept = keep.nonzero().flatten()
    Wout = torch.zeros_like(W)
    Wout[span(kept)] = M[span(kept), d1:]
    return {"support": kept.to(torch.int32), "W": Wout, "obj_trace": torch.tensor(trace, dtype=torch.float64, device="cuda"),
            "swap_trace": torch.tensor(swaps, dtype=torch.int32, device="cuda").view(-1, 2), "obj_init": trace[0], "obj_final": obj,
            "const": const, "H": H, "G": G}
