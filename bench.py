"""Benchmark of the OSSCAR per-layer solve on B200.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--workload c5] [--impl ours|reference]

One "step" is one whole layer solve (Gram over all token chunks, cross term, starting support and state,
device-resident swap search, result) on one synthetic layer.  With N > 1 (torchrun) every rank solves an
independent replica of the layer (seed = rank): the solve does not shard, so scaling is weak and there is
no collective on the data path.  Prints one JSON line on rank 0.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import torch  # noqa: E402

import workloads  # noqa: E402

METRIC = "swaps/s of the device-resident swap search (layer-solve seconds in ms_per_step)"
UNIT = "swaps/s"


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        p = json.load(open(path))
        return {"hbm_gbs": p["hbm_gbs"], "bf16_tflops": p["bf16_tflops"],
                "bf16_tflops_sustained": p.get("bf16_tflops_sustained", p["bf16_tflops"]), "source": "measured"}
    return {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0, "source": "fallback"}


# ------------------------------------------------------------------------------------------ helpers
class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi while the timed region runs."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index, self.proc, self.lines = index, None, []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._pump, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None

    def _pump(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1])); smax.append(float(f[2]))
            except ValueError:
                continue
            for name, val in zip(("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"), f[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        busy = [c for c in sm if c > 0]
        return {"sm_mhz": statistics.median(busy) if busy else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def dist_env():
    rank = int(os.environ.get("RANK", "0")); world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def reduce_over_ranks(values: dict, world: int, backend_device):
    """max over ranks for keys starting with 'max_', sum for 'sum_' (all-reduce; identity when world == 1)."""
    if world == 1:
        return dict(values)
    import torch.distributed as dist
    out = {}
    for key, val in values.items():
        t = torch.tensor([float(val)], dtype=torch.float64, device=backend_device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX if key.startswith("max_") else dist.ReduceOp.SUM)
        out[key] = float(t.item())
    return out


LAZY_ROUND = 4     # steps between two writes of the matrices in the launch chain of single-row groups



def swap_bytes(nI, nJ, m, fused_y=False, lazy=False, per_batch=0.0):
    """Algorithmic HBM bytes of one swap: V and R_J read+write and H[J,I] read once in fp32; the inverse read+write
    in fp64 with the next y fused into that pass (single-row groups), or in fp32 with a separate y pass.  `lazy`: V, R and
    the inverse are read in every step and written in every LAZY_ROUND-th.  `per_batch`: swaps per batch of the delayed loop, which reads all of
    them once per batch."""
    if per_batch:
        return int((8 * nI * nI + 4 * (nI + nJ) * m + 4 * nJ * nI) / per_batch)
    if lazy:
        held = 8 * nI * nI + 4 * (nI + nJ) * m
        return held + 4 * nJ * nI + held // LAZY_ROUND
    if fused_y:
        return 16 * nI * nI + 4 * (2 * nI * m + 2 * nJ * m + nJ * nI)
    return 4 * (3 * nI * nI + 2 * nI * m + 2 * nJ * m + nJ * nI)


KERNEL_BYTES = {   # algorithmic bytes per launch of the streaming kernels of a step
    "y_pass": lambda nI, nJ, m: 4 * nI * nI,
    "h_pass": lambda nI, nJ, m: 4 * nJ * nI,
    "update_hinv": lambda nI, nJ, m: 8 * nI * nI,
    "swap_loop": lambda nI, nJ, m: swap_bytes(nI, nJ, m, True),
    "update_v": lambda nI, nJ, m: 8 * nI * m,
    "update_r": lambda nI, nJ, m: 8 * nJ * m,
    # launch chain of single-row groups: H pass; rows of V and R; y and, in every LAZY_ROUND-th step, the write of the inverse
    "l1_hpass_update_v": lambda nI, nJ, m: 4 * nJ * nI,
    "l2_update_r_swap": lambda nI, nJ, m: 4 * (nI + nJ) * m * (LAZY_ROUND + 1) // LAZY_ROUND,
    "l4_update_hinv_y": lambda nI, nJ, m: 8 * nI * nI * (LAZY_ROUND + 1) // LAZY_ROUND,
}


# ------------------------------------------------------------------------------------------ CPU oracle legs
def workload_label(wl, max_swaps, accept_always=False, greedy=0, block_pairs=0):
    return (f"{wl.name}: d1={wl.d1} m={wl.m} g={wl.g} k={wl.k} n={wl.n} in {wl.n_chunks} chunks, "
            f"max_swaps={max_swaps}, accept={'always' if accept_always else 'improving'} (eps {wl.eps_acc:g}), damp={wl.damp}, "
            f"init={'greedy t_hat=%d' % greedy if greedy else 'energy'}"
            + (f", block exchanges of {block_pairs} groups" if block_pairs > 1 else ""))


def oracle_swaps_at_size(H, G, const, wl, n_swaps):
    """Times the oracle's low-rank mode on a layer of the workload's own size: the fresh solve that starts it (set-up)
    and `n_swaps` steps (propose + apply).  H, G are fp64 arrays of the full layer."""
    import numpy as np
    from oracle import osscar_oracle as orc
    t0 = time.perf_counter()
    S0, _ = orc.init_support(H, wl.weight().numpy().astype(np.float64), wl.g, wl.k)
    srch = orc.Search(H, G, const, wl.g, S0, mode="lowrank", eps_acc=wl.eps_acc, accept="always")
    t1 = time.perf_counter()
    per = []
    for _ in range(n_swaps):
        ts = time.perf_counter()
        info = srch.propose()
        if info is None:
            break
        srch.apply(info.slot, info.j_in)
        per.append(time.perf_counter() - ts)
    return {"setup_s": t1 - t0, "swap_s": per}


def synthetic_spd_layer(wl, tokens=512):
    """A full-width SPD H for the CPU legs that have no device: the Gram of `tokens` calibration rows plus the damping
    term (full rank through the damping; the oracle's cost per swap does not depend on the values), and G = H W."""
    import numpy as np
    keep = wl.chunk_rows
    wl.chunk_rows = tokens
    X = wl.x_chunk(0).float().numpy().astype(np.float64)
    wl.chunk_rows = keep
    H = X.T @ X
    H += max(wl.damp, 1e-2) * np.mean(np.diag(H)) * np.eye(wl.d1)
    W = wl.weight().numpy().astype(np.float64)
    G = H @ W
    return H, G, float(np.sum(W * G))


def strict_step_seconds(H, G, const, wl, steps, score_mode="independent"):
    """Seconds per step of the strict oracle (fresh Cholesky solve per step) on fp64 H, G of a whole layer."""
    import numpy as np
    from oracle import osscar_oracle as orc
    W = wl.weight().numpy().astype(np.float64)
    S0, _ = orc.init_support(H, W, wl.g, wl.k)
    srch = orc.Search(H, G, const, wl.g, S0, mode="strict", score_mode=score_mode, accept="always")
    per = []
    for _ in range(steps):
        ts = time.perf_counter()
        info = srch.propose()
        if info is None:
            break
        srch.apply(info.slot, info.j_in)
        per.append(time.perf_counter() - ts)
    return per


def run_reference(args):
    """The oracle as it stands, on the host cores, on the benchmark's own layer size: one step = one swap of its
    low-rank mode (propose + apply) on a full-width layer; the fresh solve that starts it is set-up, outside the steps."""
    rank, world, _ = dist_env()
    if rank != 0:
        return
    wl = workloads.config(args.workload)
    max_swaps = args.max_swaps if args.max_swaps is not None else wl.max_swaps
    H, G, const = synthetic_spd_layer(wl)
    r = oracle_swaps_at_size(H, G, const, wl, args.warmup + args.steps)
    timed = r["swap_s"][args.warmup:]
    tot = sum(timed)
    value = len(timed) / max(tot, 1e-9)
    cores = torch.get_num_threads()
    sample = (f"fp64 NumPy oracle (low-rank-update mode) at the layer's own size d1={wl.d1}, m={wl.m}, k={wl.k}: one swap per step, "
              f"{len(timed)} timed swaps after {args.warmup} warm-up swaps; H = Gram of 512 synthetic tokens + damping, G = H W; "
              f"set-up (fresh fp64 solve) {r['setup_s']:.1f} s outside the steps")
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * tot / max(len(timed), 1), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": workload_label(wl, max_swaps)},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0}))


def cpu_baseline_at_size(wl, H_dev, G_dev, const, n_swaps=3):
    """The oracle on the host cores at the benchmark layer's own size, fed the device's H and G (fp32 -> fp64):
    `n_swaps` steps of its low-rank mode after the fresh fp64 solve that starts it, plus the fp64 Gram of a slice of
    one token chunk (the Gram is linear in tokens, so the slice scales to the layer)."""
    import numpy as np
    H = H_dev.cpu().numpy().astype(np.float64)
    G = G_dev.cpu().numpy().astype(np.float64)
    r = oracle_swaps_at_size(H, G, const, wl, n_swaps)
    del H, G
    rows = max(64, min(wl.chunk_rows, int(2.0e12 / (2.0 * wl.d1 * wl.d1))))        # about 2 TFLOP of fp64 work
    keep = wl.chunk_rows
    wl.chunk_rows = rows
    X = wl.x_chunk(0).float().numpy().astype(np.float64)
    wl.chunk_rows = keep
    t0 = time.perf_counter()
    Hs = X.T @ X
    gram_s = time.perf_counter() - t0
    del Hs, X
    per = r["swap_s"]
    s_per_swap = sum(per) / max(len(per), 1)
    return {"value": 1.0 / max(s_per_swap, 1e-9), "unit": UNIT, "cores": torch.get_num_threads(), "kind": "oracle",
            "sample": (f"fp64 NumPy oracle (low-rank-update mode) at the layer's own size (d1={wl.d1}, m={wl.m}, k={wl.k}) on the device's H and G: "
                       f"{len(per)} swaps, {s_per_swap:.2f} s per swap, after a fresh fp64 solve of the start state ({r['setup_s']:.1f} s, not counted)"),
            "s_per_swap": s_per_swap, "setup_s": r["setup_s"],
            "gram_fp64": {"rows": rows, "seconds": gram_s, "scale_to_layer": wl.n / rows,
                          "layer_seconds_extrapolated": gram_s * wl.n / rows}}


def other_configs(pkg, b, solver, dev, with_cpu):
    """The other named layers, one warm-up and one timed solve each (outside the headline's timed region), and, with
    `with_cpu`, seconds per step of the strict oracle (fresh Cholesky solve per step) on the device's H and G."""
    import numpy as np
    from threadpoolctl import threadpool_limits
    import contextlib
    out = {}
    for name, strict_steps in (("c1", 4), ("c2", 1), ("c3", 2), ("c4", 2), ("c6", 4)):
        wl = workloads.config(name)
        W = wl.weight(dev)
        x = [wl.x_chunk(c, dev) for c in range(wl.n_chunks)]
        pair = wl.score_mode == "pair_exact"
        kw = dict(damp=wl.damp, accept_rel_tol=wl.eps_acc, score_mode=b.SCORE_PAIR_EXACT if pair else b.SCORE_INDEPENDENT)
        pkg.solve_layer(solver, x, W, wl.g, wl.k, wl.max_swaps, **kw)
        f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        f0.record()
        r = pkg.solve_layer(solver, x, W, wl.g, wl.k, wl.max_swaps, **kw)
        f1.record()
        torch.cuda.synchronize()
        nI, nJ = wl.k * wl.g, wl.d1 - wl.k * wl.g
        fused = wl.g == 1 and not pair
        loop_s = r.ms["search_loop"] * 1e-3
        rec = {"workload": workload_label(wl, wl.max_swaps), "layer_solve_s": f0.elapsed_time(f1) / 1e3, "swaps": r.n_swaps,
               "stop_reason": r.stop_reason, "phases_ms": r.ms, "loop_driver": r.loop_driver, "batches": r.n_batches,
               "swaps_per_s": r.n_swaps / max(loop_s, 1e-9) if r.n_swaps else 0.0,
               "loop_gbs": swap_bytes(nI, nJ, wl.m, fused, fused and r.loop_driver == "launches", r.n_swaps / max(r.n_batches, 1) if r.loop_driver == "delayed" else 0.0) * r.n_swaps / max(loop_s, 1e-9) / 1e9 if r.n_swaps else 0.0}
        if name == "c3":        # no improving swap from the energy start: the paper's fixed-iteration form gives the step time
            rf = pkg.solve_layer(solver, x, W, wl.g, wl.k, 8, accept_mode=b.ACCEPT_ALWAYS, **kw)
            rec["forced_swaps"] = {"swaps": rf.n_swaps, "ms_per_swap": rf.ms["search_loop"] / max(rf.n_swaps, 1)}
        if with_cpu:
            H64 = r.H.cpu().numpy().astype(np.float64); G64 = r.G.cpu().numpy().astype(np.float64)
            ctxm = threadpool_limits(1) if wl.d1 <= 3000 else contextlib.nullcontext()
            with ctxm:
                per = strict_step_seconds(H64, G64, r.const_term, wl, strict_steps, "pair_exact" if pair else "independent")
            rec["cpu_strict_oracle"] = {"steps": len(per), "s_per_step": sum(per) / max(len(per), 1),
                                        "cores": 1 if wl.d1 <= 3000 else torch.get_num_threads(),
                                        "what": "strict fp64 oracle (fresh Cholesky solve per step) on the device's H and G"}
            del H64, G64
        out[name] = rec
        del x, W, r
        torch.cuda.empty_cache()
    return out


# ------------------------------------------------------------------------------------------ our arm
def run_ours(args):
    rank, world, local = dist_env()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py: no CUDA device; the solve has no CPU path")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    import paper_2403_12983_b200 as pkg
    from paper_2403_12983_b200 import binding as b

    over = {}
    if args.tokens:
        over["n"] = args.tokens
    for key in ("d1", "m", "k"):
        if getattr(args, key) is not None:
            over[key] = getattr(args, key)
    wl = workloads.config(args.workload, seed=rank, **over)
    max_swaps = args.max_swaps if args.max_swaps is not None else wl.max_swaps
    accept = b.ACCEPT_ALWAYS if args.accept_always else b.ACCEPT_IMPROVING
    solver = pkg.Solver(local)
    W = wl.weight(dev)
    x_dev = [wl.x_chunk(c, dev) for c in range(wl.n_chunks)]          # inputs resident in HBM
    torch.cuda.synchronize()
    H = torch.empty(wl.d1, wl.d1, dtype=torch.float32, device=dev)
    G = torch.empty(wl.d1, wl.m, dtype=torch.float32, device=dev)
    nI, nJ, m = wl.k * wl.g, wl.d1 - wl.k * wl.g, wl.m

    shard = args.shard and wl.g == 1 and wl.score_mode != "pair_exact" and args.block_pairs <= 1 and not args.greedy
    if shard:
        # one layer over all ranks: every rank keeps its columns of W and its token chunks (same seed everywhere)
        from paper_2403_12983_b200 import sharding
        wl = workloads.config(args.workload, seed=0, **over)
        W_full = wl.weight(dev)
        c0, c1 = sharding.column_range(wl.m, rank, world)
        W = W_full[:, c0:c1].contiguous()
        del W_full
        x_dev = [wl.x_chunk(c, dev) for c in sharding.chunk_indices(wl.n_chunks, rank, world)]
        m = c1 - c0
        G = None
        if world > 1:
            import torch.distributed as dist
            hook = sharding.dist_reduce_hook()
            reduce_H = lambda Hm: dist.all_reduce(Hm)
        else:
            hook = lambda view, sptr: None
            reduce_H = lambda Hm: None

    def step(x_chunks, W_in, prof=0):
        if shard:
            return sharding.solve_layer_sharded(solver, x_chunks, W_in, wl.d1, wl.g, wl.k, max_swaps, hook, reduce_H, damp=wl.damp,
                                                accept_mode=accept, accept_rel_tol=wl.eps_acc, H=H)
        return pkg.solve_layer(solver, x_chunks, W_in, wl.g, wl.k, max_swaps, damp=wl.damp, accept_mode=accept, accept_rel_tol=wl.eps_acc,
                               score_mode=b.SCORE_PAIR_EXACT if wl.score_mode == "pair_exact" else b.SCORE_INDEPENDENT,
                               profile_samples=prof, H=H, G=G, greedy_t_hat=args.greedy, block_pairs=args.block_pairs,
                               loop_mode=args.loop_mode)

    def barrier():
        if world > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()

    for _ in range(args.warmup):
        res = step(x_dev, W)
    # ---------------- device-resident timing
    sampler = ClockSampler(local)
    barrier()
    sampler.start()
    launches0 = b.launch_count()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    phase = {"gram": 0.0, "gram_end": 0.0, "init": 0.0, "search": 0.0, "search_loop": 0.0}
    kern = {}
    swaps = 0
    e0.record()
    for _ in range(args.steps):
        res = step(x_dev, W)
        for key in phase:
            phase[key] += res.ms[key]
        swaps += res.n_swaps
    e1.record()
    barrier()
    launches = b.launch_count() - launches0
    clocks = sampler.stop()
    total_ms = e0.elapsed_time(e1)
    K = max(args.steps, 1)
    # phase / kernel times of a step come from one more solve outside the timed region (the launch-chain driver records
    # events around sampled steps, the delayed loop around the parts of its first batches; the persistent loop reads the device
    # clock at its barriers)
    prof_res = step(x_dev, W, prof=8)
    for key, val in prof_res.ms_kernel.items():
        kern[key] = val * K

    # ---------------- the same layer with the paper's larger local-search steps (outside the timed region above)
    block_extra = None
    if world == 1 and not shard and args.block_pairs <= 1 and not args.no_block_extra and wl.g * 16 <= 96 and wl.score_mode != "pair_exact":
        block_extra = []
        for s_pairs in (16, 50):
            if s_pairs * wl.g > 96 or s_pairs > min(wl.k, wl.ngroups - wl.k):
                continue
            f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            for rep in range(2):          # the first solve warms this code path up (attributes, first-touch of the panels)
                torch.cuda.synchronize()
                f0.record()
                rb = pkg.solve_layer(solver, x_dev, W, wl.g, wl.k, max_swaps, damp=wl.damp, accept_mode=accept,
                                     accept_rel_tol=wl.eps_acc, H=H, G=G, block_pairs=s_pairs)
                f1.record()
                torch.cuda.synchronize()
            block_extra.append({"pairs_per_iteration": s_pairs, "swaps": rb.n_swaps, "iterations": rb.n_swaps // s_pairs,
                                "layer_solve_s": f0.elapsed_time(f1) / 1e3, "search_ms": rb.ms["search"],
                                "swaps_per_s": rb.n_swaps / max(rb.ms["search"] * 1e-3, 1e-9),
                                "obj_init": rb.obj_init, "obj_final": rb.obj_final, "stop_reason": rb.stop_reason})

    # ---------------- end to end: host buffers, copies inside the timed region
    e2e = None
    if not args.no_e2e and not shard:
        try:
            x_host = [c.to("cpu").pin_memory() for c in x_dev]
            W_host = W.to("cpu").pin_memory()
            pinned = {"W": torch.empty(wl.d1, wl.m, dtype=torch.float32).pin_memory()}
            del x_dev
            torch.cuda.empty_cache()
            r = step(x_host, W_host)                         # warm-up of the copy path
            pkg.result_to_host(r, pinned)
            barrier()
            f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e_swaps, e_search, h2d, d2h = 0, 0.0, 0, 0
            nrep = max(1, min(K, 2))
            f0.record()
            for _ in range(nrep):
                r = step(x_host, W_host)
                back = pkg.result_to_host(r, pinned)
                e_swaps += r.n_swaps; h2d += r.io["h2d"]; d2h += back["bytes"]
            f1.record()
            barrier()
            e_ms = f0.elapsed_time(f1)
            e2e = {"ms_per_step": e_ms / nrep, "swaps": e_swaps, "h2d": h2d // nrep, "d2h": d2h // nrep}
        except RuntimeError as exc:                           # e.g. pinned allocation refused
            e2e = {"error": str(exc)[:200]}

    if shard and world > 1:
        swaps = swaps / world          # every rank reports the swaps of the one shared layer
    red = reduce_over_ranks({"max_total_ms": total_ms, "sum_swaps": swaps, "max_search_ms": phase["search_loop"],
                             "max_e2e_ms": (e2e or {}).get("ms_per_step", 0.0), "sum_e2e_swaps": (e2e or {}).get("swaps", 0)},
                            world, dev)
    if rank != 0:
        if world > 1:
            torch.distributed.destroy_process_group()
        return

    pk = peaks()
    # bf16 activations: one MMA per product; fp32 activations: three digits, eight digit products executed per product
    gram_terms = 1 if wl.x_dtype == torch.bfloat16 else 8
    ms_step = red["max_total_ms"] / K
    search_s = red["max_search_ms"] / 1e3
    value = red["sum_swaps"] / max(search_s, 1e-9)
    # dominant kernel among the streaming kernels of a swap, and the Gram kernel, by share of the step
    kern_avg = {k2: v / K for k2, v in kern.items()}
    per_step_swaps = swaps / K
    shares = {k2: v * (prof_res.n_batches or per_step_swaps / max(args.block_pairs, 1)) for k2, v in kern_avg.items()}
    shares["gram_tcgen05"] = phase["gram"] / K
    dom = max(shares, key=shares.get) if shares else "gram_tcgen05"
    fused_path = wl.g == 1 and wl.score_mode != "pair_exact" and args.block_pairs <= 1
    loop_ms = phase["search_loop"] / K
    # delayed updates: matrices are read once per batch, and the Gram is the largest kernel
    delayed = fused_path and res.loop_driver == "delayed"
    per_batch = res.n_swaps / max(res.n_batches, 1) if delayed else 0.0
    if fused_path and not delayed and loop_ms > 0 and loop_ms >= phase["gram"] / K:
        # the swap loop is the dominant kernel: one cooperative launch per solve (or its six-launch-per-step form),
        # timed by the library with CUDA events on its own stream around the loop
        persistent = res.loop_driver == "persistent"
        bytes_per_launch = swap_bytes(nI, nJ, m, True, not persistent and not (shard and world > 1)) * (swaps / K)
        ach = bytes_per_launch / (loop_ms * 1e-3) / 1e9
        roof = {"kernel": "k_swap_loop_g1 (persistent cooperative loop, one launch per solve)" if persistent
                          else "swap loop as six launches per step (k_lz_decide, k_lz_hpass, k_lz_rows, k_lz_finish, k_lz_select, k_lz_y)",
                "bound": "hbm", "achieved": ach, "peak": pk["hbm_gbs"], "unit": "GB/s", "frac": ach / pk["hbm_gbs"],
                "traffic": None,
                "bytes_per_launch": int(bytes_per_launch), "ms_per_launch": loop_ms,
                "bytes_per_swap": swap_bytes(nI, nJ, m, True, not persistent and not (shard and world > 1)), "peak_source": pk["source"]}
    elif dom in KERNEL_BYTES and kern_avg.get(dom, 0) > 0:
        bytes_per_launch = KERNEL_BYTES[dom](nI, nJ, m)
        ach = bytes_per_launch / (kern_avg[dom] * 1e-3) / 1e9
        roof = {"kernel": dom, "bound": "hbm", "achieved": ach, "peak": pk["hbm_gbs"], "unit": "GB/s",
                "frac": ach / pk["hbm_gbs"], "traffic": None,
                "bytes_per_launch": bytes_per_launch,
                "ms_per_launch": kern_avg[dom], "peak_source": pk["source"]}
    else:
        tm_, tn_ = -(-wl.d1 // 128), -(-wl.d1 // 256)
        tiles = sum(tn_ - t // 2 for t in range(tm_))
        flops = 2.0 * 128 * 256 * tiles * wl.n * gram_terms
        ach = flops / (phase["gram"] / K * 1e-3) / 1e12
        roof = {"kernel": "k_mma_pipe<GRAM>", "bound": "tensor", "achieved": ach, "peak": pk["bf16_tflops_sustained"],
                "unit": "TFLOP/s", "frac": ach / pk["bf16_tflops_sustained"], "traffic": None,
                "flops_per_step": flops, "peak_source": pk["source"] + " (sustained)"}
    tm_, tn_ = -(-wl.d1 // 128), -(-wl.d1 // 256)
    tiles = sum(tn_ - t // 2 for t in range(tm_))
    gram_exec_tflops = 2.0 * 128 * 256 * tiles * wl.n * gram_terms / max(phase["gram"] / K * 1e-3, 1e-12) / 1e12
    fused = wl.g == 1 and wl.score_mode != "pair_exact"
    lazy = fused_path and res.loop_driver == "launches" and not (shard and world > 1)
    if args.block_pairs > 1:     # one pass over every matrix per ITERATION, plus the read of V and R for the scores
        it_bytes = swap_bytes(nI, nJ, m, False) + 4 * (nI + nJ) * m
        loop_gbs = it_bytes * (per_step_swaps / args.block_pairs) / max(phase["search_loop"] / K * 1e-3, 1e-12) / 1e9
    else:
        loop_gbs = swap_bytes(nI, nJ, m, fused, lazy, per_batch) * per_step_swaps / max(phase["search_loop"] / K * 1e-3, 1e-12) / 1e9
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_step, "higher_is_better": True, "scaling": "strong" if shard and world > 1 else "weak", "vs_baseline": None,
        "dtype": "f32 (bf16 tensor-core Gram, fp32 accumulate)" if wl.x_dtype == torch.bfloat16
                 else "f32 (Gram as a three-term bf16 split on the tensor cores, fp32 accumulate)", "data": "synthetic",
        "config": {"workload": workload_label(wl, max_swaps, args.accept_always, args.greedy, args.block_pairs),
                   },
        "notes": {"l2": "inputs larger than L2 (X, H and the search state are each > 126 MB)" if wl.d1 >= 8192 else
                        "state smaller than L2; numbers are cache-resident",
                  "replicas": 1 if shard else world, "column_shards": world if shard else 1, "loop_driver": res.loop_driver},
        "clocks": clocks,
        "layer_solve_s": ms_step / 1e3,
        "swaps_per_step": per_step_swaps, "stop_reason": res.stop_reason,
        "obj_init": res.obj_init, "obj_final": res.obj_final,
        "phases_ms": {k2: v / K for k2, v in phase.items()},
        "kernel_ms": kern_avg,
        "gram": {"executed_tflops": gram_exec_tflops, "dense_equiv_tflops": 2.0 * wl.n * wl.d1 ** 2 / max(phase["gram"] / K * 1e-3, 1e-12) / 1e12,
                 "executed_mma_per_product": gram_terms,
                 "frac_of_bf16_peak": gram_exec_tflops / pk["bf16_tflops_sustained"], "peak": pk["bf16_tflops_sustained"],
                 "peak_source": pk["source"] + " (sustained)"},
        "swap_loop": {"gbs": loop_gbs, "bytes_per_swap": swap_bytes(nI, nJ, m, fused, lazy, per_batch), "swaps_per_batch": per_batch, "frac_of_hbm": loop_gbs / pk["hbm_gbs"],
                      "peak": pk["hbm_gbs"], "peak_source": pk["source"]},
        "roofline": roof,
        "gpu_launches": int(launches),
    }
    if e2e and "ms_per_step" in e2e:
        e_val = red["sum_e2e_swaps"] / max(min(K, 2), 1) / max(red["max_e2e_ms"] * 1e-3, 1e-9)
        out["e2e"] = {"value": e_val, "unit": UNIT, "what": "swaps per second of whole-solve time, host buffers", "ms_per_step": red["max_e2e_ms"],
                      "h2d_bytes_per_step": e2e["h2d"], "d2h_bytes_per_step": e2e["d2h"]}
    else:
        out["e2e"] = {"value": None, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0,
                      "note": (e2e or {}).get("error", "skipped")}
    if block_extra:
        out["block_exchange"] = block_extra
    if world == 1 and not shard and not args.no_other_configs and args.workload == "c5":
        out["other_configs"] = other_configs(pkg, b, solver, dev, with_cpu=not args.no_cpu)
    if world == 1 and not shard and not args.no_cpu:
        out["cpu_baseline"] = cpu_baseline_at_size(wl, H, G, res.const_term)
    print(json.dumps(out))
    if world > 1:
        torch.distributed.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="c5")
    ap.add_argument("--tokens", type=int, default=None, help="override the number of calibration rows")
    ap.add_argument("--d1", type=int, default=None, help="override the layer width (profiling cases)")
    ap.add_argument("--m", type=int, default=None)
    ap.add_argument("--k", type=int, default=None)
    ap.add_argument("--max-swaps", type=int, default=None)
    ap.add_argument("--greedy", type=int, default=0, help="start from the nested phase of Algorithm 1 with this t_hat")
    ap.add_argument("--block-pairs", type=int, default=0, help="groups exchanged per iteration (t_hat = 2 s, p_hat = 0); 0 = single swaps")
    ap.add_argument("--no-block-extra", action="store_true", help="skip the extra solves with block exchanges of 16 and 50 groups")
    ap.add_argument("--accept-always", action="store_true", help="paper-literal fixed number of iterations")
    ap.add_argument("--loop-mode", type=int, default=0, help="0 auto, 1 persistent cooperative loop, 2 a chain of launches per step (single-row groups)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--shard", action="store_true", help="with --gpus N: ONE layer over all ranks (token-split Gram, column-sharded "
                    "swap search with two all-reduces per swap) instead of N independent replicas")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-other-configs", action="store_true", help="skip the extra solves of c1, c2, c3, c4 and c6")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
