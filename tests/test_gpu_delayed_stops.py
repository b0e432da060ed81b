"""How the swap loop with delayed updates ends: stops between rebuilds, a wait that runs out, scores that are not finite, ties; what it reports."""
import pytest
import torch

import paper_2403_12983_b200 as pkg
from paper_2403_12983_b200 import binding as b
from tests.test_gpu_refresh_stop import _check, _problem
from tests.test_gpu_refresh_stop import test_weights_when_a_search_stops_between_rebuilds as check_stops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [64, 41])
def test_weights_when_a_delayed_search_stops_between_rebuilds(m):
    check_stops(m, 1, 150, 300, b.LOOP_DELAYED, 0)


def test_barrier_that_runs_out_is_a_status_and_the_context_goes_on():
    H, G, W = _problem(300, 64, 1)
    solver = pkg.Solver(0)
    solver.init_support(H, G, W, 1, 150, b.INIT_MAGNITUDE)
    with pytest.raises(pkg.OsscarError) as e:
        solver.local_search(40, loop_mode=b.LOOP_DELAYED, wait_limit_cycles=4)
    assert e.value.status == b.E_TIMEOUT
    solver.init_support(H, G, W, 1, 150, b.INIT_MAGNITUDE)
    out = solver.local_search(40, accept_mode=b.ACCEPT_ALWAYS, loop_mode=b.LOOP_DELAYED)
    assert out.n_swaps == 40 and out.loop_driver == "delayed"
    _check(out, H, G, W, 1)
    solver.close()


def test_refused_search_leaves_the_wait_budget_as_it_was():
    H, G, W = _problem(432, 64, 9)
    solver = pkg.Solver(0)
    for mode in (b.LOOP_PERSISTENT, b.LOOP_DELAYED):
        solver.init_support(H, G, W, 9, 24, b.INIT_MAGNITUDE)
        with pytest.raises(pkg.OsscarError) as e:                # loops of single-row groups
            solver.local_search(4, loop_mode=mode, wait_limit_cycles=4)
        assert e.value.status == b.E_ARG
        solver.init_support(H, G, W, 1, 216, b.INIT_MAGNITUDE)
        assert solver.local_search(12, accept_mode=b.ACCEPT_ALWAYS, loop_mode=mode).n_swaps == 12
    solver.close()


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_groups_without_a_finite_score_stay_where_they_are(value):
    H, G, W = _problem(300, 64, 1)
    solver = pkg.Solver(0)
    S = solver.init_support(H, G, W, 1, 150, b.INIT_MAGNITUDE)[0]
    pruned = [q for q in range(300) if q not in set(S.tolist())]
    bad = torch.tensor(pruned[3:140:9], device="cuda")
    Gb = G.clone()
    Gb[bad, 5] = value                              # their residual has no finite norm
    solver.set_const_term(1e9)
    outs = []
    # (the cooperative loop takes its first entering group from all scores and ends the search at an infinite one)
    for mode in (b.LOOP_DELAYED, b.LOOP_LAUNCHES):
        solver.init_support(H, Gb, W, 1, 150, b.INIT_USER, S)
        outs.append(solver.local_search(40, accept_mode=b.ACCEPT_ALWAYS, loop_mode=mode))
    for o in outs:
        assert o.n_swaps == 40 and torch.equal(o.swap_trace, outs[0].swap_trace)
        assert not set(bad.tolist()) & set(o.support.tolist())
        assert torch.isfinite(o.W).all()
    allbad = G.clone()
    allbad[torch.tensor(pruned, device="cuda")] = value
    for mode in (b.LOOP_DELAYED, b.LOOP_PERSISTENT, b.LOOP_LAUNCHES):
        solver.init_support(H, allbad, W, 1, 150, b.INIT_USER, S)
        o = solver.local_search(40, accept_mode=b.ACCEPT_ALWAYS, loop_mode=mode)
        assert (o.n_swaps, o.stop_reason) == (0, "guard") and torch.equal(o.support, S)
    solver.set_const_term(0.0, False)
    solver.close()


def test_ties_go_to_the_smaller_group():
    """All rows alike and most of them zero: more equal scores than a batch has candidates."""
    d1, k = 400, 190
    H = torch.eye(d1, device="cuda") * 3
    G = torch.zeros(d1, 32, device="cuda")
    G[:7] = 1.5
    S = torch.arange(5, 5 + k, dtype=torch.int32)
    solver = pkg.Solver(0)
    outs = []
    for mode in (b.LOOP_DELAYED, b.LOOP_PERSISTENT):
        solver.init_support(H, G, G / 3, 1, k, b.INIT_USER, S)
        outs.append(solver.local_search(60, accept_mode=b.ACCEPT_ALWAYS, loop_mode=mode))
    solver.close()
    assert outs[0].n_swaps == 60 and torch.equal(outs[0].swap_trace, outs[1].swap_trace)


def test_parts_of_the_first_batches_are_timed():
    H, G, W = _problem(300, 64, 1)
    solver = pkg.Solver(0)
    for samples, swaps in ((2, 60), (8, 20), (0, 20)):
        solver.init_support(H, G, W, 1, 150, b.INIT_MAGNITUDE)
        out = solver.local_search(swaps, accept_mode=b.ACCEPT_ALWAYS, profile_samples=samples)
        assert out.loop_driver == "delayed" and out.n_batches >= 1
        assert list(out.ms_kernel) == (b.STEP_KERNELS_DELAYED if samples else [])
        assert all(v > 0 for v in out.ms_kernel.values()) and sum(out.ms_kernel.values()) <= out.ms_search
    solver.close()
