"""Large frontiers, where a warp reserves its output slots in runs and leaves
holes behind: an exhaustive search evaluates every composition exactly once,
and its plan is the one that the pruned searches find; children that fit the
capacity fit whatever holes the runs leave; and a batch that runs out of slots
while runs are open is finished exactly.  A search keeps its work buffers (here
up to 25 GB), so each check is a process of its own."""
import math
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu


def workload(L, S, M):
    """One slice (every stage on one type), memory never binding."""
    import gen
    w = gen.config3()
    w.L = L
    for n in ("fwd", "bwd", "dsync", "mem_w", "mem_a"):
        setattr(w, n, getattr(w, n)[:, :L].copy())
    w.S, w.M_list, w.placement, w.type_counts = S, [M], 1, [S, 0]
    w.mem_w, w.mem_a = w.mem_w // 1024, w.mem_a // 1024
    return w


def few_completions():
    """Four heavy layers at the end: the bound cuts a plan with two of them in
    one stage, so most prefixes of 13 of the 15 stages, the largest frontier,
    have no completion."""
    w = workload(29, 15, 20)
    w.fwd[:, :-4] //= 50
    w.bwd[:, :-4] //= 50
    return w


def prefixes(L, S, x):
    """Placements of x stages that leave a layer for each of the other S - x."""
    return math.comb(L - S + x, x)


def check_1f1b_runs():
    import gen
    import paper_2609_06086_gb300 as P
    L, S = 36, 10
    w = workload(L, S, 12)
    n_map = gen.n_compositions(L, S)
    prob, keep = P.make_problem(w, warmup=0, prune=0, frontier_cap=n_map + 4_000_000)
    plan, st = P.poseidon_search(prob)
    assert st["reruns"] == 0 and st["evaluated"] == st["leaves"] == n_map
    assert st["prefixes"] == sum(prefixes(L, S, x) for x in range(1, S - 1))
    assert st["parents_complete"] == prefixes(L, S, S - 2)
    for prune in (1, 2):
        prob, keep = P.make_problem(w, warmup=100, prune=prune)
        assert P.poseidon_search(prob)[0] == plan


def check_interleaved_runs():
    import gen
    import paper_2609_06086_gb300 as P
    L, N, V = 34, 5, 2
    J = N * V
    w = workload(L, N, 10)
    n_map = gen.n_compositions(L, J)
    sched = P.binding.POS_SCHED_INTERLEAVED_1F1B
    prob, keep = P.make_problem(w, warmup=0, prune=0, schedule=sched, V=V,
                                frontier_cap=8 * prefixes(L, J, J - 2))
    plan, st = P.poseidon_search(prob)
    assert st["leaves"] == n_map and st["evaluated"] == n_map + 1  # and the slice's seed
    assert st["prefixes"] == sum(prefixes(L, J, x) for x in range(1, J - 1))
    prob, keep = P.make_problem(w, warmup=0, prune=2, schedule=sched, V=V)
    assert P.poseidon_search(prob)[0] == plan


def check_exact_fit():
    """The largest frontier has 14.8 million entries, from 9.6 million parents
    by warps that open runs of 512 slots: a capacity of exactly that many
    entries still holds them."""
    import paper_2609_06086_gb300 as P
    w = few_completions()
    prob, keep = P.make_problem(w, warmup=100_000, prune=1)
    plan, st = P.poseidon_search(prob)
    children = st["children_depth"][:w.S - 1]
    assert st["reruns"] == 0 and 9_000_000 < children[-3] < max(children) == children[-2] < 1 << 24
    prob, keep = P.make_problem(w, warmup=100_000, prune=1, frontier_cap=max(children))
    again, st = P.poseidon_search(prob)
    assert st["reruns"] == 0 and st["children_depth"][:w.S - 1] == children
    assert again == plan


def check_no_room_with_open_runs():
    """Slots run out while warps have open runs: at an expansion level, and at
    the completion level of an exhaustive search.  What the pipelined pass wrote
    is evaluated once, holes are not, and the batch is run again exactly."""
    import gen
    import paper_2609_06086_gb300 as P
    w = few_completions()
    prob, keep = P.make_problem(w, warmup=100_000, prune=1)
    want, _ = P.poseidon_search(prob)
    for cap in (11_000_000, 12_345_678):
        prob, keep = P.make_problem(w, warmup=100_000, prune=1, frontier_cap=cap)
        plan, st = P.poseidon_search(prob)
        assert st["reruns"] == 1 and st["evaluated"] == st["leaves"] + st["warmup_evaluated"]
        assert plan == want, cap
    L, S = 36, 10
    w = workload(L, S, 12)
    prob, keep = P.make_problem(w, warmup=100, prune=1)
    want, _ = P.poseidon_search(prob)
    prob, keep = P.make_problem(w, warmup=0, prune=0, frontier_cap=prefixes(L, S, S - 2) + 1_000_000)
    plan, st = P.poseidon_search(prob)
    # the completion level alone overflowed: its parents all fit
    assert prefixes(L, S, S - 2) > 15_000_000 and st["reruns"] == 1
    assert gen.n_compositions(L, S) < st["evaluated"] == st["leaves"]
    assert plan == want


def in_child(check):
    r = subprocess.run([sys.executable, os.path.abspath(__file__), check], capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr


def test_1f1b_runs():
    in_child("check_1f1b_runs")


def test_interleaved_runs():
    in_child("check_interleaved_runs")


def test_exact_fit():
    in_child("check_exact_fit")


def test_no_room_with_open_runs():
    in_child("check_no_room_with_open_runs")


if __name__ == "__main__":
    sys.path.insert(0, ROOT)
    globals()[sys.argv[1]]()
