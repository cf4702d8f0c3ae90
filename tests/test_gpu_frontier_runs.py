"""Large frontiers, where a warp reserves its output slots in runs and leaves
holes behind: an exhaustive search evaluates every composition exactly once,
and its plan is the one that the pruned searches find."""
import math

import pytest

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


def prefixes(L, S, x):
    """Placements of x stages that leave a layer for each of the other S - x."""
    return math.comb(L - S + x, x)


def test_1f1b_runs():
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


def test_interleaved_runs():
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
