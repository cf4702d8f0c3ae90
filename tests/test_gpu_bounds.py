"""The makespan kernels end a plan's steady steps when an upper and a lower
bound of its makespan meet, and put plans whose bounds stay apart on a queue
of their warp.  Cost tables where the bounds meet at once, late and never
(ties, near-ties, transfers that dominate, zero costs), at the fewest steady
steps and the most micro-batches, in batches small enough for one group of
plans per warp and large enough for the queue, against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TABLES = ["ties", "near_ties", "transfers", "zeros", "spread"]


def tables(kind, L, rng):
    """Two types, one TP degree; memory plays no part here."""
    K = 2
    f = np.full((K, L), 100)
    b = np.full((K, L), 200)
    d = np.zeros((K, L), int)
    p = np.zeros((K, K), int)
    if kind == "near_ties":
        f, b = f * 1000 + rng.integers(0, 3, (K, L)), b * 1000 + rng.integers(0, 3, (K, L))
        p = rng.integers(0, 50, (K, K))
    elif kind == "transfers":
        f, b = rng.integers(1, 20, (K, L)), rng.integers(1, 20, (K, L))
        p = rng.integers(500, 1500, (K, K))
        d = rng.integers(0, 4000, (K, L))
    elif kind == "zeros":
        f, b = rng.integers(0, 2, (K, L)), rng.integers(0, 2, (K, L))
        f[:, : L // 2] = 0
    elif kind == "spread":
        f, b = rng.integers(1, 60_000, (K, L)), rng.integers(1, 120_000, (K, L))
        p = rng.integers(0, 80_000, (K, K))
        d = rng.integers(0, 500_000, (K, L))
    one = np.ones((K, L), np.int64)
    return dict(L=L, n_types=K, n_tp=1, fwd=f, bwd=b, dsync=d, p2p_f=p, p2p_b=p.T.copy(),
                mem_w=one, mem_a=one, cap=np.full(K, 3 * L, np.int64))


@pytest.mark.parametrize("sched", [0, 1])
@pytest.mark.parametrize("kind", TABLES)
def test_bounds_and_queue(kind, sched):
    import gen
    import oracle
    import paper_2609_06086_gb300 as P
    from gpu_util import eval_device
    rng = np.random.default_rng(TABLES.index(kind))
    L = 48
    tab = tables(kind, L, rng)
    cands = gen.random_candidates(6000, L=L, n_types=2, S_range=(1, 16), M_range=(1, 255), seed=3)
    # a third of them with 0..3 steady steps
    first = cands["S"].astype(int) * (1 if sched == 0 else 2) - (0 if sched == 0 else 1)
    few = np.arange(len(cands)) % 3 == 0
    cands["M"][few] = np.clip(first + rng.integers(0, 4, len(cands)), 1, 255)[few]
    T_ref, F_ref = oracle.eval_batch(oracle.OracleTables(**tab, schedule=sched), cands)
    h = P.Handle(P.Tables(**tab), sched)
    for n in (len(cands), 1_500_000):
        pick = rng.integers(0, len(cands), n) if n > len(cands) else np.arange(n)
        T, F = eval_device(P, h, cands[pick])
        bad = np.flatnonzero((T != T_ref[pick]) | (F != F_ref[pick]))
        assert len(bad) == 0, (n, len(bad), cands[pick[bad[:3]]], T[bad[:3]], T_ref[pick[bad[:3]]])
    h.close()
