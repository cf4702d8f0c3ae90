"""Unranking in the decode pass: the ranks around every binomial that a
stage's layer count is found from, for the smallest and largest layer counts
and stage counts, against the oracle.  The handle's schedule is Interleaved
1F1B, whose batches of every size take that pass."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _ranks(L, J):
    """Ranks whose first Y = C(L-1, J-1) - rank is C(j, J-1) or one more, the
    first and the last, and a few in between."""
    k, n = J - 1, math.comb(L - 1, J - 1)
    ys = {1, n, n // 2 + 1, n - n // 3}
    for j in range(k, L):
        ys |= {math.comb(j, k), math.comb(j, k) + 1}
    return [n - y for y in sorted(ys) if 1 <= y <= n]


@pytest.mark.parametrize("n_types", [1, 4])  # 4 types x 8 TP indices: no memory-limit table
@pytest.mark.parametrize("L", [1, 2, 9, 33, 64, 80, 127])
def test_ranks_at_the_binomials(L, n_types):
    import gen
    import oracle
    import paper_2609_06086_gb300 as P
    from gpu_util import eval_device
    n_tp = 1 if n_types == 1 else 8
    K = n_types * n_tp
    rng = np.random.default_rng(L)
    tab = dict(L=L, n_types=n_types, n_tp=n_tp, fwd=rng.integers(1, 1000, (K, L)),
               bwd=rng.integers(1, 2000, (K, L)), dsync=rng.integers(0, 3000, (K, L)),
               p2p_f=rng.integers(0, 50, (K, K)), p2p_b=rng.integers(0, 50, (K, K)),
               mem_w=rng.integers(0, 100, (K, L)), mem_a=rng.integers(0, 20, (K, L)),
               cap=rng.integers(60 * L, 120 * L, K))
    rows = []
    for S in range(1, min(L, 16) + 1):
        rows += [(r, int(rng.integers(n_types)), S, S + 3, 0, 0) for r in _ranks(L, S)]
    for N, V in ((1, 2), (1, 16), (2, 4), (3, 3), (4, 4), (5, 3)):
        if N * V <= L:
            rows += [(r, 0, N, 2 * N, 0, V) for r in _ranks(L, N * V)]
    c = np.array(rows, dtype=gen.CANDIDATE_DTYPE)
    c = c[rng.permutation(len(c))]
    T_ref, F_ref = oracle.eval_batch(oracle.OracleTables(**tab, schedule=2), c)
    h = P.Handle(P.Tables(**tab), 2)
    T, F = eval_device(P, h, c)
    h.close()
    bad = np.flatnonzero((T != T_ref) | (F != F_ref))
    assert len(bad) == 0, (len(bad), c[bad[:5]], T[bad[:5]], T_ref[bad[:5]])
