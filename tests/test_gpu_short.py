"""Short pipelines (M < S under 1F1B, M < 2S-1 under Eager 1F1B): every
(S, M), and the first M beyond, against the oracle, in a batch of the
lane-per-stage kernel and, repeated, in one of the sorted path's kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_stage", [False, True])
@pytest.mark.parametrize("sched", [0, 1])
def test_every_short_pipeline(sched, per_stage):
    import gen
    import oracle
    import paper_2609_06086_gb300 as P
    from gpu_util import SORTED, eval_device, eval_device_ex, repeated
    w = gen.config4(seed=5)
    rng = np.random.default_rng(sched)
    tab = w.tables_dict()
    tab["dsync"] = rng.integers(0, 2_000_000, tab["dsync"].shape)
    tab["p2p_f"] = rng.integers(0, 200_000, tab["p2p_f"].shape)
    tab["p2p_b"] = rng.integers(0, 200_000, tab["p2p_b"].shape)
    pairs = [(S, M) for S in range(1, 17) for M in range(1, (S if sched == 0 else 2 * S - 1) + 1)]
    reps = 6
    n = len(pairs) * reps
    if per_stage:
        c = gen.per_stage_tp_candidates(n, w.L, w.n_types, w.n_tp, seed=9, S_range=(16, 16))
    else:
        c = gen.random_candidates(n, L=w.L, n_types=w.n_types, S_range=(16, 16), seed=9)
        c["tp_idx"] = rng.integers(0, w.n_tp, n)
    SM = np.repeat(np.array(pairs), reps, axis=0)
    c["S"], c["M"] = SM[:, 0], SM[:, 1]
    c["map_rank"] %= np.array([gen.n_compositions(w.L, S) for S in SM[:, 0]], np.uint64)
    c = c[rng.permutation(n)]
    ot = oracle.OracleTables(**tab, schedule=sched)
    T_ref, F_ref = (oracle.eval_batch_ex if per_stage else oracle.eval_batch)(ot, c)
    h = P.Handle(P.Tables(**tab), sched)
    for pick in (np.arange(n), repeated(n, SORTED)):
        T, F = (eval_device_ex if per_stage else eval_device)(P, h, c[pick])
        bad = np.flatnonzero((T != T_ref[pick]) | (F != F_ref[pick]))
        assert len(bad) == 0, (len(pick), len(bad), c[pick[bad[:5]]], T[bad[:5]],
                               T_ref[pick[bad[:5]]])
    h.close()
