"""Batches up to the lane-per-stage kernel's limits (36864 candidates under
1F1B, 24576 under Eager 1F1B) and just above them, where the sorted path
takes over: every stage count with the fewest and the most micro-batches,
invalid and overflowing records among them, odd batch sizes, both record
forms, against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def batch(gen, w, n, per_stage, rng):
    if per_stage:
        c = gen.per_stage_tp_candidates(n, w.L, w.n_types, w.n_tp, seed=n, M_range=(1, 255))
        bad = rng.random(n) < 0.05
        c["tp_code"][bad] |= np.uint32(0xC0000000)
    else:
        c = gen.random_candidates(n, L=w.L, n_types=w.n_types, S_range=(1, 16), M_range=(1, 255),
                                  seed=n)
        c["tp_idx"] = rng.integers(0, w.n_tp, n)
        c["tp_idx"][rng.random(n) < 0.02] = w.n_tp
    c["S"][rng.random(n) < 0.02] = 0
    c["S"][rng.random(n) < 0.02] = 17
    c["M"][rng.random(n) < 0.02] = 0
    c["map_rank"][rng.random(n) < 0.02] = np.uint64(2 ** 64 - 1)
    return c


@pytest.mark.parametrize("per_stage", [False, True])
@pytest.mark.parametrize("sched", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 5001, 24576, 24577, 36864, 36865])
def test_small_batches(n, sched, per_stage):
    import gen
    import oracle
    import paper_2609_06086_gb300 as P
    from gpu_util import eval_device, eval_device_ex
    w = gen.config4(seed=2)
    rng = np.random.default_rng(n + sched)
    tab = w.tables_dict()
    # M up to 255 at 65 TFLOPS passes 2^31 for the larger M: flagged 3
    tab["dsync"] = rng.integers(0, 2_000_000, tab["dsync"].shape)
    c = batch(gen, w, n, per_stage, rng)
    ot = oracle.OracleTables(**tab, schedule=sched)
    pick = rng.permutation(n)[:6000]  # the oracle's share
    T_ref, F_ref = (oracle.eval_batch_ex if per_stage else oracle.eval_batch)(ot, c[pick])
    h = P.Handle(P.Tables(**tab), sched)
    T, F = (eval_device_ex if per_stage else eval_device)(P, h, c)
    bad = np.flatnonzero((T[pick] != T_ref) | (F[pick] != F_ref))
    assert len(bad) == 0, (len(bad), c[pick[bad[:5]]], T[pick[bad[:5]]], T_ref[bad[:5]])
    h.close()


@pytest.mark.parametrize("sched", [0, 1])
def test_small_and_large_batches_agree(sched):
    """The same candidates alone and as part of a batch that takes the sorted
    path, on tables whose plans reach the steady state late."""
    import gen
    import paper_2609_06086_gb300 as P
    from gpu_util import eval_device
    from test_gpu_bounds import TABLES, tables
    for kind in TABLES:
        tab = tables(kind, 48, np.random.default_rng(1))
        c = gen.random_candidates(60_000, L=48, n_types=2, S_range=(1, 16), M_range=(1, 255), seed=4)
        h = P.Handle(P.Tables(**tab), sched)
        T, F = eval_device(P, h, c)
        for lo in range(0, len(c), 10_000):
            Ts, Fs = eval_device(P, h, c[lo:lo + 10_000])
            assert np.array_equal(Ts, T[lo:lo + 10_000]) and np.array_equal(Fs, F[lo:lo + 10_000])
        h.close()
