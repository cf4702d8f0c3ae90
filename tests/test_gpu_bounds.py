"""The makespan kernels end a plan's steady steps when an upper and a lower
bound of its makespan meet, and put plans whose bounds stay apart on a queue
of their warp.  Cost tables where the bounds meet at once, late and never
(ties, near-ties, transfers that dominate, zero costs), at the fewest steady
steps and the most micro-batches, against the oracle: in batches of the
lane-per-stage kernel, with at most two groups of plans per warp (no queue),
with a queue per warp, and so many plans of one kernel that its warps take
tiles of the range from a counter."""
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


def candidates(L, sched, S_range, rng):
    import gen
    cands = gen.random_candidates(6000, L=L, n_types=2, S_range=S_range, M_range=(1, 255), seed=3)
    # a third of them with 0..3 steady steps
    first = cands["S"].astype(int) * (1 if sched == 0 else 2) - (0 if sched == 0 else 1)
    few = np.arange(len(cands)) % 3 == 0
    cands["M"][few] = np.clip(first + rng.integers(0, 4, len(cands)), 1, 255)[few]
    return cands, first


@pytest.mark.parametrize("sched", [0, 1])
@pytest.mark.parametrize("kind", TABLES)
def test_bounds_and_queue(kind, sched):
    import oracle
    import paper_2609_06086_gb300 as P
    from gpu_util import SORTED, eval_device
    rng = np.random.default_rng(TABLES.index(kind))
    L = 48
    tab = tables(kind, L, rng)
    cands, _ = candidates(L, sched, (1, 16), rng)
    T_ref, F_ref = oracle.eval_batch(oracle.OracleTables(**tab, schedule=sched), cands)
    h = P.Handle(P.Tables(**tab), sched)
    for n in (len(cands), SORTED, 1_500_000):
        pick = rng.integers(0, len(cands), n) if n > len(cands) else np.arange(n)
        T, F = eval_device(P, h, cands[pick])
        bad = np.flatnonzero((T != T_ref[pick]) | (F != F_ref[pick]))
        assert len(bad) == 0, (n, len(bad), cands[pick[bad[:3]]], T[bad[:3]], T_ref[pick[bad[:3]]])
    h.close()


# the stage ranges of the makespan kernels
RANGES = [(0, 1, 4), (0, 5, 8), (0, 9, 12), (0, 13, 16), (1, 1, 6), (1, 7, 10), (1, 11, 13),
          (1, 14, 16)]


@pytest.mark.parametrize("sched,S_lo,S_hi", RANGES)
@pytest.mark.parametrize("kind", TABLES)
def test_tiles_of_one_range(kind, sched, S_lo, S_hi):
    """Above 32 groups of 32 plans per warp, whatever the kernel's occupancy
    (at most 16 blocks of four warps per SM)."""
    import oracle
    import paper_2609_06086_gb300 as P
    import torch
    rng = np.random.default_rng(TABLES.index(kind))
    L = 48
    tab = tables(kind, L, rng)
    cands, first = candidates(L, sched, (S_lo, S_hi), rng)
    cands["M"] = np.maximum(cands["M"], first)  # no short pipelines
    T_ref, F_ref = oracle.eval_batch(oracle.OracleTables(**tab, schedule=sched), cands)
    n = 32 * 32 * 4 * 16 * torch.cuda.get_device_properties(0).multi_processor_count + 4321
    pick = torch.randint(len(cands), (n,), generator=torch.Generator().manual_seed(1)).cuda()
    d_c = torch.from_numpy(cands.view(np.uint8).reshape(len(cands), 16)).cuda()[pick].contiguous()
    d_T = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    d_F = torch.full((n,), 99, dtype=torch.uint8, device="cuda")
    h = P.Handle(P.Tables(**tab), sched)
    P.poseidon_eval_batch(h, d_c.data_ptr(), n, d_T.data_ptr(), d_F.data_ptr(),
                          torch.cuda.current_stream().cuda_stream)
    assert torch.equal(d_T, torch.from_numpy(T_ref).cuda()[pick])
    assert torch.equal(d_F, torch.from_numpy(F_ref).cuda()[pick])
    h.close()
