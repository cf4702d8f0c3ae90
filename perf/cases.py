"""The measured workloads: what a user of the library has it do, through the
Python binding of its C ABI.

Two families.  An "eval" case is one batch of encoded candidate plans
evaluated for makespan and memory feasibility, then reduced to the best
feasible plan; a "search" case is one exact parallelism search.  Sizes and
cost tables follow the repository's own workloads (7B-like and 70B-like
layers, two or three device types, 1F1B, Eager 1F1B and Interleaved 1F1B).
Every result is a whole number and is compared exactly.

Fields of a case
  kind      "eval" or "search"
  sched     "1f1b", "eager" or "interleaved"
  L         layers; types: device types; tps: TP degrees (1, 2, 4, 8 in order)
  hidden    model width of the cost tables
  eval      n records; form "tp16" (one TP index per plan, 16 bytes) or "tp24"
            (one per stage, 24 bytes); place "device" or "host" buffers;
            S_lo..S_hi stages (devices when interleaved), M_lo..M_hi
            micro-batches
  search    S stages; M: comma-separated micro-batch counts; place "free",
            "exact" (counts: stages per type) or "devices" (counts: devices per
            type, D: data-parallel degrees); prune 1 (Eq. 2) or 2 (tightened);
            V chunks per device (interleaved); warmup: random plans
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2609_06086_gb300 as P

SCHED = {"1f1b": 0, "eager": 1, "interleaved": 2}
PLACE = {"free": 0, "exact": 1, "devices": 2}
# per device type: peak TFLOPS and memory in GB
TFLOPS = (312.0, 125.0, 65.0, 200.0)
GIGABYTES = (80, 32, 16, 48)
SEQ = 4096


def _eval(name, sched, n, *, L=64, types=2, tps=1, hidden=4096, form="tp16", place="device",
          S_lo=2, S_hi=16, M_lo=8, M_hi=128):
    return dict(name=name, kind="eval", sched=sched, n=n, L=L, types=types, tps=tps, hidden=hidden,
                form=form, place=place, S_lo=S_lo, S_hi=S_hi, M_lo=M_lo, M_hi=M_hi)


def _search(name, sched, S, M, *, L, types, tps=1, hidden=4096, place="free", counts="", D="",
            prune=2, V=0, warmup=500):
    return dict(name=name, kind="search", sched=sched, S=S, M=M, L=L, types=types, tps=tps,
                hidden=hidden, place=place, counts=counts, D=D, prune=prune, V=V, warmup=warmup)


def listed():
    return [
        # the smallest search, 14 plans: a tool that asks again after every
        # change of its inputs; latency of the call alone
        _search("search_tiny", "1f1b", 2, "4", L=8, types=2, hidden=1024, place="exact",
                counts="1,1", prune=1, warmup=16),
        # a 7B-like model on two device types, any type on any stage, three
        # micro-batch counts, the paper's bound
        _search("search_7b", "1f1b", 4, "8,16,32", L=32, types=2, prune=1),
        # the headline: a 70B-like model on three device types with TP 1..8,
        # the tightened bound
        _search("search_70b", "1f1b", 8, "32", L=80, types=3, tps=4, hidden=8192, place="exact",
                counts="2,2,4"),
        # the same with the paper's bound as printed (far more plans to look at)
        _search("search_70b_eq2", "1f1b", 8, "32", L=80, types=3, tps=4, hidden=8192,
                place="exact", counts="2,2,4", prune=1),
        # the same cluster with a TP degree chosen per stage: 168,000 slices
        _search("search_70b_stage_tp", "1f1b", 8, "32", L=80, types=3, tps=4, hidden=8192,
                place="devices", counts="32,32,64", D="2,4,8,16"),
        # Interleaved 1F1B plans of the 7B-like model, three chunks per device
        _search("search_7b_interleaved", "interleaved", 4, "8,16,32", L=32, types=2, V=3),
        # a small batch: a planner that scores a few thousand plans per step
        # and waits for them; latency and launches
        _eval("eval_small", "1f1b", 3001, hidden=2048),
        # an ordinary batch in host memory (the synchronous entry point)
        _eval("eval_host", "1f1b", 100_003, hidden=2048, place="host"),
        # an ordinary batch of plans with a TP degree per stage on the 70B-like
        # tables (12 classes), few micro-batches among them
        _eval("eval_stage_tp", "1f1b", 250_007, L=80, types=3, tps=4, hidden=8192, form="tp24",
              S_lo=1, S_hi=16, M_lo=1, M_hi=64),
        # a large batch under Eager 1F1B
        _eval("eval_eager", "eager", 2_000_003),
        # a large batch under Interleaved 1F1B, every (devices, chunks) pair
        _eval("eval_interleaved", "interleaved", 1_000_003, hidden=2048, S_lo=1, S_hi=8),
        # the largest: a random sweep of the plan space
        _eval("eval_sweep", "1f1b", 20_000_003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.65:
        sched = rng.choice(("1f1b", "1f1b", "eager", "interleaved"))
        types, tps = rng.randint(1, 4), rng.choice((1, 1, 2, 3, 4))
        L = rng.randint(16, 120)
        # the makespans of the slowest type's layers stay below 2^31 us
        m_top = min(255, 20_000 // L)
        S_lo = rng.randint(1, 8)
        S_hi = rng.randint(S_lo, 8 if sched == "interleaved" else 16)
        M_lo = _log_int(rng, 1, min(32, m_top))
        c = _eval("", sched, _log_int(rng, 257, 10_000_000), L=L, types=types, tps=tps,
                  hidden=rng.choice((2048, 4096)), form="tp24" if rng.random() < 0.3 else "tp16",
                  S_lo=S_lo, S_hi=S_hi, M_lo=M_lo, M_hi=rng.randint(M_lo, m_top))
        if c["form"] == "tp16" and rng.random() < 0.25:
            c["place"] = "host"
            c["n"] = min(c["n"], 2_000_000)
    else:
        kind = rng.choice(("free", "free", "exact", "interleaved", "devices"))
        if kind == "free":
            S = rng.randint(2, 5)
            c = _search("", rng.choice(("1f1b", "eager")), S,
                        ",".join(str(v) for v in sorted(rng.sample(range(2, 65), rng.randint(1, 3)))),
                        L=rng.randint(max(12, S), 36), types=2, prune=rng.choice((1, 2)),
                        warmup=rng.choice((0, 100, 500)))
        elif kind == "exact":
            c = _search("", rng.choice(("1f1b", "eager")), 8, str(rng.randint(8, 48)),
                        L=rng.randint(60, 88), types=3, tps=4, hidden=8192, place="exact",
                        counts="2,2,4", warmup=rng.choice((100, 500)))
        elif kind == "interleaved":
            S = rng.randint(2, 4)
            c = _search("", "interleaved", S,
                        ",".join(str(S * v) for v in sorted(rng.sample(range(2, 9), 2))),
                        L=rng.randint(16, 28), types=2, V=2)
        else:
            c = _search("", "1f1b", 8, str(rng.randint(16, 48)), L=rng.randint(74, 84), types=3,
                        tps=4, hidden=8192, place="devices", counts="32,32,64",
                        D=rng.choice(("2", "2,4", "2,8", "2,4,8")))
    c.pop("name")
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _ints(text):
    return [int(v) for v in text.split(",")] if text else []


def _tables(case, seed):
    """Cost tables of a transformer with L layers of width `hidden`, sequence
    4096: [K][L] rows per class k = type * n_tp + tp index, with a random
    factor per (type, layer) as profiles show it."""
    rng = np.random.default_rng(seed)
    L, h, T, n_tp = case["L"], case["hidden"], case["types"], case["tps"]
    tp = [1, 2, 4, 8][:n_tp]
    K = T * n_tp
    noise = np.exp(0.1 * rng.standard_normal((T, L)))
    flops = 24.0 * SEQ * h * h + 4.0 * SEQ * SEQ * h
    act = SEQ * h * 2.0
    fwd, bwd, dsync = (np.zeros((K, L), np.int32) for _ in range(3))
    mem_w, mem_a = (np.zeros((K, L), np.int64) for _ in range(2))
    cap = np.zeros(K, np.int64)
    for k in range(K):
        ty, t = k // n_tp, tp[k % n_tp]
        comp = flops / (TFLOPS[ty] * 1e12 * t) * 1e6 * noise[ty]
        ring = 2.0 * (t - 1) / t * act / 300e9 * 1e6  # one TP all-reduce
        fwd[k] = np.maximum(1, np.rint(comp + 2 * ring))
        bwd[k] = np.maximum(1, np.rint(2 * comp + 2 * ring))
        dsync[k] = np.rint(2.0 * (24.0 * h * h / t) / 100e9 * 1e6)
        mem_w[k] = 16 * 12 * h * h // t
        mem_a[k] = 34 * SEQ * h // t
        cap[k] = int(GIGABYTES[ty] * 1e9)
    ty = np.arange(K) // n_tp
    link = np.where(ty[:, None] == ty[None, :], 25e9, 9.375e9)
    p2p = np.rint(act / link * 1e6).astype(np.int32)
    return dict(L=L, n_types=T, n_tp=n_tp, fwd=fwd, bwd=bwd, dsync=dsync, p2p_f=p2p,
                p2p_b=p2p.copy(), mem_w=mem_w, mem_a=mem_a, cap=cap)


def _fields(case, seed):
    """The plans of a batch, as int64 tensors on the GPU: stages (devices) S,
    chunks V (1 unless interleaved), micro-batches M, a type and a TP index
    per stage, the composition's rank."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n, L = case["n"], case["L"]

    def uniform(lo, hi, shape):  # lo, hi inclusive, numbers or tensors
        u = torch.randint(0, 1 << 62, shape, generator=g, device="cuda")
        return lo + u % (hi - lo + 1)

    il = case["sched"] == "interleaved"
    S = uniform(case["S_lo"], case["S_hi"], (n,))
    M = uniform(case["M_lo"], case["M_hi"], (n,))
    V = torch.ones_like(S)
    if il:  # 2 chunks or more, at most 16 virtual stages, M a multiple of S
        V = uniform(2, 16 // S, (n,))
        M = torch.maximum(S, M // S * S)
    types = uniform(0, case["types"] - 1, (n, 16))
    tps = uniform(0, case["tps"] - 1, (n, 16))
    if case["form"] == "tp16":
        tps = tps[:, :1].expand(n, 16)
    J = S * V
    most = torch.tensor([1] + [math.comb(L - 1, j - 1) if j <= L else 1 for j in range(1, 17)],
                        device="cuda")
    rank = uniform(0, most[J] - 1, (n,))
    return S, V, M, types, tps, rank


def _records(case, seed):
    S, V, M, types, tps, rank = _fields(case, seed)
    n = case["n"]
    used = torch.arange(16, device="cuda")[None, :] < S[:, None]
    shift = 2 * torch.arange(16, device="cuda")[None, :]
    vbyte = V if case["sched"] == "interleaved" else torch.zeros_like(V)
    tcode = torch.where(used, types << shift, 0).sum(1)
    if case["form"] == "tp16":
        word = S | M << 8 | tps[:, 0] << 16 | vbyte << 24
        rec = torch.stack((rank, tcode | word << 32), 1)
    else:
        tpcode = torch.where(used, tps << shift, 0).sum(1)
        rec = torch.stack((rank, tcode | tpcode << 32, S | M << 8 | vbyte << 16), 1)
    return rec.contiguous().view(torch.uint8).view(n, -1)


def prepare(case, seed):
    tab = _tables(case, seed)
    if case["kind"] == "search":
        w = SimpleNamespace(
            tables_dict=lambda: tab, n_types=case["types"], n_tp=case["tps"], S=case["S"],
            M_list=_ints(case["M"]), tp_list=[1, 2, 4, 8][:case["tps"]],
            dp_list=[16 // t for t in (1, 2, 4, 8)[:case["tps"]]] if case["tps"] > 1 else [1],
            placement=PLACE[case["place"]], type_counts=_ints(case["counts"]),
            D_list=_ints(case["D"]))
        problem, keep = P.make_problem(w, warmup=case["warmup"], prune=case["prune"], seed=seed,
                                       schedule=SCHED[case["sched"]], V=case["V"])
        return dict(kind="search", problem=problem, keep=keep)
    handle = P.Handle(P.Tables(**tab), SCHED[case["sched"]])
    rec = _records(case, seed)
    n = case["n"]
    if case["place"] == "host":
        dt = np.dtype([("map_rank", "<u8"), ("type_code", "<u4"), ("S", "u1"), ("M", "u1"),
                       ("tp_idx", "u1"), ("V", "u1")])
        return dict(kind="host", handle=handle, records=rec.cpu().numpy().view(dt).reshape(n))
    return dict(kind=case["form"], handle=handle, records=rec, n=n,
                T=torch.empty(n, dtype=torch.int32, device="cuda"),
                F=torch.empty(n, dtype=torch.uint8, device="cuda"),
                best=torch.empty(1, dtype=torch.int64, device="cuda"))


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(state):
    if state["kind"] == "search":
        plan, _ = P.poseidon_search(state["problem"])
        return plan
    if state["kind"] == "host":
        T, F = P.poseidon_eval_batch_host(state["handle"], state["records"])
        return dict(T=T, F=F)
    stream = torch.cuda.current_stream().cuda_stream
    n, T, F, best = state["n"], state["T"], state["F"], state["best"]
    call = P.poseidon_eval_batch if state["kind"] == "tp16" else P.poseidon_eval_batch_ex
    call(state["handle"], state["records"].data_ptr(), n, T.data_ptr(), F.data_ptr(), stream)
    P.poseidon_argmin(T.data_ptr(), F.data_ptr(), n, best.data_ptr(), stream)
    return dict(T=T, F=F, best=best)


def work(case):
    """Bytes: records in, makespans and flags out; for a search its tables.
    Operations (whole numbers, 32 bits): the weights of every plan's stages
    (three differences, two transfer times, an edge each way: about 12 per
    stage); for a search the same for one plan of every slice it has to look
    at."""
    if case["kind"] == "eval":
        size = 16 if case["form"] == "tp16" else 24
        stages = 9 if case["sched"] == "interleaved" else (case["S_lo"] + case["S_hi"]) / 2
        return {"bytes": float(case["n"] * (size + 5)), "flops": 12.0 * stages * case["n"]}
    K, L, S = case["types"] * case["tps"], case["L"], case["S"]
    if case["place"] == "free":
        places = case["types"] ** S
    else:
        places = math.factorial(S)
        for c in _ints(case["counts"]) if case["place"] == "exact" else (2, 2, 4):
            places //= math.factorial(c)
    slices = places * case["tps"] * len(_ints(case["M"]))
    return {"bytes": float(K * (28 * L + 8 * K + 8)),
            "flops": 12.0 * S * max(1, case["V"]) * slices}


def tolerance(case):
    return "exact"


# --------------------------------------------------------------------------
# the same results in plain torch, 64-bit integers
# --------------------------------------------------------------------------
def exact(case, seed):
    """The DAG of every plan run op by op: in each round every stage (device)
    whose next op has its inter-stage predecessor finished runs it."""
    if case["kind"] == "search" or case["n"] > 300_000:
        return None  # all plans of a space, or a batch that takes too long
    tab = {k: torch.as_tensor(v).cuda().long() if isinstance(v, np.ndarray) else v
           for k, v in _tables(case, seed).items()}
    fields = _fields(case, seed)
    step = 8192
    parts = [_exact_part(case, tab, [f[i:i + step] for f in fields])
             for i in range(0, case["n"], step)]
    T = torch.cat([p[0] for p in parts])
    F = torch.cat([p[1] for p in parts])
    if case["place"] == "host":
        return dict(T=T.int().cpu().numpy(), F=F.to(torch.uint8).cpu().numpy())
    key = torch.where(F == 1, T, torch.iinfo(torch.int64).max)
    low = (key == key.min()).nonzero()[:1, 0]
    best = torch.where(F.max() == 1, low, torch.full_like(low, -1))
    return dict(T=T.int(), F=F.to(torch.uint8), best=best)


def _cuts(L, J, rank):
    """[n, 17] ends of the stages of the composition of each rank (lexicographic)."""
    n = len(rank)
    cut = torch.zeros((n, 17), dtype=torch.int64, device="cuda")
    layer = torch.arange(L, device="cuda")[None, :]
    for j in range(1, 17):
        rows = (J == j).nonzero()[:, 0]
        r, c = rank[rows], torch.zeros_like(rows)
        for s in range(j - 1):
            k = j - s - 2  # stages after the next one
            # plans whose stage s ends at c + v: the rest splits over k + 1 stages
            table = torch.tensor([math.comb(m, k) if m >= 0 else 0 for m in range(-1, L)],
                                 device="cuda")
            left = L - c[:, None] - (layer + 1)  # layers left after v = layer + 1
            count = torch.where(left >= 1, table[left.clamp(min=0)], 0)
            below = count.cumsum(1)
            v = (below <= r[:, None]).sum(1)  # v - 1
            r = r - torch.where(v > 0, below.gather(1, (v - 1).clamp(min=0)[:, None])[:, 0], 0)
            c = c + v + 1
            cut[rows, s + 1] = c
        cut[rows, j] = L
    return cut


def _exact_part(case, tab, fields):
    S, V, M, types, tps, rank = fields
    n, L, il = len(S), case["L"], case["sched"] == "interleaved"
    J = S * V
    cut = _cuts(L, J, rank)
    cls = types * case["tps"] + tps  # class of stage (device) s
    stage = torch.arange(16, device="cuda")[None, :].expand(n, 16)
    on = stage < J[:, None]
    dev = stage % S[:, None]
    k = cls.gather(1, dev)
    lo, hi = cut[:, :16], cut[:, 1:]

    def total(rows):  # sums of a [K][L] table over each stage's layers
        pre = torch.cat((torch.zeros_like(rows[:, :1]), rows.cumsum(1)), 1)
        return torch.where(on, pre[k, hi.clamp(min=0)] - pre[k, lo], 0)

    w = torch.stack((total(tab["fwd"]), total(tab["bwd"])), 2)  # [n, 16, 2]
    d, mw, ma = total(tab["dsync"]), total(tab["mem_w"]), total(tab["mem_a"])
    k2 = cls.gather(1, (stage + 1) % S[:, None])
    edge = torch.stack((tab["p2p_f"][k, k2], tab["p2p_b"][k2, k]), 2)  # j -> j+1, j+1 -> j
    # chain of unit u (stage, or device): W forwards, pairs, the rest backward
    unit = stage
    live = unit < S[:, None]
    ops = (V * M)[:, None]  # forwards of a unit
    if il:
        W = torch.minimum(2 * (S[:, None] - unit - 1) + (V * S - S)[:, None], ops)
        W = torch.where((M == S)[:, None], ops, W)
    elif case["sched"] == "eager":
        W = torch.minimum(2 * (S[:, None] - unit - 1) + 1, ops)
    else:
        W = torch.minimum(S[:, None] - unit, ops)
    first_f = (V > 1)[:, None]  # the steady pairs start with the forward
    m_top = int(M.max())
    fin = torch.full((n, 16 * 2 * m_top), -1, dtype=torch.int64, device="cuda")
    clock, held, peak, at = (torch.zeros((n, 16), dtype=torch.int64, device="cuda")
                             for _ in range(4))
    units = S[:, None]
    span = J[:, None]
    while bool(((at < 2 * ops) & live).any()):
        r = at - W
        steady = (r >= 0) & (r < 2 * (ops - W))
        fwd_turn = (r % 2 == 0) == first_f
        back = torch.where(steady, ~fwd_turn, r >= 0)
        num = torch.where(r < 0, at, torch.where(
            steady, torch.where(fwd_turn, W + r // 2, r // 2), at - ops))
        chunk = (num % span) // units
        chunk = torch.where(back, V[:, None] - 1 - chunk, chunk)
        mb = num // span * units + num % units
        mb = torch.where((V > 1)[:, None], mb, num)
        chunk = torch.where((V > 1)[:, None], chunk, 0)
        j = (chunk * units + unit).clamp(max=15)
        b = back.long()
        pj = torch.where(back, j + 1, j - 1)
        free = torch.where(back, pj >= span, pj < 0)  # no inter-stage predecessor
        pjc = pj.clamp(0, 15)
        mbc = mb.clamp(max=m_top - 1)
        pred = fin.gather(1, (pjc * 2 + b) * m_top + mbc)
        go = (free | (pred >= 0)) & (at < 2 * ops) & live
        src = torch.where(back, j, pjc)  # the edge between stages src and src + 1
        e = edge.view(n, 32).gather(1, src * 2 + b)
        start = torch.where(free, clock, torch.maximum(clock, pred + e))
        end = start + w.view(n, 32).gather(1, j * 2 + b)
        clock = torch.where(go, end, clock)
        slot = torch.where(go, (j * 2 + b) * m_top + mbc, 0)
        # a stage belongs to one unit, so the slots of a round differ; idle
        # units write slot 0 back unchanged through a scatter of the maximum
        fin.scatter_reduce_(1, slot, torch.where(go, end, -1), "amax")
        a = ma.gather(1, j)
        held = held + torch.where(go, torch.where(back, -a, a), 0)
        peak = torch.maximum(peak, held)
        at = at + go.long()
    per_unit = torch.zeros((n, 16), dtype=torch.int64, device="cuda")
    dsum = per_unit.scatter_add(1, dev, d)
    resident = per_unit.scatter_add(1, dev, mw)
    T = torch.where(live, clock + dsum, 0).max(1).values
    fits = ((peak + resident <= tab["cap"][cls]) | ~live).all(1)
    return T, fits.long()
