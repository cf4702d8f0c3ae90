// Evaluation kernels of poseidon_eval_batch (hot-path steps a2-a5).
//
// One thread evaluates one candidate, in two passes: a decode pass (field
// checks, overflow guard, unranking, memory check; few registers, so the
// latency of its dependent shared-memory lookups is hidden by many warps)
// writes every candidate's cut positions to its place in the (S, M)-sorted
// order, and the makespan pass reads them coalesced.  The makespan code is
// unrolled over the stages and its live registers grow with S (about 7*S),
// so the batch is first counting-sorted by S and M (stream-ordered scratch:
// every candidate's sorted position), and then a family of kernels, each
// owning the candidates of one S range with M >= S (eval_kernel: ramps
// unrolled, steady steps until the bounds meet) or of one M range with M < S
// (short_kernel), walks its contiguous range of the sorted records with
// launch bounds matched to its register need.  Warps therefore see one S
// except at bucket boundaries, and no kernel waits at a block barrier after
// staging the cost tables.  Small batches skip the sort (lane_max).
//
// Sort keys: fast path (M >= S for 1F1B, M >= 2S-1 for Eager 1F1B) ->
// (S-1)*32 + M/8 (a warp's plans end after about the same steps whatever M is,
// see makespan_fast, so neighbouring M share a key); short path -> 512 + M*16 +
// S-1; Interleaved 1F1B records with V >= 2 get keys after those
// (interleaved.cuh); records with S outside 1..16 or M = 0 are flagged invalid
// by the sort pass and get no key.
#pragma once
#include <algorithm>

#include "common.cuh"

namespace pos {

constexpr int kKeys = 512 + 32 * 16;  // fast keys, then short-path keys
constexpr int kEvalThreads = 128;

__host__ __device__ inline int fast_key_begin(int S) { return (S - 1) * 32; }
__host__ __device__ inline int short_key_begin(int M) { return 512 + M * 16; }

struct EvalParams {
    const uint4 *cands;    // 16-byte records (poseidon_eval_batch), or
    const uint2 *cands_ex; // 24-byte records with a TP index per stage
                           // (poseidon_eval_batch_ex; cands is then NULL)
    int64_t n;
    int32_t *T;
    uint8_t *F;
    const uint32_t *dest;  // sorted position of every candidate (kNoDest:
                           // no key, answered by the histogram pass)
    const uint32_t *offs;  // [keys + 1] start of every key in sorted order
                           // (written by the scatter pass, the decode pass
                           // after it)
    int offs_last;         // 1: offs come from the kernel right before the
                           // makespan kernel instead (interleaved search)
    uint4 *cuts;           // per sorted position j, two 16-byte words (read once,
                           // with evict-first loads, so that the outputs'
                           // sectors stay in L2):
                           // cuts[2j]: the cut positions (push_cut's layout;
                           // ascending bytes 0..14 for interleaved records),
                           // byte 15 = 1 when the result is already written;
                           // cuts[2j+1]: (candidate index, type_code, the
                           // record's S|M|tp|V word, per-stage TP code), so the makespan
                           // kernels read 32 contiguous bytes and no record
    const void *blob;
    BlobLayout lay;
    // the part of the blob that the makespan kernels stage: the timing
    // tables, or with the memory tables before them for the interleaved ones
    const void *tblob, *cblob;
    BlobLayout tlay, clay;
    // guard_m[J]: the smallest M (1..255; 256 for none) at which the
    // overflow guard (guard_trips) trips for J (virtual) stages: U(J, M)
    // grows with M since every cost is non-negative
    uint16_t guard_m[POS_MAX_STAGES + 1];
    int sms;               // SMs of the device
    uint32_t *tiles;       // [17] next tile of the range that starts at stage count
                           // S (GroupWalk), zero at the start
    int per_stage_tp;      // 1: records carry a TP index per stage (n_tp <= 4)
    // the handle's memory-limit table (Handle::lim_*): the decode pass stages
    // the binomials and this table and checks memory with one byte per stage
    int lim_w, lim_bytes;
    int inv_off, inv_bytes, inv_narrow;  // Handle::inv_*
};

// The record fields every pass reads, in the 16-byte record's word layout:
// x, y = composition rank, z = type code, w = S | M << 8 | tp << 16 | V << 24
// (tp = 0 for a 24-byte record), plus the per-stage TP code of a 24-byte
// record (TP index of stage s in bits [2s, 2s+2); 0 for 16-byte records).
struct RecView {
    uint4 rec;
    uint32_t tpc;
};
__device__ __forceinline__ RecView load_record(const EvalParams &p, uint32_t i) {
    RecView v;
    if (p.per_stage_tp) {
        // 24 bytes: u64 rank, u32 type code, u32 TP code, u8 S, M, V, pad, u32 pad
        const uint2 a = __ldg(p.cands_ex + 3 * (size_t)i), b = __ldg(p.cands_ex + 3 * (size_t)i + 1),
                    c = __ldg(p.cands_ex + 3 * (size_t)i + 2);
        v.rec = make_uint4(a.x, a.y, b.x, (c.x & 0xffffu) | ((c.x & 0xff0000u) << 8));
        v.tpc = b.y;
    } else {
        v.rec = __ldg(p.cands + i);
        v.tpc = 0;
    }
    return v;
}

// Class of stage s: type_s * n_tp + its TP index, which is tp for a 16-byte
// record (whose per-stage TP code reads 0) and the stage's field of the TP
// code for a 24-byte record (whose tp reads 0), so no select is needed.
__device__ __forceinline__ int stage_class(uint32_t tcode, uint32_t tpc, int tp, int n_tp, int s) {
    return (int)((tcode >> (2 * s)) & 3u) * n_tp + tp + (int)((tpc >> (2 * s)) & 3u);
}

// Are the 2-bit type fields of stages 0..S-1 (1 <= S <= 16) all below
// n_types (1..4)?  A field is >= n_types when its high bit is set
// (n_types <= 2), when both bits are set (n_types = 3), or, for one type,
// when it is not zero.
__device__ __forceinline__ bool types_ok(uint32_t tcode, int S, int n_types) {
    const uint32_t mask = S >= 16 ? 0xffffffffu : (1u << (2 * S)) - 1u;
    const uint32_t f = tcode & mask;
    const uint32_t bad = n_types >= 4   ? 0u
                         : n_types == 3 ? (f & (f >> 1) & 0x55555555u)
                         : n_types == 2 ? (f & 0xaaaaaaaau)
                                        : f;
    return bad == 0u;
}

// The decode pass packs the cut positions of a (non-interleaved) record
// (each below 256) into the bytes of a 16-byte word by shifting them in from
// the bottom: after pushing
// cut[1], ..., cut[n-1] (n - 1 <= 15 pushes), cut[q] sits in byte n-1-q and
// byte 15 is still 0 (the "answered by the decode pass" flag).  A push is
// three funnel shifts and a shift-or, whatever the stage index.
__device__ __forceinline__ void push_cut(uint4 &v, int c) {
    v.w = __funnelshift_l(v.z, v.w, 8);
    v.z = __funnelshift_l(v.y, v.z, 8);
    v.y = __funnelshift_l(v.x, v.y, 8);
    v.x = (v.x << 8) | (uint32_t)c;
}

// cut[q] (1 <= q <= n-1) of n stages from the packed word (n a constant
// after unrolling, so this is a constant shift of a constant word)
__device__ __forceinline__ int packed_cut(const uint32_t (&pw)[4], int n, int q) {
    const int b = n - 1 - q;
    return (int)((pw[b >> 2] >> (8 * (b & 3))) & 0xffu);
}

// One unranking step of the decode pass, k stages after the one that it places
// (unrank_step's contract): by the inverse table, or without it by the estimate.
template <bool LIM>
__device__ __forceinline__ int unrank_k(const Tab &t, const uint8_t *inv, int narrow, int rem,
                                        int k, uint64_t &Y) {
    if constexpr (LIM) {
        if (k == 1) {  // C(j, 1) = j
            const int j = (int)Y;
            Y = 1;
            return j;
        }
        return k > narrow ? unrank_table<false>(t, inv, k, Y) : unrank_table<true>(t, inv, k, Y);
    } else {
        return unrank_step(t, rem, k, Y);
    }
}

// Decode pass for an Interleaved 1F1B record (pad byte V >= 2, S = N
// devices): checks its fields (N*V <= 16 virtual stages, at most L, M a
// multiple of N) and the overflow guard over the N*V virtual stages, and
// unranks the composition of L layers into the virtual stages.  Memory is
// checked by the makespan kernel (it needs the device chains).
template <bool LIM>
__device__ __forceinline__ uint4 decode_il(const Tab &t, const uint4 &rec, uint32_t tpc,
                                           const EvalParams &p, uint32_t i, const uint8_t *inv) {
    const uint64_t rank = (uint64_t)rec.x | ((uint64_t)rec.y << 32);
    const uint32_t tcode = rec.z;
    const int S = rec.w & 0xff;
    const int M = (rec.w >> 8) & 0xff;
    const int tp = (rec.w >> 16) & 0xff;
    const int V = (int)(rec.w >> 24);
    const int J = S * V, L = t.L();
    bool ok = S >= 1 && J <= POS_MAX_STAGES && J <= L && M >= 1 && M % S == 0 &&
              tp < t.n_tp();
    const uint64_t n_map = ok ? binom(t, L - 1, J - 1) : 0;
    ok = ok && rank < n_map;
    ok = ok && types_ok(tcode, S, t.n_types()) &&
         types_ok(tpc, S, t.n_tp());  // tpc = 0 for 16-byte records
    const uint4 done = make_uint4(0, 0, 0, 1u << 24);
    if (!ok) {
        p.T[i] = -1;
        p.F[i] = POS_FEAS_INVALID;
        return done;
    }
    if (M >= (int)p.guard_m[J]) {  // the overflow guard
        p.T[i] = -1;
        p.F[i] = POS_FEAS_OVERFLOW;
        return done;
    }
    // cut[1..J-1] in ascending bytes 0..14, the layout the interleaved
    // search writes its leaf records in
    uint64_t Y = n_map - rank;
    uint64_t lo8 = 0, hi8 = 0;
    int c = 0;
#pragma unroll 1
    for (int j = 0; j < J - 1; ++j) {
        const int rem = L - c, k = J - j - 1;
        c += rem - unrank_k<LIM>(t, inv, p.inv_narrow, rem, k, Y);
        if (j < 8) lo8 |= (uint64_t)c << (8 * j);
        else hi8 |= (uint64_t)c << (8 * (j - 8));
    }
    return make_uint4((uint32_t)lo8, (uint32_t)(lo8 >> 32), (uint32_t)hi8,
                      (uint32_t)(hi8 >> 32) & 0x00ffffffu);
}

// Decode pass for one candidate: checks its fields and the overflow guard,
// unranks the composition stage by stage (carrying Y; LIM: by the inverse
// table staged at `inv`), checks each stage's memory as soon as its cut is
// known (LIM: by the memory-limit table staged at `lim`), and packs the cut positions
// (push_cut).  Invalid and overflowing candidates are answered here.  S is
// a runtime value and the stage loop is not unrolled, which keeps the
// kernel small enough to run many warps per SM.
template <bool LIM>
__device__ __forceinline__ uint4 decode_one(const Tab &t, const uint4 &rec, uint32_t tpc,
                                            const EvalParams &p, uint32_t i,
                                            const uint8_t *inv, const uint8_t *lim) {
    const uint64_t rank = (uint64_t)rec.x | ((uint64_t)rec.y << 32);
    const uint32_t tcode = rec.z;
    const int S = rec.w & 0xff;
    const int M = (rec.w >> 8) & 0xff;
    const int tp = (rec.w >> 16) & 0xff;
    const int L = t.L();
    if (t.ly->sched == POS_SCHED_INTERLEAVED_1F1B && (rec.w >> 24) >= 2)
        return decode_il<LIM>(t, rec, tpc, p, i, inv);
    bool ok = S >= 1 && S <= POS_MAX_STAGES && M >= 1 && S <= L && tp < t.n_tp();
    const uint64_t n_map = ok ? binom(t, L - 1, S - 1) : 0;
    ok = ok && rank < n_map;
    ok = ok && types_ok(tcode, S, t.n_types()) &&
         (!p.per_stage_tp || types_ok(tpc, S, t.n_tp()));  // tpc = 0 for 16-byte records
    const uint4 done = make_uint4(0, 0, 0, 1u << 24);  // byte 15 = 1: answered here
    if (!ok) {
        p.T[i] = -1;
        p.F[i] = POS_FEAS_INVALID;
        return done;
    }
    if (M >= (int)p.guard_m[S]) {  // the overflow guard
        p.T[i] = -1;
        p.F[i] = POS_FEAS_OVERFLOW;
        return done;
    }
    uint64_t Y = n_map - rank;
    uint4 cuts = make_uint4(0, 0, 0, 0);
    const int n_tp = t.n_tp();
    // in-flight micro-batches of stage s before the cap at M: S - s under
    // 1F1B, 2(S-1-s)+1 under Eager 1F1B (inflight()), stepped per stage
    const bool eager = t.ly->sched == POS_SCHED_EAGER_1F1B;
    const int dw = eager ? 2 : 1;
    int wl = eager ? 2 * S - 1 : S;
    // the stage's memory check, with the type and TP fields shifted down as
    // the stages go
    uint32_t tc = tcode, tq = tpc;
    auto fits_stage = [&](int a, int b) {
        const int cls = (int)(tc & 3u) * n_tp + tp + (int)(tq & 3u);  // stage_class
        const int w = min(wl, M);
        tc >>= 2;
        tq >>= 2;
        wl -= dw;
        if constexpr (LIM) return b <= (int)lim[(cls * p.lim_w + w - 1) * (L + 1) + a];
        else return stage_fits_w(t, w, cls, a, b);
    };
    bool fits = true;
    int c = 0;
    // stages 0..S-2 (k stages after each; L - c layers are left), then the last
    // one up to L
    auto place = [&](int c2) {
        push_cut(cuts, c2);
        fits &= fits_stage(c, c2);
        c = c2;
    };
    int k = S - 1;
    if constexpr (LIM) {
#pragma unroll 1
        for (; k > max(p.inv_narrow, 1); --k) place(L - unrank_table<false>(t, inv, k, Y));
#pragma unroll 1
        for (; k >= 2; --k) place(L - unrank_table<true>(t, inv, k, Y));
        if (k == 1) place(L - (int)Y);  // C(j, 1) = j
    } else {
#pragma unroll 1
        for (; k >= 1; --k) place(L - unrank_step(t, L - c, k, Y));
    }
    fits &= fits_stage(c, L);
    p.F[i] = fits ? POS_FEAS_YES : POS_FEAS_NO;
    return cuts;
}

template <int PATH>
struct EvalWith {
    template <int S>
    struct One {
        // makespan of a decoded candidate (cuts packed by the decode pass);
        // false when it was given up (to_end false, see makespan_fast)
        static __device__ __forceinline__ bool run(const Tab &t, const uint4 &rec,
                                                   const uint4 &packed, bool to_end,
                                                   int32_t &T) {
            // rec: x = per-stage TP code (0 for 16-byte records), z = type
            // code, w = S | M << 8 | tp << 16 | V << 24 (tp = 0 for 24-byte
            // records)
            const uint32_t tcode = rec.z;
            const int M = (rec.w >> 8) & 0xff;
            const int tp = (rec.w >> 16) & 0xff;
            int cls[S], cut[S + 1];
#pragma unroll
            for (int s = 0; s < S; ++s)
                cls[s] = stage_class(tcode, rec.x, tp, t.n_tp(), s);
            const uint32_t pw[4] = {packed.x, packed.y, packed.z, packed.w};
            cut[0] = 0;
#pragma unroll
            for (int s = 0; s < S - 1; ++s) cut[s + 1] = packed_cut(pw, S, s + 1);
            cut[S] = t.L();
            StageW<S> w;
            stage_weights<S>(t, cut, cls, w);
            return makespan_path<S, PATH>(w, M, Programs{}, to_end, NoLimit{}, T);
        }
    };
};

template <int SLO, int SHI, int PATH>
__device__ __forceinline__ bool dispatch_range(int S, const Tab &t, const uint4 &rec,
                                               const uint4 &packed, bool to_end, int32_t &T) {
#define POS_EV(n)                                                                            \
    if (n >= SLO && n <= SHI && S == n)                                                      \
        return EvalWith<PATH>::template One<(n >= SLO && n <= SHI) ? n : SLO>::run(          \
            t, rec, packed, to_end, T);
    POS_EV(1) POS_EV(2) POS_EV(3) POS_EV(4) POS_EV(5) POS_EV(6) POS_EV(7) POS_EV(8)
    POS_EV(9) POS_EV(10) POS_EV(11) POS_EV(12) POS_EV(13) POS_EV(14) POS_EV(15) POS_EV(16)
#undef POS_EV
    return true;
}

// A warp's walk over the sorted positions [begin, end), 32 at a time.
//
// Most plans need a few steady steps and some need nearly all (makespan_fast),
// so a warp that ran each of its 32 plans to the end would run as long as the
// slowest.  A plan whose bounds still differ at their first comparison is put
// on a queue of its warp instead (later), and 32 of those are run to their end
// together.  A warp with at most two groups of 32 plans has too few to fill
// such a group and runs every plan to its end at once.
//
// With a queue and many groups per warp (more than 32) the warps take tiles of
// eight neighbouring groups from a counter, from the range's end down: the most
// expensive plans first, so the warps finish together, and all warps at the
// same part of the range, so that the plans of a queue and the code that an SM
// runs have nearly one stage count at a time.  With fewer a warp walks one
// stretch of the range, whose plans have one stage count; blocks sms apart
// usually run on one SM and take neighbouring stretches, again so that an SM's
// warps run the same code.  (13..16 stages, 16 million 1F1B plans: 822 us with
// stretches in launch order, issue slots 39 % busy for want of instructions,
// 449 us with neighbouring ones; the whole sweep of 20 million 2364 -> 2259 us
// with tiles; 2 million Eager plans 413 us with stretches, 439 us with tiles.)
struct GroupWalk {
    static constexpr uint32_t kTile = 8, kTiled = 32;
    uint32_t begin, end, g, g_end, tiles, groups, stride;
    uint32_t *queue, *counter;  // 64 entries; next tile
    int queued;
    bool use_queue, more;
    // queued_from <= kTiled: groups per warp above which plans are queued
    __device__ __forceinline__ GroupWalk(uint32_t b, uint32_t e, uint32_t *q, uint32_t *c,
                                         uint32_t sms, uint32_t queued_from)
        : begin(b), end(e), queue(q), counter(c), queued(0) {
        constexpr uint32_t kWarps = kEvalThreads / 32;
        stride = gridDim.x * kWarps;
        groups = (end - begin + 31) / 32;
        use_queue = groups > queued_from * stride;
        more = groups > kTiled * stride;
        tiles = (groups + kTile - 1) / kTile;
        if (more) {
            g = g_end = 0;
        } else if (use_queue) {
            const uint32_t block = gridDim.x % sms == 0
                                       ? (blockIdx.x % sms) * (gridDim.x / sms) + blockIdx.x / sms
                                       : blockIdx.x;
            const uint32_t len = (groups + stride - 1) / stride;
            g = (block * kWarps + (threadIdx.x >> 5)) * len;
            g_end = min(groups, g + len);
        } else {  // every stride-th group
            g = blockIdx.x * kWarps + (threadIdx.x >> 5);
            g_end = groups;
        }
    }
    // The next 32 positions (whole warp): j and whether the lane has one;
    // to_end: run the plans to their end.
    __device__ __forceinline__ bool next(uint32_t &j, bool &active, bool &to_end) {
        const int lane = threadIdx.x & 31;
        if (g >= g_end && more && queued < 32) {
            uint32_t t = 0;
            if (lane == 0) t = atomicAdd(counter, 1u);
            t = __shfl_sync(0xffffffffu, t, 0);
            more = t < tiles;
            if (more) {
                g = (tiles - 1 - t) * kTile;
                g_end = min(groups, g + kTile);
            }
        }
        const bool again = queued >= 32 || (queued > 0 && g >= g_end);
        to_end = again || !use_queue;
        if (again) {
            active = lane < queued;
            j = active ? queue[lane] : 0u;
            const uint32_t rest = queue[32 + lane];
            __syncwarp();
            queue[lane] = rest;  // the oldest entries leave first
            __syncwarp();
            queued = max(queued - 32, 0);
            return true;
        }
        if (g >= g_end) return false;
        j = begin + 32 * g + lane;
        active = j < end;
        g += use_queue ? 1 : stride;
        return true;
    }
    __device__ __forceinline__ void later(uint32_t j, bool put) {
        const unsigned m = __ballot_sync(0xffffffffu, put);
        if (put) queue[queued + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = j;
        queued += __popc(m);
        __syncwarp();
    }
};

// With two groups per warp or fewer a queue has too few plans.  The plans of a
// range without bounds (Eager 1F1B, 14 stages and more) have nothing to queue,
// and their time grows with M, so up to the tiles each warp takes its share of
// every M (2 million Eager plans on a GB300: 333 us with a stretch of the range
// per warp, 310 us with every stride-th group; tiles from 8 groups on: 340 us).
__host__ __device__ constexpr uint32_t queued_from(int path, int slo) {
    return path == kPathEager && !eager_bounds(slo) ? GroupWalk::kTiled : 2u;
}

// Evaluates the sorted positions [offs[key_lo], offs[key_hi]): all
// candidates with S in [SLO, SHI] on path PATH.  Bound by issue slots (ramp,
// tail and first steps are straight-line code per stage) and, from 13 stages
// on, by instruction fetch.  Ranges of 20 million 1F1B plans on a GB300, every
// step run / with the bounds: 13..16 stages 1054 / 621 us, 9..12 595 / 365,
// 5..8 374 / 235.
template <int SLO, int SHI, int PATH, int MINB>
__global__ void __launch_bounds__(kEvalThreads, MINB) eval_kernel(EvalParams p) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ uint32_t s_queue[kEvalThreads / 32][64];
    // the key offsets come from the scatter pass, two or more kernels back
    const uint32_t begin = p.offs[fast_key_begin(SLO)], end = p.offs[fast_key_begin(SHI + 1)];
    // blocks with no candidate (all of them when the range is empty) leave
    // without staging the tables, after the decode pass has completed
    if (end == begin) {
        grid_dep_wait();
        return;
    }
    stage_blob(sm, p.tblob, p.tlay.bytes);
    __syncthreads();
    grid_dep_wait();  // the decoded records
    grid_dep_trigger();
    const Tab t = tab_at(sm, p.tlay);
    GroupWalk walk(begin, end, s_queue[threadIdx.x >> 5], p.tiles + SLO, (uint32_t)p.sms,
                   queued_from(PATH, SLO));
    uint32_t j;
    bool active, to_end;
    while (walk.next(j, active, to_end)) {
        uint32_t i = 0;
        uint4 rec = make_uint4(0, 0, 0, 0), packed = make_uint4(0, 0, 0, 0);
        if (active) {
            packed = __ldcs(p.cuts + 2 * (size_t)j);
            const uint4 meta = __ldcs(p.cuts + 2 * (size_t)j + 1);
            active = (packed.w >> 24) == 0;  // not answered by the decode pass
            i = meta.x;
            rec = make_uint4(meta.w, 0u, meta.y, meta.z);
        }
        const int S = active ? (int)(rec.w & 0xff) : 0;
        int32_t T = -1;
        bool done = true;
        unsigned pending = __ballot_sync(0xffffffffu, active);
        while (pending) {
            const int leader = __ffs(pending) - 1;
            const int Sg = __shfl_sync(0xffffffffu, S, leader);
            const bool mine = active && S == Sg;
            const unsigned grp = __ballot_sync(0xffffffffu, mine);
            if (mine) done = dispatch_range<SLO, SHI, PATH>(Sg, t, rec, packed, to_end, T);
            pending &= ~grp;
        }
        if (active && done) p.T[i] = T;
        walk.later(j, !done);
    }
}

// Byte b (a runtime index) of a packed word, see push_cut.
__device__ __forceinline__ int packed_byte(const uint4 &v, int b) {
    const uint32_t w = b < 4 ? v.x : b < 8 ? v.y : b < 12 ? v.z : v.w;
    return (int)((w >> (8 * (b & 3))) & 0xffu);
}

// Makespan of a decoded candidate of a short pipeline (see ShortProgram): S
// and the grid stages at run time, the last C stages unrolled for this M.
template <bool EAGER, int M>
__device__ __forceinline__ int32_t makespan_short_one(const Tab &t, const uint4 &rec,
                                                      const uint4 &packed) {
    constexpr int C = short_stages(EAGER, M);
    const int S = (int)(rec.w & 0xff), tp = (int)((rec.w >> 16) & 0xff), n_tp = t.n_tp();
    const int G = S - C;  // grid stages 0..G-1
    const uint32_t tcode = rec.z, tpc = rec.x;
    auto class_of = [&](int s) { return stage_class(tcode, tpc, tp, n_tp, s); };
    int32_t at[M];
#pragma unroll
    for (int m = 0; m < M; ++m) at[m] = 0;
    int k = class_of(0), c = 0;
#pragma unroll 1
    for (int s = 0; s < G; ++s) {  // G < S: the next stage exists
        const int c2 = packed_byte(packed, S - 2 - s), k2 = class_of(s + 1);
        const Sums v = sums_from(t, k, sums(t, k, c), c2);
        const int32_t pf = p2p(t, k, k2).x;
        int32_t clock = 0;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            clock = max(at[m], clock) + v.f;
            at[m] = clock + pf;
        }
        k = k2;
        c = c2;
    }
    int32_t T = 0;
    {
        // the last C stages: cut[G + q] in byte C - 1 - q (1 <= q < C)
        const uint32_t pw[4] = {packed.x, packed.y, packed.z, packed.w};
        int cls[C], cut[C + 1];
        cut[0] = c;
#pragma unroll
        for (int q = 1; q < C; ++q) cut[q] = packed_cut(pw, C, q);
        cut[C] = t.L();
#pragma unroll
        for (int q = 0; q < C; ++q) cls[q] = class_of(G + q);
        StageW<C> w;
        stage_weights<C>(t, cut, cls, w);
        int32_t Fo[C], Fp[C], Bo[C];
#pragma unroll
        for (int q = 0; q < C; ++q) Fo[q] = Fp[q] = Bo[q] = 0;
        short_run<EAGER, M>(at, Fo, Fp, Bo, w,
                            std::make_integer_sequence<int, ShortTab<EAGER, M>::value.n_levels>{});
#pragma unroll
        for (int q = 0; q < C; ++q) T = max(T, Bo[q] + w.d[q]);
    }
    int end = c;  // first layer of stage s + 1; k: its class
#pragma unroll 1
    for (int s = G - 1; s >= 0; --s) {
        const int b = s > 0 ? packed_byte(packed, S - 1 - s) : 0, ks = class_of(s);
        const Sums v = sums_from(t, ks, sums(t, ks, b), end);
        const int32_t pb = p2p(t, ks, k).y;
        int32_t clock = 0;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            clock = add_max(at[m], pb, clock) + v.b;
            at[m] = clock;
        }
        T = max(T, clock + v.d);
        k = ks;
        end = b;
    }
    return T;
}

// runtime M in MLO..MHI -> its instance
template <bool EAGER, int MLO, int... m>
__device__ __forceinline__ int32_t short_dispatch(int M, const Tab &t, const uint4 &rec,
                                                  const uint4 &packed,
                                                  std::integer_sequence<int, m...>) {
    int32_t T = -1;
    ((M == MLO + m ? (T = makespan_short_one<EAGER, MLO + m>(t, rec, packed), 0) : 0), ...);
    return T;
}

// Evaluates the sorted positions of the short pipelines with M in [MLO, MHI]
// (sorted by M, then S: a warp's plans have one M except at a boundary).  Bound
// by instruction fetch, so the code is one per M and not one per (S, M) (the
// short plans of 20 million 1F1B plans on a GB300: 144 us unrolled per (S, M),
// 61 us so; of 2 million Eager plans 166 / 60 us).
template <bool EAGER, int MLO, int MHI, int MINB>
__global__ void __launch_bounds__(kEvalThreads, MINB) short_kernel(EvalParams p) {
    extern __shared__ __align__(16) unsigned char sm[];
    // the key offsets come from the scatter pass, two or more kernels back
    const uint32_t begin = p.offs[short_key_begin(MLO)], end = p.offs[short_key_begin(MHI + 1)];
    if (blockIdx.x * blockDim.x >= end - begin) {
        grid_dep_wait();
        return;
    }
    stage_blob(sm, p.tblob, p.tlay.bytes);
    __syncthreads();
    grid_dep_wait();  // the decoded records
    grid_dep_trigger();
    const Tab t = tab_at(sm, p.tlay);
    const uint32_t stride = gridDim.x * blockDim.x;
    const uint32_t span = (end - begin + 31) & ~31u;  // whole warps iterate together
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < span; j += stride) {
        bool active = j < end - begin;
        uint32_t i = 0;
        uint4 rec = make_uint4(0, 0, 0, 0), packed = make_uint4(0, 0, 0, 0);
        if (active) {
            packed = __ldcs(p.cuts + 2 * (size_t)(begin + j));
            const uint4 meta = __ldcs(p.cuts + 2 * (size_t)(begin + j) + 1);
            active = (packed.w >> 24) == 0;  // not answered by the decode pass
            i = meta.x;
            rec = make_uint4(meta.w, 0u, meta.y, meta.z);
        }
        const int M = active ? (int)((rec.w >> 8) & 0xff) : 0;
        unsigned pending = __ballot_sync(0xffffffffu, active);
        while (pending) {
            const int Mg = __shfl_sync(0xffffffffu, M, __ffs(pending) - 1);
            const bool mine = active && M == Mg;
            if (mine)
                p.T[i] = short_dispatch<EAGER, MLO>(Mg, t, rec, packed,
                                                    std::make_integer_sequence<int, MHI - MLO + 1>{});
            pending &= ~__ballot_sync(0xffffffffu, mine);
        }
    }
}

// Launch of a makespan kernel over the sorted records, as many blocks as fit.
inline pos_status launch_ranged(void (*kern)(EvalParams), const EvalParams &p, int smem,
                                cudaStream_t stream) {
    POS_TRY(ensure_smem(reinterpret_cast<const void *>(kern), smem));
    int per_sm = 0;
    POS_TRY(blocks_per_sm(reinterpret_cast<const void *>(kern), kEvalThreads, smem, &per_sm));
    if (per_sm < 1) return fail(POS_ECUDA, "eval kernel does not fit on an SM");
    const int64_t blocks = (p.n + kEvalThreads - 1) / kEvalThreads;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(blocks, (int64_t)per_sm * sm_count()));
    POS_CUDA(launch_dependent(kern, grid, kEvalThreads, smem, stream, p));
    return POS_OK;
}

template <int SLO, int SHI, int PATH, int MINB>
pos_status launch_eval_range(const EvalParams &p, cudaStream_t stream) {
    return launch_ranged(eval_kernel<SLO, SHI, PATH, MINB>, p, p.tlay.bytes, stream);
}
template <bool EAGER, int MLO, int MHI, int MINB>
pos_status launch_short_range(const EvalParams &p, cudaStream_t stream) {
    return launch_ranged(short_kernel<EAGER, MLO, MHI, MINB>, p, p.tlay.bytes, stream);
}

// Sets the blob and the layouts of the parts that the kernels stage.
inline void set_tables(EvalParams &p, const void *blob, const BlobLayout &lay) {
    const unsigned char *b = static_cast<const unsigned char *>(blob);
    p.blob = blob;
    p.lay = lay;
    p.tblob = b + lay.off_P;
    p.tlay = timing_layout(lay);
    p.cblob = b + lay.off_Pw;
    p.clay = cost_layout(lay);
}

pos_status launch_decode(const EvalParams &p, cudaStream_t stream);

// Batches up to this many candidates take the lane-per-stage kernel of
// eval_lanes.cu.  The lanes' time grows with the micro-batches, the sorted
// path's hardly does, so the line lies where long pipelines cross.  Random plans
// of 64 layers and 2..16 stages on a GB300, lanes / sorted path: 1F1B with 8..128
// micro-batches 15.0 / 55.6 us at 3,001, 36.6 / 43.5 at 32,768, 49.5 / 46.1 at
// 49,152; with 120..255 22.5 / 46.8, 46.6 / 50.3 and 60.5 / 53.2.  Eager 1F1B
// 18.6 / 101, 48.2 / 71.8 at 24,576, 70.8 / 67.8 at 40,960; with 120..255 25.2 /
// 59.6, 63.4 / 63.4 and 90.0 / 66.3.  Few stages suit the lanes better (1F1B,
// 36,864 plans of 1..2 stages 12 us, of 2..4 23..31), batches of 16 stages
// alone worse: their Eager plans with 120..255 micro-batches take 82 us at
// 24,576, more than the sorted path did before its queues and bounds (63), and
// the rule, which sees the batch's size alone, leaves them to the lanes.
inline int64_t lane_max(int sched) {
    return sched == POS_SCHED_1F1B ? 36864 : sched == POS_SCHED_EAGER_1F1B ? 24576 : 0;
}
pos_status launch_lanes(const EvalParams &p, cudaStream_t stream);

// one launcher per instantiation unit (eval_range_*.cu)
pos_status eval_fast_1_4(const EvalParams &p, cudaStream_t s);
pos_status eval_fast_5_8(const EvalParams &p, cudaStream_t s);
pos_status eval_fast_9_12(const EvalParams &p, cudaStream_t s);
pos_status eval_fast_13_16(const EvalParams &p, cudaStream_t s);
pos_status eval_short_1_9(const EvalParams &p, cudaStream_t s);
pos_status eval_short_10_15(const EvalParams &p, cudaStream_t s);
pos_status eval_eager_1_6(const EvalParams &p, cudaStream_t s);
pos_status eval_eager_7_10(const EvalParams &p, cudaStream_t s);
pos_status eval_eager_11_13(const EvalParams &p, cudaStream_t s);
pos_status eval_eager_14_16(const EvalParams &p, cudaStream_t s);
pos_status eval_eager_short_1_14(const EvalParams &p, cudaStream_t s);
pos_status eval_eager_short_15_22(const EvalParams &p, cudaStream_t s);
pos_status eval_eager_short_23_30(const EvalParams &p, cudaStream_t s);

}  // namespace pos
