// Evaluation of small batches (1F1B and Eager 1F1B): half a warp per
// candidate, a lane per stage, one launch and no scratch.
//
// The sorted path (eval_kernel.cuh) takes ten launches one after another,
// which is all that a batch of a few thousand candidates costs.  Here nothing
// has to be sorted: the lanes of a half-warp step through the levels of their
// candidate's schedule together, each doing its stage's op of the level, and
// pass finishes to their neighbours by one shuffle per level.  With every
// forward at the steady rate,
//     F_{s,m} at level 2m + s - 2        (1F1B)
//     F_{s,m} at level 2m - 2S + 3s - 2  (Eager 1F1B)
//     B_{s,m} at level 2S - s + 2m - 1
// (s, m 1-based), an order that suits every M, short pipelines included: a
// stage's forward and backward levels alternate, its chain order holds
// (F_{s,W} is one level before B_{s,1}), B_{s+1,m} is one level before
// B_{s,m}, and F_{s-1,m} is one level before F_{s,m} under 1F1B; under Eager
// 1F1B it is three levels before, so stage s-1 has done one more forward
// since and passes on its last but one (a forward past the last micro-batch
// shifts that history too, so that F_{s,M} reads F_{s-1,M}).
//
// A level costs about 16 instructions for two candidates, far more than the
// sorted kernels' register wavefront, so the path is the faster one up to
// lane_max() candidates only.  What bounds a small batch is the latency of
// the levels of its longest candidate: a shuffle, an add-max, an add and a
// select each (with the lanes branching on their stage's parity instead:
// 23 us for 3,001 candidates, 14.9 us as it is).
#include "eval_kernel.cuh"

namespace pos {

constexpr int kLaneThreads = 128;

template <bool EAGER>
__global__ void __launch_bounds__(kLaneThreads) lane_kernel(EvalParams p) {
    // the tables straight from global memory (L1 and L2): staging them would
    // take longer than the few reads of a block's eight candidates
    const Tab t = tab_at(static_cast<const unsigned char *>(p.blob), p.lay);
    const int s0 = threadIdx.x & 15, s = s0 + 1;
    const uint32_t i = blockIdx.x * (kLaneThreads / 16) + (threadIdx.x >> 4);
    RecView v;
    v.rec = make_uint4(0, 0, 0, 0);
    v.tpc = 0;
    const bool in = i < p.n;
    if (in) v = load_record(p, i);
    const uint64_t rank = (uint64_t)v.rec.x | ((uint64_t)v.rec.y << 32);
    const uint32_t tcode = v.rec.z;
    const int M = (v.rec.w >> 8) & 0xff, tp = (v.rec.w >> 16) & 0xff, L = t.L();
    int S = v.rec.w & 0xff;
    bool ok = S >= 1 && S <= POS_MAX_STAGES && M >= 1 && S <= L && tp < t.n_tp();
    const uint64_t n_map = ok ? binom(t, L - 1, S - 1) : 0;
    ok = ok && rank < n_map && types_ok(tcode, S, t.n_types()) &&
         (!p.per_stage_tp || types_ok(v.tpc, S, t.n_tp()));
    const bool fits_32 = ok && M < (int)p.guard_m[S];  // the overflow guard
    if (in && !fits_32 && s0 == 0) {
        p.T[i] = -1;
        p.F[i] = ok ? POS_FEAS_OVERFLOW : POS_FEAS_INVALID;
    }
    if (!fits_32) S = 0;
    // the composition, by every lane of the half-warp; lane s0 keeps its
    // stage's layers [a, b)
    int a = 0, b = 0, c = 0;
    uint64_t left = n_map - rank;
#pragma unroll 1
    for (int k = S - 1; k >= 1; --k) {
        const int rem = L - c, c2 = c + (rem - unrank_step(t, rem, k, left));
        if (s0 == S - 1 - k) {
            a = c;
            b = c2;
        }
        c = c2;
    }
    if (s0 == S - 1) {
        a = c;
        b = L;
    }
    // this stage's weights and memory; lanes without a stage stay at zero
    const bool on = s0 < S;
    int32_t wF = 0, wB = 0, d = 0, eF = INT32_MIN, eB = INT32_MIN;
    bool fits = true;
    const int k = on ? stage_class(tcode, v.tpc, tp, t.n_tp(), s0) : 0;
    if (on) {
        const Sums w = sums_from(t, k, sums(t, k, a), b);
        wF = w.f;
        wB = w.b;
        d = w.d;
        fits = stage_fits(t, S, M, s0, k, a, b);
        if (s0 > 0) eF = p2p(t, stage_class(tcode, v.tpc, tp, t.n_tp(), s0 - 1), k).x;
        if (s < S) eB = p2p(t, k, stage_class(tcode, v.tpc, tp, t.n_tp(), s)).y;
    }
    __syncwarp();
    const int half = threadIdx.x & 16;
    const unsigned all_fit = __ballot_sync(0xffffffffu, fits) >> half;
    // Levels in pairs (even, odd): on the even one the even stages run their
    // forward and the odd ones their backward, on the odd one the reverse.  X
    // is the finish of the op kind that the lane's stage runs on even levels,
    // Y the other one.  A stage that runs a forward reads the previous stage's
    // forwards, which that stage updates on the other levels, and likewise
    // for backwards: so on even levels every lane publishes its Y and updates
    // X, on odd levels the reverse, and no lane branches on its parity.
    // Published is, under Eager 1F1B, the last but one of the forwards (Q of
    // the kind that is the lane's forward).  A stage without a predecessor has
    // an edge of INT32_MIN, which the clock always beats (finishes are not
    // negative).
    const bool f_even = (s & 1) == 0;  // forwards on even levels
    const int f_lo = EAGER ? 3 * s - 2 * S : s, b_lo = 2 * S - s + 1;
    const int32_t eX = f_even ? eF : eB, eY = f_even ? eB : eF;
    const int32_t wX = f_even ? wF : wB, wY = f_even ? wB : wF;
    const int loX = f_even ? f_lo : b_lo, loY = f_even ? b_lo : f_lo;
    const int srcX = f_even ? s0 - 1 : s0 + 1, srcY = f_even ? s0 + 1 : s0 - 1;
    // levels lo .. lo + span run the lane's op (none without a stage)
    const unsigned span = on ? 2u * (M - 1) : 0u;
    const int off = on ? 0 : 1 << 20;
    const int steady_end = EAGER ? 2 * M - 2 * S + 1 : 2 * M - 1, end = 2 * (S + M - 1);
    int32_t X = 0, Y = 0, PX = 0, PY = 0, clock = 0, skipped = 0;  // P: published
    auto even_level = [&](int lv) {
        const int32_t got = __shfl_sync(0xffffffffu, EAGER ? PY : Y, srcX, 16);
        const int32_t fin = add_max(got, eX, clock) + wX;
        const int at = lv - loX - off;
        const bool run = (unsigned)at <= span;
        if (EAGER) PX = f_even ? (at >= 0 ? X : PX) : (run ? fin : PX);
        X = run ? fin : X;
        clock = run ? fin : clock;
    };
    auto odd_level = [&](int lv) {
        const int32_t got = __shfl_sync(0xffffffffu, EAGER ? PX : X, srcY, 16);
        const int32_t fin = add_max(got, eY, clock) + wY;
        const int at = lv - loY - off;
        const bool run = (unsigned)at <= span;
        if (EAGER) PY = f_even ? (run ? fin : PY) : (at >= 0 ? Y : PY);
        Y = run ? fin : Y;
        clock = run ? fin : clock;
    };
    int lv = EAGER ? 2 - 2 * S : 0;
    const int last = S == 0 ? lv - 1 : end;
    while (__any_sync(0xffffffffu, lv <= last)) {
        // four pairs at a time; levels past the end run nothing
#pragma unroll
        for (int u = 0; u < 3; ++u, lv += 2) {
            even_level(lv);
            odd_level(lv + 1);
        }
        const int32_t x0 = X, y0 = Y, px0 = PX, py0 = PY;
        even_level(lv);
        odd_level(lv + 1);
        // Both levels inside the steady state and every finish grown by the
        // same amount: so will every further steady pair (the step is max-plus
        // linear), and they need not run.
        const int32_t grow = __shfl_sync(0xffffffffu, X - x0, 0, 16);
        const bool same = !on || (X - x0 == grow && Y - y0 == grow &&
                                  (!EAGER || (PX - px0 == grow && PY - py0 == grow)));
        const unsigned agree = __ballot_sync(0xffffffffu, same) >> half;
        if (lv >= 2 * S && lv + 1 < steady_end && (agree & 0xffffu) == 0xffffu) {
            const int pairs = (steady_end - lv - 1) / 2;
            skipped += pairs * grow;
            lv += 2 * pairs;
        }
        lv += 2;
    }
    const int32_t Bo = f_even ? Y : X;
    int32_t T = on ? Bo + d : 0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) T = max(T, __shfl_xor_sync(0xffffffffu, T, o));
    if (s0 == 0 && S > 0) {
        p.T[i] = T + skipped;
        p.F[i] = (all_fit & 0xffffu) == 0xffffu ? POS_FEAS_YES : POS_FEAS_NO;
    }
}

pos_status launch_lanes(const EvalParams &p, cudaStream_t stream) {
    const int grid = (int)((p.n + kLaneThreads / 16 - 1) / (kLaneThreads / 16));
    if (p.lay.sched == POS_SCHED_EAGER_1F1B)
        lane_kernel<true><<<grid, kLaneThreads, 0, stream>>>(p);
    else
        lane_kernel<false><<<grid, kLaneThreads, 0, stream>>>(p);
    POS_CUDA(cudaGetLastError());
    return POS_OK;
}

}  // namespace pos
