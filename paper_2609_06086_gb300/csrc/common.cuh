// Shared internals of libposeidon: error state, the device table blob and
// the per-candidate device routines (composition unranking/ranking, stage
// weights, memory feasibility, the 1F1B makespan wavefront).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <utility>
#include <vector>

#include "../../include/poseidon.h"

namespace pos {

// ---------------------------------------------------------------------------
// Error state (per host thread)
// ---------------------------------------------------------------------------
void set_error(const std::string &msg);
pos_status fail(pos_status st, const std::string &msg);
pos_status cuda_fail(cudaError_t e, const char *what);
// Raises a kernel's dynamic shared-memory limit to `smem` on the current
// device unless an earlier call already set at least that much (the
// attribute call costs host time that a launch-bound pipeline feels).
pos_status ensure_smem(const void *kernel, int smem);
// Resident blocks per SM of `kernel` at (threads, smem), from the occupancy
// calculator once per device and configuration, then from a cache (the
// query costs host time on every launch otherwise).
pos_status blocks_per_sm(const void *kernel, int threads, int smem, int *out);

// Programmatic dependent launch (sm_90 and later).  A kernel launched by
// launch_dependent may be scheduled while the kernel queued before it on
// the stream is still running; before it reads anything that kernel wrote
// it executes grid_dep_wait(), which returns once that grid has completed
// and its memory is visible.  It then calls grid_dep_trigger(), which lets
// the next such kernel be scheduled: a kernel's pre-wait part can therefore
// only overlap the post-wait part of its predecessor, so it may read
// whatever was written two or more kernels earlier (the cost tables, slice
// records and bound tables of a search; a kernel that can also follow the
// writer itself waits first: level_kernel at depth 0, il_eval_kernel in a
// search).  Every block of such a kernel
// executes grid_dep_wait() before it exits, even when it has no work: a grid
// completes only after its predecessor has, which keeps the chain's order
// transitive for the kernels after it.  Without the launch attribute the two
// instructions do nothing.
__device__ __forceinline__ void grid_dep_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void grid_dep_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent(void (*kern)(KArgs...), int grid, int block, int smem,
                                    cudaStream_t stream, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

#define POS_CUDA(call)                                           \
    do {                                                         \
        cudaError_t e_ = (call);                                 \
        if (e_ != cudaSuccess) return pos::cuda_fail(e_, #call); \
    } while (0)

// Propagate a non-OK pos_status.
#define POS_TRY(call)                             \
    do {                                          \
        const pos_status st_ = (call);            \
        if (st_ != POS_OK) return st_;            \
    } while (0)

// ---------------------------------------------------------------------------
// Table blob: one contiguous device buffer, staged whole into shared memory
// by every kernel.  Offsets are bytes from the blob start, 16-byte aligned.
//   binom  u64 [16][128]        C(n, k) at [k][n], k <= 15 (0 for n < k)
//   Pw, Pa i64 [K][L+1] each    exclusive prefix sums of mem_w, mem_a
//   cap    i64 [K]
//   P      i32x4 [K][L+1]       exclusive prefix sums of fwd, bwd, dsync (and a
//                               0): a stage's three sums take one 16-byte load
//                               per end instead of three loads
//   pp     i32x2 [K][K]         transfer times of the edge between a stage on
//                               class a and the next one on class b, at [a][b]:
//                               (p2p_f[a][b], p2p_b[b][a])
// ---------------------------------------------------------------------------
constexpr int kBinomN = 128;
constexpr int kBinomK = 16;

struct BlobLayout {
    int L, K, n_types, n_tp;
    int sched;  // POS_SCHED_* (stage chains, in-flight counts; Interleaved 1F1B
                // evaluates records with V < 2 as 1F1B)
    int off_binom, off_Pw, off_Pa, off_cap, off_P, off_pp;
    int bytes;  // multiple of 16
};

BlobLayout make_layout(int L, int n_types, int n_tp);
// The timing part of a blob (P, pp: its last two tables), rebased to start
// at byte 0, for kernels that read nothing else; the timing part starts at
// byte ly.off_P of the full blob.
BlobLayout timing_layout(const BlobLayout &ly);
// The same with the memory part before it (everything but the binomials);
// it starts at byte ly.off_Pw of the full blob.
BlobLayout cost_layout(const BlobLayout &ly);

struct Handle {
    int device;
    BlobLayout lay;
    void *d_blob;  // device copy of the blob
    // overflow guard terms: sum_l max_k(fwd+bwd), sum_l max_k dsync, max p2p
    int64_t guard_A, guard_D, guard_P;
    // memory-limit table of the evaluation's decode pass (after the blob in
    // the same allocation, byte lim_off): lim[k][w-1][a] = the largest b with
    // sum_{l in [a,b)} (mem_w + w mem_a) <= cap[k] (a when no layer fits), for
    // w = 1..lim_w in-flight micro-batches; lim_bytes = 0 when the table
    // would exceed kLimMaxBytes and the pass checks the sums directly
    int lim_off, lim_w, lim_bytes;
    // the decode pass's inverse of the binomials (fill_inverse; right before
    // the memory-limit table, byte inv_off; 0 bytes without that table), and
    // the largest k up to which every C(L-1, k) is below 2^32
    int inv_off, inv_bytes, inv_narrow;
};
constexpr int kLimMaxBytes = 32768;
// Threads per block of the argmin kernels (poseidon_argmin and
// poseidon_argmin_noalloc): their shared arrays hold one entry per warp of a
// block of this size, so every launch uses exactly this many threads.
constexpr int kArgminThreads = 256;
// Partial results of an argmin over n entries (1: none are stored), and its
// launches (eval.cu).
int64_t argmin_parts(const int32_t *T, const uint8_t *F, int64_t n);
pos_status launch_argmin(const int32_t *T, const uint8_t *F, int64_t n, int32_t *part_t,
                         long long *part_i, int64_t *out, cudaStream_t stream);

pos_status validate_tables(const pos_tables *t);
pos_status create_handle(const pos_tables *t, int sched, Handle **out);
// host part of create_handle: validated blob with raw rows, plus guard terms
pos_status build_blob(const pos_tables *t, int sched, std::vector<unsigned char> &host,
                      BlobLayout &ly, int64_t &guard_A, int64_t &guard_D, int64_t &guard_P);
// device part: per-class prefix sums in place, asynchronous on `stream`
pos_status launch_prefix_rows(void *d_blob, const BlobLayout &ly, cudaStream_t stream);
// lim[k][w-1][a] (K * wmax * (L+1) bytes, see Handle): asynchronous, after
// the kernel queued before it on the stream (the prefix sums)
pos_status launch_lim(const void *d_blob, const BlobLayout &ly, int wmax, uint8_t *lim,
                      cudaStream_t stream);
void destroy_handle(Handle *h);
int sm_count();

// One block (kPrefixThreads threads) per row of the five per-class tables, a
// thread per layer: the raw per-layer row sits at entries 1..L of the row;
// turn it into an exclusive prefix sum with P[0] = 0.  Bound by latency: one
// load, a scan by shuffles within the warps and over the four warp totals,
// one store per thread (a thread walking its row took 13 us for 80 layers,
// now under 4).
constexpr int kPrefixThreads = 128;
static_assert(kPrefixThreads > POS_MAX_LAYERS, "a thread per layer");
__device__ __forceinline__ void prefix_row(unsigned char *blob, const BlobLayout &ly, int row) {
    const int K = ly.K, Lp1 = ly.L + 1;
    const int table = row / K, k = row % K, l = threadIdx.x;
    int64_t *P8 = reinterpret_cast<int64_t *>(blob + (table == 0 ? ly.off_Pw : ly.off_Pa)) +
                  (int64_t)k * Lp1;
    int32_t *P4 = reinterpret_cast<int32_t *>(blob + ly.off_P) + (int64_t)k * Lp1 * 4 + (table - 2);
    int64_t v = 0;
    if (l >= 1 && l <= ly.L) v = table < 2 ? P8[l] : (int64_t)P4[4 * l];
    const int lane = l & 31, wid = l >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    __shared__ int64_t total[kPrefixThreads / 32];
    if (lane == 31) total[wid] = v;
    __syncthreads();
    for (int w = 0; w < wid; ++w) v += total[w];
    if (l <= ly.L) {
        if (table < 2) P8[l] = v;
        else P4[4 * l] = (int32_t)v;
    }
}

// View of the blob staged in shared memory.  It keeps the shared-memory
// base and a pointer to the layout in kernel parameter space; every access
// adds an offset read from there, so no table pointer occupies a register.
struct Tab {
    const unsigned char *base;  // the staged blob (dynamic shared memory)
    const BlobLayout *ly;       // points into kernel parameter space
    __device__ __forceinline__ int L() const { return ly->L; }
    __device__ __forceinline__ int Lp1() const { return ly->L + 1; }
    __device__ __forceinline__ int K() const { return ly->K; }
    __device__ __forceinline__ int n_tp() const { return ly->n_tp; }
    __device__ __forceinline__ int n_types() const { return ly->n_types; }
};

__device__ __forceinline__ int64_t ld64(const unsigned char *base, uint32_t off) {
    return *reinterpret_cast<const int64_t *>(base + off);
}

__device__ __forceinline__ Tab tab_at(const unsigned char *base, const BlobLayout &ly) {
    Tab t;
    t.base = base;
    t.ly = &ly;
    return t;
}

// (forward, backward, all-reduce) sums over layers [0, c) on class k
struct Sums {
    int32_t f, b, d;
};
__device__ __forceinline__ Sums sums(const Tab &t, int k, int c) {
    const int4 v = *reinterpret_cast<const int4 *>(t.base + t.ly->off_P +
                                                   16u * (uint32_t)(k * (t.ly->L + 1) + c));
    return {v.x, v.y, v.z};
}
// ... over layers [a, c), the sums at a known
__device__ __forceinline__ Sums sums_from(const Tab &t, int k, const Sums &at, int c) {
    const Sums v = sums(t, k, c);
    return {v.f - at.f, v.b - at.b, v.d - at.d};
}
__device__ __forceinline__ int64_t Pw(const Tab &t, int k, int c) {
    return ld64(t.base, t.ly->off_Pw + 8u * (uint32_t)(k * (t.ly->L + 1) + c));
}
__device__ __forceinline__ int64_t Pa(const Tab &t, int k, int c) {
    return ld64(t.base, t.ly->off_Pa + 8u * (uint32_t)(k * (t.ly->L + 1) + c));
}
__device__ __forceinline__ int64_t cap_of(const Tab &t, int k) {
    return ld64(t.base, t.ly->off_cap + 8u * (uint32_t)k);
}
// transfer times between a stage on class a and the next stage on class b:
// x of the forward edge, y of the backward edge
__device__ __forceinline__ int2 p2p(const Tab &t, int a, int b) {
    return *reinterpret_cast<const int2 *>(t.base + t.ly->off_pp +
                                           8u * (uint32_t)(a * t.ly->K + b));
}
// stored k-major ([k][n]) as 64-bit words, so that a warp reading
// C(n_lane, k) for one k touches consecutive 8-byte words
__device__ __forceinline__ uint64_t binom(const Tab &t, int n, int k) {
    return (uint64_t)ld64(t.base, t.ly->off_binom + 8u * (uint32_t)(k * kBinomN + n));
}

// One stage of the combinatorial-number-system unranking.  With rem layers
// left for k+1 stages (k >= 1), the remaining rank is carried as
// Y = C(rem-1, k) - rank, 1 <= Y <= C(rem-1, k).  The stage takes rem - j
// layers, j the smallest value in [k, rem-1] with C(j, k) >= Y; the next
// stage's Y (rem' = j layers, k' = k-1) is Y - C(j-1, k), since
// C(j, k) = C(j-1, k) + C(j-1, k-1) (Pascal's rule) puts it in
// [1, C(j-1, k-1)].  So a stage reads only C(j-1, k) and C(j, k).
//
// j is first estimated from C(x, k) ~ m^k / k! * exp(-k(k^2-1) / (12 m^2)),
// m = x - (k-1)/2 (the product of the k factors m +- d around their mean):
// m0 = (Y k!)^(1/k), x ~ m0 + (k-1)/2 + (k^2-1) / (24 m0) (half the
// second-order term, which over-corrects), and j = ceil(x - 0.01) (a margin
// for rounding error), taken as the nearest integer to x + 0.49.  Over
// uniform ranks of 64 layers in 2..16 stages this lands on j in about 99 %
// of the stages (else one step low); exact comparisons then move it to the
// answer whatever the estimate.
struct UnrankCoef {
    float log2_fact;  // log2(k!)
    float inv_k;      // 1/k
    float shift;      // (k-1)/2 + 0.49
    float corr;       // (k^2-1)/24
};
__device__ __constant__ static const UnrankCoef kUnrankCoef[16] = {
    {0.000000000f, 0.000000000f, 0.00f, 0.000000000f},
    {0.000000000f, 1.000000000f, 0.49f, 0.000000000f},
    {1.000000000f, 0.500000000f, 0.99f, 0.125000000f},
    {2.584962501f, 0.333333333f, 1.49f, 0.333333333f},
    {4.584962501f, 0.250000000f, 1.99f, 0.625000000f},
    {6.906890596f, 0.200000000f, 2.49f, 1.000000000f},
    {9.491853096f, 0.166666667f, 2.99f, 1.458333333f},
    {12.299208018f, 0.142857143f, 3.49f, 2.000000000f},
    {15.299208018f, 0.125000000f, 3.99f, 2.625000000f},
    {18.469133020f, 0.111111111f, 4.49f, 3.333333333f},
    {21.791061115f, 0.100000000f, 4.99f, 4.125000000f},
    {25.250492733f, 0.090909091f, 5.49f, 5.000000000f},
    {28.835455234f, 0.083333333f, 5.99f, 5.958333333f},
    {32.535894952f, 0.076923077f, 6.49f, 7.000000000f},
    {36.343249874f, 0.071428571f, 6.99f, 8.125000000f},
    {40.250140470f, 0.066666667f, 7.49f, 9.333333333f}};

// the hardware's approximate base-2 logarithm, power and reciprocal (PTX
// lg2 / ex2 / rcp .approx): an estimate only, the comparisons fix any error
__device__ __forceinline__ float approx_lg2(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float approx_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float approx_rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ int unrank_guess(uint64_t Y, int k, int rem) {
    const UnrankCoef c = kUnrankCoef[k];
    // Y as a float from its two 32-bit words: a 64-bit integer conversion
    // issues to the FP64 pipe, a small fraction of the FP32 rate here
    const float yf = __fmaf_rz(__uint2float_rz((uint32_t)(Y >> 32)), 4294967296.0f,
                               __uint2float_rz((uint32_t)Y));
    const float lg = approx_lg2(yf);
    const float m0 = approx_ex2((lg + c.log2_fact) * c.inv_k);
    const float x = m0 + c.shift + c.corr * approx_rcp(m0);
    // nearest integer by the float adder: 1.5 * 2^23 + x (0 <= x < 2^22)
    // has unit spacing, so its low bits are round(x)
    const int j = __float_as_int(x + 12582912.0f) - 0x4B400000;
    return min(max(j, k), rem - 1);
}

__device__ __forceinline__ int unrank_step(const Tab &t, int rem, int k, uint64_t &Y) {
    int j = unrank_guess(Y, k, rem);
    uint64_t below = binom(t, j - 1, k), at = binom(t, j, k);
    while (below >= Y) {  // stops at j = k at the latest: C(k-1, k) = 0 < Y
        --j;
        at = below;
        below = binom(t, j - 1, k);
    }
    while (at < Y && j < rem - 1) {  // C(rem-1, k) >= Y stops it first
        ++j;
        below = at;
        at = binom(t, j, k);
    }
    Y -= below;
    return j;
}

// The same step for k >= 2 with the estimate read from a table, for kernels
// that unrank many ranks.  A bucket holds the Y that share their exponent and
// first few mantissa bits as a float; inverse_bits makes it narrower than the
// gap between C(j, k) and C(j+1, k) for every j < 127, so with g the answer for
// its lowest Y the answer is g or g + 1, and one comparison with C(g, k)
// decides: about 12 instructions where the estimate and its two loops take 45
// and five of them go to the transcendental unit.  (The decode pass is bound by
// issue slots; whole calls on a GB300, estimate / table: 20 million 1F1B plans
// 2122 / 1973 us, 2 million Eager 364 / 346, 250,007 with 24-byte records 77.1 /
// 69.8.)  NARROW: Y is below 2^32 (k is at most Handle::inv_narrow).
//
// inv: an int2 (shift, base) for each k < 16, then the bytes g; the bucket of Y
// is byte (bits of Y as a float >> shift) + base of inv.  The conversion
// truncates, so the bucket's bits are Y's own.
__host__ __device__ constexpr int inverse_bits(int k) { return k <= 3 ? 6 : k <= 7 ? 5 : 4; }
constexpr int kInverseHeader = 16 * 8;

template <bool NARROW>
__device__ __forceinline__ int unrank_table(const Tab &t, const uint8_t *inv, int k, uint64_t &Y) {
    const int2 row = reinterpret_cast<const int2 *>(inv)[k];
    float yf = __uint2float_rz((uint32_t)Y);
    if constexpr (!NARROW) yf = __fmaf_rz(__uint2float_rz((uint32_t)(Y >> 32)), 4294967296.0f, yf);
    const int g = inv[(__float_as_int(yf) >> row.x) + row.y];
    const unsigned char *c = t.base + t.ly->off_binom + 8u * (uint32_t)(k * kBinomN + g);
    if constexpr (NARROW) {
        const uint32_t y = (uint32_t)Y, below = (uint32_t)*reinterpret_cast<const int32_t *>(c - 8),
                       at = (uint32_t)*reinterpret_cast<const int32_t *>(c);
        Y = y - (at < y ? at : below);
        return g + (at < y ? 1 : 0);
    } else {
        const uint64_t below = (uint64_t)ld64(c - 8, 0), at = (uint64_t)ld64(c, 0);
        const bool up = at < Y;
        Y -= up ? at : below;
        return g + (up ? 1 : 0);
    }
}

// Cooperative 16-byte copy of the blob into shared memory, four loads in
// flight per thread (a load-store pair per iteration would wait a full
// memory latency each time).
__device__ __forceinline__ void stage_blob(unsigned char *dst, const void *src, int bytes) {
    const uint4 *s = reinterpret_cast<const uint4 *>(src);
    uint4 *d = reinterpret_cast<uint4 *>(dst);
    const int n = bytes / 16, bd = blockDim.x;
    int i = threadIdx.x;
    for (; i + 3 * bd < n; i += 4 * bd) {
        const uint4 a = __ldg(s + i), b = __ldg(s + i + bd), c = __ldg(s + i + 2 * bd),
                    e = __ldg(s + i + 3 * bd);
        d[i] = a;
        d[i + bd] = b;
        d[i + 2 * bd] = c;
        d[i + 3 * bd] = e;
    }
    for (; i < n; i += bd) d[i] = __ldg(s + i);
}

// Bulk copies global -> this CTA's shared memory on the TMA engine
// (cp.async.bulk), completion counted in bytes on one mbarrier.  Thread 0
// calls bulk_begin with the total byte count, then issues the copies
// (16-byte aligned addresses, sizes multiples of 16); then every thread of
// the block calls bulk_wait, which returns the same value in all threads:
// false if the copies did not complete within kBulkWaitLimit polls.  That is
// a last-resort exit (2^24 polls, far beyond any copy of at most a few
// hundred KB): the caller counts it and leaves, the search then reports
// POS_ETIMEOUT, and a copy still in flight may land in shared memory that
// the block no longer owns; nothing exercises it on a GPU.
constexpr int kBulkWaitLimit = 1 << 24;

__device__ __forceinline__ void bulk_begin(uint64_t *bar, uint32_t total_bytes) {
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b),
                 "r"(total_bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_copy(void *dst_smem, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst_smem);
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(d),
        "l"(src), "r"(bytes), "r"(b)
        : "memory");
}

__device__ __forceinline__ bool bulk_wait(uint64_t *bar) {
    __syncthreads();  // the barrier is initialised before anyone polls it
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
    uint32_t done = 0;
    for (int it = 0; it < kBulkWaitLimit && !done; ++it) {
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n"
            " selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(b)
            : "memory");
    }
    return __syncthreads_and(done) != 0;
}

// The whole blob (or a rebased part of it) by one bulk copy.
__device__ __forceinline__ bool stage_blob_bulk(unsigned char *dst, const void *src, int bytes,
                                                uint64_t *bar) {
    if (threadIdx.x == 0) {
        bulk_begin(bar, (uint32_t)bytes);
        bulk_copy(dst, src, (uint32_t)bytes, bar);
    }
    return bulk_wait(bar);
}

// ---------------------------------------------------------------------------
// Composition <-> lexicographic rank (combinatorial number system).
// With p stages left and rem layers left, the compositions whose current
// stage takes fewer than v layers number C(rem-1, p-1) - C(rem-v, p-1)
// (hockey-stick sum of C(rem-u-1, p-2) over u < v).
// cut[0] = 0, cut[s+1] = layers of stages 0..s, cut[S] = L.
// ---------------------------------------------------------------------------
// Rank of the composition given by cut[0..S] (the numbering unrank_step
// walks stage by stage).
template <int S>
__device__ __forceinline__ uint64_t rank_cuts(const Tab &t, const int (&cut)[S + 1]) {
    uint64_t r = 0;
#pragma unroll
    for (int s = 0; s < S - 1; ++s) {
        const int rem = t.L() - cut[s];
        const int l = cut[s + 1] - cut[s];
        const int k = S - s - 1;
        r += binom(t, rem - 1, k) - binom(t, rem - l, k);
    }
    return r;
}

// ---------------------------------------------------------------------------
// Stage weights (Sec. 4.1.3) from prefix-sum differences; memory (Sec. 3.2).
// ---------------------------------------------------------------------------
// max(a + b, c) as one fused integer add-max (the CUDA intrinsic
// __viaddmax_s32); the makespan relaxations are built from it.
__device__ __forceinline__ int32_t add_max(int32_t a, int32_t b, int32_t c) {
    return __viaddmax_s32(a, b, c);
}

template <int S>
struct StageW {
    int32_t F[S], B[S], d[S];
    int32_t pf[S], pb[S];  // pf[s]: F edge s->s+1; pb[s]: B edge s+1->s
};

// In-flight micro-batches of 0-based stage s under 1F1B: min(S - s, M).
// Micro-batches a 0-based stage s holds at once = its warm-up forwards:
// N-s+1 (1F1B) or 2(N-s)+1 (Eager 1F1B) in 1-based numbering, at most M.
__host__ __device__ __forceinline__ int inflight(int sched, int S, int M, int s) {
    const int w = sched == POS_SCHED_EAGER_1F1B ? 2 * (S - 1 - s) + 1 : S - s;
    return w < M ? w : M;
}

// Does 0-based stage s of an S-stage pipeline on class k fit layers [a, b)?
// ... with w micro-batches in flight
__device__ __forceinline__ bool stage_fits_w(const Tab &t, int w, int k, int a, int b) {
    const int64_t need = (Pw(t, k, b) - Pw(t, k, a)) + (int64_t)w * (Pa(t, k, b) - Pa(t, k, a));
    return need <= cap_of(t, k);
}
__device__ __forceinline__ bool stage_fits(const Tab &t, int S, int M, int s, int k, int a,
                                           int b) {
    return stage_fits_w(t, inflight(t.ly->sched, S, M, s), k, a, b);
}

template <int S>
__device__ __forceinline__ void stage_weights(const Tab &t, const int (&cut)[S + 1],
                                              const int (&cls)[S], StageW<S> &w) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const Sums v = sums_from(t, cls[s], sums(t, cls[s], cut[s]), cut[s + 1]);
        w.F[s] = v.f;
        w.B[s] = v.b;
        w.d[s] = v.d;
        w.pf[s] = w.pb[s] = 0;
        if (s + 1 < S) {
            const int2 e = p2p(t, cls[s], cls[s + 1 < S ? s + 1 : s]);
            w.pf[s] = e.x;
            w.pb[s] = e.y;
        }
    }
}

// ---------------------------------------------------------------------------
// 1F1B makespan as a max-plus wavefront (Sec. 4.1, longest path by DP).
//
// Stage s (1-based) runs W_s = min(S-s+1, M) forwards, then (B_i, F_{W+i})
// pairs, then the remaining backwards.  Every op is one relaxation
//     finish = max(finish of the stage's previous op,
//                  finish of the inter-stage predecessor + edge) + weight.
// The ops are visited in the level order of the unit-weight schedule,
//     F_{s,m}: m + s - 1 (m <= W_s), 2m + s - 2 (m > W_s);
//     B_{s,m}: 2S - s + 2m - 1,
// a topological order with at most one op per stage per level in which,
// visiting the stages of a level in descending order, the inter-stage
// predecessor of an op is always the latest op of that kind on the
// neighbouring stage.  So per stage only the finish of its last forward (Fo)
// and last backward (Bo) are kept, in registers.  For M >= S the levels
// split into a ramp-up (levels 1..2S-1), M-S steady two-level steps in which
// every stage does one F and one B, and a ramp-down (levels 2M..2M+2S-2);
// the ramps depend on S only and are fully unrolled.  M < S takes a
// separate instantiation (kPathGeneric) whose schedule is unrolled for
// each M in 1..S-1.
// ---------------------------------------------------------------------------
// Paths: 1F1B with M >= S (ramps + steady loop), 1F1B with M < S (the search's
// leaf kernel: unrolled per M), Eager 1F1B with M >= 2S-1 (ramps + steady
// loop), Eager 1F1B with M < 2S-1 (leaf kernel: a level program).  The
// evaluator's short pipelines have kernels of their own (ShortProgram).
enum { kPathFast = 0, kPathGeneric = 1, kPathEager = 2, kPathEagerShort = 3 };

// Op of 1-based stage s1 at ramp-up level t (1 <= t <= 2S-1) and at
// ramp-down level 2M + tau (0 <= tau <= 2S-2), for M >= S: 0 none, 1 F, 2 B.
__host__ __device__ constexpr int ramp_up_op(int S, int s1, int t) {
    return (t >= s1 && t <= S) ? 1
           : ((t >= 2 * S - s1 + 2) && ((t + s1) & 1) == 0) ? 1
           : ((t >= 2 * S - s1 + 1) && ((t + s1) & 1) == 1) ? 2
                                                              : 0;
}
__host__ __device__ constexpr int ramp_down_op(int S, int s1, int tau) {
    return ((tau <= s1 - 2) && ((tau + s1) & 1) == 0) ? 1
           : ((tau <= 2 * S - s1 - 1) && ((tau + s1) & 1) == 1) ? 2
                                                                : 0;
}
// Was the last op of stage s1 before ramp-up level t a backward?  (No op
// yet counts as a forward: Fo starts at 0, the finish time of node S.)
__host__ __device__ constexpr bool up_last_is_b(int S, int s1, int t) {
    for (int u = t - 1; u >= 1; --u)
        if (ramp_up_op(S, s1, u)) return ramp_up_op(S, s1, u) == 2;
    return false;
}
// Same before ramp-down level 2M + tau; at the end of the steady state odd
// stages (1-based) last ran F and even stages B.
__host__ __device__ constexpr bool down_last_is_b(int S, int s1, int tau) {
    for (int u = tau - 1; u >= 0; --u)
        if (ramp_down_op(S, s1, u)) return ramp_down_op(S, s1, u) == 2;
    return (s1 & 1) == 0;
}

// One relaxation of stage s (0-based) on the forward or backward side:
// finish = max(stage clock, predecessor's finish + edge) + node weight, the
// add-max fused into one integer instruction (add_max).  Every time is >= 0
// (non-negative weights from time 0), so a stage without an inter-stage
// predecessor takes its clock alone.
template <int S, int s>
__device__ __forceinline__ void relax_f(int32_t (&Fo)[S], const StageW<S> &w, int32_t clock) {
    if constexpr (s > 0) Fo[s] = add_max(Fo[s - 1], w.pf[s - 1], clock) + w.F[s];
    else Fo[s] = clock + w.F[s];
}
template <int S, int s>
__device__ __forceinline__ void relax_b(int32_t (&Bo)[S], const StageW<S> &w, int32_t clock) {
    if constexpr (s + 1 < S) Bo[s] = add_max(Bo[s + 1], w.pb[s], clock) + w.B[s];
    else Bo[s] = clock + w.B[s];
}

// Ramp op of 1-based stage s1 at level t (UP) or at level 2M + t (DOWN);
// the clock is the finish of the stage's last op, known at compile time.
template <int S, bool UP, int t, int s1>
__device__ __forceinline__ void ramp_op(int32_t (&Fo)[S], int32_t (&Bo)[S], const StageW<S> &w) {
    constexpr int op = UP ? ramp_up_op(S, s1, t) : ramp_down_op(S, s1, t);
    constexpr bool last_b = UP ? up_last_is_b(S, s1, t) : down_last_is_b(S, s1, t);
    constexpr int s = s1 - 1;
    if constexpr (op == 1) relax_f<S, s>(Fo, w, last_b ? Bo[s] : Fo[s]);
    else if constexpr (op == 2) relax_b<S, s>(Bo, w, last_b ? Bo[s] : Fo[s]);
}
// one level, stages in descending order (i = 0 is stage S)
template <int S, bool UP, int t, int... i>
__device__ __forceinline__ void ramp_level(int32_t (&Fo)[S], int32_t (&Bo)[S], const StageW<S> &w,
                                           std::integer_sequence<int, i...>) {
    (ramp_op<S, UP, t, S - i>(Fo, Bo, w), ...);
}
template <int S, bool UP, int T0, int... t>
__device__ __forceinline__ void ramp(int32_t (&Fo)[S], int32_t (&Bo)[S], const StageW<S> &w,
                                     std::integer_sequence<int, t...>) {
    (ramp_level<S, UP, T0 + t>(Fo, Bo, w, std::make_integer_sequence<int, S>{}), ...);
}
// steady level: at level parity P (0 even) stage s1 runs F when s1 has the
// same parity, B otherwise; an F follows the stage's B and vice versa
template <int S, int P, int i>
__device__ __forceinline__ void steady_op(int32_t (&Fo)[S], int32_t (&Bo)[S], const StageW<S> &w) {
    constexpr int s1 = S - i, s = s1 - 1;
    if constexpr ((s1 & 1) == P) relax_f<S, s>(Fo, w, Bo[s]);
    else relax_b<S, s>(Bo, w, Fo[s]);
}
// M < S: the same level order, with W_s = min(S-s1+1, M); every op and the
// type of each stage's previous op are known at compile time for a given
// (S, M), so the whole schedule is unrolled (M < S <= 16 keeps it small).
__host__ __device__ constexpr int short_op(int S, int M, int s1, int t) {
    const int ws = S - s1 + 1 < M ? S - s1 + 1 : M;
    const bool odd = ((t + s1) & 1) != 0;
    if ((t >= s1 && t <= s1 + ws - 1) || (!odd && t >= 2 * ws + s1 && t <= 2 * M + s1 - 2))
        return 1;
    if (odd && t >= 2 * S - s1 + 1 && t <= 2 * S - s1 + 2 * M - 1) return 2;
    return 0;
}
__host__ __device__ constexpr bool short_last_is_b(int S, int M, int s1, int t) {
    for (int u = t - 1; u >= 1; --u)
        if (short_op(S, M, s1, u)) return short_op(S, M, s1, u) == 2;
    return false;
}
template <int S, int M, int t, int s1>
__device__ __forceinline__ void short_step(int32_t (&Fo)[S], int32_t (&Bo)[S], const StageW<S> &w) {
    constexpr int op = short_op(S, M, s1, t);
    constexpr bool last_b = short_last_is_b(S, M, s1, t);
    constexpr int s = s1 - 1;
    if constexpr (op == 1) relax_f<S, s>(Fo, w, last_b ? Bo[s] : Fo[s]);
    else if constexpr (op == 2) relax_b<S, s>(Bo, w, last_b ? Bo[s] : Fo[s]);
}
template <int S, int M, int t, int... i>
__device__ __forceinline__ void short_level(int32_t (&Fo)[S], int32_t (&Bo)[S], const StageW<S> &w,
                                            std::integer_sequence<int, i...>) {
    (short_step<S, M, t, S - i>(Fo, Bo, w), ...);
}
template <int S, int M, int... t>
__device__ __forceinline__ void short_all(int32_t (&Fo)[S], int32_t (&Bo)[S], const StageW<S> &w,
                                          std::integer_sequence<int, t...>) {
    (short_level<S, M, t + 1>(Fo, Bo, w, std::make_integer_sequence<int, S>{}), ...);
}
template <int S, int M>
__device__ __forceinline__ int32_t makespan_short(const StageW<S> &w) {
    int32_t Fo[S], Bo[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        Fo[s] = 0;
        Bo[s] = 0;
    }
    short_all<S, M>(Fo, Bo, w, std::make_integer_sequence<int, 2 * (M + S - 1)>{});
    int32_t T = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) T = max(T, Bo[s] + w.d[s]);
    return T;
}
// runtime M in 1..S-1 -> its unrolled instance
template <int S, int... m>
__device__ __forceinline__ int32_t makespan_short_dispatch(const StageW<S> &w, int M,
                                                           std::integer_sequence<int, m...>) {
    int32_t T = -1;
    ((M == m + 1 ? (T = makespan_short<S, m + 1>(w), 0) : 0), ...);
    return T;
}

// ---------------------------------------------------------------------------
// M >= S without running every steady step.  Let x be the finishes (Fo, Bo)
// after some steady step, R the number of steady steps left.
//  * Ramp-down.  T is a max-plus linear function of the state that enters
//    the ramp-down: T = max_s max(Fo[s] + rF[s], Bo[s] + rB[s]), rF and rB
//    the longest paths from those finishes to the end (all-reduce included).
//    They depend on the weights alone and are built by walking the
//    ramp-down's ops backwards, once per plan (tail_*).  A finish that no
//    later op reads gets 0, which is valid too: T is at least every finish.
//  * Upper bound.  A steady step is monotone and adds a constant to its
//    result when the constant is added to its input, so no finish ever grows
//    by more in a later step than the largest growth D of one step:
//    T <= max_s max(Fo[s] + rF[s], Bo[s] + rB[s]) + R D.
//  * Lower bound.  Stage s runs one forward and one backward per step, so its
//    finishes grow by at least F[s] + B[s] in each:
//    T >= max_s (max(Fo[s] + rF[s], Bo[s] + rB[s]) + R (F[s] + B[s])).
// When the two are equal they are T and the remaining steps need not run;
// at R = 0 they always are.  Whole numbers throughout, so nothing is
// approximated.  On random plans (64 layers, 2..16 stages, 8..128
// micro-batches) the bounds meet after three steps of the 61 on average
// for 86 % (13..16 stages) to 99 % (1..4) of the plans.
// ---------------------------------------------------------------------------
template <int S>
struct Tail {
    int32_t F[S], B[S];
};
template <int S, int tau, int s1>
__device__ __forceinline__ void tail_op(Tail<S> &r, const StageW<S> &w) {
    constexpr int op = ramp_down_op(S, s1, tau);
    constexpr bool last_b = down_last_is_b(S, s1, tau);
    constexpr int s = s1 - 1;
    if constexpr (op == 1) {
        const int32_t t = r.F[s] + w.F[s];
        if constexpr (last_b) {
            r.F[s] = 0;  // the forward before this one is read by no later op
            r.B[s] = max(r.B[s], t);
        } else {
            r.F[s] = t;
        }
        if constexpr (s > 0) r.F[s - 1] = add_max(t, w.pf[s - 1], r.F[s - 1]);
    } else if constexpr (op == 2) {
        const int32_t t = r.B[s] + w.B[s];
        if constexpr (last_b) {
            r.B[s] = t;
        } else {
            r.B[s] = 0;
            r.F[s] = max(r.F[s], t);
        }
        if constexpr (s + 1 < S) r.B[s + 1] = add_max(t, w.pb[s], r.B[s + 1]);
    }
}
// one level backwards: stages in ascending order
template <int S, int tau, int... i>
__device__ __forceinline__ void tail_level(Tail<S> &r, const StageW<S> &w,
                                           std::integer_sequence<int, i...>) {
    (tail_op<S, tau, i + 1>(r, w), ...);
}
template <int S, int... t>
__device__ __forceinline__ void tail_ramp(Tail<S> &r, const StageW<S> &w,
                                          std::integer_sequence<int, t...>) {
    (tail_level<S, 2 * S - 2 - t>(r, w, std::make_integer_sequence<int, S>{}), ...);
}

// One steady step (two levels); GROWTH: its largest growth of a finish.
template <int S, int P, bool GROWTH, int i>
__device__ __forceinline__ void steady_op_growth(int32_t (&Fo)[S], int32_t (&Bo)[S],
                                                 const StageW<S> &w, int32_t &grow) {
    constexpr int s = S - i - 1;
    const int32_t f = Fo[s], b = Bo[s];
    steady_op<S, P, i>(Fo, Bo, w);
    if constexpr (GROWTH) {
        if constexpr (((s + 1) & 1) == P) grow = max(grow, Fo[s] - f);
        else grow = max(grow, Bo[s] - b);
    }
}
template <int S, bool GROWTH, int... i>
__device__ __forceinline__ void steady_step(int32_t (&Fo)[S], int32_t (&Bo)[S], const StageW<S> &w,
                                            int32_t &grow, std::integer_sequence<int, i...>) {
    (steady_op_growth<S, 0, GROWTH, i>(Fo, Bo, w, grow), ...);
    (steady_op_growth<S, 1, GROWTH, i>(Fo, Bo, w, grow), ...);
}

// Steady steps before the bounds are first compared and between later
// comparisons (one of them costs about two and a half plain steps), the
// fastest of 2, 3, 4, 6, 8 and 10 with 4, 12, 16 and 24 on random plans; the
// bounds of Eager 1F1B meet for nine plans in ten after the second step.
__host__ __device__ constexpr int first_steps(int S) { return S <= 4 ? 3 : 6; }
constexpr int kFirstStepsEager = 2;
constexpr int kNextSteps = 16;

// What a caller does with a makespan: with no limit it needs the value; with
// one it only needs to know that T * scale is above the limit (the search's
// incumbent), so a lower bound above it ends the plan, and any value whose
// product is above the limit may be returned.  The bounds are then compared
// before the first steady step, where the lower one already ends 97 % of the
// complete plans of the 70B-like search, and after every few steps from then.
struct NoLimit {
    static constexpr bool kOn = false;
    __device__ __forceinline__ bool above(int32_t) const { return false; }
};
struct ObjLimit {
    static constexpr bool kOn = true;
    uint64_t scale, limit;
    __device__ __forceinline__ bool above(int32_t T) const {
        return (uint64_t)(uint32_t)T * scale > limit;
    }
};

// Makespan of a plan with M >= S.  to_end: runs until the bounds meet;
// otherwise the plan is given up after their first comparison and false is
// returned when they differ there.
template <int S, class Limit>
__device__ __forceinline__ bool makespan_fast(const StageW<S> &w, int M, bool to_end,
                                              const Limit &limit, int32_t &T) {
    Tail<S> r;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        r.F[s] = 0;
        r.B[s] = w.d[s];
    }
    tail_ramp<S>(r, w, std::make_integer_sequence<int, 2 * S - 1>{});
    int32_t Fo[S], Bo[S];
    // Warm-up, levels 1 .. S: no backward yet.  The longest path to F_{s,m}
    // visits every stage up to s once and repeats stages m - 1 times in all,
    // so it repeats the slowest of them:
    //   finish(F_{s,m}) = sum_{j<=s} F_j + sum_{j<s} pf_j + (m-1) max_{j<=s} F_j;
    // stage s runs its m = S-s+1 warm-up forwards.
    int32_t path = 0, slow = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        slow = max(slow, w.F[s]);
        path += w.F[s];
        Fo[s] = path + (S - 1 - s) * slow;
        Bo[s] = 0;
        path += w.pf[s];
    }
    // the rest of the ramp-up: levels S+1 .. 2S-1
    ramp<S, true, S + 1>(Fo, Bo, w, std::make_integer_sequence<int, S - 1>{});
    int left = M - S, steps = Limit::kOn ? 0 : first_steps(S);
    if constexpr (Limit::kOn) {
        int32_t lo = 0;
#pragma unroll
        for (int s = 0; s < S; ++s)
            lo = max(lo, add_max(Fo[s], r.F[s], Bo[s] + r.B[s]) + left * (w.F[s] + w.B[s]));
        T = lo;
        if (limit.above(lo)) return true;
    }
    for (;;) {
        const int n = min(steps, left);
        left -= n;
        int32_t grow = 0;
#pragma unroll 1
        for (int j = 0; j < n; ++j)
            steady_step<S, false>(Fo, Bo, w, grow, std::make_integer_sequence<int, S>{});
        if (left > 0) {
            steady_step<S, true>(Fo, Bo, w, grow, std::make_integer_sequence<int, S>{});
            --left;
        }
        int32_t hi = 0, lo = 0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int32_t m = add_max(Fo[s], r.F[s], Bo[s] + r.B[s]);
            hi = max(hi, m);
            lo = max(lo, m + left * (w.F[s] + w.B[s]));
        }
        T = lo;
        // hi + left * grow == lo, without overflow
        if ((int64_t)left * grow == (int64_t)(lo - hi) || limit.above(lo)) return true;
        if (!to_end) return false;
        steps = Limit::kOn ? 3 : kNextSteps;
    }
}

// ---------------------------------------------------------------------------
// Eager 1F1B (App. B): stage s (1-based) runs W_s = min(2(S-s)+1, M)
// forwards, then (B_i, F_{W_s+i}) pairs, then the remaining backwards.  In
// the unit-weight level order (stages descending within a level)
//     F_{s,m}: s + m - 1 (m <= W_s), 2m - 2S + 3s - 2 (m > W_s);
//     B_{s,m}: 2S - s + 2m - 1,
// each stage runs at most one op per level, but a stage can be two forwards
// ahead of the next one: the forward predecessor of F_{s,m} is the latest
// or the previous forward of stage s-1 (its lag, 1 or 2, is known at
// compile time).  So each stage keeps Fo (last forward), Fp (the one before)
// and Bo.  For M >= 2S-1 the levels split into a ramp-up (levels 1..2S-1),
// M-2S+1 steady two-level steps in which every stage alternates B and F
// (lag 2), and a ramp-down (levels 2M+tau, tau = -2S+2..2S-2).
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int eager_up_op(int S, int s1, int t) {
    return (t >= s1 && t <= 2 * S - s1) ? 1
           : (t >= 2 * S - s1 + 1 && ((t + s1) & 1) == 1) ? 2
           : (t >= 2 * S - s1 + 2 && ((t + s1) & 1) == 0) ? 1
                                                            : 0;
}
__host__ __device__ constexpr int eager_down_op(int S, int s1, int tau) {
    return ((((tau + s1) % 2) + 2) % 2 == 0 && tau <= 3 * s1 - 2 * S - 2) ? 1
           : ((((tau + s1) % 2) + 2) % 2 == 1 && tau <= 2 * S - s1 - 1) ? 2
                                                                          : 0;
}
__host__ __device__ constexpr bool eager_up_last_is_b(int S, int s1, int t) {
    for (int u = t - 1; u >= 1; --u)
        if (eager_up_op(S, s1, u)) return eager_up_op(S, s1, u) == 2;
    return false;
}
// before the ramp-down, the last steady level 2M-2S+1 ran F on odd stages
__host__ __device__ constexpr bool eager_down_last_is_b(int S, int s1, int tau) {
    for (int u = tau - 1; u >= -2 * S + 2; --u)
        if (eager_down_op(S, s1, u)) return eager_down_op(S, s1, u) == 2;
    return (s1 & 1) == 0;
}
// forwards of stage s1 in ramp-up levels < t / ramp-down levels < 2M+tau
__host__ __device__ constexpr int eager_up_nf(int S, int s1, int t) {
    int n = 0;
    for (int u = 1; u < t; ++u) n += eager_up_op(S, s1, u) == 1;
    return n;
}
__host__ __device__ constexpr int eager_down_nf(int S, int s1, int tau) {
    int n = 0;
    for (int u = -2 * S + 2; u < tau; ++u) n += eager_down_op(S, s1, u) == 1;
    return n;
}
// Is this op one of the warm-up forwards?  They are all done before the
// ramp-up's other ops run.
__host__ __device__ constexpr bool eager_up_warm(int S, int s1, int t) {
    return t >= s1 && t <= 2 * S - s1;
}
// forwards stage s1-1 has done beyond stage s1 before this (later) forward
__host__ __device__ constexpr int eager_up_lag(int S, int s1, int t) {
    const int warm = 2 * (S - (s1 - 1)) + 1, nf = eager_up_nf(S, s1 - 1, t);
    return (nf > warm ? nf : warm) - eager_up_nf(S, s1, t);
}
__host__ __device__ constexpr int eager_down_lag(int S, int s1, int tau) {
    return (eager_down_nf(S, s1, 2 * S - 1) - eager_down_nf(S, s1 - 1, 2 * S - 1)) +
           eager_down_nf(S, s1 - 1, tau) - eager_down_nf(S, s1, tau);
}

template <int S, int s, int LAG>
__device__ __forceinline__ void relax_f_lag(int32_t (&Fo)[S], int32_t (&Fp)[S],
                                            const StageW<S> &w, int32_t clock) {
    Fp[s] = Fo[s];
    if constexpr (s > 0) {
        static_assert(LAG == 1 || LAG == 2, "forward lag");
        Fo[s] = add_max(LAG == 2 ? Fp[s - 1] : Fo[s - 1], w.pf[s - 1], clock) + w.F[s];
    } else {
        Fo[s] = clock + w.F[s];
    }
}

template <int S, bool UP, int t, int s1>
__device__ __forceinline__ void eager_ramp_op(int32_t (&Fo)[S], int32_t (&Fp)[S], int32_t (&Bo)[S],
                                              const StageW<S> &w) {
    constexpr int op = UP ? eager_up_op(S, s1, t) : eager_down_op(S, s1, t);
    constexpr bool last_b = UP ? eager_up_last_is_b(S, s1, t) : eager_down_last_is_b(S, s1, t);
    constexpr int s = s1 - 1;
    if constexpr (UP && op == 1 && eager_up_warm(S, s1, t)) {
        // done already
    } else if constexpr (op == 1) {
        constexpr int lag = s1 == 1 ? 1 : (UP ? eager_up_lag(S, s1, t) : eager_down_lag(S, s1, t));
        relax_f_lag<S, s, lag>(Fo, Fp, w, last_b ? Bo[s] : Fo[s]);
    } else if constexpr (op == 2) {
        relax_b<S, s>(Bo, w, last_b ? Bo[s] : Fo[s]);
    }
}
template <int S, bool UP, int t, int... i>
__device__ __forceinline__ void eager_ramp_level(int32_t (&Fo)[S], int32_t (&Fp)[S],
                                                 int32_t (&Bo)[S], const StageW<S> &w,
                                                 std::integer_sequence<int, i...>) {
    (eager_ramp_op<S, UP, t, S - i>(Fo, Fp, Bo, w), ...);
}
template <int S, bool UP, int T0, int... t>
__device__ __forceinline__ void eager_ramp(int32_t (&Fo)[S], int32_t (&Fp)[S], int32_t (&Bo)[S],
                                           const StageW<S> &w, std::integer_sequence<int, t...>) {
    (eager_ramp_level<S, UP, T0 + t>(Fo, Fp, Bo, w, std::make_integer_sequence<int, S>{}), ...);
}
// steady level of parity P: stage s1 with the parity of P runs F (after its
// B, forward lag 2), the others B (after their F)
template <int S, int P, int i>
__device__ __forceinline__ void eager_steady_op(int32_t (&Fo)[S], int32_t (&Fp)[S],
                                                int32_t (&Bo)[S], const StageW<S> &w) {
    constexpr int s1 = S - i, s = s1 - 1;
    if constexpr ((s1 & 1) == P) relax_f_lag<S, s, 2>(Fo, Fp, w, Bo[s]);
    else relax_b<S, s>(Bo, w, Fo[s]);
}
// Tail, bounds and early end of the steady steps as in makespan_fast, with
// the previous forward Fp as a third finish per stage.
template <int S>
struct EagerTail {
    int32_t F[S], P[S], B[S];  // longest paths from Fo, Fp, Bo to the end
};
template <int S, int tau, int s1>
__device__ __forceinline__ void eager_tail_op(EagerTail<S> &r, const StageW<S> &w) {
    constexpr int op = eager_down_op(S, s1, tau);
    constexpr bool last_b = eager_down_last_is_b(S, s1, tau);
    constexpr int s = s1 - 1;
    if constexpr (op == 1) {
        constexpr int lag = s1 == 1 ? 1 : eager_down_lag(S, s1, tau);
        const int32_t t = r.F[s] + w.F[s];
        // the forward before this one becomes Fp; the older one is gone
        r.F[s] = last_b ? r.P[s] : max(r.P[s], t);
        r.P[s] = 0;
        if constexpr (last_b) r.B[s] = max(r.B[s], t);
        if constexpr (s > 0) {
            if constexpr (lag == 2) r.P[s - 1] = add_max(t, w.pf[s - 1], r.P[s - 1]);
            else r.F[s - 1] = add_max(t, w.pf[s - 1], r.F[s - 1]);
        }
    } else if constexpr (op == 2) {
        const int32_t t = r.B[s] + w.B[s];
        if constexpr (last_b) {
            r.B[s] = t;
        } else {
            r.B[s] = 0;
            r.F[s] = max(r.F[s], t);
        }
        if constexpr (s + 1 < S) r.B[s + 1] = add_max(t, w.pb[s], r.B[s + 1]);
    }
}
template <int S, int tau, int... i>
__device__ __forceinline__ void eager_tail_level(EagerTail<S> &r, const StageW<S> &w,
                                                 std::integer_sequence<int, i...>) {
    (eager_tail_op<S, tau, i + 1>(r, w), ...);
}
template <int S, int... t>
__device__ __forceinline__ void eager_tail_ramp(EagerTail<S> &r, const StageW<S> &w,
                                                std::integer_sequence<int, t...>) {
    (eager_tail_level<S, 2 * S - 2 - t>(r, w, std::make_integer_sequence<int, S>{}), ...);
}

template <int S, int P, bool GROWTH, int i>
__device__ __forceinline__ void eager_steady_op_growth(int32_t (&Fo)[S], int32_t (&Fp)[S],
                                                       int32_t (&Bo)[S], const StageW<S> &w,
                                                       int32_t &grow) {
    constexpr int s = S - i - 1;
    const int32_t f = Fo[s], q = Fp[s], b = Bo[s];
    eager_steady_op<S, P, i>(Fo, Fp, Bo, w);
    if constexpr (GROWTH) {
        if constexpr (((s + 1) & 1) == P) grow = max(grow, max(Fo[s] - f, f - q));
        else grow = max(grow, Bo[s] - b);
    }
}
template <int S, bool GROWTH, int... i>
__device__ __forceinline__ void eager_steady_step(int32_t (&Fo)[S], int32_t (&Fp)[S],
                                                  int32_t (&Bo)[S], const StageW<S> &w,
                                                  int32_t &grow, std::integer_sequence<int, i...>) {
    (eager_steady_op_growth<S, 0, GROWTH, i>(Fo, Fp, Bo, w, grow), ...);
    (eager_steady_op_growth<S, 1, GROWTH, i>(Fo, Fp, Bo, w, grow), ...);
}

// Stage counts whose Eager plans use the bounds.  Their tail costs about 6.5 S^2
// instructions (the ramp-down is 4S - 3 levels), more than the steady steps
// that it saves from 14 stages on (16 million plans of 14..16 stages on a GB300:
// 585 us with the bounds, 517 us without).
__host__ __device__ constexpr bool eager_bounds(int S) { return S <= 13; }

// Eager 1F1B, M >= 2S-1
template <int S, class Limit>
__device__ __forceinline__ bool makespan_eager(const StageW<S> &w, int M, bool to_end,
                                               const Limit &limit, int32_t &T) {
    EagerTail<S> r;
    if constexpr (eager_bounds(S)) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            r.F[s] = 0;
            r.P[s] = 0;
            r.B[s] = w.d[s];
        }
        eager_tail_ramp<S>(r, w, std::make_integer_sequence<int, 4 * S - 3>{});
    }
    // every stage's 2(S-s)+1 warm-up forwards by the closed form of
    // makespan_fast (they precede its backwards in the chain and depend on
    // forwards of earlier stages' warm-ups only), then the ramp-up's other ops
    int32_t Fo[S], Fp[S], Bo[S];
    int32_t path = 0, slow = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        slow = max(slow, w.F[s]);
        path += w.F[s];
        Fo[s] = path + 2 * (S - 1 - s) * slow;
        Fp[s] = s + 1 < S ? Fo[s] - slow : 0;
        Bo[s] = 0;
        path += w.pf[s];
    }
    eager_ramp<S, true, 1>(Fo, Fp, Bo, w, std::make_integer_sequence<int, 2 * S - 1>{});
    int left = M - 2 * S + 1, steps = Limit::kOn ? 1 : kFirstStepsEager;
    if constexpr (!eager_bounds(S)) {
        int32_t grow = 0;
#pragma unroll 1
        for (; left > 0; --left)
            eager_steady_step<S, false>(Fo, Fp, Bo, w, grow, std::make_integer_sequence<int, S>{});
        eager_ramp<S, false, -2 * S + 2>(Fo, Fp, Bo, w, std::make_integer_sequence<int, 4 * S - 3>{});
        T = 0;
#pragma unroll
        for (int s = 0; s < S; ++s) T = max(T, Bo[s] + w.d[s]);
        return true;
    } else for (;;) {
        const int n = min(steps, left);
        left -= n;
        int32_t grow = 0;
#pragma unroll 1
        for (int j = 0; j < n; ++j)
            eager_steady_step<S, false>(Fo, Fp, Bo, w, grow, std::make_integer_sequence<int, S>{});
        if (left > 0) {
            eager_steady_step<S, true>(Fo, Fp, Bo, w, grow, std::make_integer_sequence<int, S>{});
            --left;
        }
        int32_t hi = 0, lo = 0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int32_t m =
                add_max(Fp[s], r.P[s], add_max(Fo[s], r.F[s], Bo[s] + r.B[s]));
            hi = max(hi, m);
            lo = max(lo, m + left * (w.F[s] + w.B[s]));
        }
        T = lo;
        if ((int64_t)left * grow == (int64_t)(lo - hi) || limit.above(lo)) return true;
        if (!to_end) return false;
        steps = Limit::kOn ? 3 : kNextSteps;
    }
}

// ---------------------------------------------------------------------------
// Short pipelines: M < S under 1F1B, M < 2S-1 under Eager 1F1B (the
// evaluator; the search's leaf kernel has its own forms).
//
// The stages whose warm-up holds all M forwards run them all before their
// first backward, so up to the last such stage the forwards form a plain
// grid: F_{s,m} starts at the later of F_{s,m-1} and F_{s-1,m} + pf.  The
// last C stages (C = M under 1F1B, M/2 + 1 under Eager 1F1B) are the ones
// with shorter warm-ups and one stage before them; they are a small pipeline
// of their own whose first stage's forwards start no earlier than the grid's
// arrivals.  Their backwards then pass down the other S - C stages as a grid
// again (B_{s,1} follows B_{s+1,1}, which follows F_{s+1,M} and so F_{s,M}:
// the stage's own forwards never delay it).  So only the small pipeline has
// to be unrolled, once per M for every S, and a plan costs its 2SM
// relaxations (unrolled per (S, M) before: 120 and 240 instances, bound by
// instruction fetch).
//
// The small pipeline's ops are visited in the unit-weight ASAP level order of
// its chains, computed at compile time.  Stage s (0-based of C) runs W =
// min(C-s, M) or min(2(C-1-s)+1, M) forwards, then (B_i, F_{W+i}) pairs,
// then the remaining backwards; an op's level is one more than the later of
// its stage's previous op and its inter-stage predecessor (F_{s-1,m} for
// F_{s,m}, B_{s+1,m} for B_{s,m}).  Within a level the stages are visited in
// descending order, and while the program is built every op is checked to
// read the finish it depends on: F_{s-1,m} from stage s-1's latest forward
// (lag 1) or the one before (lag 2), B_{s+1,m} from stage s+1's latest
// backward.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int short_stages(bool eager, int M) { return eager ? M / 2 + 1 : M; }

struct ShortOp {
    int kind;      // 0 none, 1 forward, 2 backward
    int m;         // micro-batch (0-based)
    int lag;       // forward of a stage s > 0: 1 or 2
    bool clock_b;  // the stage's previous op is a backward (else a forward)
};
template <bool EAGER, int M>
struct ShortProgram {
    static constexpr int C = short_stages(EAGER, M);
    static constexpr int kMaxLevels = 2 * (M + C) + 2;
    ShortOp op[kMaxLevels][C];
    int n_levels;
    bool ok;
    __host__ __device__ constexpr ShortProgram() : op{}, n_levels(0), ok(true) {
        int kind[C][2 * M] = {}, mb[C][2 * M] = {};  // chains: op kind and micro-batch
        for (int s = 0; s < C; ++s) {
            const int w = EAGER ? 2 * (C - 1 - s) + 1 : C - s;
            const int W = w < M ? w : M;
            int n = 0;
            for (int m = 0; m < W; ++m) kind[s][n] = 1, mb[s][n++] = m;
            for (int i = 0; i < M - W; ++i) {
                kind[s][n] = 2, mb[s][n++] = i;
                kind[s][n] = 1, mb[s][n++] = W + i;
            }
            for (int m = M - W; m < M; ++m) kind[s][n] = 2, mb[s][n++] = m;
            if (s == 0 && W != M) ok = false;  // the first stage runs every forward first
        }
        int lf[C][M] = {}, lb[C][M] = {};  // ASAP levels (1-based)
        for (bool changed = true; changed;) {
            changed = false;
            for (int s = 0; s < C; ++s) {
                int prev = 0;
                for (int n = 0; n < 2 * M; ++n) {
                    const int m = mb[s][n];
                    int p = prev;
                    if (kind[s][n] == 2 && s + 1 < C && lb[s + 1][m] > p) p = lb[s + 1][m];
                    if (kind[s][n] == 1 && s > 0 && lf[s - 1][m] > p) p = lf[s - 1][m];
                    int &v = kind[s][n] == 2 ? lb[s][m] : lf[s][m];
                    if (v != p + 1) {
                        v = p + 1;
                        changed = true;
                    }
                    prev = p + 1;
                }
            }
        }
        for (int s = 0; s < C; ++s)
            for (int m = 0; m < M; ++m) {
                if (lf[s][m] > n_levels) n_levels = lf[s][m];
                if (lb[s][m] > n_levels) n_levels = lb[s][m];
            }
        if (n_levels > kMaxLevels) {
            ok = false;
            n_levels = kMaxLevels;
        }
        // registers: the micro-batch whose finish Fo / Fp / Bo of a stage
        // holds (-1: none yet) and whether its last op was a backward
        int fo[C] = {}, fp[C] = {}, bo[C] = {};
        bool last_b[C] = {};
        for (int s = 0; s < C; ++s) fo[s] = fp[s] = bo[s] = -1;
        for (int l = 1; l <= n_levels; ++l)
            for (int s = C - 1; s >= 0; --s) {
                int k = 0, m = -1;
                for (int u = 0; u < M; ++u) {
                    if (lf[s][u] == l) k = k ? 3 : 1, m = u;
                    if (lb[s][u] == l) k = k ? 3 : 2, m = u;
                }
                if (k == 3) ok = false;  // two ops of one stage in a level
                if (k == 1) {
                    int lag = 1;
                    if (s > 0) {
                        if (fo[s - 1] == m) lag = 1;
                        else if (fp[s - 1] == m) lag = 2;
                        else ok = false;
                    }
                    op[l - 1][s] = ShortOp{1, m, lag, last_b[s]};
                    fp[s] = fo[s];
                    fo[s] = m;
                    last_b[s] = false;
                } else if (k == 2) {
                    if (s + 1 < C && bo[s + 1] != m) ok = false;
                    op[l - 1][s] = ShortOp{2, m, 0, last_b[s]};
                    bo[s] = m;
                    last_b[s] = true;
                }
            }
    }
};
template <bool EAGER, int M>
struct ShortTab {
    static constexpr ShortProgram<EAGER, M> value{};
    static_assert(value.ok, "short pipeline: an op would read the wrong finish");
};

// One op of the small pipeline.  at[m]: earliest start of the first stage's
// forward m; once that has run, the finish of its backward m.
template <bool EAGER, int M, int l, int i, int C>
__device__ __forceinline__ void short_op_run(int32_t (&at)[M], int32_t (&Fo)[C], int32_t (&Fp)[C],
                                             int32_t (&Bo)[C], const StageW<C> &w) {
    constexpr int s = C - 1 - i;
    constexpr ShortOp o = ShortTab<EAGER, M>::value.op[l][s];
    if constexpr (o.kind == 1) {
        const int32_t clock = o.clock_b ? Bo[s] : Fo[s];
        if constexpr (s > 0) {
            relax_f_lag<C, s, o.lag>(Fo, Fp, w, clock);
        } else {
            Fp[0] = Fo[0];
            Fo[0] = max(at[o.m], clock) + w.F[0];
        }
    } else if constexpr (o.kind == 2) {
        relax_b<C, s>(Bo, w, o.clock_b ? Bo[s] : Fo[s]);
        if constexpr (s == 0) at[o.m] = Bo[0];
    }
}
template <bool EAGER, int M, int l, int C, int... i>
__device__ __forceinline__ void short_run_level(int32_t (&at)[M], int32_t (&Fo)[C],
                                                int32_t (&Fp)[C], int32_t (&Bo)[C],
                                                const StageW<C> &w,
                                                std::integer_sequence<int, i...>) {
    (short_op_run<EAGER, M, l, i>(at, Fo, Fp, Bo, w), ...);
}
template <bool EAGER, int M, int C, int... l>
__device__ __forceinline__ void short_run(int32_t (&at)[M], int32_t (&Fo)[C], int32_t (&Fp)[C],
                                          int32_t (&Bo)[C], const StageW<C> &w,
                                          std::integer_sequence<int, l...>) {
    (short_run_level<EAGER, M, l>(at, Fo, Fp, Bo, w, std::make_integer_sequence<int, C>{}), ...);
}

// Level program of one (schedule, S, M): per level one 64-bit word, bit s of
// bits 0-15 = stage s runs a forward, bits 16-31 = a backward, bits 32-47 =
// that forward's predecessor is the previous forward of stage s-1 (lag 2).
// Built on the host from the unit-weight ASAP levels of the schedule's
// chains (schedules.cu); used for Eager 1F1B with M < 2S-1.
template <int S>
__device__ __forceinline__ int32_t makespan_program(const StageW<S> &w, const uint64_t *prog,
                                                    int n_levels) {
    // A stage's last op finished at max(Fo, Bo) (finishes grow along its
    // chain), so no separate clock is kept.  The ops of one level are
    // independent (at most one per stage, and an op's inter-stage
    // predecessor lies on an earlier level), so a level's forwards run
    // first and its backwards second, each phase skipped when empty.
    int32_t Fo[S], Fp[S], Bo[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        Fo[s] = 0;
        Fp[s] = 0;
        Bo[s] = 0;
    }
    // the next level's word is loaded one level ahead, so the load latency
    // overlaps the current level's relaxations
    uint64_t next = n_levels > 0 ? __ldg(prog) : 0ull;
#pragma unroll 1
    for (int l = 0; l < n_levels; ++l) {
        const uint64_t word = next;
        if (l + 1 < n_levels) next = __ldg(prog + l + 1);
        const uint32_t fm = (uint32_t)word & 0xffffu, bm = (uint32_t)(word >> 16) & 0xffffu;
        const uint32_t lm = (uint32_t)(word >> 32) & 0xffffu;
        if (fm) {
#pragma unroll
            for (int s = S - 1; s >= 0; --s) {
                if ((fm >> s) & 1u) {
                    int32_t start = max(Fo[s], Bo[s]);
                    if (s > 0)
                        start = max(start, (((lm >> s) & 1u) ? Fp[s > 0 ? s - 1 : 0]
                                                             : Fo[s > 0 ? s - 1 : 0]) +
                                               w.pf[s > 0 ? s - 1 : 0]);
                    Fp[s] = Fo[s];
                    Fo[s] = start + w.F[s];
                }
            }
        }
        if (bm) {
#pragma unroll
            for (int s = S - 1; s >= 0; --s) {
                if ((bm >> s) & 1u) {
                    int32_t start = max(Fo[s], Bo[s]);
                    if (s + 1 < S) start = max(start, Bo[s + 1 < S ? s + 1 : s] + w.pb[s]);
                    Bo[s] = start + w.B[s];
                }
            }
        }
    }
    int32_t T = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) T = max(T, Bo[s] + w.d[s]);
    return T;
}

// Level programs on the device: index[(S-1)*32 + M] = (first word, levels)
// for the (S, M) pairs a schedule's short path covers.
struct Programs {
    const uint64_t *words;
    const uint2 *index;
};
// Programs of a schedule on the current device (built and uploaded on first
// use, kept for the process); words = index = NULL for 1F1B.
pos_status schedule_programs(int sched, Programs *out);

// Makespan of one decoded plan on path PATH (see makespan_fast for to_end,
// the limit and the result; the short paths always finish).
template <int S, int PATH, class Limit>
__device__ __forceinline__ bool makespan_path(const StageW<S> &w, int M, const Programs &pg,
                                              bool to_end, const Limit &limit, int32_t &T) {
    T = -1;  // S = 1 has no short path
    if constexpr (PATH == kPathFast) {
        return makespan_fast<S>(w, M, to_end, limit, T);
    } else if constexpr (PATH == kPathEager) {
        return makespan_eager<S>(w, M, to_end, limit, T);
    } else if constexpr (PATH == kPathEagerShort) {
        const uint2 ix = __ldg(pg.index + (S - 1) * 32 + M);
        T = makespan_program<S>(w, pg.words + ix.x, (int)ix.y);
    } else {
        if constexpr (S > 1)
            T = makespan_short_dispatch<S>(w, M, std::make_integer_sequence<int, S - 1>{});
    }
    return true;
}

// Path of (schedule, S, M) and the first M of the fast path.
__host__ __device__ __forceinline__ int fast_min_m(int sched, int S) {
    return sched == POS_SCHED_EAGER_1F1B ? 2 * S - 1 : S;
}
__host__ __device__ __forceinline__ int path_of(int sched, int S, int M) {
    const bool fast = M >= fast_min_m(sched, S);
    return sched == POS_SCHED_EAGER_1F1B ? (fast ? kPathEager : kPathEagerShort)
                                         : (fast ? kPathFast : kPathGeneric);
}

// ---------------------------------------------------------------------------
// Layer-level pruning (Theorem 2): for each device type the layer counts of
// its stages, in stage order, rise and then fall ("ridge-like").  A partial
// plan keeps one byte per type: bits 0-6 = layers of the type's last placed
// stage (0 = none yet), bit 7 = its counts have fallen; a type whose counts
// have fallen caps its next stage at its last count.
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ int ridge_cap(uint32_t state, int type) {
    const uint32_t b = (state >> (8 * type)) & 0xffu;
    return (b & 0x80u) ? (int)(b & 0x7fu) : 127;
}
__host__ __device__ __forceinline__ uint32_t ridge_next(uint32_t state, int type, int l) {
    const uint32_t b = (state >> (8 * type)) & 0xffu, last = b & 0x7fu;
    const uint32_t fallen = (b & 0x80u) | ((last != 0u && (uint32_t)l < last) ? 0x80u : 0u);
    return (state & ~(0xffu << (8 * type))) | ((fallen | (uint32_t)l) << (8 * type));
}
// Is a complete plan ridge-like?  cut[0..S], cls[s] = type * n_tp + tp.
template <int S>
__device__ __forceinline__ bool ridge_plan_ok(const int (&cut)[S + 1], const int (&cls)[S],
                                              int n_tp) {
    uint32_t st = 0;
    bool ok = true;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const int ty = cls[s] / n_tp, l = cut[s + 1] - cut[s];
        ok &= l <= ridge_cap(st, ty);
        st = ridge_next(st, ty, l);
    }
    return ok;
}

// Overflow guard U(S, M) >= 2^31 ?
__host__ __device__ __forceinline__ bool guard_trips(int64_t A, int64_t D, int64_t P, int S,
                                                     int M) {
    const int64_t U = (int64_t)M * A + D + 2 * (int64_t)M * (S - 1) * P;
    return U >= ((int64_t)1 << 31);
}

}  // namespace pos
