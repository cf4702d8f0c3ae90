// poseidon_eval_batch, poseidon_eval_batch_host and poseidon_argmin (hot-path
// step a9).  The evaluation kernels live in eval_kernel.cuh and the
// eval_range_*.cu instantiation units.
#include <iterator>
#include <mutex>
#include <utility>

#include "interleaved.cuh"

namespace pos {

// ---------------------------------------------------------------------------
// argmin over (makespan, index) among feasible entries, ties -> lowest index
// ---------------------------------------------------------------------------
__device__ __forceinline__ void better_of(int32_t &bt, long long &bi, int32_t t, long long i) {
    if (i >= 0 && (bi < 0 || t < bt || (t == bt && i < bi))) {
        bt = t;
        bi = i;
    }
}

// The block's best entry, in thread 0.
__device__ __forceinline__ void argmin_block(int32_t &bt, long long &bi) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int32_t ot = __shfl_down_sync(0xffffffffu, bt, o);
        const long long oi = __shfl_down_sync(0xffffffffu, bi, o);
        better_of(bt, bi, ot, oi);
    }
    __shared__ int32_t st[kArgminThreads / 32];
    __shared__ long long si[kArgminThreads / 32];
    if ((threadIdx.x & 31) == 0) {
        st[threadIdx.x >> 5] = bt;
        si[threadIdx.x >> 5] = bi;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < kArgminThreads / 32; ++w) better_of(bt, bi, st[w], si[w]);
}

// Best entry of every block, or, launched as one block, the answer itself
// (out).  Bound by the latency of its loads: a thread takes 16 entries at a
// time, the flags as one 16-byte word (VEC: flags and makespans 16-byte
// aligned), and reads the makespans of a word of four flags only when one of
// them is feasible.  A 20-million-candidate evaluation with its argmin went
// from 2948 to 2851 us on a GB300 with these kernels, one of 250,007 from
// 146.5 to 105.2 us (one entry per thread and iteration, the partial results
// reduced by one thread, scratch from the device's default pool before).
template <bool VEC>
__global__ void __launch_bounds__(kArgminThreads) argmin_partial(const int32_t *T, const uint8_t *F,
                                                                 int64_t n, int32_t *part_t,
                                                                 long long *part_i, int64_t *out) {
    int32_t bt = 0;
    long long bi = -1;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n16 = VEC ? n / 16 : 0;
    if constexpr (VEC) {
        const uint4 *F16 = reinterpret_cast<const uint4 *>(F);
        const int4 *T4 = reinterpret_cast<const int4 *>(T);
#pragma unroll 2
        for (int64_t g = tid; g < n16; g += stride) {
            const uint4 f = __ldg(F16 + g);
            const uint32_t w[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t yes = __vcmpeq4(w[q], POS_FEAS_YES * 0x01010101u);
                if (yes == 0u) continue;
                const int4 t = __ldg(T4 + 4 * g + q);
                const long long i = 16 * g + 4 * q;
                if (yes & 0x000000ffu) better_of(bt, bi, t.x, i);
                if (yes & 0x0000ff00u) better_of(bt, bi, t.y, i + 1);
                if (yes & 0x00ff0000u) better_of(bt, bi, t.z, i + 2);
                if (yes & 0xff000000u) better_of(bt, bi, t.w, i + 3);
            }
        }
    }
    for (int64_t i = 16 * n16 + tid; i < n; i += stride)
        if (F[i] == POS_FEAS_YES) better_of(bt, bi, T[i], i);
    argmin_block(bt, bi);
    grid_dep_trigger();
    if (threadIdx.x == 0) {
        if (out) {
            *out = bi;
        } else {
            part_t[blockIdx.x] = bt;
            part_i[blockIdx.x] = bi;
        }
    }
}

// One block over the partial results (a single thread took 75 us for 608
// of them, one dependent load after another).
__global__ void __launch_bounds__(kArgminThreads) argmin_final(const int32_t *part_t,
                                                               const long long *part_i, int parts,
                                                               int64_t *out) {
    grid_dep_wait();  // the partial results
    int32_t bt = 0;
    long long bi = -1;
    for (int q = threadIdx.x; q < parts; q += kArgminThreads)
        better_of(bt, bi, part_t[q], part_i[q]);
    argmin_block(bt, bi);
    if (threadIdx.x == 0) *out = bi;
}

// Does the partial kernel read 16 entries at a time?
static bool argmin_vec(const int32_t *T, const uint8_t *F) {
    return ((reinterpret_cast<uintptr_t>(T) | reinterpret_cast<uintptr_t>(F)) & 15) == 0;
}

// Blocks of the partial kernel: one where each thread has few dependent loads
// (up to 16384 entries in words of 16, 1024 one by one: less than a second
// launch costs), else a thread per word or entry up to four blocks per SM.
// Entries one by one, all in one block / so, on a GB300: 8.2 / 6.2 us for
// 3,001, 14.3 / 6.9 for 8,192, 24.6 / 7.3 for 16,384.
int64_t argmin_parts(const int32_t *T, const uint8_t *F, int64_t n) {
    const bool vec = argmin_vec(T, F);
    if (n <= (vec ? 64 : 4) * kArgminThreads) return 1;
    const int64_t per = (vec ? 16 : 1) * kArgminThreads;
    return std::min<int64_t>((n + per - 1) / per, 4LL * sm_count());
}

// part_t, part_i: argmin_parts() entries each (not used when that is 1).
pos_status launch_argmin(const int32_t *T, const uint8_t *F, int64_t n, int32_t *part_t,
                         long long *part_i, int64_t *out, cudaStream_t stream) {
    const int parts = (int)argmin_parts(T, F, n);
    int64_t *direct = parts == 1 ? out : nullptr;
    if (argmin_vec(T, F))
        argmin_partial<true><<<parts, kArgminThreads, 0, stream>>>(T, F, n, part_t, part_i, direct);
    else
        argmin_partial<false><<<parts, kArgminThreads, 0, stream>>>(T, F, n, part_t, part_i, direct);
    POS_CUDA(cudaGetLastError());
    if (parts > 1)
        POS_CUDA(launch_dependent(argmin_final, 1, kArgminThreads, 0, stream, part_t, part_i, parts,
                                  out));
    return POS_OK;
}

// ---------------------------------------------------------------------------
// counting sort of the candidates by (S, M) key
// ---------------------------------------------------------------------------
// il_key: kIlKeyOf staged in shared memory (a __constant__ read whose index
// differs between the lanes of a warp is served one address at a time)
__device__ __forceinline__ int eval_key(int sched, uint32_t w, const int16_t *il_key) {
    const int S = w & 0xff, M = (w >> 8) & 0xff, V = (int)(w >> 24);
    if (S < 1 || S > POS_MAX_STAGES || M < 1) return -1;
    if (sched == POS_SCHED_INTERLEAVED_1F1B && V >= 2) {
        // N = S devices, V chunks each: key block of (N, V), index q = M / N
        if (S * V > POS_MAX_STAGES || M % S != 0) return -1;
        return kKeys + il_key[(S - 1) * 17 + V] + M / S;
    }
    return M >= fast_min_m(sched, S) ? fast_key_begin(S) + M / 8 : short_key_begin(M) + S - 1;
}

// global key histogram; invalid records are answered right here
// 2-byte key per candidate, written by the histogram pass and read by the
// scatter pass (instead of the 16-byte record, twice)
constexpr uint16_t kNoKey = 0xffff;

// The S | M << 8 | tp << 16 | V << 24 word of record i (24-byte records:
// S, M, V at bytes 16..18, tp = 0).
__device__ __forceinline__ uint32_t record_word(const EvalParams &p, int64_t i) {
    if (p.per_stage_tp) {
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(p.cands_ex) + 6 * i + 4);
        return (w & 0xffffu) | ((w & 0xff0000u) << 8);
    }
    return __ldg(&p.cands[i].w);
}

template <int NK>
__global__ void sort_hist_kernel(EvalParams p, int64_t n, uint32_t *hist, uint16_t *keys,
                                 int32_t *T, uint8_t *F) {
    const int sched = p.lay.sched;
    __shared__ uint32_t h[NK];
    __shared__ int16_t il_key[8 * 17];
    for (int i = threadIdx.x; i < NK; i += blockDim.x) h[i] = 0;
    if (sched == POS_SCHED_INTERLEAVED_1F1B)
        for (int i = threadIdx.x; i < 8 * 17; i += blockDim.x) il_key[i] = kIlKeyOf[i / 17][i % 17];
    __syncthreads();
    // four record words in flight per thread (the pass is bound by HBM
    // latency: one load per thread and iteration kept too few bytes in flight)
    const int64_t bd = blockDim.x;
    for (int64_t i0 = blockIdx.x * 4 * bd + threadIdx.x; i0 < n; i0 += (int64_t)gridDim.x * 4 * bd) {
        uint32_t wv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) wv[u] = i0 + u * bd < n ? record_word(p, i0 + u * bd) : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t i = i0 + u * bd;
            if (i >= n) break;
            const int k = eval_key(sched, wv[u], il_key);
            keys[i] = k >= 0 ? (uint16_t)k : kNoKey;
            if (k >= 0) {
                atomicAdd(&h[k], 1u);
            } else {
                T[i] = -1;
                F[i] = POS_FEAS_INVALID;
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < NK; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// Each block takes chunks of `chunk` candidates: counts their keys, reserves
// one range per key with a single atomic, then gives every candidate its
// sorted position (written in input order, so coalesced).  Chunks of up to
// 16384 for large batches (measured against 4096, 8192 and 32768: within
// 0.5 % of a config-5 call, 16384 the fastest), smaller ones (down to 1024)
// so that small batches still spread over the SMs.
// Within a chunk the candidates of one key get consecutive positions, so
// the decode pass's scattered record writes come in short runs.
__host__ inline int64_t scatter_chunk(int64_t n, int sms) {
    int64_t c = (n / (8 * (int64_t)sms) + 511) & ~(int64_t)511;
    return c < 1024 ? 1024 : (c > 16384 ? 16384 : c);
}

constexpr uint32_t kNoDest = 0xffffffffu;

// Every block first makes the start of each key, the exclusive prefix sum of
// the histogram, for itself (a scan kernel of one block between the two passes
// took 6 us, 14 us with the interleaved keys); block 0 writes it to offs for
// the makespan kernels.  cursor: the positions of each key taken so far.
constexpr int kScatterThreads = 512;
template <int NK>
__global__ void __launch_bounds__(kScatterThreads) sort_scatter_kernel(
    const uint16_t *keys, int64_t n, int64_t chunk, const uint32_t *hist, uint32_t *offs,
    uint32_t *cursor, uint32_t *dest) {
    extern __shared__ uint32_t s_sort[];
    uint32_t *start = s_sort, *h = s_sort + NK;
    __shared__ uint32_t warp_total[kScatterThreads / 32];
    grid_dep_wait();  // the keys and their histogram
    grid_dep_trigger();
    {
        constexpr int per = (NK + kScatterThreads - 1) / kScatterThreads;
        const int lo = threadIdx.x * per, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        uint32_t v[per], sum = 0;
#pragma unroll
        for (int i = 0; i < per; ++i) {
            v[i] = lo + i < NK ? __ldg(hist + lo + i) : 0u;
            sum += v[i];
        }
        uint32_t incl = sum;  // over the warp's lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) warp_total[wid] = incl;
        __syncthreads();
        uint32_t run = incl - sum;
        for (int w = 0; w < wid; ++w) run += warp_total[w];
#pragma unroll
        for (int i = 0; i < per; ++i) {
            if (lo + i < NK) {
                start[lo + i] = run;
                if (blockIdx.x == 0) offs[lo + i] = run;
            }
            run += v[i];
        }
        if (blockIdx.x == 0 && threadIdx.x == kScatterThreads - 1) offs[NK] = run;
    }
    for (int64_t c0 = blockIdx.x * chunk; c0 < n; c0 += (int64_t)gridDim.x * chunk) {
        const int64_t c1 = min(n, c0 + chunk);
        for (int i = threadIdx.x; i < NK; i += blockDim.x) h[i] = 0;
        __syncthreads();
        for (int64_t i = c0 + threadIdx.x; i < c1; i += blockDim.x) {
            const uint16_t k = __ldg(keys + i);
            if (k != kNoKey) atomicAdd(&h[k], 1u);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < NK; i += blockDim.x)
            if (h[i]) h[i] = start[i] + atomicAdd(&cursor[i], h[i]);
        __syncthreads();
        for (int64_t i = c0 + threadIdx.x; i < c1; i += blockDim.x) {
            const uint16_t k = __ldg(keys + i);
            dest[i] = k != kNoKey ? atomicAdd(&h[k], 1u) : kNoDest;
        }
        __syncthreads();
    }
}

template <int NK>
static pos_status launch_sort(const EvalParams &p, int64_t m, uint32_t *hist, uint32_t *offs,
                              uint32_t *cursor, uint32_t *dest, uint16_t *keys,
                              cudaStream_t stream) {
    // histogram pass: 256 threads, four candidates per thread and round
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((m + 1023) / 1024, 4LL * sm_count()));
    const int64_t chunk = scatter_chunk(m, sm_count());
    const int sgrid = (int)std::max<int64_t>(
        1, std::min<int64_t>((m + chunk - 1) / chunk, 8LL * sm_count()));
    auto scatter = sort_scatter_kernel<NK>;
    const int smem = 2 * NK * (int)sizeof(uint32_t);
    POS_TRY(ensure_smem(reinterpret_cast<const void *>(scatter), smem));
    // the histogram follows a memset; the kernels after it are chained by
    // programmatic dependent launch
    sort_hist_kernel<NK><<<grid, 256, 0, stream>>>(p, m, hist, keys, p.T, p.F);
    POS_CUDA(cudaGetLastError());
    POS_CUDA(launch_dependent(scatter, sgrid, kScatterThreads, smem, stream,
                              static_cast<const uint16_t *>(keys), m, chunk,
                              static_cast<const uint32_t *>(hist), offs, cursor, dest));
    return POS_OK;
}

// Decode pass.  Blocks take windows of `window` consecutive candidates:
// their records and sorted positions are read coalesced into shared memory,
// and each decoded 32-byte record is written to its sorted position.  The
// decode's cost grows with the number of unranking stages (S, or N*V for an
// interleaved record) and a window mixes them, so the block orders the
// window's candidates by that count (a counting sort over 16 buckets) and
// its warps then decode 32 consecutive entries of that order at a time:
// the lanes of a warp loop over (nearly) the same number of stages.
// Bound by issue slots (the steps' integer work; 20 million 1F1B plans on a
// GB300, in blocks of 256: 438 us, 609 us with estimated binomial inverses).
// Blocks of 512 on windows of 1536: half the table copies and rounder warps than
// 256 on 768 at the same 32 warps per SM (calls, 256 / 512: 16 million 1496 / 1469
// us, 250,007 with 24-byte records 60.1 / 56.1; three blocks of 512 with 40
// registers 1473 and 56.4, but a million interleaved plans 254 / 250 / 260).
// LIM: only the binomials (the blob's first off_Pw bytes), their inverse and
// the memory-limit table are staged, one after the other.
constexpr int kDecodeThreads = 512;
constexpr int kDecodeWindowMax = 1536;
constexpr int kDecodeBuckets = POS_MAX_STAGES + 1;  // stage counts 1..16 (0 unused)

__device__ __forceinline__ int decode_bucket(int sched, uint32_t w) {
    const int S = w & 0xff, V = (int)(w >> 24);
    const int J = (sched == POS_SCHED_INTERLEAVED_1F1B && V >= 2) ? S * V : S;
    return min(max(J, 1), POS_MAX_STAGES);  // records beyond are answered at once
}

// the two 16-byte words of a decoded record in one 32-byte store
__device__ __forceinline__ void store_decoded(uint4 *dst, const uint4 &a, const uint4 &b) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst),
                 "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}

struct DecodeWindow {
    uint4 rec[kDecodeWindowMax];       // RecView::rec of each candidate
    uint32_t tpc[kDecodeWindowMax];    // RecView::tpc
    uint32_t dest[kDecodeWindowMax];   // sorted position (kNoDest: no key)
    uint16_t order[kDecodeWindowMax];  // window offsets in bucket order
    uint8_t bucket[kDecodeWindowMax];  // bucket of each candidate (0: no key)
    uint32_t slot[kDecodeBuckets + 1]; // bucket counts, then next free slots
    uint32_t n_valid;
};

template <bool LIM>
__global__ void __launch_bounds__(kDecodeThreads, 2) decode_kernel(EvalParams p, int window) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ DecodeWindow win;
    if constexpr (LIM) {
        stage_blob(sm, p.blob, p.lay.off_Pw);
        stage_blob(sm + p.lay.off_Pw, static_cast<const unsigned char *>(p.blob) + p.inv_off,
                   p.inv_bytes + p.lim_bytes);
    } else {
        stage_blob(sm, p.blob, p.lay.bytes);
    }
    __syncthreads();
    grid_dep_wait();  // the sorted positions (scatter pass)
    grid_dep_trigger();
    const Tab t = tab_at(sm, p.lay);
    const uint8_t *inv = sm + p.lay.off_Pw, *lim = inv + p.inv_bytes;
    const int sched = p.lay.sched;
    const int lane = threadIdx.x & 31;
    for (int64_t w0 = blockIdx.x * (int64_t)window; w0 < p.n; w0 += (int64_t)gridDim.x * window) {
        const int wn = (int)min((int64_t)window, p.n - w0);
        // 1. the window's records and positions, and the candidates per
        // bucket (those without a key are already answered)
        if (threadIdx.x <= kDecodeBuckets) win.slot[threadIdx.x] = 0;
        __syncthreads();
#pragma unroll 4
        for (int li = threadIdx.x; li < wn; li += kDecodeThreads) {
            const uint32_t i = (uint32_t)(w0 + li);
            const RecView v = load_record(p, i);
            const uint32_t d = __ldg(p.dest + i);
            win.rec[li] = v.rec;
            win.tpc[li] = v.tpc;
            win.dest[li] = d;
            const int b = d != kNoDest ? decode_bucket(sched, v.rec.w) : 0;
            win.bucket[li] = (uint8_t)b;
            if (b) atomicAdd(&win.slot[b], 1u);
        }
        __syncthreads();
        // 2. exclusive prefix over the buckets (first warp)
        if (threadIdx.x < 32) {
            const uint32_t c = lane <= kDecodeBuckets ? win.slot[lane] : 0u;
            uint32_t incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane <= kDecodeBuckets) win.slot[lane] = incl - c;
            if (lane == 31) win.n_valid = incl;
        }
        __syncthreads();
        // 3. the window's offsets in bucket order
        for (int li = threadIdx.x; li < wn; li += kDecodeThreads) {
            const int b = win.bucket[li];
            if (b) win.order[atomicAdd(&win.slot[b], 1u)] = (uint16_t)li;
        }
        __syncthreads();
        // 4. decode: each warp takes 32 consecutive entries of the order
        const int nv = (int)win.n_valid;
        for (int k = threadIdx.x; k < nv; k += kDecodeThreads) {
            const int li = win.order[k];
            const uint32_t i = (uint32_t)(w0 + li);
            const uint4 rec = win.rec[li];
            const uint32_t tpc = win.tpc[li];
            const uint4 out = decode_one<LIM>(t, rec, tpc, p, i, inv, lim);
            store_decoded(p.cuts + 2 * (size_t)win.dest[li], out, make_uint4(i, rec.z, rec.w, tpc));
        }
        __syncthreads();  // the window's arrays are rewritten for the next one
    }
}

pos_status launch_decode(const EvalParams &p, cudaStream_t stream) {
    const bool lim = p.lim_bytes > 0;
    const void *kern = lim ? reinterpret_cast<const void *>(decode_kernel<true>)
                           : reinterpret_cast<const void *>(decode_kernel<false>);
    const int smem = lim ? p.lay.off_Pw + p.inv_bytes + p.lim_bytes : p.lay.bytes;
    POS_TRY(ensure_smem(kern, smem));
    int per_sm = 0;
    POS_TRY(blocks_per_sm(kern, kDecodeThreads, smem, &per_sm));
    // blocks of at least 1024 candidates; the same number of windows for
    // every block (up to one), so that the blocks finish together
    const int64_t blocks = std::max<int64_t>(
        1, std::min<int64_t>((p.n + 1023) / 1024, (int64_t)std::max(per_sm, 1) * sm_count()));
    const int64_t rounds = (p.n + blocks * kDecodeWindowMax - 1) / (blocks * kDecodeWindowMax);
    const int window = (int)((p.n + blocks * rounds - 1) / (blocks * rounds));
    if (lim) POS_CUDA(launch_dependent(decode_kernel<true>, (int)blocks, kDecodeThreads, smem, stream, p, window));
    else POS_CUDA(launch_dependent(decode_kernel<false>, (int)blocks, kDecodeThreads, smem, stream, p, window));
    return POS_OK;
}

// Stream-ordered scratch comes from a library-owned pool per device that
// keeps its memory between calls (release threshold: unlimited), so what is
// taken from it is bounded: 39 bytes per candidate of a chunk of 2^24, an
// argmin's partial results, and host batches up to kHostPoolBytes.
constexpr size_t kHostPoolBytes = 64ull << 20;
static std::mutex g_pool_mutex;
static cudaMemPool_t g_pool[64];

static pos_status scratch_pool(cudaMemPool_t *out) {
    int dev = 0;
    POS_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(POS_EINVAL, "device index above 63");
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    if (!g_pool[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool;
        POS_CUDA(cudaMemPoolCreate(&pool, &props));
        uint64_t keep = ~0ull;
        POS_CUDA(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep));
        g_pool[dev] = pool;
    }
    *out = g_pool[dev];
    return POS_OK;
}

// Side streams per device.  Every makespan kernel depends only on the decode
// pass, so the ranges of a batch run on the caller's stream and on these: none
// keeps every issue slot busy (small batches: the latency of a range's slowest
// warps; large ones: the kernels' ends, and instruction fetch), the longest on
// the caller's stream.  One side stream / three on a GB300: 1F1B 93 / 73 us at
// 250,007 plans, 910 / 882 us at 8 million; Eager 245 / 205 us at a million;
// Interleaved 297 / 258 us at a million, but 1748 / 1870 us at 8 million, where
// its large kernels evict one another's code.  The fork and join events are
// shared per device, so a call holds the device's side mutex from the fork to
// the join (two calls from different host threads must not interleave their
// record / wait pairs).
constexpr int kSides = 3;
constexpr int64_t kSpreadMaxIl = 1 << 22;  // interleaved batches on all streams
struct SideStream {
    cudaStream_t s[kSides] = {};
    cudaEvent_t fork = nullptr, join[kSides] = {};
    std::mutex mu;
};
static std::mutex g_side_mutex;
static SideStream g_side[64];

static pos_status side_stream(SideStream **out) {
    int dev = 0;
    POS_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(POS_EINVAL, "device index above 63");
    std::lock_guard<std::mutex> lock(g_side_mutex);
    SideStream &ss = g_side[dev];
    if (!ss.fork) POS_CUDA(cudaEventCreateWithFlags(&ss.fork, cudaEventDisableTiming));
    for (int i = 0; i < kSides; ++i) {
        if (!ss.join[i]) POS_CUDA(cudaEventCreateWithFlags(&ss.join[i], cudaEventDisableTiming));
        if (!ss.s[i]) POS_CUDA(cudaStreamCreateWithFlags(&ss.s[i], cudaStreamNonBlocking));
    }
    *out = &ss;
    return POS_OK;
}

// A makespan kernel and its stream: 0 the caller's, 1.. a side stream.
struct RangeLaunch {
    pos_status (*launch)(const EvalParams &, cudaStream_t);
    int at;
};
static const RangeLaunch kRanges1F1B[] = {
    {eval_short_1_9, 1}, {eval_short_10_15, 1}, {eval_fast_13_16, 0},
    {eval_fast_9_12, 2}, {eval_fast_5_8, 3},    {eval_fast_1_4, 3}};
static const RangeLaunch kRangesEager[] = {
    {eval_eager_short_23_30, 1}, {eval_eager_short_15_22, 1}, {eval_eager_short_1_14, 1},
    {eval_eager_14_16, 0},       {eval_eager_11_13, 2},       {eval_eager_7_10, 3},
    {eval_eager_1_6, 2}};
// interleaved handle: the 1F1B ranges hold its records with V < 2, usually none
static const RangeLaunch kRangesIl[] = {
    {eval_il_12_22, 0},   {eval_il_23_29, 2},    {eval_il_32_33, 3}, {eval_il_0_11, 3},
    {eval_short_1_9, 1},  {eval_short_10_15, 1}, {eval_fast_1_4, 1}, {eval_fast_5_8, 1},
    {eval_fast_9_12, 1},  {eval_fast_13_16, 1},  {eval_il_30_31, 2}};
static const RangeLaunch kRangesIlLarge[] = {
    {eval_short_1_9, 1},  {eval_short_10_15, 1}, {eval_fast_1_4, 1}, {eval_fast_5_8, 1},
    {eval_fast_9_12, 1},  {eval_fast_13_16, 1},  {eval_il_30_31, 1}, {eval_il_0_11, 0},
    {eval_il_12_22, 0},   {eval_il_23_29, 0},    {eval_il_32_33, 0}};

static pos_status launch_ranges(const EvalParams &p, cudaStream_t stream) {
    const RangeLaunch *r = kRanges1F1B;
    int n = (int)std::size(kRanges1F1B), sides = kSides;
    if (p.lay.sched == POS_SCHED_EAGER_1F1B) {
        r = kRangesEager;
        n = (int)std::size(kRangesEager);
    } else if (p.lay.sched == POS_SCHED_INTERLEAVED_1F1B) {
        const bool large = p.n > kSpreadMaxIl;
        r = large ? kRangesIlLarge : kRangesIl;
        n = (int)std::size(kRangesIl);
        if (large) sides = 1;
    }
    SideStream *ss = nullptr;
    POS_TRY(side_stream(&ss));
    std::lock_guard<std::mutex> lock(ss->mu);
    // fork: the side streams start after the decode pass
    POS_CUDA(cudaEventRecord(ss->fork, stream));
    pos_status st = POS_OK;
    cudaError_t e = cudaSuccess;
    int forked = 0;
    for (; forked < sides && e == cudaSuccess; ++forked)
        e = cudaStreamWaitEvent(ss->s[forked], ss->fork, 0);
    for (int i = 0; i < n && e == cudaSuccess && st == POS_OK; ++i) {
        st = r[i].launch(p, r[i].at == 0 ? stream : ss->s[r[i].at - 1]);
    }
    // join, also after a failed launch (the side streams' queued work stays
    // ordered before the scratch is freed)
    for (int i = 0; i < forked; ++i) {
        cudaError_t ej = cudaEventRecord(ss->join[i], ss->s[i]);
        if (ej == cudaSuccess) ej = cudaStreamWaitEvent(stream, ss->join[i], 0);
        if (e == cudaSuccess) e = ej;
    }
    POS_TRY(st);
    POS_CUDA(e);
    return POS_OK;
}

// Kernel parameters of candidates [base, base + m) of a batch, without the
// sorted path's scratch.
static EvalParams eval_params(const Handle *h, const void *d_cands, bool per_stage_tp, int64_t base,
                              int64_t m, int32_t *d_T, uint8_t *d_F) {
    EvalParams p = {};
    p.per_stage_tp = per_stage_tp ? 1 : 0;
    p.cands = per_stage_tp ? nullptr : static_cast<const uint4 *>(d_cands) + base;
    p.cands_ex = per_stage_tp ? static_cast<const uint2 *>(d_cands) + 3 * base : nullptr;
    p.n = m;
    p.T = d_T + base;
    p.F = d_F + base;
    set_tables(p, h->d_blob, h->lay);
    for (int J = 1; J <= POS_MAX_STAGES; ++J) {  // smallest tripping M, by bisection
        int lo = 1, hi = 256;
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (guard_trips(h->guard_A, h->guard_D, h->guard_P, J, mid)) hi = mid;
            else lo = mid + 1;
        }
        p.guard_m[J] = (uint16_t)lo;
    }
    p.guard_m[0] = 0;
    p.sms = sm_count();
    p.lim_w = h->lim_w;
    p.lim_bytes = h->lim_bytes;
    p.inv_off = h->inv_off;
    p.inv_bytes = h->inv_bytes;
    p.inv_narrow = h->inv_narrow;
    return p;
}

// d_cands: 16-byte records, or 24-byte records when per_stage_tp.
pos_status launch_eval(Handle *h, const void *d_cands, bool per_stage_tp, int64_t n,
                       int32_t *d_T, uint8_t *d_F, cudaStream_t stream) {
    if (n == 0) return POS_OK;
    const bool il = h->lay.sched == POS_SCHED_INTERLEAVED_1F1B;
    if (n <= lane_max(h->lay.sched))
        return launch_lanes(eval_params(h, d_cands, per_stage_tp, 0, n, d_T, d_F), stream);
    cudaMemPool_t pool;
    pos_status st = scratch_pool(&pool);
    if (st != POS_OK) return st;
    // batches above 2^24 candidates go in chunks of 2^24: a chunk's outputs
    // (5 bytes per candidate, 80 MB), written in sorted order and so
    // scattered over the output arrays, stay in L2 until whole sectors are
    // written back (the 32-bit sorted positions would allow 2^31)
    const int64_t chunk = (int64_t)1 << 24;
    for (int64_t base = 0; base < n; base += chunk) {
        const int64_t m = std::min(chunk, n - base);
        void *scratch = nullptr;
        const int nk = il ? kKeysIl : kKeys;
        // scratch: decoded records (32 B per candidate), the sort arrays, the keys
        constexpr int kTiles = POS_MAX_STAGES + 1;
        const size_t sbytes = 32 * (size_t)m +
                              sizeof(uint32_t) * (kTiles + 3 * (size_t)nk + 1 + (size_t)m) +
                              sizeof(uint16_t) * (size_t)m;
        POS_CUDA(cudaMallocFromPoolAsync(&scratch, sbytes, pool, stream));
        uint4 *cuts = static_cast<uint4 *>(scratch);
        uint32_t *tiles = reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + 32 * (size_t)m);
        uint32_t *hist = tiles + kTiles;
        uint32_t *cursor = hist + nk;
        uint32_t *offs = cursor + nk;
        uint32_t *dest = offs + nk + 1;
        uint16_t *keys = reinterpret_cast<uint16_t *>(dest + m);
        EvalParams p = eval_params(h, d_cands, per_stage_tp, base, m, d_T, d_F);
        p.dest = dest;
        p.offs = offs;
        p.cuts = cuts;
        p.tiles = tiles;
        cudaError_t e = cudaMemsetAsync(tiles, 0, sizeof(uint32_t) * (kTiles + 2 * (size_t)nk), stream);
        if (e == cudaSuccess)
            st = il ? launch_sort<kKeysIl>(p, m, hist, offs, cursor, dest, keys, stream)
                    : launch_sort<kKeys>(p, m, hist, offs, cursor, dest, keys, stream);
        if (e == cudaSuccess && st == POS_OK) st = launch_decode(p, stream);
        if (e == cudaSuccess && st == POS_OK) st = launch_ranges(p, stream);
        const cudaError_t e2 = cudaFreeAsync(scratch, stream);
        if (e != cudaSuccess) return cuda_fail(e, "eval sort launch");
        if (st != POS_OK) return st;
        if (e2 != cudaSuccess) return cuda_fail(e2, "eval scratch free");
    }
    return POS_OK;
}

}  // namespace pos

extern "C" {

pos_status poseidon_eval_batch(void *handle, const pos_candidate *d_cands, int64_t n,
                               int32_t *d_makespan, uint8_t *d_feasible, void *stream) {
    if (!handle) return pos::fail(POS_EINVAL, "handle is NULL");
    if (n < 0) return pos::fail(POS_EINVAL, "n < 0");
    if (n > 0 && (!d_cands || !d_makespan || !d_feasible))
        return pos::fail(POS_EINVAL, "NULL buffer");
    if ((reinterpret_cast<uintptr_t>(d_cands) & 15) != 0)
        return pos::fail(POS_EINVAL, "candidates must be 16-byte aligned");
    return pos::launch_eval(static_cast<pos::Handle *>(handle), d_cands, false, n, d_makespan,
                            d_feasible, static_cast<cudaStream_t>(stream));
}

pos_status poseidon_eval_batch_ex(void *handle, const pos_candidate_ex *d_cands, int64_t n,
                                  int32_t *d_makespan, uint8_t *d_feasible, void *stream) {
    if (!handle) return pos::fail(POS_EINVAL, "handle is NULL");
    if (n < 0) return pos::fail(POS_EINVAL, "n < 0");
    if (n > 0 && (!d_cands || !d_makespan || !d_feasible))
        return pos::fail(POS_EINVAL, "NULL buffer");
    if ((reinterpret_cast<uintptr_t>(d_cands) & 7) != 0)
        return pos::fail(POS_EINVAL, "candidates must be 8-byte aligned");
    pos::Handle *h = static_cast<pos::Handle *>(handle);
    if (h->lay.n_tp > 4)
        return pos::fail(POS_EINVAL, "per-stage TP records need n_tp <= 4 (2-bit TP fields)");
    return pos::launch_eval(h, d_cands, true, n, d_makespan, d_feasible,
                            static_cast<cudaStream_t>(stream));
}

pos_status poseidon_eval_batch_host(void *handle, const pos_candidate *cands, int64_t n,
                                    int32_t *makespan, uint8_t *feasible) {
    if (!handle) return pos::fail(POS_EINVAL, "handle is NULL");
    if (n < 0) return pos::fail(POS_EINVAL, "n < 0");
    if (n == 0) return POS_OK;
    if (!cands || !makespan || !feasible) return pos::fail(POS_EINVAL, "NULL buffer");
    // stream-ordered on the default stream.  Up to kHostPoolBytes the buffers
    // come from the library's pool (a cudaMalloc and cudaFree pair takes 60 us
    // per call); larger ones, whose copies take 100 times that, are given back,
    // since the pool keeps what it once held
    cudaMemPool_t pool;
    POS_TRY(pos::scratch_pool(&pool));
    void *d = nullptr;
    const size_t bc = sizeof(pos_candidate) * (size_t)n, bt = sizeof(int32_t) * (size_t)n;
    const size_t bytes = bc + bt + (size_t)n;
    const bool pooled = bytes <= pos::kHostPoolBytes;
    POS_CUDA(pooled ? cudaMallocFromPoolAsync(&d, bytes, pool, 0) : cudaMalloc(&d, bytes));
    pos_candidate *dc = static_cast<pos_candidate *>(d);
    int32_t *dt = reinterpret_cast<int32_t *>(static_cast<char *>(d) + bc);
    uint8_t *df = reinterpret_cast<uint8_t *>(static_cast<char *>(d) + bc + bt);
    pos_status st = POS_OK;
    cudaError_t e = cudaMemcpyAsync(dc, cands, bc, cudaMemcpyHostToDevice, 0);
    if (e == cudaSuccess) {
        st = pos::launch_eval(static_cast<pos::Handle *>(handle), dc, false, n, dt, df, 0);
        if (st == POS_OK) e = cudaMemcpyAsync(makespan, dt, bt, cudaMemcpyDeviceToHost, 0);
        if (st == POS_OK && e == cudaSuccess)
            e = cudaMemcpyAsync(feasible, df, (size_t)n, cudaMemcpyDeviceToHost, 0);
    }
    cudaError_t e2 = pooled ? cudaFreeAsync(d, 0) : cudaSuccess;
    const cudaError_t e3 = cudaStreamSynchronize(0);
    if (!pooled) e2 = cudaFree(d);
    if (e == cudaSuccess) e = e2 != cudaSuccess ? e2 : e3;
    if (e != cudaSuccess) return pos::cuda_fail(e, "eval_batch_host copies");
    return st;
}

pos_status poseidon_argmin(const int32_t *d_makespan, const uint8_t *d_feasible, int64_t n,
                           int64_t *d_out, void *stream) {
    if (n < 0 || !d_out || (n > 0 && (!d_makespan || !d_feasible)))
        return pos::fail(POS_EINVAL, "bad argmin arguments");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int64_t parts = pos::argmin_parts(d_makespan, d_feasible, n);
    if (parts == 1) return pos::launch_argmin(d_makespan, d_feasible, n, nullptr, nullptr, d_out, s);
    // from the library's pool, which keeps its memory: the device's default
    // pool gives its memory back at every synchronisation, and a call then
    // paid for a new mapping (about 100 us)
    cudaMemPool_t pool;
    POS_TRY(pos::scratch_pool(&pool));
    void *scratch = nullptr;
    POS_CUDA(cudaMallocFromPoolAsync(&scratch, (size_t)parts * 16, pool, s));
    int32_t *pt = static_cast<int32_t *>(scratch);
    long long *pi = reinterpret_cast<long long *>(static_cast<char *>(scratch) + parts * 8);
    const pos_status st = pos::launch_argmin(d_makespan, d_feasible, n, pt, pi, d_out, s);
    const cudaError_t e2 = cudaFreeAsync(scratch, s);
    if (st != POS_OK) return st;
    if (e2 != cudaSuccess) return pos::cuda_fail(e2, "argmin free");
    return POS_OK;
}

}  // extern "C"
