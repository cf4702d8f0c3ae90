// The slices of a search: the graph of their stage sequences (host), and the
// set-up kernel that makes the prefix sums and every slice record.
#include <algorithm>
#include <array>
#include <cstring>
#include <unordered_map>
#include <vector>

#include "search_host.h"

namespace pos {

namespace {

// What is left to place, per device type.
using Left = std::array<int32_t, POS_MAX_TYPES>;
struct LeftHash {
    size_t operator()(const Left &v) const {
        uint64_t h = 0x9E3779B97F4A7C15ull;
        for (int32_t x : v) h = (h ^ (uint32_t)x) * 0xBF58476D1CE4E5B9ull;
        return (size_t)(h ^ (h >> 29));
    }
};
struct Choice {
    uint8_t val;  // type or class
    Left left;    // what is left after it
};
constexpr uint32_t kDead = 0xffffffffu;  // no completion
constexpr uint64_t kMaxSequences = 1ull << 22;

// Appends the graph of the sequences of `units` choices from `start` to sp.
// choices(left, out) lists a state's choices in ascending order;
// completes(left, r): can r more stages use up what is left?  Returns the
// number of sequences (0: none, no root is appended), kMaxSequences + 1 when
// there are more than kMaxSequences.  Every state kept lies on a sequence, so
// a level never holds more states than there are sequences.
template <class Choices, class Completes>
uint64_t add_graph(SliceSpace &sp, int units, const Left &start, Choices choices,
                   Completes completes) {
    if (!completes(start, units)) return 0;
    std::vector<std::vector<Left>> level(units + 1);
    struct Edge {
        uint8_t val;
        uint32_t to;  // index within the next level
    };
    std::vector<std::vector<Edge>> edges(units);         // per level, state by state
    std::vector<std::vector<uint32_t>> start_of(units);  // first edge of each state
    level[0].push_back(start);
    std::vector<Choice> ch;
    for (int u = 0; u < units; ++u) {
        std::unordered_map<Left, uint32_t, LeftHash> id;
        for (const Left &st : level[u]) {
            start_of[u].push_back((uint32_t)edges[u].size());
            ch.clear();
            choices(st, ch);
            for (const Choice &c : ch) {
                const auto it = id.find(c.left);
                uint32_t to;
                if (it != id.end()) {
                    to = it->second;
                } else {
                    to = completes(c.left, units - u - 1) ? (uint32_t)level[u + 1].size() : kDead;
                    id.emplace(c.left, to);
                    if (to != kDead) level[u + 1].push_back(c.left);
                }
                if (to != kDead) edges[u].push_back({c.val, to});
            }
        }
        start_of[u].push_back((uint32_t)edges[u].size());
        if (level[u + 1].size() > kMaxSequences) return kMaxSequences + 1;
    }
    // sequences from every state, from the last level back
    std::vector<std::vector<uint64_t>> count(units + 1);
    count[units].assign(level[units].size(), 1);
    for (int u = units - 1; u >= 0; --u) {
        count[u].assign(level[u].size(), 0);
        for (size_t i = 0; i < level[u].size(); ++i)
            for (uint32_t e = start_of[u][i]; e < start_of[u][i + 1]; ++e)
                count[u][i] = std::min(kMaxSequences + 1, count[u][i] + count[u + 1][edges[u][e].to]);
    }
    const uint64_t total = count[0][0];
    if (total > kMaxSequences) return kMaxSequences + 1;
    // states level by level after those there are (sp.first ends with the
    // number of choices)
    std::vector<uint32_t> base(units + 1);
    uint32_t n_states = (uint32_t)sp.first.size() - 1;
    for (int u = 0; u <= units; ++u) {
        base[u] = n_states;
        n_states += (uint32_t)level[u].size();
    }
    sp.root.push_back(base[0]);
    for (int u = 0; u <= units; ++u)
        for (size_t i = 0; i < level[u].size(); ++i) {
            uint64_t before = 0;
            for (uint32_t e = u < units ? start_of[u][i] : 0u;
                 u < units && e < start_of[u][i + 1]; ++e) {
                sp.before.push_back((uint32_t)before);
                sp.next.push_back(base[u + 1] + edges[u][e].to);
                sp.val.push_back(edges[u][e].val);
                before += count[u + 1][edges[u][e].to];
            }
            sp.first.push_back((uint32_t)sp.next.size());
        }
    return total;
}

// POS_PLACE_DEVICES, one D: class k = (t, j) takes tp_list[j] of type t's
// devices in units of D, all of which are to be used.
uint64_t add_device_graph(const pos_problem *p, int units, int D, SliceSpace &sp) {
    const int T = p->tables.n_types, n_tp = p->tables.n_tp;
    Left start{};
    int vmax = 0;
    for (int t = 0; t < T; ++t) {
        if (p->type_counts[t] % D != 0) return 0;  // no stage split uses them up
        start[t] = p->type_counts[t] / D;
        vmax = std::max(vmax, (int)start[t]);
    }
    // reach[v], bit n: v is a sum of exactly n TP degrees (n <= units)
    std::vector<uint32_t> reach((size_t)vmax + 1, 0u);
    reach[0] = 1u;
    for (int v = 1; v <= vmax; ++v)
        for (int j = 0; j < n_tp; ++j) {
            const int d = p->tp_list[j];
            if (d <= v) reach[v] |= (reach[v - d] << 1) & ((2u << units) - 1u);
        }
    auto completes = [&](const Left &left, int r) {
        uint32_t mask = 1u;  // bit n: n stages used by the types seen so far
        for (int t = 0; t < T && mask; ++t) {
            uint32_t next = 0, m = reach[left[t]] & ((2u << r) - 1u);
            while (m) {
                next |= mask << __builtin_ctz(m);
                m &= m - 1u;
            }
            mask = next & ((2u << r) - 1u);
        }
        return ((mask >> r) & 1u) != 0u;
    };
    auto choices = [&](const Left &left, std::vector<Choice> &out) {
        for (int t = 0; t < T; ++t)
            for (int j = 0; j < n_tp; ++j) {
                const int d = p->tp_list[j];
                if (d > left[t]) continue;
                Choice c{(uint8_t)(t * n_tp + j), left};
                c.left[t] -= d;
                out.push_back(c);
            }
    };
    return add_graph(sp, units, start, choices, completes);
}

}  // namespace

pos_status build_slice_space(const pos_problem *p, int units, SliceSpace &sp) {
    const int T = p->tables.n_types, n_tp = p->tables.n_tp;
    sp = SliceSpace();
    sp.units = units;
    sp.per_stage = p->placement == POS_PLACE_DEVICES;
    sp.n_grp = sp.per_stage ? p->n_D : n_tp;
    sp.first.push_back(0);
    sp.grp_off.assign(sp.n_grp + 1, 0);
    if (sp.per_stage) {
        for (int g = 0; g < sp.n_grp; ++g) {
            const size_t roots = sp.root.size();
            const uint64_t n = add_device_graph(p, units, p->D_list[g], sp);
            sp.grp_off[g + 1] = sp.grp_off[g] + n;
            if (sp.grp_off[g + 1] > kMaxSequences)
                return fail(POS_EINVAL, "more than 2^22 class sequences");
            if (sp.root.size() == roots) sp.root.push_back(0);  // an empty group
            sp.D.push_back(p->D_list[g]);
        }
    } else {
        const bool exact = p->placement == POS_PLACE_EXACT;
        Left start{};
        int sum = 0;
        for (int t = 0; t < T && exact; ++t) {
            start[t] = p->type_counts[t];
            sum += start[t];
        }
        if (exact && sum != units) return fail(POS_EINVAL, "type_counts must sum to S");
        const uint64_t n = add_graph(
            sp, units, start,
            [&](const Left &left, std::vector<Choice> &out) {
                for (int t = 0; t < T; ++t) {
                    if (exact && left[t] == 0) continue;
                    Choice c{(uint8_t)t, left};
                    if (exact) --c.left[t];
                    out.push_back(c);
                }
            },
            [](const Left &, int) { return true; });
        if (n > kMaxSequences) return fail(POS_EINVAL, "too many placements");
        for (int g = 0; g < n_tp; ++g) {
            if (g > 0) sp.root.push_back(sp.root[0]);
            sp.grp_off[g + 1] = sp.grp_off[g] + n;
            sp.D.push_back(p->dp_list[g]);
        }
    }
    sp.per_m = sp.grp_off[sp.n_grp];
    if ((uint64_t)p->n_M * sp.per_m > kMaxSequences)
        return fail(POS_EINVAL, "more than 2^22 slices");
    return POS_OK;
}

void plan_slice_fields(const pos_problem *p, const SliceSpace &sp, uint64_t ord, pos_plan *out) {
    int mi = 0, g = 0;
    uint64_t pr = 0;
    sp.decode(ord, &mi, &g, &pr);
    const int n_tp = p->tables.n_tp;
    out->m_idx = mi;
    out->M = p->M_list[mi];
    out->D = sp.D[g];
    out->place_rank = pr;
    out->tp_idx = sp.per_stage ? -1 : g;
    out->tp = sp.per_stage ? -1 : p->tp_list[g];
    out->d_idx = sp.per_stage ? g : -1;
    int cls[POS_MAX_STAGES];
    sp.classes(g, pr, n_tp, cls);
    for (int x = 0; x < POS_MAX_STAGES; ++x) {
        const int k = x < sp.units ? cls[x] : -1;
        out->type[x] = k < 0 ? -1 : k / n_tp;
        out->tp_stage[x] = k < 0 ? -1 : k % n_tp;
    }
}

void pack_setup(const pos_problem *p, const SliceSpace &sp, const std::vector<int32_t> &mis,
                uint64_t Q, const std::vector<unsigned char> &blob, SetupPack &out) {
    out.bytes = blob;
    auto put = [&](const void *src, size_t bytes) {
        const size_t at = (out.bytes.size() + 15) & ~(size_t)15;
        out.bytes.resize(at + bytes);
        if (bytes) std::memcpy(out.bytes.data() + at, src, bytes);
        return at;
    };
    out.n_slices = (uint32_t)(mis.size() * sp.per_m);
    out.off_first = put(sp.first.data(), 4 * sp.first.size());
    out.off_before = put(sp.before.data(), 4 * sp.before.size());
    out.off_next = put(sp.next.data(), 4 * sp.next.size());
    out.off_val = put(sp.val.data(), sp.val.size());
    out.off_root = put(sp.root.data(), 4 * sp.root.size());
    std::vector<uint32_t> grp(sp.grp_off.begin(), sp.grp_off.end());
    out.off_grp = put(grp.data(), 4 * grp.size());
    std::vector<uint64_t> scale;
    std::vector<int32_t> M;
    std::vector<uint64_t> counts(mis.size(), sp.per_m);
    for (int32_t mi : mis) {
        M.push_back(p->M_list[mi]);
        for (int g = 0; g < sp.n_grp; ++g)
            scale.push_back(Q / ((uint64_t)sp.D[g] * p->M_list[mi]));
    }
    out.off_scale = put(scale.data(), 8 * scale.size());
    out.off_mi = put(mis.data(), 4 * mis.size());
    out.off_M = put(M.data(), 4 * M.size());
    out.off_counts = put(counts.data(), 8 * counts.size());
}

struct SetupParams {
    unsigned char *pack;  // tables, graph
    BlobLayout ly;
    const uint32_t *first, *before, *next, *root, *grp;
    const uint8_t *val;
    const uint64_t *scale;
    const int32_t *mi, *M;
    int n_grp, units, n_tp, per_stage;
    uint32_t per_m, n_slices;
    SliceRec *slices;
    unsigned long long *best, *ctr;
    Key128 *inc;
};

// Blocks 0 .. 5K-1: a prefix-sum row each; the others: a thread per slice,
// which walks the graph with its rank (a few dependent loads per stage, all
// in L1 after the first warps).  Listing 168,000 class sequences and their
// records on the host, and uploading them, took 10 ms of a 12 ms search; the
// kernel takes 13 us (4 us for 48 slices, bound by its launch and the tables'
// prefix sums).
__global__ void __launch_bounds__(kPrefixThreads) setup_kernel(SetupParams p) {
    const int rows = 5 * p.ly.K;
    if ((int)blockIdx.x < rows) {
        prefix_row(p.pack, p.ly, blockIdx.x);
        return;
    }
    const uint32_t i = (blockIdx.x - rows) * kPrefixThreads + threadIdx.x;
    if (i < kCounters) p.ctr[i] = 0;
    if (i == 0) p.inc->idx = p.inc->obj = ~0ull;
    if (i >= p.n_slices) return;
    const uint32_t v = i / p.per_m, r = i - v * p.per_m;
    int g = 0;
    while (g + 1 < p.n_grp && __ldg(p.grp + g + 1) <= r) ++g;
    uint32_t rank = r - __ldg(p.grp + g), st = __ldg(p.root + g);
    uint32_t cw[4] = {0u, 0u, 0u, 0u};
    for (int u = 0; u < p.units; ++u) {
        uint32_t q = __ldg(p.first + st);
        const uint32_t e = __ldg(p.first + st + 1);
        uint32_t bq = 0;
        while (q + 1 < e) {
            const uint32_t b = __ldg(p.before + q + 1);
            if (b > rank) break;
            bq = b;
            ++q;
        }
        rank -= bq;
        const uint32_t k = p.per_stage ? __ldg(p.val + q) : __ldg(p.val + q) * p.n_tp + g;
#pragma unroll
        for (int w = 0; w < 4; ++w) cw[w] |= (u >> 2) == w ? k << (8 * (u & 3)) : 0u;
        st = __ldg(p.next + q);
    }
    SliceRec rec;
    rec.ordinal = (uint64_t)__ldg(p.mi + v) * p.per_m + r;
    rec.scale = __ldg(p.scale + v * p.n_grp + g);
    rec.M = __ldg(p.M + v);
    rec.gid = i;
    rec.vslot = i;  // bound-table row when every slice has one
    rec.pad = 0;
    uint4 *out = reinterpret_cast<uint4 *>(p.slices + i);
    out[0] = make_uint4((uint32_t)rec.ordinal, (uint32_t)(rec.ordinal >> 32), (uint32_t)rec.scale,
                        (uint32_t)(rec.scale >> 32));
    out[1] = make_uint4(cw[0], cw[1], cw[2], cw[3]);
    out[2] = make_uint4((uint32_t)rec.M, rec.gid, rec.vslot, rec.pad);
    if (p.best) p.best[i] = ~0ull;
}

pos_status launch_setup(const SetupPack &pk, const SliceSpace &sp, int n_tp, const BlobLayout &ly,
                        void *d_pack, SliceRec *slices, unsigned long long *best, Key128 *inc,
                        unsigned long long *ctr, cudaStream_t stream) {
    unsigned char *d = static_cast<unsigned char *>(d_pack);
    SetupParams p;
    p.pack = d;
    p.ly = ly;
    p.first = reinterpret_cast<const uint32_t *>(d + pk.off_first);
    p.before = reinterpret_cast<const uint32_t *>(d + pk.off_before);
    p.next = reinterpret_cast<const uint32_t *>(d + pk.off_next);
    p.val = d + pk.off_val;
    p.root = reinterpret_cast<const uint32_t *>(d + pk.off_root);
    p.grp = reinterpret_cast<const uint32_t *>(d + pk.off_grp);
    p.scale = reinterpret_cast<const uint64_t *>(d + pk.off_scale);
    p.mi = reinterpret_cast<const int32_t *>(d + pk.off_mi);
    p.M = reinterpret_cast<const int32_t *>(d + pk.off_M);
    p.n_grp = sp.n_grp;
    p.units = sp.units;
    p.n_tp = n_tp;
    p.per_stage = sp.per_stage ? 1 : 0;
    p.per_m = (uint32_t)std::max<uint64_t>(1, sp.per_m);
    p.n_slices = pk.n_slices;
    p.slices = slices;
    p.best = best;
    p.ctr = ctr;
    p.inc = inc;
    const uint32_t n = std::max<uint32_t>(pk.n_slices, kCounters);
    setup_kernel<<<5 * ly.K + (n + kPrefixThreads - 1) / kPrefixThreads, kPrefixThreads, 0,
                   stream>>>(p);
    POS_CUDA(cudaGetLastError());
    return POS_OK;
}

}  // namespace pos
