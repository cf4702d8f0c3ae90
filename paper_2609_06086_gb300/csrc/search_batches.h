// How a search splits the memory-feasible slices of one micro-batch count
// into batches (host only, no CUDA).
#pragma once
#include <algorithm>
#include <cstddef>
#include <vector>

namespace pos {

// A prefix names its slice by its slot in the batch, 16 bits of which the
// largest value marks a hole.
constexpr size_t kMaxBatchSlices = 65535;

// Sizes of the batches of n slices, in processing order (most promising
// slices first).
// Eq. 2 alone: eight batches, best first, so that the incumbent improves
// between them.  With the completion bounds (prune mode 2) the warm-up already
// holds each slice's argmin completion and every launch costs more than a
// little extra pruning saves: a first batch of the 1/16 of the slices with the
// smallest root bounds (most likely to hold the optimum), then the rest in one
// batch.  No batch exceeds the slots.
inline std::vector<size_t> batch_sizes(size_t n, int prune) {
    const size_t bsz = prune == 2 ? std::min<size_t>(kMaxBatchSlices, n)
                                  : std::min<size_t>(kMaxBatchSlices,
                                                     std::max<size_t>(32, (n + 7) / 8));
    const size_t first = prune == 2 ? std::min(bsz, (n + 15) / 16) : bsz;
    std::vector<size_t> out;
    for (size_t b0 = 0; b0 < n; b0 += out.back())
        out.push_back(std::min(b0 == 0 ? first : bsz, n - b0));
    return out;
}

}  // namespace pos
