// host_sched.h -- host-side scheduling rules of the library, plain C++ (no
// CUDA), so that they are also compiled and checked on a host without a GPU
// (tests/host_sched_harness.cpp):
//   - which batches of a one-warp length conv_circular runs with one thread
//     block per pair (k_conv_small) instead of one warp per pair;
//   - how conv_circular_host cuts a batch into the chunks of its copy /
//     convolve / copy-back pipeline;
//   - the scratch of a batch plan's split classes.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

namespace ntt {

// Largest batch of length 2^L (L <= rw, the one-warp lengths) that runs one
// block per pair; 0 for longer lengths.  The one-warp kernels win once the
// batch fills the GPU: measured on GB300, the crossover lies near 16 KB of
// input per SM (2^10, 32-bit words: 608 pairs; 64-bit words at 2^9: between
// 608 and 1216), and beyond 32 pairs per SM the block-per-pair kernel's idle
// threads at the shortest lengths cost more.
inline long long small_batch_max(int L, int rw, int word_bytes, int nsm)
{
    if (L > rw || L < 0 || word_bytes <= 0 || nsm <= 0) return 0;
    const long long by_bytes = (long long)nsm * 16384 / ((1LL << L) * word_bytes);
    return std::max<long long>(1, std::min<long long>(by_bytes, (long long)nsm * 32));
}

// Pairs per chunk of the host-buffer pipeline: about 48 MB of input (f and
// g) for whole-sequence lengths, 32 MB on the split path, at least one pair,
// at most the batch.
inline size_t host_chunk_pairs(size_t seq_bytes, bool split, size_t batch)
{
    const size_t bytes = split ? (size_t)32 << 20 : (size_t)48 << 20;
    return std::min(std::max<size_t>(1, bytes / (2 * seq_bytes)), std::max<size_t>(1, batch));
}

// Chunk sizes (pairs) covering `pairs`: full chunks, then 1/2, 1/4 and 1/8
// of one at the end when `shrink_tail` and the batch holds at least four
// full chunks of at least 8 pairs, so that the convolution and outbound copy
// still to run after the last inbound copy are short.
inline std::vector<size_t> host_chunk_sizes(size_t pairs, size_t chunk, bool shrink_tail)
{
    std::vector<size_t> sizes;
    if (chunk == 0) return sizes;
    const size_t tail = (shrink_tail && chunk >= 8 && pairs >= 4 * chunk) ? chunk / 2 + chunk / 4 + chunk / 8 : 0;
    for (size_t body = pairs - tail; body > 0;) {
        const size_t c = std::min(chunk, body);
        sizes.push_back(c);
        body -= c;
    }
    if (tail) sizes.insert(sizes.end(), {chunk / 2, chunk / 4, chunk / 8});
    return sizes;
}

// Scratch of a batch plan's split classes: one piece per stream, used by its
// classes in turn, for every pair of a class in one wave up to SCRATCH_MAX
// (fewer, fuller launches: measured on GB300, 143 x 2^19 in waves of 64 pairs
// 721 us, in one 679 us), and for the plan's own wave at least.
constexpr size_t SCRATCH_MAX = (size_t)1 << 30;

struct ScratchClass {
    int stream = 0;
    size_t per_pair = 0;        // bytes per pair of a wave
    size_t count = 0;           // pairs of the class
    uint32_t least = 0;         // the plan's own wave
    uint32_t wave = 0;          // result: pairs per wave
};

// Takes every stream's piece from alloc(bytes) (null when there is no room).
// When one fails, all that were taken go back and every stream gets by with
// the plans' own waves; false, with nothing taken, when those do not fit either.
template <class Alloc, class Free>
bool take_scratch(std::vector<ScratchClass> &classes, std::vector<void *> &pieces, Alloc alloc, Free release)
{
    for (size_t limit : {SCRATCH_MAX, (size_t)0}) {
        bool ok = true;
        for (size_t k = 0; k < pieces.size() && ok; ++k) {
            size_t bytes = 0;
            for (ScratchClass &c : classes) {
                if (c.stream != (int)k) continue;
                c.wave = (uint32_t)std::min(std::max<size_t>(c.least, limit / c.per_pair), c.count);
                bytes = std::max(bytes, c.wave * c.per_pair);
            }
            if (bytes) ok = (pieces[k] = alloc(bytes)) != nullptr;
        }
        if (ok) return true;
        for (void *&p : pieces) {
            if (p) release(p);
            p = nullptr;
        }
    }
    return false;
}

}  // namespace ntt
