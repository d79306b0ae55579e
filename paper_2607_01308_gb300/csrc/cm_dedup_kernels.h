// Internal interface between the host core (cm_host.cpp) and the byte-comparison
// kernels of the optional re-delivery fast path (dedup.cu). Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace cm {

constexpr int kMaxComparePairs = 128;         // pairs (members) per launch
constexpr uint64_t kCompareChunkVecs = 2048;   // 16-byte vectors of each array per chunk

// Two fragments of one shape, told apart by their K arrays' first 4 KiB: `vecs` 16-byte
// vectors long. All pointers below are 16-byte aligned.
struct ComparePair {
    const uint4 *a_k, *b_k;
    uint64_t vecs;
};
struct ComparePrefix {
    uint32_t count;                               // pairs, <= kMaxComparePairs
    uint32_t pad_;
    ComparePair pair[kMaxComparePairs];
    uint32_t *differ;                             // one word per pair; may be mapped host memory
};

// Deliveries (members) that may equal one candidate (the group's base). K and V arrays are
// `vecs` 16-byte vectors long, a member's as long as its base's.
struct CompareMember {
    const uint4 *k, *v;
    uint64_t vecs;
};
struct CompareGroup {
    const uint4 *k, *v;                           // the base
    uint64_t vecs;
    uint32_t begin, end;                          // its members
};
struct CompareFull {
    uint32_t groups;                              // <= members <= kMaxComparePairs
    uint32_t pad_;
    // prefix sums of the groups' chunk counts: 2 ceil(vecs / kCompareChunkVecs) per group
    uint64_t chunk_begin[kMaxComparePairs + 1];
    CompareGroup group[kMaxComparePairs];
    CompareMember member[kMaxComparePairs];
    uint32_t *differ;                             // device, one word per member, zeroed before
};

// differ[p] = 1 if the first 4 KiB of pair p's K arrays differ, else 0 (one block per pair).
cudaError_t launch_compare_prefix(const ComparePrefix &c, cudaStream_t stream);

// differ[m] |= 1 if member m's K or V array differs from its group's base anywhere (a
// persistent grid of blocks_per_sm blocks per SM over all chunks of all groups; a member
// already found to differ is skipped).
cudaError_t launch_compare_full(const CompareFull &c, int num_sms, int blocks_per_sm, cudaStream_t stream);

// Bounds-checked builds: reads and zeroes these kernels' violation count on the current device
// (0 in other builds).
cudaError_t take_dedup_bounds_violations(unsigned int *out);

}  // namespace cm
