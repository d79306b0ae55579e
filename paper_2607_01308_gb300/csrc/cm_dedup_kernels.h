// Internal interface between the host core (cm_host.cpp) and the byte-comparison
// kernels of the optional re-delivery fast path (dedup.cu). Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace cm {

constexpr int kMaxComparePairs = 128;         // pairs (members) per launch
constexpr uint32_t kMaxCompareGroup = 32;     // members of a group: a lane keeps track of each
constexpr uint64_t kCompareChunkVecs = 2048;   // 16-byte vectors of each array per chunk

// Two fragments of one shape, K and V `vecs` 16-byte vectors long each. All pointers below are
// 16-byte aligned.
struct ComparePair {
    const uint4 *a_k, *a_v, *b_k, *b_v;
    uint64_t vecs;
};
struct CompareLook {
    uint32_t count;                               // pairs, <= kMaxComparePairs
    uint32_t pad_;
    ComparePair pair[kMaxComparePairs];
    uint32_t *differ;                             // one word per pair; may be mapped host memory
};

// Deliveries (members) that are compared in one walk: each with the group's base, or (a chain)
// the first with the base and each other one with the member before it. K and V arrays are
// `vecs` 16-byte vectors long, a member's as long as its base's.
struct CompareMember {
    const uint4 *kv[2];
    uint64_t vecs;
};
struct CompareGroup {
    const uint4 *kv[2];                           // the base
    uint64_t vecs;
    uint32_t begin, end;                          // its members, at most kMaxCompareGroup
    uint32_t chain, pad_;
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

// A first look at every pair: differ[p] = 1 if pair p's K arrays differ in their first 4 KiB, or
// one of 16 pieces of 256 bytes spread over K and V to their ends differs, else 0 (one block per
// pair). The start alone is the same in fragments whose tokens begin alike; their ends are not.
cudaError_t launch_compare_look(const CompareLook &c, cudaStream_t stream);

// differ[m] |= 1 if member m's K or V array differs anywhere from what it is compared with (a
// persistent grid of blocks_per_sm blocks per SM over all chunks of all groups; what is already
// known to differ is no longer read).
cudaError_t launch_compare_full(const CompareFull &c, int num_sms, int blocks_per_sm, cudaStream_t stream);

// Bounds-checked builds: reads and zeroes these kernels' violation count on the current device
// (0 in other builds).
cudaError_t take_dedup_bounds_violations(unsigned int *out);

}  // namespace cm
