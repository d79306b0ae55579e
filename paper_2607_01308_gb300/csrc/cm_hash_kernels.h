// Internal interface between the host core (cm_host.cpp) and the content-address
// kernels (blake2s_tree.cu). Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "cm.h"

namespace cm {

// ---------------------------------------------------------------- content address
// BLAKE2s tree mode (RFC 7693 compression; tree parameters of the BLAKE2 paper):
// 1024-byte leaves, fanout 16, 16-byte node digests.
constexpr int kDigestBytes = 16;
constexpr int kLeafBytes = 1024;
constexpr int kFanout = 16;

// Chaining value a node starts from: IV xor the 32-byte parameter block with the
// node offset and node depth fields zero. Kernels xor in offset and depth.
struct TreeParams {
    uint32_t h_base[8];
};

struct LeafLaunch {
    const uint8_t *k;              // fragment K, device
    const uint8_t *v;              // fragment V, device
    uint64_t plane_bytes;          // bytes of one layer of K (= of V): H*T*d*2
    uint64_t stream_bytes;         // 2 * L * plane_bytes
    uint64_t num_leaves;           // ceil(stream_bytes / 1024)
    uint64_t norm_begin;           // stream offset of K[l*]; its length is plane_bytes
    uint32_t row_bytes;            // d*2; a power of two in [32, 1024]
    uint32_t seq_len;              // T
    uint32_t heads;                // H
    uint32_t num_arrivals;         // arrival counters of the tree levels >= 2
    uint32_t *arrivals;            // zeroed by the leaf launch
    unsigned long long *norm_key;  // Q[T] out: every entry is written, once
    uint8_t *digests;              // num_leaves * 16 bytes out
    TreeParams tree;
};

// Level 0 of up to kMaxLeafGroup fragments in one launch: one thread per leaf, the
// leaf blocks of fragment i being [block_begin[i], block_begin[i + 1]) (set by the
// caller); then one block per fragment that zeroes its arrival counters.
constexpr int kMaxLeafGroup = 32;
constexpr int kLeafBlockThreads = 128;   // threads (= leaves) per block of the leaf launch
// Threads of a norm block that share one token's heads (the block's other tokens side by side).
__host__ __device__ constexpr uint32_t norm_lanes(uint32_t heads) { return heads < 32u ? (heads ? heads : 1u) : 32u; }
struct LeafGroup {
    uint32_t count;
    uint32_t pad_;
    uint64_t block_begin[kMaxLeafGroup + 1];
    uint64_t norm_block_begin[kMaxLeafGroup + 1];
    LeafLaunch frag[kMaxLeafGroup];
};
// with_norms: the group's norm keys too, in a launch of their own beside the leaves. Otherwise
// they are launched elsewhere (launch_norm_keys).
cudaError_t launch_leaf_hash_group(const LeafGroup &g, bool with_norms, int num_sms, cudaStream_t stream);
// The routing-layer norm keys of the group, norm_lanes(H) threads to a token, by at most
// max_blocks blocks. They read only K[l*], 1/(2L) of the bytes. (Norm block i of fragment f is
// norm_block_begin[f] + i, set by the launcher.)
cudaError_t launch_norm_keys(const LeafGroup &g, uint64_t max_blocks, cudaStream_t stream);
// Leaf-hash blocks that fit on one SM at once (the least of leaf_hash_kernel's instances; the
// four-lane kernel has at most two an SM), or 0 on error.
int leaf_hash_blocks_per_sm();

constexpr int kMaxGroup = 32;

// Every tree level above the leaves, for up to kMaxGroup fragments. Four lanes hash a level-s
// node, a block the nodes of one parent and then the parent; then, level by level, the warp that
// completes a parent's last child (a per-node arrival counter, zeroed by the leaf launch)
// hashes that parent, up to the root. No thread ever waits for another block's. With fewer
// than kSplitLevel1Nodes level-1 nodes in all, one launch with s = 1. With more, a first
// launch hashes level 1 with a lane to a node, which takes the fewest instructions, and a
// second runs the scheme above with s = 2: one ingest with 26k level-1 nodes 298 us in one
// launch, 290 in two, with 13k 175 and 175.
constexpr int kMaxLevels = 12;
struct TreeTopFragment {
    uint8_t *level[kMaxLevels];       // digests of level k; level[levels - 1] is the root
    uint64_t size[kMaxLevels];        // nodes of level k
    uint32_t *arrivals[kMaxLevels];   // per node of level k >= 2: children finished so far (0 before)
    uint32_t levels;                  // >= 2
    TreeParams tree;
};
struct TreeTop {
    uint32_t count;
    // prefix sums of the nodes of the level that a launch starts from (set by launch_tree_top)
    uint64_t node_begin[kMaxGroup + 1];
    TreeTopFragment frag[kMaxGroup];
};
constexpr uint64_t kSplitLevel1Nodes = 16384;
cudaError_t launch_tree_top(const TreeTop &t, cudaStream_t stream);
int tree_top_kernels(const TreeTop &t);   // kernels launch_tree_top launches for t

// *flag |= 1 if the `bytes` bytes at a and b differ (16-byte aligned, bytes % 16 == 0).
cudaError_t launch_compare(const void *a, const void *b, uint64_t bytes, unsigned int *flag,
                           cudaStream_t stream);

// Bounds-checked builds: reads and zeroes the content-address kernels' violation count on
// the current device (0 in other builds).
cudaError_t take_hash_bounds_violations(unsigned int *out);

// Host-core helpers used by the allocation-free entry point in blake2s_tree.cu.
TreeParams make_tree_params(int32_t L, int32_t H, int32_t d, int32_t T);
cm_status check_fragment(const cm_fragment *f);
cm_status report_error(cm_status st, const char *msg);

}  // namespace cm
