// Which full comparisons share a launch group (the re-delivery fast path's host side; no CUDA
// call). Not part of the public ABI.
#pragma once

#include <cstring>
#include <functional>

#include "cm.h"
#include "cm_dedup_kernels.h"

namespace cm {

// A delivery that may equal a fragment of its shape, the base.
struct Comparison {
    cm_fragment base, member;
};

inline uint64_t fragment_vecs(const cm_fragment &f) {   // 16-byte vectors of its K (= of its V)
    return (uint64_t)f.num_layers * (uint64_t)f.num_kv_heads * (uint64_t)f.seq_len * (uint64_t)f.head_dim / 8;
}

// A fragment is its buffers and its shape: a part of a fragment (its first layers, or with one
// layer and head its first tokens) starts at the same addresses and is another fragment.
inline int compare_fragments(const cm_fragment &a, const cm_fragment &b) {
    if (a.k != b.k) return std::less<const void *>()(a.k, b.k) ? -1 : 1;
    if (a.v != b.v) return std::less<const void *>()(a.v, b.v) ? -1 : 1;
    if (a.num_layers != b.num_layers) return a.num_layers < b.num_layers ? -1 : 1;
    if (a.num_kv_heads != b.num_kv_heads) return a.num_kv_heads < b.num_kv_heads ? -1 : 1;
    if (a.seq_len != b.seq_len) return a.seq_len < b.seq_len ? -1 : 1;
    if (a.head_dim != b.head_dim) return a.head_dim < b.head_dim ? -1 : 1;
    return 0;
}

// Fills the launch of n comparisons (n <= kMaxComparePairs): member m is comparison m's. A
// comparison joins the group before it, unless that is full, if they have one base, or (a chain)
// if it is with that group's last member. False if a member is not of its base's size.
inline bool group_comparisons(const Comparison *c, size_t n, CompareFull &out) {
    std::memset(&out, 0, sizeof out);
    if (n > (size_t)kMaxComparePairs) return false;
    for (size_t m = 0; m < n; ++m) {
        const cm_fragment &b = c[m].base, &f = c[m].member;
        const uint64_t vecs = fragment_vecs(b);
        if (fragment_vecs(f) != vecs) return false;
        out.member[m] = {{static_cast<const uint4 *>(f.k), static_cast<const uint4 *>(f.v)}, vecs};
        CompareGroup *g = out.groups != 0 ? &out.group[out.groups - 1] : nullptr;
        if (g != nullptr && g->end - g->begin == kMaxCompareGroup) g = nullptr;
        const bool one = g != nullptr && g->end - g->begin == 1;   // not yet a chain or not
        if (g != nullptr && (one || g->chain != 0) && compare_fragments(c[m - 1].member, b) == 0) {
            g->chain = 1;
        } else if (g == nullptr || g->chain != 0 || compare_fragments(c[m - 1].base, b) != 0) {
            g = &out.group[out.groups];
            *g = {{static_cast<const uint4 *>(b.k), static_cast<const uint4 *>(b.v)}, vecs, (uint32_t)m, 0, 0, 0};
            out.chunk_begin[out.groups + 1] =
                out.chunk_begin[out.groups] + 2 * ((vecs + kCompareChunkVecs - 1) / kCompareChunkVecs);
            ++out.groups;
        }
        g->end = (uint32_t)m + 1;
    }
    return true;
}

}  // namespace cm
