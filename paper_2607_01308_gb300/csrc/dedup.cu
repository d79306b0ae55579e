// Byte comparison of delivered fragments against candidates of the same shape, for
// the optional re-delivery fast path of Ingest (Algorithm 2): a byte-identical
// re-delivery has the same content address by definition (Section 4.3: the address
// is a function of the bytes, shapes and dtype), so once its bytes are shown equal to
// a fragment whose address is known or being computed, it need not be hashed. The
// comparison reads both fragments once at HBM speed; the hash is bound by the
// integer ALU. Pairs that differ are usually told apart by their first 4 KiB.
#include "cm_bounds.h"
#include "cm_dedup_kernels.h"

namespace cm {
namespace {

constexpr int kThreads = 256;
constexpr uint64_t kPrefixVecs = 256;                   // 4 KiB
constexpr uint64_t kChunkVecs = kCompareChunkVecs;      // 32 KiB of each array per chunk
constexpr int kStepVecs = 4;                            // vectors per thread at a time
static_assert(kChunkVecs % ((uint64_t)kThreads * kStepVecs) == 0, "a chunk is a number of whole steps");
static_assert(sizeof(CompareFull) <= 32764, "comparison parameters exceed the kernel parameter limit");

__device__ __forceinline__ uint32_t diff4(const uint4 &x, const uint4 &y) {
    return (x.x ^ y.x) | (x.y ^ y.y) | (x.z ^ y.z) | (x.w ^ y.w);
}

// Vector i of an array of n.
__device__ __forceinline__ uint4 load_vec(const uint4 *p, uint64_t i, [[maybe_unused]] uint64_t n) {
    return CM_IN_BOUNDS(p + i, 16, p, n * 16) ? __ldcs(p + i) : make_uint4(0, 0, 0, 0);
}

// One block per pair: the first 4 KiB of K.
__global__ void __launch_bounds__(kThreads) prefix_kernel(const __grid_constant__ ComparePrefix c) {
    const ComparePair &p = c.pair[blockIdx.x];
    const uint64_t n = p.vecs < kPrefixVecs ? p.vecs : kPrefixVecs;
    uint32_t d = 0;
    for (uint64_t i = threadIdx.x; i < n; i += kThreads) d |= diff4(load_vec(p.a_k, i, p.vecs), load_vec(p.b_k, i, p.vecs));
    const int any = __syncthreads_or(d != 0);
    if (threadIdx.x == 0) c.differ[blockIdx.x] = any ? 1u : 0u;
}

// Persistent grid over the chunks of all groups (K then V of each): a warp loads its part of
// the base's chunk and compares every member's with it, so the base is read once for all its
// members (bound by HBM: (members + 1) reads of a fragment instead of 2 per member). Members
// that another warp has found to differ are skipped.
__global__ void __launch_bounds__(kThreads) full_kernel(const __grid_constant__ CompareFull c) {
    const uint64_t total = c.chunk_begin[c.groups];
    uint32_t gi = 0;
    for (uint64_t x = blockIdx.x; x < total; x += gridDim.x) {
        while (x >= c.chunk_begin[gi + 1]) ++gi;
        const CompareGroup &g = c.group[gi];
        // chunk index within the group: the K chunks, then the V chunks
        const uint64_t per_array = (g.vecs + kChunkVecs - 1) / kChunkVecs;
        const uint64_t local = x - c.chunk_begin[gi];
        const bool is_v = local >= per_array;
        const uint64_t begin = (is_v ? local - per_array : local) * kChunkVecs;
        const uint64_t end = begin + kChunkVecs < g.vecs ? begin + kChunkVecs : g.vecs;
        const uint4 *base = is_v ? g.v : g.k;
#pragma unroll 1
        for (uint64_t i = begin + threadIdx.x; i < end; i += (uint64_t)kThreads * kStepVecs) {
            uint4 b[kStepVecs];
#pragma unroll
            for (int u = 0; u < kStepVecs; ++u)
                b[u] = i + (uint64_t)u * kThreads < end ? load_vec(base, i + (uint64_t)u * kThreads, g.vecs)
                                                        : make_uint4(0, 0, 0, 0);
            for (uint32_t m = g.begin; m < g.end; ++m) {
                if (__ldcg(c.differ + m) != 0) continue;
                const uint4 *a = is_v ? c.member[m].v : c.member[m].k;
                uint32_t d = 0;
#pragma unroll
                for (int u = 0; u < kStepVecs; ++u)
                    if (i + (uint64_t)u * kThreads < end)
                        d |= diff4(load_vec(a, i + (uint64_t)u * kThreads, c.member[m].vecs), b[u]);
                if (d != 0) atomicOr(c.differ + m, 1u);
            }
        }
    }
}

}  // namespace

CM_DEFINE_BOUNDS_READER(take_dedup_bounds_violations)

cudaError_t launch_compare_prefix(const ComparePrefix &c, cudaStream_t stream) {
    if (c.count == 0) return cudaSuccess;
    prefix_kernel<<<c.count, kThreads, 0, stream>>>(c);
    return cudaGetLastError();
}

cudaError_t launch_compare_full(const CompareFull &c, int num_sms, int blocks_per_sm, cudaStream_t stream) {
    if (c.groups == 0) return cudaSuccess;
    for (uint32_t g = 0; g < c.groups; ++g)   // a member of another size would be read past its end
        for (uint32_t m = c.group[g].begin; m < c.group[g].end; ++m)
            if (c.member[m].vecs != c.group[g].vecs) return cudaErrorInvalidValue;
    const uint64_t total = c.chunk_begin[c.groups];
    const uint64_t most = (uint64_t)num_sms * (uint64_t)blocks_per_sm;
    const uint64_t grid = total < most ? total : most;
    if (grid == 0) return cudaSuccess;
    full_kernel<<<(unsigned)grid, kThreads, 0, stream>>>(c);
    return cudaGetLastError();
}

}  // namespace cm
