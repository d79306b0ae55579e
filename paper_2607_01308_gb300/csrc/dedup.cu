// Byte comparison of delivered fragments against candidates of the same shape, for
// the optional re-delivery fast path of Ingest (Algorithm 2): a byte-identical
// re-delivery has the same content address by definition (Section 4.3: the address
// is a function of the bytes, shapes and dtype), so once its bytes are shown equal to
// a fragment whose address is known or being computed, it need not be hashed. The
// comparison reads both fragments once at HBM speed; the hash is bound by the
// integer ALU. Pairs that differ are usually told apart by a first look at 8 KiB of them.
#include "cm_bounds.h"
#include "cm_dedup_kernels.h"

namespace cm {
namespace {

constexpr int kThreads = 256;
constexpr uint32_t kPieces = 16, kPieceVecs = 16;       // of the first look: 256 bytes each
static_assert(kPieces * kPieceVecs == (uint32_t)kThreads, "a thread compares one vector of a piece");
constexpr uint64_t kChunkVecs = kCompareChunkVecs;      // 32 KiB of each array per chunk
constexpr int kStepVecs = 4;                            // vectors per thread at a time
constexpr uint64_t kStep = (uint64_t)kThreads * kStepVecs;
static_assert(kChunkVecs % kStep == 0, "a chunk is a number of whole steps");
static_assert(sizeof(CompareFull) <= 32764, "comparison parameters exceed the kernel parameter limit");

__device__ __forceinline__ uint32_t diff4(const uint4 &x, const uint4 &y) {
    return (x.x ^ y.x) | (x.y ^ y.y) | (x.z ^ y.z) | (x.w ^ y.w);
}

// Vector i of an array of n.
__device__ __forceinline__ uint4 load_vec(const uint4 *p, uint64_t i, [[maybe_unused]] uint64_t n) {
    return CM_IN_BOUNDS(p + i, 16, p, n * 16) ? __ldcs(p + i) : make_uint4(0, 0, 0, 0);
}

// One block per pair: a vector of K's first 4 KiB and one of the spread pieces per thread.
__global__ void __launch_bounds__(kThreads) look_kernel(const __grid_constant__ CompareLook c) {
    const ComparePair &p = c.pair[blockIdx.x];
    const uint32_t t = threadIdx.x, piece = t / kPieceVecs;
    const bool in_v = piece >= kPieces / 2;
    const uint64_t room = p.vecs > kPieceVecs ? p.vecs - kPieceVecs : 0;   // the last piece begins here
    const uint64_t i = piece % (kPieces / 2) * room / (kPieces / 2 - 1) + t % kPieceVecs;
    // indices brought into range, so that the four reads are in flight together: 3.1 us for nine
    // pairs, 3.7 with a test before each two
    const uint64_t last = p.vecs - 1, j = t < p.vecs ? t : last, k = i < p.vecs ? i : last;
    const uint4 a0 = load_vec(p.a_k, j, p.vecs), b0 = load_vec(p.b_k, j, p.vecs);
    const uint4 a1 = load_vec(in_v ? p.a_v : p.a_k, k, p.vecs), b1 = load_vec(in_v ? p.b_v : p.b_k, k, p.vecs);
    const int any = __syncthreads_or((diff4(a0, b0) | diff4(a1, b1)) != 0);
    if (t == 0) c.differ[blockIdx.x] = any ? 1u : 0u;
}

// Persistent grid over the chunks of all groups (K then V of each): a warp loads its part of
// the base's chunk and of every member's, so that a fragment is read once for all its copies
// (bound by HBM: (members + 1) reads instead of 2 per member). What other warps have found to
// differ is learnt once per chunk, a lane to a member; such a member is read only where the next
// of its chain is compared with it, and a group whose members all differ is left. Beside the
// hash, which is bound by issue slots, instructions and registers count: six copies alone take
// 152 us at 8 vectors a step, 185 at 4, but a merge of nine deliveries hashed beside it 420 and
// 367; with a test per vector (29 instead of 23 M instructions) 373.
__global__ void __launch_bounds__(kThreads) full_kernel(const __grid_constant__ CompareFull c) {
    const uint64_t total = c.chunk_begin[c.groups];
    const uint32_t lane = threadIdx.x % 32;
    uint32_t gi = 0, closed = 0;   // the group's members known to differ
    for (uint64_t x = blockIdx.x; x < total; x += gridDim.x) {
        for (; x >= c.chunk_begin[gi + 1]; ++gi) closed = 0;
        const CompareGroup &g = c.group[gi];
        const uint32_t members = g.end - g.begin, all = 0xFFFFFFFFu >> (32 - members);
        if (closed == all) {
            // to this block's first chunk past the group: x + k gridDim with
            // k = ceil((end of group - x) / gridDim) >= 1 (the loop adds the last gridDim)
            x += ((c.chunk_begin[gi + 1] - x + gridDim.x - 1) / gridDim.x - 1) * (uint64_t)gridDim.x;
            continue;
        }
        const uint32_t found = lane < members ? __ldcg(c.differ + g.begin + lane) : 0u;   // for the next chunk
        // the members to read, and whether the base
        const uint32_t open = ~closed & all, read = g.chain != 0 ? open | open >> 1 : open;
        const bool read_base = g.chain == 0 || (open & 1u) != 0;
        // chunk index within the group: the K chunks, then the V chunks
        const uint64_t per_array = (g.vecs + kChunkVecs - 1) / kChunkVecs;
        const uint64_t local = x - c.chunk_begin[gi];
        const uint32_t is_v = local >= per_array;
        const uint64_t begin = (is_v ? local - per_array : local) * kChunkVecs;
        const uint64_t end = begin + kChunkVecs < g.vecs ? begin + kChunkVecs : g.vecs;
        const bool whole = g.vecs >= kStep;
#pragma unroll 1
        for (uint64_t at = begin; at < end; at += kStep) {
            // an array's last step begins early enough to be a whole one, so that none but an
            // array shorter than a step needs a test per vector
            const uint64_t i = (whole && at + kStep > g.vecs ? g.vecs - kStep : at) + threadIdx.x;
            auto load = [&](const uint4 *p, uint64_t vecs, uint4 (&r)[kStepVecs]) {
                if (whole) {
#pragma unroll
                    for (int u = 0; u < kStepVecs; ++u) r[u] = load_vec(p, i + (uint64_t)u * kThreads, vecs);
                } else {
#pragma unroll
                    for (int u = 0; u < kStepVecs; ++u)
                        r[u] = i + (uint64_t)u * kThreads < vecs ? load_vec(p, i + (uint64_t)u * kThreads, vecs)
                                                                 : make_uint4(0, 0, 0, 0);
                }
            };
            uint4 b[kStepVecs], a[kStepVecs];
            if (read_base) load(g.kv[is_v], g.vecs, b);
            // member m into `a`, compared with `b`, which may be anything if m is known to differ
            auto member = [&](uint32_t m, const uint4 (&b)[kStepVecs], uint4 (&a)[kStepVecs]) {
                if ((read >> m & 1u) == 0) return;
                const CompareMember &f = c.member[g.begin + m];
                load(f.kv[is_v], f.vecs, a);
                uint32_t d = 0;
#pragma unroll
                for (int u = 0; u < kStepVecs; ++u) d |= diff4(a[u], b[u]);
                if ((open >> m & 1u) != 0 && __any_sync(0xFFFFFFFFu, d != 0) && lane == 0)
                    atomicOr(c.differ + g.begin + m, 1u);
            };
#pragma unroll 1
            for (uint32_t m = 0; m < members; ++m) {
                member(m, b, a);
                if (g.chain != 0 && ++m < members) member(m, a, b);   // in turn: no copies
            }
        }
        closed |= __ballot_sync(0xFFFFFFFFu, found != 0);
    }
}

}  // namespace

CM_DEFINE_BOUNDS_READER(take_dedup_bounds_violations)

cudaError_t launch_compare_look(const CompareLook &c, cudaStream_t stream) {
    if (c.count == 0) return cudaSuccess;
    look_kernel<<<c.count, kThreads, 0, stream>>>(c);
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
