// Content address Id(C) (Section 4.3; Algorithm 2, Id) and the routing-layer
// norm key (Eq. rho).
//
// Id is a BLAKE2s tree hash (RFC 7693 compression function; tree parameters of
// the BLAKE2 paper, Section 2.10) of the byte stream K[0] V[0] ... K[L-1] V[L-1]:
// 1024-byte leaves (depth 0), inner nodes over 16 child digests, 16-byte
// digests, shapes and dtype in the salt, seq_len in the personalisation.
//
// Level 0 runs one thread per leaf (four lanes, where there are few): 16 compressions of
// 64-byte blocks, loaded as 128-bit vectors straight from the fragment buffers. A launch beside
// it computes the norm key from K[l*]: a row's squared norm in fp64 in ascending element
// order by one thread, then the quantised norm (round-half-even of 2^20 * sqrt,
// saturated at 2^44 - 1) summed over heads into Q[t] as 64-bit integers: integer
// addition is associative, so Q does not depend on the order of the heads.
#include "cm_bounds.h"
#include "cm_hash_kernels.h"

#include <cstring>

#include <vector>

namespace cm {
namespace {

constexpr uint32_t kIV0 = 0x6A09E667u, kIV1 = 0xBB67AE85u, kIV2 = 0x3C6EF372u, kIV3 = 0xA54FF53Au;
constexpr uint32_t kIV4 = 0x510E527Fu, kIV5 = 0x9B05688Cu, kIV6 = 0x1F83D9ABu, kIV7 = 0x5BE0CD19u;
constexpr unsigned long long kQMax = (1ull << 44) - 1;

__device__ __forceinline__ uint32_t rotr16(uint32_t x) { return __byte_perm(x, 0, 0x1032); }
__device__ __forceinline__ uint32_t rotr8(uint32_t x) { return __byte_perm(x, 0, 0x0321); }
__device__ __forceinline__ uint32_t rotr12(uint32_t x) { return __funnelshift_r(x, x, 12); }
__device__ __forceinline__ uint32_t rotr7(uint32_t x) { return __funnelshift_r(x, x, 7); }

// Where G's operations run. An SM sub-partition issues one warp instruction per cycle; its
// integer ALU pipe and the half of its FMA pipe that multiplies integers each accept one
// every two cycles. G's four xors and four rotations belong to the ALU pipe (16 cycles a
// warp), which bounds the leaf kernel; the additions are moved to the FMA pipe as
// multiply-adds by a 1 the compiler cannot see through (a __constant__ it must load, so it
// cannot fold the product into an add; inline, so that it keeps the shape below).
//
// a + b + x: x is added first. b is the last word that the previous half of G produced, so
// this leaves one addition instead of two on G's chain of dependent operations: one warp
// alone took 0.89 instead of 1.08 us per compression.
//
// The rotation by 16 can move as well: x * 2^16 is its upper half, and a two-way 16-bit dot
// product with (0, 1) adds its lower half: two multiply-type instructions for one byte
// permutation. Moved in three of a round's eight G's it leaves a block 630 ALU, 542 FMA and 1186
// instructions in all (656, 485 and 1155 with none; counted on 604 MB of leaves): ALU 95 %, the
// multiplying half of the FMA pipe 81 % and issue 90 % busy. Moved further (five or all eight)
// the ALU count stays, since the compiler gives other additions back to that pipe, and only the
// instructions grow (1207, 1237): 2.4 GB of leaves and their norm keys 1.317 ms with none, 1.261
// with three, 1.265 with five, 1.262 with eight; beside a render, which takes issue slots too, the
// Qwen3-4B-shaped merge of 4 x 4096 tokens 1.631, 1.598 and (five) 1.633.
__constant__ uint32_t g_one = 1, g_64k = 65536, g_upper_half = 0x0100;
__device__ __forceinline__ uint32_t mad1(uint32_t x, uint32_t y) {
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(g_one), "r"(y));
    return r;
}
__device__ __forceinline__ uint32_t add3(uint32_t a, uint32_t b, uint32_t x) { return mad1(b, mad1(x, a)); }

__device__ __forceinline__ uint32_t rotr16_fma(uint32_t x) {
    uint32_t r;
    asm("dp2a.lo.u32.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(g_upper_half), "r"(x * g_64k));
    return r;
}

// Which G's rotate by 16 on the FMA pipe (bit g: the round's G number g). Which three they are
// makes half a per cent or less.
constexpr uint32_t kFmaMask = 0x94u;
template <int kG>
__device__ __forceinline__ uint32_t rotate16(uint32_t x) {
    return (kFmaMask >> kG) & 1u ? rotr16_fma(x) : rotr16(x);
}

// The G mixing function of RFC 7693, Section 3.1 (rotation distances 16, 12, 8, 7); g is
// G's place in its round.
#define CM_G(g, a, b, c, d, x, y)   \
    a = add3(a, b, (x));            \
    d = rotate16<g>(d ^ a);         \
    c = c + d;                      \
    b = rotr12(b ^ c);              \
    a = add3(a, b, (y));            \
    d = rotr8(d ^ a);               \
    c = c + d;                      \
    b = rotr7(b ^ c);

// One round: four column mixes, then four diagonal mixes, message words taken in
// the order of that round's SIGMA row (RFC 7693, Section 2.7).
#define CM_ROUND(s0, s1, s2, s3, s4, s5, s6, s7, s8, s9, s10, s11, s12, s13, s14, s15) \
    CM_G(0, v0, v4, v8, v12, m[s0], m[s1])                                             \
    CM_G(1, v1, v5, v9, v13, m[s2], m[s3])                                             \
    CM_G(2, v2, v6, v10, v14, m[s4], m[s5])                                            \
    CM_G(3, v3, v7, v11, v15, m[s6], m[s7])                                            \
    CM_G(4, v0, v5, v10, v15, m[s8], m[s9])                                            \
    CM_G(5, v1, v6, v11, v12, m[s10], m[s11])                                          \
    CM_G(6, v2, v7, v8, v13, m[s12], m[s13])                                           \
    CM_G(7, v3, v4, v9, v14, m[s14], m[s15])

// Compression function F (RFC 7693, Section 3.2), 10 rounds. t = bytes hashed
// so far including this block; the last-node flag is applied together with the
// last-block flag, on the node's final compression.
__device__ __forceinline__ void compress(uint32_t h[8], const uint32_t m[16], uint64_t t,
                                         bool last_block, bool last_node) {
    uint32_t v0 = h[0], v1 = h[1], v2 = h[2], v3 = h[3];
    uint32_t v4 = h[4], v5 = h[5], v6 = h[6], v7 = h[7];
    uint32_t v8 = kIV0, v9 = kIV1, v10 = kIV2, v11 = kIV3;
    uint32_t v12 = kIV4 ^ (uint32_t)t, v13 = kIV5 ^ (uint32_t)(t >> 32);
    uint32_t v14 = last_block ? ~kIV6 : kIV6;
    uint32_t v15 = (last_block && last_node) ? ~kIV7 : kIV7;
    CM_ROUND(0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15)
    CM_ROUND(14, 10, 4, 8, 9, 15, 13, 6, 1, 12, 0, 2, 11, 7, 5, 3)
    CM_ROUND(11, 8, 12, 0, 5, 2, 15, 13, 10, 14, 3, 6, 7, 1, 9, 4)
    CM_ROUND(7, 9, 3, 1, 13, 12, 11, 14, 2, 6, 5, 10, 4, 0, 15, 8)
    CM_ROUND(9, 0, 5, 7, 2, 4, 10, 15, 14, 1, 11, 12, 6, 8, 3, 13)
    CM_ROUND(2, 12, 6, 10, 0, 11, 8, 3, 4, 13, 7, 5, 15, 14, 1, 9)
    CM_ROUND(12, 5, 1, 15, 14, 13, 4, 10, 0, 7, 6, 3, 9, 2, 8, 11)
    CM_ROUND(13, 11, 7, 14, 12, 1, 3, 9, 5, 0, 15, 4, 8, 6, 2, 10)
    CM_ROUND(6, 15, 14, 9, 11, 3, 0, 8, 12, 2, 13, 7, 1, 4, 10, 5)
    CM_ROUND(10, 2, 8, 4, 7, 6, 1, 5, 15, 11, 9, 14, 3, 12, 13, 0)
    h[0] ^= v0 ^ v8;
    h[1] ^= v1 ^ v9;
    h[2] ^= v2 ^ v10;
    h[3] ^= v3 ^ v11;
    h[4] ^= v4 ^ v12;
    h[5] ^= v5 ^ v13;
    h[6] ^= v6 ^ v14;
    h[7] ^= v7 ^ v15;
}

#undef CM_ROUND
#undef CM_G

// Chaining value of node (offset, depth): the base words with the 48-bit node
// offset (parameter bytes 8..13) and the node depth (byte 14) xored in.
__device__ __forceinline__ void node_init(uint32_t h[8], const TreeParams &tp, uint64_t offset,
                                          uint32_t depth) {
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = tp.h_base[i];
    h[2] ^= (uint32_t)offset;
    h[3] ^= ((uint32_t)(offset >> 32) & 0xFFFFu) | (depth << 16);
}

__device__ __forceinline__ uint4 load_nc(const uint8_t *p) {
    return __ldg(reinterpret_cast<const uint4 *>(p));
}

__device__ __forceinline__ void store_digest(uint8_t *dst, const uint32_t h[8]) {
    *reinterpret_cast<uint4 *>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
}

// Bounds-checked builds: [p, p + n) lies inside the fragment's K or V array (each
// stream_bytes / 2 long); otherwise a violation is counted.
__device__ __forceinline__ bool in_fragment(const LeafLaunch &a, const uint8_t *p, uint64_t n) {
#ifdef CM_DEBUG_BOUNDS
    const uint64_t half = a.stream_bytes / 2, x = reinterpret_cast<uint64_t>(p);
    const uint64_t k = reinterpret_cast<uint64_t>(a.k), v = reinterpret_cast<uint64_t>(a.v);
    if (n <= half && ((x >= k && x - k <= half - n) || (x >= v && x - v <= half - n))) return true;
    bounds_fail();
    return false;
#else
    (void)a;
    (void)p;
    (void)n;
    return true;
#endif
}

// fl(ss + x^2) for the 8 bf16 of one 16-byte vector, in ascending element order (x^2
// is exact in fp64, so each step is the one rounding of the sum). A normal bf16 (exponent
// field 1..254) is 2^(e-127) (1 + m/128) in magnitude; as an fp64 its exponent field is
// e + 896 and its 7 fraction bits lead the 52-bit fraction, so the high word of |x| is
// ((e << 7 | m) << 13) + (896 << 20) and the low word is 0: integer operations instead of
// a conversion on the FP64 pipe, which is the slow one on this part. A vector holding a
// zero, subnormal, infinity or NaN converts through fp32 instead.
__device__ __forceinline__ double accumulate_squares(uint4 w, double ss) {
    const uint32_t words[4] = {w.x, w.y, w.z, w.w};
    bool normal = true;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t elo = words[i] & 0x7F80u, ehi = words[i] & 0x7F800000u;
        normal = normal && elo != 0u && elo != 0x7F80u && ehi != 0u && ehi != 0x7F800000u;
    }
    if (normal) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double lo = __hiloint2double((int)(((words[i] & 0x7FFFu) << 13) + 0x38000000u), 0);
            const double hi = __hiloint2double((int)(((words[i] >> 3) & 0x0FFFE000u) + 0x38000000u), 0);
            ss = __fma_rn(lo, lo, ss);
            ss = __fma_rn(hi, hi, ss);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double lo = (double)__uint_as_float(words[i] << 16);
            const double hi = (double)__uint_as_float(words[i] & 0xFFFF0000u);
            ss = __fma_rn(lo, lo, ss);
            ss = __fma_rn(hi, hi, ss);
        }
    }
    return ss;
}

// Quantised norm of row r of K[l*] (Eq. rho; the plane is [H][T][d], so r = h*T + t).
__device__ __forceinline__ unsigned long long row_norm(const LeafLaunch &a, uint64_t r) {
    const uint8_t *row = a.k + a.norm_begin / 2 + r * a.row_bytes;   // K[l*] at stream offset 2 l* plane
    const uint32_t nvec = a.row_bytes >> 4;
    double ss = 0.0;
    for (uint32_t v = 0; v < nvec; v += 8) {   // a 128-byte line's loads in flight together
        uint4 w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (v + q < nvec)
                w[q] = CM_IN_BOUNDS(row + 16 * (v + q), 16, a.k + a.norm_begin / 2, a.plane_bytes)
                           ? load_nc(row + 16 * (v + q))
                           : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (v + q < nvec) ss = accumulate_squares(w[q], ss);
    }
    const double scaled = __dsqrt_rn(ss) * 1048576.0;     // exact scaling by 2^20
    return (scaled < (double)kQMax) ? __double2ull_rn(scaled) : kQMax;   // NaN saturates too
}

// Norm keys of the tokens of norm block `block` of one fragment: norm_lanes(H) threads share a
// token's heads, each summing its rows' quantised norms; the integer sums are then added in
// shared memory. Every Q[t] is written once, by a plain store, so Q needs no zeroing and may
// lie in host memory that the device maps.
__device__ __forceinline__ void norm_block(const LeafLaunch &a, uint32_t block) {
    __shared__ unsigned long long part[kLeafBlockThreads];
    const uint32_t lanes = norm_lanes(a.heads), tokens = kLeafBlockThreads / lanes;
    const uint32_t tl = threadIdx.x % tokens, hl = threadIdx.x / tokens;
    const uint64_t t = (uint64_t)block * tokens + tl;
    unsigned long long q = 0;
    if (hl < lanes && t < a.seq_len)
        for (uint32_t h = hl; h < a.heads; h += lanes) q += row_norm(a, (uint64_t)h * a.seq_len + t);
    part[threadIdx.x] = q;
    __syncthreads();
    if (hl == 0 && t < a.seq_len) {
        for (uint32_t k = 1; k < lanes; ++k) q += part[tl + k * tokens];
        if (CM_IN_BOUNDS(a.norm_key + t, 8, a.norm_key, (uint64_t)a.seq_len * 8)) a.norm_key[t] = q;
    }
}

// Cursor over the fragment's byte stream K[0] V[0] K[1] V[1] ...: every segment
// (one layer of K or of V) is plane_bytes long, a multiple of 32, so 32 bytes of the stream
// from a multiple of 32 never straddle two segments.
struct StreamCursor {
    const uint8_t *ptr;
    uint64_t left;       // bytes left in the current segment
    uint32_t layer;
    bool in_v;
};

__device__ __forceinline__ StreamCursor cursor_at(const LeafLaunch &a, uint64_t pos) {
    StreamCursor c;
    const uint64_t two_p = 2 * a.plane_bytes;
    c.layer = (uint32_t)(pos / two_p);
    const uint64_t within = pos - (uint64_t)c.layer * two_p;
    c.in_v = within >= a.plane_bytes;
    const uint64_t seg_off = c.in_v ? within - a.plane_bytes : within;
    c.ptr = (c.in_v ? a.v : a.k) + (uint64_t)c.layer * a.plane_bytes + seg_off;
    c.left = a.plane_bytes - seg_off;
    return c;
}

// The next 32 bytes.
__device__ __forceinline__ const uint8_t *cursor_next(const LeafLaunch &a, StreamCursor &c) {
    if (c.left == 0) {
        if (c.in_v) ++c.layer;
        c.in_v = !c.in_v;
        c.ptr = (c.in_v ? a.v : a.k) + (uint64_t)c.layer * a.plane_bytes;
        c.left = a.plane_bytes;
    }
    const uint8_t *p = c.ptr;
    c.ptr += 32;
    c.left -= 32;
    return p;
}

// Four lanes to a node, for levels with few nodes, where the chain of dependent operations
// bounds a compression: lane q holds column q of the state (words q, q + 4, q + 8, q + 12) and
// does one G of every half round, so the chain is G's twelve operations and not four G's taking
// turns on the half-rate ALU pipe. Between the halves the diagonals are lined up by moving a, c
// and d to the lanes that hold their b: b is the last word that G produces, and the moves of the
// others hide behind it. One warp alone takes 0.61 us per compression this way, 0.89 with a
// lane to a node.
//
// The message words lie in shared memory; g_schedule[q][r] holds, a byte each, the offsets of
// the words that lane q's two G's of round r add (RFC 7693, Section 2.7: column G q, then
// diagonal G q - 1, whose b is in column q).
#define CM_Q4(x0, y0, x1, y1) (4u * (x0) | 4u * (y0) << 8 | 4u * (x1) << 16 | 4u * (y1) << 24)
#define CM_QUAD(s0, s1, s2, s3, s4, s5, s6, s7, s8, s9, s10, s11, s12, s13, s14, s15)          \
    {CM_Q4(s0, s1, s14, s15), CM_Q4(s2, s3, s8, s9), CM_Q4(s4, s5, s10, s11), CM_Q4(s6, s7, s12, s13)}
__constant__ uint32_t g_schedule[10][4] = {
    CM_QUAD(0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15),
    CM_QUAD(14, 10, 4, 8, 9, 15, 13, 6, 1, 12, 0, 2, 11, 7, 5, 3),
    CM_QUAD(11, 8, 12, 0, 5, 2, 15, 13, 10, 14, 3, 6, 7, 1, 9, 4),
    CM_QUAD(7, 9, 3, 1, 13, 12, 11, 14, 2, 6, 5, 10, 4, 0, 15, 8),
    CM_QUAD(9, 0, 5, 7, 2, 4, 10, 15, 14, 1, 11, 12, 6, 8, 3, 13),
    CM_QUAD(2, 12, 6, 10, 0, 11, 8, 3, 4, 13, 7, 5, 15, 14, 1, 9),
    CM_QUAD(12, 5, 1, 15, 14, 13, 4, 10, 0, 7, 6, 3, 9, 2, 8, 11),
    CM_QUAD(13, 11, 7, 14, 12, 1, 3, 9, 5, 0, 15, 4, 8, 6, 2, 10),
    CM_QUAD(6, 15, 14, 9, 11, 3, 0, 8, 12, 2, 13, 7, 1, 4, 10, 5),
    CM_QUAD(10, 2, 8, 4, 7, 6, 1, 5, 15, 11, 9, 14, 3, 12, 13, 0),
};
#undef CM_QUAD
#undef CM_Q4
__constant__ uint32_t g_iv[8] = {kIV0, kIV1, kIV2, kIV3, kIV4, kIV5, kIV6, kIV7};

struct QuadLane {
    uint32_t q, before, after, across;   // lane in its node, and the node's lanes q - 1, q + 1, q + 2
    uint32_t iv_c, iv_d;
    uint32_t schedule[10];
};

__device__ __forceinline__ QuadLane quad_lane(uint32_t lane) {
    QuadLane l;
    l.q = lane & 3u;
    const uint32_t base = lane & 28u;
    l.before = base | ((l.q + 3u) & 3u);
    l.after = base | ((l.q + 1u) & 3u);
    l.across = base | (l.q ^ 2u);
    l.iv_c = g_iv[l.q];
    l.iv_d = g_iv[4u + l.q];
#pragma unroll
    for (int r = 0; r < 10; ++r) l.schedule[r] = g_schedule[r][l.q];
    return l;
}

__device__ __forceinline__ uint32_t move(uint32_t x, uint32_t from) { return __shfl_sync(0xFFFFFFFFu, x, (int)from); }

__device__ __forceinline__ void quad_g(uint32_t &a, uint32_t &b, uint32_t &c, uint32_t &d, uint32_t x, uint32_t y) {
    a = add3(a, b, x);
    d = rotr16(d ^ a);
    c = c + d;
    b = rotr12(b ^ c);
    a = add3(a, b, y);
    d = rotr8(d ^ a);
    c = c + d;
    b = rotr7(b ^ c);
}

// One compression by the four lanes of a node: (h0, h1) are words q and q + 4 of the chaining
// value, the block's words lie at m, t = bytes hashed so far including this block (below 2^32).
// Every lane of the warp calls.
__device__ __forceinline__ void quad_compress(const QuadLane &l, uint32_t &h0, uint32_t &h1, const uint8_t *m,
                                              uint32_t t, bool last_block, bool last_node) {
    uint32_t a = h0, b = h1, c = l.iv_c, d = l.iv_d;
    if (l.q == 0) d ^= t;
    if (l.q == 2 && last_block) d = ~d;
    if (l.q == 3 && last_block && last_node) d = ~d;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t s = l.schedule[r];
        auto word = [&](uint32_t k) {
            return *reinterpret_cast<const uint32_t *>(m + __byte_perm(s, 0, 0x4440u + k));
        };
        quad_g(a, b, c, d, word(0), word(1));
        a = move(a, l.before), c = move(c, l.after), d = move(d, l.across);
        quad_g(a, b, c, d, word(2), word(3));
        a = move(a, l.after), c = move(c, l.before), d = move(d, l.across);
    }
    h0 ^= a ^ c;
    h1 ^= b ^ d;
}

// Words q and q + 4 of the chaining value that node (offset, depth) starts from.
__device__ __forceinline__ void quad_init(const QuadLane &l, uint32_t &h0, uint32_t &h1, const TreeParams &tp,
                                          uint64_t offset, uint32_t depth) {
    h0 = tp.h_base[l.q];
    h1 = tp.h_base[4 + l.q];
    if (l.q == 2) h0 ^= (uint32_t)offset;
    if (l.q == 3) h0 ^= ((uint32_t)(offset >> 32) & 0xFFFFu) | (depth << 16);
}

// A launch with programmatic stream serialisation may start while the launch before it on the
// stream drains: its blocks wait here until that launch has completed and its writes are
// visible.
__device__ __forceinline__ void wait_for_previous_launch() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// Lets the launch after this one start once every block has come this far (or ended).
__device__ __forceinline__ void allow_next_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

constexpr int kLeafThreads = kLeafBlockThreads;

// A block of the leaf launch: zeroes a fragment's arrival counters for the tree launch, and ends
// after the launch before this one, so that the tree launch comes after both.
__device__ __forceinline__ void zero_arrivals(const LeafLaunch &a) {
    for (uint32_t i = threadIdx.x; i < a.num_arrivals; i += kLeafThreads)
        if (CM_IN_BOUNDS(a.arrivals + i, 4, a.arrivals, (uint64_t)a.num_arrivals * 4)) a.arrivals[i] = 0;
    wait_for_previous_launch();
}

// kWhole: every plane of the group is a multiple of a leaf, so each leaf is 1 KiB of one
// segment. Otherwise a leaf may run into the next segments and a fragment's last leaf may be
// short (a multiple of 64 bytes, as 2 L planes are): every leaf then walks its blocks in
// halves of 32 bytes, one loop for all, so that a warp never hashes its straddling leaves
// after the others (as it once did: the tiny merge's leaves took 42 us, now 21).
template <bool kWhole>
__global__ void __launch_bounds__(kLeafThreads)
leaf_hash_kernel(const __grid_constant__ LeafGroup grp) {
    // the blocks after the leaf blocks, one per fragment (done by the leaf threads this cost
    // them 8 registers)
    const uint32_t x = blockIdx.x;
    const uint32_t leaf_blocks = (uint32_t)grp.block_begin[grp.count];
    if (x >= leaf_blocks) {
        zero_arrivals(grp.frag[x - leaf_blocks]);
        return;
    }
    uint32_t fi = 0;                                   // the block's fragment (uniform)
    while (fi + 1 < grp.count && x >= grp.block_begin[fi + 1]) ++fi;
    const LeafLaunch &a = grp.frag[fi];
    const uint64_t leaf = (uint64_t)(x - grp.block_begin[fi]) * kLeafThreads + threadIdx.x;
    if (leaf >= a.num_leaves) return;
    const uint64_t begin = leaf * kLeafBytes;
    const bool last_node = leaf + 1 == a.num_leaves;
    uint32_t h[8];
    node_init(h, a.tree, leaf, 0);
    StreamCursor cur = cursor_at(a, begin);
    if (kWhole) {
        const uint8_t *p = cur.ptr;
        if (!in_fragment(a, p, kLeafBytes)) return;
#pragma unroll 1
        for (uint32_t at = 0; at < (uint32_t)kLeafBytes; at += 64) {
            const uint4 w0 = load_nc(p + at), w1 = load_nc(p + at + 16), w2 = load_nc(p + at + 32),
                        w3 = load_nc(p + at + 48);
            const uint32_t m[16] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w,
                                    w2.x, w2.y, w2.z, w2.w, w3.x, w3.y, w3.z, w3.w};
            compress(h, m, at + 64, at + 64 == (uint32_t)kLeafBytes, last_node);
        }
    } else {
        const uint64_t rem = a.stream_bytes - begin;
        const uint32_t nblocks = rem < (uint64_t)kLeafBytes ? (uint32_t)rem / 64 : (uint32_t)kLeafBytes / 64;
#pragma unroll 1
        for (uint32_t b = 0; b < nblocks; ++b) {
            const uint8_t *p = cursor_next(a, cur), *q = cursor_next(a, cur);
            if (!in_fragment(a, p, 32) || !in_fragment(a, q, 32)) return;
            const uint4 w0 = load_nc(p), w1 = load_nc(p + 16), w2 = load_nc(q), w3 = load_nc(q + 16);
            const uint32_t m[16] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w,
                                    w2.x, w2.y, w2.z, w2.w, w3.x, w3.y, w3.z, w3.w};
            compress(h, m, (b + 1) * 64, b + 1 == nblocks, last_node);
        }
    }
    if (CM_IN_BOUNDS(a.digests + leaf * kDigestBytes, kDigestBytes, a.digests,
                     a.num_leaves * kDigestBytes))
        store_digest(a.digests + leaf * kDigestBytes, h);
}

// Level 0 with four lanes to a leaf, for groups of so few leaves that the chain of a leaf's 16
// compressions bounds them: kLeafThreads / 4 leaves to a block, so four blocks here for one of
// block_begin, then the blocks that zero the arrival counters as above. Lane q loads its 16
// bytes of the next block while this one is hashed.
__global__ void __launch_bounds__(kLeafThreads)
leaf_quad_kernel(const __grid_constant__ LeafGroup grp) {
    constexpr uint32_t kSlotBytes = 2 * 64 + 16;   // two blocks, 16 bytes to spread the leaves over the banks
    __shared__ __align__(16) uint8_t stage_all[kLeafThreads / 4][kSlotBytes];
    const uint32_t leaf_blocks = (uint32_t)grp.block_begin[grp.count];
    const uint32_t x = blockIdx.x >> 2;
    if (x >= leaf_blocks) {
        zero_arrivals(grp.frag[blockIdx.x - 4 * leaf_blocks]);
        return;
    }
    uint32_t fi = 0;                                   // the block's fragment (uniform)
    while (fi + 1 < grp.count && x >= grp.block_begin[fi + 1]) ++fi;
    const LeafLaunch &a = grp.frag[fi];
    const QuadLane l = quad_lane(threadIdx.x & 31u);
    const uint64_t leaf = (uint64_t)(x - grp.block_begin[fi]) * kLeafThreads +
                          (blockIdx.x & 3u) * (kLeafThreads / 4) + (threadIdx.x >> 2);
    const uint64_t begin = leaf * kLeafBytes;
    const uint64_t rem = leaf < a.num_leaves ? a.stream_bytes - begin : 0;
    const uint32_t nblocks = rem < (uint64_t)kLeafBytes ? (uint32_t)rem / 64 : (uint32_t)kLeafBytes / 64;
    uint8_t *stage = stage_all[threadIdx.x >> 2];
    uint64_t pos = begin + 16 * l.q;
    StreamCursor cur{};
    auto load = [&](uint32_t n) {   // this lane's part of block n, the block after the last one loaded
        if (n >= nblocks) return make_uint4(0, 0, 0, 0);
        if (n == 0 || cur.left <= 64) {
            cur = cursor_at(a, pos);
        } else {
            cur.ptr += 64;
            cur.left -= 64;
        }
        pos += 64;
        return in_fragment(a, cur.ptr, 16) ? load_nc(cur.ptr) : make_uint4(0, 0, 0, 0);
    };
    uint32_t h0, h1;
    quad_init(l, h0, h1, a.tree, leaf, 0);
    uint4 next = load(0);
#pragma unroll 1
    for (uint32_t n = 0; n < (uint32_t)kLeafBytes / 64; ++n) {
        if (!__any_sync(0xFFFFFFFFu, n < nblocks)) break;
        uint8_t *m = stage + 64 * (n & 1u);   // the other half may still be read
        *reinterpret_cast<uint4 *>(m + 16 * l.q) = next;
        __syncwarp();
        next = load(n + 1);
        const uint32_t k0 = h0, k1 = h1;
        quad_compress(l, h0, h1, m, (n + 1) * 64, n + 1 == nblocks, leaf + 1 == a.num_leaves);
        if (n >= nblocks) h0 = k0, h1 = k1;
    }
    uint8_t *out = a.digests + leaf * kDigestBytes + 4 * l.q;
    if (leaf < a.num_leaves && CM_IN_BOUNDS(out, 4, a.digests, a.num_leaves * kDigestBytes))
        *reinterpret_cast<uint32_t *>(out) = h0;
}

// The norm keys of a group: the blocks walk over the group's norm blocks. Ahead of a leaf
// launch they are at most one to an SM (the FP64 pipe bounds them, the ALU and FMA pipes the
// leaves), and the leaves start as soon as they run.
__global__ void __launch_bounds__(kLeafThreads)
norm_key_kernel(const __grid_constant__ LeafGroup grp) {
    allow_next_launch();
    const uint32_t total = (uint32_t)grp.norm_block_begin[grp.count];
    uint32_t fi = 0;
    for (uint64_t k = blockIdx.x; k < total; k += gridDim.x) {
        while (fi + 1 < grp.count && k >= grp.norm_block_begin[fi + 1]) ++fi;
        norm_block(grp.frag[fi], (uint32_t)(k - grp.norm_block_begin[fi]));
        __syncthreads();   // the sums in shared memory have been read
    }
}

constexpr int kTopThreads = 64;   // of a tree-top block

// Bytes of children under node j of a level above one of num_children nodes.
__device__ __forceinline__ uint32_t child_bytes(uint64_t num_children, uint64_t j) {
    const uint64_t left = num_children - j * kFanout;
    return (left < (uint64_t)kFanout ? (uint32_t)left : (uint32_t)kFanout) * kDigestBytes;
}

__device__ __forceinline__ uint32_t arrive_acq_rel(uint32_t *counter) {
    uint32_t old;
    asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], 1;" : "=r"(old) : "l"(counter) : "memory");
    return old;
}

constexpr int kLevel1Threads = 128;

// Level 1 of up to kMaxGroup fragments: one thread per node (node_begin: prefix sums of
// the level-1 sizes, each rounded up to the children of one parent), its children read
// straight into registers. Every lane of a warp hashes a node, and with no shared memory many
// warps fit on an SM.
__global__ void __launch_bounds__(kLevel1Threads)
level1_kernel(const __grid_constant__ TreeTop t) {
    wait_for_previous_launch();
    const uint64_t g = (uint64_t)blockIdx.x * kLevel1Threads + threadIdx.x;
    if (g >= t.node_begin[t.count]) return;
    uint32_t fi = 0;
    while (fi + 1 < t.count && g >= t.node_begin[fi + 1]) ++fi;
    const TreeTopFragment &f = t.frag[fi];
    const uint64_t j = g - t.node_begin[fi];
    if (j >= f.size[1]) return;
    const uint32_t len = child_bytes(f.size[0], j);
    const uint32_t nblocks = (len + 63) / 64;
    const bool last_node = j + 1 == f.size[1];
    const uint8_t *src = f.level[0] + j * kFanout * kDigestBytes;
    uint32_t h[8];
    node_init(h, f.tree, j, 1);
#pragma unroll 1
    for (uint32_t b = 0; b < nblocks; ++b) {
        uint4 w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t off = b * 64 + q * 16;
            w[q] = off < len && CM_IN_BOUNDS(src + off, 16, f.level[0], f.size[0] * kDigestBytes)
                       ? __ldcg(reinterpret_cast<const uint4 *>(src + off))
                       : make_uint4(0, 0, 0, 0);
        }
        const uint32_t m[16] = {w[0].x, w[0].y, w[0].z, w[0].w, w[1].x, w[1].y, w[1].z, w[1].w,
                                w[2].x, w[2].y, w[2].z, w[2].w, w[3].x, w[3].y, w[3].z, w[3].w};
        const uint32_t end = (b + 1) * 64 < len ? (b + 1) * 64 : len;
        compress(h, m, end, b + 1 == nblocks, last_node);
    }
    if (CM_IN_BOUNDS(f.level[1] + j * kDigestBytes, kDigestBytes, f.level[1], f.size[1] * kDigestBytes))
        store_digest(f.level[1] + j * kDigestBytes, h);
}

// Digest of a node by the four lanes that call with its arguments (the warp's lanes all call,
// with `blocks` the most of any): lane q's word of it. The node's len bytes of children's digests
// lie at `stage`, zero-padded to whole blocks.
__device__ __forceinline__ uint32_t quad_digest(const QuadLane &l, const uint8_t *stage, uint32_t len,
                                                uint32_t blocks, uint64_t j, uint64_t num_nodes,
                                                uint32_t depth, const TreeParams &tp) {
    const uint32_t mine = (len + 63) / 64;
    uint32_t h0, h1;
    quad_init(l, h0, h1, tp, j, depth);
#pragma unroll 1
    for (uint32_t n = 0; n < blocks; ++n) {
        const uint32_t k0 = h0, k1 = h1, end = (n + 1) * 64 < len ? (n + 1) * 64 : len;
        quad_compress(l, h0, h1, stage + 64 * n, end, n + 1 == mine, j + 1 == num_nodes);
        if (n >= mine) h0 = k0, h1 = k1;
    }
    return h0;
}

constexpr uint32_t kStageBytes = kFanout * kDigestBytes + 16;   // 16 to spread the nodes over the banks

// Levels kStart and up (node_begin: prefix sums of the level-kStart sizes, each rounded up to
// the children of one parent, 0 for a fragment without that level): a block hashes the level-
// kStart nodes of one parent, four lanes each, then its first warp the parent, handed over in
// shared memory; from there, level by level, the warp that completes a parent's last child
// hashes the parent. The chain of levels bounds it: four compressions to a node, and between
// levels a store, an arrival and the loads of 16 digests, which the hand-over saves once.
template <int kStart>
__global__ void __launch_bounds__(kTopThreads)
tree_top_kernel(const __grid_constant__ TreeTop t) {
    static_assert(kTopThreads == 4 * kFanout, "a block hashes the children of one parent");
    static_assert(kFanout * kDigestBytes == 256, "an inner node is at most four blocks");
    __shared__ __align__(16) uint8_t stage_all[kFanout][kStageBytes];
    __shared__ __align__(16) uint8_t stage_parent[kStageBytes];
    const QuadLane l = quad_lane(threadIdx.x & 31u);
    const uint64_t g = (uint64_t)blockIdx.x * kFanout;
    uint32_t fi = 0;
    while (fi + 1 < t.count && g >= t.node_begin[fi + 1]) ++fi;
    const TreeTopFragment &f = t.frag[fi];
    const uint32_t slot = threadIdx.x >> 2;
    uint64_t j = (g - t.node_begin[fi]) / kFanout;   // the parent
    uint32_t k = kStart;
    wait_for_previous_launch();
    {
        const uint64_t node = j * kFanout + slot;
        const bool mine = node < f.size[k];
        const uint32_t len = mine ? child_bytes(f.size[k - 1], node) : 0;
        const uint8_t *src = f.level[k - 1] + node * kFanout * kDigestBytes;
#pragma unroll
        for (int v = 0; v < 4; ++v) {   // read through L2: the launch that this one overlaps wrote them
            const uint32_t at = 64 * v + 16 * l.q;
            const uint4 w = at < len && CM_IN_BOUNDS(src + at, 16, f.level[k - 1], f.size[k - 1] * kDigestBytes)
                                ? __ldcg(reinterpret_cast<const uint4 *>(src + at))
                                : make_uint4(0, 0, 0, 0);
            *reinterpret_cast<uint4 *>(stage_all[slot] + at) = w;
        }
        __syncwarp();
        const uint32_t word = quad_digest(l, stage_all[slot], len, 4, node, f.size[k], k, f.tree);
        if (k + 1 == f.levels) {   // the root
            if (mine && CM_IN_BOUNDS(f.level[k] + 4 * l.q, 4, f.level[k], kDigestBytes))
                reinterpret_cast<uint32_t *>(f.level[k])[l.q] = word;
            return;
        }
        *reinterpret_cast<uint32_t *>(stage_parent + slot * kDigestBytes + 4 * l.q) = mine ? word : 0;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    uint32_t len = child_bytes(f.size[k], j);
    for (;;) {
        ++k;
        // every four lanes hash the same node
        const uint32_t word = quad_digest(l, stage_parent, len, (len + 63) / 64, j, f.size[k], k, f.tree);
        uint8_t *out = f.level[k] + j * kDigestBytes;
        if (threadIdx.x < 4 && CM_IN_BOUNDS(out + 4 * l.q, 4, f.level[k], f.size[k] * kDigestBytes))
            reinterpret_cast<uint32_t *>(out)[l.q] = word;
        if (k + 1 >= f.levels) return;
        // this warp finished node j of level k; the one that finishes the last child of
        // parent j / 16 hashes the parent
        const uint64_t parent = j / kFanout;
        len = child_bytes(f.size[k], parent);
        __syncwarp();
        // one acquire-release add: it publishes this node's digest and, for the warp
        // that counts the last sibling, makes every sibling's digest visible
        uint32_t done = 0;
        if (threadIdx.x == 0 && CM_IN_BOUNDS(f.arrivals[k + 1] + parent, 4, f.arrivals[k + 1], f.size[k + 1] * 4))
            done = arrive_acq_rel(f.arrivals[k + 1] + parent) + 1;
        done = __shfl_sync(0xFFFFFFFFu, done, 0);
        __syncwarp();   // lane 0's acquire comes before the other lanes' loads
        if (done * kDigestBytes != len) return;
        j = parent;
        if (threadIdx.x < (uint32_t)kFanout) {
            const uint8_t *src = f.level[k] + (j * kFanout + threadIdx.x) * kDigestBytes;
            const bool in = threadIdx.x * kDigestBytes < len &&
                            CM_IN_BOUNDS(src, 16, f.level[k], f.size[k] * kDigestBytes);
            const uint4 w = in ? __ldcg(reinterpret_cast<const uint4 *>(src)) : make_uint4(0, 0, 0, 0);
            *reinterpret_cast<uint4 *>(stage_parent + threadIdx.x * kDigestBytes) = w;
        }
        __syncwarp();
    }
}

__global__ void compare_kernel(const uint4 *__restrict__ a, const uint4 *__restrict__ b,
                               uint64_t n, unsigned int *flag) {
    uint32_t diff = 0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint4 x = __ldg(a + i), y = __ldg(b + i);
        diff |= (x.x ^ y.x) | (x.y ^ y.y) | (x.z ^ y.z) | (x.w ^ y.w);
    }
    if (__any_sync(0xFFFFFFFFu, diff != 0) && (threadIdx.x & 31) == 0) atomicOr(flag, 1u);
}

}  // namespace

CM_DEFINE_BOUNDS_READER(take_hash_bounds_violations)

int leaf_hash_blocks_per_sm() {
    void (*const kernels[])(LeafGroup) = {leaf_hash_kernel<true>, leaf_hash_kernel<false>};
    int least = 0;
    for (void (*const kernel)(LeafGroup) : kernels) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kLeafThreads, 0) != cudaSuccess) return 0;
        if (least == 0 || n < least) least = n;
    }
    return least;
}

namespace {

// Launches a kernel that may start once every block of the launch before it on `stream` has
// ended or called allow_next_launch; it waits for that launch where it has to
// (wait_for_previous_launch). The kernels that a tree launch follows do not call it: its
// one-warp blocks, placed while the leaves still hold most SMs, would crowd on the free ones
// (one 1021-token ingest 200 us with the call, 160 us without, 167 us launched plainly).
template <class P>
cudaError_t launch_after(void (*kernel)(P), uint64_t blocks, int threads, cudaStream_t stream, const P &p) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

}  // namespace

cudaError_t launch_leaf_hash_group(const LeafGroup &g, bool with_norms, int num_sms, cudaStream_t stream) {
    if (g.count > (uint32_t)kMaxLeafGroup) return cudaErrorInvalidValue;
    if (g.count == 0) return cudaSuccess;
    // four lanes to a leaf up to half a leaf block per SM (two such warps per scheduler; beyond,
    // they take more issue slots than the chain leaves free): tiny merge 63 -> 58 us, one
    // 60-token ingest of the Qwen3-4B shape 56 -> 54.5, but of 100 tokens 56 -> 61
    const bool few = g.block_begin[g.count] * 2 <= (uint64_t)num_sms;
    const uint64_t blocks = (few ? 4 : 1) * g.block_begin[g.count] + g.count;   // leaves, then arrival counters
    if (blocks > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    bool whole = true;
    for (uint32_t i = 0; i < g.count; ++i) whole = whole && g.frag[i].plane_bytes % kLeafBytes == 0;
    void (*const kernel)(LeafGroup) = few     ? leaf_quad_kernel
                                      : whole ? leaf_hash_kernel<true>
                                              : leaf_hash_kernel<false>;
    if (!with_norms) {
        kernel<<<(unsigned)blocks, kLeafThreads, 0, stream>>>(g);
        return cudaGetLastError();
    }
    const cudaError_t e = launch_norm_keys(g, (uint64_t)num_sms, stream);
    return e != cudaSuccess ? e : launch_after(kernel, blocks, kLeafThreads, stream, g);
}

cudaError_t launch_norm_keys(const LeafGroup &in, uint64_t max_blocks, cudaStream_t stream) {
    if (in.count > (uint32_t)kMaxLeafGroup) return cudaErrorInvalidValue;
    if (in.count == 0) return cudaSuccess;
    LeafGroup g = in;
    for (uint32_t i = 0; i < g.count; ++i) {
        const uint64_t tokens = kLeafBlockThreads / norm_lanes(g.frag[i].heads);   // per block
        g.norm_block_begin[i + 1] = g.norm_block_begin[i] + (g.frag[i].seq_len + tokens - 1) / tokens;
    }
    const uint64_t total = g.norm_block_begin[g.count];
    if (total > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    const uint64_t blocks = total < max_blocks ? total : max_blocks;
    norm_key_kernel<<<(unsigned)blocks, kLeafThreads, 0, stream>>>(g);
    return cudaGetLastError();
}

static uint64_t level1_nodes(const TreeTop &t) {
    uint64_t n = 0;
    for (uint32_t i = 0; i < t.count; ++i) n += t.frag[i].size[1];
    return n;
}

int tree_top_kernels(const TreeTop &t) {
    const uint64_t nodes = t.count > (uint32_t)kMaxGroup ? 0 : level1_nodes(t);
    if (nodes < kSplitLevel1Nodes) return nodes == 0 ? 0 : 1;
    for (uint32_t i = 0; i < t.count; ++i)
        if (t.frag[i].levels >= 3) return 2;
    return 1;
}

namespace {

// node_begin for level `k`: each fragment's nodes rounded up to the children of one parent, so
// that no tree-top block holds nodes of two.
void count_level(TreeTop &t, uint32_t k) {
    for (uint32_t i = 0; i < t.count; ++i) {
        const uint64_t nodes = k < t.frag[i].levels ? t.frag[i].size[k] : 0;
        t.node_begin[i + 1] = t.node_begin[i] + (nodes + kFanout - 1) / kFanout * kFanout;
    }
}

}  // namespace

cudaError_t launch_tree_top(const TreeTop &in, cudaStream_t stream) {
    if (in.count > (uint32_t)kMaxGroup) return cudaErrorInvalidValue;
    const int kernels = tree_top_kernels(in);
    if (kernels == 0) return cudaSuccess;
    TreeTop t = in;
    count_level(t, 1);
    const uint64_t total1 = t.node_begin[t.count];
    if (level1_nodes(in) < kSplitLevel1Nodes)
        // one launch from level 1: the level-2 parents are hashed by the warps that hash their
        // children, with no second launch
        return launch_after(tree_top_kernel<1>, total1 / kFanout, kTopThreads, stream, t);
    const cudaError_t e = launch_after(level1_kernel, (total1 + kLevel1Threads - 1) / kLevel1Threads,
                                       kLevel1Threads, stream, t);
    if (e != cudaSuccess || kernels == 1) return e;
    count_level(t, 2);
    return launch_after(tree_top_kernel<2>, t.node_begin[t.count] / kFanout, kTopThreads, stream, t);
}

cudaError_t launch_compare(const void *a, const void *b, uint64_t bytes, unsigned int *flag,
                           cudaStream_t stream) {
    const uint64_t n = bytes / 16;
    if (n == 0) return cudaSuccess;
    uint64_t blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    compare_kernel<<<(unsigned)blocks, 256, 0, stream>>>(static_cast<const uint4 *>(a),
                                                         static_cast<const uint4 *>(b), n, flag);
    return cudaGetLastError();
}

}  // namespace cm

// ---------------------------------------------------------------- allocation-free Id(C)
//
// cm_fragment_id_static computes what cm_fragment_id computes, for callers that
// cannot allocate device memory: its scratch (the digests of every tree level
// below the root and the arrival counters) lives in the file-scope array below, which every GPU that loads
// this library holds for the life of the process. Host code never uses the
// array's name as an address: every call looks the array's device address up with
// cudaGetSymbolAddress, with the calling thread's device current, and keeps no copy
// of it, so a device reset or another context on the device, either of which can
// move the array, never leaves a stale address in use.

namespace cm {
namespace {

constexpr uint64_t kStaticMaxLeaves = 1ull << 20;                // byte stream of at most 1 GiB
constexpr size_t kStaticScratchBytes = (17u << 20) + (256u << 10);   // 17.25 MiB
}  // namespace

static __device__ __align__(256) uint8_t g_static_scratch[kStaticScratchBytes];

}  // namespace cm

extern "C" cm_status cm_fragment_id_static(const cm_fragment *frag, int32_t routing_layer,
                                           cm_stream_t stream, void *id_out,
                                           uint64_t *norm_key_out) {
    using namespace cm;
    try {
        cm_status st = check_fragment(frag);
        if (st != CM_OK) return st;
        if (!id_out || !norm_key_out)
            return report_error(CM_ERR_INVALID_ARG, "id_out and norm_key_out must be device pointers");
        if ((reinterpret_cast<uintptr_t>(id_out) & 15u) != 0 ||
            (reinterpret_cast<uintptr_t>(norm_key_out) & 7u) != 0)
            return report_error(CM_ERR_ALIGNMENT,
                                "id_out must be 16-byte and norm_key_out 8-byte aligned");
        const int32_t L = frag->num_layers, H = frag->num_kv_heads, T = frag->seq_len,
                      d = frag->head_dim;
        const int32_t rl = routing_layer < 0 ? L / 2 : routing_layer;
        if (rl >= L) return report_error(CM_ERR_INVALID_ARG, "routing layer >= num_layers");
        const uint64_t plane = (uint64_t)H * T * d * 2;
        const uint64_t stream_bytes = 2ull * L * plane;
        std::vector<uint64_t> sizes{(stream_bytes + kLeafBytes - 1) / kLeafBytes};
        if (sizes[0] > kStaticMaxLeaves)
            return report_error(CM_ERR_UNSUPPORTED,
                                "cm_fragment_id_static: the fragment's K and V bytes exceed the "
                                "1 GiB that its static scratch covers; use cm_fragment_id");
        while (sizes.size() == 1 || sizes.back() > 1)
            sizes.push_back((sizes.back() + kFanout - 1) / kFanout);
        // levels below the root in the static array, each 256-byte aligned, then the arrival
        // counters of the levels >= 2; the root (the last level, one node) is written straight
        // to id_out
        std::vector<size_t> off;
        size_t used = 0;
        for (size_t k = 0; k + 1 < sizes.size(); ++k) {
            off.push_back(used);
            used += ((size_t)sizes[k] * kDigestBytes + 255) & ~(size_t)255;
        }
        const size_t arrivals_off = used;
        uint32_t num_arrivals = 0;
        for (size_t k = 2; k < sizes.size(); ++k) num_arrivals += (uint32_t)sizes[k];
        used += (size_t)num_arrivals * 4;
        if (used > kStaticScratchBytes)
            return report_error(CM_ERR_UNSUPPORTED, "static scratch layout overflow");
        cudaError_t e = cudaSuccess;
        const cudaStream_t cs = reinterpret_cast<cudaStream_t>(stream);
        void *addr = nullptr;
        e = cudaGetSymbolAddress(&addr, g_static_scratch);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return report_error(CM_ERR_CUDA, cudaGetErrorString(e));
        }
        uint8_t *scratch = static_cast<uint8_t *>(addr);
        LeafLaunch a;
        a.k = static_cast<const uint8_t *>(frag->k);
        a.v = static_cast<const uint8_t *>(frag->v);
        a.plane_bytes = plane;
        a.stream_bytes = stream_bytes;
        a.num_leaves = sizes[0];
        a.norm_begin = 2ull * (uint64_t)rl * plane;
        a.row_bytes = (uint32_t)d * 2;
        a.seq_len = (uint32_t)T;
        a.norm_key = reinterpret_cast<unsigned long long *>(norm_key_out);
        a.heads = (uint32_t)H;
        a.num_arrivals = num_arrivals;
        a.arrivals = reinterpret_cast<uint32_t *>(scratch + arrivals_off);
        a.digests = scratch + off[0];
        a.tree = make_tree_params(L, H, d, T);
        LeafGroup g;
        std::memset(&g, 0, sizeof g);
        g.count = 1;
        g.block_begin[1] = (a.num_leaves + kLeafThreads - 1) / kLeafThreads;
        g.frag[0] = a;
        int device = 0, num_sms = 0;
        e = cudaGetDevice(&device);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, device);
        if (e == cudaSuccess) e = launch_leaf_hash_group(g, true, num_sms, cs);
        if (e != cudaSuccess) return report_error(CM_ERR_CUDA, cudaGetErrorString(e));
        TreeTop top;
        std::memset(&top, 0, sizeof top);
        top.count = 1;
        TreeTopFragment &tf = top.frag[0];
        tf.levels = (uint32_t)sizes.size();
        uint32_t *arrivals = a.arrivals;
        for (size_t k = 0; k < sizes.size(); ++k) {
            tf.size[k] = sizes[k];
            tf.level[k] = k + 1 == sizes.size() ? static_cast<uint8_t *>(id_out) : scratch + off[k];
            if (k >= 2) {
                tf.arrivals[k] = arrivals;
                arrivals += sizes[k];
            }
        }
        tf.tree = a.tree;
        e = launch_tree_top(top, cs);
        if (e != cudaSuccess) return report_error(CM_ERR_CUDA, cudaGetErrorString(e));
        return CM_OK;
    } catch (...) {
        return report_error(CM_ERR_OOM, "host allocation failed");
    }
}

// ---------------------------------------------------------------- integer-ALU throughput
//
// Register-only kernels that measure the ceiling of the content-address kernels on the
// current GPU (a profiling aid for their roofline): chains of three-input xors, one
// integer-ALU instruction each, and the compression function above applied to register
// data with no memory traffic, counted as the 648 xors and rotations of a 64-byte block
// (10 rounds x 8 G x (4 xors + 4 rotations) + 8 xors).

namespace cm {
namespace {

__global__ void __launch_bounds__(kLeafThreads)
xor3_probe_kernel(uint32_t *out, int iters) {
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t a[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = tid * (2u * i + 3u);
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = a[i] ^ a[(i + 1) & 7] ^ a[(i + 3) & 7];
    }
    uint32_t x = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) x ^= a[i];
    out[tid] = x;
}

__global__ void __launch_bounds__(kLeafThreads)
compress_probe_kernel(uint32_t *out, int blocks) {
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t h[8], m[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = tid * 2654435761u + (uint32_t)i;
#pragma unroll
    for (int i = 0; i < 16; ++i) m[i] = tid ^ ((uint32_t)i * 0x9E3779B9u);
    for (int b = 0; b < blocks; ++b) {
        compress(h, m, (uint64_t)(b + 1) * 64, false, false);
        m[0] ^= h[0];
        m[7] ^= h[3];
        m[11] ^= h[6];
    }
    out[tid] = h[0] ^ h[1] ^ h[2] ^ h[3] ^ h[4] ^ h[5] ^ h[6] ^ h[7];
}

}  // namespace
}  // namespace cm

extern "C" cm_status cm_measure_int_alu(int32_t device, double *xor3_tops, double *compress_tops) {
    using namespace cm;
    if (!xor3_tops || !compress_tops)
        return report_error(CM_ERR_INVALID_ARG, "xor3_tops and compress_tops are required");
    int prev = 0;
    cudaError_t e = cudaGetDevice(&prev);
    if (e != cudaSuccess) return report_error(CM_ERR_CUDA, cudaGetErrorString(e));
    e = cudaSetDevice(device);
    if (e != cudaSuccess) return report_error(CM_ERR_CUDA, cudaGetErrorString(e));
    cm_status st = CM_OK;
    uint32_t *out = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    auto check = [&](cudaError_t err) {
        if (err != cudaSuccess && st == CM_OK) st = report_error(CM_ERR_CUDA, cudaGetErrorString(err));
        return err == cudaSuccess;
    };
    int sms = 0, per_sm_x = 0, per_sm_c = 0;
    if (check(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device)) &&
        check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_x, xor3_probe_kernel,
                                                            kLeafThreads, 0)) &&
        check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_c, compress_probe_kernel,
                                                            kLeafThreads, 0))) {
        // four full waves of each kernel
        const int grid_x = 4 * sms * per_sm_x, grid_c = 4 * sms * per_sm_c;
        const int grid = grid_x > grid_c ? grid_x : grid_c;
        const int xor_iters = 4096, comp_blocks = 64;
        if (check(cudaMalloc(&out, (size_t)grid * kLeafThreads * sizeof(uint32_t))) &&
            check(cudaEventCreate(&e0)) && check(cudaEventCreate(&e1))) {
            auto best_ms = [&](auto launch) {
                float best = 0.0f;
                for (int rep = 0; rep < 4 && st == CM_OK; ++rep) {   // rep 0 warms up
                    check(cudaEventRecord(e0));
                    launch();
                    check(cudaGetLastError());
                    check(cudaEventRecord(e1));
                    float ms = 0.0f;
                    if (check(cudaEventSynchronize(e1)) && check(cudaEventElapsedTime(&ms, e0, e1)) &&
                        rep > 0 && (best == 0.0f || ms < best))
                        best = ms;
                }
                return (double)best;
            };
            const double ms_x = best_ms([&] {
                xor3_probe_kernel<<<grid_x, kLeafThreads>>>(out, xor_iters);
            });
            const double ms_c = best_ms([&] {
                compress_probe_kernel<<<grid_c, kLeafThreads>>>(out, comp_blocks);
            });
            if (st == CM_OK) {
                const double ops_x = (double)grid_x * kLeafThreads * xor_iters * 8;
                const double ops_c = (double)grid_c * kLeafThreads * comp_blocks * 648;
                *xor3_tops = ops_x / (ms_x * 1e-3) / 1e12;
                *compress_tops = ops_c / (ms_c * 1e-3) / 1e12;
            }
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (out) cudaFree(out);
    cudaSetDevice(prev);
    return st;
}
