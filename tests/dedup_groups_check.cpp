// Host check of cm_dedup_groups.h (no GPU): the launch groups of full comparisons between
// fragments that start at one address. Prints "ok" or the first line that does not hold.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "cm_dedup_groups.h"

#define CHECK(x)                                                  \
    do {                                                          \
        if (!(x)) {                                               \
            std::printf("line %d: %s\n", __LINE__, #x);           \
            return 1;                                             \
        }                                                         \
    } while (0)

namespace {

alignas(16) unsigned char buffers[16][64];   // addresses only: nothing is read

cm_fragment fragment(int k, int L, int H, int T, int d) { return {L, H, T, d, buffers[2 * k], buffers[2 * k + 1]}; }

// Every member in one group, compared with its own base (the one before it, in a chain) over its
// own size; chunks as long as the sizes say.
int check_in_order(const std::vector<cm::Comparison> &c, uint32_t want_groups, uint32_t want_chains) {
    static cm::CompareFull out;
    CHECK(cm::group_comparisons(c.data(), c.size(), out));
    CHECK(out.groups == want_groups);
    uint32_t m = 0;
    for (uint32_t g = 0; g < out.groups; ++g) {
        const cm::CompareGroup &q = out.group[g];
        CHECK(q.begin == m && q.end > m && q.end - q.begin <= cm::kMaxCompareGroup);
        for (; m < q.end; ++m) {
            const uint64_t vecs = cm::fragment_vecs(c[m].member);
            const bool first = m == q.begin || q.chain == 0;
            CHECK((first ? q.kv[0] : out.member[m - 1].kv[0]) == c[m].base.k);
            CHECK((first ? q.kv[1] : out.member[m - 1].kv[1]) == c[m].base.v);
            CHECK(q.vecs == vecs && out.member[m].vecs == vecs);
            CHECK(out.member[m].kv[0] == c[m].member.k && out.member[m].kv[1] == c[m].member.v);
        }
        const uint64_t chunks = 2 * ((q.vecs + cm::kCompareChunkVecs - 1) / cm::kCompareChunkVecs);
        CHECK(out.chunk_begin[g + 1] - out.chunk_begin[g] == chunks);
    }
    CHECK(m == c.size());
    uint32_t chains = 0;
    for (uint32_t g = 0; g < out.groups; ++g) chains += out.group[g].chain;
    CHECK(chains == want_chains);
    return 0;
}

int check(std::vector<cm::Comparison> c, uint32_t want_groups) {
    std::stable_sort(c.begin(), c.end(), [](const cm::Comparison &a, const cm::Comparison &b) {
        return cm::compare_fragments(a.base, b.base) < 0;
    });
    return check_in_order(c, want_groups, 0);
}

}  // namespace

int main() {
    // a fragment of 3 layers and its first 2 layers; one of 900 tokens and its first 700 (one
    // layer and head); the same bytes as 2 layers x 3 heads and as 3 x 2: a copy of each
    const cm_fragment pairs[3][2] = {{fragment(0, 3, 2, 50, 64), fragment(0, 2, 2, 50, 64)},
                                     {fragment(0, 1, 1, 900, 64), fragment(0, 1, 1, 700, 64)},
                                     {fragment(0, 2, 3, 50, 64), fragment(0, 3, 2, 50, 64)}};
    for (const auto &p : pairs) {
        std::vector<cm::Comparison> c;
        for (int i = 0; i < 6; ++i) {
            cm_fragment copy = p[i & 1];
            copy.k = buffers[2 * (i + 1)], copy.v = buffers[2 * (i + 1) + 1];
            c.push_back({p[i & 1], copy});
        }
        if (check(c, 2) != 0) return 1;                                    // one base, three copies each
        std::reverse(c.begin(), c.end());
        if (check(c, 2) != 0) return 1;
    }
    // one fragment's copies share a group; other buffers do not
    const cm_fragment a = fragment(0, 3, 2, 50, 64), b = fragment(1, 3, 2, 50, 64);
    if (check({{a, fragment(2, 3, 2, 50, 64)}, {b, fragment(3, 3, 2, 50, 64)}, {a, fragment(4, 3, 2, 50, 64)}}, 2) != 0)
        return 1;
    // a chain is one group; its end, another chain and a base with several copies are not in it
    const cm_fragment f[6] = {a, b, fragment(2, 3, 2, 50, 64), fragment(3, 3, 2, 50, 64), fragment(4, 3, 2, 50, 64),
                              fragment(5, 3, 2, 50, 64)};
    if (check_in_order({{f[0], f[1]}, {f[1], f[2]}, {f[2], f[3]}}, 1, 1) != 0) return 1;
    if (check_in_order({{f[0], f[1]}, {f[1], f[2]}, {f[3], f[4]}, {f[4], f[5]}}, 2, 2) != 0) return 1;
    if (check_in_order({{f[0], f[1]}, {f[0], f[2]}, {f[2], f[3]}, {f[3], f[4]}}, 2, 1) != 0) return 1;
    if (check_in_order({{f[0], f[1]}, {f[1], f[2]}, {f[1], f[3]}}, 2, 1) != 0) return 1;
    // (a part of a fragment that ends a chain is another fragment)
    if (check_in_order({{f[0], f[1]}, {fragment(1, 2, 2, 50, 64), fragment(2, 2, 2, 50, 64)}}, 2, 0) != 0) return 1;
    // sizes that differ are refused, and so are more than a launch holds
    static cm::CompareFull out;
    const cm::Comparison wrong{a, fragment(2, 2, 2, 50, 64)};
    CHECK(!cm::group_comparisons(&wrong, 1, out));
    const std::vector<cm::Comparison> many(cm::kMaxComparePairs + 1, {a, b});
    CHECK(!cm::group_comparisons(many.data(), many.size(), out));
    CHECK(cm::group_comparisons(many.data(), many.size() - 1, out) && out.groups == 4);   // full ones
    std::printf("ok\n");
    return 0;
}
