// Host-only check of which streams store colour words beside their entries (widest_colours, quads_bound,
// words_fit).  Exit code 0: all as stated.
#include <cstdio>

#include "rept_common.cuh"

using namespace rept;

static int bad = 0;
static void expect(bool ok, const char* what) {
    if (!ok) std::printf("not so: %s\n", what), ++bad;
}

int main() {
    uint32_t bits = 0;
    expect(widest_colours(100, 100, 1u << 24, false, bits) == kColInEntry, "one group, 100 colours: in the entry");
    expect(widest_colours(100, 100, (1u << 24) + 1u, false, bits) == kColWords && bits == 7, "one group, many nodes");
    expect(widest_colours(300, 120, 10, false, bits) == kColWords && bits == 9, "one group, 300 colours");
    expect(widest_colours(20, 100, 10, false, bits) == kColMulti && bits == 5, "five groups of 20 colours: 25 bits");
    expect(widest_colours(20, 140, 10, false, bits) == kColNone, "seven groups of 20 colours: 35 bits");
    expect(widest_colours(10, 32, 10, true, bits) == kColMulti && bits == 1, "32 samplers");
    expect(widest_colours(10, 33, 10, true, bits) == kColNone, "33 samplers");
    expect(widest_colours(1000, 1, 10, true, bits) == kColMulti && bits == 1, "one sampler of 1,000 colours");
    expect(widest_colours(10, 1, 10, true, bits) == kColInEntry, "one sampler of ten colours");
    expect(widest_colours(1, 1, 10, false, bits) == kColMulti && bits == 1, "one processor that keeps everything");
    expect(widest_colours(4294967295u, 4096, 10, false, bits) == kColWords && bits == 32, "the largest m");
    // Offsets of 32 bits span 536 million edges' blocks without words, 357 million with them.
    const unsigned long long most = kMaxQuads, gb = 1ull << 30;
    expect(quads_bound(357000000ull, kColMulti) <= most && quads_bound(359000000ull, kColMulti) > most, "with words");
    expect(quads_bound(536000000ull, kColNone) <= most && quads_bound(538000000ull, kColNone) > most, "without");
    // A pool with words leaves room for the one that takes over from it (4/3 of it) beside itself.
    expect(words_fit(1000000000ull, 280 * gb, most), "32 GB of 280");
    expect(!words_fit(most + 1ull, 2800 * gb, most), "beyond the offsets");
    expect(words_fit(3 * gb / 32ull, 7 * gb, most) && !words_fit(3 * gb / 32ull + 32ull, 7 * gb, most), "three sevenths");
    expect(!words_fit(~0ull, ~0ull, ~0ull), "no wrap");
    std::printf("wrong: %d\n", bad);
    return bad != 0;
}
