// Host-only check of the block layouts (block_quads, key_word, eidx_of, list_of, aux_of, cw_of) at every table
// size up to 2^31 slots: the table, the list and what stands beside it follow one another inside the block,
// none reaching into the next.  Exit code 0: they do.
#include <cstdint>
#include <cstdio>

#include "rept_common.cuh"

using namespace rept;

int main() {
    long bad = 0;
    for (uint32_t colours : {kColNone, kColInEntry, kColWords, kColMulti}) {
        for (uint32_t lg = 2; lg <= 31u; ++lg) {
            const uint64_t slots = 1ull << lg, entries = lg >= 3u ? slots / 2u : 4u;
            const uint64_t table = (colours == kColMulti ? 3u : 2u) * slots;  // words
            const uint64_t beside = colours == kColMulti ? 2u * entries : entries, end = table + entries + beside;
            const uint64_t words = colours == kColWords ? (lg >= 4u ? slots / 4u : 4u) * 2u : 0u;
            const uint64_t block = 8ull * block_quads(lg, colours);
            const uint32_t last = (uint32_t)(slots - 1u);
            bool ok = block >= end + words && block < end + words + 8u;
            const uint32_t* at = nullptr;
            auto words_to = [&](const uint32_t* p) { return (uint64_t)(reinterpret_cast<uintptr_t>(p) / 4u); };
            ok = ok && words_to(list_of(at, lg, colours)) == table && words_to(aux_of(at, lg, colours)) == table + entries;
            if (colours == kColWords) ok = ok && words_to(cw_of(at, lg)) == end;
            ok = ok && key_word(0u, colours) == 0u && key_word(last, colours) < table;
            ok = ok && words_to(eidx_of(at, last, lg, colours)) + (colours == kColMulti ? 2u : 1u) == table;
            ok = ok && words_to(eidx_of(at, 0u, lg, colours)) == (interleaved(colours) ? 4u : slots);
            if (!ok) std::printf("layout %u: tables of 2^%u slots\n", colours, lg);
            bad += !ok;
        }
    }
    std::printf("wrong: %ld\n", bad);
    return bad != 0;
}
