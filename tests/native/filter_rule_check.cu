// Host-only check of the rule for the intersection's filters (filter_pays): none where its building costs more than
// the scan it serves.  Exit code 0: all as stated.
#include <cstdio>

#include "rept_common.cuh"

using namespace rept;

int main() {
    int bad = 0;
    for (uint32_t colours : {kColNone, kColInEntry, kColWords, kColMulti}) {
        bad += filter_pays(colours, 1000000u, 16u * 60u);       // a hub of a million entries, 16 short lists
        bad += filter_pays(colours, 20000u, 40u);               // 20,000 entries for one short list
        bad += filter_pays(colours, 2000000u, 1000000u);        // more entries than the filter has bits
        bad += !filter_pays(colours, 4096u, 64u * 100u);        // the ordinary unit
        bad += !filter_pays(colours, 20000u, 64u * 1000u);
        bad += !filter_pays(colours, 300u, 100u);
    }
    bad += filter_pays(kColInEntry, 24577u, 1u << 20) + filter_pays(kColMulti, 262145u, 1u << 20);
    bad += !filter_pays(kColInEntry, 24576u, 1u << 20) + !filter_pays(kColMulti, 262144u, 1u << 20);
    std::printf("wrong: %d\n", bad);
    return bad != 0;
}
