// Prints the library's layout choice for configurations read from the standard input, a line each of
// m c n_nodes edges: the pool bytes per edge of a handle made for them.
#include <cstdio>

#include "rept_common.cuh"

using namespace rept;

int main() {
    unsigned m, c, n;
    unsigned long long edges;
    while (std::scanf("%u %u %u %llu", &m, &c, &n, &edges) == 4) {
        uint32_t bits = 0, colours = widest_colours(m, c, n, false, bits);
        if (colours == kColMulti && quads_bound(edges, kColMulti) > kMaxQuads) colours = kColNone;
        std::printf("%llu\n", 32ull * (quads_bound(1u, colours) - quads_bound(0u, colours)));
    }
    return 0;
}
