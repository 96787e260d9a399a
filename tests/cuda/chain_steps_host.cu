// The engine's count of a Metropolis chain's steps and tiles, called on the
// host: reads "n C tile" lines, writes "steps tiles" lines.
#include <cstdio>

#include "common.cuh"

int main() {
    unsigned n, C, tile;
    while (std::scanf("%u %u %u", &n, &C, &tile) == 3)
        std::printf("%u %u\n", gdpm::chain_steps(n, C), gdpm::chain_tiles(n, C, tile));
    return 0;
}
