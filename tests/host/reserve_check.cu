// Host-side check of the histogram room that a tile-ordered state's binning
// needs: it always bins in BIN_TILE tiles with BIN_MIN_SPAN, so a reservation by
// another span of the plan's does not cover it.  Runs on the CPU only.
#include <cstdint>
#include <cstdio>

#include "common.cuh"

int main() {
    int failures = 0, short_by_plan = 0;
    const int grids[][2] = {{8, 8}, {100, 77}, {1024, 1024}, {2048, 1800}};
    const int64_t counts[] = {0, 1, 1024, 1025, 4097, 100000, 622591, 622592, 4000000};
    for (auto& g : grids)
        for (int64_t nv : counts) {
            const int tiles = ((g[0] + BIN_TILE - 1) / BIN_TILE) * ((g[1] + BIN_TILE - 1) / BIN_TILE);
            const int64_t launched = (int64_t)bin_blocks(nv) * tiles;                   // rows that the passes write
            if (bin_off_ints(g[0], g[1], BIN_TILE, nv, BIN_MIN_SPAN) < launched) ++failures;
            for (int span : {2048, 4096}) short_by_plan += bin_off_ints(g[0], g[1], BIN_TILE, nv, span) < launched;
        }
    if (failures || !short_by_plan) {
        std::printf("%d reservations too small, %d by another span\n", failures, short_by_plan);
        return 1;
    }
    std::printf("OK\n");
    return 0;
}
