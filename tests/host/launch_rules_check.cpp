// Host-only check of the arithmetic behind the choice of kernels.
#include <cstdio>
#include <cstdlib>

#include "launch_rules.h"

using namespace uoe;

int main() {
    std::srand(1);
    // the fewest row tiles: no routing has fewer, and regions without padding have just as many
    for (int trial = 0; trial < 200000; ++trial) {
        const int n = 1 + std::rand() % 31, l_a = 1 + std::rand() % 600;
        long long rows = 0, tiles = 0;
        for (int e = 0; e < n; ++e) {
            const long long r = (long long)(std::rand() % 12) * l_a;
            rows += r;
            tiles += (r + kRowTile - 1) / kRowTile;
        }
        const long long rows_max = (rows + (long long)n * (kRowTile - 1)) / kRowTile * kRowTile, least = least_row_tiles(rows_max, n);
        if (least > tiles || tiles * kRowTile > rows_max) return 1;
        if (rows % kRowTile == 0 && rows > 0 && least != rows / kRowTile) return 2;
        // one tile for q, k and v only where three would be more than a wave
        if (qkv_as_one_tile(rows_max, n, 148) && 3 * tiles <= 148) return 3;
    }
    const long long pad = 8 * (kRowTile - 1);
    auto bound = [&](long long rows) { return (rows + pad) / kRowTile * kRowTile; };
    if (qkv_as_one_tile(bound(49 * 128), 8, 148) || !qkv_as_one_tile(bound(50 * 128), 8, 148)) return 4;
    // a sample of many slabs gets all warps, whatever the number of weight-gradient tiles
    if (router_grad_threads(false, 4, 1280) != 512 || router_grad_threads(false, 300, 1280) != 512 || router_grad_threads(false, 8, 240) != 512) return 5;
    if (router_grad_threads(false, 24, 240) != 256 || router_grad_threads(false, 8, 32) != 256 || router_grad_threads(true, 8, 32) != 512) return 6;
    std::printf("ok\n");
    return 0;
}
