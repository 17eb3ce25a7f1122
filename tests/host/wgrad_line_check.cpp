// Host-only check of the bounds on the line of weight-gradient tiles: the line that the kernel builds, for every kind of
// expert load, is no longer than the bound, and its positions and piece ends fit 32 bits where wgrad_line_fits says so.
#include <cstdio>
#include <cstdlib>

#include "wgrad_line.h"

using namespace uoe;

int main() {
    std::srand(1);
    int full = 0, refused = 0;
    for (int trial = 0; trial < 20000; ++trial) {
        const int n = 1 + std::rand() % 32, nprob = 1 + std::rand() % 2, pieces = 1 + std::rand() % 148;
        WTileShape t[2];
        int wmax = 0;
        for (int p = 0; p < nprob; ++p) {
            t[p] = wgrad_tile_shape(128 * (1 + std::rand() % 64), 64 * (1 + std::rand() % 64));
            if (t[p].w > wmax) wmax = t[p].w;
        }
        // loads in 128-row units: from none at all to a few experts with everything
        const long long units = (1ll << (std::rand() % 24)) - 1;
        long long kb[32] = {}, left = units;
        for (int e = 0; e < n && left > 0; ++e) {
            const long long take = std::rand() % 3 ? 0 : (e == n - 1 ? left : std::rand() % (left + 1));
            kb[e] = 2 * take;
            left -= take;
        }
        long long line = 0;          // as wsched_build adds it up
        for (int p = 0; p < nprob; ++p)
            for (int e = 0; e < n; ++e) line += (kb[e] > kMinTileKb ? kb[e] : kMinTileKb) * t[p].m_tiles * t[p].n_tiles * t[p].w;
        const long long bound = wgrad_line_bound(t, nprob, n, units * 128);
        if (line > bound) { std::printf("line %lld, bound %lld, n %d\n", line, bound, n); return 1; }
        if (!wgrad_line_fits(bound, wmax, pieces)) { ++refused; continue; }
        long long Q = (line + pieces - 1) / pieces;
        if (Q < 4ll * wmax) Q = 4ll * wmax;
        // the pieces the line can fill are as long as with more of them, and hold the whole line
        const int used = wgrad_pieces(bound, wmax, pieces);
        long long Qu = (line + used - 1) / used;
        if (Qu < 4ll * wmax) Qu = 4ll * wmax;
        if (used > pieces || (Qu != Q && used < pieces) || used * Qu < line) { std::printf("%d of %d pieces\n", used, pieces); return 5; }
        if (pieces * Q > 0x7fffffffll || line + pieces > 0x7fffffffll) { std::printf("piece end %lld\n", pieces * Q); return 2; }
        full += bound < 0x7fffffffll / 2 ? 0 : 1;
    }
    // widths that only the workspace query sees
    if (wgrad_tile_shape(32, 8).BN != 64 || wgrad_tile_shape(32, 8).m_tiles != 0) return 3;
    if (full == 0 || refused == 0) { std::printf("full %d refused %d\n", full, refused); return 4; }
    std::printf("ok\n");
    return 0;
}
