// Host-side check of the forward kernel's work items (tile_pair in s2a_params.h): every query tile of a
// group is in exactly one pair (or is a single item of its own), with exactly the key tiles it attends,
// heaviest of a range first.
// Prints "ok" and returns 0, or says what failed.
#include <cstdio>
#include <vector>

#include "s2a_params.h"

using namespace s2a;

int main() {
    for (int G : {8, 128, 200, 256, 384, 640, 1000, 1024})
        for (int groups : {1, 2, 3})
            for (int shift : {0, G / 2, -(G / 4) * 4 / 2 * 2, 4})
                for (int variant : {0, 1, 2}) {
                    if (G * groups < 128 || shift % 4 != 0) continue;
                    Geometry geo{};
                    geo.B = 1, geo.N = G * groups, geo.H = 2, geo.Hkv = 2, geo.G = G, geo.groups = groups, geo.shift = shift;
                    geo.leak_free = variant == 1, geo.swap_wrapped = variant == 2;
                    for (int g = 0; g < groups; ++g) {
                      for (bool single : {false, true}) {
                        const GroupLayout L = group_layout(geo, shift, g);
                        std::vector<int> seen(L.nTiles, 0);
                        int prev = 1 << 30;
                        for (int r = 0; r < pairs_of_group(L, single); ++r) {
                            const TilePair t = tile_pair(L, r, single);
                            if (t.n[1] < 1 || t.n[0] != (single ? 0 : t.n[1] - 1) || t.i[0] != t.i[1] - 1) return std::printf("FAIL shape %d %d %d\n", G, g, r), 1;
                            const bool new_range = L.cut > 0 && t.i[1] == L.cut - 1;
                            if (t.n[1] > prev && !new_range) return std::printf("FAIL order %d %d %d\n", G, g, r), 1;
                            prev = t.n[1];
                            for (int x = 0; x < 2; ++x) {
                                if (t.n[x] == 0) continue;
                                if (t.i[x] < 0 || t.i[x] >= L.nTiles || seen[t.i[x]]++) return std::printf("FAIL cover %d %d %d\n", G, g, r), 1;
                                if (t.j_begin != first_key_tile(L, t.i[x]) || t.n[x] != t.i[x] + 1 - t.j_begin)
                                    return std::printf("FAIL keys %d %d %d\n", G, g, r), 1;
                            }
                        }
                        for (int s : seen)
                            if (s != 1) return std::printf("FAIL tile left out %d %d\n", G, g), 1;
                      }
                    }
                }
    std::printf("ok\n");
    return 0;
}
