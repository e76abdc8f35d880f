// Host-side rules of the wide full-range passes, for the tests: reads "shape W H D views paths
// truncation radius" lines and prints "G NQ" ("0 0" where the passes don't apply); "elements"
// checks the elements that a warp loads from a step's shared memory.
#include <cstdio>
#include <cstring>

#include "volume_layout.cuh"

namespace {

// Every byte of a step of 128 nq bytes is loaded exactly once, and no other.
bool elements_ok(int nq)
{
    const int step = 128 * nq, ne = (nq + 1) / 2;
    unsigned char seen[128 * 8 + 256] = {};
    for (int lane = 0; lane < 32; ++lane)
        for (int k = 0; k < ne; ++k) {
            if (!mpv::wide_elem(nq, lane, k)) continue;
            const int at = 8 * (lane + 32 * k);
            if (at + 8 > step) return false;
            for (int b = 0; b < 8; ++b) ++seen[at + b];
        }
    for (int b = 0; b < step; ++b)
        if (seen[b] != 1) return false;
    return true;
}

}  // namespace

int main()
{
    char word[16];
    while (std::scanf("%15s", word) == 1) {
        if (!std::strcmp(word, "elements")) {
            for (int nq = 3; nq <= 8; ++nq) std::printf("%d %d\n", nq, (int)elements_ok(nq));
        } else {
            mpv::LevelArgs a{};
            if (std::scanf("%d %d %d %d %d %d %d", &a.W, &a.H, &a.D, &a.nviews, &a.npaths, &a.trunc,
                           &a.radius) != 7)
                return 1;
            a.Dw = a.D;
            a.Dws = (a.Dw + 15) / 16 * 16;
            int G = 0, NQ = 0;
            if (!mpv::wide_shape(a, G, NQ)) G = NQ = 0;
            std::printf("%d %d\n", G, NQ);
        }
    }
    return 0;
}
