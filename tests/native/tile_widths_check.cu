// Lines per tile along each axis of the grids given (n1 n2 n3 ...), one line of
// nine numbers per grid: the split, hi-only and paired passes.
#include <cstdio>
#include <cstdlib>

#include "tfde_tc.h"

int main(int argc, char** argv) {
    for (int i = 1; i + 2 < argc; i += 3) {
        const int n[3] = {std::atoi(argv[i]), std::atoi(argv[i + 1]), std::atoi(argv[i + 2])};
        for (int kind = 0; kind < tfde::tc::TILES_KINDS; ++kind)
            for (int a = 0; a < 3; ++a)
                std::printf("%d ", tfde::tc::tile_lines(tfde::tc::wide_tiles(n, a), kind));
        std::printf("\n");
    }
    return 0;
}
