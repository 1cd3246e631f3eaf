// Every descriptor of the split contraction that a batch or its problems keep
// names the tile width that the launches over it take: the batch's grouped
// launches one per layout, a problem's pairs (four descriptors) their own.
// Prints one line per failed check; exit status 1 on any.
#include <cstdio>
#include <map>
#include <vector>

#include "fake_cudart.h"
#include "tfde.h"
#include "tfde_tc.h"

using tfde::tc::Params;

int main() {
    const int sizes[3] = {16, 64, 128};   // 64-line tiles for the smaller ones alone, wider ones in the batch
    std::vector<tfde_params> prm;
    for (int k = 0; k < 12; ++k) {
        tfde_params p{};
        for (int a = 0; a < 3; ++a) {
            p.n[a] = sizes[k % 3];
            p.hi[a] = 1.0;
            p.delta[a] = 0.5;
            p.kp[a] = 1.0;
            p.km[a] = k % 2 ? 1.0 : 0.5;
        }
        p.dt = 0.1;
        prm.push_back(p);
    }
    std::map<void*, size_t> tables;   // device arrays of descriptors
    fake.on_copy = [&](void* dst, size_t bytes) {
        if (bytes && bytes % sizeof(Params) == 0) tables[dst] = bytes / sizeof(Params);
    };
    tfde_batch* B = nullptr;
    int failures = tfde_batch_create(prm.data(), (int)prm.size(), 20, nullptr, &B) != TFDE_OK;
    std::map<int, int> width;   // of the batch, by the x / other layout; every axis is alike here
    size_t seen = 0, pairs = 0;
    for (auto& t : tables) {
        if (!fake.live.count(t.first)) continue;
        for (size_t i = 0; i < t.second; ++i) {
            const Params& p = static_cast<const Params*>(t.first)[i];
            if (p.n != 16 && p.n != 64 && p.n != 128) continue;   // another array of the same length
            const int n[3] = {p.n, p.n, p.n}, axis = p.b_kmajor ? 0 : 1;
            int w;
            if (t.second == 4) {
                w = tfde::tc::tile_lines(tfde::tc::wide_tiles(n, axis), tfde::tc::TILES_PAIR);
                ++pairs;
            } else {
                if (!width[p.b_kmajor]) width[p.b_kmajor] = p.bn;
                w = width[p.b_kmajor];
            }
            ++seen;
            const long long per = p.b_kmajor ? w : w / 64, all = p.b_kmajor ? p.lines : p.nblocks;
            if (p.bn != w || p.ntiles != (all + per - 1) / per) {
                std::printf("n = %d, layout %d: %d lines and %lld tiles, launches take %d lines\n", p.n, p.b_kmajor,
                            p.bn, p.ntiles, w);
                ++failures;
            }
        }
    }
    if (pairs != 12 * 4 || seen < 12 * 20) ++failures;
    std::printf("%zu descriptors, widths %d and %d\n", seen, width[1], width[0]);
    tfde_batch_destroy(B);
    return failures != 0;
}
