// Host check of the brick table's addressing (itm_internal.cuh): blocks entered
// by brick_share and brick_place into a table of the smallest size, and every
// block's 2x2x2 neighbourhood read back at the fixed offsets of brick_local.
#include <stdio.h>

#include <map>
#include <set>
#include <tuple>
#include <vector>

#include "itm_internal.cuh"

using namespace itm;
using Block = std::tuple<int, int, int>;

int main()
{
    uint64_t r = 88172645463325252ull;  // xorshift64 (Marsaglia 2003)
    auto next = [&]() { r ^= r << 13; r ^= r >> 7; r ^= r << 17; return r; };
    const uint32_t mask = kBrickMin - 1;
    for (int origin : {0, -4, -32768, 32767 - 23, 8 * 512 - 12}) {
        // a dense random half of 24^3 blocks, at the ends of the range and across brick edges
        std::map<Block, int> have;
        for (int i = 0; i < 24 * 24 * 24 / 2; ++i) {
            const uint64_t v = next();
            have[{origin + (int)(v % 24), (int)((v >> 16) % 24) - 12, -32768 + (int)((v >> 32) % 24)}] = i;
        }
        std::vector<unsigned long long> owner(kBrickMin, 0);
        std::vector<int> cell((size_t)kBrickMin * kBrickCells, -1);
        std::set<uint32_t> shared;
        for (auto &e : have)
            for (int c = 0; c < 8; ++c) {
                int X, Y, Z, local;
                if (!brick_share(std::get<0>(e.first), std::get<1>(e.first), std::get<2>(e.first), c, X, Y, Z, local)) continue;
                if (local < 0 || local >= kBrickCells) return printf("cell %d\n", local), 1;
                const uint32_t p = brick_place(X, Y, Z, mask);
                if (p > mask) return printf("place\n"), 1;
                if (!owner[p]) owner[p] = brick_key(X, Y, Z);
                if (owner[p] == brick_key(X, Y, Z)) cell[(size_t)p * kBrickCells + local] = e.second;
                else shared.insert(p);
            }
        long long checked = 0;
        for (int dx = -2; dx < 26; ++dx)
            for (int dy = -14; dy < 14; ++dy)
                for (int dz = -2; dz < 26; ++dz) {
                    const int b[3] = {origin + dx, dy, -32768 + dz};
                    if (b[0] < -32768 || b[0] > 32766 || b[2] < -32768) continue;
                    const int X = b[0] >> 3, Y = b[1] >> 3, Z = b[2] >> 3;
                    const uint32_t p = brick_place(X, Y, Z, mask);
                    for (int k = 0; k < 8; ++k) {
                        auto it = have.find({b[0] + (k & 1), b[1] + ((k >> 1) & 1), b[2] + (k >> 2)});
                        const int want = it == have.end() ? -1 : it->second;
                        int got;
                        if (owner[p] == brick_key(X, Y, Z))
                            got = cell[(size_t)p * kBrickCells + brick_local((b[0] & 7) + (k & 1), (b[1] & 7) + ((k >> 1) & 1), (b[2] & 7) + (k >> 2))];
                        else if (shared.count(p))
                            continue;  // the hash table answers
                        else
                            got = -1;
                        if (got != want) return printf("(%d %d %d) + %d: %d, not %d\n", b[0], b[1], b[2], k, got, want), 1;
                        ++checked;
                    }
                }
        if (checked < 50000) return printf("only %lld checked\n", checked), 1;
    }
    // a brick's owner word tells bricks apart over the whole range, and is never 0 nor marked shared
    for (int i = 0; i < 2000000; ++i) {
        const uint64_t v = next();
        const int X = (int)(int16_t)(v & 0xffff) >> 3, Y = (int)(int16_t)((v >> 16) & 0xffff) >> 3, Z = (int)(int16_t)((v >> 32) & 0xffff) >> 3;
        const unsigned long long k = brick_key(X, Y, Z);
        if (!(k & kBrickValid) || (k & kBrickShared) || (int)(int16_t)(k & 0xffff) != X || (int)(int16_t)((k >> 16) & 0xffff) != Y ||
            (int)(int16_t)((k >> 32) & 0xffff) != Z)
            return printf("key\n"), 1;
    }
    printf("ok\n");
    return 0;
}
