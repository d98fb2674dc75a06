// GPU check of the brick table's entry and removal (itm_internal.cuh): a camera
// that travels.  Clusters of blocks enter and leave in the order of a queue, far
// more bricks in all than the smallest table has places, so that bricks meet at
// places all the time, as owner and as the one that comes later, and leave in
// either order.  After every change the table is read back: each block present
// is in its own brick's cells or its brick's place is marked; a place is marked
// only while a block is not in its cells, and taken only while a block counts on
// it.  At the end nothing is left.
#include <cstdio>
#include <deque>
#include <map>
#include <set>
#include <tuple>
#include <vector>

#include "itm_internal.cuh"

using namespace itm;
using Block = std::tuple<int, int, int>;

__global__ void change(SceneDev s, const short4 *b, int n, bool put)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= 8 * n) return;
    const short4 v = b[j >> 3];
    if (put) brick_put(s, v.x, v.y, v.z, (int)(unsigned short)v.w, j & 7);
    else brick_take(s, v.x, v.y, v.z, j & 7);
}

int main()
{
    uint64_t r = 88172645463325252ull;  // xorshift64 (Marsaglia 2003)
    auto next = [&]() { r ^= r << 13; r ^= r >> 7; r ^= r << 17; return r; };
    SceneDev s;
    memset(&s, 0, sizeof(s));
    s.brick_mask = kBrickMin - 1;
    s.nv = 1 << 16;
    short4 *dev = nullptr;
    const size_t cells = (size_t)kBrickMin * kBrickCells;
    const size_t count_bytes = sizeof(*s.brick_count) * kBrickMin;
    if (cudaMalloc(&s.brick_owner, 8 * kBrickMin) || cudaMalloc(&s.brick_count, count_bytes) ||
        cudaMalloc(&s.brick_cell, 4 * cells) || cudaMalloc(&dev, sizeof(short4) * 4096))
        return 2;
    cudaMemset(s.brick_owner, 0, 8 * kBrickMin);
    cudaMemset(s.brick_count, 0, count_bytes);
    cudaMemset(s.brick_cell, 0xff, 4 * cells);
    std::vector<unsigned long long> owner(kBrickMin);
    std::vector<int> cell(cells);
    std::map<Block, int> have;
    std::deque<std::vector<short4>> present;
    int id = 0, shared_seen = 0;
    auto apply = [&](const std::vector<short4> &v, bool put) {
        cudaMemcpy(dev, v.data(), sizeof(short4) * v.size(), cudaMemcpyHostToDevice);
        change<<<(8 * (int)v.size() + 255) / 256, 256>>>(s, dev, (int)v.size(), put);
        for (auto &b : v)
            if (put) have[{b.x, b.y, b.z}] = (int)(unsigned short)b.w;
            else have.erase({b.x, b.y, b.z});
    };
    auto look = [&]() {
        if (cudaMemcpy(owner.data(), s.brick_owner, 8 * kBrickMin, cudaMemcpyDeviceToHost) != cudaSuccess ||
            cudaMemcpy(cell.data(), s.brick_cell, 4 * cells, cudaMemcpyDeviceToHost) != cudaSuccess)
            return printf("cuda\n"), false;
        std::set<uint32_t> used, other;
        size_t in_cells = 0;
        for (auto &e : have)
            for (int c = 0; c < 8; ++c) {
                int X, Y, Z, local;
                if (!brick_share(std::get<0>(e.first), std::get<1>(e.first), std::get<2>(e.first), c, X, Y, Z, local)) continue;
                const uint32_t p = brick_place(X, Y, Z, s.brick_mask);
                used.insert(p);
                if ((owner[p] & ~kBrickShared) == brick_key(X, Y, Z)) {
                    if (cell[(size_t)p * kBrickCells + local] != e.second) return printf("cell of place %u\n", p), false;
                    ++in_cells;
                } else {
                    other.insert(p);
                }
            }
        size_t full = 0;
        for (int v : cell) full += v >= 0;
        if (full != in_cells) return printf("%zu cells, not %zu\n", full, in_cells), false;
        for (uint32_t p = 0; p < (uint32_t)kBrickMin; ++p) {
            if ((owner[p] != 0) != (used.count(p) != 0)) return printf("place %u taken for nobody, or not taken\n", p), false;
            if (((owner[p] & kBrickShared) != 0) != (other.count(p) != 0)) return printf("mark of place %u\n", p), false;
        }
        shared_seen += (int)other.size();
        return true;
    };
    for (int step = 0; step < 60; ++step) {
        // a cluster of new blocks in 40 bricks around a point of the walk, with bricks whose places others have
        std::vector<short4> v;
        std::set<Block> mine;
        for (int k = 0; k < 1500; ++k) {
            const uint64_t a = next();
            const int brick = (int)(a % 40), far = (a >> 8) % 4 == 0 ? 1 : 0;
            const int bx = 8 * (step * 5 + brick % 5 + 43 * far) + (int)((a >> 16) % 8);
            const int by = 8 * (brick / 5 + far) + (int)((a >> 24) % 8), bz = -8 * 4 * far + (int)((a >> 32) % 8);
            if (have.count({bx, by, bz}) || !mine.insert({bx, by, bz}).second) continue;
            v.push_back(make_short4((short)bx, (short)by, (short)bz, (short)(id++ & 0x7fff)));
        }
        apply(v, true);
        present.push_back(v);
        if (!look()) return 1;
        if (present.size() > 12) {  // the oldest, or one in the middle, leaves
            const size_t at = step & 1 ? 0 : present.size() / 2;
            apply(present[at], false);
            present.erase(present.begin() + at);
            if (!look()) return 1;
        }
    }
    while (!present.empty()) {
        const size_t at = next() % present.size();
        apply(present[at], false);
        present.erase(present.begin() + at);
        if (!look()) return 1;
    }
    std::vector<unsigned char> count(count_bytes);
    cudaMemcpy(count.data(), s.brick_count, count_bytes, cudaMemcpyDeviceToHost);
    for (unsigned char c : count)
        if (c) return printf("counts left\n"), 1;
    if (shared_seen < 500) return printf("only %d shared places\n", shared_seen), 1;
    printf("ok\n");
    return 0;
}
