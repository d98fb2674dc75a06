// GPU check of the march's stop (itm::march_stops): the lanes of a warp must
// decide alike while other warps append to the list whose length decides.
// Every lane writes its decisions after 16, 32 and 48 iterations; the lanes come
// to each of them apart from one another (work that depends on the lane before
// it), and every warp adds to the length in between.  Loops are counted, so
// every warp ends.  Prints how often lanes disagreed, and how many warps stopped
// and went on (both must occur, or nothing was decided).
#include <cstdio>
#include <vector>

#include "itm_ops.cuh"

constexpr int kWarps = 1 << 15, kRoom = 1 << 14;

__global__ void check(int32_t *len, unsigned char *out, unsigned *sink)
{
    const int lane = threadIdx.x & 31, warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    unsigned x = lane + 1;
    for (int k = 1; k <= 3; ++k) {
        for (int i = 0; i < (lane * 37 + warp) % 61; ++i) x = x * 1664525u + 1013904223u;
        if (lane == (warp & 31)) atomicAdd(len, 1);
        out[(k - 1) * 32 * kWarps + 32 * warp + lane] = itm::march_stops(len, 16 * k, kRoom);
    }
    if (x == 0u) *sink = x;
}

int main()
{
    int32_t *len = nullptr;
    unsigned char *out = nullptr;
    unsigned *sink = nullptr;
    std::vector<unsigned char> h(3 * 32 * kWarps);
    if (cudaMalloc(&len, 4) != cudaSuccess || cudaMalloc(&sink, 4) != cudaSuccess ||
        cudaMalloc(&out, h.size()) != cudaSuccess)
        return 2;
    cudaMemset(len, 0, 4);
    check<<<kWarps / 8, 256>>>(len, out, sink);
    if (cudaDeviceSynchronize() != cudaSuccess) return 3;
    cudaMemcpy(h.data(), out, h.size(), cudaMemcpyDeviceToHost);
    int apart = 0, stopped = 0, went_on = 0;
    for (int w = 0; w < 3 * kWarps; ++w) {
        int c = 0;
        for (int l = 0; l < 32; ++l) c += h[32 * (size_t)w + l];
        apart += c != 0 && c != 32;
        stopped += c == 32;
        went_on += c == 0;
    }
    printf("%d %d %d\n", apart, stopped, went_on);
    return 0;
}
