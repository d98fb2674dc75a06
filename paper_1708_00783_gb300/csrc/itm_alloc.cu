// Sec. 4.2 allocation on the GPU, in three launches per frame:
//
//  1. alloc_enumerate  one thread per pixel walks the blocks crossed by its
//     segment d-mu .. d+mu (3D DDA), a warp per 8x4 pixel tile.  The blocks
//     are looked up in the brick table, those of a walk together.  A missing
//     block claims its bucket's request word with one 64-bit CAS (the paper's
//     per-entry allocation array, Sec. 4.2; equal keys of a warp grouped by
//     __match_any_sync); the winner of a bucket appends the bucket to the
//     request list, a block that finds its bucket claimed by another key goes
//     to the overflow list (warp-aggregated appends).
//  2. alloc_commit     one thread per requested bucket inserts its key
//     (Sec. 3.3 insertion).  Each bucket's chain has exactly one writer, so
//     chains are extended without locks; blocks and excess slots come from
//     prepopulated free lists through warp-aggregated atomic counters (the
//     paper's "atomic subtraction on a stack").  In a frame with an overflow
//     list the CTA that finishes last resolves it in rounds: look up, claim
//     the bucket, let winners insert, repeat with the losers.  The paper
//     leaves such intra-frame collisions for the next frame; resolving them
//     makes the allocated set the complete union over all pixels.
//  3. build_visible    every allocated block whose voxels can project into the
//     image with z > 0 and lie within the frame's depth range + mu is
//     appended to the visible list (Sec. 4.2, third part); eight lanes per
//     block, one per corner.  When the raycast will use the allocation pose,
//     the same pass also rasterises each block's search range.  It also enters
//     the blocks this allocation handed out (a few dozen in a usual frame) in
//     the brick table.
//
// The kernels run once through their code, so their length is dependent
// accesses and code size: the insertion in the enumeration's warps took the
// commit's launch out but cost a frame with thousands of new blocks more
// (131 us against 38 + 38 in the 2 mm hall), in the visible pass it made that
// pass 17 us instead of 8.
//
// Counts produced on the device are read by the next kernel from device
// memory (persistent grid-stride loops), so no host synchronisation and no
// allocation happen per frame.
#include "itm_ops.cuh"

namespace itm {

namespace {

// Also clears the search-range tiles of this frame (n_range_tiles of them;
// nothing reads them before the visible-list pass).
__global__ void __launch_bounds__(256) alloc_enumerate_kernel(SceneDev s, const float *__restrict__ depth,
                                                              Intr in, Mat34 T, float inv_b, int n_range_tiles,
                                                              const uint16_t *__restrict__ raw,
                                                              float *__restrict__ depth_out)
{
    __shared__ int depth_max[8];
    const int cta = blockIdx.y * gridDim.x + blockIdx.x, ctas = gridDim.x * gridDim.y;
    grid_dep_wait();  // the previous raycast may still read the range tiles
    FrameCounters *fc = &s.ctr->frame[__ldcg(&s.ctr->entered) & 1u];
    if (cta == 0 && threadIdx.x == 0) frame_begin(s);
    for (int i = cta * blockDim.x + threadIdx.x; i < n_range_tiles; i += ctas * blockDim.x) {
        s.range_min[i] = 0xffffffffu;
        s.range_max[i] = 0u;
    }
    const int dm = enumerate_tile<4>(s, depth, in, T, inv_b, blockIdx.x, blockIdx.y, raw, depth_out, fc);
    // one maximum per CTA: thousands on one word would wait for each other
    if ((threadIdx.x & 31) == 0) depth_max[threadIdx.x >> 5] = dm;
    __syncthreads();
    if (threadIdx.x == 0) {
        int m = 0;
        for (int w = 0; w < 8; ++w) m = max(m, depth_max[w]);
        if (m > 0) atomicMax(&fc->depth_max_bits, m);
    }
    grid_dep_launch();
}

__global__ void __launch_bounds__(256) alloc_commit_kernel(SceneDev s)
{
    __shared__ int is_last, remaining;
    grid_dep_wait();
    FrameCounters *fc = frame_set(s);
    const int n = min(__ldcg(&fc->n_req), s.nb), n_overflow = __ldcg(&fc->n_overflow);
    const int stride = gridDim.x * blockDim.x;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) commit_request(s, i);
    if (blockIdx.x == 0 && threadIdx.x == 0) frame_end(s);
    if (n_overflow > 0) {
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) is_last = atomicAdd(&fc->done, 1) == (int)gridDim.x - 1;
        __syncthreads();
        if (is_last) {
            __threadfence();
            overflow_scene(s, n_overflow, remaining);
        }
    }
    grid_dep_launch();
}

// RANGE: also fill the search range of a raycast from this pose (zc, tiles).
// The loop is uniform per CTA; a warp's four groups of eight lanes hold a
// block each.
template <bool RANGE>
__global__ void __launch_bounds__(256) build_visible_kernel(SceneDev s, Mat34 M, Intr in, float zc, int tiles_x,
                                                            int tiles_y)
{
    grid_dep_wait();
    const int n = min(__ldcg(&s.ctr->block_head), s.nv), head_before = __ldcg(&s.ctr->head_before);
    const float zfar = visible_zfar(s, frame_set(s));
    const int groups = gridDim.x * (blockDim.x >> 3);
    // a group's next block is fetched (two dependent loads) beside the test of this one
    int i = blockIdx.x * (blockDim.x >> 3) + (threadIdx.x >> 3);
    int ptr = i < n ? __ldg(&s.block_free[i]) : 0;
    short4 b = i < n ? __ldcg(&s.block_pos[ptr]) : make_short4(0, 0, 0, 0);
    for (int g0 = blockIdx.x * (blockDim.x >> 3); g0 < n; g0 += groups) {
        const int i_next = i + groups;
        const int ptr_next = i_next < n ? __ldg(&s.block_free[i_next]) : 0;
        const short4 b_next = i_next < n ? __ldcg(&s.block_pos[ptr_next]) : make_short4(0, 0, 0, 0);
        visible_8<RANGE>(s, M, in, zfar, i >= head_before, ptr, b, zc, tiles_x, tiles_y);
        i = i_next;
        ptr = ptr_next;
        b = b_next;
    }
    grid_dep_launch();
}

int sm_count()
{
    static int cached_sm = 0;
    if (!cached_sm) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&cached_sm, cudaDevAttrMultiProcessorCount, dev);
        if (cached_sm <= 0) cached_sm = 1;
    }
    return cached_sm;
}

int persistent_grid(int threads, const void *kernel)
{
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
    if (per_sm < 1) per_sm = 1;
    return sm_count() * per_sm;
}

}  // namespace

cudaError_t launch_allocate(const SceneDev &s, const float *depth, const Intr &in, const Mat34 &T_wc,
                            const Mat34 &M_d, bool with_range, cudaStream_t st, const uint16_t *raw, bool &half)
{
    half = false;
    const float inv_b = (float)(1.0 / (8.0 * (double)s.voxel_size));
    dim3 grid((in.W + 31) / 32, (in.H + 7) / 8);
    const int n_range_tiles = with_range ? ((in.W + 7) / 8) * ((in.H + 3) / 4) : 0;
    // with raw, depth is the output of the frame's conversion
    cudaError_t e = launch_pdl(alloc_enumerate_kernel, grid, dim3(256), 0, st, s, raw ? nullptr : depth, in, T_wc, inv_b,
                   n_range_tiles, raw, raw ? const_cast<float *>(depth) : nullptr);
    if (e != cudaSuccess) return e;
    static int g_commit = 0, g_visible = 0, g_visrange = 0;
    // one CTA per SM: a frame's requests (usually a few thousand) fit in one pass
    if (!g_commit) g_commit = sm_count();
    if (!g_visible) g_visible = persistent_grid(256, (const void *)build_visible_kernel<false>);
    if (!g_visrange) g_visrange = persistent_grid(256, (const void *)build_visible_kernel<true>);
    e = launch_pdl(alloc_commit_kernel, dim3(g_commit), dim3(256), 0, st, s);
    if (e != cudaSuccess) return e;
    if (with_range) {
        const int tx = (in.W + 7) / 8, ty = (in.H + 3) / 4;
        e = launch_pdl(build_visible_kernel<true>, dim3(g_visrange), dim3(256), 0, st, s, M_d, in, s.z_min - 1e-3f,
                       tx, ty);
    } else {
        e = launch_pdl(build_visible_kernel<false>, dim3(g_visible), dim3(256), 0, st, s, M_d, in, 0.0f, 1, 1);
    }
    half = e != cudaSuccess;
    return e;
}

int overflow_capacity() { return kOvfCapacity; }

}  // namespace itm
