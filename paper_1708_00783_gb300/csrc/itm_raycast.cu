// Sec. 4.4 raycast: one thread per pixel, a warp covering an 8x4 pixel tile.
//
// The march is the state machine of Sec. 4.4 (SEARCH_BLOCK_COARSE ->
// SEARCH_BLOCK_FINE -> SEARCH_SURFACE -> BEHIND_SURFACE, or WRONG_SIDE), with
// these step rules (the paper names the states, not the constants):
//   ray o + t dir, dir = R ((u-cx)/fx, (v-cy)/fy, 1): t is z-depth;
//   len = |((u-cx)/fx, (v-cy)/fy, 1)|, tB = 8s/len, tmu = mu/len, ts = s/len;
//   t starts at z_min; the ray misses when t > z_max or after
//   4 (z_max - z_min)/s + 64 iterations;
//   "the block at p" is the block of the nearest voxel floor(p/s + 1/2);
//   COARSE : unallocated -> t += tB; allocated -> t -= tB, FINE;
//   FINE   : unallocated -> t += tmu; allocated -> F (trilinear) <= 0 ->
//            WRONG_SIDE, else SURFACE at the same t;
//   SURFACE: unallocated -> COARSE; F <= 0 -> BEHIND; else
//            t += max(F tmu, ts);
//   BEHIND : twice t += F(t) tmu (trilinear), hit = o + t dir.
// The TSDF field outside allocated blocks is the default voxel value 1
// (Sec. 3.3 retrieval of a missing block).  Normals: central differences of
// the trilinear field at +-1 voxel per axis, emitted only when all 48 voxels
// read are allocated and observed (weight > 0).
//
// Search range (Sec. 4.4, second half): before the march, every allocated
// block is projected into the image and each 8x4-pixel tile (the pixels of
// one warp) records the nearest and farthest camera depth of the blocks that
// cover it.  A block's extent here is its query region -- the points whose
// nearest voxel lies in it, [8b - 1/2, 8b + 15/2] voxels per axis -- clipped
// to z >= z_min, grown by a small margin.  The march uses the range without
// changing its result: coarse steps in front of the tile's nearest depth are
// replayed as additions (no hash probes, the same t sequence and iteration
// count), and a ray in COARSE or FINE beyond the tile's farthest depth can
// only miss.  The paper renders 16x16-pixel fragments with per-pixel atomic
// min/max; here the fragment is the warp's tile and the atomics go to one
// word per tile.
//
// The blocks of a sample -- the nearest voxel's, which decides whether the
// space is allocated, and those of its trilinear stencil -- come from the
// brick table (itm_internal.cuh) with loads that are issued together, so a
// step has two dependent loads: cells, voxels.  Every arithmetic step of the
// march uses IEEE round-to-nearest operations in a fixed order.
#include "itm_ops.cuh"

namespace itm {

namespace {

// One warp takes 32 allocated blocks and rasterises their tile rectangles.
__global__ void __launch_bounds__(256) range_kernel(SceneDev s, Mat34 M, Intr in, float zc, int tiles_x,
                                                    int tiles_y, uint32_t *__restrict__ rmin,
                                                    uint32_t *__restrict__ rmax)
{
    const int n = min(__ldcg(&s.ctr->block_head), s.nv);
    const int lane = threadIdx.x & 31;
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (int base = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < n; base += warps * 32) {
        const int i = base + lane;
        TileRange r{0, -1, 0, -1, 0.f, 0.f};
        bool ok = false;
        if (i < n) {
            const int ptr = __ldg(&s.block_free[i]);
            const short4 b = __ldg(&s.block_pos[ptr]);
            if (b.w) ok = block_tile_range(b, M, in, s.voxel_size, zc, tiles_x, tiles_y, r);
        }
        range_rasterize(ok, r, tiles_x, rmin, rmax);
    }
}

// Persistent raycast, first phase (the march): each warp takes the next 8x4
// tile from a device counter until none is left, so warps that finish early
// pick up more work.  Rays that are not through after a while go to the slow
// list (room: the list's length up to which warps give rays up early, see
// march_warp; 0: no list).
//
// Most rays end within 6 to 10 iterations, but those that skim a wall or leave
// the mapped part take 80 (room) to 190 (2 mm hall), each two dependent memory
// accesses long (0.7 us): marched to their end in their own tiles they were
// most of the raycast (56 to 80 us of it in the room, 28 to 36 us at 160x120),
// with the chip idle.  Now they continue in the second kernel with four lanes a
// ray (march_slow), beside the finish of the others.
template <int MODE>
__global__ void __launch_bounds__(256, 4) raycast_march_kernel(SceneDev s, Intr in, Mat34 T, float4 *__restrict__ vtx,
                                                               int max_iter, float tB_m, float inv_sv,
                                                               const uint32_t *__restrict__ rmin,
                                                               const uint32_t *__restrict__ rmax, int tiles_x,
                                                               int n_tiles, int room)
{
    const int lane = threadIdx.x & 31;
    grid_dep_wait();
    const uint32_t entered = __ldcg(&s.ray_ctr->entered);
    auto *c = &s.ray_ctr->set[entered & 1u];
    if (blockIdx.x == 0 && threadIdx.x == 0) s.ray_ctr->begun = entered + 1u;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(&c->next, 1);
        t = __shfl_sync(kFull, t, 0);
        if (t >= n_tiles) break;
        raycast_march_tile<MODE>(s, in, T, vtx, max_iter, tB_m, inv_sv, rmin, rmax, tiles_x, t % tiles_x, t / tiles_x,
                                 room > 0 ? &c->n_slow : nullptr, room);
    }
    grid_dep_launch();
}

// Second phase: refinement, hit point and normal of the rays that ended (two
// kernels with smaller code each measured faster than the one that did both),
// beside the slow rays to their end.  The first slow_ctas CTAs take the groups
// of the slow list, the first warp of each before the second, ...: of eight
// rays while there are warps for them, of up to 32 beyond that, where filled
// finish passes count for more than latency.
template <int MODE>
__global__ void __launch_bounds__(256, 4) raycast_finish_kernel(SceneDev s, Intr in, Mat34 T, float4 *vtx, float4 *nrm,
                                                                int max_iter, float tB_m, float inv_sv,
                                                                const uint32_t *__restrict__ rmin,
                                                                const uint32_t *__restrict__ rmax, int tiles_x,
                                                                int tiles, int slow_ctas)
{
    grid_dep_wait();
    RayCounters *c = s.ray_ctr;
    const uint32_t begun = __ldcg(&c->begun);
    const int warp = threadIdx.x >> 5, cta = (int)blockIdx.x - slow_ctas;
    if (cta == 0 && threadIdx.x == 0) {
        // the next raycast's set; nothing reads it before that
        c->set[begun & 1u].next = c->set[begun & 1u].n_slow = 0;
        c->entered = begun;
    }
    const int n_slow = cta < 0 ? min(__ldcg(&c->set[(begun - 1u) & 1u].n_slow), kSlowMax) : 0;
    const int rounds = n_slow > 0 ? min((n_slow - 1) / (64 * slow_ctas) + 1, 4) : 1;
    for (int g = cta < 0 ? (int)blockIdx.x + slow_ctas * warp : cta * 8 + warp;
         cta < 0 ? g * 8 * rounds < n_slow : g < tiles; g += cta < 0 ? 8 * slow_ctas : tiles) {
        const EndedRay e = cta < 0 ? raycast_slow_rays<MODE>(s, in, T, vtx, max_iter, tB_m, inv_sv, rmin, rmax, tiles_x,
                                                             g * 8 * rounds, rounds, n_slow)
                                   : raycast_tile_rays(in, vtx, g % tiles_x, g / tiles_x);
        finish_ray<MODE>(s, in, T, tB_m, inv_sv, e, vtx, nrm);
    }
}

// Without a search range (images beyond the range tiles): the whole raycast
// of one pixel per thread.
template <int MODE>
__global__ void __launch_bounds__(256) raycast_kernel(SceneDev s, Intr in, Mat34 T, float4 *__restrict__ vtx,
                                                      float4 *__restrict__ nrm, int max_iter, float tB_m, float inv_sv)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u = (blockIdx.x * 4 + (warp & 3)) * 8 + (lane & 7), v = (blockIdx.y * 2 + (warp >> 2)) * 4 + (lane >> 3);
    const bool inside = u < in.W && v < in.H;
    const Ray r = make_ray(s, in, T, tB_m, u, v);
    float t;
    int state, it;
    march_warp<MODE, false>(s, r, inside, max_iter, inv_sv, nullptr, nullptr, 0, nullptr, 0, t, state, it);
    if (inside) finish_pixel<MODE>(s, r, state == BEHIND, t, inv_sv, (size_t)v * in.W + u, vtx, nrm);
}

int range_grid()
{
    static int g = 0;
    if (!g) {
        int dev = 0, sms = 1;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        g = sms * 4;
    }
    return g;
}

}  // namespace

bool range_fits(const Intr &in) { return in.W <= kRangeMaxW && in.H <= kRangeMaxH; }

cudaError_t launch_raycast_range(const SceneDev &s, const Intr &in, const Mat34 &M_d, uint32_t *rmin, uint32_t *rmax,
                                 cudaStream_t st)
{
    const int tx = (in.W + 7) / 8, ty = (in.H + 3) / 4;
    cudaError_t e = cudaMemsetAsync(rmin, 0xff, sizeof(uint32_t) * (size_t)tx * ty, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(rmax, 0, sizeof(uint32_t) * (size_t)tx * ty, st);
    if (e != cudaSuccess) return e;
    const float zc = s.z_min - 1e-3f;
    range_kernel<<<range_grid(), 256, 0, st>>>(s, M_d, in, zc, tx, ty, rmin, rmax);
    return cudaGetLastError();
}

cudaError_t launch_raycast(const SceneDev &s, const Intr &in, const Mat34 &T_wc, const Mat34 &M_d, float4 *vtx,
                           float4 *nrm, bool range_ready, cudaStream_t st, bool &half)
{
    half = false;
    // host-side constants with the same float operations as the oracle
    volatile float span = s.z_max - s.z_min;
    volatile float four_span = 4.0f * span;
    volatile float ratio = four_span / s.voxel_size;
    const int max_iter = (int)ratio + 64;
    volatile float tB_v = 8.0f * s.voxel_size;
    const float tB_m = tB_v;
    const float inv_sv = (float)(1.0 / (double)s.voxel_size);  // voxel coordinates: p * (1/s), 1/s rounded once
    dim3 grid((in.W + 31) / 32, (in.H + 7) / 8);
    const int tx = (in.W + 7) / 8, ty = (in.H + 3) / 4;
    if (range_fits(in)) {
        // the allocation of this frame may have filled the range already
        cudaError_t e = range_ready ? cudaSuccess : launch_raycast_range(s, in, M_d, s.range_min, s.range_max, st);
        if (e != cudaSuccess) return e;
        static int g_dyn[2] = {0, 0}, sms = 1;
        const int mode = s.weight_mode ? 1 : 0;
        if (!g_dyn[mode]) {
            int dev = 0, per = 1;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                &per, mode ? (const void *)raycast_march_kernel<1> : (const void *)raycast_march_kernel<0>, 256, 0);
            g_dyn[mode] = sms * (per > 0 ? per : 1);
        }
        const int n_tiles = tx * ty, ctas = (n_tiles + 7) / 8;
        const int g = g_dyn[mode] < ctas ? g_dyn[mode] : ctas;
        // CTAs for the slow rays, three per SM (of four that fit beside each
        // other); none for an image that could have more than the list holds.
        // room, the list's length up to which warps give rays up early: as many
        // as these CTAs take at once, but at most 48 per SM.  Whole frames in
        // us, each pair on the same inputs, this setting first; 160x120, the
        // 640x480 room, the 2 mm hall, a third of whose rays are slow:
        //   one CTA per SM for slow rays  48.5 : 48.5, 112.7 : 112.0, 522 : 572
        //   room up to all 192 per SM     42.7 : 42.7, 102.4 : 102.3, 600 : 629
        //   room 1 (48 iterations first)  54.3 : 59.7, 148.6 : 150.4, 637 : 641
        const int slow_ctas = (long long)in.W * in.H > kSlowMax ? 0 : 3 * sms < ctas ? 3 * sms : ctas;
        const uint32_t *rmin = s.range_min, *rmax = s.range_max;
        const auto march = mode ? raycast_march_kernel<1> : raycast_march_kernel<0>;
        const auto finish = mode ? raycast_finish_kernel<1> : raycast_finish_kernel<0>;
        e = launch_pdl(march, dim3(g), dim3(256), 0, st, s, in, T_wc, vtx, max_iter, tB_m, inv_sv, rmin, rmax, tx,
                       n_tiles, 64 * slow_ctas < 48 * sms ? 64 * slow_ctas : 48 * sms);
        if (e != cudaSuccess) return e;
        e = launch_pdl(finish, dim3(slow_ctas + ctas), dim3(256), 0, st, s, in, T_wc, vtx, nrm, max_iter, tB_m,
                       inv_sv, rmin, rmax, tx, n_tiles, slow_ctas);
        half = e != cudaSuccess;
        return e;
    }
    const auto whole = s.weight_mode ? raycast_kernel<1> : raycast_kernel<0>;
    whole<<<grid, 256, 0, st>>>(s, in, T_wc, vtx, nrm, max_iter, tB_m, inv_sv);
    return cudaGetLastError();
}

// Parts' raycasts of a split scene merged per pixel: the hit nearest to the
// camera (camera depth = row 2 of M_d applied to the vertex, each operation
// rounded on its own), equal depths to the lower part; no hit: zeros.
__global__ void __launch_bounds__(256) merge_kernel(const float4 *__restrict__ vtx, const float4 *__restrict__ nrm,
                                                    int parts, long long npix, Mat34 M, float4 *__restrict__ vo,
                                                    float4 *__restrict__ no)
{
    for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < npix;
         o += (long long)gridDim.x * blockDim.x) {
        int best = -1;
        float best_z = 0.0f;
        for (int k = 0; k < parts; ++k) {
            const float4 V = __ldg(&vtx[(size_t)k * npix + o]);
            if (!(V.w > 0.0f)) continue;
            const float z = row_apply(&M.m[8], V.x, V.y, V.z);
            if (best < 0 || z < best_z) {
                best = k;
                best_z = z;
            }
        }
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        vo[o] = best < 0 ? zero : __ldg(&vtx[(size_t)best * npix + o]);
        no[o] = best < 0 ? zero : __ldg(&nrm[(size_t)best * npix + o]);
    }
}

cudaError_t launch_raycast_merge(const float4 *vtx, const float4 *nrm, int parts, long long npix, const Mat34 &M_d,
                                 float4 *vo, float4 *no, cudaStream_t st)
{
    if (npix <= 0) return cudaSuccess;
    const long long blocks = (npix + 255) / 256;
    merge_kernel<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(vtx, nrm, parts, npix, M_d, vo, no);
    return cudaGetLastError();
}

}  // namespace itm
