// Sec. 4 mesh generation by Marching Cubes (Lorensen & Cline 1987) over the
// zero level set of the TSDF (inside: F < 0).
//
// Cells are the voxel cubes g + {0,1}^3 whose eight corners are allocated
// and observed (weight > 0); cells that straddle blocks read the neighbour
// blocks.  The triangulation of each of the 256 inside/outside corner
// patterns is built once on the host (build_table): the crossings of the
// sign-changing edges are linked face by face, a face with two diagonal
// inside corners separating them (a rule that depends only on the face, so
// neighbouring cells agree and the mesh is closed); the links form loops,
// each oriented by a geometric test and fanned from its crossing on the
// lowest-numbered edge, counter-clockwise seen from outside (F > 0).
// Edge 4 a + o1 + 2 o2 runs along axis a from the corner whose other two
// coordinates are o1 (lower axis) and o2 (higher axis).  A crossing sits at
// t = F_a / (F_a - F_b) from the edge's lower corner: coordinate
// (g + t) * s along the edge's axis, g * s on the others, each operation
// rounded on its own (built with -fmad=false).
//
// One warp per allocated block (persistent grid-stride): the block's 9x9x9
// voxel neighbourhood (the block and the +1 layers of up to seven neighbours)
// is staged in the warp's part of shared memory; the cells' patterns are read
// off bit masks, one atomic reserves the block's triangles, and the lanes
// write the vertices side by side.
#include "itm_ops.cuh"

namespace itm {

namespace {

struct McTable {
    uint8_t count[256];
    uint8_t edge[256][15];  // 3 edge indices per triangle
};

// Corner k of a cell sits at (k & 1, (k >> 1) & 1, k >> 2); edge e = 4 a + o1 +
// 2 o2 runs along axis a from its lower corner.
int edge_lo(int e)
{
    const int a = e >> 2, o1 = e & 1, o2 = (e >> 1) & 1;
    const int ua = a == 0 ? 1 : 0, va = a == 2 ? 1 : 2;  // the other axes, lower first
    return (o1 << ua) | (o2 << va);
}
int edge_hi(int e) { return edge_lo(e) | (1 << (e >> 2)); }

// The case table, derived as a graph: the crossings (edges with one inside and
// one outside corner) are its nodes, and each face of the cube links the
// crossings on its four sides -- two crossings are linked to each other, four
// (two inside corners on a diagonal) are linked in pairs around each inside
// corner, which separates the diagonal corners (a choice that depends on the
// face alone, so the two cells sharing the face agree and the mesh is closed).
// Every crossing has one link on each of its two faces, so the links form
// loops.  A loop is oriented by geometry: on the face of its first link, seen
// from outside the cube, the inside corner of the first crossing must lie to
// the left of the step from the first crossing's midpoint to the second's
// (inside on the left: the loop runs clockwise seen from the F > 0 side).  It
// is then fanned from its crossing on the lowest-numbered edge, each triangle
// (first, next, current) so that it faces the F > 0 side.
void build_table(McTable &T)
{
    memset(&T, 0, sizeof(T));
    for (int cfg = 0; cfg < 256; ++cfg) {
        auto inside = [cfg](int k) { return ((cfg >> k) & 1) != 0; };
        int link[12][2], face_of[12][2], nl[12] = {0};
        for (int f = 0; f < 6; ++f) {
            const int a = f >> 1, side = f & 1;
            int sides[4], ns = 0;
            for (int e = 0; e < 12; ++e) {
                if ((e >> 2) == a) continue;  // an edge along the face normal is not on the face
                const int lo = edge_lo(e), hi = edge_hi(e);
                if (((lo >> a) & 1) != side) continue;
                if (inside(lo) != inside(hi)) sides[ns++] = e;
            }
            int pairs[2][2], np = 0;
            if (ns == 2) {
                pairs[np][0] = sides[0];
                pairs[np++][1] = sides[1];
            } else if (ns == 4) {
                // pair the two crossings at each inside corner of the face
                for (int i = 0; i < 4; ++i)
                    for (int j = i + 1; j < 4; ++j) {
                        const int c0[2] = {edge_lo(sides[i]), edge_hi(sides[i])};
                        const int c1[2] = {edge_lo(sides[j]), edge_hi(sides[j])};
                        for (int x = 0; x < 2; ++x)
                            for (int y = 0; y < 2; ++y)
                                if (c0[x] == c1[y] && inside(c0[x]) && np < 2) {
                                    pairs[np][0] = sides[i];
                                    pairs[np++][1] = sides[j];
                                }
                    }
            }
            for (int q = 0; q < np; ++q)
                for (int h = 0; h < 2; ++h) {
                    const int e = pairs[q][h];
                    link[e][nl[e]] = pairs[q][1 - h];
                    face_of[e][nl[e]++] = f;
                }
        }
        bool seen[12] = {false};
        int nt = 0;
        for (int e0 = 0; e0 < 12; ++e0) {
            if (nl[e0] != 2 || seen[e0]) continue;
            int loop[12], n = 0, prev = -1, cur = e0;
            do {  // follow the links: each crossing has two, leave by the one not arrived on
                seen[cur] = true;
                loop[n++] = cur;
                const int nxt = link[cur][0] == prev ? link[cur][1] : link[cur][0];
                prev = cur;
                cur = nxt;
            } while (cur != e0 && n < 12);
            // orientation: outward normal of the face linking loop[0] and loop[1]
            const int f = link[loop[0]][0] == loop[1] ? face_of[loop[0]][0] : face_of[loop[0]][1];
            const int a = f >> 1;
            const double nrm = (f & 1) ? 1.0 : -1.0;
            auto mid = [](int e, double *m) {
                const int lo = edge_lo(e), hi = edge_hi(e);
                for (int k = 0; k < 3; ++k) m[k] = 0.5 * (((lo >> k) & 1) + ((hi >> k) & 1));
            };
            double m0[3], m1[3], c[3];
            mid(loop[0], m0);
            mid(loop[1], m1);
            const int in0 = inside(edge_lo(loop[0])) ? edge_lo(loop[0]) : edge_hi(loop[0]);
            for (int k = 0; k < 3; ++k) c[k] = (double)((in0 >> k) & 1);
            const double d[3] = {m1[0] - m0[0], m1[1] - m0[1], m1[2] - m0[2]};
            const double w[3] = {c[0] - m0[0], c[1] - m0[1], c[2] - m0[2]};
            const double cross_a = d[(a + 1) % 3] * w[(a + 2) % 3] - d[(a + 2) % 3] * w[(a + 1) % 3];
            if (cross_a * nrm < 0.0)  // inside corner on the right: reverse the loop
                for (int i = 0, j = n - 1; i < j; ++i, --j) {
                    const int t = loop[i];
                    loop[i] = loop[j];
                    loop[j] = t;
                }
            int first = 0;
            for (int i = 1; i < n; ++i)
                if (loop[i] < loop[first]) first = i;
            for (int i = 1; i + 1 < n; ++i) {
                T.edge[cfg][3 * nt] = (uint8_t)loop[first];
                T.edge[cfg][3 * nt + 1] = (uint8_t)loop[(first + i + 1) % n];
                T.edge[cfg][3 * nt + 2] = (uint8_t)loop[(first + i) % n];
                ++nt;
            }
        }
        T.count[cfg] = (uint8_t)nt;
    }
}

constexpr int kHalo = 9;  // a block plus the +1 layers
constexpr int kMeshWarps = 8, kMeshThreads = 32 * kMeshWarps;
constexpr int kMeshChunk = 256;  // triangles listed at a time

// One warp's working set: its block's values with the +1 layers, the signs and
// observed flags of each x-row of nine (bits 0..8 and 16..24), the triangles
// listed for output and a round of vertices on their way out.
struct MeshWarp {
    float F[kHalo * kHalo * kHalo];
    uint32_t row[kHalo * kHalo];
    uint32_t list[kMeshChunk];
    float out[96];
};

// Bits 0..3: which bytes of w are not 0.
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t w)
{
    const uint32_t t = ((((w & 0x7f7f7f7fu) + 0x7f7f7f7fu) | w) >> 7) & 0x01010101u;
    return (t * 0x10204080u) >> 28;  // byte i's bit to bit 28 + i; no other product reaches bit 28
}

// An x-row of nine voxels on its way to the working set: eight of block p0
// from its voxel at, one of block p1 (-1: not in device memory; sdf 1,
// unobserved).
template <int MODE>
struct RowVoxels {
    float4 a, b, wa, wb;
    uint2 w;
    float f8, w8;
    __device__ __forceinline__ void load(const SceneDev &s, int p0, int p1, int at)
    {
        a = b = make_float4(1.f, 1.f, 1.f, 1.f);
        wa = wb = make_float4(0.f, 0.f, 0.f, 0.f);
        w = make_uint2(0u, 0u);
        f8 = 1.0f;
        w8 = 0.0f;
        if (p0 >= 0) {
            const size_t i = (size_t)p0 * kBlockVoxels + at;
            a = __ldg(reinterpret_cast<const float4 *>(s.sdf + i));
            b = __ldg(reinterpret_cast<const float4 *>(s.sdf + i) + 1);
            if (MODE == 0) {
                w = __ldg(reinterpret_cast<const uint2 *>(s.w8 + i));
            } else {
                wa = __ldg(reinterpret_cast<const float4 *>(s.w32 + i));
                wb = __ldg(reinterpret_cast<const float4 *>(s.w32 + i) + 1);
            }
        }
        if (p1 >= 0) {
            const size_t i = (size_t)p1 * kBlockVoxels + at;
            f8 = __ldg(&s.sdf[i]);
            w8 = MODE == 0 ? (float)__ldg(&s.w8[i]) : __ldg(&s.w32[i]);
        }
    }
    // the nine values to F; returns their sign bits (0..8) and observed bits (16..24)
    __device__ __forceinline__ uint32_t store(float *F) const
    {
        const float v[9] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, f8};
        uint32_t bits = MODE == 0 ? (nonzero_bytes(w.x) | (nonzero_bytes(w.y) << 4)) << 16 : 0u;
        if (MODE == 1) {
            const float o[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
            for (int x = 0; x < 8; ++x) bits |= o[x] > 0.0f ? 0x10000u << x : 0u;
        }
        bits |= w8 > 0.0f ? 0x1000000u : 0u;
#pragma unroll
        for (int x = 0; x < 9; ++x) {
            F[x] = v[x];
            bits |= v[x] < 0.0f ? 1u << x : 0u;
        }
        return bits;
    }
};

// One block per warp, no barriers: its eight blocks are looked up by eight lanes, its 9^3 voxels staged as 81 x-rows (a lane takes three, as vectors),
// the cells' sign patterns read off the rows' bit masks (a lane takes two
// x-rows of eight cells), one atomic reserves the block's triangles, and the lanes then take one vertex
// each and write 96 consecutive floats per round.
//
// What bounds it: latency (cells, voxels, the reservation), hidden by up
// to 40 warps per SM that each keep a block in flight.  Before, a CTA of 256
// threads took a block between four barriers, reserved space with sixteen
// atomics on the one counter and wrote each triangle's nine floats from one
// thread: 156 us on average of the sizing and the filling call for rooms of
// 9.5 to 27 thousand blocks (1.1 to 3.3 million triangles), 93 us by warps with
// one voxel per lane and load, 56 us with rows as vectors.
template <int MODE>
__global__ void __launch_bounds__(kMeshThreads) mesh_kernel(SceneDev s, const McTable tab, float *__restrict__ out,
                                                            long long cap, unsigned long long *__restrict__ counter)
{
    extern __shared__ __align__(16) unsigned char mesh_smem[];
    McTable &st = *reinterpret_cast<McTable *>(mesh_smem);
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(&tab);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&st);
        for (int i = threadIdx.x; i < (int)(sizeof(McTable) / 4); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    MeshWarp &w = reinterpret_cast<MeshWarp *>(mesh_smem + sizeof(McTable))[warp];
    const int n = min(__ldcg(&s.ctr->block_head), s.nv);
    const float vs = s.voxel_size;
    for (int i = blockIdx.x * kMeshWarps + warp; i < n; i += gridDim.x * kMeshWarps) {
        const int ptr = __ldg(&s.block_free[i]);
        const short4 b = __ldg(&s.block_pos[ptr]);
        if (!b.w) continue;  // uniform over the warp
        // lane l < 8: the block at (l & 1, l >> 1 & 1, l >> 2) from it
        const int nx = b.x + (lane & 1), ny = b.y + ((lane >> 1) & 1), nz = b.z + ((lane >> 2) & 1);
        const int nb = lane < 8 && in_i16(nx) && in_i16(ny) && in_i16(nz) ? brick_find(s, nx, ny, nz) : -1;
        __syncwarp();  // the previous block's working set is no longer read
        // a lane takes the x-rows lane, lane + 32, lane + 64 of the 9 x 9: eight
        // voxels of one block as vectors and the first of the block beside it
        RowVoxels<MODE> rv[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int r = min(lane + 32 * k, kHalo * kHalo - 1), z = r / kHalo, y = r - kHalo * z;
            const int h = ((y >> 3) << 1) | ((z >> 3) << 2);
            const int p0 = __shfl_sync(kFull, nb, h), p1 = __shfl_sync(kFull, nb, h | 1);
            rv[k].load(s, p0, p1, 8 * (y & 7) + 64 * (z & 7));
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int r = lane + 32 * k;
            if (r < kHalo * kHalo) w.row[r] = rv[k].store(&w.F[kHalo * r]);
        }
        __syncwarp();
        // triangles of the lane's cells: x-rows lane and lane + 32 (y = row & 7, z = row >> 3)
        uint32_t cfgs[4] = {0u, 0u, 0u, 0u};  // one byte per cell, 0 where the cell has none
        int nt = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r0 = kHalo * ((lane >> 3) + 4 * h) + (lane & 7);
            const uint32_t a = w.row[r0], c = w.row[r0 + 1], d = w.row[r0 + kHalo], e = w.row[r0 + kHalo + 1];
            const uint32_t obs = (a & c & d & e) >> 16;
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const uint32_t cfg = ((a >> x) & 3u) | (((c >> x) & 3u) << 2) | (((d >> x) & 3u) << 4) |
                                     (((e >> x) & 3u) << 6);
                if (((obs >> x) & 3u) == 3u && cfg != 0u && cfg != 255u) {
                    nt += st.count[cfg];
                    cfgs[2 * h + (x >> 2)] |= cfg << (8 * (x & 3));
                }
            }
        }
        int incl = nt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        const int total = __shfl_sync(kFull, incl, 31);
        if (total == 0) continue;
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(counter, (unsigned long long)total);
        base = __shfl_sync(kFull, base, 0);
        const long long room = cap - (long long)base;  // triangles that still fit
        const int fits = room < (long long)total ? (room > 0 ? (int)room : 0) : total;
        for (int c0 = 0; c0 < fits; c0 += kMeshChunk) {
            __syncwarp();
            int at = incl - nt - c0;
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const uint32_t cfg = (cfgs[q >> 2] >> (8 * (q & 3))) & 0xffu;
                if (!cfg) continue;
                const int m = st.count[cfg];
                const uint32_t cell = (uint32_t)((q & 7) + 8 * (lane & 7) + 64 * ((lane >> 3) + 4 * (q >> 3)));
                for (int t = 0; t < m; ++t, ++at)
                    if ((unsigned)at < (unsigned)kMeshChunk) w.list[at] = cell | ((uint32_t)t << 9) | (cfg << 12);
            }
            __syncwarp();
            const int nv = 3 * min(kMeshChunk, fits - c0);  // vertices of this chunk
            float *dst = out + ((size_t)base + c0) * 9;
            for (int v0 = 0; v0 < nv; v0 += 32) {
                const int v = v0 + lane;
                if (v < nv) {
                    const int tri = v / 3, j = v - 3 * tri;
                    const uint32_t item = w.list[tri];
                    const uint32_t cfg = item >> 12, t = (item >> 9) & 7u;
                    const int cx = item & 7, cy = (item >> 3) & 7, cz = (item >> 6) & 7;
                    // edge 4 a + o1 + 2 o2 along axis a: its lower corner ka, the next one's step
                    const int e = st.edge[cfg][3 * t + j];
                    const int axis = e >> 2;
                    const int ka = (int)((0x321054106420ull >> (4 * e)) & 7);
                    const int gx = cx + (ka & 1), gy = cy + ((ka >> 1) & 1), gz = cz + (ka >> 2);
                    const int at_a = gx + kHalo * (gy + kHalo * gz);
                    const float Fa = w.F[at_a];
                    const float Fb = w.F[at_a + ((0x510901 >> (8 * axis)) & 0x7f)];
                    const float tt = fdiv(Fa, fsub(Fa, Fb));
                    const int g[3] = {8 * b.x + gx, 8 * b.y + gy, 8 * b.z + gz};
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        float coord = (float)g[k];
                        if (k == axis) coord = fadd(coord, tt);
                        w.out[3 * lane + k] = fmul(coord, vs);
                    }
                }
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    if (32 * k + lane < 3 * (nv - v0)) dst[3 * v0 + 32 * k + lane] = w.out[32 * k + lane];
                __syncwarp();
            }
        }
    }
}

constexpr size_t kMeshSmem = sizeof(McTable) + kMeshWarps * sizeof(MeshWarp);
static_assert(sizeof(McTable) % 16 == 0 && sizeof(MeshWarp) % 4 == 0, "aligned working sets");

// CTAs of mesh_kernel<MODE> resident at once
template <int MODE>
int mesh_grid()
{
    static int g = 0;
    if (!g) {
        int dev = 0, sms = 1, per = 1;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaFuncSetAttribute(mesh_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMeshSmem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, mesh_kernel<MODE>, kMeshThreads, kMeshSmem);
        g = sms * (per > 0 ? per : 1);
    }
    return g;
}

// built on first use (a function-local static: thread-safe initialisation)
const McTable &mc_table()
{
    static const McTable T = [] {
        McTable t;
        build_table(t);
        return t;
    }();
    return T;
}

}  // namespace

int mesh_case_table(uint8_t *count, uint8_t *edges)
{
    const McTable &t = mc_table();
    memcpy(count, t.count, sizeof(t.count));
    memcpy(edges, t.edge, sizeof(t.edge));
    return ITM_OK;
}

cudaError_t launch_mesh(const SceneDev &s, float *out, long long cap, unsigned long long *counter, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    if (s.weight_mode == 0)
        mesh_kernel<0><<<mesh_grid<0>(), kMeshThreads, kMeshSmem, st>>>(s, mc_table(), out, cap, counter);
    else
        mesh_kernel<1><<<mesh_grid<1>(), kMeshThreads, kMeshSmem, st>>>(s, mc_table(), out, cap, counter);
    return cudaGetLastError();
}

}  // namespace itm

extern "C" int itm_mesh_case_table(uint8_t *count, uint8_t *edges)
{
    if (!count || !edges) return ITM_ERR_ARG;
    return itm::mesh_case_table(count, edges);
}
