// Internal definitions shared by the CUDA translation units of libitm.
//
// Device layout of one scene (all arrays allocated once by itm_scene_create):
//   entries     Entry[nb + ne]      16 B each; buckets then excess entries (Sec. 3.2)
//   req         uint64[nb]          per-bucket allocation request (packed key, 0 = none)
//   req_list    int32[nb]           buckets that received a request this frame
//   overflow    uint64[ovf_cap]     requests that lost their bucket to another key
//   visible     int32[nv]           visible block indices of the current frame
//   block_pos   short4[nv]          coordinates of the block held at each index (w = 1 in use)
//   sdf         float[nv][512]      TSDF, voxel index x + 8y + 64z (Sec. 3.1)
//   w8 / w32    uint8 / float [nv][512]  weights (constant / learned observation weight)
//   block_free  int32[nv]           free block list, handed out front to back
//   excess_free int32[ne]           free excess slots, handed out front to back
//   ctr         Counters            device counters and the sticky status word
//   brick_*     per brick place     block indices by block coordinates (brick_fetch8), for the
//                                   kernels that only look blocks up
//   swap_state  uint8[nb + ne]      Sec. 5 swapping (itm_swap_enable): kSw* per entry
//   touch       int32[nv]           last allocation whose segments met the block (-1: freed
//                                   by the running swap-out)
//   rgbw        uint32[nv][512]     colour voxels (itm_colour_enable): bytes r, g, b, colour weight
//   host store  pinned host memory mapped into the device, one slot per entry:
//               float[nb + ne][512] sdf and uint8 / float [nb + ne][512] weights
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include "itm.h"

namespace itm {

constexpr int kBlockVoxels = 512;
// largest image whose raycast uses the search-range tiles (8x4 pixels each)
constexpr int kRangeMaxW = 4096, kRangeMaxH = 4096;
constexpr int kRangeMaxTiles = (kRangeMaxW / 8) * (kRangeMaxH / 4);
// rays that the raycast's slow list has room for (larger images march every ray in the first phase)
constexpr int kSlowMax = 1 << 21;
constexpr int kCombinedMax = ITM_COMBINED_MAX;
constexpr int kIcpSums = ITM_ICP_SUMS;
constexpr int kIcpWorkDoubles = ITM_ICP_WORK_DOUBLES;
constexpr int kIcpMaxPartials = ITM_ICP_WORK_DOUBLES / ITM_ICP_SUMS - 1;
constexpr int kTrackMaxLevels = ITM_TRACK_MAX_LEVELS;
constexpr unsigned kFull = 0xffffffffu;

// Sec. 5 swap state of a hash entry
constexpr uint8_t kSwDevice = 0;  // current data in the device block (or none)
constexpr uint8_t kSwHost = 1;    // swapped out: data in the host slot only, entry ptr -1
constexpr uint8_t kSwMerge = 2;   // host data waiting to be fused into the device block

// Sec. 3.2 hash entry.  Bytes 0..7 (x, y, z, flag) form the packed block key
// compared and claimed as one 64-bit word; flag = 1 marks an entry that holds
// a block, so the all-zero word means "never used".
struct __align__(16) Entry {
    int16_t x, y, z, flag;
    int32_t offset;  // 0: end of chain; k >= 1: next entry at nb + k - 1 (Sec. 3.3)
    int32_t ptr;     // >= 0 block index; -1 swapped out; < -1 unallocated (Sec. 3.2)
};

// Counts of one allocation.
struct FrameCounters {
    int32_t n_req;          // buckets requested
    int32_t n_overflow;     // requests that lost their bucket
    int32_t depth_max_bits; // largest valid depth (float bits, >= 0)
    int32_t done;           // CTAs of the commit that finished (frames with an overflow)
};

// Two sets of frame counts take turns, so that no launch in front of an
// allocation has to clear them.  The enumeration reads `entered` and counts in
// set entered & 1; it writes `begun`, from which the passes after it know the
// set (frame_set); the first of them to follow clears the other set and
// writes `entered`.  Neither word is read by a kernel that writes it.
struct Counters {
    uint32_t status;
    int32_t block_head;     // blocks handed out (may run past nv when the array is full)
    int32_t excess_head;    // excess slots handed out
    int32_t n_visible;      // visible blocks
    int32_t head_before;    // blocks handed out before the last allocation
    uint32_t begun, entered;  // allocations whose enumeration / whose commit has run
    FrameCounters frame[2];
    unsigned long long updated;  // cumulative voxel updates
    unsigned long long visited;  // cumulative voxels visited by integration
    unsigned long long frames;   // cumulative integrated frames
    unsigned long long mesh_tris;  // per-mesh: triangles found
};

// Counts of one raycast: its next tile, its slow rays.  Two sets take turns as
// in Counters: the first phase reads `entered` and writes `begun`, the second
// reads `begun`, clears the other set and writes `entered`.
struct RayCounters {
    uint32_t begun, entered;
    struct {
        int32_t next, n_slow;
    } set[2];
};

struct SceneDev {
    Entry *entries;
    unsigned long long *req;
    int32_t *req_list;
    unsigned long long *overflow;
    int32_t *visible;
    short4 *block_pos;
    float *sdf;
    uint8_t *w8;
    float *w32;
    int32_t *block_free;
    int32_t *excess_free;
    Counters *ctr;
    unsigned long long *brick_owner;  // the brick of each place (brick_key), 0: none yet
    unsigned long long *brick_count;  // cells of the place that hold a block, kBrickOther for each block not entered
    int32_t *brick_cell;              // kBrickCells block indices per place, -1: none
    uint32_t brick_mask;              // places - 1
    uint32_t *range_min;  // per 8x4 tile: nearest / farthest depth (float bits) of covering blocks
    uint32_t *range_max;
    RayCounters *ray_ctr;
    int32_t *slow_list;  // kSlowMax pixels: rays not through with the raycast's first phase
    // Sec. 5 swapping: null while swapping is off
    uint8_t *swap_state;
    int32_t *touch;
    int swap_frame;  // allocations since swapping was enabled
    uint32_t *rgbw;  // colour voxels (Sec. 3.1): null while colour is off
    int nb, ne, nv;
    int ovf_cap;
    float voxel_size, mu, z_min, z_max;
    float inv_mu;  // RN(1 / mu)
    int max_w, weight_mode;
    // one part of a scene split by slabs of block columns (itm_scene_set_shard);
    // shard_n <= 1: the whole scene
    int shard_n, shard_i, shard_w;
};

struct Intr {
    int W, H;
    float fx, fy, cx, cy;
};

// Rows 0..2 of a 4x4 rigid transform, row-major.
struct Mat34 {
    float m[12];
};

// ---------------------------------------------------------------- hashing

// Sec. 3.2 hashIndex: unsigned coordinates times three primes, xor, mask.
__host__ __device__ __forceinline__ uint32_t hash_bucket(int x, int y, int z, uint32_t mask)
{
    return (((uint32_t)x * 73856093u) ^ ((uint32_t)y * 19349669u) ^ ((uint32_t)z * 83492791u)) & mask;
}

__host__ __device__ __forceinline__ unsigned long long pack_key(int x, int y, int z)
{
    return (unsigned long long)(uint16_t)x | ((unsigned long long)(uint16_t)y << 16) |
           ((unsigned long long)(uint16_t)z << 32) | (1ull << 48);
}

__device__ __forceinline__ void unpack_key(unsigned long long k, int &x, int &y, int &z)
{
    x = (int)(int16_t)(k & 0xffff);
    y = (int)(int16_t)((k >> 16) & 0xffff);
    z = (int)(int16_t)((k >> 32) & 0xffff);
}

__device__ __forceinline__ unsigned long long entry_key(const int4 &e)
{
    return (unsigned long long)(uint32_t)e.x | ((unsigned long long)(uint32_t)e.y << 32);
}

// Sec. 3.3 retrieval through the read-only path (tables not modified by the
// running kernel).  Returns the block index or -1.
__device__ __forceinline__ void set_status(const SceneDev &s, uint32_t bits)
{
    atomicOr(&s.ctr->status, bits);
}

// Builds with -DITM_CHECK_BOUNDS check the indices into the hash table, the
// voxel block array, the depth image and the per-frame lists before the
// access; a failed check sets ITM_ST_BOUNDS and the access is skipped.  In
// normal builds the checks compile to nothing.
#ifdef ITM_CHECK_BOUNDS
#define ITM_IN_BOUNDS(s, cond) ((cond) ? true : (set_status((s), ITM_ST_BOUNDS), false))
#else
#define ITM_IN_BOUNDS(s, cond) true
#endif

__device__ __forceinline__ int lookup_ro(const SceneDev &s, int bx, int by, int bz)
{
    const unsigned long long key = pack_key(bx, by, bz);
    int idx = (int)hash_bucket(bx, by, bz, (uint32_t)(s.nb - 1));
    const int4 *E = reinterpret_cast<const int4 *>(s.entries);
    for (int guard = 0; guard <= s.ne; ++guard) {
        int4 e = __ldg(&E[idx]);
        if (entry_key(e) == key && e.w >= 0) return ITM_IN_BOUNDS(s, e.w < s.nv) ? e.w : -1;
        if (e.z < 1) return -1;
        if (!ITM_IN_BOUNDS(s, e.z - 1 < s.ne)) return -1;
        idx = s.nb + e.z - 1;
    }
    return -1;
}

// Same, through L2 (coherent with writes made earlier by the same kernel).
__device__ __forceinline__ int lookup_cg(const SceneDev &s, int bx, int by, int bz)
{
    const unsigned long long key = pack_key(bx, by, bz);
    int idx = (int)hash_bucket(bx, by, bz, (uint32_t)(s.nb - 1));
    const int4 *E = reinterpret_cast<const int4 *>(s.entries);
    for (int guard = 0; guard <= s.ne; ++guard) {
        int4 e = __ldcg(&E[idx]);
        if (entry_key(e) == key && e.w >= 0) return ITM_IN_BOUNDS(s, e.w < s.nv) ? e.w : -1;
        if (e.z < 1) return -1;
        if (!ITM_IN_BOUNDS(s, e.z - 1 < s.ne)) return -1;
        idx = s.nb + e.z - 1;
    }
    return -1;
}

// ----------------------------------------------------------- brick table
// The blocks in device memory by their coordinates, for the kernels that look
// blocks up without changing them: the raycasts, the mesh, the colour of
// points, and the enumeration, which requests a block when it is not found
// here, so that every block of the hash table has to be here as well (or its
// brick marked) before the next allocation begins.  A brick is 8 x 8
// x 8 blocks, brick (X, Y, Z) = (bx, by, bz) >> 3; its place in the table is a
// hash of its coordinates.  A place has room for one brick, the first that
// came (brick_owner), and holds 9 x 9 x 9 block indices: the brick's blocks
// and the blocks one further along each axis, so that the up to eight blocks
// that a 2x2x2 voxel stencil reaches are cells of one brick at fixed offsets.
// Blocks of a brick whose place is taken are not entered; the place is marked
// (kBrickShared) and lookups in that brick go to the hash table.  They are
// counted, so that the mark goes with the last of them, and a place that no
// block counts on is free again: a camera that travels, with swapping, leaves
// no places behind that are taken or marked for bricks that have left.
//
// Why: through the hash table each of those eight blocks was a key, a hash
// and a scattered 16-byte load of its own, one after the other wherever any
// lane of the warp crossed a block face; here they are 4-byte loads of
// neighbouring words that are issued together with the owner's, so that a
// sample has two dependent loads, cells and voxels.  (Neighbour indices kept
// with each block, found through the hash, made three and measured slower:
// 153 us against 151 us before and 129 us now for a 640x480 frame of
// the room; cells with a tag of their own instead of the place's owner took a
// fifth more instructions.)
//
// Blocks enter in the last pass of the allocation that hands them out (and
// after an import), and leave in the swap-out; the kernels that change the
// table and those that read it never run at the same time.  When that pass
// cannot be launched, the scene notes it and the next call enters all blocks
// anew (recover).
constexpr int kBrickSide = 9;      // blocks along a brick's edge with the one further
constexpr int kBrickCells = 736;   // 9^3 cells, rounded up to whole 32-byte sectors
constexpr int kBrickMin = 4096;    // smallest number of places (12 MB)
constexpr unsigned long long kBrickValid = 1ull << 48, kBrickShared = 1ull << 63, kBrickOther = 1ull << 32;

// places for nv blocks: one for every 16 blocks (a surface fills a brick with
// about a hundred, and the bricks before it by their ninth cells), 185 bytes
// per block beside its 2560 bytes of voxels.  Bricks that find their place
// taken cost the walks the table is there to save: with one place for 32
// blocks, 512 at least, a camera turning round in a room of 350 bricks took
// 196 us per frame instead of 168.
inline int brick_places(int nv)
{
    int n = kBrickMin;
    while (n < nv / 16) n *= 2;
    return n;
}

// the owner word of brick (X, Y, Z) = block coordinates >> 3
__host__ __device__ __forceinline__ unsigned long long brick_key(int X, int Y, int Z)
{
    return (unsigned long long)((uint32_t)(X & 0xffff) | ((uint32_t)Y << 16)) |
           ((unsigned long long)(uint32_t)(Z & 0xffff) << 32) | kBrickValid;
}
// its place: neighbouring bricks lie apart from each other, distant ones at random
__host__ __device__ __forceinline__ uint32_t brick_place(int X, int Y, int Z, uint32_t mask)
{
    return ((uint32_t)X + (uint32_t)Y * 0x9e3779b1u + (uint32_t)Z * 0x85ebca77u) & mask;
}
__host__ __device__ __forceinline__ int brick_local(int lx, int ly, int lz)
{
    return lx + kBrickSide * ly + kBrickSide * kBrickSide * lz;
}

// The hash table's answer for a block of a brick whose place is shared; a call
// of its own, as it is rare and would be inlined for every block of a stencil.
static __device__ __noinline__ int lookup_chain(const SceneDev &s, int bx, int by, int bz)
{
    return lookup_ro(s, bx, by, bz);
}

// The block index at (bx, by, bz), or -1; in two parts, so that the loads of
// several blocks can be issued together.
struct BrickCell {
    unsigned long long own;
    int ptr;
};
__device__ __forceinline__ BrickCell brick_load(const SceneDev &s, int bx, int by, int bz)
{
    const uint32_t place = brick_place(bx >> 3, by >> 3, bz >> 3, s.brick_mask);
    return {__ldg(&s.brick_owner[place]),
            __ldg(&s.brick_cell[(size_t)place * kBrickCells + brick_local(bx & 7, by & 7, bz & 7)])};
}
__device__ __forceinline__ int brick_answer(const SceneDev &s, int bx, int by, int bz, const BrickCell &c)
{
    if ((c.own & ~kBrickShared) == brick_key(bx >> 3, by >> 3, bz >> 3))
        return ITM_IN_BOUNDS(s, c.ptr < s.nv) ? c.ptr : -1;
    return c.own & kBrickShared ? lookup_chain(s, bx, by, bz) : -1;
}
__device__ __forceinline__ int brick_find(const SceneDev &s, int bx, int by, int bz)
{
    return brick_answer(s, bx, by, bz, brick_load(s, bx, by, bz));
}

// The blocks of the 2x2x2 neighbourhood of block (bx, by, bz) towards +x, +y,
// +z: P[dx + 2 dy + 4 dz], where an axis without its cross flag stays at the
// block itself.
__device__ __forceinline__ void brick_fetch8(const SceneDev &s, int bx, int by, int bz, bool cx, bool cy, bool cz,
                                             int (&P)[8])
{
    const int X = bx >> 3, Y = by >> 3, Z = bz >> 3;
    const uint32_t place = brick_place(X, Y, Z, s.brick_mask);
    const int32_t *cell = s.brick_cell + (size_t)place * kBrickCells + brick_local(bx & 7, by & 7, bz & 7);
    const unsigned long long own = __ldg(&s.brick_owner[place]), key = brick_key(X, Y, Z);
    constexpr int dx = 1, dy = kBrickSide, dz = kBrickSide * kBrickSide;
    int R[8];
    R[0] = __ldg(cell);
#pragma unroll
    for (int k = 1; k < 8; ++k) {
        R[k] = -1;
        if ((!(k & 1) || cx) && (!(k & 2) || cy) && (!(k & 4) || cz))
            R[k] = __ldg(cell + ((k & 1) ? dx : 0) + ((k & 2) ? dy : 0) + ((k & 4) ? dz : 0));
    }
    if ((own & ~kBrickShared) != key) {
        // no block of this brick is in the table: none exists, or they are only in the hash table
        const bool chain = (own & kBrickShared) != 0ull;
        const int skip = (cx ? 0 : 1) | (cy ? 0 : 2) | (cz ? 0 : 4);
#pragma unroll 1
        for (int k = 0; k < 8; ++k) {
            const int p = chain && !(k & skip) ? lookup_chain(s, bx + (k & 1), by + ((k >> 1) & 1), bz + (k >> 2)) : -1;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (j == k) R[j] = p;
        }
    }
#ifdef ITM_CHECK_BOUNDS
    for (int k = 0; k < 8; ++k)
        if (!ITM_IN_BOUNDS(s, R[k] < s.nv)) R[k] = -1;
#endif
    P[0] = R[0];
    P[1] = cx ? R[1] : R[0];
    P[2] = cy ? R[2] : R[0];
    P[3] = cy ? (cx ? R[3] : R[2]) : P[1];
    P[4] = cz ? R[4] : R[0];
    P[5] = cz ? (cx ? R[5] : R[4]) : P[1];
    P[6] = cz ? (cy ? R[6] : R[4]) : P[2];
    P[7] = cz ? (cy ? (cx ? R[7] : R[6]) : P[5]) : P[3];
}

// Block (bx, by, bz) is a cell of its own brick and, on each axis where it is
// the brick's first, the ninth cell of the brick before: c = 0..7 takes the
// brick that is one before on the axes of c's bits.  False when there is no
// such brick (also outside the int16 block coordinates).
__host__ __device__ __forceinline__ bool brick_share(int bx, int by, int bz, int c, int &X, int &Y, int &Z, int &local)
{
    int b[3] = {bx, by, bz}, B[3], l[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        B[i] = b[i] >> 3;
        l[i] = b[i] & 7;
        if (c & (1 << i)) {
            if (l[i] != 0 || B[i] == -4096) return false;
            B[i] -= 1;
            l[i] = 8;
        }
    }
    X = B[0];
    Y = B[1];
    Z = B[2];
    local = brick_local(l[0], l[1], l[2]);
    return true;
}

// Block ptr enters at (bx, by, bz): the share of lane or thread c (0..7).
__device__ __forceinline__ void brick_put(const SceneDev &s, int bx, int by, int bz, int ptr, int c)
{
    int X, Y, Z, local;
    if (!brick_share(bx, by, bz, c, X, Y, Z, local)) return;
    const uint32_t place = brick_place(X, Y, Z, s.brick_mask);
    const unsigned long long key = brick_key(X, Y, Z);
    const unsigned long long old = atomicCAS(&s.brick_owner[place], 0ull, key);
    const bool own = old == 0ull || (old & ~kBrickShared) == key;
    if (own) s.brick_cell[(size_t)place * kBrickCells + local] = ptr;
    else atomicOr(&s.brick_owner[place], kBrickShared);
    atomicAdd(&s.brick_count[place], own ? 1ull : kBrickOther);
}

// The block at (bx, by, bz) leaves: the share of thread c (0..7).  While any
// block counts on the place its owner stays, so this finds the owner that
// brick_put found.  The one that takes the last count frees the place; the mark
// may be taken off before or after that (a free place's word stays 0).
__device__ __forceinline__ void brick_take(const SceneDev &s, int bx, int by, int bz, int c)
{
    int X, Y, Z, local;
    if (!brick_share(bx, by, bz, c, X, Y, Z, local)) return;
    const uint32_t place = brick_place(X, Y, Z, s.brick_mask);
    const bool own = (__ldcg(&s.brick_owner[place]) & ~kBrickShared) == brick_key(X, Y, Z);
    if (own) s.brick_cell[(size_t)place * kBrickCells + local] = -1;
    const unsigned long long one = own ? 1ull : kBrickOther;
    const unsigned long long left = atomicAdd(&s.brick_count[place], 0ull - one) - one;
    if (left == 0ull) s.brick_owner[place] = 0ull;
    else if (left < kBrickOther && !own) atomicAnd(&s.brick_owner[place], ~kBrickShared);
}

// ------------------------------------------------------ slab partition
// Block column x belongs to part floor(x / w) mod n; a part keeps its own
// columns and kShardGhost columns on either side (whose voxels every sample
// around a point of its own columns reads), and reports only raycast hits in
// its own columns.
constexpr int kShardGhost = 1;

__host__ __device__ __forceinline__ int slab_owner(int bx, int n, int w)
{
    const int q = bx >= 0 ? bx / w : -((-bx + w - 1) / w);  // floor(bx / w)
    const int r = q % n;
    return r < 0 ? r + n : r;
}

__device__ __forceinline__ bool shard_keeps(const SceneDev &s, int bx)
{
    if (s.shard_n <= 1) return true;
    bool keep = false;
#pragma unroll
    for (int d = -kShardGhost; d <= kShardGhost; ++d) keep = keep || slab_owner(bx + d, s.shard_n, s.shard_w) == s.shard_i;
    return keep;
}

__device__ __forceinline__ bool shard_owns(const SceneDev &s, int bx)
{
    return s.shard_n <= 1 || slab_owner(bx, s.shard_n, s.shard_w) == s.shard_i;
}

// ------------------------------------------ programmatic dependent launch
// The per-frame kernels are launched with programmatic stream serialization
// (launch_pdl): a kernel may be scheduled while the kernel before it on the
// stream drains, runs only what touches no memory until grid_dep_wait()
// (which returns once the previous kernel has completed and its writes are
// visible), and calls grid_dep_launch() when its own main work is done so
// that the next kernel can be scheduled early.  Both are no-ops for a kernel
// launched the ordinary way.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ------------------------------------------------ IEEE round-to-nearest ops
// Every operation that decides an integer (which block, which pixel, whether
// a voxel is updated) is written with these so that no multiply-add is fused.
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdiv_rn(a, b); }

// ((m0 x + m1 y) + m2 z) + m3, each operation rounded on its own.
__device__ __forceinline__ float row_apply(const float *m, float x, float y, float z)
{
    return fadd(fadd(fadd(fmul(m[0], x), fmul(m[1], y)), fmul(m[2], z)), m[3]);
}

// --------------------------------------------------------------- atomics


// Warp-aggregated append: the lanes active at the call each get a distinct
// slot of their counter; lanes naming the same counter share one atomic
// (lanes of one warp may work for different scenes in a batch).
__device__ __forceinline__ int warp_append(int32_t *counter)
{
    const unsigned active = __activemask();
    const int lane = threadIdx.x & 31;
    const unsigned peers = __match_any_sync(active, (unsigned long long)counter);
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(counter, __popc(peers));
    base = __shfl_sync(active, base, leader);
    return base + __popc(peers & ((1u << lane) - 1u));
}

}  // namespace itm

// Opaque handle behind the C ABI.
struct itm_scene {
    itm_scene_params params;
    itm::SceneDev d;
    cudaStream_t last_stream;
    int device;
    // the search-range tiles hold the range of a raycast from range_pose /
    // range_intr over the blocks allocated at epoch range_epoch
    long long alloc_epoch;
    long long range_epoch;
    float range_pose[16];
    itm_intrinsics range_intr;
    // the visible list's interior flags were computed for vis_pose /
    // vis_intr (vis_ok: by the last allocation, with no block moved or freed
    // since)
    bool vis_ok;
    float vis_pose[16];
    itm_intrinsics vis_intr;
    // Sec. 5 swapping (itm_swap_enable): the host store (pinned, mapped) and
    // the device scratch of the selection
    void *host_sdf, *host_w;
    void *swap_scratch;
    int swap_k, swap_idle;
    // weight mode 1: a second stream and fork / join events, so that
    // itm_process_frame_weighted runs the per-pixel weights beside the
    // allocation (made by itm_scene_create)
    cudaStream_t aux;
    cudaEvent_t ev_fork, ev_join;
    // a raycast's march was launched and its finish could not be: the counts
    // of rays (ray_ctr) are those of a raycast under way (recover)
    bool rays_behind;
    // the same of an allocation's commit and its visible-list pass: blocks that
    // the hash table has are not in the brick table
    bool bricks_behind;
};

// An NVTX range named after a C-ABI call for the duration of the call, so
// profiler timelines group each call's kernels (no cost without a profiler).
struct Range {
    explicit Range(const char *name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
};

// Host helpers implemented in itm_scene.cu.
namespace itm {
int check_cuda(cudaError_t e);
void pose_rows(const float T[16], Mat34 &out);        // rows 0..2 of T
void rigid_inverse_rows(const float T[16], Mat34 &out); // rows 0..2 of T^-1 (fp64, rounded once)
int valid_intr(const itm_intrinsics *in);
Intr to_intr(const itm_intrinsics *in);
// the visible list's interior flags hold for an integration with this pose
// and these intrinsics (launch_integrate's interior_ok)
bool interior_flags_hold(const itm_scene *sc, const float T_wc[16], const itm_intrinsics *intr);
// Puts right what a call that failed between two of its launches left behind;
// every call that reads or changes the brick table or the ray counts begins with it.
cudaError_t recover(itm_scene *sc, cudaStream_t st);
}  // namespace itm

// Launchers implemented in the kernel translation units.
namespace itm {
// half: the commit was launched and the visible-list pass was not
cudaError_t launch_allocate(const SceneDev &s, const float *depth, const Intr &in, const Mat34 &T_wc,
                            const Mat34 &M_d, bool with_range, cudaStream_t st, const uint16_t *raw, bool &half);
// interior_ok: the visible list was built by an allocation with this pose and
// these intrinsics, and no block changed since, so its interior flags hold
cudaError_t launch_integrate(const SceneDev &s, const float *depth, const float *wpx, const Intr &in,
                             const Mat34 &M_d, bool interior_ok, cudaStream_t st);
// half: the march was launched and the finish was not
cudaError_t launch_raycast(const SceneDev &s, const Intr &in, const Mat34 &T_wc, const Mat34 &M_d, float4 *vtx,
                           float4 *nrm, bool range_ready, cudaStream_t st, bool &half);
cudaError_t launch_raycast_range(const SceneDev &s, const Intr &in, const Mat34 &M_d, uint32_t *rmin, uint32_t *rmax,
                                 cudaStream_t st);
bool range_fits(const Intr &in);
cudaError_t launch_mesh(const SceneDev &s, float *out, long long cap, unsigned long long *counter, cudaStream_t st);
// Sec. 5 swapping state of a scene: freed by itm_scene_destroy, cleared by
// itm_scene_reset (itm_swap.cu)
void swap_free(itm_scene *sc);
cudaError_t swap_reset(itm_scene *sc, cudaStream_t st);
cudaError_t launch_depth_halve(const float *in, int W, int H, float *out, cudaStream_t st);
cudaError_t launch_icp_reduce(const float *depth, const Intr &in, const Mat34 &T_g, const float4 *V, const float4 *N,
                              const Intr &ref, const Mat34 &M_ref, float dist_thresh, double *work, cudaStream_t st);
size_t track_scratch_bytes(int W, int H, int levels);
cudaError_t launch_track(const float *depth, const Intr &in0, int levels, const int *iters, const float *thresh,
                         const float4 *V, const float4 *N, const Intr &ref, const Mat34 &M_ref, float T[16],
                         int *steps, void *scratch, cudaStream_t st);
cudaError_t launch_raycast_combined(const SceneDev *subs, const Mat34 *P, int n, const Intr &in, const Mat34 &T_wc,
                                    float4 *vtx, float4 *nrm, cudaStream_t st);
cudaError_t launch_depth_u16(const uint16_t *raw, float *out, int64_t n, cudaStream_t st);
cudaError_t launch_raycast_merge(const float4 *vtx, const float4 *nrm, int parts, long long npix, const Mat34 &M_d,
                                 float4 *vo, float4 *no, cudaStream_t st);
cudaError_t launch_reset(const SceneDev &s, cudaStream_t st);
// enters blocks 0 .. n-1 (block_pos) in the brick table
cudaError_t launch_brick_fill(const SceneDev &s, int n, cudaStream_t st);
// empties the brick table and enters every block in use
cudaError_t launch_brick_refill(const SceneDev &s, cudaStream_t st);
}  // namespace itm
