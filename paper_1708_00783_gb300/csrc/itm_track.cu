// Sec. 4.1.1 depth tracker (ITMDepthTracker): point-to-plane alignment of a
// depth frame to the raycast vertex/normal maps, coarse to fine.
//
//  * depth_halve_kernel: one pyramid level, the mean of the valid depths of
//    each 2x2 block (summed in raster order, one rounded division).
//  * icp_step_kernel: per pixel, the camera point d ((u-cx)/fx,
//    (v-cy)/fy, 1) mapped to the world by the current estimate T, projected
//    into the reference view (nearest pixel); with both maps valid there and
//    |T p - V| within the outlier distance, the residual r = (T p - V) . N and
//    J = (T p x N, N) give J J^T, J r, r^2 and a count.  The per-pixel
//    arithmetic is float with each operation rounded on its own (built with
//    -fmad=false), so the selection of pixels is the same on any IEEE
//    machine; a thread accumulates its pixels (about eight) in float and a
//    warp adds its lanes by a float shuffle tree (FP64 is a small fraction
//    of the FP32 rate here); the CTA adds its warps in double and writes one
//    partial row.  Each float sum is within 13 roundings of 2^-24 of the
//    magnitude of its terms.  Where a track does not converge, 19 steps make
//    1e-4 of the pose out of the last bit of a sum, so the split of the
//    pixels and the order of the sums are kept as they are (about eight pixels
//    per thread at every level: more threads with fewer pixels at the coarse
//    levels took the same time).
//  * the CTA that finishes last adds the partial rows in a fixed order (the
//    result does not depend on scheduling), then one of its warps solves
//    H x = -g in double and applies the motion x = (omega, tau) on the world
//    side, T <- [R(omega) | tau] T with R by Rodrigues' formula.  The pose
//    stays in device memory, so a whole coarse-to-fine track runs without a
//    host round trip per step (the paper solves on the host), one launch per
//    step, chained by programmatic dependent launch.
//
// What bounds a step is latency: the wait for the step before, the gathers of
// V and N at the projected pixel (L2), then the serial end (completion count,
// rows, 6x6 solve).  FP64 instructions cost about 16 issue cycles per warp,
// so sums run with lanes as columns and few rows, and the solve keeps one
// element of the symmetric system per lane.  640x480, three levels, 19 steps:
// 800 us per track with one kernel for the sums and one for a serial solve by
// a single thread (9 + 26 us per step), 328 us with this one (362 with IEEE
// divisions in the solve); 800 and 325 in later runs of both on one box.
#include "itm_ops.cuh"

namespace itm {

namespace {

constexpr int kIcpThreads = 256, kIcpWarps = kIcpThreads / 32;
constexpr int kBatch = 8;  // pixels of a thread per pass

__global__ void __launch_bounds__(256) depth_halve_kernel(const float *__restrict__ in, int W, int H,
                                                          float *__restrict__ out)
{
    const int w = W / 2, h = H / 2;
    grid_dep_wait();
    for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < w * h; o += gridDim.x * blockDim.x) {
        const int i = o % w, j = o / w;
        float sum = 0.0f;
        int n = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float d = __ldg(&in[(size_t)(2 * j + (k >> 1)) * W + 2 * i + (k & 1)]);
            if (d > 0.0f) {
                sum = fadd(sum, d);
                ++n;
            }
        }
        out[o] = n > 0 ? fdiv(sum, (float)n) : 0.0f;
    }
    grid_dep_launch();
}

struct IcpState {
    float T[16];     // current camera-to-world estimate
    int done_level;  // the level (from 1) that stopped: too few pixels or no solution
    int steps;       // steps applied
    int arrived;     // CTAs of the running step that wrote their row
};

__global__ void __launch_bounds__(32) track_begin_kernel(IcpState *st, Mat34 T)
{
    grid_dep_wait();
    if (threadIdx.x < 16) st->T[threadIdx.x] = threadIdx.x < 12 ? T.m[threadIdx.x] : (threadIdx.x == 15 ? 1.0f : 0.0f);
    if (threadIdx.x == 0) st->done_level = st->steps = st->arrived = 0;
    grid_dep_launch();
}

// Sum over the warp of v[0 .. 31], value l ending in lane l: each stage halves
// the values a lane holds (31 shuffles and adds instead of 5 per value).  The
// lanes 16, 8, 4, 2, 1 apart are added in that order.
__device__ __forceinline__ float warp_sum32(float (&v)[32], int lane)
{
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
        const bool up = lane & h;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float keep = up ? v[i + h] : v[i], send = up ? v[i] : v[i + h];
            v[i] = fadd(keep, __shfl_xor_sync(kFull, send, h));
        }
    }
    return v[0];
}

// Columns of the n_part partial rows, added by the whole CTA: lane l of warp 0
// gets column l.  Rows r, r + 32, ... are added in order for each r < 32, then
// the 32 sums by halves (r with r + 16, 8, 4, 2, 1): the order in which a warp
// with a row per lane adds them, here with a column per lane.
__device__ __forceinline__ double row_sums(const double *__restrict__ partials, int n_part, double (*red)[32], int lane,
                                           int warp)
{
    double x[4] = {0.0, 0.0, 0.0, 0.0};  // r = warp + 8 q
    if (lane < kIcpSums) {
        // 160 rows at a time, their loads issued together
        for (int b0 = warp; b0 < n_part; b0 += 160) {
            double v[20];
#pragma unroll
            for (int k = 0; k < 20; ++k) {
                const int b = b0 + 8 * k;
                v[k] = b < n_part ? __ldcg(&partials[(size_t)b * kIcpSums + lane]) : 0.0;
            }
#pragma unroll
            for (int k = 0; k < 20; ++k)
                if (b0 + 8 * k < n_part) x[k & 3] += v[k];  // uniform over the warp
        }
    }
    __syncthreads();  // red may still be read
    red[warp][lane] = (x[0] + x[2]) + (x[1] + x[3]);
    __syncthreads();
    if (warp != 0) return 0.0;
    return ((red[0][lane] + red[4][lane]) + (red[2][lane] + red[6][lane])) +
           ((red[1][lane] + red[5][lane]) + (red[3][lane] + red[7][lane]));
}
static_assert(kIcpWarps == 8, "row_sums adds eight warps' sums");

// 1 / a to within an ulp of double: Newton's iteration y + y (1 - a y) from
// the float reciprocal, whose error 2^-23 it squares twice (four FP64
// operations; the IEEE division costs several times as many).
__device__ __forceinline__ double rcp_double(double a)
{
    const float f = (float)a;
    if (!(f > 0x1p-100f && f < 0x1p100f)) return 1.0 / a;
    double y = (double)__frcp_rn(f);
    y = __fma_rn(y, __fma_rn(-a, y, 1.0), y);
    return __fma_rn(y, __fma_rn(-a, y, 1.0), y);
}

// One Gauss-Newton step by one warp: lane l holds sums[l] in x, that is
// element (i, j), i <= j, of the upper triangle of H row by row, then -g's
// entries as column 6.  Elimination keeps one element per lane: with pivot p,
// a_ij -= a_pi a_pj / a_pp for p < i <= j (H = L D L^T; the pivots are the
// squares of Cholesky's, so the system is refused in the same cases).
// Returns false when it has no solution; else T and the motion are applied.
__device__ __forceinline__ bool gauss_newton_warp(double x, IcpState *st, int lane)
{
    if (__shfl_sync(kFull, x, 28) < 6.0) return false;
    // this lane's row and column: sums 0..20 are (i, j), 21..26 are (i, 6)
    int i = 0, j = 0;
    {
        int k = 0;
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int c = r; c < 6; ++c, ++k)
                if (k == lane) i = r, j = c;
        if (lane >= 21) i = min(lane - 21, 5), j = 6;
    }
    const auto at = [](int r, int c) { return c == 6 ? 21 + r : 6 * r - r * (r - 1) / 2 + (c - r); };  // r <= c
    double inv[6];
#pragma unroll
    for (int p = 0; p < 6; ++p) {
        const double a = __shfl_sync(kFull, x, at(p, p));
        if (!(a > 0.0)) return false;  // uniform
        inv[p] = rcp_double(a);
        if (p == 5) break;
        const double aj = __shfl_sync(kFull, x, j < p ? 0 : at(p, j)), ai = __shfl_sync(kFull, x, i < p ? 0 : at(p, i));
        if (i > p && lane < 27) x = __fma_rn(-ai, aj * inv[p], x);
    }
    // U x = -g by columns from the last
    double s[6];
#pragma unroll
    for (int c = 5; c >= 0; --c) {
        s[c] = __shfl_sync(kFull, x, at(c, 6)) * inv[c];
        const double u = __shfl_sync(kFull, x, i <= c ? at(i, c) : 0);
        if (j == 6 && i < c) x = __fma_rn(-u, s[c], x);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) s[c] = -s[c];
    // R = I + s1 K + s2 K^2, K = [omega]_x, K^2 = omega omega^T - th^2 I, with
    // s1 = sin(th) / th, s2 = (1 - cos(th)) / th^2: their Taylor series in
    // th^2 for the usual small steps, to below 2^-60 relative (th < 1/64: the
    // term t2^4 / 9! is the last above it; th < 1/4: t2^7 / 15!)
    const double t2 = __fma_rn(s[0], s[0], __fma_rn(s[1], s[1], s[2] * s[2]));
    double s1, s2;
    if (t2 < 0x1p-4) {
        constexpr double c1[8] = {1.0, -1.0 / 6, 1.0 / 120, -1.0 / 5040, 1.0 / 362880, -1.0 / 39916800,
                                  1.0 / 6227020800.0, -1.0 / 1307674368000.0};
        constexpr double c2[8] = {1.0 / 2, -1.0 / 24, 1.0 / 720, -1.0 / 40320, 1.0 / 3628800, -1.0 / 479001600,
                                  1.0 / 87178291200.0, -1.0 / 20922789888000.0};
        s1 = c1[4];
        s2 = c2[4];
        if (t2 >= 0x1p-12) {
            s1 = __fma_rn(t2, __fma_rn(t2, __fma_rn(t2, c1[7], c1[6]), c1[5]), c1[4]);
            s2 = __fma_rn(t2, __fma_rn(t2, __fma_rn(t2, c2[7], c2[6]), c2[5]), c2[4]);
        }
#pragma unroll
        for (int k = 3; k >= 0; --k) {
            s1 = __fma_rn(t2, s1, c1[k]);
            s2 = __fma_rn(t2, s2, c2[k]);
        }
    } else {
        const double th = sqrt(t2);
        s1 = sin(th) / th;
        s2 = (1.0 - cos(th)) / t2;
    }
    // lane 4 r + c < 12: element (r, c) of [R | tau] T
    float Tn = 0.0f;
    if (lane < 12) {
        const int r = lane >> 2, c = lane & 3;
        const float Tc[3] = {__ldcg(&st->T[c]), __ldcg(&st->T[4 + c]), __ldcg(&st->T[8 + c])};
        const double wr = r == 0 ? s[0] : (r == 1 ? s[1] : s[2]);
        double acc = c == 3 ? (r == 0 ? s[3] : (r == 1 ? s[4] : s[5])) : 0.0;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const int o = 3 - r - m;  // off the diagonal, K[r][m] = -+ omega_o
            const double w = o == 0 ? s[0] : (o == 1 ? s[1] : s[2]);
            const double k = m == r ? -s2 * t2 : ((m - r + 3) % 3 == 1 ? -s1 : s1) * w;
            const double R = __fma_rn(s2 * wr, s[m], m == r ? 1.0 + k : k);
            acc = __fma_rn(R, (double)Tc[m], acc);
        }
        Tn = (float)acc;
    }
    __syncwarp();  // every lane has read T
    if (lane < 12) st->T[lane] = Tn;
    if (lane == 0) st->steps += 1;
    return true;
}

// Partial sums of CTA blockIdx.x: partials[b * kIcpSums + k].  The pose is
// read from the tracker state st, and the CTA that finishes last takes the
// step; or, with st null, from T_arg.  A thread takes the pixels p, p +
// stride, ... in order, kBatch per pass: their depth loads, then their map
// loads, are issued together.  prefetch: the depth frame was complete before
// the previous kernel of the stream began, so the first pass's camera points
// (which need no pose) are computed before the wait for that kernel, on the
// SMs that its last CTA's solve leaves idle.
__global__ void __launch_bounds__(kIcpThreads) icp_step_kernel(
    const float *__restrict__ depth, int W, int H, Intr in, IcpState *st, int level, Mat34 T_arg,
    const float4 *__restrict__ V, const float4 *__restrict__ N, Intr ref, Mat34 M, float dist_thresh,
    double *__restrict__ partials, bool prefetch)
{
    __shared__ double red[kIcpWarps][32];
    __shared__ int is_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_pix = W * H, stride = gridDim.x * blockDim.x;
    int p0 = blockIdx.x * blockDim.x + threadIdx.x;
    float pc[kBatch][3];  // camera points, z = 0: no depth
    auto camera_points = [&]() {
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int p = p0 + b * stride;
            const float d = p < n_pix ? __ldg(&depth[p]) : 0.0f;
            pc[b][2] = d > 0.0f ? d : 0.0f;
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int p = p0 + b * stride;
            const int u = p % W, v = p / W;
            pc[b][0] = fmul(fdiv(fsub((float)u, in.cx), in.fx), pc[b][2]);
            pc[b][1] = fmul(fdiv(fsub((float)v, in.cy), in.fy), pc[b][2]);
        }
    };
    if (prefetch) camera_points();
    grid_dep_wait();
    Mat34 T = T_arg;
    if (st) {
        // the pose with the level's flag, not after it
        const int done_level = __ldcg(&st->done_level);
#pragma unroll
        for (int k = 0; k < 12; ++k) T.m[k] = __ldcg(&st->T[k]);
        if (done_level == level) return;
    }
    if (!prefetch) camera_points();
    const float t2 = fmul(dist_thresh, dist_thresh);
    float acc[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) acc[k] = 0.0f;
    int count = 0;
    while (p0 < n_pix) {
        float pw[kBatch][3];
        int o[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            o[b] = -1;
            float pr[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) pw[b][r] = row_apply(T.m + 4 * r, pc[b][0], pc[b][1], pc[b][2]);
#pragma unroll
            for (int r = 0; r < 3; ++r) pr[r] = row_apply(M.m + 4 * r, pw[b][0], pw[b][1], pw[b][2]);
            if (pc[b][2] > 0.0f && pr[2] > 0.0f) {
                const float ur = fadd(fdiv(fmul(ref.fx, pr[0]), pr[2]), ref.cx);
                const float vr = fadd(fdiv(fmul(ref.fy, pr[1]), pr[2]), ref.cy);
                if (ur >= 0.0f && ur <= (float)(ref.W - 1) && vr >= 0.0f && vr <= (float)(ref.H - 1))
                    o[b] = (int)fadd(vr, 0.5f) * ref.W + (int)fadd(ur, 0.5f);
            }
        }
        float4 Vk[kBatch], Nk[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            Vk[b] = make_float4(0.f, 0.f, 0.f, 0.f);
            Nk[b] = Vk[b];
            if (o[b] >= 0) {
                Vk[b] = __ldg(&V[o[b]]);
                Nk[b] = __ldg(&N[o[b]]);
            }
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            if (o[b] < 0) continue;
            const float4 Vp = Vk[b], Np = Nk[b];
            if (!(Vp.w > 0.0f && Np.w > 0.0f)) continue;
            const float dx = fsub(pw[b][0], Vp.x), dy = fsub(pw[b][1], Vp.y), dz = fsub(pw[b][2], Vp.z);
            const float dist2 = fadd(fadd(fmul(dx, dx), fmul(dy, dy)), fmul(dz, dz));
            if (!(dist2 <= t2)) continue;
            const float res = fadd(fadd(fmul(dx, Np.x), fmul(dy, Np.y)), fmul(dz, Np.z));
            const float J[6] = {fsub(fmul(pw[b][1], Np.z), fmul(pw[b][2], Np.y)),
                                fsub(fmul(pw[b][2], Np.x), fmul(pw[b][0], Np.z)),
                                fsub(fmul(pw[b][0], Np.y), fmul(pw[b][1], Np.x)), Np.x, Np.y, Np.z};
            int k = 0;
#pragma unroll
            for (int i = 0; i < 6; ++i)
#pragma unroll
                for (int j = i; j < 6; ++j, ++k) acc[k] = fadd(acc[k], fmul(J[i], J[j]));
#pragma unroll
            for (int i = 0; i < 6; ++i) acc[21 + i] = fadd(acc[21 + i], fmul(J[i], res));
            acc[27] = fadd(acc[27], fmul(res, res));
            ++count;
        }
        p0 += kBatch * stride;
        if (p0 < n_pix) camera_points();
    }
    // warps by float shuffle trees (the count is a whole number below 2^24:
    // exact), then the CTA's warp rows in double, in order
    static_assert(kIcpSums == 29, "28 sums and the count");
    acc[28] = (float)count;
    red[warp][lane] = (double)warp_sum32(acc, lane);
    __syncthreads();
    if (warp == 0) {
        double x = 0.0;
#pragma unroll
        for (int w = 0; w < kIcpWarps; ++w) x += red[w][lane];
        if (lane < kIcpSums) {
            partials[(size_t)blockIdx.x * kIcpSums + lane] = x;
            __threadfence();
        }
        __syncwarp();
        if (lane == 0) is_last = st && atomicAdd(&st->arrived, 1) == (int)gridDim.x - 1;
    }
    if (!st) return;  // icp_sum_kernel adds the rows
    __syncthreads();
    grid_dep_launch();
    if (!is_last) return;
    __threadfence();
    const double sum = row_sums(partials, gridDim.x, red, lane, warp);
    if (warp != 0) return;
    if (lane == 0) st->arrived = 0;
    if (!gauss_newton_warp(sum, st, lane) && lane == 0) st->done_level = level;
}

// The n_part partial rows added into sums (one CTA).
__global__ void __launch_bounds__(kIcpThreads) icp_sum_kernel(const double *__restrict__ partials, int n_part,
                                                              double *__restrict__ sums)
{
    __shared__ double red[kIcpWarps][32];
    grid_dep_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double x = row_sums(partials, n_part, red, lane, warp);
    if (warp == 0 && lane < kIcpSums) sums[lane] = x;
}

// CTAs of a step: about eight pixels per thread, at most two CTAs per SM and
// kIcpMaxPartials rows.  The split also fixes the order of the sums.
int icp_grid(int n_pix)
{
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms < 1) sms = 1;
    }
    int g = (n_pix + 8 * kIcpThreads - 1) / (8 * kIcpThreads);
    if (g > 2 * sms) g = 2 * sms;
    if (g > kIcpMaxPartials) g = kIcpMaxPartials;
    return g > 0 ? g : 1;
}

}  // namespace

cudaError_t launch_depth_halve(const float *in, int W, int H, float *out, cudaStream_t st)
{
    const int n = (W / 2) * (H / 2);
    if (n <= 0) return cudaSuccess;
    int g = (n + 255) / 256;
    if (g > 1216) g = 1216;
    return launch_pdl(depth_halve_kernel, dim3(g), dim3(256), 0, st, in, W, H, out);
}

cudaError_t launch_icp_reduce(const float *depth, const Intr &in, const Mat34 &T_g, const float4 *V, const float4 *N,
                              const Intr &ref, const Mat34 &M_ref, float dist_thresh, double *work, cudaStream_t st)
{
    const int g = icp_grid(in.W * in.H);
    double *partials = work + kIcpSums;
    cudaError_t e = launch_pdl(icp_step_kernel, dim3(g), dim3(kIcpThreads), 0, st, depth, in.W, in.H, in,
                               (IcpState *)nullptr, 0, T_g, V, N, ref, M_ref, dist_thresh, partials, false);
    if (e != cudaSuccess) return e;
    return launch_pdl(icp_sum_kernel, dim3(1), dim3(kIcpThreads), 0, st, (const double *)partials, g, work);
}

size_t track_scratch_bytes(int W, int H, int levels)
{
    size_t b = sizeof(double) * (size_t)kIcpWorkDoubles + 256;  // work, then the state
    int w = W, h = H;
    for (int l = 1; l < levels; ++l) {
        w /= 2;
        h /= 2;
        b += sizeof(float) * (size_t)(w > 0 ? w : 0) * (size_t)(h > 0 ? h : 0);
        b = (b + 255) & ~(size_t)255;
    }
    return b;
}

cudaError_t launch_track(const float *depth, const Intr &in0, int levels, const int *iters, const float *thresh,
                         const float4 *V, const float4 *N, const Intr &ref, const Mat34 &M_ref, float T[16],
                         int *steps, void *scratch, cudaStream_t st)
{
    char *base = static_cast<char *>(scratch);
    double *work = reinterpret_cast<double *>(base);
    IcpState *state = reinterpret_cast<IcpState *>(base + sizeof(double) * (size_t)kIcpWorkDoubles);
    size_t off = sizeof(double) * (size_t)kIcpWorkDoubles + 256;
    const float *lev[kTrackMaxLevels];
    Intr li[kTrackMaxLevels];
    lev[0] = depth;
    li[0] = in0;
    Mat34 T0;
    pose_rows(T, T0);
    cudaError_t e = launch_pdl(track_begin_kernel, dim3(1), dim3(32), 0, st, state, T0);
    if (e != cudaSuccess) return e;
    for (int l = 1; l < levels; ++l) {
        float *out = reinterpret_cast<float *>(base + off);
        li[l].W = li[l - 1].W / 2;
        li[l].H = li[l - 1].H / 2;
        // pixel i of the next level covers pixels 2i, 2i+1: f / 2, (c - 1/2) / 2
        volatile float fx = li[l - 1].fx / 2.0f, fy = li[l - 1].fy / 2.0f;
        volatile float cxm = li[l - 1].cx - 0.5f, cym = li[l - 1].cy - 0.5f;
        li[l].fx = fx;
        li[l].fy = fy;
        li[l].cx = cxm / 2.0f;
        li[l].cy = cym / 2.0f;
        e = launch_depth_halve(lev[l - 1], li[l - 1].W, li[l - 1].H, out, st);
        if (e != cudaSuccess) return e;
        lev[l] = out;
        off += sizeof(float) * (size_t)li[l].W * (size_t)li[l].H;
        off = (off + 255) & ~(size_t)255;
    }
    double *partials = work + kIcpSums;
    bool first = true;
    for (int l = levels - 1; l >= 0; --l) {
        if (iters[l] <= 0 || li[l].W < 1 || li[l].H < 1) continue;
        const int g = icp_grid(li[l].W * li[l].H);
        for (int it = 0; it < iters[l]; ++it) {
            // the first step follows the pyramid's last kernel, which may have written its depth
            e = launch_pdl(icp_step_kernel, dim3(g), dim3(kIcpThreads), 0, st, lev[l], li[l].W, li[l].H, li[l], state,
                           l + 1, Mat34{}, V, N, ref, M_ref, thresh[l], partials, !first);
            if (e != cudaSuccess) return e;
            first = false;
        }
    }
    IcpState h_state;
    e = cudaMemcpyAsync(&h_state, state, sizeof(h_state), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    memcpy(T, h_state.T, sizeof(float) * 12);
    T[12] = T[13] = T[14] = 0.0f;
    T[15] = 1.0f;
    *steps = h_state.steps;
    return cudaGetLastError();
}

}  // namespace itm
