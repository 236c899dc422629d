// Pyramid build: the storage-typed levels of a batch of frames, their means, and for the nonrigid
// model the border and the B-spline model of every level.
//
// Every kernel takes all frames (grid.z or grid.x = frame).  The work is memory traffic for a long
// series and launch latency for one pair of frames, so it is few launches: level 0 with level 1 in
// one pass over the frame, one box average per further level, the means of all levels, and border
// and model of all levels.  For a pair of 512x512 frames (nonrigid, two levels) that is 3 launches
// instead of the 8 of one per level and step, which took 211 us, most of it the means summed by a
// single CTA each: the pair's registration went from 1,217 to 1,031 us, that of a 741x1003 pair (BF16)
// from 3,933 to 2,784 us, and a series' pyramids stay within 3 % of what they took.
#include <cooperative_groups.h>

#include "reg_dev.cuh"
#include "reg_internal.h"

namespace cg = cooperative_groups;

namespace reg {

// Level 0 in storage type and (DOWN) level 1 from it.  A CTA covers kTopRows rows of kTopCols
// columns; a thread holds columns kTopThreads apart, every load issued before the first store.  The
// 2x2 average takes the column to the right from the next lane (kTopThreads is a multiple of 32 and
// a tile starts at an even column), with the operations of pyr_down in its order; rows and columns
// past the frame repeat the last one, the clamp of an odd size.
constexpr int kTopThreads = 256, kTopRows = 8, kTopCols = 512;
template <typename S, bool DOWN>
__global__ void __launch_bounds__(kTopThreads) pyr_top(const float *frames, size_t fstride, int W, int H, int pitch,
                                                       S *out, size_t ostride, int opitch, S *dn, size_t dstride,
                                                       int dpitch)
{
    constexpr int CB = kTopCols / kTopThreads;
    const int c0 = blockIdx.x * kTopCols + threadIdx.x, r0 = blockIdx.y * kTopRows;
    const float *src = frames + blockIdx.z * fstride;
    out += blockIdx.z * ostride;
    dn += blockIdx.z * dstride;
    float v[kTopRows][CB];
#pragma unroll
    for (int i = 0; i < kTopRows; ++i)
#pragma unroll
        for (int j = 0; j < CB; ++j)
            v[i][j] = __ldg(src + (size_t)min(r0 + i, H - 1) * pitch + min(c0 + j * kTopThreads, W - 1));
#pragma unroll
    for (int i = 0; i < kTopRows; ++i)
#pragma unroll
        for (int j = 0; j < CB; ++j) {
            const int r = r0 + i, c = c0 + j * kTopThreads;
            const S x = toS<S>(v[i][j]);
            if (r < H && c < W) out[(size_t)r * opitch + c] = x;
            v[i][j] = fromS(x);   // the average is that of the stored samples
        }
    if constexpr (DOWN) {
        const int w2 = (W + 1) / 2, h2 = (H + 1) / 2;
#pragma unroll
        for (int i = 0; i < kTopRows; i += 2)
#pragma unroll
            for (int j = 0; j < CB; ++j) {
                const float a = __shfl_down_sync(0xffffffffu, v[i][j], 1), b = __shfl_down_sync(0xffffffffu, v[i + 1][j], 1);
                const int r = (r0 + i) / 2, c = (c0 + j * kTopThreads) / 2;
                if ((threadIdx.x & 1) == 0 && r < h2 && c < w2)
                    dn[(size_t)r * dpitch + c] = toS<S>(0.25f * (((v[i][j] + a) + v[i + 1][j]) + b));
            }
    }
}

// Level l+1 from level l: 2x2 box average, last odd row/column clamped.  A thread makes kDnRows
// samples of one column, every load issued before the first store.
constexpr int kDnThreads = 128, kDnRows = 8;
template <typename S>
__global__ void __launch_bounds__(kDnThreads) pyr_down(const S *src, size_t sstride, int spitch, int W, int H,
                                                       S *dst, size_t dstride, int dpitch)
{
    const int w2 = (W + 1) / 2, h2 = (H + 1) / 2;
    const int c = blockIdx.x * kDnThreads + threadIdx.x, rb = blockIdx.y * kDnRows;
    if (c >= w2) return;
    src += blockIdx.z * sstride;
    dst += blockIdx.z * dstride;
    const int c0 = 2 * c, c1 = min(2 * c + 1, W - 1);
    float v[kDnRows];
#pragma unroll
    for (int k = 0; k < kDnRows; ++k) {
        v[k] = 0.f;
        const int r = rb + k;
        if (r < h2) {
            const int r0 = 2 * r, r1 = min(2 * r + 1, H - 1);
            v[k] = ((ldS<S>(src + (size_t)r0 * spitch + c0) + ldS<S>(src + (size_t)r0 * spitch + c1)) +
                    ldS<S>(src + (size_t)r1 * spitch + c0)) + ldS<S>(src + (size_t)r1 * spitch + c1);
        }
    }
#pragma unroll
    for (int k = 0; k < kDnRows; ++k)
        if (rb + k < h2) dst[(size_t)(rb + k) * dpitch + c] = toS<S>(0.25f * v[k]);
}

// The levels of a pyramid, for the kernels that take all of them in one launch (grid.y = level).
template <typename S> struct Levels {
    S *lvl[kMaxLevels];      // pixel (0, 0) of frame 0
    size_t stride[kMaxLevels];
    S *smooth[kMaxLevels];   // B-spline model at the pixel centres, W x H, or null
    size_t sstride[kMaxLevels];
    int W[kMaxLevels], H[kMaxLevels], pitch[kMaxLevels];
    int nxb[kMaxLevels], nsb[kMaxLevels];   // pyr_finish: column blocks of the model, and its blocks
};

// Samples counted, their mean and sum of squared deviations; the union of two sets by Chan, Golub and LeVeque,
// "Updating formulae and a pairwise algorithm for computing sample variances", 1979: no cancellation, whatever
// the mean.
struct Spread {
    float n, mean, dev;
};
__device__ __forceinline__ Spread joined(Spread a, Spread b)
{
    const float n = a.n + b.n, d = b.mean - a.mean, w = n > 0.f ? b.n / n : 0.f;
    return Spread{n, fmaf(d, w, a.mean), a.dev + b.dev + d * d * (a.n * w)};
}

// Mean and standard deviation of every level of each frame; the mean a deterministic float-float sum: a cluster of kMeanCtas CTAs
// sums the rows of one level (a warp takes every kMeanCtas * kMeanWarps-th row, a lane every 32nd
// column with kMeanBatch loads in flight), and its first CTA adds the CTAs' sums in rank order.  The
// split is the same for every batch size, so a frame's means do not depend on the call it is in.
// One CTA sums at the rate a single SM loads, about 80 us for a 512x512 level: most of the call of a
// small pair.  A CTA stores into the first one's shared memory only once every CTA of the cluster is
// known to run: each arrives at the cluster barrier first and waits there after its sums.  The deviation's
// sums ride on the same loads: with the passes' use of them, 2.7 of the 97 us of a 160x128 pair.
constexpr int kMeanCtas = 8, kMeanWarps = 8, kMeanBatch = 8;
template <typename S>
__global__ void __launch_bounds__(32 * kMeanWarps) level_means(Levels<S> L, LevelStat *means, int levels)
{
    __shared__ float2 ws[kMeanWarps];
    __shared__ float2 part[kMeanCtas];
    __shared__ Spread wsp[kMeanWarps], spart[kMeanCtas];
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_arrive();
    const int l = blockIdx.y, f = blockIdx.x / kMeanCtas, rank = cl.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int W = L.W[l], H = L.H[l], pitch = L.pitch[l];
    const S *img = L.lvl[l] + (size_t)f * L.stride[l];
    float hi = 0.f, lo = 0.f;
    float x0 = 0.f, n = 0.f, s1 = 0.f, s2 = 0.f;   // the lane's first sample, and its samples' differences from it
    for (int r = rank * kMeanWarps + warp; r < H; r += kMeanCtas * kMeanWarps) {
        const S *row = img + (size_t)r * pitch;
        for (int c0 = lane; c0 < W; c0 += 32 * kMeanBatch) {
            float x[kMeanBatch], a = 0.f;
#pragma unroll
            for (int k = 0; k < kMeanBatch; ++k) x[k] = c0 + 32 * k < W ? ldS<S>(row + c0 + 32 * k) : 0.f;
            if (n == 0.f) x0 = x[0];
#pragma unroll
            for (int k = 0; k < kMeanBatch; ++k) {
                a += x[k];
                const float d = c0 + 32 * k < W ? x[k] - x0 : 0.f;
                s1 += d;
                s2 = fmaf(d, d, s2);
            }
            n += (float)min(kMeanBatch, (W - c0 + 31) / 32);
            ff_acc(hi, lo, a);
        }
    }
    const float m1 = n > 0.f ? s1 / n : 0.f;
    Spread sp{n, x0 + m1, fmaxf(fmaf(-s1, m1, s2), 0.f)};
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, off), l2 = __shfl_xor_sync(0xffffffffu, lo, off);
        ff_add(hi, lo, h2, l2);
        sp = joined(sp, Spread{__shfl_xor_sync(0xffffffffu, sp.n, off), __shfl_xor_sync(0xffffffffu, sp.mean, off),
                               __shfl_xor_sync(0xffffffffu, sp.dev, off)});
    }
    if (lane == 0) { ws[warp] = make_float2(hi, lo); wsp[warp] = sp; }
    __syncthreads();
    cl.barrier_wait();
    if (threadIdx.x == 0) {
        float h = 0.f, l2 = 0.f;
        for (int k = 0; k < kMeanWarps; ++k) ff_add(h, l2, ws[k].x, ws[k].y);
        *cl.map_shared_rank(&part[rank], 0) = make_float2(h, l2);
        for (int k = 1; k < kMeanWarps; ++k) sp = joined(sp, wsp[k]);
        *cl.map_shared_rank(&spart[rank], 0) = sp;
    }
    cl.sync();
    if (rank == 0 && threadIdx.x == 0) {
        float h = 0.f, l2 = 0.f;
        for (int k = 0; k < kMeanCtas; ++k) ff_add(h, l2, part[k].x, part[k].y);
        for (int k = 1; k < kMeanCtas; ++k) sp = joined(sp, spart[k]);
        means[(size_t)f * levels + l] = LevelStat{(float)(((double)h + (double)l2) / ((double)W * (double)H)), sqrtf(sp.dev / sp.n)};
    }
}

// Border and B-spline model of every level (grid.y = level, grid.z = frame).  Beyond its border a
// frame is taken to be its mean: a border of `pad` samples holds it, in storage type.  The model at
// the pixel centres is the separable filter (1/8, 3/4, 1/8), with the operations of bspline2 at a
// zero offset, so that a frame registered to itself matches bit for bit; it is written as a plain
// W x H level.  The first nsb blocks of a level make the model: a thread walks kSmoothRows rows down
// one column and carries the horizontal filter of the rows above and at the current one, so each
// output row reads one row of three taps; a tap in the border is the mean itself, so the model does
// not wait for the border.  The other blocks write the border, one sample a thread: the top and
// bottom bands first, then the left and right ones.
constexpr int kSmoothRows = 16, kFinishThreads = 128;
template <typename S>
__global__ void __launch_bounds__(kFinishThreads) pyr_finish(Levels<S> L, int pad, const LevelStat *means, int levels)
{
    const int l = blockIdx.y;
    const int W = L.W[l], H = L.H[l], pitch = L.pitch[l];
    S *lvl = L.lvl[l] + blockIdx.z * L.stride[l];
    const S edge = toS<S>(means[(size_t)blockIdx.z * levels + l].mean);
    if ((int)blockIdx.x >= L.nsb[l]) {
        const int bands = 2 * pad * pitch, sides = 2 * pad * H;
        const int t = ((int)blockIdx.x - L.nsb[l]) * kFinishThreads + threadIdx.x;
        if (t >= bands + sides) return;
        int r, c;
        if (t < bands) {
            const int q = t / pitch;                      // 0 .. 2 pad - 1
            r = q < pad ? q - pad : H + (q - pad);        // -pad .. -1, then H .. H + pad - 1
            c = t - q * pitch - pad;                      // -pad .. W + pad - 1
        } else {
            const int u = t - bands, q = u / H;           // 0 .. 2 pad - 1
            r = u - q * H;
            c = q < pad ? q - pad : W + (q - pad);
        }
        lvl[(ptrdiff_t)r * pitch + c] = edge;
        return;
    }
    const int by = (int)blockIdx.x / L.nxb[l], bx = (int)blockIdx.x - by * L.nxb[l];
    const int c = bx * kFinishThreads + threadIdx.x, r0 = by * kSmoothRows;
    if (c >= W) return;
    const float m = fromS(edge);
    const S *p = lvl + c;
    S *q = L.smooth[l] + blockIdx.z * L.sstride[l] + (size_t)r0 * W + c;
    // the horizontal filter of row r0 + k (k = -1 .. kSmoothRows)
    auto hrow = [&](int k) {
        const int r = r0 + k;
        const bool in = r >= 0 && r < H;
        const S *x = p + (ptrdiff_t)min(max(r, 0), H - 1) * pitch;
        const float t0 = in && c > 0 ? ldS<S>(x - 1) : m, t1 = in ? ldS<S>(x) : m, t2 = in && c + 1 < W ? ldS<S>(x + 1) : m;
        return fmaf(0.125f, t0 + t2, 0.75f * t1);
    };
    float a = hrow(-1), b = hrow(0);
#pragma unroll
    for (int k = 0; k < kSmoothRows; ++k) {
        if (r0 + k >= H) break;
        const float d = hrow(k + 1);
        q[(size_t)k * W] = toS<S>(fmaf(0.125f, a + d, 0.75f * b));
        a = b;
        b = d;
    }
}

// Row i of a level table (frame i / levels).
__device__ __forceinline__ void level_row(LevelDesc *tab, const LevelTable &t, const LevelStat *means, int i)
{
    const int f = i / t.levels, l = i - f * t.levels;
    LevelDesc d;
    d.ptr = t.raw[l] + (size_t)f * t.raw_stride[l];
    d.rptr = t.ref[l] + (size_t)f * t.ref_stride[l];
    d.W = t.W[l];
    d.H = t.H[l];
    d.pitch = t.pitch[l];
    d.rpitch = t.rpitch[l];
    d.mean = means[i].mean;
    d.sd = means[i].sd;
    tab[i] = d;
}

// Made on the device, the table costs a launch; with the means read back and the rows made by the host it
// cost two copies and two waits, of a 160x128 pair's call some 40 us.
__global__ void level_table_kernel(LevelDesc *tab, LevelTable t, const LevelStat *means, int rows)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < rows) level_row(tab, t, means, i);
}

cudaError_t launch_level_table(LevelDesc *tab, const LevelTable &t, const LevelStat *means, int frames, cudaStream_t s)
{
    const int rows = frames * t.levels;
    level_table_kernel<<<(rows + 127) / 128, 128, 0, s>>>(tab, t, means, rows);
    return cudaGetLastError();
}

__global__ void pair_setup_kernel(PairBlock *b, OpDesc op, double i0, double i1, double i2, LevelDesc *tab, LevelTable t,
                                  const LevelStat *means)
{
    if (threadIdx.x < 2 * t.levels) level_row(tab, t, means, threadIdx.x);
    unsigned *w = reinterpret_cast<unsigned *>(&b->stats);
    for (int i = threadIdx.x; i < (int)(sizeof(OpStats) / sizeof(unsigned)); i += blockDim.x) w[i] = 0u;
    if (threadIdx.x == 0) {
        b->theta[0] = b->theta[1] = b->theta[2] = 0.0;
        b->theta[3] = i0; b->theta[4] = i1; b->theta[5] = i2;
        b->status[0] = b->status[1] = b->status[2] = b->status[3] = 0;
        b->op = op;
        b->node0 = 0;
    }
}

cudaError_t launch_pair_setup(PairBlock *b, const OpDesc &op, const double *init3, LevelDesc *tab, const LevelTable &t,
                              const LevelStat *means, cudaStream_t s)
{
    pair_setup_kernel<<<1, 64, 0, s>>>(b, op, init3[0], init3[1], init3[2], tab, t, means);
    return cudaGetLastError();
}

// The level means of a freshly built pyramid into its rows of a level table.
__global__ void set_level_means_kernel(LevelDesc *tab, const LevelStat *means, int L)
{
    const int l = threadIdx.x;
    if (l < L) { tab[l].mean = means[l].mean; tab[l].sd = means[l].sd; }
}

cudaError_t launch_set_level_means(LevelDesc *tab, const LevelStat *means, int L, cudaStream_t s)
{
    set_level_means_kernel<<<1, 32, 0, s>>>(tab, means, L);
    return cudaGetLastError();
}

int pyramid_launches(int levels, bool means, int pad)
{
    return 1 + (levels > 2 ? levels - 2 : 0) + (means ? 1 : 0) + (pad > 0 ? 1 : 0);
}

template <typename S>
static cudaError_t pyramid_t(const float *frames, int N, size_t fstride, int W, int H, int pitch, int levels,
                             const PyrOut &o, LevelStat *means, cudaStream_t s)
{
    Levels<S> L = {};
    int w = W, h = H, most = 0;
    for (int l = 0; l < levels; ++l) {
        L.W[l] = w;
        L.H[l] = h;
        L.pitch[l] = level_pitch(w, o.pad);
        L.lvl[l] = (S *)o.raw[l] + level_origin(w, o.pad);
        L.stride[l] = o.raw_stride[l];
        L.smooth[l] = (S *)o.smooth[l];
        L.sstride[l] = o.smooth_stride[l];
        L.nxb[l] = (w + kFinishThreads - 1) / kFinishThreads;
        L.nsb[l] = L.smooth[l] ? L.nxb[l] * ((h + kSmoothRows - 1) / kSmoothRows) : 0;
        const int border = 2 * o.pad * (L.pitch[l] + h);
        const int nb = L.nsb[l] + (border + kFinishThreads - 1) / kFinishThreads;
        most = nb > most ? nb : most;
        w = (w + 1) / 2;
        h = (h + 1) / 2;
    }
    const dim3 top((W + kTopCols - 1) / kTopCols, (H + kTopRows - 1) / kTopRows, N);
    if (levels > 1)
        pyr_top<S, true><<<top, kTopThreads, 0, s>>>(frames, fstride, W, H, pitch, L.lvl[0], L.stride[0], L.pitch[0],
                                                     L.lvl[1], L.stride[1], L.pitch[1]);
    else
        pyr_top<S, false><<<top, kTopThreads, 0, s>>>(frames, fstride, W, H, pitch, L.lvl[0], L.stride[0], L.pitch[0],
                                                      nullptr, 0, 0);
    for (int l = 1; l + 1 < levels; ++l)
        pyr_down<S><<<dim3((L.W[l + 1] + kDnThreads - 1) / kDnThreads, (L.H[l + 1] + kDnRows - 1) / kDnRows, N),
                      kDnThreads, 0, s>>>(L.lvl[l], L.stride[l], L.pitch[l], L.W[l], L.H[l], L.lvl[l + 1],
                                          L.stride[l + 1], L.pitch[l + 1]);
    if (means) {
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3((unsigned)N * kMeanCtas, levels);
        lc.blockDim = dim3(32 * kMeanWarps);
        lc.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kMeanCtas;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        lc.attrs = attr;
        lc.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&lc, level_means<S>, L, means, levels);
        if (e != cudaSuccess) return e;
    }
    if (o.pad > 0) pyr_finish<S><<<dim3(most, levels, N), kFinishThreads, 0, s>>>(L, o.pad, means, levels);
    return cudaGetLastError();
}

cudaError_t launch_pyramid(const float *frames, int N, size_t fstride, int W, int H, int pitch, int levels,
                           int storage, const PyrOut &out, LevelStat *means, cudaStream_t s)
{
    if (out.pad != 0) {
        // the smoothed levels read the 3x3 window of a bordered level; the border holds the mean
        if (out.pad < 1 || !means) return cudaErrorInvalidValue;
    } else {
        for (int l = 0; l < levels; ++l)
            if (out.smooth[l]) return cudaErrorInvalidValue;
    }
    switch (storage) {
    case REG_F32: return pyramid_t<float>(frames, N, fstride, W, H, pitch, levels, out, means, s);
    case REG_BF16: return pyramid_t<__nv_bfloat16>(frames, N, fstride, W, H, pitch, levels, out, means, s);
    case REG_F16: return pyramid_t<__half>(frames, N, fstride, W, H, pitch, levels, out, means, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace reg
