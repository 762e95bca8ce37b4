// rect.cu -- Sec. 5.1 auto-rectification offset, with census matching in place
// of block matching: for every vertical offset delta and every ROI pixel, the
// winner-take-all disparity of the left pixel read delta rows lower, checked by
// the backward search; the offset with the most consistent disparities above a
// threshold wins.  Not on the per-frame path; run now and then on a stream of
// its own.  Also the temporal filter of the per-frame estimates (host code).
#include <cuda_runtime.h>
#include <stdlib.h>

#include <algorithm>
#include <vector>

#include "ctm_internal.cuh"

namespace ctm {
namespace {

__device__ __forceinline__ uint64_t code_or_zero(const uint64_t *C, long long pitch, int W, int H, int x, int y)
{
    return (x >= 0 && x < W && y >= 0 && y < H) ? __ldg(C + (long long)y * pitch + x) : 0ull;
}

constexpr int kRectThreads = 128;

// Thread per ROI pixel of one row and one offset (grid: x tiles, rows, offsets).
// The CTA stages the two code rows its pixels search: the right row y over
// columns x0 - dmax .. x0 + 127 - dmin (forward candidates x - d) and the left
// row y + delta over x0 + dmin - dmax .. x0 + 127 + dmax - dmin (backward
// candidates x - d_f + d for any d_f), codes outside the image as 0.  Each scan
// keeps the first minimum as the least key (cost << 11 | candidate index).
__global__ void __launch_bounds__(kRectThreads) rect_kernel(const uint64_t *CL, const uint64_t *CR, long long pitch,
                                                            int W, int H, int sx, int sy, int rx0, int rx1, int ry0,
                                                            int dmin, int dmax, int delta_min, int d_thresh,
                                                            int fb_tol, unsigned long long *counts)
{
    extern __shared__ uint64_t rect_smem[];
    const int nd = dmax - dmin + 1;
    const int x0 = rx0 + blockIdx.x * kRectThreads;
    const int x = x0 + threadIdx.x;
    const int y = ry0 + blockIdx.y;
    const int delta = delta_min + blockIdx.z;
    const int yl = y + delta;
    uint64_t *rrow = rect_smem;                     // columns x0 - dmax + i
    uint64_t *lrow = rect_smem + kRectThreads + nd;  // columns x0 + dmin - dmax + i
    const int nr = kRectThreads + nd - 1, nl = kRectThreads + 2 * (nd - 1);
    for (int i = threadIdx.x; i < nr; i += kRectThreads) rrow[i] = code_or_zero(CR, pitch, W, H, x0 - dmax + i, y);
    for (int i = threadIdx.x; i < nl; i += kRectThreads)
        lrow[i] = code_or_zero(CL, pitch, W, H, x0 + dmin - dmax + i, yl);
    __syncthreads();
    bool hit = false;
    if (x < rx1 && x - sx >= 0 && x + sx < W && yl - sy >= 0 && yl + sy < H) {
        const int t = threadIdx.x;
        const uint64_t cl = lrow[t + dmax - dmin];  // column x
        unsigned kf = 0xffffffffu;
        for (int i = 0; i < nd; ++i)  // candidate d = dmin + i at column x - d: rrow[t + dmax - d]
            kf = min(kf, ((unsigned)__popcll(cl ^ rrow[t + nd - 1 - i]) << 11) | (unsigned)i);
        const int i_f = (int)(kf & 2047u);
        const uint64_t cq = rrow[t + nd - 1 - i_f];   // column x - d_f
        const int b0 = t + nd - 1 - i_f;              // lrow index of column x - d_f + dmin
        unsigned kb = 0xffffffffu;
        for (int i = 0; i < nd; ++i) kb = min(kb, ((unsigned)__popcll(cq ^ lrow[b0 + i]) << 11) | (unsigned)i);
        const int d_f = dmin + i_f, d_b = dmin + (int)(kb & 2047u);
        hit = abs(d_b - d_f) <= fb_tol && d_f > d_thresh;
    }
    const int n = __syncthreads_count(hit);
    if (threadIdx.x == 0 && n) atomicAdd(counts + blockIdx.z, (unsigned long long)n);
}

// The same counts from one pass over the costs.  The backward cost of a right pixel
// x_r at d' is the forward cost of the left pixel x_r + d' at d', so both minima are
// minima over one band of costs, c(x_l, d) = popcount(C_L(x_l) ^ C_R(x_l - d)): the
// forward one along d, the backward one along x_l at fixed x_r = x_l - d.  A warp
// walks d for 32 kBandGroups consecutive left pixels; the running backward minimum of
// a right pixel moves one lane up per step (x_r = x_l - d stays), enters at the lowest
// lane and leaves at the highest into shared memory.  The left pixels reach nd - 1
// beyond the CTA's pixels on both sides, so that every right pixel they match has all
// its candidates: (n + 2 nd - 2) nd costs instead of 2 n nd, half for a wide segment.
// Half the population counts (the bound of rect_kernel, at 0.72 of their peak; 0.70 here)
// for one shuffle, select and minimum more a cost.  A 1920x128 band of a 1920x1200
// pair, 64 disparities, 9 offsets: the call 0.156 -> 0.100 ms, 0.088 of it this kernel;
// the census of both images' band rows is one launch of 8 us (0.106 ms with two).
constexpr int kBandThreads = 256;
constexpr int kBandGroups = 2;       // 32-pixel groups per warp step
constexpr int kBandPixels = 2048;    // pixels of a CTA's segment

// The band is taken where a segment holds three ranges of disparities.
constexpr int kBandRatio = 3;

// Shared memory of a segment of w pixels.
constexpr size_t band_smem_bytes(int w, int ndisp)
{
    return (size_t)12 * (w + 3 * ndisp + 32 * kBandGroups) + sizeof(unsigned) * (size_t)w;
}
// of the widest segment and the longest range it is taken for: the limit every call sets,
// so that no call's is below what another thread's launch needs
constexpr size_t kBandSmemMax = band_smem_bytes(kBandPixels, kBandPixels / kBandRatio);
static_assert(kBandSmemMax <= 227 * 1024, "shared memory of a CTA");
static_assert(sizeof(uint64_t) * (2 * kRectThreads + 3 * 1024) <= 48 * 1024, "rect_kernel needs no raised limit");

__global__ void __launch_bounds__(kBandThreads) rect_band_kernel(const uint64_t *CL, const uint64_t *CR,
                                                                 long long pitch, int W, int H, int sx, int sy,
                                                                 int rx0, int rx1, int ry0, int dmin, int dmax,
                                                                 int delta_min, int d_thresh, int fb_tol,
                                                                 unsigned long long *counts)
{
    extern __shared__ uint64_t rect_smem[];
    const unsigned full = 0xffffffffu;
    const int nd = dmax - dmin + 1;
    const int xs = rx0 + blockIdx.x * kBandPixels, xe = min(xs + kBandPixels, rx1);
    const int y = ry0 + blockIdx.y, yl = y + delta_min + (int)blockIdx.z;
    if (yl - sy < 0 || yl + sy >= H) return;  // no left pixel of this row is defined
    constexpr int kStep = 32 * kBandGroups;
    const int a0 = xs - (nd - 1);                                    // first left pixel
    const int steps = (xe - xs + 2 * (nd - 1) + kStep - 1) / kStep;  // warp steps of kStep left pixels
    const int n_l = steps * kStep, n_r = n_l + nd - 1;               // right pixels: a0 - dmax + i
    uint64_t *rrow = rect_smem;
    unsigned *bkey = reinterpret_cast<unsigned *>(rrow + n_r);
    unsigned *fkey = bkey + n_r;
    for (int i = threadIdx.x; i < n_r; i += kBandThreads) {
        rrow[i] = code_or_zero(CR, pitch, W, H, a0 - dmax + i, y);
        bkey[i] = full;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int st = warp; st < steps; st += kBandThreads / 32) {
        uint32_t lo[kBandGroups], hi[kBandGroups];
        unsigned kf[kBandGroups], acc[kBandGroups];
        const int i0 = st * kStep;  // index of the step's first left pixel
#pragma unroll
        for (int g = 0; g < kBandGroups; ++g) {
            const uint64_t c = code_or_zero(CL, pitch, W, H, a0 + i0 + 32 * g + lane, yl);
            lo[g] = (uint32_t)c;
            hi[g] = (uint32_t)(c >> 32);
            kf[g] = acc[g] = full;
        }
        const uint64_t *rp = rrow + (i0 + lane + nd - 1);  // candidate i of group g: rp[32 g - i]
#pragma unroll 4
        for (int i = 0; i < nd; ++i) {
#pragma unroll
            for (int g = 0; g < kBandGroups; ++g) {
                const uint64_t r = rp[32 * g - i];
                const unsigned k = (unsigned)(__popc(lo[g] ^ (uint32_t)r) + __popc(hi[g] ^ (uint32_t)(r >> 32))) << 11;
                kf[g] = min(kf[g], k + (unsigned)i);
                acc[g] = min(acc[g], k + (unsigned)i);
            }
            // the right pixel of the step's last left pixel leaves, the others move up
            if (lane == 31) atomicMin(bkey + (i0 + kStep - 1 + nd - 1 - i), acc[kBandGroups - 1]);
            unsigned up[kBandGroups];
#pragma unroll
            for (int g = 0; g < kBandGroups; ++g) up[g] = __shfl_sync(full, acc[g], (lane + 31) & 31);
#pragma unroll
            for (int g = 0; g < kBandGroups; ++g) acc[g] = lane ? up[g] : (g ? up[g - 1] : full);
        }
        // after the last step the pixels that have not left sit one lane up
#pragma unroll
        for (int g = 0; g < kBandGroups; ++g) {
            atomicMin(bkey + (i0 + 32 * g + lane - 1 < 0 ? 0 : i0 + 32 * g + lane - 1), acc[g]);
            const int x = a0 + i0 + 32 * g + lane;
            if (x >= xs && x < xe) fkey[x - xs] = kf[g];
        }
    }
    __syncthreads();
    int hits = 0;
    for (int i = threadIdx.x; i < xe - xs; i += kBandThreads) {
        const int x = xs + i;
        if (x - sx < 0 || x + sx >= W) continue;
        const int i_f = (int)(fkey[i] & 2047u);
        const int i_b = (int)(bkey[x - a0 + nd - 1 - i_f] & 2047u);
        hits += abs(i_b - i_f) <= fb_tol && dmin + i_f > d_thresh;
    }
    hits = __reduce_add_sync(full, hits);
    if (lane == 0 && hits) atomicAdd(counts + blockIdx.z, (unsigned long long)hits);
}

// First offset with the largest count.
__global__ void rect_argmax_kernel(const unsigned long long *counts, int n, int delta_min, int *delta_out)
{
    if (threadIdx.x != 0) return;
    int best = 0;
    for (int i = 1; i < n; ++i)
        if (counts[i] > counts[best]) best = i;
    *delta_out = delta_min + best;
}

}  // namespace
}  // namespace ctm

using namespace ctm;

// The part of an image that the census of its rows [y0, y1) (clipped to it) reads: it
// starts at an even row, so that its rows stay word-aligned.  Rows of that part outside
// [y0, y1) get codes no one reads.  False: no rows.
static bool census_part(const ctm_params &p, const uint8_t *img, int width, int height, int pitch, long long y0,
                        long long y1, uint64_t *codes, ctm::CensusImage *part)
{
    const int sy = p.win_h / 2;
    const long long a = std::max(y0 - sy, 0ll) & ~1ll, b = std::min(y1 + sy, (long long)height);
    if (b <= a) return false;
    *part = ctm::CensusImage{img + a * pitch, width, (int)(b - a), codes + a * width};
    return true;
}

extern "C" int ctm_auto_rect(const ctm_params *p, const uint8_t *left_dev, const uint8_t *right_dev, int width,
                             int height, int pitch, int rx0, int ry0, int rx1, int ry1, int dmin, int dmax,
                             int delta_min, int delta_max, int d_thresh, int fb_tol, uint64_t *census_dev,
                             unsigned long long *counts_dev, int *delta_dev, ctm_stream stream)
{
    if (!p || !left_dev || !right_dev || !census_dev || !counts_dev || !delta_dev) return CTM_EINVAL;
    if (width < 1 || height < 1 || pitch < width || dmin > dmax || dmax - dmin + 1 > 1024 ||
        delta_min > delta_max || delta_max - delta_min + 1 > 65535 || fb_tol < 0)
        return CTM_EINVAL;
    if (p->win_w < 1 || p->win_h < 1 || (p->win_w & 1) == 0 || (p->win_h & 1) == 0 || p->win_w > kMaxWin ||
        p->win_h > kMaxWin || p->win_w * p->win_h + (p->sentinel ? 1 : 0) > 64)
        return CTM_EINVAL;
    rx0 = std::max(rx0, 0);
    ry0 = std::max(ry0, 0);
    rx1 = std::min(rx1, width);
    ry1 = std::min(ry1, height);
    cudaStream_t s = (cudaStream_t)stream;
    const int nd = delta_max - delta_min + 1;
    const long long cpitch = width;  // census planes: width codes per row, left then right
    uint64_t *CL = census_dev, *CR = census_dev + (long long)width * height;
    cudaError_t e = cudaMemsetAsync(counts_dev, 0, sizeof(unsigned long long) * nd, s);
    if (e == cudaSuccess && rx1 > rx0 && ry1 > ry0) {
        // the rows the search reads: the ROI's on the right, moved by every offset on the left
        CensusImage parts[2];
        int n = 0;
        n += census_part(*p, left_dev, width, height, pitch, (long long)ry0 + delta_min, (long long)ry1 + delta_max, CL,
                         parts + n);
        n += census_part(*p, right_dev, width, height, pitch, ry0, ry1, CR, parts + n);
        if (n > 0) e = launch_census_images(parts, n, pitch, 1, p->win_w, p->win_h, p->sentinel, cpitch, s);
        const int ndisp = dmax - dmin + 1, w = rx1 - rx0;
        // one band of costs for both searches where the pixels are wide enough against the
        // nd - 1 pixels it adds on both sides: (w + 2 nd) nd costs against 2 w nd, equal at
        // two ranges, so from three on
        if (e == cudaSuccess && std::min(w, kBandPixels) >= kBandRatio * ndisp) {
            const dim3 grid((w + kBandPixels - 1) / kBandPixels, ry1 - ry0, nd);
            const size_t smem = band_smem_bytes(std::min(w, kBandPixels), ndisp);
            e = cudaFuncSetAttribute(rect_band_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBandSmemMax);
            if (e == cudaSuccess)
                rect_band_kernel<<<grid, kBandThreads, smem, s>>>(CL, CR, cpitch, width, height, p->win_w / 2,
                                                                  p->win_h / 2, rx0, rx1, ry0, dmin, dmax, delta_min,
                                                                  d_thresh, fb_tol, counts_dev);
        } else if (e == cudaSuccess) {
            const dim3 grid((w + kRectThreads - 1) / kRectThreads, ry1 - ry0, nd);
            const size_t smem = sizeof(uint64_t) * (size_t)(2 * kRectThreads + 3 * ndisp);
            rect_kernel<<<grid, kRectThreads, smem, s>>>(CL, CR, cpitch, width, height, p->win_w / 2, p->win_h / 2,
                                                         rx0, rx1, ry0, dmin, dmax, delta_min, d_thresh, fb_tol,
                                                         counts_dev);
        }
        e = e == cudaSuccess ? cudaGetLastError() : e;
    }
    if (e == cudaSuccess) {
        rect_argmax_kernel<<<1, 32, 0, s>>>(counts_dev, nd, delta_min, delta_dev);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? CTM_OK : CTM_ECUDA;
}

extern "C" int ctm_rect_filter(const int *estimates, int n, int prev, int max_step)
{
    if (!estimates || n < 1) return prev;
    if (max_step < 0) max_step = 0;
    std::vector<int> v(estimates, estimates + n);
    std::sort(v.begin(), v.end());
    const int med = v[(n - 1) / 2];
    const int step = std::min(std::max(med - prev, -max_step), max_step);
    return prev + step;
}
