// plan.cu -- device-side planning of Algorithm 2's per-box steps.
//
// plan_kernel (several CTAs per frame, each a slice of the frame's boxes), a warp per
// box: clip each box to its frame, classify it FAR or CLOSE by its larger side against
// tau_s (Sec. 4.3.4), map it to its matching grid (full resolution for FAR, the decimated
// grid for CLOSE), count its blocks, and select its occluders -- overlapping boxes of the
// same frame with a larger bottom y (Sec. 4.3.5), nearest (largest bottom y) first, at
// most max_occluders.  Boxes that are empty after clipping get their outputs here.  Then a
// warp per row of a box's block grid: the blocks' point grids and usable points; blocks
// with fewer than min_pts usable points are finished here, the others go to the work
// queue (large work first) and mark the census tiles their search can read.  All counts
// come from device memory so a captured graph replays with new inputs.
#include <math.h>

#include <algorithm>

#include "aggregate.cuh"
#include "ctm_internal.cuh"

namespace ctm {
namespace {

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__device__ __forceinline__ int4 clip_box(const ctm_box &b, int W, int H)
{
    int4 r;
    r.x = b.x0 < 0 ? 0 : b.x0;
    r.y = b.y0 < 0 ? 0 : b.y0;
    r.z = b.x1 > W ? W : b.x1;
    r.w = b.y1 > H ? H : b.y1;
    if (r.z <= r.x || r.w <= r.y) r = make_int4(0, 0, 0, 0);
    return r;
}

// Priority rule of Sec. 4.3.5: an occluder is frontal if its clipped box
// centre lies in the centred crop [W (1 - c) / 2, W (1 + c) / 2) x [H (1 - c) / 2,
// H (1 + c) / 2), compared on doubled coordinates in fp32.
__device__ __forceinline__ bool frontal(int4 q, int W, int H, float c)
{
    if (!(c > 0.0f)) return false;
    const float sx = (float)(q.x + q.z), sy = (float)(q.y + q.w);
    const float om = __fsub_rn(1.0f, c), op = __fadd_rn(1.0f, c);
    return sx >= __fmul_rn((float)W, om) && sx < __fmul_rn((float)W, op) && sy >= __fmul_rn((float)H, om) &&
           sy < __fmul_rn((float)H, op);
}

__device__ __forceinline__ bool overlaps(int4 a, int4 b)
{
    const int ix0 = max(a.x, b.x), ix1 = min(a.z, b.z);
    const int iy0 = max(a.y, b.y), iy1 = min(a.w, b.w);
    return ix1 > ix0 && iy1 > iy0;
}

constexpr int kStageBoxes = 1024;  // boxes of one frame staged in shared memory
constexpr int kKeyCache = 8;       // occluder keys per lane held in registers

constexpr int kPlanWarps = kPlanThreads / 32;

// A planned box and its occluders, for the warps that sample its rows.
struct PlannedBox {
    BoxPlan P;
    int4 occ[kMaxOcc];
};

// Mark the census row tiles of plane q that columns [c0, c1] of row y lie in.
__device__ __forceinline__ void mark_range(const MatchArgs &a, int f, int q, int y, int c0, int c1,
                                           int Ws, int Hs)
{
    if (y < 0 || y >= Hs) return;
    c0 = max(c0, 0);
    c1 = min(c1, Ws - 1);
    if (c1 < c0) return;
    const int t0 = c0 / kCensusTilePx, t1 = c1 / kCensusTilePx;
    uint32_t *row = a.ws.bitmap + (long long)f * a.ws.bm_frame_words + a.ws.bm_plane_off[q] +
                    (long long)y * a.ws.bm_row_words[q];
    for (int wi = t0 >> 5; wi <= (t1 >> 5); ++wi) {
        const int lo = max(t0 - wi * 32, 0), hi = min(t1 - wi * 32, 31);
        const uint32_t upto = hi == 31 ? 0xffffffffu : ((1u << (hi + 1)) - 1u);
        atomicOr(row + wi, upto & ~((1u << lo) - 1u));
    }
}

// Mark what the searches of neighbouring blocks of one grid row can read, whose sampled
// columns span [x_first, x_last]: the left plane at the sampled rows (lane m holds row
// m; plus the vertical spread of the backward pass) over [x_first - (dmax - dmin),
// x_last + (dmax - dmin)], which holds the points and every backward strip; the right
// plane at rows Y_m + dy over [x_first - dmax, x_last - dmin], which holds every forward
// strip and the backward queries.
__device__ __forceinline__ void mark_blocks(const MatchArgs &a, const BoxPlan &P, int ny, int Yl, int x_first,
                                            int x_last)
{
    const int lane = threadIdx.x & 31;
    const int qL = (P.far || a.p.close_factor == 1) ? 0 : 2;
    const int span = P.dmax - P.dmin;
    const int dyr = a.p.dy_max - a.p.dy_min;
    const int nl = 2 * dyr + 1, nr = dyr + 1;
    const int items = ny * (nl + nr);
    for (int it0 = 0; it0 < items; it0 += 32) {  // uniform trip count: the shuffle needs every lane
        const int it = it0 + lane;
        const int m = dyr == 0 ? (it >> 1) & 15 : (it < items ? it : 0) / (nl + nr);
        const int e = it - m * (nl + nr);
        const int y = __shfl_sync(0xffffffffu, Yl, m);
        if (it >= items) continue;
        if (e < nl)
            mark_range(a, P.frame, qL, y + e - dyr, x_first - span, x_last + span, P.Ws, P.Hs);
        else
            mark_range(a, P.frame, qL + 1, y + a.p.dy_min + (e - nl), x_first - P.dmax, x_last - P.dmin, P.Ws,
                       P.Hs);
    }
}

// Row gb of a box's block grid (FAR boxes: one row of one block), by a warp: a half-warp
// per block.  The row's blocks share the sampled rows, their occluded rows and mostly
// their census tiles.  Bound by its instructions (the point grids' divisions, the
// occluders, the records) and the census marks' atomics, of which neighbouring blocks
// with touching ranges make one set.
__device__ __forceinline__ void sample_row(const MatchArgs &a, const PlannedBox &planned, int box, int gb)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const BoxPlan P = planned.P;
    const int base = block_base(a, box) + gb * P.g;
    // the sampled rows; rows beyond ny repeat the last one (no point of theirs is usable)
    const int bw = P.sx1 - P.sx0, bh = P.sy1 - P.sy0;
    const int by0 = P.sy0 + div_small(gb * bh, P.g), by1 = P.sy0 + div_small((gb + 1) * bh, P.g);
    const int ny = min(by1 - by0, a.p.pts_side);
    const int Yl = ny > 0 ? point_coord(by0, by1, ny, min(lane, ny - 1)) : 0;
    // usable: left census defined (window inside the grid) and full-res position
    // k (x, y) in no kept occluder.  Each occluder covers a column range x a row range of
    // the point grid: lane q holds occluder q and the rows it covers.
    const int sxw = a.p.win_w >> 1, syw = a.p.win_h >> 1;
    const unsigned rowok = __ballot_sync(full, lane < ny && Yl - syw >= 0 && Yl + syw < P.Hs);
    int4 occ = make_int4(0, 0, 0, 0);
    if (lane < P.nocc) occ = planned.occ[lane];
    unsigned occrows = 0u;
    const int fy = lane < ny ? P.k * Yl : -1;
    for (int q = 0; q < P.nocc; ++q) {
        const int oy0 = __shfl_sync(full, occ.y, q), oy1 = __shfl_sync(full, occ.w, q);
        const unsigned rows = __ballot_sync(full, fy >= oy0 && fy < oy1);
        if (lane == q) occrows = rows;
    }
    const unsigned live = __ballot_sync(full, occrows != 0u);  // occluders that touch these rows
    const int nd = P.dmax - P.dmin + 1;
    const int ndy = a.p.dy_max - a.p.dy_min + 1;
    int work = 0;  // lane ga: usable points x candidates of a searchable block, else 0
    int m0 = 1, m1 = 0;  // columns of the blocks not marked yet (none)
    const int half = lane >> 4, hl = lane & 15;
    const int Yh = __shfl_sync(full, Yl, hl);
    for (int ga0 = 0; ga0 < P.g; ga0 += 2) {
        const int ga = ga0 + half;  // this half-warp's block, its lanes the block's columns
        const bool on = ga < P.g;
        const int bx0 = P.sx0 + div_small(ga * bw, P.g), bx1 = P.sx0 + div_small((ga + 1) * bw, P.g);
        const int nx = on ? min(bx1 - bx0, a.p.pts_side) : 0;
        const int Xl = nx > 0 ? point_coord(bx0, bx1, nx, min(hl, nx - 1)) : 0;
        unsigned colmask = hl < nx && Xl - sxw >= 0 && Xl + sxw < P.Ws ? rowok : 0u;
        const int fx = P.k * Xl;
        for (unsigned o = live; o; o &= o - 1u) {
            const int q = __ffs(o) - 1;
            const int ox0 = __shfl_sync(full, occ.x, q), ox1 = __shfl_sync(full, occ.z, q);
            const unsigned rows = __shfl_sync(full, occrows, q);
            if (fx >= ox0 && fx < ox1) colmask &= ~rows;
        }
        const int cnt = __popc(colmask);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < kMaxPtsSide; o <<= 1) {
            const int y = __shfl_up_sync(full, incl, o, kMaxPtsSide);
            if (hl >= o) incl += y;
        }
        const int n_valid = __shfl_sync(full, incl, 15, kMaxPtsSide);
        const int x_first = __shfl_sync(full, Xl, 0, kMaxPtsSide), x_last = __shfl_sync(full, Xl, 15, kMaxPtsSide);
        // column chunks whose strip (plus alignment) fits the popcount matchers' strip
        unsigned cstart = 1u;
        if (__any_sync(full, x_last - x_first + nd + 2 > a.strip_cols)) {
            int x0 = x_first;
            for (int j = 1; j < kMaxPtsSide; ++j) {
                const int xj = __shfl_sync(full, Xl, j, kMaxPtsSide);
                if (j < nx && xj - x0 + nd + 2 > a.strip_cols) {
                    cstart |= 1u << j;
                    x0 = xj;
                }
            }
        }
        const bool few = n_valid < a.p.min_pts;
        if (on) {
            BlockGeom *g = a.ws.geom + (base + ga);
            g->X[hl] = (int16_t)Xl;
            g->Y[hl] = (int16_t)Yh;
            g->colmask[hl] = (uint16_t)colmask;
            g->colprefix[hl] = (uint16_t)(incl - cnt);
            if (hl == 0) {
                g->n_valid = n_valid;
                g->nx = nx;
                g->ny = ny;
                g->cstart = cstart;
                g->box = box;
                g->slot = gb * P.g + ga;
                g->frame = P.frame;
                g->k = P.k;
                g->far = P.far;
                g->dmin = P.dmin;
                g->dmax = P.dmax;
                g->Ws = P.Ws;
                g->Hs = P.Hs;
                if (few) {
                    ctm_block rec;
                    rec.n_pts = nx * ny;
                    rec.n_valid = n_valid;
                    rec.d_f = rec.dy_f = rec.d_b = rec.dy_b = 0;
                    rec.s_m = rec.s_0 = rec.s_p = 0;
                    rec.d_sub = 0.0f;
                    rec.d_full = 0.0f;
                    rec.flags = CTM_BLK_PRESENT | CTM_BLK_FEW_POINTS;
                    write_block(a, box, gb * P.g + ga, rec);
                }
            }
        }
        const unsigned found = __ballot_sync(full, on && !few);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!((found >> (16 * h)) & 1u)) continue;
            const int nv = __shfl_sync(full, n_valid, 16 * h);
            if (lane == ga0 + h) work = nv * nd * ndy;
            // census demand: joined with the searchable block before it where the ranges touch
            const int xf = __shfl_sync(full, x_first, 16 * h), xl = __shfl_sync(full, x_last, 16 * h);
            if (m0 <= m1 && xf - m1 > nd) {
                mark_blocks(a, P, ny, Yl, m0, m1);
                m0 = 1;
                m1 = 0;
            }
            if (m0 > m1) m0 = xf;
            m1 = xl;
        }
    }
    if (m0 <= m1) mark_blocks(a, P, ny, Yl, m0, m1);
    // queue the searchable blocks, one reservation per end for the whole row
    const unsigned big = __ballot_sync(full, work >= kBigWork), small = __ballot_sync(full, work > 0 && work < kBigWork);
    int qb = 0, qs = 0;
    if (lane == 0 && big) qb = atomicAdd(&a.ws.counts->n_big, __popc(big));
    if (lane == 0 && small) qs = atomicAdd(&a.ws.counts->n_small, __popc(small));
    qb = __shfl_sync(full, qb, 0);
    qs = __shfl_sync(full, qs, 0);
    const unsigned lt = (1u << lane) - 1u;
    if (work >= kBigWork)
        a.ws.queue[qb + __popc(big & lt)] = base + lane;
    else if (work > 0)
        a.ws.queue[a.caps.max_blocks - 1 - qs - __popc(small & lt)] = base + lane;
}

// S CTAs per frame, each a slice of the frame's boxes.  First a warp plans a box: clip,
// classify, map to the matching grid, select its occluders (the frame's clipped boxes are
// staged in shared memory for the pairwise test).  Then the warps take the rows of the
// planned boxes' block grids.  Block slot s of box i is block i * grid_g^2 + s, so
// nothing is counted across CTAs.  Bound by latency (one box's occluder rounds, then one
// row); the sampling was a kernel of its own, a warp per row with plans and occluders
// through memory: both 13.4 -> 6.8 us on four boxes, 15.8 -> 9.1 on four 720p frames; a
// 1279x719 frame 47.9 -> 44.9 us a call, four 720p frames 58.1 -> 56.5, eight 4K frames
// 294.8 -> 291.5.  64 registers a thread: at the 122 it takes freely, two CTAs an SM, the
// 4K frames lose it again (293.4).
__global__ void __launch_bounds__(kPlanThreads, 4) plan_kernel(MatchArgs a, int S)
{
    __shared__ int4 sbox[kStageBoxes];
    __shared__ PlannedBox planned[kPlanWarps];
    const int f = blockIdx.x / S, slice = blockIdx.x % S;
    const int nf = a.frames ? clampi(a.counts_in[0], 0, a.caps.max_frames) : 1;
    const int nb_total = clampi(a.frames ? a.counts_in[1] : a.n_boxes1, 0, a.caps.max_boxes);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (blockIdx.x == 0 && tid == 0) {
        a.ws.counts->n_frames = nf;
        a.ws.counts->n_boxes = nb_total;
        a.ws.counts->error = 0;  // the previous call's flag stays until here (see aggregate_kernel)
    }
    if (f >= nf) return;
    const ctm_frame fr = a.frames ? a.frames[f] : a.frame1;
    const bool bad_frame = fr.width < 1 || fr.height < 1 || fr.width > a.caps.max_width ||
                           fr.height > a.caps.max_height || fr.pitch < fr.width ||
                           fr.left == nullptr || fr.right == nullptr;
    if (slice == 0 && tid < 4) {  // census plane descriptors of this frame: L1, R1, Lk, Rk
        PlaneDesc d;
        const int q = tid;
        d.img = (q & 1) ? fr.right : fr.left;
        d.W = fr.width;
        d.H = fr.height;
        d.pitch = fr.pitch;
        d.k = q < 2 ? 1 : a.p.close_factor;
        d.Ws = ceil_div_nn(fr.width, d.k);
        d.Hs = ceil_div_nn(fr.height, d.k);
        uint64_t *cb = a.ws.census + (long long)f * a.ws.frame_stride;
        d.out = q < 2 ? cb + q * a.ws.plane1_elems : cb + 2 * a.ws.plane1_elems + (q - 2) * a.ws.planek_elems;
        d.opitch = (int)(q < 2 ? a.ws.pitch1 : a.ws.pitchk);
        d.vec_load = (d.k == 1 || d.k == 2) && (fr.pitch % 4 == 0) &&
                     ((reinterpret_cast<uintptr_t>(d.img) & 7u) == 0);
        a.ws.planes[f * 4 + q] = d;
    }
    const int begin = clampi(fr.box_begin, 0, nb_total);
    const int end = clampi(fr.box_begin + fr.box_count, begin, nb_total);
    const int nloc = end - begin;
    const bool staged = nloc <= kStageBoxes;
    if (staged)
        for (int t = tid; t < nloc; t += blockDim.x) sbox[t] = clip_box(a.boxes[begin + t], fr.width, fr.height);
    __syncthreads();
    const ctm_params &p = a.p;
    const int K = p.max_occluders < kMaxOcc ? p.max_occluders : kMaxOcc;
    // this CTA's slice of the frame's boxes, as many at a time as it has warps
    const int per = (nloc + S - 1) / S;
    const int sb = begin + min(slice * per, nloc), se = begin + min((slice + 1) * per, nloc);

    for (int i0 = sb; i0 < se; i0 += kPlanWarps) {
        // a warp per box
        const int i = i0 + warp;
        if (i < se) {
            const int4 r = staged ? sbox[i - begin] : clip_box(a.boxes[i], fr.width, fr.height);
            const int w = r.z - r.x, h = r.w - r.y;
            const int side = w > h ? w : h;
            const int far = side < p.far_side_px ? 1 : 0;
            const int k = far ? 1 : p.close_factor;
            BoxPlan P;
            P.cx0 = r.x; P.cy0 = r.y; P.cx1 = r.z; P.cy1 = r.w;
            // decimated pixel x belongs to the box iff its source pixel k x does
            P.sx0 = ceil_div_nn(r.x, k); P.sx1 = ceil_div_nn(r.z, k);
            P.sy0 = ceil_div_nn(r.y, k); P.sy1 = ceil_div_nn(r.w, k);
            P.frame = f;
            P.far = far;
            P.k = k;
            P.g = far ? 1 : p.grid_g;
            P.dmin = far ? p.far_dmin : p.close_dmin;
            P.dmax = far ? p.far_dmax : p.close_dmax;
            P.Ws = ceil_div_nn(fr.width, k);
            P.Hs = ceil_div_nn(fr.height, k);
            P.fb = __fmul_rn(fr.f_px, fr.baseline_m);
            const bool empty = bad_frame || w <= 0 || h <= 0 || P.sx1 <= P.sx0 || P.sy1 <= P.sy0;
            P.nblk = empty ? 0 : P.g * P.g;

            // occluders: overlap with positive area and strictly larger bottom y; keep
            // K of them: frontal ones first (frontal_crop > 0), then by largest bottom
            // y, ties to the lower index.  Key (frontal, bottom y, -index) is unique
            // per box, so round t takes the largest key below round t-1's: each lane
            // scans its share of the frame's boxes.
            // key of box j as an occluder of box i (0: it is not one)
            auto occ_key = [&](int j) -> unsigned long long {
                if (j >= end || j == i) return 0ull;
                const int4 q = staged ? sbox[j - begin] : clip_box(a.boxes[j], fr.width, fr.height);
                if (!(q.w > r.w) || !overlaps(r, q)) return 0ull;
                const unsigned front = frontal(q, fr.width, fr.height, p.frontal_crop) ? 0x80000000u : 0u;
                return ((unsigned long long)(front | (unsigned)q.w) << 32) | (unsigned)(0x7fffffff - (j - begin));
            };
            int nocc = 0;
            int4 occ = make_int4(0, 0, 0, 0);  // lane q: occluder q
            if (!empty && K > 0) {
                // frames of up to 32 * kKeyCache boxes keep every lane's keys in registers,
                // so a round is a register scan and two warp reductions
                const bool cached = nloc <= 32 * kKeyCache;
                unsigned long long kc[kKeyCache];
#pragma unroll
                for (int u = 0; u < kKeyCache; ++u) kc[u] = cached ? occ_key(begin + lane + 32 * u) : 0ull;
                unsigned long long prev = ~0ull;
                for (; nocc < K; ++nocc) {
                    unsigned long long best = 0ull;
                    if (cached) {
#pragma unroll
                        for (int u = 0; u < kKeyCache; ++u)
                            if (kc[u] < prev && kc[u] > best) best = kc[u];
                    } else {
                        for (int j = begin + lane; j < end; j += 32) {
                            const unsigned long long key = occ_key(j);
                            if (key < prev && key > best) best = key;
                        }
                    }
                    // warp maximum of the 64-bit keys (two 32-bit reductions)
                    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32));
                    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32) == hi ? (unsigned)best : 0u);
                    best = ((unsigned long long)hi << 32) | lo;
                    if (best == 0ull) break;
                    prev = best;
                    if (lane == nocc) {
                        const int j = begin + (0x7fffffff - (int)lo);
                        occ = staged ? sbox[j - begin] : clip_box(a.boxes[j], fr.width, fr.height);
                    }
                }
            }
            P.nocc = nocc;
            if (lane == 0) {
                if (P.nblk == 0) {
                    a.disp[i] = __int_as_float(0x7fc00000);
                    a.depth[i] = __int_as_float(0x7fc00000);
                    a.flags[i] = (uint8_t)((far ? CTM_BOX_FAR : 0) | CTM_BOX_EMPTY);
                } else if (atomicCAS(a.ws.nblk + i, 0, P.nblk) == 0) {
                    a.ws.plans[i] = P;
                    atomicAdd(&a.ws.counts->n_blocks, P.nblk);
                } else {
                    P.nblk = 0;  // frames whose boxes overlap: the box is another frame's
                }
                planned[warp].P = P;
            }
            planned[warp].occ[lane] = occ;
        }
        __syncthreads();
        // a warp per row of their block grids
        const int rows = a.p.grid_g, n = min(se - i0, kPlanWarps);
        for (int t = warp; t < n * rows; t += kPlanWarps) {
            const int q = t / rows, gb = t - q * rows;
            if (planned[q].P.nblk > 0 && gb < planned[q].P.g) sample_row(a, planned[q], i0 + q, gb);
        }
        __syncthreads();
    }
}

}  // namespace

// One warp per planned box with blocks: Sec. 4.3.4 over its block records and
// Eq. 1 (boxes without blocks got their outputs from the planner).
//
// When a bounded wait of the matching kernel expired (counts->error), some
// blocks were never searched and their records are stale, so no box with
// blocks is aggregated: each gets NaN disparity and depth and flags 0 (neither
// VALID nor any reason bit), and the call's status says why.
//
// It is the last kernel of a call, so it also leaves the workspace ready for
// the next one: block 0 moves the counters to the stats record and zeroes
// them -- all but the error flag, which every CTA reads here and the next
// call's plan_kernel clears -- and every box's block count goes back to zero (no memset nodes at the start of a call).
__global__ void __launch_bounds__(256) aggregate_kernel(MatchArgs a)
{
    __shared__ float scratch[8][2 * kMaxSlots];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int failed = *reinterpret_cast<volatile int *>(&a.ws.counts->error);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const Counts c = *a.ws.counts;
        if (a.stats_accumulate) {  // a later sub-batch of one call
            Counts t = *a.ws.stats;
            t.n_frames += c.n_frames;
            t.n_boxes += c.n_boxes;
            t.n_blocks += c.n_blocks;
            t.queue_head += c.queue_head;
            t.error |= c.error;
            t.evals += c.evals;
            t.n_big += c.n_big;
            t.n_small += c.n_small;
            t.n_tiles += c.n_tiles;
            t.n_units += c.n_units;
            t.host_bytes += c.host_bytes;
            *a.ws.stats = t;
        } else {
            *a.ws.stats = c;
        }
        Counts z{};
        z.error = c.error;  // unchanged: other CTAs read it
        *a.ws.counts = z;
    }
    const int box = blockIdx.x * 8 + warp;
    if (box >= clampi(a.frames ? a.counts_in[1] : a.n_boxes1, 0, a.caps.max_boxes)) return;
    if (a.ws.nblk[box] == 0) return;
    if (failed) {
        if (lane == 0) {
            a.disp[box] = __int_as_float(0x7fc00000);
            a.depth[box] = __int_as_float(0x7fc00000);
            a.flags[box] = 0;
        }
    } else {
        aggregate_box(a, box, scratch[warp], lane);
    }
    __syncwarp();
    if (lane == 0) a.ws.nblk[box] = 0;
}

cudaError_t launch_aggregate(const MatchArgs &a, cudaStream_t s)
{
    aggregate_kernel<<<ceil_div_nn(a.caps.max_boxes, 8), 256, 0, s>>>(a);
    return cudaGetLastError();
}

// The counters and block counts start at zero: the workspace is created zeroed
// and every call's aggregate_kernel zeroes them again.  Two boxes a CTA at the context's
// capacity (their rows then fill its warps; with four a 1279x719 frame takes 49.3 us, with
// one 32 frames of 1920x1200 221.8 instead of 218.9), 4 to 64 CTAs per frame.
cudaError_t launch_plan(const MatchArgs &a, cudaStream_t s)
{
    const int nf = std::max(a.caps.max_frames, 1);
    const int slices = std::min(std::max(ceil_div_nn(a.caps.max_boxes, 2 * nf), 4), 64);
    plan_kernel<<<nf * slices, kPlanThreads, 0, s>>>(a, slices);
    return cudaGetLastError();
}

}  // namespace ctm
