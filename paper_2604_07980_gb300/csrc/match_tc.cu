// match_tc.cu -- the Hamming-cost search of Algorithm 2 on the tensor cores (the
// matcher of every call but the plain per-box path, match.cu, and the two-pass
// variant, match_pipe.cu).
//
// Why a product: with the points (j, m) of a block (column X_j, row Y_m) and x a column
// of the searched strip,
//     D[x][j] = sum over rows m and code bits b of r(x, m, b) l(j, m, b)
// is a (strip columns) x 16 x (16 rows * 64 bits) contraction, and the cost of a
// candidate is one diagonal of it, S(d) = K0 + sum_j D[X_j - d][j] / 2.  Every strip
// code is then read and unpacked once per pass instead of once per point column (16
// times), and the xors and population counts (16 per SM clock; the popcount kernel ran
// at 0.6 of that pipe's peak with two thirds of the issue slots taken) go to
// tcgen05.mma.  Measured here, per SM clock: kind::mxf4, M 128, N 16, K 64, A in tensor
// memory, one per 15 clocks with four CTAs (59 in one dependent chain); f8f6f4 the same
// per instruction at half the K; mma.sync fp8 runs as two fp16 products with
// conversions, b1 and s4 are emulated, s8 is a quarter of fp16's rate.
//
// Operands, exact in e2m1 with unit scales: bit p (0 .. 2) of a nibble of a strip code
// word alone is 0 or 2^(p-1), so a bit plane is one AND; bit 3, the sign, over the
// constant 1.0 is +-1.  The point side holds s 2^(2-p), s = 1 - 2 l, so a product is
// 2 r s; with r = (1 - v) / 2 for the sign plane its operand is -s.  Then
// popc(l ^ r) = l + r s summed, K0 = sum over usable points of popc(l without the
// sign plane) + 8; unusable points have operand 0.  A code's 64 values are one row's K,
// in the same order on both sides.  |D| <= 1792, whole numbers: the fp32 sums are exact.
//
// Work split.  A worker holds one block: four builder warps -- thread x is strip column
// x: it reads the column's code of each sampled row from the strip (staged by
// tile::gather4), unpacks it (8 logic instructions) and stores the 8 words to its
// tensor-memory lane -- and a control warp that copies strips and records, issues the
// products (one per sampled row) and takes the next block.  Rows go through a ring of
// two stages of four; D is read back once per 128 columns, and the diagonals are 16
// shared-memory reads per candidate.  Tensor memory holds six workers an SM (64 ring +
// 16 accumulator columns each, three to a CTA so that the power-of-two allocation
// fits), shared memory too (35 KB each).
//
// What bounds it: issue slots (6040 warp instructions a searched block on the 32 frames
// below, 8730 on the 4K ones, half of them in the per-block work around the unpacking)
// and, with six workers, the chain of barriers of a block.  Measured (matching kernel, popcount kernel before it): 32 frames of
// 1920x1200 0.145 -> 0.096 ms, eight 4K frames 0.27 -> 0.152 ms; the whole calls 0.289 ->
// 0.235 and 0.440 -> 0.340 ms, four 720p frames 0.0735 -> 0.0585 ms.  Slower variants:
// a warp per block on mma.sync fp8 (0.41 ms on the first batch), one barrier of the
// CTA per stage (0.16), strips by plain loads into registers (0.13, spills),
// builders polling mbarriers instead of waiting in named barriers.
#include "aggregate.cuh"
#include "ctm_internal.cuh"
#include "match_common.cuh"

namespace ctm {
namespace {

constexpr int kBuilders = 128;                   // builder threads of a worker: one per strip column of a tile
constexpr int kWorkers = 3;                      // workers (blocks in progress) per CTA
constexpr int kTcThreads = kWorkers * (kBuilders + 32);  // and a control warp each
constexpr int kTcCtas = 2;                       // resident CTAs per SM
constexpr int kTcCols = 128;                     // columns of a product (its rows, M)
constexpr int kTileCols = 256;                   // columns of a tile: up to two products
constexpr int kStageRows = 4;                    // sampled rows per ring stage (two stages)
constexpr int kRowCols = 8;                      // tensor-memory columns of one sampled row (64 e2m1)
constexpr int kTmD = 2 * kStageRows * kRowCols;  // a worker's accumulator (16 columns), after its ring
constexpr int kTmWorker = kTmD + 16;             // tensor-memory columns of a worker
constexpr int kTmSf = kWorkers * kTmWorker;      // unit scale factors: 16 columns
constexpr int kTmCols = 256;
static_assert(kTmSf + 16 <= kTmCols && kTmCols * kTcCtas <= 512, "tensor memory of an SM");
static_assert(kMaxPtsSide % kStageRows == 0, "whole stages");

struct __align__(128) Shared {
    uint64_t strip[kMaxPtsSide * kTcCols];       // codes of one product's columns, row by row
    uint4 points[kMaxPtsSide * 32];              // point operand: [2 m + h][j] 16-byte pieces
    int16_t tile[kMaxPtsSide * kTileCols];       // D of one tile, [j][x]
    int cost[kMaxCand];
    BlockGeom geom[2];
    int xoff[kMaxPtsSide];                       // byte offset of D[j][X_j]
    int kpart[kBuilders / 32];                   // K0's parts, each builder warp's first minimum
    unsigned keys[kBuilders / 32];
    uint64_t empty[2];                           // products that read the ring stage are done
    uint64_t done;                               // the products of all rows are done
    uint64_t landed;                             // the strip has landed
    uint64_t last;                               // after a failed wait: every product is done
    int next_b;                                  // the next block; -1: none
    int d_f, dy_f;                               // forward match of the block
    int fail;                                    // a bounded wait expired (read after worker_sync)
    int *err;                                    // the call's error flag
    int give_up;                                 // the same within a pass: nothing is waited for any more
};

// Bit planes of a strip code as e2m1 values, 8 words in the order (plane, half).
template <int P>
__device__ __forceinline__ uint32_t strip_plane(uint32_t w)
{
    return P < 3 ? w & (0x11111111u << P) : (w & 0x88888888u) | 0x22222222u;
}

__device__ __forceinline__ void tmem_store8(uint32_t addr, uint2 c)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n"
                 ::"r"(addr), "r"(strip_plane<0>(c.x)), "r"(strip_plane<0>(c.y)), "r"(strip_plane<1>(c.x)),
                 "r"(strip_plane<1>(c.y)), "r"(strip_plane<2>(c.x)), "r"(strip_plane<2>(c.y)),
                 "r"(strip_plane<3>(c.x)), "r"(strip_plane<3>(c.y)) : "memory");
}

__device__ __forceinline__ void tmem_load16(uint32_t addr, float (&v)[16])
{
    uint32_t u[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                 "[%16];\n"
                 : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
                   "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
                 : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(u[i]);
}

// One sampled row's product: D[128 x 16] (+)= strip[128 x 64] points[16 x 64]^T.
__device__ __forceinline__ void mma_row(uint32_t d, uint32_t strip, uint64_t points, uint32_t sf, bool add)
{
    // e2m1 x e2m1, ue8m0 scales, N = 16, M = 128
    constexpr uint32_t idesc = (1u << 7) | (1u << 10) | (2u << 17) | (1u << 23) | (8u << 24);
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], %2, %3, [%5], [%6], p;\n}\n"
                 ::"r"(d), "r"(strip), "l"(points), "r"(idesc), "r"((unsigned)add), "r"(sf), "r"(sf + 4) : "memory");
}

// One lane of a converged warp; the compiler then issues tensor-core and bulk-copy
// instructions without a loop over the lanes' operands.
__device__ __forceinline__ bool elect_one()
{
    unsigned p;
    asm volatile("{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n selp.u32 %0, 1, 0, e;\n}\n" : "=r"(p));
    return p != 0;
}

// Named barriers of worker w (barrier 0 is __syncthreads): its builder warps; all its
// warps; the control warp's signals to the builders (strip landed, products done); the
// builders' signals that a ring stage is written.  A warp that waits in a barrier
// issues nothing, where one that polls an mbarrier took issue slots from the others.
__device__ __forceinline__ int bar_id(int w, int i) { return 5 * w + 1 + i; }
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void builders_sync(int w) { bar_sync(bar_id(w, 0), 128); }
__device__ __forceinline__ void worker_sync(int w) { bar_sync(bar_id(w, 1), 160); }
constexpr int kBarSignal = 2, kBarStage = 3;  // kBarStage + stage

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

__device__ __forceinline__ void mma_commit(uint64_t *mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                 ::"r"(smem_addr(mbar)) : "memory");
}

// One pass of a block: its point codes are plane PA at (X_j + ax, Y_m + ay); the
// candidate (e, c) of point (j, m) is the other plane at column X_j + off + sgn * c of
// row Y_m + by + bstep * e (0 outside the plane).  Forward: the left codes over the
// right plane; backward: the right codes at the matched positions over the left plane.
struct Pass {
    int ax, ay, by, bstep, off, sgn;
    int nd, lo, hi;  // candidates of a row; first and last column of the strip
};

__device__ __forceinline__ Pass forward_pass(const MatchArgs &a, const BlockGeom &g)
{
    const int nd = g.dmax - g.dmin + 1;
    return Pass{0, 0, a.p.dy_min, 1, -g.dmin, -1, nd, g.X[0] - g.dmax, g.X[kMaxPtsSide - 1] - g.dmin};
}

__device__ __forceinline__ Pass backward_pass(const MatchArgs &a, const BlockGeom &g, int d_f, int dy_f)
{
    const int nd = g.dmax - g.dmin + 1;
    return Pass{-d_f, dy_f, dy_f - a.p.dy_min, -1, g.dmin - d_f, 1, nd, g.X[0] - d_f + g.dmin,
                g.X[kMaxPtsSide - 1] - d_f + g.dmax};
}

// A tile: the strip's columns [base, base + cols), base even, cols <= kTileCols.  The
// strip of most blocks is one tile.  Points further apart than the range leave columns
// no candidate reads: a tile of a wider strip starts at the first column needed from
// `cur` on and ends before such a gap.
struct Tile {
    int base, cols;
};

__device__ __noinline__ Tile wide_tile(const BlockGeom &g, int lo, int nd, int cur)
{
    const int reach = lo - g.X[0];  // candidate columns of point j: [X_j + reach, X_j + reach + nd)
    int j = 0;
    while (g.X[j] + reach + nd - 1 < cur) ++j;
    cur = max(cur, g.X[j] + reach);
    int end = g.X[j] + reach + nd - 1;
    while (j + 1 < g.nx && g.X[j + 1] + reach <= end + 16) {
        ++j;
        end = g.X[j] + reach + nd - 1;
    }
    Tile t;
    t.base = cur & ~1;
    t.cols = min(kTileCols, end - t.base + 1);
    return t;
}

// The tile of the columns from `cur` on (ps.lo <= cur <= ps.hi).
__device__ __forceinline__ Tile tile_at(const BlockGeom &g, const Pass &ps, int cur)
{
    Tile t;
    t.base = ps.lo & ~1;
    t.cols = ps.hi - t.base + 1;
    if (t.cols > kTileCols) t = wide_tile(g, ps.lo, ps.nd, cur);
    return t;
}

// Census planes of a record's block.
struct Planes {
    const uint64_t *L, *R;
    int pitch;
    int map;  // tensor map of L (R's follows)
};

__device__ __forceinline__ Planes planes_of(const MatchArgs &a, const BlockGeom &g)
{
    const bool full = g.far || a.p.close_factor == 1;
    const uint64_t *base = a.ws.census + (long long)g.frame * a.ws.frame_stride;
    Planes p;
    p.L = full ? base : base + 2 * a.ws.plane1_elems;
    p.R = p.L + (full ? a.ws.plane1_elems : a.ws.planek_elems);
    p.pitch = (int)(full ? a.ws.pitch1 : a.ws.pitchk);
    p.map = 4 * g.frame + (full ? 0 : 2);
    return p;
}

__device__ __forceinline__ int strip_stride(int cols) { return (cols + 31) & ~31; }

// After worker_sync: a bounded wait of this worker expired.
__device__ __forceinline__ bool failed(const Shared &sh) { return *reinterpret_cast<const volatile int *>(&sh.fail) != 0; }

// A bounded wait of the worker.  The first that expires ends the waiting of all its
// warps: the pass keeps up its named barriers to the end, and an expiry costs two seconds
// once instead of in each of the pass's products (up to 256 offsets x the strip's width).
// Only a wait that does not succeed at once looks at give_up: the 4K batch's call takes the
// 288.5 us it took before; with a look per product in every warp 300.0, with the error
// flag's address handed to each wait 291.1.
__device__ __noinline__ bool wait_slow(Shared &sh, uint64_t *mbar, unsigned parity)
{
    volatile int *stop = &sh.give_up;
    if (*stop) return false;
    if (mbar_wait_for(mbar, parity)) return true;
    *stop = 1;
    atomicOr(sh.err, 1);
    mbar_wait_for(mbar, parity);
    return false;
}

__device__ __forceinline__ bool wait_worker(Shared &sh, uint64_t *mbar, unsigned parity)
{
    return mbar_try_wait(mbar, parity) || wait_slow(sh, mbar, parity);
}

// ---------------------------------------------------------------- control warp

// Copy the strip of one product -- `cols` columns from `base`, rows Y_m + dy -- into
// sh.strip, four rows per gather4 where the planes have tensor maps, else row by row.
// What lies outside the plane is not written or not zero; the builders replace it.
__device__ __forceinline__ void issue_strip(const MatchArgs &a, const BlockGeom &g, Shared &sh, const Planes &pl,
                                            bool left, int base, int cols, int dy)
{
    const int lane = threadIdx.x & 31;
    const int stride = strip_stride(cols);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    int y = g.Y[lane & (kMaxPtsSide - 1)] + dy;  // rows beyond ny repeat the last one
    if (a.ws.tmaps != nullptr) {
        const int groups = (g.ny + 3) >> 2;
        const CUtensorMap *tm = a.ws.tmaps + (pl.map + (left ? 0 : 1)) * kBoxClasses + (stride / 32 - 1);
        if ((unsigned)y >= (unsigned)g.Hs) y = 0;
        int yy[kMaxPtsSide];
#pragma unroll
        for (int i = 0; i < kMaxPtsSide; ++i) yy[i] = __shfl_sync(0xffffffffu, y, i);
        if (elect_one()) {
            mbar_arrive_expect_tx(&sh.landed, (unsigned)(groups * 4 * stride * 8));
#pragma unroll
            for (int q = 0; q < kMaxPtsSide / 4; ++q)
                if (q < groups)
                    gather4_g2s(sh.strip + 4 * q * stride, tm, base, yy[4 * q], yy[4 * q + 1], yy[4 * q + 2],
                                yy[4 * q + 3], &sh.landed);
        }
        __syncwarp();
        return;
    }
    const int x_lo = max(base, 0), x_hi = min(base + cols + 1, g.Ws + 1) & ~1;  // the pitch is even
    const bool on = lane < g.ny && (unsigned)y < (unsigned)g.Hs && x_hi > x_lo;
    const unsigned bytes = on ? 8u * (unsigned)(x_hi - x_lo) : 0u;
    const unsigned total = __reduce_add_sync(0xffffffffu, bytes);
    if (lane == 0) mbar_arrive_expect_tx(&sh.landed, total);
    __syncwarp();
    if (on)
        bulk_g2s(sh.strip + lane * stride + (x_lo - base), (left ? pl.L : pl.R) + (long long)y * pl.pitch + x_lo,
                 bytes, &sh.landed);
    __syncwarp();
}

// The first product's strip of a pass.
__device__ __forceinline__ void issue_first(const MatchArgs &a, const BlockGeom &g, Shared &sh, const Planes &pl,
                                            bool left, const Pass &ps)
{
    const Tile t = tile_at(g, ps, ps.lo);
    issue_strip(a, g, sh, pl, left, t.base, min(t.cols, kTcCols), ps.by);
}

// A block's sampling record, 16 bytes per lane.
__device__ __forceinline__ void copy_record(BlockGeom *dst, const BlockGeom *src)
{
    const int lane = threadIdx.x & 31;
    if (lane < (int)(sizeof(BlockGeom) / 16))
        cp_async16(reinterpret_cast<char *>(dst) + 16 * lane, reinterpret_cast<const char *>(src) + 16 * lane);
}

// Issue the products of one pass, each product's strip when the previous one has been
// read.  next: the record of the next block, whose first strip follows the pass's
// last; null: none.  ph: parities of landed (bit 0) and done (bit 1).  tm, sf: tensor
// memory of the worker and of the scale factors.  False if a bounded wait expired:
// the barriers are kept up to the end of the pass, without products.
__device__ __forceinline__ bool issue_pass(const MatchArgs &a, const BlockGeom &g, Shared &sh, int w, const Pass &ps,
                                           const Planes &pl, bool left, const BlockGeom *next, unsigned &ph,
                                           uint32_t tm, uint32_t sf, bool withhold)
{
    const int ndy = a.p.dy_max - a.p.dy_min + 1;
    const int stages = (g.ny + kStageRows - 1) / kStageRows;
    const uint64_t desc0 = (uint64_t)((smem_addr(sh.points) & 0x3ffff) >> 4) | ((uint64_t)(256 >> 4) << 16) |
                           ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
    bool ok = true, more = true;
    int e = 0, h = 0;
    Tile t = tile_at(g, ps, ps.lo);
#pragma unroll 1
    while (more) {
        // one verdict for the warp, whose lanes may see a phase end on both sides of the limit:
        // what follows elects a lane of all
        ok = ok && __all_sync(0xffffffffu, wait_worker(sh, &sh.landed, ph & 1u));
        if (ok) ph ^= 1u;
        bar_arrive(bar_id(w, kBarSignal), 160);
        // the product after this one
        const Tile t0 = t;
        ++h;
        if (kTcCols * h >= t.cols) {
            h = 0;
            const bool end = t.base + t.cols > ps.hi;
            if (end) ++e;
            more = e < ndy;
            if (more) t = tile_at(g, ps, end ? ps.lo : t0.base + t0.cols);
        }
#pragma unroll 1
        for (int q = 0; q < stages; ++q) {
            const int st = q & 1;
            bar_sync(bar_id(w, kBarStage + st), 160);
            if (ok && elect_one()) {
                fence_after();
                const uint32_t strip = tm + st * kStageRows * kRowCols;
                const uint64_t desc = desc0 + 32 * kStageRows * q;
#pragma unroll
                for (int i = 0; i < kStageRows; ++i)
                    mma_row(tm + kTmD, strip + i * kRowCols, desc + 32 * i, sf, q + i > 0);
                mma_commit(&sh.empty[st]);
                if (q == stages - 1 && !withhold) mma_commit(&sh.done);
            }
            __syncwarp();
        }
        // every builder has read the strip
        if (ok && more) issue_strip(a, g, sh, pl, left, t.base + kTcCols * h, min(kTcCols, t.cols - kTcCols * h),
                                    ps.by + ps.bstep * e);
        ok = ok && __all_sync(0xffffffffu, wait_worker(sh, &sh.done, (ph >> 1) & 1u));
        if (ok) ph ^= 2u;
        bar_sync(bar_id(w, kBarSignal), 160);
    }
    if (ok && next != nullptr) {
        cp_async_wait_all();
        __syncwarp();
        issue_first(a, *next, sh, planes_of(a, *next), false, forward_pass(a, *next));
    }
    return ok;
}

// The control warp of worker w: block after block from queue position `first`.
__device__ __forceinline__ void control_warp(const MatchArgs &a, Shared &sh, int w, int first, int n_big, int nq,
                                             uint32_t tm, uint32_t sf)
{
    const int lane = threadIdx.x & 31;
    unsigned ph = 0u;
    const bool withhold = a.inject_expiry != 0 && first == 0;
#pragma unroll 1
    for (int buf = 0;; buf ^= 1) {
        const BlockGeom &g = sh.geom[buf];
        const Planes pl = planes_of(a, g);
        int i = 0, nb = -1;
        if (lane == 0) i = (int)gridDim.x * kWorkers + atomicAdd(&a.ws.counts->queue_head, 1);
        Pass ps = forward_pass(a, g);
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            const bool ok = issue_pass(a, g, sh, w, ps, pl, pass == 1, nb >= 0 ? &sh.geom[buf ^ 1] : nullptr, ph, tm,
                                       sf, withhold);
            if (!ok && lane == 0) sh.fail = 1;
            if (pass == 0) {  // the next block and its record
                if (lane == 0) {
                    if (i < nq) nb = queue_at(a, n_big, i);
                    sh.next_b = nb;
                }
                nb = __shfl_sync(0xffffffffu, nb, 0);
                if (nb >= 0) copy_record(&sh.geom[buf ^ 1], a.ws.geom + nb);
            } else {
                cp_async_wait_all();
            }
            worker_sync(w);  // 0: the forward match is known; 1: the block is finished, the next record visible
            if (failed(sh)) break;
            if (pass == 0) {
                ps = backward_pass(a, g, sh.d_f, sh.dy_f);
                issue_first(a, g, sh, pl, true, ps);
            }
        }
        if (failed(sh) || nb < 0) break;
    }
    cp_async_wait_all();
    __syncwarp();
    if (failed(sh)) {  // what is in flight ends before the CTA's memory is given back
        if (elect_one()) mma_commit(&sh.last);
        __syncwarp();
        mbar_wait_for(&sh.last, 0u);
        mbar_wait_for(&sh.landed, 0u);
        mbar_wait_for(&sh.landed, 1u);
        __syncwarp();
    }
}

// --------------------------------------------------------------- builder warps

// The point operand of a pass (two points per thread) and K0's parts.
__device__ __forceinline__ void store_points(const Pass &ps, const BlockGeom &g, Shared &sh, const uint64_t *plane,
                                             int pitch)
{
    const int tid = threadIdx.x % kBuilders, j = tid & 15, m0 = tid >> 4;
    const unsigned mask = (unsigned)g.colmask[j] >> m0;  // bits 0 and 8: this thread's points
    const int x = g.X[j] + ps.ax, y0 = g.Y[m0] + ps.ay, y1 = g.Y[m0 + 8] + ps.ay;
    const bool in = (unsigned)x < (unsigned)g.Ws;
    const uint2 *src = reinterpret_cast<const uint2 *>(plane + x);
    uint2 c[2] = {make_uint2(0u, 0u), make_uint2(0u, 0u)};
    if (in && (mask & 1u) && (unsigned)y0 < (unsigned)g.Hs) c[0] = __ldg(src + (long long)y0 * pitch);
    if (in && (mask & 256u) && (unsigned)y1 < (unsigned)g.Hs) c[1] = __ldg(src + (long long)y1 * pitch);
    uint4 *dst = sh.points + 32 * m0 + j;
    int k0 = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t on = 0u - ((mask >> (8 * h)) & 1u);
        const uint32_t sign = 0x88888888u & on;
        const uint32_t w0 = 0x66666666u & on, w1 = 0x44444444u & on, w2 = 0x22222222u & on;
        dst[256 * h] = make_uint4(((c[h].x << 3) & sign) | w0, ((c[h].y << 3) & sign) | w0,
                                  ((c[h].x << 2) & sign) | w1, ((c[h].y << 2) & sign) | w1);
        dst[256 * h + 16] = make_uint4(((c[h].x << 1) & sign) | w2, ((c[h].y << 1) & sign) | w2,
                                       (~c[h].x & sign) | w2, (~c[h].y & sign) | w2);
        k0 += __popc(c[h].x & 0x77777777u) + __popc(c[h].y & 0x77777777u);  // codes of unusable points are 0
    }
    k0 = __reduce_add_sync(0xffffffffu, k0);
    if ((tid & 31) == 0) sh.kpart[tid >> 5] = k0;
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}

__device__ __forceinline__ uint2 lds64(uint32_t addr)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
    return v;
}

// Unpack one product's strip (`cols` columns from `base`, rows Y_m + dy) into the ring,
// then its D into columns x0 .. of sh.tile.  empty: parities of sh.empty (bit per
// stage).  False if a bounded wait expired.
__device__ __forceinline__ bool build_product(const MatchArgs &a, const BlockGeom &g, Shared &sh, int w,
                                              unsigned &empty, int base, int cols, int x0, int dy, uint32_t lanes)
{
    const int tid = threadIdx.x % kBuilders;
    const bool busy = (tid & ~31) < cols;  // this warp's columns are needed
    const int stride = strip_stride(cols);
    const int stages = (g.ny + kStageRows - 1) / kStageRows;
    bool ok = true;
    bar_sync(bar_id(w, kBarSignal), 160);  // the strip has landed
    if (busy && (base < 0 || base + cols > g.Ws || g.Y[0] + dy < 0 || g.Y[kMaxPtsSide - 1] + dy >= g.Hs)) {
        const bool on = (unsigned)(base + tid) < (unsigned)g.Ws;  // 0 outside the plane
        for (int m = 0; m < g.ny; ++m)
            if (!on || (unsigned)(g.Y[m] + dy) >= (unsigned)g.Hs) sh.strip[m * stride + tid] = 0ull;
    }
    uint32_t src = smem_addr(sh.strip) + 8u * (unsigned)tid;
    const uint32_t row = 8u * (unsigned)stride;
#pragma unroll 1
    for (int q = 0; q < stages; ++q) {
        const int st = q & 1;
        // the products of the stage's previous rows are done
        if (q >= 2) ok = ok && wait_worker(sh, &sh.empty[st], ((empty >> st) & 1u) ^ 1u);
        empty ^= 1u << st;
        if (busy) {
            const uint32_t dst = lanes + st * kStageRows * kRowCols;
            uint2 c[kStageRows];
#pragma unroll
            for (int i = 0; i < kStageRows; ++i) {
                c[i] = lds64(src);
                src += row;
            }
#pragma unroll
            for (int i = 0; i < kStageRows; ++i) tmem_store8(dst + i * kRowCols, c[i]);
            asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
        }
        fence_before();
        bar_arrive(bar_id(w, kBarStage + st), 160);
    }
    bar_sync(bar_id(w, kBarSignal), 160);  // the products are done
    if (busy) {
        fence_after();
        float d[16];
        tmem_load16(lanes + kTmD, d);
        // whole numbers below 2^15: added to 1.5 * 2^23, the low half of the sum is the 16-bit integer
        int16_t *t = sh.tile + (x0 + tid);
#pragma unroll
        for (int j = 0; j < 16; ++j) t[j * kTileCols] = (int16_t)(uint16_t)__float_as_uint(__fadd_rn(d[j], 12582912.0f));
        fence_before();
    }
    return ok;
}

// One pass: costs of every candidate into sh.cost (index e * nd + c), and the key
// (cost << 16 | index) of the first minimum, in every thread.
// Ends after a barrier of the builders.  ok: cleared if a bounded wait expired.
__device__ __forceinline__ unsigned build_pass(const MatchArgs &a, const Pass &ps, const BlockGeom &g, Shared &sh,
                                               unsigned &empty, int w, const uint64_t *plane, int pitch,
                                               uint32_t lanes, bool &ok)
{
    const int tid = threadIdx.x % kBuilders;
    store_points(ps, g, sh, plane, pitch);
    unsigned key = 0xffffffffu;
    int e = 0;
    const int ndy = a.p.dy_max - a.p.dy_min + 1;
#pragma unroll 1
    do {
        const int dy = ps.by + ps.bstep * e;
        int cur = ps.lo;
#pragma unroll 1
        do {
            const Tile t = tile_at(g, ps, cur);
#pragma unroll 1
            for (int x0 = 0; x0 < t.cols; x0 += kTcCols)
                ok = build_product(a, g, sh, w, empty, t.base + x0, min(kTcCols, t.cols - x0), x0, dy, lanes) && ok;
            builders_sync(w);
            const int4 kp = *reinterpret_cast<const int4 *>(sh.kpart);
            const int K0 = kp.x + kp.y + kp.z + kp.w + 8 * g.n_valid;
            const bool whole = t.base <= ps.lo && ps.hi < t.base + t.cols;  // one tile holds the strip
            const bool end = ps.hi < t.base + t.cols;
#pragma unroll 1
            for (int c = tid; c < ps.nd; c += kBuilders) {
                const int x = ps.off - t.base + ps.sgn * c;
                const char *p = reinterpret_cast<const char *>(sh.tile + x);
                int *dst = sh.cost + e * ps.nd + c;
                int s = 0;
                if (whole) {
#pragma unroll
                    for (int j = 0; j < kMaxPtsSide; j += 4) {
                        const int4 o = *reinterpret_cast<const int4 *>(sh.xoff + j);
                        s += *reinterpret_cast<const int16_t *>(p + o.x) + *reinterpret_cast<const int16_t *>(p + o.y) +
                             *reinterpret_cast<const int16_t *>(p + o.z) + *reinterpret_cast<const int16_t *>(p + o.w);
                    }
                    s = K0 + (s >> 1);
                } else {  // 2 K0 and the tiles' sums (all even), halved with the last
                    for (int j = 0; j < g.nx; ++j)
                        if ((unsigned)(g.X[j] + x) < (unsigned)t.cols)
                            s += *reinterpret_cast<const int16_t *>(p + sh.xoff[j]);
                    s += cur == ps.lo ? 2 * K0 : *dst;
                    if (end) s >>= 1;
                }
                *dst = s;
                if (end) key = min(key, ((unsigned)s << 16) | (unsigned)(e * ps.nd + c));
            }
            cur = t.base + t.cols;
            if (cur <= ps.hi || e + 1 < ndy) builders_sync(w);  // D has been read
        } while (cur <= ps.hi);
    } while (++e < ndy);
    key = __reduce_min_sync(0xffffffffu, key);
    if ((tid & 31) == 0) sh.keys[tid >> 5] = key;
    builders_sync(w);
    const uint4 k = *reinterpret_cast<const uint4 *>(sh.keys);
    return min(min(k.x, k.y), min(k.z, k.w));
}

__device__ __forceinline__ void builder_warps(const MatchArgs &a, Shared &sh, int w, uint32_t tm)
{
    const int tid = threadIdx.x % kBuilders;
    const uint32_t lanes = tm + ((uint32_t)(tid & ~31) << 16);
    unsigned empty = 0u;
    unsigned long long evals = 0ull;
    const int ndy = a.p.dy_max - a.p.dy_min + 1;
#pragma unroll 1
    for (int buf = 0;; buf ^= 1) {
        const BlockGeom &g = sh.geom[buf];
        const Planes pl = planes_of(a, g);
        if (tid < kMaxPtsSide) sh.xoff[tid] = 2 * (tid * kTileCols + g.X[tid]);
        Pass ps = forward_pass(a, g);
        int d_f = 0, dy_f = 0, s_0 = 0, s_m = 0, s_p = 0;
        bool ok = true;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            const unsigned key = build_pass(a, ps, g, sh, empty, w, pass == 0 ? pl.L : pl.R, pl.pitch, lanes, ok);
            if (!ok) sh.fail = 1;
            const int c = (int)(key & 0xffffu);
            const int e = ndy == 1 ? 0 : c / ps.nd;
            const int di = c - e * ps.nd;
            int32_t *dbg = pass == 0 ? a.dbg.cost_f : a.dbg.cost_b;
            if (dbg) {
                dbg += ((long long)g.box * (a.p.grid_g * a.p.grid_g) + g.slot) * a.nc_stride;
                for (int i = tid; i < ps.nd * ndy; i += kBuilders) dbg[i] = sh.cost[i];
            }
            if (pass == 0) {
                d_f = g.dmin + di;
                dy_f = a.p.dy_min + e;
                s_0 = (int)(key >> 16);
                if (tid == 0) {
                    sh.d_f = d_f;
                    sh.dy_f = dy_f;
                    s_m = di > 0 ? sh.cost[c - 1] : 0;
                    s_p = di < ps.nd - 1 ? sh.cost[c + 1] : 0;
                }
                worker_sync(w);  // the control warp has the forward match
                if (failed(sh)) return;
                ps = backward_pass(a, g, d_f, dy_f);
            } else if (tid == 0) {
                write_record(a, g, d_f, dy_f, g.dmin + di, a.p.dy_min + e, s_m, s_0, s_p);
                evals += 2ull * (unsigned)g.n_valid * (unsigned)(ps.nd * ndy);
            }
        }
        worker_sync(w);  // the block is finished, the next record visible
        if (failed(sh) || sh.next_b < 0) break;
    }
    if (tid == 0 && evals) atomicAdd(&a.ws.counts->evals, evals);
}

__global__ void __launch_bounds__(kTcThreads, kTcCtas) match_tc_kernel(MatchArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint32_t tmem;
    const int n_big = a.ws.counts->n_big;
    const int nq = n_big + a.ws.counts->n_small;
    if ((int)blockIdx.x >= nq) return;
    // warps 0 .. 11: the builders of the workers, four each (a warp reaches the
    // tensor-memory lanes of its index modulo 4); then the control warps
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const bool control = warp >= 4 * kWorkers;
    const int w = control ? warp - 4 * kWorkers : warp / 4;
    Shared &sh = reinterpret_cast<Shared *>(smem_raw)[w];
    const int first = (int)(blockIdx.x + gridDim.x * w);  // the worker's first queue position
    if (control) {
        if (first < nq) copy_record(&sh.geom[0], a.ws.geom + queue_at(a, n_big, first));
        if (w == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                         ::"r"(smem_addr(&tmem)), "r"(kTmCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
        }
        if (lane < 2) mbar_init(&sh.empty[lane], 1);
        if (lane == 2) mbar_init(&sh.done, 1);
        if (lane == 3) mbar_init(&sh.landed, 1);
        if (lane == 4) mbar_init(&sh.last, 1);
        if (lane == 5) sh.fail = sh.give_up = 0;
        if (lane == 6) sh.err = &a.ws.counts->error;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        cp_async_wait_all();
        __syncwarp();
        if (first < nq) issue_first(a, sh.geom[0], sh, planes_of(a, sh.geom[0]), false, forward_pass(a, sh.geom[0]));
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    if (warp < 4) {
        const uint32_t one = 0x7f7f7f7fu;  // unit scale factors
        asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
                     "{%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};\n"
                     ::"r"(tm + kTmSf + ((uint32_t)warp << 21)), "r"(one) : "memory");
        asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (first < nq) {
        if (control)
            control_warp(a, sh, w, first, n_big, nq, tm + w * kTmWorker, tm + kTmSf);
        else
            builder_warps(a, sh, w, tm + w * kTmWorker);
    }
    fence_before();
    __syncthreads();
    if (warp == 4 * kWorkers)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tm), "r"(kTmCols));
}

}  // namespace

cudaError_t match_tc_configure()
{
    return cudaFuncSetAttribute(match_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kWorkers * sizeof(Shared)));
}

cudaError_t launch_match_tc(const MatchArgs &a, cudaStream_t s)
{
    const int ctas = a.sm_count * kTcCtas;
    const int grid = a.caps.max_blocks < ctas ? a.caps.max_blocks : ctas;
    match_tc_kernel<<<grid, kTcThreads, kWorkers * sizeof(Shared), s>>>(a);
    return cudaGetLastError();
}

}  // namespace ctm
