// match.cu -- the Hamming-cost search of Algorithm 2 with population counts, one CTA
// per block end to end: the plain per-box path (ctm_match_boxes_plain, one launch per
// box, the comparison for the batched path; match_tc.cu searches the blocks of every
// other call, match_pipe.cu has the two-pass variant):
//   1. the block's sampling record (point grid, usable-point masks from the
//      occlusion test of Sec. 4.3.5) is in shared memory; copy the left census
//      at every usable point (compacted column-major) and the first forward
//      strip chunk into shared memory with asynchronous copies issued together;
//   2. forward pass over the right-image strip the block can reach (sampled rows
//      x [x - dmax, x - dmin]): Eq. census_cost,
//      S(dy, d) = sum_p popc(C_L(p) ^ C_R(p.x - d, p.y + dy)), for every
//      candidate; lanes own consecutive candidates (conflict-free strip reads),
//      warps own point subsets, each thread keeps up to 8 candidate sums in
//      registers, and the warps' sums are combined in two shared rows by ordered
//      stores and adds (no atomics);
//   3. first argmin over (dy, d): after the last combining barrier every warp
//      reduces the rows to the minimum (cost << 16 | index) key itself, so the
//      result needs no broadcast; Eq. subpixel in fp32 with IEEE division;
//   4. backward pass (Sec. 4.3.3): the left strip [q.x + dmin, q.x + dmax] (bulk
//      copies, issued first) and the right codes at the matched positions (plain
//      loads) arrive in one round trip;
//   5. consistency |d_b - d_f| <= fb_tol and the block record; boxes are
//      aggregated afterwards (aggregate_kernel).
// Blocks wider than the strip are split into column chunks; chunk sums add up
// because Eq. census_cost is a sum over points.
#include <math.h>

#include "aggregate.cuh"
#include "ctm_internal.cuh"
#include "match_common.cuh"

namespace ctm {
namespace {

struct Shared {
    BlockGeom geom;         // the block's sampled grid
    uint64_t mbar;          // completion of the strip bulk copies
    int X[kMaxPtsSide];
    int Y[kMaxPtsSide];
    int colstart[kMaxPtsSide + 1];
    int spend;              // a strip copy is in flight on mbar
    unsigned cstart;        // bit j set: a strip column chunk starts at point column j
};

struct BlockCtx {
    int box, slot, b;
    int k, far;
    int dmin, dmax, nd, ndy, nc;
    int nx, ny, Ws, Hs;
    int tm_l, tm_r;           // tensor maps of the left and right planes (tile::gather4 loads)
    long long pitch;
    const uint64_t *CL;
    const uint64_t *CR;
};

// Geometry of a strip chunk whose columns start at colbase, SWc wide: rows load by
// tile::gather4 with the narrowest box that holds them when it fits the strip's
// shared-memory width, else by 1-D copies at the chunk's own width.
__device__ __forceinline__ ChunkGeom strip_geom(const MatchArgs &a, int colbase, int SWc)
{
    return chunk_geom(colbase, SWc, a.ws.tmaps != nullptr ? min(a.strip_cols, 32 * kBoxClasses) : 0);
}

// Row r = (m, e) of a strip chunk: the right plane at Y_m + dy_min + e (forward)
// or the left plane at Y_m + dy_f - (dy_min + e) (backward).
__device__ __forceinline__ int chunk_row_y(const MatchArgs &a, const BlockCtx &bc, const int *Y, bool fwd,
                                           int dy_f, int r)
{
    const int m = bc.ndy == 1 ? r : r / bc.ndy;
    const int e = r - m * bc.ndy;
    return fwd ? Y[m] + a.p.dy_min + e : Y[m] + dy_f - (a.p.dy_min + e);
}

// Warp 0: issue the bulk copies of one strip chunk (completion on sh.mbar).
template <int NT>
__device__ __forceinline__ void issue_chunk(const MatchArgs &a, const BlockCtx &bc, const Smem &sm,
                                            Shared &sh, bool fwd, int dy_f, const ChunkGeom &g)
{
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid >= 32) return;
    const int rows = bc.ny * bc.ndy;
    if (g.box > 0) {
        // tile::gather4: four rows per copy, each the map's box of g.box codes from
        // colbase_a (columns outside the plane's allocation read as zero); rows outside
        // the grid are fetched as row 0 and zeroed by land_chunk, like the other columns
        // outside [0, Ws)
        const CUtensorMap *tm = a.ws.tmaps + (fwd ? bc.tm_r : bc.tm_l) * kBoxClasses + (g.box / 32 - 1);
        const int groups = (rows + 3) >> 2;
        const unsigned total = (unsigned)groups * 4u * (unsigned)g.box * 8u;
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        if (lane == 0) {
            mbar_arrive_expect_tx(&sh.mbar, total);
            sh.spend = 1;
        }
        __syncwarp();
        for (int q = lane; q < groups; q += 32) {
            int y[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = min(4 * q + i, rows - 1);
                const int yy = chunk_row_y(a, bc, sh.Y, fwd, dy_f, r);
                y[i] = (yy >= 0 && yy < bc.Hs) ? yy : 0;
            }
            gather4_g2s(sm.strip + 4 * q * g.stride, tm, g.colbase_a, y[0], y[1], y[2], y[3], &sh.mbar);
        }
        return;
    }
    const uint64_t *plane = fwd ? bc.CR : bc.CL;
    const int Ws_even = (bc.Ws + 1) & ~1;   // the padding column after an odd width is readable
    const int x_lo = max(g.colbase_a, 0);
    const int x_hi = min(g.colbase_a + g.SWa, Ws_even);
    const unsigned row_bytes = x_hi > x_lo ? 8u * (unsigned)(x_hi - x_lo) : 0u;
    unsigned total = 0;
    for (int r = lane; r < rows; r += 32) {
        const int y = chunk_row_y(a, bc, sh.Y, fwd, dy_f, r);
        if (y >= 0 && y < bc.Hs) total += row_bytes;
    }
    total = __reduce_add_sync(0xffffffffu, total);
    // order earlier generic-proxy accesses of the strip before the bulk writes
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    if (lane == 0) {
        mbar_arrive_expect_tx(&sh.mbar, total);
        sh.spend = 1;
    }
    __syncwarp();
    if (row_bytes > 0) {
        for (int r = lane; r < rows; r += 32) {
            const int y = chunk_row_y(a, bc, sh.Y, fwd, dy_f, r);
            if (y >= 0 && y < bc.Hs)
                bulk_g2s(sm.strip + r * g.stride + (x_lo - g.colbase_a), plane + (long long)y * bc.pitch + x_lo,
                         row_bytes, &sh.mbar);
        }
    }
}

// All threads: wait for the chunk issued last, then zero what lies outside the
// plane (rows outside it; columns < 0 or >= Ws), a warp per row (only edge
// chunks have any).  Returns false if the bounded wait expired.  The phase is
// only consumed when the wait succeeded, so a drain after a failure waits for
// the same copies.
template <int NT>
__device__ __forceinline__ bool land_chunk(const MatchArgs &a, const BlockCtx &bc, const Smem &sm,
                                           Shared &sh, unsigned &phase, bool fwd, int dy_f,
                                           const ChunkGeom &g)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const bool ok = mbar_wait_bounded(&sh.mbar, phase, &a.ws.counts->error);
    if (ok) phase ^= 1u;
    if (ok && tid == 0) sh.spend = 0;
    const int rows = bc.ny * bc.ndy;
    const bool edge = g.colbase_a < 0 || g.colbase_a + g.SWa > bc.Ws ||
                      sh.Y[0] + (fwd ? a.p.dy_min : dy_f - a.p.dy_max) < 0 ||
                      sh.Y[bc.ny - 1] + (fwd ? a.p.dy_max : dy_f - a.p.dy_min) >= bc.Hs;
    if (edge) {
        const int warp = tid >> 5;
        const int c_lo = min(max(-g.colbase_a, 0), g.SWa);             // [0, c_lo): x < 0
        const int c_hi = max(min(bc.Ws - g.colbase_a, g.SWa), c_lo);   // [c_hi, SWa): x >= Ws
        for (int r = warp; r < rows; r += NT / 32) {
            const int y = chunk_row_y(a, bc, sh.Y, fwd, dy_f, r);
            uint64_t *row = sm.strip + r * g.stride;
            if (y < 0 || y >= bc.Hs) {
                for (int c = lane; c < g.SWa; c += 32) row[c] = 0ull;
            } else {
                for (int c = lane; c < c_lo; c += 32) row[c] = 0ull;
                for (int c = c_hi + lane; c < g.SWa; c += 32) row[c] = 0ull;
            }
        }
    }
    return ok;
}

// Load one strip chunk: rows (m, e) of the right plane at Y_m + dy_min + e
// (forward) or of the left plane at Y_m + dy_f - (dy_min + e) (backward);
// issue, wait, zero-fill.
template <int NT>
__device__ __forceinline__ bool load_chunk(const MatchArgs &a, const BlockCtx &bc, const Smem &sm,
                                           Shared &sh, unsigned &phase, bool fwd, int dy_f,
                                           const ChunkGeom &g)
{
    issue_chunk<NT>(a, bc, sm, sh, fwd, dy_f, g);
    return land_chunk<NT>(a, bc, sm, sh, phase, fwd, dy_f, g);
}

// The scans of one search pass after its first strip chunk has landed and the
// point bases of the first chunk are set: every chunk (later ones loaded into
// the strip after the previous chunk's scan), sums kept in registers.  Returns
// false if a bounded wait expired.
template <int NT>
__device__ bool scan_chunks(const MatchArgs &a, const BlockCtx &bc, const Smem &sm, Shared &sh,
                            unsigned &phase, bool fwd, ChunkGeom g, int (&acc)[8], int d_f, int dy_f)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31;
    const int T = (bc.nc + 31) >> 5;
    const bool fast = bc.ndy == 1 && (bc.nd & 31) == 0;
#pragma unroll
    for (int t = 0; t < 8; ++t) acc[t] = 0;
    const unsigned cs = sh.cstart;
    int j0 = 0;
    bool ok = true;
    while (j0 < bc.nx) {
        const unsigned later = cs & ~((2u << j0) - 1u);
        const int j1 = later ? __ffs(later) - 1 : bc.nx;
        const int xj0 = sh.X[j0];
        const int p0 = sh.colstart[j0], p1 = sh.colstart[j1];
        if (j0 > 0) {  // later chunks: load now (the first chunk was prefetched)
            const int SWc = sh.X[j1 - 1] - xj0 + bc.nd;
            g = strip_geom(a, fwd ? xj0 - bc.dmax : xj0 - d_f + bc.dmin, SWc);
            ok = load_chunk<NT>(a, bc, sm, sh, phase, fwd, dy_f, g) && ok;
            set_bases<NT>(sm, sh.X, p0, p1, bc.ndy, g.stride, xj0, g.delta);
            __syncthreads();
        }
        if (fast) {
            if (fwd)
                scan_dispatch_fast<NW, -1>(T, sm, p0, p1, bc.nd - 1 - lane, acc);
            else
                scan_dispatch_fast<NW, 1>(T, sm, p0, p1, lane, acc);
        } else {
            int coff[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                int c = t * 32 + lane;
                int o = 0;
                if (c < bc.nc) {
                    int e = 0;
                    while (c >= bc.nd) { c -= bc.nd; ++e; }
                    o = e * g.stride + (fwd ? (bc.nd - 1 - c) : c);
                }
                coff[t] = o;
            }
            scan_dispatch<NW>(T, sm, p0, p1, coff, acc);
        }
        __syncthreads();
        j0 = j1;
    }
    return ok;
}

// The end of a pass: the warps' sums are combined in two rows, sm.cost and
// sm.cost_b, without atomics -- warps 0 and 1 store theirs, then each further pair
// of warps adds its sums to the rows in turn, a barrier between steps -- and
// every warp then reduces the whole row pair to the first argmin key
// (cost << 16 | c), so every thread holds it without a broadcast.  Warp 0 writes
// the debug costs.  The rows' previous readers (the other pass's argmin) are
// separated from the first store by a barrier of the caller.  False if a
// bounded wait expired anywhere.
template <int NT>
__device__ __forceinline__ bool combine_pass(const MatchArgs &a, const BlockCtx &bc, const Smem &sm, bool fwd,
                                             const int (&acc)[8], bool ok, unsigned &key)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int T = (bc.nc + 31) >> 5;
    int *row = (warp & 1) ? sm.cost_b : sm.cost;
    if (warp < 2) {
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int c = t * 32 + lane;
            if (t < T && c < bc.nc) row[c] = acc[t];
        }
    }
    if (!__syncthreads_and(ok)) return false;
#pragma unroll
    for (int step = 1; step < NW / 2; ++step) {
        if ((warp >> 1) == step) {
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int c = t * 32 + lane;
                if (t < T && c < bc.nc) row[c] += acc[t];
            }
        }
        __syncthreads();
    }
    int32_t *dbgc = warp == 0 ? (fwd ? a.dbg.cost_f : a.dbg.cost_b) : nullptr;
    const int slots = a.p.grid_g * a.p.grid_g;
    unsigned k = 0xffffffffu;
    for (int c = lane; c < bc.nc; c += 32) {
        const int s = sm.cost[c] + sm.cost_b[c];
        k = min(k, ((unsigned)s << 16) | (unsigned)c);
        if (dbgc) dbgc[((long long)bc.box * slots + bc.slot) * a.nc_stride + c] = s;
    }
    key = __reduce_min_sync(0xffffffffu, k);
    return true;
}

// Block context from the block's sampling record (which carries its box plan).
__device__ __forceinline__ BlockCtx make_ctx(const MatchArgs &a, const BlockGeom &g, int b)
{
    BlockCtx bc;
    bc.box = g.box;
    bc.slot = g.slot;
    bc.b = b;
    bc.k = g.k;
    bc.far = g.far;
    bc.dmin = g.dmin;
    bc.dmax = g.dmax;
    bc.nd = g.dmax - g.dmin + 1;
    bc.ndy = a.p.dy_max - a.p.dy_min + 1;
    bc.nc = bc.nd * bc.ndy;
    bc.Ws = g.Ws;
    bc.Hs = g.Hs;
    bc.nx = g.nx;
    bc.ny = g.ny;
    const bool full = g.far || a.p.close_factor == 1;
    bc.tm_l = 4 * g.frame + (full ? 0 : 2);
    bc.tm_r = bc.tm_l + 1;
    const uint64_t *base = a.ws.census + (long long)g.frame * a.ws.frame_stride;
    bc.CL = full ? base : base + 2 * a.ws.plane1_elems;
    bc.CR = full ? base + a.ws.plane1_elems : base + 2 * a.ws.plane1_elems + a.ws.planek_elems;
    bc.pitch = full ? a.ws.pitch1 : a.ws.pitchk;
    return bc;
}

// Point layout of a block whose sampling record is in g: the column-major
// compaction of its usable points (sm.pmj), its sampled columns and rows, the left
// codes at its points (cp.async) and their strip bases in its first forward strip
// chunk g0.  Ends with a barrier.
template <int NT>
__device__ __forceinline__ void layout_block(const BlockCtx &bc, const BlockGeom &g, const Smem &sm, Shared &sh,
                                             int j1_first, const ChunkGeom &g0)
{
    const int tid = threadIdx.x;
    const int x0 = g.X[0];
    for (int t = tid; t < kMaxPts; t += NT) {
        const int j = t >> 4, m = t & 15;
        if (j < bc.nx && ((g.colmask[j] >> m) & 1u)) {
            const int idx = g.colprefix[j] + __popc(g.colmask[j] & ((1u << m) - 1u));
            const int x = g.X[j], y = g.Y[m];
            cp_async8(&sm.pcode[idx], bc.CL + (long long)y * bc.pitch + x);
            if (j < j1_first) sm.pbase[idx] = 8 * (m * bc.ndy * g0.stride + x - x0 + g0.delta);
            sm.pmj[idx] = (m << 8) | j;
        }
    }
    if (tid < kMaxPtsSide) {
        sh.X[tid] = g.X[tid];
        sh.Y[tid] = g.Y[tid];
    }
    if (tid <= kMaxPtsSide) sh.colstart[tid] = tid < bc.nx ? g.colprefix[tid] : g.n_valid;
    if (tid == 0) sh.cstart = g.cstart;
    __syncthreads();  // sh.Y is read by the issuing warp
}

// First column chunk of a block: its end column and its forward strip geometry.
__device__ __forceinline__ int first_chunk_end(const BlockGeom &g, int nx)
{
    const unsigned later0 = g.cstart & ~1u;
    return later0 ? __ffs(later0) - 1 : nx;
}

// One block end to end, its record in sh.geom.  Returns false if a bounded wait
// expired.  evals: thread 0 adds this block's evaluation count.
template <int NT>
__device__ bool process_block(const MatchArgs &a, int b, const Smem &sm, Shared &sh, unsigned &phase,
                              unsigned long long &evals)
{
    const int tid = threadIdx.x;
    const BlockGeom &g = sh.geom;
    const BlockCtx bc = make_ctx(a, g, b);
    const int total = g.n_valid;
    const int j1_first = first_chunk_end(g, bc.nx);
    const int x0 = g.X[0];
    const int SW0 = g.X[j1_first - 1] - x0 + bc.nd;
    const ChunkGeom g0 = strip_geom(a, x0 - bc.dmax, SW0);

    // 1. the left codes and the first forward strip chunk
    layout_block<NT>(bc, g, sm, sh, j1_first, g0);
    issue_chunk<NT>(a, bc, sm, sh, true, 0, g0);
    bool ok = land_chunk<NT>(a, bc, sm, sh, phase, true, 0, g0);
    cp_async_wait_all();
    if (!__syncthreads_and(ok)) return false;

    // 2-3. forward pass, argmin (every thread), parabola inputs
    int acc[8];
    ok = scan_chunks<NT>(a, bc, sm, sh, phase, true, g0, acc, 0, 0);
    unsigned key;
    if (!combine_pass<NT>(a, bc, sm, true, acc, ok, key)) return false;
    const int cf = (int)(key & 0xffffu);
    const int ef = bc.ndy == 1 ? 0 : cf / bc.nd;
    const int dif = cf - ef * bc.nd;
    const int d_f = bc.dmin + dif, dy_f = a.p.dy_min + ef;
    int s_m = 0, s_p = 0;
    if (tid == 0) {
        s_m = dif > 0 ? sm.cost[cf - 1] + sm.cost_b[cf - 1] : 0;
        s_p = dif < bc.nd - 1 ? sm.cost[cf + 1] + sm.cost_b[cf + 1] : 0;
    }

    // 4. backward pass: the right codes at the matched positions and the first left
    //    strip (every warp's forward scans ended at combine_pass's barrier); the codes'
    //    plain loads overlap the copies' round trip
    const ChunkGeom gb = strip_geom(a, x0 - d_f + bc.dmin, SW0);
    issue_chunk<NT>(a, bc, sm, sh, false, dy_f, gb);
    for (int t = tid; t < total; t += NT) {
        const int mj = sm.pmj[t];
        const int qx = sh.X[mj & 255] - d_f, qy = sh.Y[mj >> 8] + dy_f;
        sm.pcode[t] = (qx >= 0 && qx < bc.Ws && qy >= 0 && qy < bc.Hs)
                          ? __ldg(bc.CR + (long long)qy * bc.pitch + qx) : 0ull;
    }
    ok = land_chunk<NT>(a, bc, sm, sh, phase, false, dy_f, gb);
    set_bases<NT>(sm, sh.X, 0, sh.colstart[j1_first], bc.ndy, gb.stride, x0, gb.delta);
    if (!__syncthreads_and(ok)) return false;
    ok = scan_chunks<NT>(a, bc, sm, sh, phase, false, gb, acc, d_f, dy_f);
    unsigned keyb;
    if (!combine_pass<NT>(a, bc, sm, false, acc, ok, keyb)) return false;
    if (tid == 0) {
        const int cb = (int)(keyb & 0xffffu);
        const int eb = bc.ndy == 1 ? 0 : cb / bc.nd;
        // 5. block record; boxes are aggregated by aggregate_kernel
        write_record(a, g, d_f, dy_f, bc.dmin + (cb - eb * bc.nd), a.p.dy_min + eb, s_m, (int)(key >> 16), s_p);
        evals += 2ull * (unsigned long long)total * (unsigned long long)bc.nc;
    }
    return true;
}

__device__ __forceinline__ Smem carve(const MatchArgs &a, unsigned char *raw)
{
    Smem sm;
    size_t off = 0;
    sm.strip = reinterpret_cast<uint64_t *>(raw + off);
    off += sizeof(uint64_t) * (size_t)a.strip_rows * a.strip_cols;
    sm.pcode = reinterpret_cast<uint64_t *>(raw + off);
    off += sizeof(uint64_t) * kMaxPts;
    sm.cost = reinterpret_cast<int *>(raw + off);
    off += sizeof(int) * kMaxCand;
    sm.cost_b = reinterpret_cast<int *>(raw + off);
    off += sizeof(int) * kMaxCand;
    sm.pmj = reinterpret_cast<int *>(raw + off);
    off += sizeof(int) * kMaxPts;
    sm.pbase = reinterpret_cast<int *>(raw + off);
    return sm;
}

template <int NT>
__global__ void __launch_bounds__(NT) match_box_kernel(MatchArgs a, int box)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(16) Shared sh;
    if ((int)blockIdx.x >= a.ws.nblk[box]) return;
    const int b = block_base(a, box) + blockIdx.x;
    if (a.ws.geom[b].n_valid < a.p.min_pts) return;  // finished by the planner
    const Smem sm = carve(a, smem_raw);
    if (threadIdx.x < (int)(sizeof(BlockGeom) / 16))
        cp_async16(reinterpret_cast<char *>(&sh.geom) + 16 * threadIdx.x,
                   reinterpret_cast<const char *>(a.ws.geom + b) + 16 * threadIdx.x);
    if (threadIdx.x == 0) {
        mbar_init(&sh.mbar, 1);
        sh.spend = 0;
    }
    cp_async_wait_all();
    __syncthreads();
    unsigned phase = 0;
    unsigned long long evals = 0ull;
    if (!process_block<NT>(a, b, sm, sh, phase, evals)) {
        // let every copy still in flight land before the CTA leaves (its shared memory
        // may go to another CTA)
        cp_async_wait_all();
        __syncthreads();
        if (sh.spend) mbar_wait_bounded(&sh.mbar, phase, &a.ws.counts->error);
    }
    if (threadIdx.x == 0 && evals) atomicAdd(&a.ws.counts->evals, evals);
}

}  // namespace

size_t match_smem_bytes(const MatchArgs &a)
{
    return sizeof(uint64_t) * (size_t)a.strip_rows * a.strip_cols + sizeof(uint64_t) * kMaxPts +
           2 * sizeof(int) * kMaxCand + 2 * sizeof(int) * kMaxPts;
}

namespace {

template <int NT>
cudaError_t raise_box_limit(int need)
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, match_box_kernel<NT>);
    if (e == cudaSuccess && fa.maxDynamicSharedSizeBytes < need)
        e = cudaFuncSetAttribute(match_box_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, need);
    return e;
}

}  // namespace

// The dynamic shared-memory limit is a per-kernel, process-wide setting: it is
// only ever raised, so contexts with different strip sizes can coexist.
cudaError_t match_configure(const MatchArgs &a, int threads)
{
    const int need = (int)match_smem_bytes(a);
    return threads == 128 ? raise_box_limit<128>(need) : raise_box_limit<256>(need);
}

cudaError_t launch_match_box(const MatchArgs &a, int threads, int box, cudaStream_t s)
{
    const int slots = a.p.grid_g * a.p.grid_g;
    if (threads == 128)
        match_box_kernel<128><<<slots, 128, match_smem_bytes(a), s>>>(a, box);
    else
        match_box_kernel<256><<<slots, 256, match_smem_bytes(a), s>>>(a, box);
    return cudaGetLastError();
}

}  // namespace ctm
