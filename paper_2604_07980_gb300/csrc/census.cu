// census.cu -- census transform kernels (Sec. 4.3.1, Algorithm 1).
//
// Codes on the grid I_k(x, y) = I(k x, k y) (k = 1 is the image itself; k > 1
// is the multi-resolution census of Sec. 4.3.1 taken by decimation).  Bits
// follow the raster order of the window (row j outer, column i inner), first
// neighbour in the highest comparison bit, with the optional sentinel above
// them; pixels whose window leaves the grid get 0.
//
// Fixed windows (5x5, 7x7, 9x7) compare bit planes of 32 pixels at a time in units of
// 128 columns: of eight rows for a full image (ctm_census_build), of the marked ones of
// sixteen rows for the matching path.  Other windows use a warp per 64-pixel tile, the
// window rows staged in shared memory as 16-bit values 0x6400 | v.
#include "ctm_internal.cuh"

namespace ctm {
namespace {

constexpr int kTile = 64;                          // pixels per warp tile of the full-image kernels
constexpr int kColsMax = kTile + kMaxWin - 1;      // staged columns (78)
constexpr int kWordsMax = (kColsMax + 1) / 2 + 1;  // half2 words per staged row (40)
constexpr int kWarpsPerCta = 8;

// Per-warp staging buffers: `rows` window rows, each as half2 pairs (c, c+1)
// starting at even c (even) and at odd c (odd), kWordsMax words per row.
struct WarpStage {
    uint32_t *even;
    uint32_t *odd;
};

__device__ __forceinline__ WarpStage warp_stage(uint32_t *smem, int warp, int rows)
{
    WarpStage st;
    st.even = smem + (size_t)warp * 2 * rows * kWordsMax;
    st.odd = st.even + rows * kWordsMax;
    return st;
}

struct Plane {
    const uint8_t *img;   // source image (full resolution)
    int W, H, pitch, k;   // source size and decimation
    int Ws, Hs;           // census grid size
    uint64_t *out;
    long long opitch;
    int vec_ok;           // 16-byte stores allowed (even pitch, 16-byte aligned base)
    int vec_load;         // word loads allowed: k in {1, 2}, 8-byte aligned base, pitch % 4 == 0
};

// Staged row layout: H[b] = 0x6400 | I_k(x0 - 8 + b, row) for b in [0, 80), kept
// twice as half2 words: even[t] = (H[2t], H[2t+1]) and odd[t] = (H[2t+1], H[2t+2]),
// so every pair of adjacent pixels is one aligned 32-bit word in one of the two.
// Lane l < 21 loads H[4l .. 4l+3] with one 32-bit load (k = 1) or one 64-bit
// load (k = 2) where the four pixels lie inside the image, else byte by byte.
__device__ __forceinline__ uint32_t load_quad(const Plane &pl, int x0, int ys, int lane)
{
    const uint8_t *row = pl.img + (long long)pl.k * ys * pl.pitch;
    uint32_t v = 0u;
    if (lane < 21) {
        const int xs = x0 - 8 + 4 * lane;
        if (pl.vec_load && pl.k == 1 && xs >= 0 && xs + 3 < pl.W) {
            v = __ldg(reinterpret_cast<const uint32_t *>(row + xs));
        } else if (pl.vec_load && pl.k == 2 && xs >= 0 && 2 * xs + 7 < pl.W) {
            const uint2 w = __ldg(reinterpret_cast<const uint2 *>(row + 2 * xs));
            v = __byte_perm(w.x, w.y, 0x6420);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int xq = xs + q;
                if (xq >= 0 && xq < pl.Ws) v |= (uint32_t)__ldg(row + (long long)pl.k * xq) << (8 * q);
            }
        }
    }
    return v;
}

// Convert one loaded row (4 pixels per lane) to the two half2 copies.
__device__ __forceinline__ void store_quad(uint32_t v, uint32_t *even, uint32_t *odd, int lane)
{
    const uint32_t nxt = __shfl_down_sync(0xffffffffu, v, 1);
    if (lane < 20) {
        const uint32_t C = 0x64646464u;
        uint2 e, o;
        e.x = __byte_perm(v, C, 0x4140);                            // H[4l],   H[4l+1]
        e.y = __byte_perm(v, C, 0x4342);                            // H[4l+2], H[4l+3]
        o.x = __byte_perm(v, C, 0x4241);                            // H[4l+1], H[4l+2]
        o.y = __byte_perm(__byte_perm(v, nxt, 0x0043), C, 0x4140);  // H[4l+3], H[4l+4]
        *reinterpret_cast<uint2 *>(even + 2 * lane) = e;
        *reinterpret_cast<uint2 *>(odd + 2 * lane) = o;
    }
}

__device__ __forceinline__ void stage_rows_any(const Plane &pl, int x0, int y, int sy,
                                               const WarpStage &st, int lane)
{
    for (int r = 0; r < 2 * sy + 1; ++r)
        store_quad(load_quad(pl, x0, y - sy + r, lane), st.even + r * kWordsMax, st.odd + r * kWordsMax, lane);
}

// Any window: plain per-pixel loop over the staged rows.
__device__ __forceinline__ uint64_t code_any(const WarpStage &st, int px, int win_w, int win_h,
                                             int sentinel)
{
    const uint16_t *ev = reinterpret_cast<const uint16_t *>(st.even);
    constexpr int rowh = 2 * kWordsMax;
    const int sx = win_w / 2, sy = win_h / 2;
    const int off = 8 - sx;
    const uint16_t centre = ev[sy * rowh + px + 8];
    uint64_t c = sentinel ? 1ull : 0ull;
    for (int j = 0; j < win_h; ++j)
        for (int i = 0; i < win_w; ++i) c = (c << 1) | (uint64_t)(ev[j * rowh + px + i + off] > centre);
    return c;
}

__device__ __forceinline__ void store_pair(const Plane &pl, int x, int y, uint64_t c0, uint64_t c1)
{
    uint64_t *dst = pl.out + (long long)y * pl.opitch + x;
    if (x + 1 < pl.Ws) {
        if (pl.vec_ok) {
            *reinterpret_cast<ulonglong2 *>(dst) = make_ulonglong2(c0, c1);
        } else {
            dst[0] = c0;
            dst[1] = c1;
        }
    } else if (x < pl.Ws) {
        dst[0] = c0;
    }
}


// ---------------------------------------------------------------------------
// Fixed windows (5x5, 7x7, 9x7): bit-sliced.
//
// A unit is 128 columns x up to 16 rows of a plane.  Its pixels are turned into bit
// planes: word j of plane p holds bit p of the 32 pixels x0 + j + 4 b (bit b of the
// word), j = 0 .. 3.  Pixels four apart share a word, so the neighbour at column offset
// dx is another word -- word j + dx, of -4 .. 7, where the words outside 0 .. 3 are the
// same words moved by one bit -- and no compare needs a shift.  [neighbour > centre] of
// 32 pixels is then one LOP3 per plane, from the lowest bit up:
//     gt = (a & ~c) | (gt & ~(a ^ c)),
// 8 instructions for 32 compares, and two 32 x 32 bit transposes turn a pixel group's 63
// results into codes.
//
// Work split: a warp takes a unit.  Four lanes slice a source row (once, for the up to
// WH rows of codes that read it): 32 pixels per lane, an 8 x 8 bit transpose within the
// bytes of its 8 words, byte exchange between the four lanes, the word and its two moved
// copies to shared memory.  Then four lanes take a marked row, a word each.
//
// What bounds it: the ALU pipe (LOP3, PRMT, SHF: half of the issue rate; about 1450
// instructions for eight rows of a unit, 912 of them the compares and transposes) and
// the L1 (124 LDS.128 for the same rows, 0.6 of its wavefronts), 60 and 75% busy on eight
// 4K frames, with twelve warps an SM (shared memory, and 64,512 of 65,536 registers).  The kernel before it compared two
// pixels per instruction in 16-bit halves, 160 instructions a pixel against 85 here
// (per marked pixel: a unit also computes the unmarked part of its 128 columns, 10 to
// 25%, and leaves lanes idle when its rows are not a multiple of eight).  Measured, list
// and census of the marked tiles: eight 4K frames 141 -> 110 us, 32 frames of 1920x1200
// 110 -> 103, four 720p frames 24.4 -> 19.5, one 1279x719 frame (rows of odd pitch, which
// the old kernel read by bytes) 18.2 -> 14.6; full images, alone: 1920x1200 15.0 -> 12.4,
// 3839x2159 at half resolution 35 -> 13.7 us.  Where sampled rows lie far apart it is the
// slower one: a unit of a few marked rows slices nearly as many source rows as a full one
// and leaves lanes idle (eight 1920x1200 frames, every box one block of 16 x 16 points,
// 28.7 -> 52 us; joining spans of columns in such units did not help).  Slower: a CTA of
// four warps per unit of 32 rows (120 us on the 32 frames), codes stored by the lanes
// instead of bulk copies (L1 at 78%), all source rows loaded before the first is sliced
// (instruction cache), two row buffers in registers (spills).
constexpr int kUnitPx = 128;      // columns of a unit
constexpr int kRoiRows = 16;      // rows of a unit of the matching path
constexpr int kUnitThreads = 64;
constexpr int kUnitCtas = 6;      // resident CTAs per SM (37 KB and 168 registers a thread: each alone stops a seventh)
constexpr int kFullThreads = 128; // full image
constexpr int kFullCtas = 4;      // 128 registers a thread
constexpr int kUnitPos = 12;      // words -4 .. 7 of a source row
// 16-byte pieces of a sliced row: planes 0 .. 3 of the 12 words, then planes 4 .. 7, and
// four unused, so that neighbouring rows' pieces lie half of the banks apart
constexpr int kUnitPieces = 2 * kUnitPos + 4;
constexpr int kStageStride = kUnitPx + 4;  // codes between staged rows: eight rows' 32-byte stores cover the banks

// 32 pixels of a row on their way in: 8 little-endian words, or (pairs) the 16 words of 64
// source bytes whose even bytes they are, and the pixels left and right of the lane's word.
struct RowPx {
    uint32_t v[16];
    uint32_t left, right;
    bool pairs;
};

// 32 pixels of grid row yr from grid column x (a multiple of 32); pixels outside the grid
// are 0.  Sixteen-byte loads where image and pitch allow them, not waited for here; else
// aligned words moved into place; bytes at the grid's right border, where a word would
// leave the image, and at other decimations.
__device__ __forceinline__ void load_px32(const PlaneDesc &d, int x, int yr, bool vec, RowPx &px)
{
    const uint8_t *row = d.img + (long long)d.k * yr * d.pitch;
    const uint8_t *end = d.img + (long long)(d.H - 1) * d.pitch + d.W;
    const bool inside = x + 32 <= d.Ws;
    const uint8_t *s = row + (long long)d.k * x;
    const unsigned mis = (unsigned)(reinterpret_cast<uintptr_t>(s) & 3u), sh = 8u * mis;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(s - mis);
    uint32_t (&v)[16] = px.v;
    if (d.k <= 2 && inside && vec && s + 32 * d.k <= end) {
        px.pairs = d.k == 2;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i >= 2 && d.k == 1) break;
            const uint4 a = __ldg(reinterpret_cast<const uint4 *>(s) + i);
            v[4 * i] = a.x;
            v[4 * i + 1] = a.y;
            v[4 * i + 2] = a.z;
            v[4 * i + 3] = a.w;
        }
    } else if (d.k == 1 && inside && s - mis >= d.img && s + 36 <= end) {
        uint32_t u[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) u[i] = __ldg(w + i);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __funnelshift_r(u[i], u[i + 1], sh);
    } else if (d.k == 2 && inside && s - mis >= d.img && s + 68 <= end) {
        uint32_t u[17];
        px.pairs = true;
#pragma unroll
        for (int i = 0; i < 17; ++i) u[i] = __ldg(w + i);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __funnelshift_r(u[i], u[i + 1], sh);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (x + 4 * i + q < d.Ws) v[i] |= (uint32_t)__ldg(s + (long long)d.k * (4 * i + q)) << (8 * q);
        }
    }
}

// Lane j of four: the pixels x0 + 32 j .. + 31 of row yr (on: it is needed and inside the
// grid) of the unit at column x0.
__device__ __forceinline__ void load_row(const PlaneDesc &d, int x0, int yr, bool on, int j, bool vec, RowPx &px)
{
#pragma unroll
    for (int i = 0; i < 16; ++i) px.v[i] = 0u;
    px.left = px.right = 0u;
    px.pairs = false;
    if (!on) return;
    if (x0 + 32 * j < d.Ws) load_px32(d, x0 + 32 * j, yr, vec, px);
    const uint8_t *row = d.img + (long long)d.k * yr * d.pitch;
    const int xl = x0 - 4 + j, xr = x0 + kUnitPx + j;
    if (xl >= 0 && xl < d.Ws) px.left = __ldg(row + (long long)d.k * xl);
    if (xr < d.Ws) px.right = __ldg(row + (long long)d.k * xr);
}

// b << S on the multiply pipe (the compiler would take the ALU, which bounds these kernels).
template <int S>
__device__ __forceinline__ uint32_t shl_fma(uint32_t b)
{
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, 0;" : "=r"(r) : "r"(b), "n"(1u << S));
    return r;
}

// Three-input logic as one instruction (written out, the compiler spends up to two on it).
template <int Lut>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(r) : "r"(a), "r"(b), "r"(c), "n"(Lut));
    return r;
}
constexpr int kSelect = 0xe4;   // (a & c) | (b & ~c)
constexpr int kGreater = 0xb2;  // (a & ~b) | (c & ~(a ^ b)): one more bit of [a > b], c the result of the bits below

// Exchange bits: a's bits of ~m (shifted down) against b's bits of m, m the low s bits of
// every 2 s.
template <int S>
__device__ __forceinline__ void swap_bits(uint32_t &a, uint32_t &b)
{
    constexpr uint32_t m = S == 1 ? 0x55555555u : (S == 2 ? 0x33333333u : 0x0f0f0f0fu);
    const uint32_t lo = lop3<kSelect>(a, shl_fma<S>(b), m);
    b = lop3<kSelect>(a >> S, b, m);
    a = lo;
}

// Transpose of a 32 x 32 bit matrix, row i in w[i].
__device__ __forceinline__ void transpose32(uint32_t (&w)[32])
{
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const uint32_t a = w[i], b = w[i + 16];
        w[i] = __byte_perm(a, b, 0x5410);
        w[i + 16] = __byte_perm(a, b, 0x7632);
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        if (i & 8) continue;
        const uint32_t a = w[i], b = w[i + 8];
        w[i] = __byte_perm(a, b, 0x6240);
        w[i + 8] = __byte_perm(a, b, 0x7351);
    }
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if (!(i & 4)) swap_bits<4>(w[i], w[i + 4]);
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if (!(i & 2)) swap_bits<2>(w[i], w[i + 2]);
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if (!(i & 1)) swap_bits<1>(w[i], w[i + 1]);
}

// Slice a loaded row into `dst`.  All lanes of a warp call it (on: this row is written).
__device__ __forceinline__ void slice_row(const RowPx &px, bool on, int j, uint4 *dst)
{
    const unsigned full = 0xffffffffu;
    const uint32_t bl = px.left, br = px.right;
    uint32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)  // the even bytes of words 2 i, 2 i + 1, or word i
        v[i] = px.pairs ? __byte_perm(px.v[2 * i], px.v[2 * i + 1], 0x6420) : px.v[i];
    // bit i of byte c of v[p]: bit p of byte c of word i
#pragma unroll
    for (int i = 0; i < 4; ++i) swap_bits<4>(v[i], v[i + 4]);
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (!(i & 2)) swap_bits<2>(v[i], v[i + 2]);
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (!(i & 1)) swap_bits<1>(v[i], v[i + 1]);
    // byte c of lane g to byte g of lane c
    const unsigned sel2 = (j & 2) ? 0x3276u : 0x5410u, sel1 = (j & 1) ? 0x3715u : 0x6240u;
#pragma unroll
    for (int p = 0; p < 8; ++p) v[p] = __byte_perm(v[p], __shfl_xor_sync(full, v[p], 2), sel2);
#pragma unroll
    for (int p = 0; p < 8; ++p) v[p] = __byte_perm(v[p], __shfl_xor_sync(full, v[p], 1), sel1);
    if (!on) return;
    uint32_t l[8], r[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        l[p] = __funnelshift_l(bl << (31 - p), v[p], 1);
        r[p] = __funnelshift_r(v[p], br >> p, 1);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint4 *o = dst + h * kUnitPos + j;
        o[0] = make_uint4(l[4 * h], l[4 * h + 1], l[4 * h + 2], l[4 * h + 3]);
        o[4] = make_uint4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
        o[8] = make_uint4(r[4 * h], r[4 * h + 1], r[4 * h + 2], r[4 * h + 3]);
    }
}

// [neighbour > centre] of 32 pixels: `a` the neighbour's planes 0 .. 3 and b its planes 4 .. 7.
__device__ __forceinline__ uint32_t greater32(uint4 a, uint4 b, const uint32_t (&c)[8])
{
    uint32_t g = a.x & ~c[0];
    g = lop3<kGreater>(a.y, c[1], g);
    g = lop3<kGreater>(a.z, c[2], g);
    g = lop3<kGreater>(a.w, c[3], g);
    g = lop3<kGreater>(b.x, c[4], g);
    g = lop3<kGreater>(b.y, c[5], g);
    g = lop3<kGreater>(b.z, c[6], g);
    return lop3<kGreater>(b.w, c[7], g);
}

// Code bits 32 H .. 32 H + 31 of the 32 pixels of a word, pixel b's in w[b].  src: piece
// (first window row, word j).  V: pixels whose window lies in the grid.
template <int WW, int WH, int H>
__device__ __forceinline__ void code_half(const uint4 *src, const uint32_t (&c)[8], uint32_t V, int sentinel,
                                          uint32_t (&w)[32])
{
    constexpr int sx = WW / 2, n = WW * WH;
#pragma unroll
    for (int q = 0; q < 32; ++q) {
        const int p = 32 * H + q, k = n - 1 - p;  // code bit and raster index of its window offset
        if (p > n || k == n / 2) {
            w[q] = 0u;
        } else if (p == n) {
            w[q] = sentinel ? V : 0u;
        } else {
            const uint4 *s = src + (k / WW) * kUnitPieces + 4 + (k % WW) - sx;
            w[q] = greater32(s[0], s[kUnitPos], c);
        }
    }
    if (V != 0xffffffffu) {
#pragma unroll
        for (int q = 0; q < 32; ++q) w[q] &= V;
    }
    transpose32(w);
}

// Codes of word j of row y (its first window row, word -4, at `rows`) of the unit at x0.
template <int WW, int WH>
__device__ __forceinline__ void word_codes(const PlaneDesc &d, int x0, int y, int j, const uint4 *rows, int sentinel,
                                           uint32_t (&lo)[32], uint32_t (&hi)[32])
{
    constexpr int sx = WW / 2, sy = WH / 2;
    static_assert(sx <= 4 && WW * WH < 64, "window");
    const int x = x0 + j;
    // pixels x + 4 b with b0 <= b < b1 have their window inside the grid
    uint32_t V = 0xffffffffu;
    if (y - sy < 0 || y + sy >= d.Hs) {
        V = 0u;
    } else if (x0 < sx || x0 + kUnitPx + sx > d.Ws) {
        const int b0 = max(0, (sx - x + 3) >> 2), b1 = min(32, (d.Ws - sx - x + 3) >> 2);
        V = b1 <= b0 ? 0u : (0xffffffffu >> (32 - b1)) & (0xffffffffu << b0);
    }
    const uint4 *src = rows + j, *mid = src + sy * kUnitPieces + 4;
    const uint4 ca = mid[0], cb = mid[kUnitPos];
    const uint32_t c[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
    code_half<WW, WH, 0>(src, c, V, sentinel, lo);
    if constexpr (WW * WH >= 32) {
        code_half<WW, WH, 1>(src, c, V, sentinel, hi);
    } else {
#pragma unroll
        for (int b = 0; b < 32; ++b) hi[b] = 0u;
    }
}

__device__ __forceinline__ void stage_codes(uint2 *st, const uint32_t (&lo)[32], const uint32_t (&hi)[32])
{
#pragma unroll
    for (int b = 0; b < 32; ++b) st[4 * b] = make_uint2(lo[b], hi[b]);
}

// One staged row to its place, 16-byte aligned, cols even.
__device__ __forceinline__ void bulk_row(uint64_t *dst, const uint2 *src, int cols)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\ncp.async.bulk.commit_group;\n"
                 ::"l"(dst), "r"((unsigned)__cvta_generic_to_shared(src)), "r"(8 * cols) : "memory");
}

// This thread's bulk copies have read their shared memory (.read) or are complete.
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

// Place of marked row `row` among the marked ones: odd and even rows in turn as long as
// both last, as two rows read together (eight lanes of a 16-byte load) meet in the same
// banks when both are even or both odd.
__device__ __forceinline__ int slot_of_row(uint32_t mask, int row)
{
    const uint32_t even = mask & 0x55555555u, odd = mask & ~0x55555555u;
    const int both = min(__popc(even), __popc(odd));
    const int i = __popc((row & 1 ? odd : even) & ((1u << row) - 1u));
    return i < both ? 2 * i + (row & 1) : both + i;
}

// Shared memory of a warp working on listed units.
template <int WH>
struct __align__(16) UnitSmem {
    static constexpr int kRows = kRoiRows + WH - 1;  // source rows of a unit
    uint4 rows[kRows * kUnitPieces];
    uint2 codes[8 * kStageStride];                   // codes of eight rows on their way out
    int need_row[2][kRows];                          // source rows read, in order: this unit's, the next one's
    int row_of[kRoiRows];                            // marked rows
};

// A unit: marked rows y0 + i (i in mask) of columns x0 .. x0 + 127 (x0 a multiple of 32)
// of a plane.
struct Unit {
    uint32_t mask;
    int x0, y0, plane;
};

__device__ __forceinline__ Unit unit_at(const uint4 *list, int u)
{
    const uint4 e = __ldg(list + u);
    return Unit{e.x, (int)e.y, (int)e.z, (int)e.w};
}

// Codes of the listed units first, first + step, ... below n, by one warp.  Workspace
// planes are 256-byte aligned and their pitch is a multiple of 32 codes, so rows leave by
// bulk copies (codes between a grid's width and the pitch, which no one reads, as 0).
// One loop over batches of eight source rows: a batch is sliced while the next one's
// loads are in flight -- the same unit's, or the first of the next unit, whose latency
// the current unit's codes then cover.
template <int WW, int WH>
__device__ __forceinline__ void census_units(const uint4 *list, const PlaneDesc *planes, int first, int n, int step,
                                             int sentinel, UnitSmem<WH> &sm)
{
    constexpr int sy = WH / 2;
    static_assert(UnitSmem<WH>::kRows <= 32, "a lane per source row");
    const int lane = threadIdx.x & 31, j = lane & 3, slot = lane >> 2;
    const uint32_t lt = (1u << lane) - 1u;
    const Unit none{0u, 0, 0, 0};
    Unit cur = none, ld = none;                          // the unit being sliced, the unit being loaded
    Unit nxt = first < n ? unit_at(list, first) : none;
    int u = first - step;                                // index of `ld`
    int t = 0, n_need = 0;                               // batch being sliced, source rows of `cur`
    int tl = 0, nl = 0, bl = 0;                          // batch being loaded, source rows of `ld`
    PlaneDesc d{};                                       // of `ld`
    bool vec = false;
    RowPx px;                                            // the batch being sliced
    int r = 0;
    bool on = false;
#pragma unroll
    for (int i = 0; i < 16; ++i) px.v[i] = 0u;
    px.left = px.right = 0u;
    px.pairs = false;
#pragma unroll 1
    for (;;) {
        // the batch after this one
        if (8 * (tl + 1) < nl) {
            ++tl;
        } else {
            u += step;
            ld = u < n ? nxt : none;
            if (u + step < n) nxt = unit_at(list, u + step);
            tl = 0;
            bl ^= 1;
            if (ld.mask) {
                d = planes[ld.plane];
                vec = ((reinterpret_cast<uintptr_t>(d.img) | (unsigned)d.pitch) & 15u) == 0;
            }
            uint32_t need = 0u;  // bit i: source row y0 - sy + i is read
#pragma unroll
            for (int i = 0; i < WH; ++i) need |= ld.mask << i;
            nl = __popc(need);
            if ((need >> lane) & 1u) {
                sm.need_row[bl][__popc(need & lt)] = lane;
                // the later batches' rows on their way to the L2 while the first is loaded
                const int yr = ld.y0 - sy + lane;
                if (yr >= 0 && yr < d.Hs) {
                    const uint8_t *p = d.img + (long long)d.k * yr * d.pitch;
                    for (int o = 0; o < kUnitPx * d.k; o += 128)
                        if (d.k * ld.x0 + o < d.W)
                            asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p + d.k * ld.x0 + o));
                }
            }
            __syncwarp();
        }
        RowPx px2;
        const int q = 8 * tl + slot, r2 = q < nl ? sm.need_row[bl][q] : 0, yr = ld.y0 - sy + r2;
        const bool on2 = q < nl && yr >= 0 && yr < d.Hs;
        load_row(d, ld.x0, yr, on2, j, vec, px2);
        if (n_need > 0) slice_row(px, on, j, sm.rows + r * kUnitPieces);
        px = px2;
        r = r2;
        on = on2;
        if (8 * (t + 1) < n_need) {
            ++t;
            continue;
        }
        if (cur.mask) {  // every source row is sliced: the codes
            const int n_rows = __popc(cur.mask);
            if ((cur.mask >> lane) & 1u) sm.row_of[slot_of_row(cur.mask, lane)] = lane;
            __syncwarp();
            const PlaneDesc c_d = planes[cur.plane];
            const int cols = min(kUnitPx, c_d.opitch - cur.x0);
#pragma unroll 1
            for (int q0 = 0; q0 < n_rows; q0 += 8) {
                bulk_wait_read();  // the codes staged before have been read
                __syncwarp();
                if (q0 + slot < n_rows) {
                    uint32_t lo[32], hi[32];
                    const int i = sm.row_of[q0 + slot];
                    word_codes<WW, WH>(c_d, cur.x0, cur.y0 + i, j, sm.rows + i * kUnitPieces, sentinel, lo, hi);
                    stage_codes(sm.codes + slot * kStageStride + j, lo, hi);
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                __syncwarp();
                if (lane < 8 && q0 + lane < n_rows)
                    bulk_row(c_d.out + (long long)(cur.y0 + sm.row_of[q0 + lane]) * c_d.opitch + cur.x0,
                             sm.codes + lane * kStageStride, cols);
            }
            __syncwarp();  // the unit's rows have been read
        }
        if (!ld.mask) break;
        cur = ld;
        t = 0;
        n_need = nl;
    }
    bulk_wait();
}

inline PlaneDesc desc_of(const Plane &pl)
{
    PlaneDesc d;
    d.img = pl.img;
    d.out = pl.out;
    d.W = pl.W;
    d.H = pl.H;
    d.pitch = pl.pitch;
    d.k = pl.k;
    d.Ws = pl.Ws;
    d.Hs = pl.Hs;
    d.opitch = (int)pl.opitch;
    d.vec_load = pl.vec_load;
    return d;
}

// Full image, fixed window: warp w of CTA (bx, by) takes columns 128 bx .. + 127 of the
// eight rows 8 (4 by + w) ..; a unit a warp, its codes staged where its rows were.
template <int WH>
union __align__(16) FullSmem {
    uint4 rows[(8 + WH - 1) * kUnitPieces];
    uint2 codes[8 * kStageStride];
};

struct PlanePair {
    PlaneDesc d[2];
};

// planes is indexed where it lies: without __grid_constant__ every thread copies it to
// local memory first (112 bytes of stack).  Images in a row, without and with it: 1920x1200
// 10.4 -> 9.6 us, 3840x2160 29.8 -> 27.0, 3839x2159 at half resolution 11.9 -> 11.5.
template <int WW, int WH>
__global__ void __launch_bounds__(kFullThreads, kFullCtas)
    census_full_unit_kernel(const __grid_constant__ PlanePair planes, int sentinel)
{
    const PlaneDesc &d = planes.d[blockIdx.z];  // one image, or two in one launch
    __shared__ FullSmem<WH> smem[kFullThreads / 32];
    constexpr int sy = WH / 2;
    const int lane = threadIdx.x & 31, j = lane & 3, slot = lane >> 2, warp = threadIdx.x >> 5;
    FullSmem<WH> &sm = smem[warp];
    const int x0 = blockIdx.x * kUnitPx, y0 = 8 * (blockIdx.y * (kFullThreads / 32) + warp);
    if (y0 >= d.Hs || x0 >= d.Ws) return;
    const bool vec = ((reinterpret_cast<uintptr_t>(d.img) | (unsigned)d.pitch) & 15u) == 0;
#pragma unroll 1
    for (int r0 = 0; r0 < 8 + WH - 1; r0 += 8) {
        const int r = r0 + slot, yr = y0 - sy + r;
        const bool on = r < 8 + WH - 1 && yr >= 0 && yr < d.Hs;
        RowPx px;
        load_row(d, x0, yr, on, j, vec, px);
        slice_row(px, on, j, sm.rows + (on ? r * kUnitPieces : 0));
    }
    __syncwarp();
    uint32_t lo[32], hi[32];
    const int rows = min(8, d.Hs - y0), cols = min(kUnitPx, d.Ws - x0);
    if (slot < rows) word_codes<WW, WH>(d, x0, y0 + slot, j, sm.rows + slot * kUnitPieces, sentinel, lo, hi);
    __syncwarp();  // the rows have been read
    if (slot < rows) stage_codes(sm.codes + slot * kStageStride + j, lo, hi);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncwarp();
    uint64_t *out = d.out + (long long)y0 * d.opitch + x0;
    if (((reinterpret_cast<uintptr_t>(d.out) & 15u) | (unsigned)(d.opitch & 1) | (unsigned)(cols & 1)) == 0) {
        if (lane < rows) bulk_row(out + (long long)lane * d.opitch, sm.codes + lane * kStageStride, cols);
        bulk_wait();
    } else {
        for (int i = 0; i < rows; ++i) {
            uint2 *dst = reinterpret_cast<uint2 *>(out + (long long)i * d.opitch);
            for (int c = lane; c < cols; c += 32) dst[c] = sm.codes[i * kStageStride + c];
        }
    }
}

// One 64-pixel tile of row y starting at x0 (x0 a multiple of 64).
__device__ __forceinline__ void census_tile(const Plane &pl, int x0, int y, int win_w, int win_h, int sentinel,
                                            const WarpStage &st)
{
    const int lane = threadIdx.x & 31;
    const int sx = win_w / 2, sy = win_h / 2;
    const int x = x0 + 2 * lane;
    if (y - sy < 0 || y + sy >= pl.Hs) {  // whole row undefined
        store_pair(pl, x, y, 0ull, 0ull);
        return;
    }
    stage_rows_any(pl, x0, y, sy, st, lane);
    __syncwarp();
    uint64_t c0 = code_any(st, 2 * lane, win_w, win_h, sentinel);
    uint64_t c1 = code_any(st, 2 * lane + 1, win_w, win_h, sentinel);
    if (x - sx < 0 || x + sx >= pl.Ws) c0 = 0ull;
    if (x + 1 - sx < 0 || x + 1 + sx >= pl.Ws) c1 = 0ull;
    store_pair(pl, x, y, c0, c1);
    __syncwarp();
}

// Full image: warp w of CTA (bx, by) takes tile bx of row by * 8 + w.
__global__ void __launch_bounds__(32 * kWarpsPerCta) census_full_kernel(Plane pl, int win_w, int win_h,
                                                                        int sentinel)
{
    extern __shared__ __align__(16) uint32_t stage_mem[];
    const int warp = threadIdx.x >> 5;
    const int y = blockIdx.y * kWarpsPerCta + warp;
    if (y >= pl.Hs) return;
    const WarpStage st = warp_stage(stage_mem, warp, win_h);
    census_tile(pl, blockIdx.x * kTile, y, win_w, win_h, sentinel, st);
}

// Region of interest.  The planner marks, per plane row, the 32-pixel tiles the
// search reads (bitmap, one bit per tile).  A list kernel compacts the marks into a
// dense list -- units for the fixed windows (unit_list_kernel), else tiles, one packed
// entry each (tile_list_kernel) -- and clears the bitmap for the next call; the census
// kernels then take their work from the list, so no warp scans empty bitmap words.
//
// Entry: bits 0-9 tile (x0 / 32), 10-25 row, 26-27 plane (L1, R1, Lk, Rk), 28- frame.
__device__ __forceinline__ unsigned long long tile_entry(int f, int q, int y, int tile)
{
    return ((unsigned long long)f << 28) | ((unsigned long long)q << 26) | ((unsigned long long)y << 10) |
           (unsigned long long)tile;
}

// Plane descriptor, tile origin and row of a list entry; false if the tile lies
// outside its plane.
__device__ __forceinline__ bool tile_of(const MatchArgs &a, unsigned long long e, PlaneDesc &d, int &x0, int &y)
{
    const int tile = (int)(e & 1023u);
    y = (int)((e >> 10) & 0xffffu);
    d = a.ws.planes[e >> 26];  // frame * 4 + plane
    x0 = tile * kCensusTilePx;
    return x0 < d.Ws && y < d.Hs;
}

__global__ void __launch_bounds__(256) tile_list_kernel(MatchArgs a)
{
    __shared__ int warp_tot[8];
    __shared__ int s_base;
    const int nf = a.ws.counts->n_frames;  // clamped by the planner
    const long long total = (long long)nf * a.ws.bm_frame_words;
    const long long w0 = (long long)blockIdx.x * blockDim.x;
    if (w0 >= total) return;  // uniform per CTA
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long w = w0 + tid;
    uint32_t bits = 0u;
    if (w < total) {
        bits = a.ws.bitmap[w];
        if (bits) a.ws.bitmap[w] = 0u;  // consumed: clear for the next call
    }
    const int cnt = __popc(bits);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    int wpre = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        wpre += i < warp ? warp_tot[i] : 0;
        tot += warp_tot[i];
    }
    if (tid == 0) s_base = tot ? atomicAdd(&a.ws.counts->n_tiles, tot) : 0;
    __syncthreads();
    if (bits == 0u) return;
    const int f = (int)(w / a.ws.bm_frame_words);
    int r = (int)(w - (long long)f * a.ws.bm_frame_words);
    int q = 0;
    while (q < 3 && r >= a.ws.bm_plane_off[q + 1]) ++q;
    r -= a.ws.bm_plane_off[q];
    const int y = r / a.ws.bm_row_words[q];
    const int wi = r - y * a.ws.bm_row_words[q];
    int pos = s_base + wpre + incl - cnt;
    while (bits) {
        const int b = __ffs(bits) - 1;
        bits &= bits - 1u;
        a.ws.tiles[pos++] = tile_entry(f, q, y, wi * 32 + b);
    }
}

// Fixed windows: the units with marked tiles, 16 bytes each in the tile list's place (a
// bitmap word's 32 rows make at most 16): marked rows of the unit, its first column and
// row, frame * 4 + plane.  A warp takes 32 rows of one bitmap word column, a row per lane.
static_assert(2 * kRoiRows == 32, "two units a bitmap word and 32 rows");

struct BandShape {
    int off[5];  // first (32-row band, word column) item of each plane in a frame, and their number
};

__global__ void __launch_bounds__(256) unit_list_kernel(MatchArgs a, BandShape bands)
{
    __shared__ int warp_units[8], warp_tiles[8];
    __shared__ int s_base;
    const unsigned full = 0xffffffffu;
    const long long total = (long long)a.ws.counts->n_frames * bands.off[4];  // clamped by the planner
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long item = (long long)blockIdx.x * 8 + warp;
    if ((long long)blockIdx.x * 8 >= total) return;  // uniform per CTA
    uint32_t mine = 0u;  // lane 16 h + u: marked rows of unit u of the h-th half of the rows
    int col = 0;         // and its first tile of the word
    int tiles = 0, f = 0, q = 0, band = 0, wi = 0;
    if (item < total) {
        f = (int)(item / bands.off[4]);
        int r = (int)(item - (long long)f * bands.off[4]);
        while (q < 3 && r >= bands.off[q + 1]) ++q;
        r -= bands.off[q];
        const int words = a.ws.bm_row_words[q], rows = (a.ws.bm_plane_off[q + 1] - a.ws.bm_plane_off[q]) / words;
        band = r / words;
        wi = r - band * words;
        const int y = band * 32 + lane;
        uint32_t bits = 0u;
        if (y < rows) {
            uint32_t *p = a.ws.bitmap + f * a.ws.bm_frame_words + a.ws.bm_plane_off[q] + (long long)y * words + wi;
            bits = *p;
            if (bits) *p = 0u;  // consumed: clear for the next call
        }
        tiles = __reduce_add_sync(full, __popc(bits));
        // per half of the rows, units from the first marked column not covered yet
        const unsigned half = lane < kRoiRows ? 0x0000ffffu : 0xffff0000u;
        uint32_t left = __reduce_or_sync(half, bits);
        for (int u = 0; __any_sync(full, left != 0u); ++u) {  // at most 8: each takes four columns
            const int c = left ? __ffs(left) - 1 : 0;
            const uint32_t m = __ballot_sync(full, left && ((bits >> c) & 15u) != 0u) & half;
            if ((lane & 15) == u) {
                mine = lane < kRoiRows ? m : m >> kRoiRows;
                col = c;
            }
            left &= ~(15u << c);
        }
    }
    const unsigned found = __ballot_sync(full, mine != 0u);
    if (lane == 0) {
        warp_units[warp] = __popc(found);
        warp_tiles[warp] = tiles;
    }
    __syncthreads();
    int pre = 0, tot = 0, ttot = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        pre += i < warp ? warp_units[i] : 0;
        tot += warp_units[i];
        ttot += warp_tiles[i];
    }
    if (tot == 0) return;  // uniform per CTA
    if (threadIdx.x == 0) {
        s_base = atomicAdd(&a.ws.counts->n_units, tot);
        atomicAdd(&a.ws.counts->n_tiles, ttot);
    }
    __syncthreads();
    if (mine != 0u)
        reinterpret_cast<uint4 *>(a.ws.tiles)[s_base + pre + __popc(found & ((1u << lane) - 1u))] =
            make_uint4(mine, (unsigned)((wi * 32 + col) * kCensusTilePx),
                       (unsigned)(band * 32 + (lane & kRoiRows)), (unsigned)(f * 4 + q));
}

template <int WW, int WH>
__global__ void __launch_bounds__(kUnitThreads, kUnitCtas) census_unit_kernel(MatchArgs a)
{
    __shared__ UnitSmem<WH> sm[kUnitThreads / 32];
    const int warp = threadIdx.x >> 5;
    census_units<WW, WH>(reinterpret_cast<const uint4 *>(a.ws.tiles), a.ws.planes,
                         (int)(blockIdx.x + gridDim.x * warp), a.ws.counts->n_units,
                         (int)gridDim.x * (kUnitThreads / 32), a.p.sentinel, sm[warp]);
}

// Any other window: a warp per listed tile, rows staged in shared memory.
__global__ void __launch_bounds__(32 * kWarpsPerCta) census_roi_kernel(MatchArgs a)
{
    extern __shared__ __align__(16) uint32_t stage_mem[];
    const int warp = threadIdx.x >> 5;
    const WarpStage st = warp_stage(stage_mem, warp, a.p.win_h);
    const int n = a.ws.counts->n_tiles;
    const int nw = gridDim.x * kWarpsPerCta;
    for (int t = blockIdx.x * kWarpsPerCta + warp; t < n; t += nw) {
        PlaneDesc d;
        int x0, y;
        if (!tile_of(a, a.ws.tiles[t], d, x0, y)) continue;
        Plane pl;
        pl.img = d.img;
        pl.W = d.W;
        pl.H = 0;
        pl.pitch = d.pitch;
        pl.k = d.k;
        pl.Ws = d.Ws;
        pl.Hs = d.Hs;
        pl.out = d.out;
        pl.opitch = d.opitch;
        pl.vec_ok = 1;  // workspace planes: 256-byte aligned, pitch a multiple of 32
        pl.vec_load = d.vec_load;
        census_tile(pl, x0, y, a.p.win_w, a.p.win_h, a.p.sentinel, st);
    }
}

template <typename K>
int resident_ctas(K kernel, int threads, size_t smem)
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = 1;
    }
    return n;
}

}  // namespace

size_t census_smem_bytes(int win_h)
{
    return sizeof(uint32_t) * (size_t)kWarpsPerCta * 2 * win_h * kWordsMax;
}

static Plane plane_of(const CensusImage &c, int pitch, int k, long long out_pitch)
{
    Plane pl;
    pl.img = c.img;
    pl.W = c.W;
    pl.H = c.H;
    pl.pitch = pitch;
    pl.k = k;
    pl.Ws = ceil_div_nn(c.W, k);
    pl.Hs = ceil_div_nn(c.H, k);
    pl.out = c.out;
    pl.opitch = out_pitch;
    pl.vec_ok = (out_pitch % 2 == 0) && ((reinterpret_cast<uintptr_t>(c.out) & 15u) == 0);
    pl.vec_load = (k == 1 || k == 2) && (pitch % 4 == 0) && ((reinterpret_cast<uintptr_t>(c.img) & 7u) == 0);
    return pl;
}

cudaError_t launch_census_images(const CensusImage *images, int n, int pitch, int k, int win_w, int win_h,
                                 int sentinel, long long out_pitch, cudaStream_t s)
{
    PlanePair pair{};
    int Ws = 0, Hs = 0;
    for (int i = 0; i < n; ++i) {
        const Plane pl = plane_of(images[i], pitch, k, out_pitch);
        pair.d[i] = desc_of(pl);
        Ws = pl.Ws > Ws ? pl.Ws : Ws;
        Hs = pl.Hs > Hs ? pl.Hs : Hs;
        if (!census_fixed_window(win_w, win_h)) {
            const dim3 grid(ceil_div_nn(pl.Ws, kTile), ceil_div_nn(pl.Hs, kWarpsPerCta));
            census_full_kernel<<<grid, 32 * kWarpsPerCta, census_smem_bytes(win_h), s>>>(pl, win_w, win_h, sentinel);
        }
    }
    const dim3 units(ceil_div_nn(Ws, kUnitPx), ceil_div_nn(Hs, 8 * (kFullThreads / 32)), n);
    if (win_w == 9 && win_h == 7)
        census_full_unit_kernel<9, 7><<<units, kFullThreads, 0, s>>>(pair, sentinel);
    else if (win_w == 7 && win_h == 7)
        census_full_unit_kernel<7, 7><<<units, kFullThreads, 0, s>>>(pair, sentinel);
    else if (win_w == 5 && win_h == 5)
        census_full_unit_kernel<5, 5><<<units, kFullThreads, 0, s>>>(pair, sentinel);
    return cudaGetLastError();
}

int census_roi_ctas_per_sm(int win_w, int win_h)
{
    static const int n97 = resident_ctas(census_unit_kernel<9, 7>, kUnitThreads, 0);
    static const int n77 = resident_ctas(census_unit_kernel<7, 7>, kUnitThreads, 0);
    static const int n55 = resident_ctas(census_unit_kernel<5, 5>, kUnitThreads, 0);
    static const int ng = resident_ctas(census_roi_kernel, 32 * kWarpsPerCta, census_smem_bytes(kMaxWin));
    if (!census_fixed_window(win_w, win_h)) return ng;
    return win_h == 5 ? n55 : (win_w == 9 ? n97 : n77);
}

cudaError_t launch_census_roi(const MatchArgs &a, int sm_count, cudaStream_t s)
{
    const int ww = a.p.win_w, wh = a.p.win_h;
    const int grid = sm_count * census_roi_ctas_per_sm(ww, wh);
    // a marked tile's codes read grid columns [x0 - 4, x0 + 36) with the fixed windows,
    // [x0 - 8, x0 + 76) with the generic kernel: census_reach_left/right, which the mapped
    // entry point's gather copies, follow census_fixed_window's choice made here
    if (!census_fixed_window(ww, wh)) {
        const long long words = (long long)a.caps.max_frames * a.ws.bm_frame_words;
        const int list_grid = (int)((words + 255) / 256);
        if (list_grid > 0) tile_list_kernel<<<list_grid, 256, 0, s>>>(a);
        census_roi_kernel<<<grid, 32 * kWarpsPerCta, census_smem_bytes(wh), s>>>(a);
        return cudaGetLastError();
    }
    BandShape b;
    b.off[0] = 0;
    for (int q = 0; q < 4; ++q) {
        const int words = a.ws.bm_row_words[q], n = a.ws.bm_plane_off[q + 1] - a.ws.bm_plane_off[q];
        b.off[q + 1] = b.off[q] + (n > 0 ? ceil_div_nn(n / words, 32) * words : 0);
    }
    const long long items = (long long)a.caps.max_frames * b.off[4];
    if (items > 0) unit_list_kernel<<<(unsigned)((items + 7) / 8), 256, 0, s>>>(a, b);
    if (ww == 9)
        census_unit_kernel<9, 7><<<grid, kUnitThreads, 0, s>>>(a);
    else if (ww == 7)
        census_unit_kernel<7, 7><<<grid, kUnitThreads, 0, s>>>(a);
    else
        census_unit_kernel<5, 5><<<grid, kUnitThreads, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace ctm
