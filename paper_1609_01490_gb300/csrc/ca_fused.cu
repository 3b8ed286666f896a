// Several steps of Conway's rule per pass through memory (temporal blocking)
// on the triangular domain {0 <= j <= i < n} (the triangular-domain automaton
// of Section 1).  One warp per tile placed by a block map (Section 3): it reads
// the tile with a halo of 8 or 16 cells on every side, once, as one bit per cell,
// keeps the region in registers, takes up to 8 or 16 steps there and writes the
// tile's domain cells back.  A cell of the region is exact after s steps when
// it lies at least s cells inside the region, so the tile itself is; the halo
// cells are computed only to get it there.  After every step the cells outside
// the domain (j > i, i >= n, j < 0) are cleared, as the rule counts them dead.
//
// Long runs keep the grid as bits between passes: a first kernel packs the
// bytes, each pass reads and writes bits, a last kernel unpacks them.  Runs of up
// to 16 steps go from bytes to bytes in one pass (second half of the file).
//
// Bit layout of a region of 128 x 128 cells.  A row's column 4 b + w is bit b of
// word w, so a cell's side neighbours are the same bit of the neighbouring words,
// and only the first and the last word of a row need a shift (two a row instead
// of two funnel shifts a word in column order).  Lane l keeps rows 4 l .. 4 l + 3.
//
// What bounds a pass: the ALU pipe, ten logic operations per word and step (two
// full adders across the row and down the three rows, four for the rule) at 64
// lanes per clock and SM; ncu counts 11.7 ALU operations per word and step and
// the pipe 84% busy at n = 16384.
// 100 steps at n = 16384: 977 -> 500 us (bytes between passes of 16 steps and
// column-order words before), 469 with the passes launched behind one another; at n =
// 2000: 180 -> 66 us.  256 x 256-cell regions
// (8 words, 8 rows a lane) took 514 us: fewer halo cells, but a step's code no
// longer fits the instruction cache and the last wave runs nearly empty.
#include <cuda_runtime.h>

#include <algorithm>

#include "tri_internal.h"
#include "pdl.cuh"
#include "tri_maps.cuh"

using namespace tri;

namespace {

constexpr uint32_t FULLMASK = 0xFFFFFFFFu;
constexpr int W = 4;             // words per region row
constexpr int RPL = 4;           // region rows per lane
constexpr int REGION = 128;      // region side in cells
static_assert(32 * W == REGION && 32 * RPL == REGION, "a square region");

__device__ __forceinline__ int clamp_small(int64_t v) { return (int)(v < -4096 ? -4096 : (v > 4096 ? 4096 : v)); }

// The domain within a lane's rows: row r holds the domain's cells j <= i up to
// bit floor((base + r - w) / W) - 1 of word w (base = i - c0 + W for the lane's
// first row i and the region's first column c0); rows r >= rows lie past the
// grid; `left` clears the columns j < 0.  Values beyond +-4096 are clamped: only
// the region's 128 matter.
struct RowDomain {
    int base, rows;
    uint32_t left;
    __device__ __forceinline__ uint32_t mask(int r, int w) const
    {
        const int bits = (base + r - w) >> 2;  // / W, rounded down
        return r < rows ? ~__funnelshift_lc(0u, FULLMASK, (uint32_t)max(bits, 0)) & left : 0u;
    }
};

// One three-input logic operation: bit 4 a + 2 b + c of LUT.  Written out because
// the compiler, left to split the rule by itself, takes thirteen of them per word.
template <int LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(LUT));
    return d;
}
constexpr int XOR3 = 0x96, MAJ = 0xE8;

// `steps` steps of the region held by the warp, one word column at a time.  The
// sum of the 3 x 3 cells is o + 2 (k + x) + 4 y: s3 + 2 c3 sums a row's three, o
// and k add the s3 of three rows, x and y their c3.  A cell lives on iff the sum
// (itself included) is 3, or 4 with the cell alive.  The sums of the rows above
// a lane's first and below its last come from the neighbouring lanes by shuffle;
// the region's first and last rows are stepped from whatever their shuffles
// return: like every cell that lacks neighbours in the region, they are wrong
// after the first step, and the wrong rim grows one cell per step.
template <bool MASKED>
__device__ __forceinline__ void run_steps(uint32_t (&c)[RPL][W], uint32_t steps, const RowDomain &dom)
{
#pragma unroll 1
    for (uint32_t s = 0; s < steps; ++s) {
        uint32_t west[RPL], wrap[RPL];  // old word w - 1; old word 0 one column on
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            west[r] = c[r][W - 1] << 1;
            wrap[r] = c[r][0] >> 1;
        }
#pragma unroll
        for (int w = 0; w < W; ++w) {
            uint32_t s3[RPL], c3[RPL];
#pragma unroll
            for (int r = 0; r < RPL; ++r) {
                const uint32_t east = w + 1 < W ? c[r][w + 1 < W ? w + 1 : 0] : wrap[r];
                s3[r] = lop3<XOR3>(west[r], c[r][w], east);
                c3[r] = lop3<MAJ>(west[r], c[r][w], east);
                west[r] = c[r][w];
            }
            const uint32_t us = __shfl_up_sync(FULLMASK, s3[RPL - 1], 1), uc = __shfl_up_sync(FULLMASK, c3[RPL - 1], 1);
            const uint32_t ds = __shfl_down_sync(FULLMASK, s3[0], 1), dc = __shfl_down_sync(FULLMASK, c3[0], 1);
#pragma unroll
            for (int r = 0; r < RPL; ++r) {
                const uint32_t sa = r ? s3[r ? r - 1 : 0] : us, sb = r + 1 < RPL ? s3[r + 1 < RPL ? r + 1 : 0] : ds;
                const uint32_t ca = r ? c3[r ? r - 1 : 0] : uc, cb = r + 1 < RPL ? c3[r + 1 < RPL ? r + 1 : 0] : dc;
                const uint32_t o = lop3<XOR3>(sa, s3[r], sb), k = lop3<MAJ>(sa, s3[r], sb);
                const uint32_t x = lop3<XOR3>(ca, c3[r], cb), y = lop3<MAJ>(ca, c3[r], cb);
                const uint32_t two = lop3<0x14>(k, x, y);   // (k ^ x) & ~y: sum 2 or 3
                const uint32_t four = lop3<0x42>(k, x, y);  // k + x + 2 y = 2: sum 4 or 5
                uint32_t v = lop3<0xCA>(o, two, four & c[r][w]);  // o ? two : four and alive
                if constexpr (MASKED) v &= dom.mask(r, w);
                c[r][w] = v;
            }
        }
    }
}

// Where a state is kept between passes: tile number T = bi (bi + 1) / 2 + bj in
// RPL pieces, piece r holding the four words of row r of each of its 32 lanes, 16
// bytes a lane, so that a warp moves up to 512 contiguous bytes per instruction
// (pieces at each row's own address cost 25 us a pass in uncoalesced accesses at n
// = 16384).  Slot z = 32 T + lane of piece r sits in the domain cells of row r0 +
// r band + (z >> lp) at column 16 (z mod 2^lp): no byte outside the domain is
// written.  The words' halo bits are zero.
struct BitStore {
    uint32_t r0, band;
    int lp;
    __device__ __forceinline__ size_t slot(uint64_t T, int lane, size_t ld) const
    {
        const uint64_t z = 32 * T + lane;
        return (size_t)(r0 + (z >> lp)) * ld + 16 * (size_t)(z & ((1ull << lp) - 1));
    }
};

__device__ __forceinline__ uint64_t tile_number(int64_t bi, int64_t bj) { return (uint64_t)(bi * (bi + 1) / 2 + bj); }

// One pass: reads a stored state, takes up to `halo` steps, stores the next.
template <int MAP>
__global__ void __launch_bounds__(32, 28)
    ca_life_run_kernel(const uint8_t *in, uint8_t *out, uint32_t n, size_t ld, BlockMap bm,
                       uint32_t rows, uint32_t steps, int halo, BitStore store)
{
    dependents_may_start();
    wait_for_previous();
    uint32_t bi, bj;
    if (!map_block<MAP>(bm, bi, bj)) return;
    if (bi >= rows) return;  // REC covers a power of two of block rows
    const int lane = threadIdx.x, side = REGION - 2 * halo, hb = halo / W;
    const int64_t i0 = (int64_t)bi * side, j0 = (int64_t)bj * side, ib = i0 - halo;
    const int l0 = halo / RPL, l1 = 32 - l0;  // the lanes that hold the tile's rows
    const size_t piece = (size_t)store.band * ld;
    uint32_t c[RPL][W];
    {
        // the words of this lane's rows in its tile row's tiles bj - 1, bj, bj + 1:
        // the first l0 lanes hold rows of the tile row above, the last l0 of the one below
        const int64_t tr = lane < l0 ? (int64_t)bi - 1 : (lane >= l1 ? (int64_t)bi + 1 : (int64_t)bi);
        const int slot = lane < l0 ? lane + l1 - l0 : (lane >= l1 ? lane - (l1 - l0) : lane);
        const bool row = tr >= 0 && tr < (int64_t)rows;
        const bool own = row && (int64_t)bj <= tr, west = row && bj > 0 && (int64_t)bj - 1 <= tr;
        const bool east = row && (int64_t)bj + 1 <= tr;
        const uint64_t T = row ? tile_number(tr, bj) : 1;
        const uint8_t *pa = in + (own ? store.slot(T, slot, ld) : 0), *pw = in + (west ? store.slot(T - 1, slot, ld) : 0);
        const uint8_t *pe = in + (east ? store.slot(T + 1, slot, ld) : 0);
        // the neighbours' edge bits, moved by multiplies: the ALU pipe has enough to do
        const uint32_t up = 1u << (32 - 2 * hb), down = 1u << (2 * hb);
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            const uint4 a = own ? *reinterpret_cast<const uint4 *>(pa + r * piece) : zero;
            const uint4 l = west ? *reinterpret_cast<const uint4 *>(pw + r * piece) : zero;
            const uint4 e = east ? *reinterpret_cast<const uint4 *>(pe + r * piece) : zero;
            c[r][0] = __umulhi(l.x, down) + (e.x * up + a.x);
            c[r][1] = __umulhi(l.y, down) + (e.y * up + a.y);
            c[r][2] = __umulhi(l.z, down) + (e.z * up + a.z);
            c[r][3] = __umulhi(l.w, down) + (e.w * up + a.w);
        }
    }
    // every cell of the region lies in the domain
    if (bj > 0 && i0 - j0 >= REGION - 1 && ib + REGION <= (int64_t)n) {
        run_steps<false>(c, steps, RowDomain{});
    } else {
        RowDomain dom;
        dom.base = clamp_small(i0 - j0) + lane * RPL + W;
        dom.rows = clamp_small((int64_t)n - (ib + lane * RPL));
        dom.left = bj == 0 ? FULLMASK << hb : FULLMASK;
        run_steps<true>(c, steps, dom);
    }
    if (lane < l0 || lane >= l1) return;
    uint8_t *dst = out + store.slot(tile_number(bi, bj), lane, ld);
    const uint32_t mid = (FULLMASK << hb) & (FULLMASK >> hb);
#pragma unroll
    for (int r = 0; r < RPL; ++r)
        *reinterpret_cast<uint4 *>(dst + r * piece) = make_uint4(c[r][0] & mid, c[r][1] & mid, c[r][2] & mid, c[r][3] & mid);
}

// Bytes to a stored state and back: one block per tile, warp r for row r of every
// lane, eight rows' loads or stores in flight per warp.  A byte row's column
// group b (4 cells) belongs to lane b; word w is the ballot of the lanes' w-th
// cells.  Bound by the grid's bytes and, next, by issue (27 instructions a row).
template <int MAP>
__global__ void __launch_bounds__(32 * RPL)
    ca_life_pack_kernel(const uint8_t *__restrict__ in, uint8_t *__restrict__ out, uint32_t n, size_t ld, BlockMap bm,
                        uint32_t rows, int halo, BitStore store)
{
    dependents_may_start();
    uint32_t bi, bj;
    if (!map_block<MAP>(bm, bi, bj)) return;
    if (bi >= rows) return;
    const int lane = threadIdx.x & 31, r = threadIdx.x >> 5, side = REGION - 2 * halo;
    const int l0 = halo / RPL, l1 = 32 - l0;
    const int64_t i0 = (int64_t)bi * side, j0 = (int64_t)bj * side, col = j0 - halo + W * lane;
    const bool mine = W * lane >= halo && W * lane < halo + side;
    uint32_t c[W] = {};
    // the tile's rows RPL apart; a tile wholly inside the domain needs no tests
    const int64_t first = i0 + r;
    const uint8_t *src = in + (mine ? (size_t)first * ld + (size_t)col : 0);
    const size_t pitch = (size_t)RPL * ld;
    const auto rows_of = [&](auto tag) {
        constexpr bool inside = decltype(tag)::value;
        const int left = clamp_small((int64_t)n - first), ahead = clamp_small(first - col);
#pragma unroll 8
        for (int l = l0; l < l1; ++l, src += pitch) {
            // a group that starts at a column in [0, n) lies inside the row (ld >= n, both multiples of 4)
            const int k = (l - l0) * RPL;
            const bool ok = mine && (inside || (k < left && ahead + k >= 0));
            const uint32_t v = ok ? *reinterpret_cast<const uint32_t *>(src) : 0u;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const uint32_t word = __ballot_sync(FULLMASK, ((v >> (8 * w)) & 0xFFu) && (inside || w <= ahead + k));
                if (lane == l) c[w] = word;
            }
        }
    };
    if (bj < bi && i0 + side <= (int64_t)n) rows_of(std::true_type{});
    else rows_of(std::false_type{});
    if (lane >= l0 && lane < l1)
        *reinterpret_cast<uint4 *>(out + store.slot(tile_number(bi, bj), lane, ld) + r * ((size_t)store.band * ld)) =
            make_uint4(c[0], c[1], c[2], c[3]);
}

template <int MAP>
__global__ void __launch_bounds__(32 * RPL)
    ca_life_unpack_kernel(const uint8_t *in, uint8_t *out, uint32_t n, size_t ld,
                          BlockMap bm, uint32_t rows, int halo, BitStore store)
{
    wait_for_previous();
    uint32_t bi, bj;
    if (!map_block<MAP>(bm, bi, bj)) return;
    if (bi >= rows) return;
    const int lane = threadIdx.x & 31, r = threadIdx.x >> 5, side = REGION - 2 * halo;
    const int l0 = halo / RPL, l1 = 32 - l0;
    const int64_t i0 = (int64_t)bi * side, j0 = (int64_t)bj * side, col = j0 - halo + W * lane;
    const bool mine = W * lane >= halo && W * lane < halo + side;
    __shared__ uint4 s_rows[RPL][32];
    if (lane >= l0 && lane < l1)
        s_rows[r][lane] = *reinterpret_cast<const uint4 *>(in + store.slot(tile_number(bi, bj), lane, ld) +
                                                           r * ((size_t)store.band * ld));
    __syncwarp();
    const int64_t first = i0 + r;
    uint8_t *dst = out + (mine ? (size_t)first * ld + (size_t)col : 0);
    const size_t pitch = (size_t)RPL * ld;
    const auto rows_of = [&](auto tag) {
        constexpr bool inside = decltype(tag)::value;
        const int left = clamp_small((int64_t)n - first), ahead = clamp_small(first - col);
#pragma unroll 8
        for (int l = l0; l < l1; ++l, dst += pitch) {
            const uint4 v = s_rows[r][l];
            const uint32_t y = ((v.x >> lane) & 1u) + 256u * ((v.y >> lane) & 1u) + 65536u * ((v.z >> lane) & 1u) +
                               16777216u * ((v.w >> lane) & 1u);
            const int k = (l - l0) * RPL;
            if (!mine || !(inside || (k < left && ahead + k >= 0))) continue;
            if (inside || ahead + k >= W - 1) {
                *reinterpret_cast<uint32_t *>(dst) = y;
            } else {
                for (int q = 0; q <= ahead + k; ++q) dst[q] = (uint8_t)(y >> (8 * q));
            }
        }
    };
    if (bj < bi && i0 + side <= (int64_t)n) rows_of(std::true_type{});
    else rows_of(std::false_type{});
}

// The rows a state's slots go to: 2^lp slots a row from row 16 2^lp - 1 on (the
// first whose domain holds them), lp the largest that leaves room for every
// piece; false when the grid is too small for them.
bool bit_store(uint32_t n, uint32_t rows, BitStore &b)
{
    for (int lp = 20; lp >= 0; --lp) {
        const uint64_t r0 = (16ull << lp) - 1, band = ((T2(rows) * 32 - 1) >> lp) + 1;
        if (r0 >= n || r0 + band * RPL > n) continue;
        b.r0 = (uint32_t)r0;
        b.band = (uint32_t)band;
        b.lp = lp;
        return true;
    }
    return false;
}

// Runs `steps` steps in passes of `halo`, from and to bytes; -1 when the grid
// cannot hold the states between passes.
int run_fused(const uint8_t *in, uint8_t *out, uint8_t *scratch, uint32_t n, size_t ld, int map, uint32_t steps,
              int halo, cudaStream_t s)
{
    const uint32_t side = REGION - 2 * halo, rows = (n + side - 1) / side, passes = (steps + halo - 1) / halo;
    BitStore store{};
    if (!bit_store(n, rows, store)) return -1;
    uint32_t m = rows;
    if (map == TRI_MAP_REC)
        for (m = 1; m < rows;) m *= 2;
    // state p (after p passes) lies in `scratch` when passes - p is even, else in
    // `out`: the last one in `scratch`, from which `out` gets its bytes
    auto at = [&](uint32_t p) { return (passes - p) % 2 == 0 ? scratch : out; };
    int r = trihost::map_launches(map, m, [&](auto tag, dim3 g, const BlockMap &bm) -> cudaError_t {
        ca_life_pack_kernel<decltype(tag)::value><<<g, 32 * RPL, 0, s>>>(in, at(0), n, ld, bm, rows, halo, store);
        return cudaGetLastError();
    });
    for (uint32_t p = 0; p < passes && r == TRI_OK; ++p) {
        const uint32_t k = std::min((uint32_t)halo, steps - p * halo);
        r = trihost::map_launches(map, m, [&](auto tag, dim3 g, const BlockMap &bm) -> cudaError_t {
            return trihost::launch_behind(ca_life_run_kernel<decltype(tag)::value>, g, 32, 0, s, at(p), at(p + 1), n, ld,
                                          bm, rows, k, halo, store);
        });
    }
    if (r != TRI_OK) return r;
    return trihost::map_launches(map, m, [&](auto tag, dim3 g, const BlockMap &bm) -> cudaError_t {
        return trihost::launch_behind(ca_life_unpack_kernel<decltype(tag)::value>, g, 32 * RPL, 0, s, scratch, out, n, ld,
                                      bm, rows, halo, store);
    });
}

// Passes of 8 steps recompute less halo (1.31 times the tiles' cells against 1.78
// for passes of 16), but there are twice as many, 5 us apart at the least: 100
// steps under lambda take, in us (16 / 8 steps a pass), n = 3000: 61 / 76, 6000:
// 121 / 148, 8000: 173 / 181, 9000: 199 / 193, 12000: 311 / 276, 16384: 561 / 469
// (the passes launched behind one another; in stream order 16384: 576 / 500).
constexpr uint32_t THIN_HALO_N = 8500;

// ------------------------------------------------------- up to 16 steps ----
// Runs of up to 16 steps (which need no scratch), and grids too small to keep a
// state between passes: one pass from bytes to bytes.  128 x 128-cell tiles, the
// region's words in column order, lane l holding region rows 5 l .. 5 l + 4.
constexpr uint32_t TS = 128;                 // tile side in cells (the rho = 32 tile of tri_ca_step)
constexpr int KH = 16;                       // halo in cells on each side, and steps per pass
constexpr uint32_t WPR = 5;                  // words per region row: columns j0 - 16 .. j0 + 143
constexpr uint32_t ROWS = TS + 2 * KH;       // region rows: i0 - 16 .. i0 + 143
constexpr uint32_t TILE_RPL = ROWS / 32;          // region rows per lane
static_assert(TILE_RPL * 32 == ROWS, "one warp holds the region");
static_assert(KH <= 16, "the halo must fit the 16-cell margins of the region's words");

// Four bytes -> four bits at 0 .. 3 (byte k non-zero -> bit k).  Bit 7 of
// each byte of t marks a non-zero byte: its low seven bits plus 0x7F carry
// into bit 7 unless all zero, and a byte >= 0x80 has it already.  Times
// 2^21 + 2^14 + 2^7 + 1, bits 7, 15, 23, 31 land at 28, 29, 30, 31; every
// other product bit lands below 28 or past 31, each at its own position, so
// nothing carries into the top four.
__device__ __forceinline__ uint32_t nib_of(uint32_t x)
{
    const uint32_t t = (((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x) & 0x80808080u;
    return (t * 0x00204081u) >> 28;
}

// 16 bytes -> 16 bits
__device__ __forceinline__ uint32_t pack16(const uint4 q)
{
    return nib_of(q.x) + 16u * (nib_of(q.y) + 16u * (nib_of(q.z) + 16u * nib_of(q.w)));
}

// bit k of a nibble -> byte k = 0 or 1: the multiply puts copies of bit k at
// k, k + 7, k + 14, k + 21, and only the copy at 8k falls on a byte's bit 0.
__device__ __forceinline__ uint32_t bits4_to_bytes(uint32_t nib) { return (nib * 0x00204081u) & 0x01010101u; }

// bits lo .. hi of a word (empty when hi < lo), for any ints
__device__ __forceinline__ uint32_t span_bits(int lo, int hi)
{
    lo = lo > 0 ? lo : 0;
    hi = hi < 31 ? hi : 31;
    if (hi < lo) return 0u;
    return (0xFFFFFFFFu >> (31 - hi)) & (0xFFFFFFFFu << lo);
}

// The domain within the region as small ints: region rows g in [ilo, ihi]
// are cell rows 0 .. n - 1, and row g holds the domain's region columns lo ..
// min(dd + g, lastrel) (dd = i0 - j0; lastrel = n - 1 - (j0 - 16); lo = 16
// in the first block column, where cell column 0 is region column 16).
// Values beyond +-4096 are clamped: only -1 .. 160 matter.
struct TileDomain {
    int lo, dd, lastrel, ilo, ihi;
    __device__ __forceinline__ uint32_t mask(int g, int w) const
    {
        if (g < ilo || g > ihi) return 0u;
        const int hi = min(dd + g, lastrel);
        return span_bits(lo - 32 * w, hi - 32 * w);
    }
    // every cell of the region lies in the domain
    __device__ __forceinline__ bool full() const
    {
        return lo == 0 && ilo == 0 && ihi >= (int)ROWS - 1 && dd >= (int)ROWS - 1 && lastrel >= (int)ROWS - 1;
    }
};

// For each word of a row: the sum of the cell and its two side neighbours as
// (s3 + 2 c3), and of the two side neighbours alone as (s2 + 2 c2), from the
// row's west and east planes (bit b of a word is region column 32 w + b).
__device__ __forceinline__ void row_sums(const uint32_t (&row)[WPR], uint32_t (&s3)[WPR], uint32_t (&c3)[WPR],
                                         uint32_t (&s2)[WPR], uint32_t (&c2)[WPR])
{
#pragma unroll
    for (uint32_t w = 0; w < WPR; ++w) {
        const uint32_t l = w ? row[w - 1] : 0u, r = w + 1 < WPR ? row[w + 1] : 0u;
        const uint32_t W = __funnelshift_l(l, row[w], 1), E = __funnelshift_r(row[w], r, 1);
        s2[w] = W ^ E;
        c2[w] = W & E;
        s3[w] = s2[w] ^ row[w];
        c3[w] = c2[w] | (row[w] & s2[w]);
    }
}

// `steps` steps of the region held by the warp.  Each row's sums are formed
// once, by the lane that holds it, and used by the rows above and below it;
// a lane gets the 3-sums of the row above its first and below its last from
// its neighbours by shuffle.  The region's first and last rows are stepped
// from whatever their shuffles return: like every cell that lacks neighbours
// in the region, they are wrong after the first step, and the wrong rim grows
// one cell per step.
template <bool MASKED>
__device__ __forceinline__ void tile_steps(uint32_t (&c)[TILE_RPL][WPR], uint32_t lane, uint32_t steps,
                                          const TileDomain &dom)
{
    for (uint32_t s = 0; s < steps; ++s) {
        // sums of the lane's first and last rows, formed once: their 3-sums go
        // to the neighbouring lanes by shuffle (as the sums of the row above
        // or below theirs) and all four are used here
        uint32_t fs3[WPR], fc3[WPR], fs2[WPR], fc2[WPR], ls3[WPR], lc3[WPR], ls2[WPR], lc2[WPR];
        row_sums(c[0], fs3, fc3, fs2, fc2);
        row_sums(c[TILE_RPL - 1], ls3, lc3, ls2, lc2);
        uint32_t ps3[WPR], pc3[WPR], ds3[WPR], dc3[WPR];
#pragma unroll
        for (uint32_t w = 0; w < WPR; ++w) {
            ps3[w] = __shfl_up_sync(0xFFFFFFFFu, ls3[w], 1);
            pc3[w] = __shfl_up_sync(0xFFFFFFFFu, lc3[w], 1);
            ds3[w] = __shfl_down_sync(0xFFFFFFFFu, fs3[w], 1);
            dc3[w] = __shfl_down_sync(0xFFFFFFFFu, fc3[w], 1);
        }
        uint32_t cs3[WPR], cc3[WPR], cs2[WPR], cc2[WPR];
#pragma unroll
        for (uint32_t w = 0; w < WPR; ++w) {
            cs3[w] = fs3[w];
            cc3[w] = fc3[w];
            cs2[w] = fs2[w];
            cc2[w] = fc2[w];
        }
#pragma unroll
        for (uint32_t r = 0; r < TILE_RPL; ++r) {
            uint32_t ns3[WPR], nc3[WPR], ns2[WPR], nc2[WPR];
            if (r + 2 < TILE_RPL) {
                row_sums(c[r + 1], ns3, nc3, ns2, nc2);
            } else if (r + 2 == TILE_RPL) {
#pragma unroll
                for (uint32_t w = 0; w < WPR; ++w) {
                    ns3[w] = ls3[w];
                    nc3[w] = lc3[w];
                    ns2[w] = ls2[w];
                    nc2[w] = lc2[w];
                }
            } else {  // the row below the lane's last: its 3-sums from the next lane
#pragma unroll
                for (uint32_t w = 0; w < WPR; ++w) {
                    ns3[w] = ds3[w];
                    nc3[w] = dc3[w];
                    ns2[w] = 0u;
                    nc2[w] = 0u;
                }
            }
#pragma unroll
            for (uint32_t w = 0; w < WPR; ++w) {
                // the 8 neighbours: (ps3 + 2 pc3) + (ns3 + 2 nc3) + (cs2 + 2 cc2)
                // = x1 + 2 (x2 + y1) + 4 y2
                const uint32_t x1 = ps3[w] ^ ns3[w] ^ cs2[w];
                const uint32_t x2 = (ps3[w] & ns3[w]) | (cs2[w] & (ps3[w] ^ ns3[w]));
                const uint32_t y1 = pc3[w] ^ nc3[w] ^ cc2[w];
                const uint32_t y2 = (pc3[w] & nc3[w]) | (cc2[w] & (pc3[w] ^ nc3[w]));
                // alive next: count 3, or count 2 and alive now (>= 4 when x2 & y1 or y2)
                uint32_t v = (x2 ^ y1) & ~((x2 & y1) | y2) & (x1 | c[r][w]);
                if constexpr (MASKED) v &= dom.mask((int)(lane * TILE_RPL + r), (int)w);
                c[r][w] = v;
            }
#pragma unroll
            for (uint32_t w = 0; w < WPR; ++w) {
                ps3[w] = cs3[w];
                pc3[w] = cc3[w];
                cs3[w] = ns3[w];
                cc3[w] = nc3[w];
                cs2[w] = ns2[w];
                cc2[w] = nc2[w];
            }
        }
    }
}

// 128 registers a thread (16 warps per SM; a few spill in the masked form):
// the ALU pipe, not occupancy, bounds the steps
template <int MAP>
__global__ void __launch_bounds__(32, 16) ca_life_tile_kernel(const uint8_t *__restrict__ in, uint8_t *__restrict__ out,
                                                             uint32_t n, size_t ld, BlockMap bm, uint32_t steps)
{
    uint32_t bi, bj;
    if (!map_block<MAP>(bm, bi, bj)) return;
    __shared__ uint32_t s_rows[ROWS * WPR];  // region row g, word w at g * WPR + w
    const uint32_t lane = threadIdx.x;
    const int64_t i0 = (int64_t)bi * TS, j0 = (int64_t)bj * TS;
    const int64_t ibase = i0 - KH, jbase = j0 - 16, last = (int64_t)n - 1;
    TileDomain dom;
    dom.lo = bj == 0 ? 16 : 0;
    dom.dd = clamp_small(i0 - j0);
    dom.lastrel = clamp_small(last - jbase);
    dom.ilo = clamp_small(ibase < 0 ? -ibase : 0);
    dom.ihi = clamp_small(last - ibase);
    const bool full = dom.full();

    // load: region word e = g * WPR + w, five words a lane at a time, every
    // load of a batch issued before any is used; a tile whose region lies
    // inside the domain needs no masks
#pragma unroll 1
    for (uint32_t b = 0; b < ROWS * WPR / 32; b += 5) {
        uint4 v[5][2];
        uint32_t mk[5];
#pragma unroll
        for (uint32_t k = 0; k < 5; ++k) {
            const uint32_t e = (b + k) * 32 + lane, g = e / WPR, w = e - g * WPR;
            if (full) {
                const uint8_t *src = in + (size_t)(ibase + g) * ld + (size_t)(jbase + 32 * (int64_t)w);
                mk[k] = 0xFFFFFFFFu;
                v[k][0] = *reinterpret_cast<const uint4 *>(src);
                v[k][1] = *reinterpret_cast<const uint4 *>(src + 16);
            } else {
                mk[k] = dom.mask((int)g, (int)w);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // a half word with a domain column starts at a column in [0, n - 1]:
                    // its 16-byte chunk lies inside the row (ld >= n, both multiples of 16)
                    v[k][h] = make_uint4(0, 0, 0, 0);
                    if ((mk[k] >> (16 * h)) & 0xFFFFu)
                        v[k][h] = *reinterpret_cast<const uint4 *>(in + (size_t)(ibase + g) * ld +
                                                                   (size_t)(jbase + 32 * (int64_t)w + 16 * h));
                }
            }
        }
#pragma unroll
        for (uint32_t k = 0; k < 5; ++k)
            s_rows[(b + k) * 32 + lane] = (pack16(v[k][0]) + 65536u * pack16(v[k][1])) & mk[k];
    }
    __syncwarp();
    // lane l takes region rows 5 l .. 5 l + 4 (a stride of 25 words: no bank conflicts)
    uint32_t c[TILE_RPL][WPR];
#pragma unroll
    for (uint32_t r = 0; r < TILE_RPL; ++r)
#pragma unroll
        for (uint32_t w = 0; w < WPR; ++w) c[r][w] = s_rows[(lane * TILE_RPL + r) * WPR + w];
    if (full)
        tile_steps<false>(c, lane, steps, dom);
    else
        tile_steps<true>(c, lane, steps, dom);
    __syncwarp();
#pragma unroll
    for (uint32_t r = 0; r < TILE_RPL; ++r)
#pragma unroll
        for (uint32_t w = 0; w < WPR; ++w) s_rows[(lane * TILE_RPL + r) * WPR + w] = c[r][w];
    __syncwarp();

    // the tile's domain cells: 128 rows x 8 chunks of 16 cells; chunk ch of
    // tile row rr is bits 16 + 16 ch .. + 15 of region row KH + rr (all of
    // them for a tile inside the domain)
#pragma unroll 4
    for (uint32_t e = lane; e < TS * 8; e += 32) {
        const uint32_t rr = e >> 3, ch = e & 7;
        const int64_t i = i0 + rr, col = j0 + 16 * (int64_t)ch;
        const uint32_t off = 16 + 16 * ch;
        const uint32_t b16 = s_rows[(KH + rr) * WPR + (off >> 5)] >> (off & 31);
        const uint4 q = make_uint4(bits4_to_bytes(b16 & 15u), bits4_to_bytes((b16 >> 4) & 15u),
                                   bits4_to_bytes((b16 >> 8) & 15u), bits4_to_bytes((b16 >> 12) & 15u));
        if (full) {
            *reinterpret_cast<uint4 *>(out + (size_t)i * ld + (size_t)col) = q;
            continue;
        }
        if (i > last || col > i) continue;
        uint8_t *dst = out + (size_t)i * ld + (size_t)col;
        const int64_t lastc = i < last ? i : last;  // the row's last domain column
        if (col + 15 <= lastc) {
            *reinterpret_cast<uint4 *>(dst) = q;
        } else {
            for (int64_t k = 0; k <= lastc - col; ++k) dst[k] = (uint8_t)((b16 >> k) & 1u);
        }
    }
}

int launch_tile_pass(int map, const uint8_t *in, uint8_t *out, uint32_t n, size_t ld, uint32_t steps, cudaStream_t s)
{
    const uint32_t m = (n + TS - 1) / TS;
    return trihost::map_launches(map, m, [&](auto tag, dim3 g, const BlockMap &bm) -> cudaError_t {
        constexpr int MAP = decltype(tag)::value;
        ca_life_tile_kernel<MAP><<<g, 32, 0, s>>>(in, out, n, ld, bm, steps);
        return cudaGetLastError();
    });
}


constexpr uint32_t LIFE_BIRTH_MASK = 1u << 3, LIFE_SURVIVE_MASK = (1u << 2) | (1u << 3);

bool overlap(const uint8_t *a, const uint8_t *b, size_t span) { return a < b + span && b < a + span; }

}  // namespace

extern "C" int tri_ca_run(const uint8_t *in, uint8_t *out, uint8_t *scratch, uint32_t n, size_t ld,
                          uint32_t birth_mask, uint32_t survive_mask, int map, uint32_t rho, uint32_t steps,
                          void *stream)
{
    if (!in || !out || n == 0 || steps == 0 || !trihost::rho_ok(rho)) return TRI_EINVAL;
    if (ld < n || (ld & 15) || ((uintptr_t)in & 15) || ((uintptr_t)out & 15) || ((uintptr_t)scratch & 15))
        return TRI_EINVAL;
    if ((birth_mask | survive_mask) >> 9) return TRI_EINVAL;
    if (map != TRI_MAP_LAMBDA && map != TRI_MAP_LAMBDA_PDELTA && map != TRI_MAP_BB && map != TRI_MAP_RB &&
        map != TRI_MAP_REC)
        return TRI_EINVAL;
    const bool fused = birth_mask == LIFE_BIRTH_MASK && survive_mask == LIFE_SURVIVE_MASK && rho == 32;
    // up to 16 steps run as one pass and need no scratch
    const uint32_t passes = fused ? (steps + 15) / 16 : steps;
    const size_t span = (size_t)(n - 1) * ld + n;
    if (overlap(in, out, span)) return TRI_EINVAL;
    if (passes > 1) {
        if (!scratch || overlap(scratch, in, span) || overlap(scratch, out, span)) return TRI_EINVAL;
    }
    // REC is placed over 128-cell block rows, fused or not: a size that those
    // do not divide into a power of two stays out of its range
    if (fused && map == TRI_MAP_REC && !trihost::is_pow2((n + 127) / 128)) return TRI_ERANGE;
    cudaStream_t s = (cudaStream_t)stream;
    if (fused && passes > 1) {
        int r = run_fused(in, out, scratch, n, ld, map, steps, n >= THIN_HALO_N ? 8 : 16, s);
        if (r < 0) r = run_fused(in, out, scratch, n, ld, map, steps, 8, s);  // fewer tiles to hold
        if (r >= 0) return r;
    }
    // pass p writes `out` when passes - 1 - p is even, `scratch` otherwise,
    // so the last pass writes `out` and `in` is only read
    const uint8_t *src = in;
    for (uint32_t p = 0; p < passes; ++p) {
        uint8_t *dst = ((passes - 1 - p) % 2 == 0) ? out : scratch;
        int r;
        if (fused)
            r = launch_tile_pass(map, src, dst, n, ld, std::min((uint32_t)KH, steps - p * KH), s);
        else
            r = tri_ca_step(src, dst, n, ld, birth_mask, survive_mask, map, rho, stream);
        if (r != TRI_OK) return r;
        src = dst;
    }
    return TRI_OK;
}
