// Collision detection of N spheres with random radii (Section 5, test 3), the
// paper's shared-memory workload: every block of a 2-D block map stages the
// spheres of its row and column tiles in shared memory and tests its pairs
// from registers.  UTM, a thread-space map, tests one pair per thread from
// global memory instead (the paper notes it cannot use the 2-D shared tile).
//
// The test of a pair i > j is s <= (r_i + r_j)^2 with
// s = (c_i0 - c_j0)^2 + (c_i1 - c_j1)^2 + ..., each step a separate FP32
// operation rounded to nearest (no fused multiply-add), so the decisions are
// exactly those of any other implementation that takes the same steps.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "f32x2.cuh"
#include "pdl.cuh"
#include "tri_internal.h"
#include "tri_maps.cuh"

using namespace tri;

namespace {

struct CollideOut {
    uint32_t *count;               // per-sphere counts, or null
    uint32_t *pairs;               // (i, j) list, or null
    uint64_t cap;                  // entries of the list
    unsigned long long *n_pairs;   // colliding pairs found
};

// The exact test in scalar FP32: the reference order of operations.
template <int DIM>
__device__ __forceinline__ bool hit_scalar(const float *a, const float *b)
{
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const float dk = __fsub_rn(a[k], b[k]);
        const float sq = __fmul_rn(dk, dk);
        s = k == 0 ? sq : __fadd_rn(s, sq);
    }
    const float rr = __fadd_rn(a[DIM], b[DIM]);
    return s <= __fmul_rn(rr, rr);
}

// A colliding pair: one slot of the list, one count for each sphere.
__device__ __forceinline__ void record(const CollideOut &o, uint32_t i, uint32_t j)
{
    const unsigned long long q = atomicAdd(o.n_pairs, 1ull);
    if (q < o.cap) {
        o.pairs[2 * q] = i;
        o.pairs[2 * q + 1] = j;
    }
    if (o.count) {
        atomicAdd(o.count + i, 1u);
        atomicAdd(o.count + j, 1u);
    }
}

// One S x S pair tile, S = RHO*R: rows i0 = bi S + [0, S), columns
// j0 = bj S + [0, S).  The 2 S spheres are staged transposed ([coordinate or
// radius][sphere]) in dynamic shared memory, the rows with each value duplicated
// into both halves of an 8-byte word.  Thread (ty, tx) owns rows ty + u RHO (u < R)
// and, for R >= 2, the column pairs 2 tx + 2 RHO v + {0, 1} (v < R/2), taken two at
// a time with f32x2 instructions.  Those only rule pairs out: ptxas fuses a packed
// product into the sum or difference after it, rounding modifiers or not, so a
// packed form of the exact test misses pairs that touch exactly (s = q).  They form
// s' - q', s' = s but for at most six roundings and q' from radii widened by
// 2^-19 of themselves and 2^-73, so that s' < q' wherever s <= q, also where squares
// vanish in FP32.  A set sign means that the pair may touch (NaNs never do); the
// thread keeps one bit per row, the OR of its pairs' signs.  Threads with such a row
// (a few per contact, plus the diagonal, where a sphere meets itself) form s' - q'
// again there and take the exact test, hit_scalar, of each such pair (i < n, j < i).
// (With one bit for all its rows a thread repeats 64 pairs for each contact: 65,536
// spheres in 3-D, reg = 8, took 0.97 ms, now 0.79; on a line 0.57, now 0.46; 9001
// discs with 400 contacts each 1.01, now 0.41.)  Sums of
// radii of either sign may cancel and lose the margin, and q' of huge ones is
// infinite: a tile with a negative radius, or one of 2^62 or more, takes the exact
// test for all its pairs.  Padding spheres past n sit at +inf (rows) and -inf
// (columns), where s' = inf.  For R = 1 each thread takes the exact test of its one
// pair.
// Not inlined: every block map calls the same body.
extern __shared__ __align__(16) unsigned char collide_smem[];

template <int RHO, int R, int DIM>
struct TileBytes {
    static constexpr int S = RHO * R, ROWS = (DIM + 1) * S * 8, BYTES = ROWS + (DIM + 1) * (S + 2) * 4;
};

template <int RHO, int R, int DIM>
__device__ __noinline__ void collide_tile(const float *__restrict__ c, const float *__restrict__ rad, uint32_t n,
                                          uint32_t bi, uint32_t bj, CollideOut o, int tx, int ty)
{
    constexpr int S = RHO * R;
    constexpr int RC = R == 1 ? 1 : R / 2;
    f2(*si)[S] = reinterpret_cast<f2(*)[S]>(collide_smem);  // rows, duplicated
    float(*sj)[S + 2] = reinterpret_cast<float(*)[S + 2]>(collide_smem + TileBytes<RHO, R, DIM>::ROWS);  // columns
    const int tid = ty * RHO + tx;
    const uint64_t i0 = (uint64_t)bi * S, j0 = (uint64_t)bj * S;
    const float inf = __int_as_float(0x7f800000);
    // coalesced staging of S consecutive spheres: centres (S DIM floats), then radii
    for (int t = tid; t < S * DIM; t += RHO * RHO) {
        const int r = t / DIM, k = t - r * DIM;
        const float a = i0 + r < n ? c[i0 * DIM + t] : inf;
        si[k][r] = f2_pack(a, a);
        sj[k][r] = j0 + r < n ? c[j0 * DIM + t] : -inf;
    }
    bool every = false;  // no margin: all pairs take the exact test
    for (int t = tid; t < S; t += RHO * RHO) {
        float a = i0 + t < n ? rad[i0 + t] : 0.0f, b = j0 + t < n ? rad[j0 + t] : 0.0f;
        every = every || fminf(a, b) < 0.0f || fmaxf(a, b) >= 4.6116860e18f;
        if constexpr (R > 1) {
            a = fmaf(a, 1.0000019f, 1.0587912e-22f);
            b = fmaf(b, 1.0000019f, 1.0587912e-22f);
        }
        si[DIM][t] = f2_pack(a, a);
        sj[DIM][t] = b;
    }
    if constexpr (R == 1) {
        __syncthreads();
        float a[DIM + 1], b[DIM + 1], dummy;
#pragma unroll
        for (int k = 0; k <= DIM; ++k) {
            f2_unpack(si[k][ty], a[k], dummy);
            b[k] = sj[k][tx];
        }
        const uint64_t i = i0 + ty, j = j0 + tx;
        if (hit_scalar<DIM>(a, b) && i < n && j < i) record(o, (uint32_t)i, (uint32_t)j);
        return;
    } else {
        every = __syncthreads_or(every);
        f2 b2[RC][DIM + 1];
#pragma unroll
        for (int v = 0; v < RC; ++v)
#pragma unroll
            for (int k = 0; k <= DIM; ++k) b2[v][k] = *reinterpret_cast<const f2 *>(&sj[k][2 * tx + 2 * RHO * v]);
        // s' - q' of the column pair v for row values a2: sign set if the pair may touch
        auto filter = [&](const f2 *a2, int v) {
            f2 s;
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                const f2 dk = f2_sub(a2[k], b2[v][k]);
                s = k == 0 ? f2_mul(dk, dk) : f2_fma(dk, dk, s);
            }
            const f2 rr = f2_add(a2[DIM], b2[v][DIM]);
            return f2_sub(s, f2_mul(rr, rr));
        };
        uint32_t near = 0;  // bit R - 1 - u: some pair of row u may touch
#pragma unroll
        for (int u = 0; u < R; ++u) {
            f2 a2[DIM + 1];
#pragma unroll
            for (int k = 0; k <= DIM; ++k) a2[k] = si[k][ty + u * RHO];
            uint32_t acc = 0;
#pragma unroll
            for (int v = 0; v < RC; ++v) {
                const f2 e = filter(a2, v);
                acc |= (uint32_t)e | (uint32_t)(e >> 32);
            }
            near = __funnelshift_l(acc, near, 1);
        }
        if (every) near = (1u << R) - 1u;
        // the exact test of the pairs that may touch.  Without a list one addition per
        // row and thread, and one of the thread's pairs.
        uint32_t found = 0;
        for (; near; near &= near - 1) {
            const int u = R - __ffs(near);
            const uint64_t i = i0 + ty + u * RHO;
            if (i >= n) continue;
            uint32_t row = 0;
            f2 a2[DIM + 1];
#pragma unroll
            for (int k = 0; k <= DIM; ++k) a2[k] = si[k][ty + u * RHO];
#pragma unroll
            for (int v = 0; v < RC; ++v) {
                const f2 e = filter(a2, v);
                const uint64_t j = j0 + 2 * tx + 2 * RHO * v;
                const bool lo = ((int)(uint32_t)e < 0 || every) && j < i;
                const bool hi = ((int)(uint32_t)(e >> 32) < 0 || every) && j + 1 < i;
                if (!lo && !hi) continue;
                float a[DIM + 1], b0[DIM + 1], b1[DIM + 1], dummy;
#pragma unroll
                for (int k = 0; k < DIM; ++k) {
                    f2_unpack(a2[k], a[k], dummy);
                    f2_unpack(b2[v][k], b0[k], b1[k]);
                }
                a[DIM] = rad[i];
                b0[DIM] = lo ? rad[j] : 0.0f;
                b1[DIM] = hi ? rad[j + 1] : 0.0f;
                const bool h0 = lo && hit_scalar<DIM>(a, b0), h1 = hi && hit_scalar<DIM>(a, b1);
                if (o.pairs) {
                    if (h0) record(o, (uint32_t)i, (uint32_t)j);
                    if (h1) record(o, (uint32_t)i, (uint32_t)(j + 1));
                } else {
                    row += (h0 ? 1u : 0u) + (h1 ? 1u : 0u);
                    if (o.count && h0) atomicAdd(o.count + j, 1u);
                    if (o.count && h1) atomicAdd(o.count + j + 1, 1u);
                }
            }
            found += row;
            if (o.count && row) atomicAdd(o.count + i, row);
        }
        if (found) atomicAdd(o.n_pairs, (unsigned long long)found);
    }
}

// ------------------------------------------------- tensor-core filter ----
// The library's own tile (reg = 0, 2-D and 3-D): FP16 tensor cores rule out the
// pairs that surely do not touch, and the few others take the exact test.
//
// With X = sigma (c - c0), R = sigma r (c0 and the power of two sigma chosen per
// block so that every |X_k|, |R| < 16),
//   sigma^2 (q - s) / 2 = u_i + u_j + R_i R_j + X_i . X_j,  u = (R^2 - |X|^2) / 2,
// is one inner product of 16 terms: X and R in two FP16 parts each (hi.hi',
// hi.lo', lo.hi' of up to four coordinates) and u in two.  Its error is below
// 2^-8: parts 2^-13, dropped lo.lo' 2^-14, u 2^-13, accumulation of terms up to
// 1792 with at least 23 fraction bits kept 2^-9, rounding of c - c0 and of the
// exact test's own operations 2^-11.  u carries 2^-9 extra per sphere, so a
// negative value proves s > q as the exact test computes it.  A sphere with an
// infinite or NaN coordinate, and every sphere of a block whose extent lies
// outside [2^-50, 2^60] (where the exact test's squares may overflow or
// vanish), gets u = 30000 and X = R = 0: its pairs always take the exact test.
// Padding past n gets u = -30000.
//
// mma.sync m16n8k16 leaves each thread its results in registers, so the test of
// 512 pairs per warp is 4 instructions on the tensor core, 8 three-input ANDs
// and a vote, against about 50 packed FP32 instructions.
// 65,536 spheres in 3-D take 215 us against 786 with the packed FP32 tile,
// 9001 in 2-D 13 against 19.  The tensor core bounds it (one m16n8k16 per SM
// takes 1.04 ns: 115 us), then the staging of each block's spheres.
// The margin is 3e-5 of the block's squared extent, so it flags few pairs unless
// most spheres crowd into a small part of that extent (or meet many others):
// each warp counts the flags of its first 512 pairs, and a block that finds more
// than 1 in 128 runs the packed FP32 tile instead: 1 in 4 where infinities or NaNs
// flag whole rows (18,000 spheres, one infinite radius: 33 us pair by pair, 104
// packed; every third a NaN: 283 and 122).  On a line (1-D) the margin
// alone flags 1 in 180 pairs (0.63 ms against 0.46): those keep the FP32 tile.
constexpr int MMA_THREADS = 256;
constexpr int MMA_BLOCKS = 4;
constexpr unsigned FULL = 0xFFFFFFFFu;

__device__ __forceinline__ float redux_min(float v)
{
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float redux_max(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// two floats rounded to FP16, a in the low half
__device__ __forceinline__ uint32_t half2_bits(float a, float b)
{
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ float2 half2_floats(uint32_t v)
{
    return __half22float2(*reinterpret_cast<const __half2 *>(&v));
}

// d (16 x 8, FP32) = a (16 x 16) b (16 x 8), FP16 operands
__device__ __forceinline__ void mma_16x8x16(const uint2 a0, const uint2 a1, const uint2 b, uint32_t (&d)[4])
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, "
        "%10, %10};"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
        : "r"(a0.x), "r"(a1.x), "r"(a0.y), "r"(a1.y), "r"(b.x), "r"(b.y), "f"(0.0f));
}

// AND of three words in one instruction (the sign tests' chain written with & took
// 229 us where this takes 218).
__device__ __forceinline__ uint32_t and3(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0x80;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// One S x S tile by 8 warps: S / 64 row groups of 64 rows (four 16-row operands
// kept in registers), the columns split among the warps that share one.
template <int S, int DIM>
__device__ __noinline__ void collide_tile_mma(const float *__restrict__ c, const float *__restrict__ rad, uint32_t n,
                                              uint32_t bi, uint32_t bj, CollideOut o)
{
    constexpr int NT = MMA_THREADS, NW = NT / 32, PER = 2 * S / NT;  // spheres staged per thread
    static_assert(S % 64 == 0 && S / 64 <= NW && PER >= 1, "row groups of 64 rows");
    // operand records (16 halves) of the S rows and S columns, then the spheres themselves
    uint4 *rec = reinterpret_cast<uint4 *>(collide_smem);
    float4 *pos = reinterpret_cast<float4 *>(collide_smem + 2 * S * 32);
    __shared__ float s_red[NW][2 * DIM + 1];
    __shared__ uint32_t s_flags[NW];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint64_t i0 = (uint64_t)bi * S, j0 = (uint64_t)bj * S;
    const float inf = __int_as_float(0x7f800000);

    // sphere e of the tile: e < S row i0 + e, else column j0 + e - S
    float v[PER][DIM + 1];
    bool live[PER], finite[PER];
    float lo[DIM], hi[DIM], rmax = 0.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        lo[k] = inf;
        hi[k] = -inf;
    }
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int e = tid + p * NT;
        const uint64_t g = e < S ? i0 + e : j0 + (e - S);
        live[p] = g < n;
        finite[p] = live[p];
#pragma unroll
        for (int k = 0; k < DIM; ++k) v[p][k] = live[p] ? c[g * DIM + k] : 0.0f;
        v[p][DIM] = live[p] ? rad[g] : 0.0f;
#pragma unroll
        for (int k = 0; k <= DIM; ++k) finite[p] = finite[p] && fabsf(v[p][k]) < inf;
        if (finite[p]) {
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                lo[k] = fminf(lo[k], v[p][k]);
                hi[k] = fmaxf(hi[k], v[p][k]);
            }
            rmax = fmaxf(rmax, fabsf(v[p][DIM]));
        }
    }
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const float a = redux_min(lo[k]), b = redux_max(hi[k]);
        if (lane == 0) {
            s_red[warp][2 * k] = a;
            s_red[warp][2 * k + 1] = b;
        }
    }
    rmax = redux_max(rmax);
    if (lane == 0) s_red[warp][2 * DIM] = rmax;
    bool odd = false;  // an infinite or NaN value
#pragma unroll
    for (int p = 0; p < PER; ++p) odd = odd || (live[p] && !finite[p]);
    odd = __syncthreads_or(odd);
    float c0[DIM], extent = 0.0f;
#pragma unroll
    for (int w = 0; w < NW; ++w) extent = fmaxf(extent, s_red[w][2 * DIM]);
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        float a = inf, b = -inf;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            a = fminf(a, s_red[w][2 * k]);
            b = fmaxf(b, s_red[w][2 * k + 1]);
        }
        c0[k] = a <= b ? 0.5f * a + 0.5f * b : 0.0f;
        if (a <= b) extent = fmaxf(extent, fmaxf(b - c0[k], c0[k] - a));
    }
    // sigma extent in [8, 16)
    const bool usable = extent >= 8.8817842e-16f && extent <= 1.1529215e18f;  // [2^-50, 2^60]
    const float sigma = usable ? __uint_as_float((uint32_t)(257 - (int)(__float_as_uint(extent) >> 23)) << 23) : 0.0f;
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int e = tid + p * NT;
        const bool ok = finite[p] && usable, column = S >= NT ? p >= S / NT : e >= S;
        // sigma c - sigma c0 rounds once, as sigma (c - c0) does: sigma is a power of two
        float X[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) X[k] = 0.0f;
#pragma unroll
        for (int k = 0; k < DIM; ++k) X[k] = ok ? fmaf(v[p][k], sigma, -sigma * c0[k]) : 0.0f;
        X[3] = ok ? v[p][DIM] * sigma : 0.0f;
        float u = X[3] * X[3];
#pragma unroll
        for (int k = 0; k < DIM; ++k) u = fmaf(-X[k], X[k], u);
        u = ok ? fmaf(0.5f, u, 0.001953125f) : (live[p] ? 30000.0f : -30000.0f);
        const uint32_t h0 = half2_bits(X[0], X[1]), h1 = half2_bits(X[2], X[3]);
        const float2 f0 = half2_floats(h0), f1 = half2_floats(h1);
        const uint32_t l0 = half2_bits(X[0] - f0.x, X[1] - f0.y), l1 = half2_bits(X[2] - f1.x, X[3] - f1.y);
        const float uh = __half2float(__float2half_rn(u));
        const uint32_t uu = half2_bits(uh, u - uh), one = 0x3C003C00u;
        // rows (hi, hi, lo, u, 1) against columns (hi, lo, hi, 1, u)
        rec[2 * e] = column ? make_uint4(h0, h1, l0, l1) : make_uint4(h0, h1, h0, h1);
        rec[2 * e + 1] = column ? make_uint4(h0, h1, one, uu) : make_uint4(l0, l1, uu, one);
        pos[e] = make_float4(v[p][0], DIM > 1 ? v[p][DIM > 1 ? 1 : 0] : 0.0f, DIM > 2 ? v[p][DIM > 2 ? 2 : 0] : 0.0f, v[p][DIM]);
    }
    __syncthreads();

    // A thread of quad t = lane % 4 takes words 2t and 2t + 1 of a record: the
    // inner index is permuted alike in both operands.
    const uint2 *words = reinterpret_cast<const uint2 *>(rec);
    constexpr int RG = S / 64, CS = NW / RG;             // row groups, warps per row group
    const int r0 = (warp % RG) * 64, part = warp / RG;   // this warp's rows, its share of the columns
    const int g = lane >> 2, t = lane & 3;
    uint2 a[4][2];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        a[m][0] = words[(r0 + 16 * m + g) * 4 + t];
        a[m][1] = words[(r0 + 16 * m + 8 + g) * 4 + t];
    }
    // a diagonal block needs no column past the group's last row
    const int jn = bi == bj ? (r0 + 64) / 8 : S / 8;
    const uint2 *bw = words + S * 4;
    uint32_t d[4][4];
    auto filter = [&](int jt) {
        const uint2 b = bw[(jt * 8 + g) * 4 + t];
#pragma unroll
        for (int m = 0; m < 4; ++m) mma_16x8x16(a[m][0], a[m][1], b, d[m]);
        uint32_t acc = d[0][0];
#pragma unroll
        for (int m = 0; m < 4; ++m) acc = and3(and3(acc, d[m][0], d[m][1]), d[m][2], d[m][3]);
        return (int)acc >= 0;
    };
    // bit 4 m + e: the value of row 16 m + g + 8 (e / 2), column 2 t + (e & 1) is not negative
    auto flags = [&]() {
        uint32_t mask = 0;
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int e = 0; e < 4; ++e) mask |= (~d[m][e] >> 31) << (4 * m + e);
        return mask;
    };
    // the trial: flags among each warp's first 512 pairs
    uint32_t first = part < jn && filter(part) ? __popc(flags()) : 0u;
    first = __reduce_add_sync(FULL, first);
    if (lane == 0) s_flags[warp] = first;
    __syncthreads();
    uint32_t total = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) total += s_flags[w];
    wait_for_previous();  // the outputs are zeroed from here on
    if (total > (odd ? NW * 512 / 4 : NW * 512 / 128)) {
        constexpr int Q = S / 128;  // packed FP32 tiles a side
        for (int w = 0; w < Q * Q; ++w) {
            const uint32_t ti = bi * Q + w / Q, tj = bj * Q + w % Q;
            if (tj > ti || (uint64_t)ti * 128 >= n) continue;
            __syncthreads();  // the previous tile's spheres have been read
            collide_tile<16, 8, DIM>(c, rad, n, ti, tj, o, tid & 15, tid >> 4);
        }
        return;
    }
    uint32_t hits = 0;
    for (int jt = part; jt < jn; jt += CS) {
        if (!__any_sync(FULL, filter(jt))) continue;
        for (uint32_t mask = flags(); mask; mask &= mask - 1) {
            const int bit = __ffs(mask) - 1;
            const int r = r0 + 16 * (bit >> 2) + g + 8 * ((bit >> 1) & 1), q = jt * 8 + 2 * t + (bit & 1);
            const uint64_t i = i0 + r, j = j0 + q;
            if (i >= n || j >= i) continue;
            const float4 pi = pos[r], pj = pos[S + q];
            const float va[4] = {pi.x, pi.y, pi.z, pi.w}, vb[4] = {pj.x, pj.y, pj.z, pj.w};
            float fa[DIM + 1], fb[DIM + 1];
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                fa[k] = va[k];
                fb[k] = vb[k];
            }
            fa[DIM] = va[3];
            fb[DIM] = vb[3];
            if (!hit_scalar<DIM>(fa, fb)) continue;
            if (o.pairs) {
                record(o, (uint32_t)i, (uint32_t)j);
            } else {
                ++hits;
                if (o.count) {
                    atomicAdd(o.count + i, 1u);
                    atomicAdd(o.count + j, 1u);
                }
            }
        }
    }
    // without a list the pairs are only counted: one atomic per warp, not one per pair
    const uint32_t w = __reduce_add_sync(FULL, hits);
    if (lane == 0 && w) atomicAdd(o.n_pairs, (unsigned long long)w);
}

template <int MAP, int S, int DIM>
__global__ void __launch_bounds__(MMA_THREADS, MMA_BLOCKS)
    collide_mma_kernel(const float *__restrict__ c, const float *__restrict__ rad, uint32_t n, CollideOut o,
                       BlockMap bm)
{
    uint32_t bi, bj;
    if (!map_block<MAP>(bm, bi, bj)) return;
    collide_tile_mma<S, DIM>(c, rad, n, bi, bj, o);
}

// Zeroes the outputs in one launch (two memsets cost two).
__global__ void collide_zero_kernel(uint32_t *__restrict__ count, uint32_t n, unsigned long long *__restrict__ n_pairs)
{
    dependents_may_start();
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) *n_pairs = 0ull;
    if (count && t < n) count[t] = 0u;
}

template <int S, int DIM>
int launch_mma(const float *c, const float *rad, uint32_t n, int map, CollideOut o, cudaStream_t s)
{
    const uint32_t m = (uint32_t)(((uint64_t)n + S - 1) / S);
    constexpr int smem = 2 * S * 48;
    return trihost::map_launches(map, m, [&](auto tag, dim3 g, const BlockMap &bm) -> cudaError_t {
        constexpr int MAP = decltype(tag)::value;
        if constexpr (MAP != MAP_REC) {
            if (smem > 40 * 1024) {
                const cudaError_t e = trihost::allow_smem(collide_mma_kernel<MAP, S, DIM>, smem);
                if (e != cudaSuccess) return e;
            }
            return trihost::launch_behind(collide_mma_kernel<MAP, S, DIM>, g, MMA_THREADS, smem, s, c, rad, n, o, bm);
        }
        return cudaErrorInvalidValue;
    });
}

// Tile side: the staging of 2 S spheres pays off over S^2 pairs, so the largest
// tile that still gives every SM several blocks.
template <int DIM>
int launch_filter(const float *c, const float *rad, uint32_t n, int map, CollideOut o, cudaStream_t s)
{
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const auto blocks = [&](uint64_t S) { return T2((n + S - 1) / S); };
    if (blocks(512) >= 4ull * nsm) return launch_mma<512, DIM>(c, rad, n, map, o, s);
    if (blocks(256) >= 2ull * nsm) return launch_mma<256, DIM>(c, rad, n, map, o, s);
    return launch_mma<128, DIM>(c, rad, n, map, o, s);
}

// 8 x 8 pairs per thread on 16 x 16 threads: registers capped at 64 so that
// four blocks share an SM (uncapped the tile takes over 100 and three fit,
// which leaves too few warps to cover the staging loads).
template <int MAP, int RHO, int R, int DIM>
__global__ void __launch_bounds__(RHO *RHO, (RHO == 16 && R == 8) ? 4 : 1)
    collide_kernel(const float *__restrict__ c, const float *__restrict__ rad, uint32_t n, CollideOut o, BlockMap bm)
{
    uint32_t bi, bj;
    if (!map_block<MAP>(bm, bi, bj)) return;
    collide_tile<RHO, R, DIM>(c, rad, n, bi, bj, o, threadIdx.x, threadIdx.y);
}

// UTM (Section 4.2): thread k of the (n+1) n / 2 pairs j <= i, one test each,
// operands from global memory; the diagonal threads (j = i) do nothing.
template <int DIM>
__global__ void collide_utm_kernel(const float *__restrict__ c, const float *__restrict__ rad, uint32_t n,
                                   CollideOut o)
{
    const uint64_t N = (uint64_t)n + 1;
    const uint64_t total = N * n / 2;
    const uint64_t k = ((uint64_t)blockIdx.y * gridDim.x + blockIdx.x) * (blockDim.x * blockDim.y) +
                       threadIdx.y * blockDim.x + threadIdx.x;
    if (k >= total) return;
    uint32_t a, b;
    utm_pair(k, N, a, b);
    const uint32_t i = b - 2, j = a - 1;
    if (j >= i) return;
    float pa[DIM + 1], pb[DIM + 1];
#pragma unroll
    for (int t = 0; t < DIM; ++t) {
        pa[t] = c[(uint64_t)i * DIM + t];
        pb[t] = c[(uint64_t)j * DIM + t];
    }
    pa[DIM] = rad[i];
    pb[DIM] = rad[j];
    if (hit_scalar<DIM>(pa, pb)) record(o, i, j);
}

template <int DIM>
int launch_dim(const float *c, const float *rad, uint32_t n, int map, uint32_t rho, uint32_t reg, CollideOut o,
               cudaStream_t s)
{
    if (map == TRI_MAP_UTM) {
        const uint64_t N = (uint64_t)n + 1, total = N * n / 2, tpb = (uint64_t)rho * rho;
        if (total > 0xFFFFFFFFull) return TRI_ERANGE;
        collide_utm_kernel<DIM><<<trihost::linear_grid((total + tpb - 1) / tpb), dim3(rho, rho), 0, s>>>(c, rad,
                                                                                                         n, o);
        return cudaGetLastError() == cudaSuccess ? TRI_OK : TRI_ECUDA;
    }
    const uint32_t S = rho * reg, m = (n + S - 1) / S;
    return trihost::map_launches(map, m, [&](auto tag, dim3 g, const BlockMap &bm) -> cudaError_t {
        constexpr int MAP = decltype(tag)::value;
#define TRI_C(RH, RG)                                                                                          \
    if (rho == RH && reg == RG) {                                                                              \
        collide_kernel<MAP, RH, RG, DIM><<<g, dim3(RH, RH), TileBytes<RH, RG, DIM>::BYTES, s>>>(c, rad, n, o, bm); \
        return cudaGetLastError();                                                                             \
    }
        TRI_C(8, 1) TRI_C(8, 4) TRI_C(8, 8) TRI_C(16, 1) TRI_C(16, 4) TRI_C(16, 8) TRI_C(32, 1) TRI_C(32, 4)
#undef TRI_C
        return cudaErrorInvalidValue;
    });
}

}  // namespace

extern "C" int tri_collide(const float *centres, const float *radii, uint32_t n, uint32_t dim, int map,
                           uint32_t rho, uint32_t reg, uint32_t *count, uint32_t *pairs, uint64_t pair_cap,
                           unsigned long long *n_pairs, void *stream)
{
    if ((n && (!centres || !radii)) || !n_pairs || (!pairs && pair_cap > 0)) return TRI_EINVAL;
    if (dim < 1 || dim > 3 || !trihost::rho_ok(rho)) return TRI_EINVAL;
    // reg = 0, the library's choice: the tensor-core filter for 2-D and 3-D spheres
    // and the maps that place any number of block rows.  Its tiles are larger, so a size it covers
    // is first checked against the packed tile's block rows, which the other
    // maps run at.
    const bool filter = reg == 0 && dim >= 2 && map != TRI_MAP_REC && map != TRI_MAP_UTM;
    if (reg == 0) reg = rho <= 16 ? 8 : 4;
    if ((reg != 1 && reg != 4 && reg != 8) || (reg == 8 && rho > 16)) return TRI_EINVAL;
    if (map < TRI_MAP_LAMBDA || map > TRI_MAP_LAMBDA_PDELTA) return TRI_EINVAL;
    if (n > 0) {  // every range check before the first call that touches the device
        const int st = map == TRI_MAP_UTM
                           ? ((uint64_t)n + 1) * n / 2 <= 0xFFFFFFFFull ? TRI_OK : TRI_ERANGE
                           : trihost::map_range(map, ((uint64_t)n + rho * reg - 1) / (rho * reg));
        if (st != TRI_OK) return st;
    }
    cudaStream_t s = (cudaStream_t)stream;
    collide_zero_kernel<<<(unsigned)((count ? (uint64_t)n : 0) / 256 + 1), 256, 0, s>>>(count, n, n_pairs);
    if (cudaGetLastError() != cudaSuccess) return TRI_ECUDA;
    if (n == 0) return TRI_OK;
    const CollideOut o{count, pairs, pairs ? pair_cap : 0, n_pairs};
    if (filter) {
        switch (dim) {
        case 2: return launch_filter<2>(centres, radii, n, map, o, s);
        default: return launch_filter<3>(centres, radii, n, map, o, s);
        }
    }
    switch (dim) {
    case 1: return launch_dim<1>(centres, radii, n, map, rho, reg, o, s);
    case 2: return launch_dim<2>(centres, radii, n, map, rho, reg, o, s);
    default: return launch_dim<3>(centres, radii, n, map, rho, reg, o, s);
    }
}
