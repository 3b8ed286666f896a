// The library's own tile of the FP32 direct-difference distance map for few
// features (Section 5, test 2, with tri_edm's reg = 0 and d <= 8): the distances
// cost far less than their stores, so the tile is built around the stores.
#pragma once

#include <cuda_runtime.h>

#include "f32x2.cuh"
#include "tri_maps.cuh"

namespace tri {
namespace rows {

constexpr int S = 128;        // tile side: a warp's 32 four-float stores
constexpr int THREADS = 256;  // 8 warps of 16 rows
constexpr int MAX_D = 8;      // the columns' features stay in registers

// One 128 x 128 tile (bi, bj).  Row i of the packed triangle starts at an offset
// T(i) that is a multiple of four floats for one row in four only, so a row's
// tile is shifted left by p = T(i) mod 4 columns (p also counts the output's own
// misalignment): it covers columns j0 - p .. j0 + 127 - p, each lane four of them
// at a 16-byte aligned address.  The shifted tiles of a row still cover it once;
// the diagonal tile adds the p last columns.  T(r) mod 4 depends on r mod 8
// only, and rows a and 7 - a of an octet share it: warp w takes those two rows of
// eight octets (a = w mod 4), keeps its lanes' columns in registers for all of
// them, and per row reads one broadcast record, computes four distances per lane
// two at a time, and stores them with one instruction.
// D: features, padded with zeros (which add exact zeros) to 2, 3, 4 or 8.
// What bounds it: the stores, up to d = 4.  At N = 65536, d = 3 it writes 7.1 TB/s
// (1214 us; a plain fill of the same 8.59 GB takes 1190), against 1995 us for the 4 x
// 4 tile, whose stores are four bytes a lane; d = 8, which issue slots bound, takes
// 1864 against 2788 us.  With one row loop for all tiles, its tests and a 64-bit T(i)
// for every row, d = 3 took 1718 us (issue slots 86% busy) and d = 8 2385 us.
template <int D>
__device__ __forceinline__ void tile(const float *__restrict__ x, uint32_t n, uint32_t d, float *__restrict__ out,
                                     uint32_t bi, uint32_t bj)
{
    constexpr int RF = D <= 4 ? 4 : 8;  // floats of a row's record
    __shared__ __align__(16) float sc[4][D][S];  // the columns as each phase shifts them
    __shared__ __align__(16) float sr[S][RF];    // the rows
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t i0 = (int64_t)bi * S, j0 = (int64_t)bj * S;
    const uint32_t base = (uint32_t)((uintptr_t)out >> 2);  // the output's own phase
    // phase of octet rows a and 7 - a: T(a) = 0, 1, 3, 6 (i0 is a multiple of 8)
    auto phase = [&](int a) { return (int)((base + (uint32_t)(a * (a + 1) / 2)) & 3u); };
    for (int t = tid; t < 4 * S; t += THREADS) {
        const int a = t / S, c = t % S;
        const int64_t j = j0 - phase(a) + c;
        const bool in = j >= 0 && j < (int64_t)n;
        const float *src = x + (size_t)(in ? j : 0) * d;
#pragma unroll
        for (int k = 0; k < D; ++k) sc[a][k][c] = in && k < (int)d ? src[k] : 0.0f;
    }
    if (tid < S) {
        const int64_t i = i0 + tid;
        const bool in = i < (int64_t)n;
        const float *src = x + (size_t)(in ? i : 0) * d;
#pragma unroll
        for (int k = 0; k < D; ++k) sr[tid][k] = in && k < (int)d ? src[k] : 0.0f;
    }
    __syncthreads();
    const int a = warp & 3, p = phase(a);
    const int64_t c0 = j0 - p + 4 * lane;  // this lane's first column
    f2 xc[D][2];
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&sc[a][k][4 * lane]);
        xc[k][0] = v.x;
        xc[k][1] = v.y;
    }
    // the four distances of row r
    auto distances = [&](int r) {
        float xr[RF];
#pragma unroll
        for (int k = 0; k < RF; k += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(&sr[r][k]);
            xr[k] = v.x;
            xr[k + 1] = v.y;
            xr[k + 2] = v.z;
            xr[k + 3] = v.w;
        }
        f2 s0 = 0ull, s1 = 0ull;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const f2 row = f2_pack(xr[k], xr[k]);
            const f2 d0 = f2_sub(row, xc[k][0]), d1 = f2_sub(row, xc[k][1]);
            s0 = f2_fma(d0, d0, s0);
            s1 = f2_fma(d1, d1, s1);
        }
        float4 v;
        f2_unpack(s0, v.x, v.y);
        f2_unpack(s1, v.z, v.w);
        v.x = sqrtf(v.x);
        v.y = sqrtf(v.y);
        v.z = sqrtf(v.z);
        v.w = sqrtf(v.w);
        return v;
    };
    const int r0 = (warp >> 2) * 64;  // this warp's octets
    // Every row of the tile lies in the grid and takes all four columns of every
    // lane: no tests, and each row's address comes from that of the row eight
    // above it, T(i + 8) - T(i) = 8 i + 36.
    if (bj > 0 && bj < bi && i0 + S <= (int64_t)n) {
        uint32_t ia = (uint32_t)i0 + r0 + a, ib = (uint32_t)i0 + r0 + 7 - a;
        float *da = out + T2((uint64_t)ia) + c0, *db = out + T2((uint64_t)ib) + c0;
#pragma unroll 2
        for (int o = 0; o < 64; o += 8) {
            __stcs(reinterpret_cast<float4 *>(da), distances(r0 + o + a));
            __stcs(reinterpret_cast<float4 *>(db), distances(r0 + o + 7 - a));
            da += 8 * (uint64_t)ia + 36;
            db += 8 * (uint64_t)ib + 36;
            ia += 8;
            ib += 8;
        }
        return;
    }
    for (int q = 0; q < 16; ++q) {
        const int r = r0 + (q >> 1) * 8 + ((q & 1) ? 7 - a : a);
        const int64_t i = i0 + r;
        if (i >= (int64_t)n) break;
        const float4 v = distances(r);
        float *dst = out + T2((uint64_t)i) + c0;
        if (c0 >= 0 && c0 + 3 <= i) {
            __stcs(reinterpret_cast<float4 *>(dst), v);
        } else {
            if (c0 >= 0 && c0 <= i) dst[0] = v.x;
            if (c0 + 1 >= 0 && c0 + 1 <= i) dst[1] = v.y;
            if (c0 + 2 >= 0 && c0 + 2 <= i) dst[2] = v.z;
            if (c0 + 3 >= 0 && c0 + 3 <= i) dst[3] = v.w;
        }
        if (bi == bj && r + p >= S && lane < p && j0 + S - p + lane <= i) {
            // the diagonal tile's last columns, shifted out of it (three rows at most)
            const int64_t j = j0 + S - p + lane;
            float s = 0.0f;
            for (uint32_t k = 0; k < d; ++k) {
                const float df = x[(size_t)i * d + k] - x[(size_t)j * d + k];
                s = fmaf(df, df, s);
            }
            out[T2((uint64_t)i) + j] = sqrtf(s);
        }
    }
}

}  // namespace rows
}  // namespace tri
