// Euclidean distance matrix on CUDA cores in FP32 by direct differences
// (Section 5, test 2): one triangle under any block map.  The tile itself is
// in edm_tile.cuh; many uneven triangles in one launch are in edm_batched.cu.
#include <cuda_runtime.h>

#include "edm_rows.cuh"
#include "edm_tile.cuh"
#include "tri_internal.h"

using namespace tri;
using namespace tri::tile;

namespace {

template <int MAP, int RHO, int R, bool PIPE>
__global__ void __launch_bounds__(RHO *RHO) edm_kernel(const float *__restrict__ x, uint32_t n, uint32_t d,
                                                       float *__restrict__ out, BlockMap bm)
{
    uint32_t bi, bj;
    if (!map_block<MAP>(bm, bi, bj)) return;
    edm_tile<RHO, R, PIPE>(x, n, d, out, bi, bj);
}

template <int MAP, int D>
__global__ void __launch_bounds__(rows::THREADS) edm_rows_kernel(const float *__restrict__ x, uint32_t n, uint32_t d,
                                                                 float *__restrict__ out, BlockMap bm)
{
    uint32_t bi, bj;
    if (!map_block<MAP>(bm, bi, bj)) return;
    rows::tile<D>(x, n, d, out, bi, bj);
}

int launch_rows(const float *x, uint32_t n, uint32_t d, float *out, int map, cudaStream_t s)
{
    const uint32_t m = (uint32_t)(((uint64_t)n + rows::S - 1) / rows::S);
    return trihost::map_launches(map, m, [&](auto tag, dim3 g, const BlockMap &bm) -> cudaError_t {
        constexpr int MAP = decltype(tag)::value;
        if constexpr (MAP != MAP_REC) {
            if (d <= 2) edm_rows_kernel<MAP, 2><<<g, rows::THREADS, 0, s>>>(x, n, d, out, bm);
            else if (d == 3) edm_rows_kernel<MAP, 3><<<g, rows::THREADS, 0, s>>>(x, n, d, out, bm);
            else if (d == 4) edm_rows_kernel<MAP, 4><<<g, rows::THREADS, 0, s>>>(x, n, d, out, bm);
            else edm_rows_kernel<MAP, 8><<<g, rows::THREADS, 0, s>>>(x, n, d, out, bm);
            return cudaGetLastError();
        }
        return cudaErrorInvalidValue;
    });
}

// UTM is a thread-space map: one thread per pair, no tile to stage.
__global__ void edm_utm_kernel(const float *__restrict__ x, uint32_t n, uint32_t d, float *__restrict__ out)
{
    const uint64_t N = (uint64_t)n + 1;
    const uint64_t total = N * n / 2;
    const uint64_t k = ((uint64_t)blockIdx.y * gridDim.x + blockIdx.x) * (blockDim.x * blockDim.y) +
                       threadIdx.y * blockDim.x + threadIdx.x;
    if (k >= total) return;
    uint32_t a, b;
    utm_pair(k, N, a, b);
    const uint64_t i = b - 2, j = a - 1;
    const float *xi = x + i * d, *xj = x + j * d;
    float acc = 0.0f;
    for (uint32_t t = 0; t < d; ++t) {
        const float df = xi[t] - xj[t];
        acc = fmaf(df, df, acc);
    }
    out[T2(i) + j] = sqrtf(acc);
}

template <int MAP, int RHO, int R>
cudaError_t launch_one(dim3 g, cudaStream_t s, const float *x, uint32_t n, uint32_t d, float *out, BlockMap bm)
{
    if (d <= (uint32_t)KC) {
        edm_kernel<MAP, RHO, R, false><<<g, dim3(RHO, RHO), TileSmem<RHO, R>::bytes(false), s>>>(x, n, d, out, bm);
        return cudaGetLastError();
    }
    constexpr size_t smem = TileSmem<RHO, R>::bytes(true);
    if (smem > 48 * 1024) {
        const cudaError_t e = trihost::allow_smem(edm_kernel<MAP, RHO, R, true>, smem);
        if (e != cudaSuccess) return e;
    }
    edm_kernel<MAP, RHO, R, true><<<g, dim3(RHO, RHO), smem, s>>>(x, n, d, out, bm);
    return cudaGetLastError();
}

template <int MAP>
cudaError_t launch_rr(uint32_t rho, uint32_t reg, dim3 g, cudaStream_t s, const float *x, uint32_t n, uint32_t d,
                      float *out, BlockMap bm)
{
#define TRI_E(RH, RG)                                                                                          \
    if (rho == RH && reg == RG) return launch_one<MAP, RH, RG>(g, s, x, n, d, out, bm);
    TRI_E(8, 1) TRI_E(8, 2) TRI_E(8, 4) TRI_E(8, 8) TRI_E(16, 1) TRI_E(16, 2) TRI_E(16, 4) TRI_E(16, 8)
    TRI_E(32, 1) TRI_E(32, 2) TRI_E(32, 4)
#undef TRI_E
    return cudaErrorInvalidValue;
}

}  // namespace

int trihost::edm_fp32(const float *x, uint32_t n, uint32_t d, float *out, int map, uint32_t rho, uint32_t reg,
                      cudaStream_t s)
{
    const bool choose = reg == 0;  // the library's choice of the tile
    if (choose) reg = 4;
    // 8 x 8 pairs per thread only with rho <= 16 (registers and shared memory)
    if ((reg != 1 && reg != 2 && reg != 4 && reg != 8) || (reg == 8 && rho > 16)) return TRI_EINVAL;
    if (map == TRI_MAP_UTM) {
        const uint64_t N = (uint64_t)n + 1, total = N * n / 2, tpb = (uint64_t)rho * rho;
        if (total > 0xFFFFFFFFull) return TRI_ERANGE;
        edm_utm_kernel<<<trihost::linear_grid((total + tpb - 1) / tpb), dim3(rho, rho), 0, s>>>(x, n, d, out);
        return cudaGetLastError() == cudaSuccess ? TRI_OK : TRI_ECUDA;
    }
    if (choose && map != TRI_MAP_REC) {
        // a size that the 4 x 4 tile's block rows put out of the map's range stays
        // out of it; REC keeps that tile, whose block rows it needs a power of two of
        const int st = trihost::map_range(map, ((uint64_t)n + 4 * rho - 1) / (4 * rho));
        if (st != TRI_OK) return st;
        // few features: the row tile once there are 800 of its blocks (d <= 4) or 1200,
        // five and eight for each of 152 SMs; 5 to 7 features take the sums of 8
        // (d = 3, us, 4 x 4 pairs a thread / row tile: n = 65536 1995 / 1209, n = 8000 32.5 /
        // 24.9, n = 5000 14.4 / 14.1, n = 4000 10.1 / 10.6, n = 2048 4.7 / 7.8;
        // d = 8: n = 7000 36.9 / 32.9, n = 6000 28.7 / 28.2, n = 5000 20.6 / 22.6; d = 5:
        // n = 6144 / 6145 23.5 / 23.6, and with the staging before that 8000 43.4 / 34.9)
        if (d <= (uint32_t)rows::MAX_D && T2(((uint64_t)n + rows::S - 1) / rows::S) >= (d <= 4 ? 800u : 1200u))
            return launch_rows(x, n, d, out, map, s);
        // more features: 8 x 8 pairs per thread, bound by arithmetic with half the
        // shared-memory reads per pair, once there are 500 of its blocks (4 x 4 / 8 x
        // 8 at rho = 16, us: n = 20011 d = 100 1627 / 1318, d = 32 616 / 488, d = 9 293 /
        // 238; d = 64 n = 4000 49 / 47, n = 2500 24.4 / 26.9)
        const uint64_t m8 = ((uint64_t)n + 8 * rho - 1) / (8 * rho);
        if (rho <= 16 && d > (uint32_t)rows::MAX_D && T2(m8) >= 500) reg = 8;
    }
    const uint32_t S = rho * reg;
    const uint32_t m = (n + S - 1) / S;
    BlockMap bm{};
    bm.m = m;
    bm.nblocks = T2(m);
    cudaError_t e = cudaSuccess;
    switch (map) {
    case TRI_MAP_LAMBDA:
        if (bm.nblocks > 0xFFFFFFFFull) return TRI_ERANGE;
        e = launch_rr<MAP_LAMBDA>(rho, reg, trihost::linear_grid(bm.nblocks), s, x, n, d, out, bm);
        break;
    case TRI_MAP_LAMBDA_PDELTA: {
        if (bm.nblocks > 0xFFFFFFFFull) return TRI_ERANGE;
        const uint64_t mp = trihost::isqrt_ceil(bm.nblocks);
        if (mp > 65535) return TRI_ERANGE;
        e = launch_rr<MAP_LAMBDA_PD>(rho, reg, dim3((unsigned)mp, (unsigned)mp), s, x, n, d, out, bm);
        break;
    }
    case TRI_MAP_BB:
        if (m > 65535) return TRI_ERANGE;
        e = launch_rr<MAP_BB>(rho, reg, dim3(m, m), s, x, n, d, out, bm);
        break;
    case TRI_MAP_RB: {
        const uint32_t h = (m & 1u) ? (m + 1) / 2 : m / 2 + 1;
        if (h > 65535) return TRI_ERANGE;
        e = launch_rr<MAP_RB>(rho, reg, dim3(m, h), s, x, n, d, out, bm);
        break;
    }
    case TRI_MAP_REC: {
        if (!trihost::is_pow2(m)) return TRI_ERANGE;
        const uint32_t k = trihost::ilog2(m);
        if (k > 0 && m / 2 > 65535) return TRI_ERANGE;
        for (uint32_t l = 0; l <= k && e == cudaSuccess; ++l) {
            bm.level = l;
            const dim3 g = l == 0 ? dim3(m) : dim3(1u << (l - 1), m / 2);
            e = launch_rr<MAP_REC>(rho, reg, g, s, x, n, d, out, bm);
        }
        break;
    }
    default:
        return TRI_EINVAL;
    }
    return e == cudaSuccess ? TRI_OK : TRI_ECUDA;
}
