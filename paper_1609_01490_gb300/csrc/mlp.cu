// Training and inference kernels of the MLP cost model that picks a map and
// block size (not part of the paper): y = W3 relu(W2 relu(W1 x + b1) + b2) + b3,
// mean-squared-error loss, Adam (Kingma and Ba, 2015).  Every reduction runs
// in a fixed order, so results do not depend on scheduling.
#include <cuda_runtime.h>

#include "../../include/tri.h"
#include "pdl.cuh"
#include "tri_internal.h"

namespace {

// theta: W1 [H1][F], b1 [H1], W2 [H2][H1], b2 [H2], W3 [H2], b3 [1]
struct Layout {
    const float *W1, *b1, *W2, *b2, *W3, *b3;
};

// The batch's intermediate values: z1 [B][H1], z2 [B][H2] (before the relu), pred
// [B] and the loss gradients with respect to pred, z2 and z1.
struct Batch {
    float *z1, *z2, *pred, *g_out, *g_z2, *g_z1;
};

constexpr int MLP_THREADS = 256;
constexpr uint32_t GROUP = 4, MAX_GROUP = 32;  // samples a block takes at a time

// Floats of shared memory of mlp_pass_kernel: the weights (rows padded by one
// word, so that neither a row per thread nor a column per thread conflicts) and a
// group's activations and gradients.
__host__ __device__ constexpr uint32_t pass_floats(uint32_t F, uint32_t H1, uint32_t H2, uint32_t group)
{
    return H1 * (F + 1) + H1 + H2 * (H1 + 1) + 2 * H2 + 1 + group * (F + H1 + 2 * H2 + 1);
}

// The most shapes_ok lets it take: larger groups belong to narrower layers.
constexpr size_t PASS_SMEM = pass_floats(64, 128, 128, GROUP) * sizeof(float);
static_assert(pass_floats(64, 128, 1, GROUP) * sizeof(float) <= PASS_SMEM &&
                  pass_floats(64, 64, 64, MAX_GROUP) * sizeof(float) <= PASS_SMEM,
              "a larger group only where the wider layer has at most 64 outputs");

// Forward pass and, with BACK, the gradients of the mean squared loss down to z1,
// in one launch: a block keeps the weights in shared memory and takes the samples
// `group` at a time through all the layers.  The passes are bound by latency (the
// whole batch of the selector's sweep is 2 Mflop): as ten dependent launches a
// training step took 113 us at B = 391, H1 = H2 = 64, as three it takes 19.  Each sum runs over
// its inputs in increasing order.
template <bool BACK>
__global__ void __launch_bounds__(MLP_THREADS)
    mlp_pass_kernel(const Layout L, const float *__restrict__ X, const float *__restrict__ y, uint32_t B, uint32_t F,
                    uint32_t H1, uint32_t H2, uint32_t group, float *__restrict__ pred, const Batch w)
{
    extern __shared__ float sm[];
    tri::dependents_may_start();
    float *W1 = sm, *b1 = W1 + H1 * (F + 1), *W2 = b1 + H1, *b2 = W2 + H2 * (H1 + 1), *W3 = b2 + H2, *b3 = W3 + H2;
    float *x = b3 + 1, *z1 = x + group * F, *z2 = z1 + group * H1, *gz2 = z2 + group * H2, *gout = gz2 + group * H2;
    const uint32_t tid = threadIdx.x;
    for (uint32_t t = tid; t < H1 * F; t += MLP_THREADS) W1[t / F * (F + 1) + t % F] = L.W1[t];
    for (uint32_t t = tid; t < H2 * H1; t += MLP_THREADS) W2[t / H1 * (H1 + 1) + t % H1] = L.W2[t];
    for (uint32_t t = tid; t < H1; t += MLP_THREADS) b1[t] = L.b1[t];
    for (uint32_t t = tid; t < H2; t += MLP_THREADS) {
        b2[t] = L.b2[t];
        W3[t] = L.W3[t];
    }
    if (tid == 0) *b3 = *L.b3;
    for (uint64_t s0 = (uint64_t)blockIdx.x * group; s0 < B; s0 += (uint64_t)gridDim.x * group) {
        const uint32_t m = (uint32_t)(B - s0 < group ? B - s0 : group);
        for (uint32_t t = tid; t < m * F; t += MLP_THREADS) x[t] = X[s0 * F + t];
        __syncthreads();
        for (uint32_t t = tid; t < m * H1; t += MLP_THREADS) {
            const uint32_t b = t / H1, o = t - b * H1;
            float s = b1[o];
            for (uint32_t i = 0; i < F; ++i) s = fmaf(W1[o * (F + 1) + i], x[b * F + i], s);
            z1[t] = s;
            if (BACK) w.z1[s0 * H1 + t] = s;
        }
        __syncthreads();
        for (uint32_t t = tid; t < m * H2; t += MLP_THREADS) {
            const uint32_t b = t / H2, o = t - b * H2;
            float s = b2[o];
#pragma unroll 8
            for (uint32_t i = 0; i < H1; ++i) s = fmaf(W2[o * (H1 + 1) + i], fmaxf(z1[b * H1 + i], 0.0f), s);
            z2[t] = s;
            if (BACK) w.z2[s0 * H2 + t] = s;
        }
        __syncthreads();
        if (tid < m) {
            float s = *b3;
#pragma unroll 8
            for (uint32_t i = 0; i < H2; ++i) s = fmaf(W3[i], fmaxf(z2[tid * H2 + i], 0.0f), s);
            pred[s0 + tid] = s;
            if (BACK) w.g_out[s0 + tid] = gout[tid] = 2.0f * (s - y[s0 + tid]) / (float)B;
        }
        if constexpr (BACK) {
            __syncthreads();
            for (uint32_t t = tid; t < m * H2; t += MLP_THREADS) {
                const uint32_t b = t / H2, o = t - b * H2;
                w.g_z2[s0 * H2 + t] = gz2[t] = z2[t] > 0.0f ? gout[b] * W3[o] : 0.0f;
            }
            __syncthreads();
            for (uint32_t t = tid; t < m * H1; t += MLP_THREADS) {
                const uint32_t b = t / H1, i = t - b * H1;
                float s = 0.0f;
#pragma unroll 8
                for (uint32_t o = 0; o < H2; ++o) s = fmaf(gz2[b * H2 + o], W2[o * (H1 + 1) + i], s);
                w.g_z1[s0 * H1 + t] = z1[t] > 0.0f ? s : 0.0f;
            }
        }
        __syncthreads();  // the group's buffers are refilled
    }
}

// Weight and bias gradients of all three layers and the loss, one launch: gW[o][i]
// = sum_b g[b][o] a[b][i] as 16 x 16 tiles of outputs (the bias is the input i = I
// that is always 1), the batch in chunks of 128 staged in shared memory.  64
// threads hold 2 x 2 outputs each, four of them share a tile's samples (sample b of
// a chunk goes to part b / 32), and the parts are added in order, so a result does
// not depend on scheduling.  One thread per output walking the batch alone took
// 16 us a layer at B = 391.
constexpr int TILE = 16, CHUNK = 128, PARTS = 4;

struct GradLayer {
    const float *g, *a;  // [B][O], [B][I]
    float *gW, *gb;
    uint32_t O, I, relu, tiles;  // tiles: ceil(O / 16) ceil((I + 1) / 16)
};

struct GradArgs {
    GradLayer layer[3];
    const float *pred, *y;
    float *loss;
    uint32_t B;
};

__global__ void __launch_bounds__(MLP_THREADS) mlp_wgrad_kernel(const GradArgs ga)
{
    __shared__ float sg[CHUNK][TILE + 1], sa[CHUNK][TILE + 1];
    const uint32_t tid = threadIdx.x;
    uint32_t tile = blockIdx.x, l = 0;
    while (l < 3 && tile >= ga.layer[l].tiles) tile -= ga.layer[l++].tiles;
    tri::wait_for_previous();
    if (l == 3) {  // the last block: loss = mean (pred - y)^2
        float *part = &sg[0][0];
        float s = 0.0f;
        for (uint32_t b = tid; b < ga.B; b += MLP_THREADS) {
            const float r = ga.pred[b] - ga.y[b];
            s = fmaf(r, r, s);
        }
        part[tid] = s;
        __syncthreads();
        for (uint32_t w = MLP_THREADS / 2; w > 0; w >>= 1) {
            if (tid < w) part[tid] += part[tid + w];
            __syncthreads();
        }
        if (tid == 0) *ga.loss = part[0] / (float)ga.B;
        return;
    }
    const GradLayer &L = ga.layer[l];
    const uint32_t across = (L.I + 1 + TILE - 1) / TILE, o0 = tile / across * TILE, i0 = tile % across * TILE;
    const uint32_t part = tid >> 6, to = (tid >> 3 & 7) * 2, ti = (tid & 7) * 2;
    const uint32_t col = tid & 15, row = tid >> 4;  // staging: 16 rows of 16 columns a sweep
    const bool has_g = o0 + col < L.O, has_a = i0 + col < L.I;
    const float one = i0 + col == L.I ? 1.0f : 0.0f;
    float c00 = 0.0f, c01 = 0.0f, c10 = 0.0f, c11 = 0.0f;
    for (uint32_t b0 = 0; b0 < ga.B; b0 += CHUNK) {
        float vg[CHUNK / 16], va[CHUNK / 16];
#pragma unroll
        for (uint32_t q = 0; q < CHUNK / 16; ++q) {
            const uint32_t b = b0 + q * 16 + row;
            const bool in = b < ga.B;
            vg[q] = in && has_g ? L.g[(size_t)b * L.O + o0 + col] : 0.0f;
            va[q] = in ? (has_a ? L.a[(size_t)b * L.I + i0 + col] : one) : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (uint32_t q = 0; q < CHUNK / 16; ++q) {
            sg[q * 16 + row][col] = vg[q];
            sa[q * 16 + row][col] = L.relu ? fmaxf(va[q], 0.0f) : va[q];
        }
        __syncthreads();
#pragma unroll 8
        for (uint32_t q = 0; q < CHUNK / PARTS; ++q) {
            const uint32_t b = part * (CHUNK / PARTS) + q;
            const float g0 = sg[b][to], g1 = sg[b][to + 1], a0 = sa[b][ti], a1 = sa[b][ti + 1];
            c00 = fmaf(g0, a0, c00);
            c01 = fmaf(g0, a1, c01);
            c10 = fmaf(g1, a0, c10);
            c11 = fmaf(g1, a1, c11);
        }
    }
    __syncthreads();
    float *sum = &sg[0][0];  // [part][16][16]
    sum[part * 256 + to * 16 + ti] = c00;
    sum[part * 256 + to * 16 + ti + 1] = c01;
    sum[part * 256 + (to + 1) * 16 + ti] = c10;
    sum[part * 256 + (to + 1) * 16 + ti + 1] = c11;
    __syncthreads();
    const float v = (sum[tid] + sum[256 + tid]) + (sum[512 + tid] + sum[768 + tid]);
    const uint32_t o = o0 + (tid >> 4), i = i0 + (tid & 15);
    if (o < L.O) {
        if (i < L.I) L.gW[(size_t)o * L.I + i] = v;
        else if (i == L.I) L.gb[o] = v;
    }
}

__global__ void adam_kernel(float *__restrict__ theta, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, uint32_t np, float lr, float b1, float b2, float eps, float c1,
                            float c2)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= np) return;
    const float gt = g[t];
    const float mt = b1 * m[t] + (1.0f - b1) * gt;
    const float vt = b2 * v[t] + (1.0f - b2) * gt * gt;
    m[t] = mt;
    v[t] = vt;
    theta[t] -= lr * (mt / c1) / (sqrtf(vt / c2) + eps);
}

__global__ void argmin_kernel(const float *__restrict__ pred, uint32_t B, uint32_t *__restrict__ best)
{
    __shared__ float bv[256];
    __shared__ uint32_t bi[256];
    float v = __int_as_float(0x7f800000);
    uint32_t k = 0xFFFFFFFFu;
    for (uint32_t b = threadIdx.x; b < B; b += blockDim.x)
        if (pred[b] < v) {
            v = pred[b];
            k = b;
        }
    bv[threadIdx.x] = v;
    bi[threadIdx.x] = k;
    __syncthreads();
    for (uint32_t w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            const float ov = bv[threadIdx.x + w];
            const uint32_t ok = bi[threadIdx.x + w];
            if (ov < bv[threadIdx.x] || (ov == bv[threadIdx.x] && ok < bi[threadIdx.x])) {
                bv[threadIdx.x] = ov;
                bi[threadIdx.x] = ok;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *best = bi[0] == 0xFFFFFFFFu ? 0 : bi[0];
}

inline unsigned nblk(size_t work) { return (unsigned)((work + 255) / 256); }

Layout layout(const float *theta, uint32_t F, uint32_t H1, uint32_t H2)
{
    Layout L;
    L.W1 = theta;
    L.b1 = L.W1 + (size_t)H1 * F;
    L.W2 = L.b1 + H1;
    L.b2 = L.W2 + (size_t)H2 * H1;
    L.W3 = L.b2 + H2;
    L.b3 = L.W3 + H2;
    return L;
}

bool shapes_ok(uint32_t B, uint32_t F, uint32_t H1, uint32_t H2)
{
    return B > 0 && F > 0 && F <= 64 && H1 > 0 && H1 <= 128 && H2 > 0 && H2 <= 128;
}

// workspace: z1 [B][H1], z2 [B][H2], pred [B], g_out [B], g_z2 [B][H2], g_z1 [B][H1]
size_t ws_floats(uint32_t B, uint32_t H1, uint32_t H2) { return (size_t)B * (2 * H1 + 2 * H2 + 2); }

Batch batch(float *ws, uint32_t B, uint32_t H1, uint32_t H2)
{
    Batch w;
    w.z1 = ws;
    w.z2 = w.z1 + (size_t)B * H1;
    w.pred = w.z2 + (size_t)B * H2;
    w.g_out = w.pred + B;
    w.g_z2 = w.g_out + B;
    w.g_z1 = w.g_z2 + (size_t)B * H2;
    return w;
}

template <bool BACK>
int pass(const float *theta, const float *X, const float *y, uint32_t B, uint32_t F, uint32_t H1, uint32_t H2,
         float *pred, const Batch &w, cudaStream_t s)
{
    // four samples a block until 1024 blocks read the weights; then as many as keep
    // the threads busy in the wider layer (B = 200,000, F = 3, H1 = 8, H2 = 5, forward:
    // 56 us in fours, 14 so)
    const uint32_t wide = MLP_THREADS / (H1 > H2 ? H1 : H2), per = (uint32_t)(((uint64_t)B + 1023) / 1024);
    uint32_t group = wide < per ? wide : per;
    group = group < GROUP ? GROUP : group > MAX_GROUP ? MAX_GROUP : group;
    const size_t smem = pass_floats(F, H1, H2, group) * sizeof(float);
    if (smem > 48 * 1024 && trihost::allow_smem(mlp_pass_kernel<BACK>, PASS_SMEM) != cudaSuccess) return TRI_ECUDA;
    const uint32_t groups = (uint32_t)(((uint64_t)B + group - 1) / group);
    mlp_pass_kernel<BACK><<<groups < 1024u ? groups : 1024u, MLP_THREADS, smem, s>>>(layout(theta, F, H1, H2), X, y, B, F,
                                                                                 H1, H2, group, pred, w);
    return cudaGetLastError() == cudaSuccess ? TRI_OK : TRI_ECUDA;
}

}  // namespace

extern "C" int tri_mlp_workspace_size(uint32_t B, uint32_t H1, uint32_t H2, size_t *bytes)
{
    if (!bytes) return TRI_EINVAL;
    *bytes = ws_floats(B, H1, H2) * sizeof(float);
    return TRI_OK;
}

extern "C" int tri_mlp_forward(const float *theta, const float *X, uint32_t B, uint32_t F, uint32_t H1, uint32_t H2,
                               float *pred, void *workspace, size_t ws_bytes, void *stream)
{
    if (!theta || !X || !pred || !workspace || !shapes_ok(B, F, H1, H2)) return TRI_EINVAL;
    if (ws_bytes < ws_floats(B, H1, H2) * sizeof(float)) return TRI_ENOSPACE;
    return pass<false>(theta, X, nullptr, B, F, H1, H2, pred, Batch{}, (cudaStream_t)stream);
}

extern "C" int tri_mlp_grad(const float *theta, const float *X, const float *y, uint32_t B, uint32_t F, uint32_t H1,
                            uint32_t H2, float *loss, float *grad, void *workspace, size_t ws_bytes, void *stream)
{
    if (!theta || !X || !y || !loss || !grad || !workspace || !shapes_ok(B, F, H1, H2)) return TRI_EINVAL;
    if (ws_bytes < ws_floats(B, H1, H2) * sizeof(float)) return TRI_ENOSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    const Batch w = batch((float *)workspace, B, H1, H2);
    const int st = pass<true>(theta, X, y, B, F, H1, H2, w.pred, w, s);
    if (st != TRI_OK) return st;
    float *gW1 = grad, *gb1 = gW1 + (size_t)H1 * F, *gW2 = gb1 + H1, *gb2 = gW2 + (size_t)H2 * H1;
    float *gW3 = gb2 + H2, *gb3 = gW3 + H2;
    const auto tiles = [](uint32_t O, uint32_t I) { return ((O + TILE - 1) / TILE) * ((I + 1 + TILE - 1) / TILE); };
    GradArgs ga{{{w.g_z2, w.z1, gW2, gb2, H2, H1, 1u, tiles(H2, H1)},
                 {w.g_z1, X, gW1, gb1, H1, F, 0u, tiles(H1, F)},
                 {w.g_out, w.z2, gW3, gb3, 1u, H2, 1u, tiles(1u, H2)}},
                w.pred, y, loss, B};
    const uint32_t blocks = ga.layer[0].tiles + ga.layer[1].tiles + ga.layer[2].tiles + 1;
    return trihost::launch_behind(mlp_wgrad_kernel, blocks, MLP_THREADS, 0, s, ga) == cudaSuccess ? TRI_OK : TRI_ECUDA;
}

extern "C" int tri_mlp_adam(float *theta, const float *grad, float *m, float *v, uint32_t nparams, uint32_t t,
                            float lr, float beta1, float beta2, float eps, void *stream)
{
    if (!theta || !grad || !m || !v || nparams == 0 || t == 0) return TRI_EINVAL;
    const float c1 = 1.0f - powf(beta1, (float)t), c2 = 1.0f - powf(beta2, (float)t);
    adam_kernel<<<nblk(nparams), 256, 0, (cudaStream_t)stream>>>(theta, grad, m, v, nparams, lr, beta1, beta2, eps,
                                                                  c1, c2);
    return cudaGetLastError() == cudaSuccess ? TRI_OK : TRI_ECUDA;
}

extern "C" int tri_mlp_argmin(const float *theta, const float *X, uint32_t B, uint32_t F, uint32_t H1, uint32_t H2,
                              uint32_t *best, void *workspace, size_t ws_bytes, void *stream)
{
    if (!theta || !X || !best || !workspace || !shapes_ok(B, F, H1, H2)) return TRI_EINVAL;
    if (ws_bytes < ws_floats(B, H1, H2) * sizeof(float)) return TRI_ENOSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    float *ws = (float *)workspace;
    float *pred = ws + (size_t)B * (H1 + H2);
    const int st = pass<false>(theta, X, nullptr, B, F, H1, H2, pred, Batch{}, s);
    if (st != TRI_OK) return st;
    argmin_kernel<<<1, 256, 0, s>>>(pred, B, best);
    return cudaGetLastError() == cudaSuccess ? TRI_OK : TRI_ECUDA;
}
