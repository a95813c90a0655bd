// A3 similarity kernels: MSE and NCC over the mask (two-phase, fixed-order
// FP64 reductions) and the LCC local-correlation tile kernel shared with
// the fused objective.
#include "launch.h"
#include "profile.h"

namespace airgb {

namespace {

constexpr int kRedThreads = 256;
// At most 4 blocks per SM of a 152-SM GB300: the count sizes the partials'
// workspace, so it is a constant, not the current device's SM count. A thread
// reads four voxels at a time and sums each of the four apart in fp32, so a
// partial sum has few terms; from there on the sums are Sum2 pairs, so no FP64
// instruction is left but the last ones. (2.4 M voxels, NCC: 17.8, 9.7, 18.5
// and 10.7 us for its four reductions with FP64 trees, 8.6, 13.3 and 7.3 us for
// the three so.)
constexpr int kRedBlocksMax = 152 * 4;

int red_blocks(int64_t nv)
{
    int64_t b = (nv + kRedThreads * 8 - 1) / (kRedThreads * 8);
    return (int)(b < 1 ? 1 : (b > kRedBlocksMax ? kRedBlocksMax : b));
}

// f(k, F, W, on) of every voxel, k the position in a group of four (every
// pointer is 16-byte aligned); the last nv % 4 voxels one by one.
template <class Fn>
__device__ __forceinline__ void each_voxel(int64_t nv, const float *__restrict__ F,
                                           const float *__restrict__ W,
                                           const uint8_t *__restrict__ m, Fn f)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
#pragma unroll 2
    for (int64_t e = t; e < nv / 4; e += stride) {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(F) + e);
        const float4 b = __ldg(reinterpret_cast<const float4 *>(W) + e);
        const uchar4 c = __ldg(reinterpret_cast<const uchar4 *>(m) + e);
        f(0, a.x, b.x, c.x != 0);
        f(1, a.y, b.y, c.y != 0);
        f(2, a.z, b.z, c.z != 0);
        f(3, a.w, b.w, c.w != 0);
    }
    for (int64_t v = nv / 4 * 4 + t; v < nv; v += stride)
        f(0, __ldg(F + v), __ldg(W + v), __ldg(m + v) != 0);
}

// g[v] = f(F, W) on the mask, 0 off it.
template <class Fn>
__device__ __forceinline__ void each_gradient(int64_t nv, const float *__restrict__ F,
                                              const float *__restrict__ W,
                                              const uint8_t *__restrict__ m,
                                              float *__restrict__ g, Fn f)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = t; e < nv / 4; e += stride) {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(F) + e);
        const float4 b = __ldg(reinterpret_cast<const float4 *>(W) + e);
        const uchar4 c = __ldg(reinterpret_cast<const uchar4 *>(m) + e);
        reinterpret_cast<float4 *>(g)[e] =
            make_float4(c.x ? f(a.x, b.x) : 0.0f, c.y ? f(a.y, b.y) : 0.0f,
                        c.z ? f(a.z, b.z) : 0.0f, c.w ? f(a.w, b.w) : 0.0f);
    }
    for (int64_t v = nv / 4 * 4 + t; v < nv; v += stride)
        g[v] = __ldg(m + v) ? f(__ldg(F + v), __ldg(W + v)) : 0.0f;
}

size_t align256(size_t b) { return (b + 255) / 256 * 256; }

__device__ __forceinline__ Sum2 sum4(const float (&v)[4])
{
    Sum2 t;
    t.s = v[0];
    t.add(v[1]);
    t.add(v[2]);
    t.add(v[3]);
    return t;
}

// The block's K sums of four per thread as its row of partials; by FP64 trees
// when a thread's sum is beyond what a Sum2 takes.
template <int K>
__device__ __forceinline__ void store_partials(const float (&v)[K][4], double *part, double *red)
{
    bool far = false;
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            far |= !(fabsf(v[k][i]) <= kSum2Most);
    double t[K];
    if (__syncthreads_or(far)) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            t[k] = ((double)v[k][0] + v[k][1]) + ((double)v[k][2] + v[k][3]);
        block_reduce_d<K>(t, red);
    } else {
        Sum2 s[K];
#pragma unroll
        for (int k = 0; k < K; ++k)
            s[k] = sum4(v[k]);
        block_reduce_s2<K>(s, t, red);
    }
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < K; ++k)
            part[(int64_t)blockIdx.x * K + k] = t[k];
}

// Sums of all blocks' K partials in fixed order, valid in thread 0.
template <int K>
__device__ __forceinline__ void sum_block_partials(const double *__restrict__ part, int nblocks,
                                                   double (&tot)[K], double *red)
{
#pragma unroll
    for (int k = 0; k < K; ++k)
        tot[k] = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
#pragma unroll
        for (int k = 0; k < K; ++k)
            tot[k] += part[(int64_t)b * K + k];
    block_reduce_d<K>(tot, red);
}

// Block sum of K Sum2 that stays a pair (sums that are far from fp32's range);
// valid in warp 0's lane 0.
template <int K>
__device__ __forceinline__ void block_reduce_pairs(Sum2 (&v)[K], float2 *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                Sum2 o;
                o.s = __shfl_down_sync(0xffffffffu, v[k].s, off);
                o.e = __shfl_down_sync(0xffffffffu, v[k].e, off);
                v[k].add(o);
            }
        if (pass == 1)
            return;
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < K; ++k)
                red[k * (kRedThreads / 32) + warp] = make_float2(v[k].s, v[k].e);
        __syncthreads();
        if (warp != 0)
            return;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float2 p = lane < kRedThreads / 32 ? red[k * (kRedThreads / 32) + lane]
                                                     : make_float2(0.0f, 0.0f);
            v[k].s = p.x;
            v[k].e = p.y;
        }
    }
}

// ---------------------------------------------------------------- MSE ------
__global__ void __launch_bounds__(kRedThreads)
    k_mse_partials(int64_t nv, const float *__restrict__ F, const float *__restrict__ W,
                   const uint8_t *__restrict__ m, double *__restrict__ part)
{
    __shared__ double red[2 * kRedThreads / 32];
    float s[2][4] = {};
    each_voxel(nv, F, W, m, [&](int k, float f, float w, bool on) {
        if (on) {
            const float d = w - f;
            s[0][k] = fmaf(d, d, s[0][k]);
            s[1][k] += 1.0f;
        }
    });
    store_partials<2>(s, part, red);
}

__global__ void __launch_bounds__(kRedThreads)
    k_mse_finalize(const double *__restrict__ part, int nblocks, double *__restrict__ value,
                   double *__restrict__ scal)
{
    __shared__ double red[2 * kRedThreads / 32];
    double t[2];
    sum_block_partials<2>(part, nblocks, t, red);
    if (threadIdx.x == 0) {
        const double n = t[1];
        value[0] = n > 0.0 ? t[0] / n : 0.0;
        value[1] = n;
        scal[0] = n > 0.0 ? 2.0 / n : 0.0;
    }
}

__global__ void __launch_bounds__(kRedThreads)
    k_mse_grad(int64_t nv, const float *__restrict__ F, const float *__restrict__ W,
               const uint8_t *__restrict__ m, const double *__restrict__ scal,
               float *__restrict__ g)
{
    const float k = (float)scal[0];
    each_gradient(nv, F, W, m, g, [&](float f, float w) { return k * (w - f); });
}

// ---------------------------------------------------------------- NCC ------
constexpr float kNccScale = 0x1p-20f;
static_assert((int64_t)kRedBlocksMax * kRedThreads * 4 <= 1 << 20, "sums of a pass");

__global__ void __launch_bounds__(kRedThreads)
    k_ncc_sums(int64_t nv, const float *__restrict__ F, const float *__restrict__ W,
               const uint8_t *__restrict__ m, float2 *__restrict__ part)
{
    __shared__ float2 red[3 * kRedThreads / 32];
    float sf[4] = {}, sw[4] = {}, c[4] = {};
    each_voxel(nv, F, W, m, [&](int k, float f, float w, bool on) {
        if (on) {
            sf[k] += f;
            sw[k] += w;
            c[k] += 1.0f;
        }
    });
    // scaled by 2^-20, at least the reciprocal of the threads' sums that are added, so that
    // no sum of sums leaves fp32's range
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        sf[k] *= kNccScale;
        sw[k] *= kNccScale;
        c[k] *= kNccScale;
    }
    Sum2 acc[3] = {sum4(sf), sum4(sw), sum4(c)};
    block_reduce_pairs<3>(acc, red);
    if (threadIdx.x == 0)
        for (int k = 0; k < 3; ++k)
            part[3 * blockIdx.x + k] = make_float2(acc[k].s, acc[k].e);
}

// The central moments about the means of the first pass, whose partials every
// block sums by itself (the same fixed order, so the same means; block 0 keeps
// them): 608 rows from L2 instead of a launch of one block.
__global__ void __launch_bounds__(kRedThreads)
    k_ncc_central(int64_t nv, const float *__restrict__ F, const float *__restrict__ W,
                  const uint8_t *__restrict__ m, const float2 *__restrict__ sums,
                  double *__restrict__ scal, double *__restrict__ part)
{
    __shared__ double red[3 * kRedThreads / 32];
    __shared__ float2 pairs[3 * kRedThreads / 32];
    __shared__ float mu[2];
    Sum2 t[3];
    for (int b = threadIdx.x; b < gridDim.x; b += kRedThreads)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float2 p = __ldg(sums + 3 * b + k);
            Sum2 o;
            o.s = p.x;
            o.e = p.y;
            t[k].add(o);
        }
    block_reduce_pairs<3>(t, pairs);
    if (threadIdx.x == 0) {
        constexpr double up = 1.0 / kNccScale;
        const double n = t[2].value() * up, sf = t[0].value() * up, sw = t[1].value() * up;
        const double mf = n > 0.0 ? sf / n : 0.0, mw = n > 0.0 ? sw / n : 0.0;
        mu[0] = (float)mf;
        mu[1] = (float)mw;
        if (blockIdx.x == 0) {
            scal[0] = mf;
            scal[1] = mw;
            scal[2] = n;
        }
    }
    __syncthreads();
    const float muf = mu[0], muw = mu[1];
    float s[3][4] = {};  // cov, vf, vw
    each_voxel(nv, F, W, m, [&](int k, float f, float w, bool on) {
        if (on) {
            const float a = f - muf, b = w - muw;
            s[0][k] = fmaf(a, b, s[0][k]);
            s[1][k] = fmaf(a, a, s[1][k]);
            s[2][k] = fmaf(b, b, s[2][k]);
        }
    });
    store_partials<3>(s, part, red);
}

// scal: {muF, muW, n} in; writes {.., .., .., kF, kW} with
// dS/dW = kF*(F - muF) + kW*(W - muW) on the mask.
__global__ void __launch_bounds__(kRedThreads)
    k_ncc_finalize(const double *__restrict__ part, int nblocks, double eps,
                   double *__restrict__ scal, double *__restrict__ value)
{
    __shared__ double red[3 * kRedThreads / 32];
    double t[3];
    sum_block_partials<3>(part, nblocks, t, red);
    if (threadIdx.x == 0) {
        const double n = scal[2];
        const double cov = t[0], vf = t[1], vw = t[2];
        const double D = vf * vw + eps;
        if (n > 0.0 && D > 0.0) {
            const double sD = sqrt(D);
            value[0] = 1.0 - cov / sD;
            scal[3] = -1.0 / sD;
            scal[4] = cov * vf / (D * sD);
        } else {
            value[0] = n > 0.0 ? 1.0 : 0.0;
            scal[3] = 0.0;
            scal[4] = 0.0;
        }
        value[1] = n;
    }
}

__global__ void __launch_bounds__(kRedThreads)
    k_ncc_grad(int64_t nv, const float *__restrict__ F, const float *__restrict__ W,
               const uint8_t *__restrict__ m, const double *__restrict__ scal,
               float *__restrict__ g)
{
    const float muf = (float)scal[0], muw = (float)scal[1];
    const float kf = (float)scal[3], kw = (float)scal[4];
    each_gradient(nv, F, W, m, g,
                  [&](float f, float w) { return fmaf(kf, f - muf, kw * (w - muw)); });
}

// The two sums of the LCC kernels' FP64 partials.
__global__ void k_lcc_finalize(const double *__restrict__ part, int nblocks,
                               double *__restrict__ value, double *__restrict__ scal)
{
    __shared__ double red[2 * 32];
    double t[2] = {0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
        t[0] += part[2 * (int64_t)b];
        t[1] += part[2 * (int64_t)b + 1];
    }
    block_reduce_d<2>(t, red);
    if (threadIdx.x == 0) {
        const double n = t[1];
        value[0] = n > 0.0 ? 1.0 - t[0] / n : 0.0;
        value[1] = n;
        scal[0] = n > 0.0 ? 1.0 / n : 0.0;
    }
}

__global__ void k_scale(int64_t nv, const double *__restrict__ scal, float *__restrict__ g)
{
    const float k = (float)scal[0];
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv;
         v += (int64_t)gridDim.x * blockDim.x)
        g[v] *= k;
}

}  // namespace

size_t similarity_ws(const Grid &g, int kind, int window)
{
    const size_t scal = 256;
    if (kind == 2)
        return scal + align256((size_t)lcc_max_blocks(g, window) * 2 * sizeof(double)) +
               lcc_coef_bytes(g);
    return scal + 2 * align256((size_t)red_blocks(g.nv) * 3 * sizeof(double));
}

cudaError_t launch_similarity_scalars(const Grid &g, int kind, int window, double eps,
                                      const float *F, const float *W, const uint8_t *m,
                                      bool w_masked, double *value, float *grad, void *ws,
                                      int *gw, cudaStream_t s)
{
    double *scal = (double *)ws;
    double *part = (double *)((char *)ws + 256);
    const int nb = red_blocks(g.nv);
    const int th = kRedThreads;
    if (kind == 0) {
        *gw = GW_MSE;
        k_mse_partials<<<nb, th, 0, s>>>(g.nv, F, W, m, part);
        k_mse_finalize<<<1, th, 0, s>>>(part, nb, value, scal);
    } else if (kind == 1) {
        *gw = GW_NCC;
        double *part2 = (double *)((char *)part + align256((size_t)nb * 3 * sizeof(double)));
        k_ncc_sums<<<nb, th, 0, s>>>(g.nv, F, W, m, (float2 *)part);
        k_ncc_central<<<nb, th, 0, s>>>(g.nv, F, W, m, (const float2 *)part, scal, part2);
        k_ncc_finalize<<<1, th, 0, s>>>(part2, nb, eps, scal, value);
    } else {
        *gw = GW_SCALED;
        const int lb = lcc_num_blocks(g, window);
        float *coef = (float *)((char *)part +
                                align256((size_t)lcc_max_blocks(g, window) * 2 * sizeof(double)));
        cudaError_t e = launch_lcc(g, window, eps, F, W, m, w_masked, grad, part, coef, s);
        if (e != cudaSuccess)
            return e;
        k_lcc_finalize<<<1, 1024, 0, s>>>(part, lb, value, scal);
    }
    return cudaGetLastError();
}

cudaError_t launch_similarity(const Grid &g, int kind, int window, double eps, const float *F,
                              const float *W, const uint8_t *m, double *value, float *grad,
                              void *ws, cudaStream_t s)
{
    int gw = GW_NONE;
    const cudaError_t e =
        launch_similarity_scalars(g, kind, window, eps, F, W, m, false, value, grad, ws, &gw, s);
    if (e != cudaSuccess || !grad)
        return e;
    const double *scal = (const double *)ws;
    const int64_t nb4 = (g.nv + 4 * kRedThreads - 1) / (4 * (int64_t)kRedThreads);
    const int nb = (int)(nb4 < 8 * device_sms() ? nb4 : 8 * device_sms());
    if (kind == 0)
        k_mse_grad<<<nb, kRedThreads, 0, s>>>(g.nv, F, W, m, scal, grad);
    else if (kind == 1)
        k_ncc_grad<<<nb, kRedThreads, 0, s>>>(g.nv, F, W, m, scal, grad);
    else
        k_scale<<<nb, kRedThreads, 0, s>>>(g.nv, scal, grad);
    return cudaGetLastError();
}

}  // namespace airgb
