// Learned initialisation: the light kernels around the convolution layers.
//
//  * k_net_input     F, M (fp32 volumes) -> the 2-channel bf16 input x
//  * k_upcat         [up(e4), e3]: nearest 2x up-sampling of the coarsest
//                    level, cropped to e3's grid, concatenated before e3
//  * k_upcat_adjoint its transpose for the up-sampled channels, times the
//                    ReLU factor of e4
//  * k_head_to_ctrl  the head's output voxel j - 1 (clamped) gives control
//                    point j of the spacing-8 lattice (point j sits at voxel
//                    8 (j - 1), where output voxel j - 1 of the head sits)
//  * k_head_adjoint  its transpose, a gather over the points each voxel feeds
//  * k_field_loss    L = (1/(3|X| nb)) sum_b sum_i e_i^T (G_z x G_y x G_x) e_i,
//                    e = c - c*, and dL/dc = (2/(3|X| nb)) (G x G x G) e.
//                    G = B^T B is the Gram matrix of the sampled 1D cubic
//                    B-spline basis (Sec. III-C), banded with 7 diagonals,
//                    so the loss is exactly the mean squared difference of
//                    the two displacement fields, computed on the lattice.
//  * k_adam_flat     Adam (Sec. III-G) on a flat fp32 parameter array
//  * k_render_blobs  training volumes: sums of isotropic Gaussian blobs (per-axis
//                    factors, terms beyond 6 sigma dropped: synthetic data)
//
// All are memory- or latency-bound elementwise/gather kernels sized to the
// data; none needs scratch beyond what its caller passes.
#include <cuda_bf16.h>
#include <stdint.h>

#include "launch.h"
#include "profile.h"

namespace airgb {

namespace {

constexpr int kT = 256;

int blocks(int64_t n)
{
    int64_t b = (n + kT - 1) / kT;
    if (b > 64 * (int64_t)device_sms())  // grid-stride loops beyond this
        b = 64 * (int64_t)device_sms();
    return (int)(b < 1 ? 1 : b);
}

__global__ void k_net_input(const float *__restrict__ F, const float *__restrict__ M, int64_t n,
                            __nv_bfloat162 *__restrict__ x)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        x[i] = __floats2bfloat162_rn(__ldg(F + i), __ldg(M + i));
}

// One thread per 8-channel group of an output voxel of cat.
__global__ void k_upcat(NetGrid g, int c4, int c3, const uint4 *__restrict__ e4,
                        const uint4 *__restrict__ e3, uint4 *__restrict__ cat)
{
    const int g4 = c4 / 8, g3 = c3 / 8, gc = g4 + g3;
    const int64_t total = (int64_t)g.nb * g.n3[0] * g.n3[1] * g.n3[2] * gc;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int q = (int)(i % gc);
        int64_t v = i / gc;  // voxel of e3's grid
        if (q >= g4) {
            cat[i] = __ldg(e3 + v * g3 + (q - g4));
            continue;
        }
        const int x = (int)(v % g.n3[2]);
        v /= g.n3[2];
        const int y = (int)(v % g.n3[1]);
        v /= g.n3[1];
        const int z = (int)(v % g.n3[0]);
        const int b = (int)(v / g.n3[0]);
        const int64_t src = (((int64_t)b * g.n4[0] + z / 2) * g.n4[1] + y / 2) * g.n4[2] + x / 2;
        cat[i] = __ldg(e4 + src * g4 + q);
    }
}

// g_e4[v][c] = (e4[v][c] > 0) * sum over the up to 8 fine voxels copied
// from v of g_cat[fine][c], c < c4, summed in a fixed order.
__global__ void k_upcat_adjoint(NetGrid g, int c4, int c3, const __nv_bfloat16 *__restrict__ gcat,
                                const __nv_bfloat16 *__restrict__ e4,
                                __nv_bfloat16 *__restrict__ ge4)
{
    const int cc = c4 + c3;
    const int64_t total = (int64_t)g.nb * g.n4[0] * g.n4[1] * g.n4[2] * c4;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % c4);
        int64_t v = i / c4;
        const int x = (int)(v % g.n4[2]);
        v /= g.n4[2];
        const int y = (int)(v % g.n4[1]);
        v /= g.n4[1];
        const int z = (int)(v % g.n4[0]);
        const int b = (int)(v / g.n4[0]);
        float acc = 0.0f;
        for (int dz = 0; dz < 2; ++dz) {
            const int fz = 2 * z + dz;
            if (fz >= g.n3[0])
                continue;
            for (int dy = 0; dy < 2; ++dy) {
                const int fy = 2 * y + dy;
                if (fy >= g.n3[1])
                    continue;
                for (int dx = 0; dx < 2; ++dx) {
                    const int fx = 2 * x + dx;
                    if (fx >= g.n3[2])
                        continue;
                    const int64_t f = (((int64_t)b * g.n3[0] + fz) * g.n3[1] + fy) * g.n3[2] + fx;
                    acc += __bfloat162float(gcat[f * cc + c]);
                }
            }
        }
        ge4[i] = __float2bfloat16_rn(__bfloat162float(e4[i]) > 0.0f ? acc : 0.0f);
    }
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__global__ void k_head_to_ctrl(NetGrid g, int ch, const float *__restrict__ h,
                               float *__restrict__ c)
{
    const int nx = g.lat[0], ny = g.lat[1], nz = g.lat[2];
    const int64_t per = (int64_t)nx * ny * nz;
    const int64_t total = (int64_t)g.nb * 3 * per;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = i;
        const int jx = (int)(r % nx);
        r /= nx;
        const int jy = (int)(r % ny);
        r /= ny;
        const int jz = (int)(r % nz);
        r /= nz;
        const int comp = (int)(r % 3);
        const int b = (int)(r / 3);
        const int hx = clampi(jx - 1, 0, g.n3[2] - 1), hy = clampi(jy - 1, 0, g.n3[1] - 1),
                  hz = clampi(jz - 1, 0, g.n3[0] - 1);
        const int64_t v = (((int64_t)b * g.n3[0] + hz) * g.n3[1] + hy) * g.n3[2] + hx;
        c[i] = h[v * ch + comp];
    }
}

// Lattice indices j whose clamp(j - 1) is output voxel o along one axis of
// n3 outputs and n lattice points: [lo, hi].
__device__ __forceinline__ void feeds(int o, int n3, int n, int &lo, int &hi)
{
    lo = o == 0 ? 0 : o + 1;
    hi = o == n3 - 1 ? n - 1 : o + 1;
}

__global__ void k_head_adjoint(NetGrid g, int ch, const float *__restrict__ gc,
                               __nv_bfloat16 *__restrict__ gh)
{
    const int nx = g.lat[0], ny = g.lat[1], nz = g.lat[2];
    const int64_t total = (int64_t)g.nb * g.n3[0] * g.n3[1] * g.n3[2] * ch;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int comp = (int)(i % ch);
        int64_t v = i / ch;
        float acc = 0.0f;
        if (comp < 3) {
            const int x = (int)(v % g.n3[2]);
            v /= g.n3[2];
            const int y = (int)(v % g.n3[1]);
            v /= g.n3[1];
            const int z = (int)(v % g.n3[0]);
            const int b = (int)(v / g.n3[0]);
            int zl, zh, yl, yh, xl, xh;
            feeds(z, g.n3[0], nz, zl, zh);
            feeds(y, g.n3[1], ny, yl, yh);
            feeds(x, g.n3[2], nx, xl, xh);
            const float *base = gc + ((int64_t)b * 3 + comp) * nx * ny * nz;
            for (int jz = zl; jz <= zh; ++jz)
                for (int jy = yl; jy <= yh; ++jy)
                    for (int jx = xl; jx <= xh; ++jx)
                        acc += base[((int64_t)jz * ny + jy) * nx + jx];
        }
        gh[i] = __float2bfloat16_rn(acc);
    }
}

// Cubic B-spline kernel k_B1D (Sec. III-C) at r (in units of the spacing).
__device__ __forceinline__ float kb3(float r)
{
    const float a = fabsf(r);
    if (a < 1.0f)
        return 2.0f / 3.0f - a * a + 0.5f * a * a * a;
    if (a < 2.0f) {
        const float t = 2.0f - a;
        return t * t * t * (1.0f / 6.0f);
    }
    return 0.0f;
}

// One block per (pair, component). Shared: the three banded Gram matrices
// (n x 7 each; fp32 sums of at most 4 delta terms), two float planes of the
// lattice, reduction scratch. With one block per SM at most (a batch of 16
// has 48 blocks), 1024 threads give each SM enough warps to cover the
// shared-memory latency of the three banded passes.
constexpr int kFieldT = 1024;

__global__ void __launch_bounds__(kFieldT) k_field_loss(FieldLossArgs a, const float *__restrict__ c,
                                                   const float *__restrict__ ct,
                                                   float *__restrict__ gc, double *__restrict__ part)
{
    extern __shared__ double fsm[];
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    const int np = nx * ny * nz;
    double *red = fsm;  // kFieldT doubles
    float *Gs = reinterpret_cast<float *>(fsm + kFieldT);
    float *G[3] = {Gs, Gs + 7 * nx, Gs + 7 * (nx + ny)};
    float *b0 = Gs + 7 * (nx + ny + nz);
    float *b1 = b0 + np;
    const int nn[3] = {nx, ny, nz};
    // Gram entries G[j][d + 3] = sum_x k((x - 8 (j-1))/8) k((x - 8 (j+d-1))/8).
    for (int e = threadIdx.x; e < 7 * (nx + ny + nz); e += blockDim.x) {
        int ax = 0, r = e;
        while (r >= 7 * nn[ax]) {
            r -= 7 * nn[ax];
            ++ax;
        }
        const int j = r / 7, d = r % 7 - 3, j2 = j + d;
        float acc = 0.0f;
        if (j2 >= 0 && j2 < nn[ax]) {
            const int D = a.delta, N = a.N[ax];
            const float inv = 1.0f / (float)D;
            const int p1 = D * (j - 1), p2 = D * (j2 - 1);
            const int lo = max(0, max(p1, p2) - 2 * D), hi = min(N - 1, min(p1, p2) + 2 * D);
            for (int x = lo; x <= hi; ++x)
                acc += kb3((float)(x - p1) * inv) * kb3((float)(x - p2) * inv);
        }
        G[ax][r] = acc;
    }
    const int64_t off = (int64_t)blockIdx.x * np;
    for (int p = threadIdx.x; p < np; p += blockDim.x)
        b0[p] = c[off + p] - ct[off + p];
    __syncthreads();
    // x pass: b1 = (I x I x G_x) b0
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
        const int x = p % nx;
        float acc = 0.0f;
        for (int d = -3; d <= 3; ++d)
            if (x + d >= 0 && x + d < nx)
                acc += G[0][x * 7 + d + 3] * b0[p + d];
        b1[p] = acc;
    }
    __syncthreads();
    // y pass: b0 = (I x G_y x I) b1
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
        const int y = (p / nx) % ny;
        float acc = 0.0f;
        for (int d = -3; d <= 3; ++d)
            if (y + d >= 0 && y + d < ny)
                acc += G[1][y * 7 + d + 3] * b1[p + d * nx];
        b0[p] = acc;
    }
    __syncthreads();
    // z pass and the quadratic form
    double dot = 0.0;
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
        const int z = p / (nx * ny);
        float acc = 0.0f;
        for (int d = -3; d <= 3; ++d)
            if (z + d >= 0 && z + d < nz)
                acc += G[2][z * 7 + d + 3] * b0[p + d * nx * ny];
        const float e = c[off + p] - ct[off + p];
        dot += (double)e * (double)acc;
        gc[off + p] = (float)(a.gscale * acc);
    }
    red[threadIdx.x] = dot;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        part[blockIdx.x] = red[0];
}

__global__ void k_field_loss_finish(const double *__restrict__ part, int n, double scale,
                                    double *__restrict__ loss)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < n; ++i)
            s += part[i];
        *loss = s * scale;
    }
}

__global__ void k_adam_flat(AdamFlatArgs a, const int64_t *__restrict__ step,
                            float *__restrict__ p, const float *__restrict__ g,
                            float *__restrict__ m, float *__restrict__ v)
{
    __shared__ float s_ib[2];
    if (threadIdx.x == 0) {
        const long long t = (long long)*step + 1;
        s_ib[0] = adam_inv_bias(a.beta1, t);
        s_ib[1] = adam_inv_bias(a.beta2, t);
    }
    __syncthreads();
    const float b1 = (float)a.beta1, b2 = (float)a.beta2;
    const float o1 = (float)(1.0 - a.beta1), o2 = (float)(1.0 - a.beta2);
    const float ib1 = s_ib[0], ib2 = s_ib[1];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float mm = m[i], vv = v[i];
        p[i] = adam_flat_update(p[i], g[i], mm, vv, b1, o1, b2, o2, a.lr, a.eps, ib1, ib2);
        m[i] = mm;
        v[i] = vv;
    }
}

__global__ void k_tick(int64_t *step)
{
    if (threadIdx.x == 0 && blockIdx.x == 0)
        *step += 1;
}

// out[v][z][y][x] = sum_b a_b exp(-|x - mu_b|^2 / (2 sigma_b^2)) for the
// blob table of volume v ([blob][mu_x, mu_y, mu_z, sigma, a]). A block owns
// a TB x TB x 32 box (x, y, z) and takes the table in chunks of 64 or 128 blobs, of
// which it keeps those that come within 6 sigma of the 16 x 16 x 32 box around
// it (in table order; the same blobs whatever TB, so the same bits): a
// dropped term is below a exp(-18) < 1.6e-8 a everywhere in the box. A Gaussian
// separates into per-axis factors,
//   a exp(-|p - mu|^2 / (2 sigma^2)) = ex(x) ey(y) (a ez(z)),
// so a kept blob takes 2 TB + 32 exponentials per box. With TB = 16 a thread owns four
// columns (x .. x + 3, y) of 8 slices; per blob two packed products ex ey, one
// 16-byte read of ex, one 8-byte read of ey, four 16-byte reads of the z factors
// (y and z factors stored twice, as the packed operands want them) and 16 packed
// f32x2 FMAs: 24 instructions for 32 voxels and a blob, the FMAs' rate (34 us for
// 16 x 128^3 voxels, 60 blobs of sigma 3-12) being the bound. That case takes 49 us;
// 92 with one column of 8 slices per thread and boxes of 8 x 8, whose factor loads
// and exponentials took half the issue slots. Calls of few boxes are chains of latencies
// instead, and take boxes of 8 x 8 with one column of 8 slices per thread: 2 volumes of
// 64 x 64 x 20 and 500 blobs 92 us with four columns, 35 so; one of 128 x 256 x 16 and 60
// blobs 10 us either way.
constexpr int kBrickZ = 32;    // z extent: 4 groups of 8 slices

template <int TB>
__global__ void __launch_bounds__(256, 4)
    k_render_blobs(int D, int H, int W, int nblobs, const float *__restrict__ table,
                   float *__restrict__ out, int vec)
{
    constexpr int NT = 256, CX = TB == 16 ? 4 : 1;  // threads; columns of a thread
    // factors of a blob: TB = 16: ex, (ey, ey), (a ez, a ez); TB = 8: ex, ey, a ez
    constexpr int OY = TB, OZ = CX == 4 ? 3 * TB : 2 * TB,
                  FAC = OZ + (CX == 4 ? 2 : 1) * kBrickZ;
    static_assert(NT == TB / CX * TB * 4 && FAC % 4 == 0 && OZ % 4 == 0, "16-byte rows");
    constexpr int CH = TB == 16 ? 64 : 128;  // blobs of a chunk
    __shared__ float4 fac4[CH * FAC / 4];
    __shared__ float par[CH][5];
    __shared__ unsigned kept[CH / 32];
    float *fac = reinterpret_cast<float *>(fac4);
    const int vol = blockIdx.y;
    const int bx = (W + TB - 1) / TB, by = (H + TB - 1) / TB;
    const int brick = blockIdx.x;
    const int x0 = (brick % bx) * TB, y0 = ((brick / bx) % by) * TB,
              z0 = (brick / (bx * by)) * kBrickZ;
    const float *tv = table + (int64_t)vol * nblobs * 5;
    const int t = threadIdx.x, lx = (t % (TB / CX)) * CX, ly = t / (TB / CX) % TB,
              zg = t / (TB / CX * TB);
    // TB = 16: columns (x, x + 1), (x + 2, x + 3) of slice i; TB = 8: slices 2 i, 2 i + 1
    float2 acc[CX == 4 ? 8 : 2][2];
#pragma unroll
    for (int i = 0; i < (CX == 4 ? 8 : 2); ++i)
        acc[i][0] = acc[i][1] = make_float2(0.0f, 0.0f);
    for (int b0 = 0; b0 < nblobs; b0 += CH) {
        float e[5];
        bool in = false;
        if (t < CH) {
            if (b0 + t < nblobs) {
#pragma unroll
                for (int k = 0; k < 5; ++k)
                    e[k] = __ldg(tv + (int64_t)(b0 + t) * 5 + k);
                // distance from the centre to the 16 x 16 x 32 box
                const int xb = x0 & ~15, yb = y0 & ~15;
                const float dx = fmaxf(fmaxf((float)xb - e[0], e[0] - (float)(xb + 15)), 0.0f);
                const float dy = fmaxf(fmaxf((float)yb - e[1], e[1] - (float)(yb + 15)), 0.0f);
                const float dz =
                    fmaxf(fmaxf((float)z0 - e[2], e[2] - (float)(z0 + kBrickZ - 1)), 0.0f);
                in = dx * dx + dy * dy + dz * dz <= 36.0f * e[3] * e[3];
            }
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (t % 32 == 0)
                kept[t / 32] = m;
        }
        __syncthreads();  // also: the previous chunk's factors are read
        int n = 0, before = 0;  // kept blobs, those of the warps before this one
#pragma unroll
        for (int w = 0; w < CH / 32; ++w) {
            before = w == t / 32 ? n : before;
            n += __popc(kept[w]);
        }
        if (in) {
            const int k = before + __popc(kept[t / 32] & ((1u << (t % 32)) - 1u));
#pragma unroll
            for (int q = 0; q < 5; ++q)
                par[k][q] = e[q];
        }
        __syncthreads();
        // the per-axis factors of the kept blobs at the box's coordinates
        constexpr int NE = 2 * TB + kBrickZ;
        for (int i = t; i < n * NE; i += NT) {
            const int k = i / NE, r = i - k * NE;
            const int axis = r < TB ? 0 : r < 2 * TB ? 1 : 2;
            const int o = r - axis * TB;
            const float c = (float)((axis == 0 ? x0 : axis == 1 ? y0 : z0) + o) - par[k][axis];
            float v = expf(-0.5f * c * c / (par[k][3] * par[k][3]));
            if (axis == 2)
                v = par[k][4] * v;
            float *f = fac + FAC * k;
            if (axis == 0)
                f[o] = v;
            else if (CX == 1)
                f[(axis == 1 ? OY : OZ) + o] = v;
            else
                reinterpret_cast<float2 *>(f + (axis == 1 ? OY : OZ))[o] = make_float2(v, v);
        }
        __syncthreads();
#pragma unroll 2
        for (int k = 0; k < n; ++k) {
            const float *f = fac + FAC * k;
            if constexpr (CX == 4) {
                const float4 ex = *reinterpret_cast<const float4 *>(f + lx);
                const float2 ey = *reinterpret_cast<const float2 *>(f + OY + 2 * ly);
                const float2 p0 = __fmul2_rn(make_float2(ex.x, ex.y), ey);
                const float2 p1 = __fmul2_rn(make_float2(ex.z, ex.w), ey);
                const float4 *zz = reinterpret_cast<const float4 *>(f + OZ + 16 * zg);
#pragma unroll
                for (int i = 0; i < 8; i += 2) {
                    const float4 z = zz[i / 2];
                    acc[i][0] = __ffma2_rn(p0, make_float2(z.x, z.y), acc[i][0]);
                    acc[i][1] = __ffma2_rn(p1, make_float2(z.x, z.y), acc[i][1]);
                    acc[i + 1][0] = __ffma2_rn(p0, make_float2(z.z, z.w), acc[i + 1][0]);
                    acc[i + 1][1] = __ffma2_rn(p1, make_float2(z.z, z.w), acc[i + 1][1]);
                }
            } else {
                const float pxy = f[lx] * f[OY + ly];
                const float2 p = make_float2(pxy, pxy);
                const float4 *zz = reinterpret_cast<const float4 *>(f + OZ + 8 * zg);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float4 z = zz[i];
                    acc[i][0] = __ffma2_rn(p, make_float2(z.x, z.y), acc[i][0]);
                    acc[i][1] = __ffma2_rn(p, make_float2(z.z, z.w), acc[i][1]);
                }
            }
        }
    }
    const int x = x0 + lx, y = y0 + ly;
    if (x >= W || y >= H)
        return;
    float *o = out + ((int64_t)vol * D * H + y) * W + x;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int z = z0 + 8 * zg + i;
        if (z >= D)
            break;
        float *oz = o + (int64_t)z * H * W;
        if constexpr (CX == 1) {
            const float2 v = acc[i / 4][i / 2 % 2];
            *oz = i % 2 ? v.y : v.x;
        } else {
            const float v[4] = {acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y};
            if (vec) {
                *reinterpret_cast<float4 *>(oz) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (x + j < W)
                        oz[j] = v[j];
            }
        }
    }
}

template <int TB>
cudaError_t run_render(int D, int H, int W, int count, int nblobs, const float *table, float *out,
                       cudaStream_t s)
{
    const int64_t boxes = (int64_t)((W + TB - 1) / TB) * ((H + TB - 1) / TB) *
                          ((D + kBrickZ - 1) / kBrickZ);
    // rows of whole 16-byte pieces (out is 16-byte aligned)
    k_render_blobs<TB><<<dim3((unsigned)boxes, count), 256, 0, s>>>(D, H, W, nblobs, table, out,
                                                                   W % 4 == 0);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_net_input(int64_t n, const float *F, const float *M, void *x, cudaStream_t s)
{
    ProfScope ps(s, "k_net_input");
    k_net_input<<<blocks(n), kT, 0, s>>>(F, M, n, static_cast<__nv_bfloat162 *>(x));
    return cudaGetLastError();
}

cudaError_t launch_upcat(const NetGrid &g, int c4, int c3, const void *e4, const void *e3,
                         void *cat, cudaStream_t s)
{
    ProfScope ps(s, "k_upcat");
    const int64_t n = (int64_t)g.nb * g.n3[0] * g.n3[1] * g.n3[2] * ((c4 + c3) / 8);
    k_upcat<<<blocks(n), kT, 0, s>>>(g, c4, c3, static_cast<const uint4 *>(e4),
                                     static_cast<const uint4 *>(e3), static_cast<uint4 *>(cat));
    return cudaGetLastError();
}

cudaError_t launch_upcat_adjoint(const NetGrid &g, int c4, int c3, const void *gcat,
                                 const void *e4, void *ge4, cudaStream_t s)
{
    ProfScope ps(s, "k_upcat_adjoint");
    const int64_t n = (int64_t)g.nb * g.n4[0] * g.n4[1] * g.n4[2] * c4;
    k_upcat_adjoint<<<blocks(n), kT, 0, s>>>(g, c4, c3, static_cast<const __nv_bfloat16 *>(gcat),
                                             static_cast<const __nv_bfloat16 *>(e4),
                                             static_cast<__nv_bfloat16 *>(ge4));
    return cudaGetLastError();
}

cudaError_t launch_head_to_ctrl(const NetGrid &g, int ch, const float *h, float *c, cudaStream_t s)
{
    ProfScope ps(s, "k_head_to_ctrl");
    const int64_t n = (int64_t)g.nb * 3 * g.lat[0] * g.lat[1] * g.lat[2];
    k_head_to_ctrl<<<blocks(n), kT, 0, s>>>(g, ch, h, c);
    return cudaGetLastError();
}

cudaError_t launch_head_adjoint(const NetGrid &g, int ch, const float *gc, void *gh,
                                cudaStream_t s)
{
    ProfScope ps(s, "k_head_adjoint");
    const int64_t n = (int64_t)g.nb * g.n3[0] * g.n3[1] * g.n3[2] * ch;
    k_head_adjoint<<<blocks(n), kT, 0, s>>>(g, ch, gc, static_cast<__nv_bfloat16 *>(gh));
    return cudaGetLastError();
}

size_t field_loss_smem(const FieldLossArgs &a)
{
    const int np = a.n[0] * a.n[1] * a.n[2];
    return sizeof(double) * kFieldT + sizeof(float) * 7 * (a.n[0] + a.n[1] + a.n[2]) +
           sizeof(float) * 2 * np;
}

cudaError_t launch_field_loss(const FieldLossArgs &a, int nb, const float *c, const float *ct,
                              float *gc, double *part, double *loss, cudaStream_t s)
{
    const size_t sm = field_loss_smem(a);
    cudaError_t e = cudaFuncSetAttribute(k_field_loss, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sm);
    if (e != cudaSuccess)
        return e;
    {
        ProfScope ps(s, "k_field_loss");
        k_field_loss<<<nb * 3, kFieldT, sm, s>>>(a, c, ct, gc, part);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    ProfScope ps(s, "k_field_loss_finish");
    k_field_loss_finish<<<1, 32, 0, s>>>(part, nb * 3, a.lscale, loss);
    return cudaGetLastError();
}

cudaError_t launch_adam_flat(const AdamFlatArgs &a, int64_t *step, float *p, const float *g,
                             float *m, float *v, cudaStream_t s)
{
    {
        ProfScope ps(s, "k_adam_flat");
        k_adam_flat<<<blocks(a.n), kT, 0, s>>>(a, step, p, g, m, v);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    return launch_step_tick(step, s);
}

cudaError_t launch_step_tick(int64_t *step, cudaStream_t s)
{
    ProfScope ps(s, "k_tick");
    k_tick<<<1, 32, 0, s>>>(step);
    return cudaGetLastError();
}

cudaError_t launch_render_blobs(int D, int H, int W, int count, int nblobs, const float *table,
                                float *out, cudaStream_t s)
{
    ProfScope ps(s, "k_render_blobs");
    const int64_t boxes16 = (int64_t)((W + 15) / 16) * ((H + 15) / 16) *
                            ((D + kBrickZ - 1) / kBrickZ) * count;
    // boxes of 16 x 16 need a third of the exponentials per voxel; below two per SM
    // the smaller ones spread better (12 us either way at 48^3: launch)
    if (boxes16 >= 2 * (int64_t)device_sms())
        return run_render<16>(D, H, W, count, nblobs, table, out, s);
    return run_render<8>(D, H, W, count, nblobs, table, out, s);
}

}  // namespace airgb
