// The optimisation loop around the objective: Adam on the control points
// (Sec. II-A, Optimization; Sec. III-G), one level of the Gaussian image
// pyramid and the dyadic refinement of the B-spline coefficients between
// levels (multi-resolution strategy of Sec. IV-A).
//
// All three are light: Adam streams 7 floats per coefficient (0.19 M
// coefficients at 256x256x160, spacing 6), the pyramid reads an image once,
// the refinement gathers at most 27 coarse coefficients per fine
// one. They are elementwise, filter and gather kernels sized to the data; what
// matters is that the whole loop stays on the device (no host round trip per
// iteration) so that a level's iterations can be captured in a CUDA graph.
#include "launch.h"
#include "profile.h"

namespace airgb {

namespace {

constexpr int kOptThreads = 256;

int blocks_for(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    return (int)(b < 1 ? 1 : b);
}

// ---- Adam ------------------------------------------------------------------
// m, v are the moments of the gradient in normalised units (the image spans
// [-1, 1] per axis, Sec. III-C); ctrl and grad stay in voxel units, so with
// h = (N_k - 1)/2 voxels per normalised unit:
//   g~ = h g, m <- b1 m + (1 - b1) g~, v <- b2 v + (1 - b2) g~^2,
//   c <- c - h lr (m / bc1) / (sqrt(v / bc2) + eps),  bc = 1 - b^t.
// t = *step + 1 is read from the device counter; k_adam_tick stores it
// afterwards, so a captured graph replays successive steps.
// A small launch is one chain of latencies: the two bias corrections are formed
// by a warp each while the block's operands are on their way (128^3 at spacing 8,
// 81 blocks: 5.9 us with the corrections one after the other before the loads,
// 4.2 so).
__global__ void __launch_bounds__(kOptThreads)
    k_adam(AdamArgs a, const int64_t *__restrict__ step, float *__restrict__ ctrl,
           const float *__restrict__ grad, float *__restrict__ m, float *__restrict__ v)
{
    __shared__ float s_inv_bc[2];
    const int64_t n = (int64_t)a.ndim * a.nc;
    const int64_t e = blockIdx.x * (int64_t)kOptThreads + threadIdx.x;  // one element a thread
    const bool on = e < n;
    float ge = 0.0f, me = 0.0f, ve = 0.0f, ce = 0.0f;
    if (on) {
        ge = grad[e];
        me = m[e];
        ve = v[e];
        ce = ctrl[e];
    }
    if (threadIdx.x % 32 == 0 && threadIdx.x < 64)
        s_inv_bc[threadIdx.x / 32] =
            adam_inv_bias(threadIdx.x == 0 ? a.beta1 : a.beta2, (long long)*step + 1);
    __syncthreads();
    if (!on)
        return;
    const float inv_bc1 = s_inv_bc[0], inv_bc2 = s_inv_bc[1];
    const float b1 = (float)a.beta1, b2 = (float)a.beta2;
    const float omb1 = (float)(1.0 - a.beta1), omb2 = (float)(1.0 - a.beta2);
    const float h = a.h[(e >= a.nc) + (e >= 2 * a.nc)];
    const float gn = ge * h;
    const float mm = fmaf(b1, me, omb1 * gn);
    const float vv = fmaf(b2, ve, omb2 * gn * gn);
    m[e] = mm;
    v[e] = vv;
    const float den = sqrtf(vv * inv_bc2) + a.eps;
    ctrl[e] = ce - (a.lr * h) * ((mm * inv_bc1) / den);
}

__global__ void k_adam_tick(int64_t *step)
{
    if (threadIdx.x == 0 && blockIdx.x == 0)
        *step += 1;
}

// ---- pyramid ---------------------------------------------------------------
// Output tile of k_pyramid_xy and the input rows and columns it stages, per
// factor F (taps -r..r, r = floor(3 F / 2); a staged row starts on 4 floats,
// so it holds up to 3 columns more).
template <int F>
struct PyrTile {
    static constexpr int R = 3 * F / 2;
    static constexpr int OX = F <= 3 ? 64 : (F == 4 ? 32 : 16);
    static constexpr int OY = F <= 2 ? 16 : (F <= 4 ? 8 : 4);
    static constexpr int ROWS = (OY - 1) * F + 2 * R + 1;
    static constexpr int COLS = ((OX - 1) * F + 2 * R + 1 + 3 + 3) / 4 * 4;
};

// Smooth along x and y with the taps w[0..2R] (indices clamped to the grid)
// and keep every F-th point from 0 of each, slice by slice: in[Z][Y][X] ->
// out[Z][OY][OX]. Memory bound: one read of the image (42 MB at
// 256 x 256 x 160, 6.2 us at the measured HBM rate) and a write F^2 smaller.
// A block stages its input rows in shared memory once, 16 bytes a load where
// they lie inside the row and X is a multiple of 4, filters them along x into
// a second buffer and that one along y. Both images' next level and the
// refinement at 256 x 256 x 160, factor 2: 264.7 us with one pass per axis
// (one thread per output, 64-bit index divisions, full-size intermediates in
// memory), 59 us of kernels with this one and k_pyramid_z. Sums run in the order of
// the taps, x then y then z, as one pass per axis forms them: the same bits.
template <int F>
__global__ void __launch_bounds__(kOptThreads)
    k_pyramid_xy(const float *__restrict__ in, float *__restrict__ out, int X, int Y, int OX,
                 int OY, int ntx, int nty, const __grid_constant__ GaussTaps t)
{
    using T = PyrTile<F>;
    __shared__ __align__(16) float raw[T::ROWS][T::COLS];
    __shared__ float fx[T::ROWS][T::OX];
    const int tile = blockIdx.x;
    const int tx = tile % ntx, ty = (tile / ntx) % nty, z = tile / (ntx * nty);
    const int ox0 = tx * T::OX, oy0 = ty * T::OY;
    const int y0 = oy0 * F - T::R;
    const int xs = ox0 * F - T::R;
    const int xa = xs & ~3;  // two's complement: rounds down, also below 0
    const float *slice = in + (int64_t)z * Y * X;
    const bool vec = (X & 3) == 0;
    constexpr int GROUPS = T::COLS / 4;
    for (int e = threadIdx.x; e < T::ROWS * GROUPS; e += kOptThreads) {
        const int r = e / GROUPS, g = e - r * GROUPS;
        const float *row = slice + (int64_t)min(max(y0 + r, 0), Y - 1) * X;
        const int x = xa + 4 * g;
        float4 v;
        if (vec && x >= 0 && x + 3 < X) {
            v = __ldg(reinterpret_cast<const float4 *>(row + x));
        } else {
            v.x = __ldg(row + min(max(x, 0), X - 1));
            v.y = __ldg(row + min(max(x + 1, 0), X - 1));
            v.z = __ldg(row + min(max(x + 2, 0), X - 1));
            v.w = __ldg(row + min(max(x + 3, 0), X - 1));
        }
        *reinterpret_cast<float4 *>(&raw[r][4 * g]) = v;
    }
    __syncthreads();
    const int sh = xs - xa;
    for (int e = threadIdx.x; e < T::ROWS * T::OX; e += kOptThreads) {
        const int r = e / T::OX, ox = e - r * T::OX;
        const float *p = &raw[r][ox * F + sh];
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k <= 2 * T::R; ++k)
            s = fmaf(t.w[k], p[k], s);
        fx[r][ox] = s;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < T::OY * T::OX; e += kOptThreads) {
        const int oy = e / T::OX, ox = e - oy * T::OX;
        if (ox0 + ox >= OX || oy0 + oy >= OY)
            continue;
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k <= 2 * T::R; ++k)
            s = fmaf(t.w[k], fx[oy * F + k][ox], s);
        out[((int64_t)z * OY + oy0 + oy) * OX + ox0 + ox] = s;
    }
}

// The z pass: in[Z][plane] -> out[OZ][plane], one thread per VEC consecutive
// values of a plane (4 when the plane is a multiple of 4, so that every slice
// starts on 16 bytes). Its input is F^2 smaller than the image and still in L2.
template <int VEC>
__global__ void __launch_bounds__(kOptThreads)
    k_pyramid_z(const float *__restrict__ in, float *__restrict__ out, int Z, int OZ, int plane,
                int factor, const __grid_constant__ GaussTaps t)
{
    const int per = plane / VEC;
    const int64_t n = (int64_t)per * OZ;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int oz = (int)(e / per), i = ((int)(e - (int64_t)oz * per)) * VEC;
        float s[VEC] = {};
#pragma unroll 4
        for (int k = 0; k <= 2 * t.r; ++k) {
            const int p = min(max(oz * factor + k - t.r, 0), Z - 1);
            const float *src = in + (int64_t)p * plane + i;
            if constexpr (VEC == 4) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(src));
                s[0] = fmaf(t.w[k], v.x, s[0]);
                s[1] = fmaf(t.w[k], v.y, s[1]);
                s[2] = fmaf(t.w[k], v.z, s[2]);
                s[3] = fmaf(t.w[k], v.w, s[3]);
            } else {
                s[0] = fmaf(t.w[k], __ldg(src), s[0]);
            }
        }
        if constexpr (VEC == 4)
            *reinterpret_cast<float4 *>(out + (int64_t)oz * plane + i) =
                make_float4(s[0], s[1], s[2], s[3]);
        else
            out[(int64_t)oz * plane + i] = s[0];
    }
}

template <int F>
void run_pyramid_xy(const Grid &g, int OX, int OY, const GaussTaps &t, const float *image,
                    float *out, cudaStream_t s)
{
    const int ntx = (OX + PyrTile<F>::OX - 1) / PyrTile<F>::OX;
    const int nty = (OY + PyrTile<F>::OY - 1) / PyrTile<F>::OY;
    k_pyramid_xy<F><<<ntx * nty * g.Z, kOptThreads, 0, s>>>(image, out, g.X, g.Y, OX, OY, ntx, nty,
                                                            t);
}

// ---- refinement ------------------------------------------------------------
// Fine coefficient i from the coarse lattice by the two-scale relation of the
// cubic B-spline: with q = i - 1, j = floor(q/2) + 1, an even q takes
// (1, 6, 1)/8 of coarse j-1, j, j+1 and an odd q takes (1, 1)/2 of j, j+1,
// per axis; the tensor product is multiplied by 2 (coarse voxel units are
// twice the fine ones). The host checks that every tap lies in the coarse
// lattice.
struct Taps1 {
    int j0, n;
    float w[3];
};

__device__ __forceinline__ Taps1 refine_taps(int i)
{
    const int q = i - 1;          // >= -1
    const int j = (q + 2) / 2;    // floor(q/2) + 1
    Taps1 t;
    if ((q & 1) == 0) {
        t.j0 = j - 1, t.n = 3;
        t.w[0] = 0.125f, t.w[1] = 0.75f, t.w[2] = 0.125f;
    } else {
        t.j0 = j, t.n = 2;
        t.w[0] = 0.5f, t.w[1] = 0.5f, t.w[2] = 0.0f;
    }
    return t;
}

__global__ void __launch_bounds__(kOptThreads)
    k_refine(const float *__restrict__ cc, float *__restrict__ cf, int ndim, int cx, int cy,
             int cz, int fx, int fy, int fz)
{
    const int64_t nff = (int64_t)fx * fy * fz, ncc = (int64_t)cx * cy * cz;
    const int64_t n = ndim * nff;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int comp = (int)(e / nff);
        const int64_t r = e - comp * nff;
        const int ix = (int)(r % fx), iy = (int)((r / fx) % fy), iz = (int)(r / ((int64_t)fx * fy));
        const Taps1 tx = refine_taps(ix), ty = refine_taps(iy);
        Taps1 tz;
        if (ndim == 3) {
            tz = refine_taps(iz);
        } else {
            tz.j0 = 0, tz.n = 1, tz.w[0] = 1.0f, tz.w[1] = tz.w[2] = 0.0f;
        }
        const float *src = cc + comp * ncc;
        float s = 0.0f;
        for (int a = 0; a < tz.n; ++a) {
            const int jz = tz.j0 + a;
            for (int b = 0; b < ty.n; ++b) {
                const int jy = ty.j0 + b;
                float sy = 0.0f;
                for (int k = 0; k < tx.n; ++k) {
                    const int jx = tx.j0 + k;
                    sy = fmaf(tx.w[k], __ldg(src + ((int64_t)jz * cy + jy) * cx + jx), sy);
                }
                s = fmaf(tz.w[a] * ty.w[b], sy, s);
            }
        }
        cf[e] = 2.0f * s;
    }
}

}  // namespace

cudaError_t launch_adam(const AdamArgs &a, int64_t *step, float *ctrl, const float *grad,
                        float *m, float *v, cudaStream_t s)
{
    const int64_t n = (int64_t)a.ndim * a.nc;
    const int blocks = blocks_for(n, kOptThreads);
    {
        ProfScope ps(s, "k_adam");
        k_adam<<<blocks, kOptThreads, 0, s>>>(a, step, ctrl, grad, m, v);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    k_adam_tick<<<1, 32, 0, s>>>(step);
    return cudaGetLastError();
}

size_t pyramid_ws(const Grid &g, int factor)
{
    if (factor == 1)
        return 0;
    const int64_t OX = (g.X - 1) / factor + 1, OY = (g.Y - 1) / factor + 1;
    const size_t a = (size_t)OX * g.Y * g.Z * 4, b = (size_t)OX * OY * g.Z * 4;
    return (a + 255) / 256 * 256 + (b + 255) / 256 * 256;
}

cudaError_t launch_pyramid(const Grid &g, int factor, const GaussTaps &t, const float *image,
                           float *level, void *ws, cudaStream_t s)
{
    if (factor == 1)
        return cudaMemcpyAsync(level, image, (size_t)g.nv * 4, cudaMemcpyDeviceToDevice, s);
    const int OX = (g.X - 1) / factor + 1, OY = (g.Y - 1) / factor + 1;
    const int OZ = g.ndim == 3 ? (g.Z - 1) / factor + 1 : 1;
    const int64_t nl = (int64_t)OX * OY * OZ;
    // the x/y pass goes to the workspace when a z pass follows it, and when the
    // level overlaps the image it is formed from
    const bool overlap = image < level + nl && level < image + g.nv;
    float *xy = g.ndim == 3 || overlap ? static_cast<float *>(ws) : level;
    ProfScope ps(s, "k_pyramid");
    switch (factor) {
    case 2: run_pyramid_xy<2>(g, OX, OY, t, image, xy, s); break;
    case 3: run_pyramid_xy<3>(g, OX, OY, t, image, xy, s); break;
    case 4: run_pyramid_xy<4>(g, OX, OY, t, image, xy, s); break;
    case 5: run_pyramid_xy<5>(g, OX, OY, t, image, xy, s); break;
    case 6: run_pyramid_xy<6>(g, OX, OY, t, image, xy, s); break;
    case 7: run_pyramid_xy<7>(g, OX, OY, t, image, xy, s); break;
    default: run_pyramid_xy<8>(g, OX, OY, t, image, xy, s); break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || xy == level)
        return e;
    if (g.ndim == 2)
        return cudaMemcpyAsync(level, xy, (size_t)nl * 4, cudaMemcpyDeviceToDevice, s);
    const int plane = OX * OY;
    if (plane % 4 == 0)
        k_pyramid_z<4><<<blocks_for(nl / 4, kOptThreads), kOptThreads, 0, s>>>(xy, level, g.Z, OZ,
                                                                               plane, factor, t);
    else
        k_pyramid_z<1><<<blocks_for(nl, kOptThreads), kOptThreads, 0, s>>>(xy, level, g.Z, OZ,
                                                                           plane, factor, t);
    return cudaGetLastError();
}

cudaError_t launch_refine(int ndim, const int *nc, const int *nf, const float *cc, float *cf,
                          cudaStream_t s)
{
    const int64_t n = (int64_t)ndim * nf[0] * nf[1] * nf[2];
    ProfScope ps(s, "k_refine");
    k_refine<<<blocks_for(n, kOptThreads), kOptThreads, 0, s>>>(cc, cf, ndim, nc[0], nc[1], nc[2],
                                                                 nf[0], nf[1], nf[2]);
    return cudaGetLastError();
}

}  // namespace airgb
