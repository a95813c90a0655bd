// Diffeomorphic B-spline transformation (Sec. III-D): f = exp(v) of the
// stationary velocity field v by scaling and squaring,
//   u_0 = v / 2^K,  u_{k+1}(x) = u_k(x) + u~_k(x + u_k(x)),  f = x + u_K,
// and the adjoint of that map. u~_k is the linear interpolant of u_k at the
// sample position clamped to the grid (a field has no mask); along a clamped
// axis the interpolant is constant, so its derivative there is 0.
//
// The adjoint of one squaring is, with p(x) = x + u_k(x),
//   g_k(y) = g_{k+1}(y) + (du~_k/dp at p(y))^T g_{k+1}(y)
//            + sum_x w_y(p(x)) g_{k+1}(x).
// The first two terms are local. The last is the transpose of the
// interpolation, a scatter from every sample to the corners of its cell.
// It is accumulated in 64-bit fixed point with integer atomics: integer
// addition is associative, so the result does not depend on the order in
// which the atomics land (deterministic, unlike float atomics). The scale
// 2^s is chosen per step from the largest |g| (an exact max reduction) so
// that a node can take 2^20 contributions of the largest size without
// overflow; the fixed point then resolves 2^-42 of that size, far below fp32
// rounding of the contributions themselves.
#include <algorithm>

#include "launch.h"
#include "profile.h"

namespace airgb {

namespace {

constexpr int kDiffeoThreads = 256;

int blocks_for(int64_t n)
{
    int64_t b = (n + kDiffeoThreads - 1) / kDiffeoThreads;
    return (int)(b < 1 ? 1 : b);
}

// Cell and offset of the position x + u along an axis of n points, clamped
// into [0, n - 1]; returns whether the position was inside (a non-finite u
// counts as outside: NaN and -inf at 0, +inf at n - 1). No branches: u is
// clamped to [lo, hi] = [-x, n - 1 - x] (exact floats, axes are shorter than
// 2^22), and one round-toward-minus-infinity add of 1.5 * 2^23 leaves floor(u)
// in the low mantissa bits; the integer part is split off first, so x + u is
// not rounded in fp32.
__device__ __forceinline__ bool field_axis(int x, float u, float lo, float hi, int n,
                                                int &cell, float &f)
{
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23, bit pattern 0x4B400000
    const float uc = fminf(fmaxf(u, lo), hi);
    const float t = __fadd_rd(uc, kMagic);
    const int iy = x + (__float_as_int(t) - 0x4B400000);
    const float fr = uc - (t - kMagic);
    cell = min(iy, n - 2);
    f = iy > cell ? fr + 1.0f : fr;  // the last face: all weight on the last point
    return u >= lo && u <= hi;
}

// Interpolant of one component (times sc) in the cell at p, every linear step
// as fma(1 - f, a, f b). In 3D the two z faces are packed pairs.
template <int D>
__device__ __forceinline__ float interp_field(const float *__restrict__ p, int sy, int sz,
                                              float fx, float fy, float fz, float sc)
{
    const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
    if constexpr (D == 2) {
        const float c0 = fmaf(gx, __ldg(p) * sc, fx * (__ldg(p + 1) * sc));
        const float c1 = fmaf(gx, __ldg(p + sy) * sc, fx * (__ldg(p + sy + 1) * sc));
        return fmaf(gy, c0, fy * c1);
    } else {
        const float *q = p + sz;
        const float2 a = make_float2(__ldg(p) * sc, __ldg(q) * sc);
        const float2 b = make_float2(__ldg(p + 1) * sc, __ldg(q + 1) * sc);
        const float2 c = make_float2(__ldg(p + sy) * sc, __ldg(q + sy) * sc);
        const float2 d = make_float2(__ldg(p + sy + 1) * sc, __ldg(q + sy + 1) * sc);
        const float2 gx2 = make_float2(gx, gx), fx2 = make_float2(fx, fx);
        const float2 c0 = __ffma2_rn(gx2, a, __fmul2_rn(fx2, b));
        const float2 c1 = __ffma2_rn(gx2, c, __fmul2_rn(fx2, d));
        const float2 r = __ffma2_rn(make_float2(gy, gy), c0, __fmul2_rn(make_float2(fy, fy), c1));
        return fmaf(gz, r.x, fz * r.y);
    }
}

__global__ void __launch_bounds__(kDiffeoThreads)
    k_scale(const float *__restrict__ in, float *__restrict__ out, float s, int64_t n)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x)
        out[e] = in[e] * s;
}

// One squaring of a 2D field: out = u + u~(x + u), the field read as u * sc
// (sc = 2^-K on the first squaring, which then reads v itself and also writes
// u_0 = v sc to u0 when given; otherwise 1). Scaling by a power of two is
// exact, so this equals scaling v in a pass of its own first.
template <bool SCALED>
__global__ void __launch_bounds__(kDiffeoThreads)
    k_compose2(Grid g, const float *__restrict__ u, float *__restrict__ out, float scale,
               float *__restrict__ u0)
{
    const float sc = SCALED ? scale : 1.0f;  // a compile-time 1 on every squaring but the first
    const int v = blockIdx.x * kDiffeoThreads + threadIdx.x;
    if (v >= g.nv)
        return;
    const int y = v / g.X, x = v - y * g.X;
    const float a0 = __ldg(u + v) * sc, a1 = __ldg(u + g.nv + v) * sc;
    int cx, cy;
    float fx, fy;
    field_axis(x, a0, -(float)x, (float)(g.X - 1 - x), g.X, cx, fx);
    field_axis(y, a1, -(float)y, (float)(g.Y - 1 - y), g.Y, cy, fy);
    const float *p = u + cy * g.X + cx;
    const float r0 = interp_field<2>(p, g.X, 0, fx, fy, 0.0f, sc);
    const float r1 = interp_field<2>(p + g.nv, g.X, 0, fx, fy, 0.0f, sc);
    if (SCALED && u0) {
        u0[v] = a0;
        u0[g.nv + v] = a1;
    }
    out[v] = a0 + r0;
    out[g.nv + v] = a1 + r1;
}

// The same squaring of a 3D field: a warp takes 32 consecutive x of a row and
// marches through zc slices, so that the index arithmetic is done once per
// column and the cells come without branches. Bound by the L1's wavefronts (24
// gathers a voxel) and their latency: 134 us a squaring at 256 x 256 x 160
// (217 us the scaled one) with 64-bit divisions and branches per voxel, 81 us
// (98 us) so; two passes over memory take 37 us. Four blocks per SM (64
// registers) against six: 525 and 544 us for the six squarings; 16 slices
// instead of 8 took 544, 32 took 830.
template <bool SCALED>
__global__ void __launch_bounds__(kDiffeoThreads, 4)
    k_compose3(Grid g, const float *__restrict__ u, float *__restrict__ out, float scale,
               float *__restrict__ u0, int ntx, int nty, int zc, int lx)
{
    const float sc = SCALED ? scale : 1.0f;
    const int tile = blockIdx.x, tx = tile % ntx, ty = (tile / ntx) % nty, tz = tile / (ntx * nty);
    const int x = (tx << lx) + (threadIdx.x & ((1 << lx) - 1)),
              y = ty * (kDiffeoThreads >> lx) + (threadIdx.x >> lx);
    if (x >= g.X || y >= g.Y)
        return;
    const int sy = g.X, sz = g.X * g.Y;
    const float xlo = -(float)x, xhi = (float)(g.X - 1 - x);
    const float ylo = -(float)y, yhi = (float)(g.Y - 1 - y);
    const int z1 = min((tz + 1) * zc, g.Z);
    const float *u1 = u + g.nv, *u2 = u1 + g.nv;
    float *o1 = out + g.nv, *o2 = o1 + g.nv;
    unsigned v = (unsigned)((tz * zc * g.Y + y) * g.X + x);
    for (int z = tz * zc; z < z1; ++z, v += sz) {
        const float a0 = __ldg(u + v) * sc, a1 = __ldg(u1 + v) * sc, a2 = __ldg(u2 + v) * sc;
        int cx, cy, cz;
        float fx, fy, fz;
        field_axis(x, a0, xlo, xhi, g.X, cx, fx);
        field_axis(y, a1, ylo, yhi, g.Y, cy, fy);
        field_axis(z, a2, -(float)z, (float)(g.Z - 1 - z), g.Z, cz, fz);
        const int base = (cz * g.Y + cy) * g.X + cx;  // nv < 2^31
        const float r0 = interp_field<3>(u + base, sy, sz, fx, fy, fz, sc);
        const float r1 = interp_field<3>(u1 + base, sy, sz, fx, fy, fz, sc);
        const float r2 = interp_field<3>(u2 + base, sy, sz, fx, fy, fz, sc);
        if (SCALED && u0) {
            u0[v] = a0;
            u0[g.nv + v] = a1;
            u0[2 * g.nv + v] = a2;
        }
        out[v] = a0 + r0;
        o1[v] = a1 + r1;
        o2[v] = a2 + r2;
    }
}

// Largest |g| over n floats, as the bits of a non-negative float (ordered
// like unsigned integers), by atomicMax: exact and order-independent.
__global__ void __launch_bounds__(kDiffeoThreads)
    k_absmax(const float *__restrict__ gin, int64_t n, unsigned int *__restrict__ out)
{
    float m = 0.0f;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const float a = fabsf(gin[e]);
        m = a > m ? a : m;  // a NaN never wins
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0)
        atomicMax(out, __float_as_uint(m));
}

// 2^s for the fixed-point scatter: |w g| < 2^e, so every contribution stays
// below 2^(s + e) = 2^42 and 2^20 of them below 2^62.
__device__ __forceinline__ float fixed_scale(unsigned int maxbits)
{
    int e = 0;
    frexpf(__uint_as_float(maxbits), &e);
    const int s = min(42 - e, 100);
    return ldexpf(1.0f, s);
}

// round(p) of |p| <= 2^42 as a 64-bit integer, ties to even like
// __float2ll_rn, by fp32 adds. The 64-bit conversion instructions issue at the
// rate of this part's FP64 pipe, 16 cycles per warp, and 24 of them per voxel
// bounded the scatter. p = hi 2^21 + lo with hi = round(p / 2^21), |hi| <= 2^21,
// and lo = p - hi 2^21, |lo| <= 2^20, exact (a multiple of p's last place);
// adding 1.5 * 2^23 leaves an integer in the low mantissa bits. hi 2^21 is
// even, so round(p) = hi 2^21 + round(lo) to even.
__device__ __forceinline__ long long fixed_of(float p)
{
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    constexpr int kBits = 0x4B400000;
    const float t = __fmaf_rn(p, 0x1p-21f, kMagic);
    const float lo = __fmaf_rn(__fsub_rn(t, kMagic), -0x1p21f, p);
    const int ih = __float_as_int(t) - kBits;
    const int il = __float_as_int(__fadd_rn(lo, kMagic)) - kBits;
    return (long long)ih * 2097152ll + il;
}

// (float)q rounded to nearest even, like __ll2float_rn, with 32-bit
// conversions only: the top 32 significant bits of |q| with the bits below
// them or-ed into the last (more than the 24 that are kept, so one rounding).
__device__ __forceinline__ float float_of(long long q)
{
    const unsigned long long m = q < 0 ? 0ull - (unsigned long long)q : (unsigned long long)q;
    const unsigned hi = (unsigned)(m >> 32), lo = (unsigned)m;
    float f;
    if (hi == 0) {
        f = __uint2float_rn(lo);
    } else {
        const int k = __clz(hi);
        const unsigned top = __funnelshift_l(lo, hi, k), rest = lo << k;
        // top has its leading bit set; times 2^(32 - k), exact
        f = __uint2float_rn(top | (rest != 0u)) * __int_as_float((127 + 32 - k) << 23);
    }
    return q < 0 ? -f : f;
}

// The scatter of one sample whose gradient component does not fit the fixed
// point, one component (its plane's accumulators from the sample's cell).
template <int D>
__device__ __noinline__ void scatter_far(unsigned long long *acc, int sy, int sz,
                                         float fx, float fy, float fz, float gv, float S)
{
    for (int c = 0; c < (1 << D); ++c) {
        const int cx = c & 1, cy = (c >> 1) & 1, cz = c >> 2;
        const float wyz = (cy ? fy : 1.0f - fy) * (D == 3 ? (cz ? fz : 1.0f - fz) : 1.0f);
        const float w = (cx ? fx : 1.0f - fx) * wyz;
        atomicAdd(acc + cz * sz + cy * sy + cx,
                  (unsigned long long)__float2ll_rn(w * gv * S));
    }
}

// Local terms of one squaring's adjoint of a 2D field into h, the scatter into
// acc.
__global__ void __launch_bounds__(kDiffeoThreads)
    k_compose_adjoint2(Grid g, const float *__restrict__ u, const float *__restrict__ gin,
                       float *__restrict__ h, unsigned long long *__restrict__ acc,
                       const unsigned int *__restrict__ maxbits)
{
    const float S = fixed_scale(*maxbits);
    const int v = blockIdx.x * kDiffeoThreads + threadIdx.x;
    if (v >= g.nv)
        return;
    const int y = v / g.X, x = v - y * g.X, sy = g.X;
    int cx, cy;
    float fx, fy;
    const bool inx = field_axis(x, __ldg(u + v), -(float)x, (float)(g.X - 1 - x), g.X, cx, fx);
    const bool iny =
        field_axis(y, __ldg(u + g.nv + v), -(float)y, (float)(g.Y - 1 - y), g.Y, cy, fy);
    const int base = cy * g.X + cx;
    const float gx = 1.0f - fx, gy = 1.0f - fy;
    const float gv[2] = {__ldg(gin + v), __ldg(gin + g.nv + v)};
    float loc[2] = {gv[0], gv[1]};
    // derivative of the interpolant of each component at the sample
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float *p = u + (int64_t)i * g.nv + base;
        const float a00 = __ldg(p), a01 = __ldg(p + 1), a10 = __ldg(p + sy),
                    a11 = __ldg(p + sy + 1);
        const float d0 = fmaf(gy, a01 - a00, fy * (a11 - a10));
        const float d1 = fmaf(gx, a10 - a00, fx * (a11 - a01));
        if (inx)
            loc[0] = fmaf(d0, gv[i], loc[0]);
        if (iny)
            loc[1] = fmaf(d1, gv[i], loc[1]);
    }
    h[v] = loc[0];
    h[g.nv + v] = loc[1];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        unsigned long long *ap = acc + (int64_t)i * g.nv + base;
        const float gs = gv[i] * S;
        if (!(fabsf(gs) <= 0x1p42f)) {  // an infinity or a NaN
            scatter_far<2>(ap, sy, 0, fx, fy, 0.0f, gv[i], S);
            continue;
        }
        auto add = [&](unsigned long long *a, float w) {
            const long long q = fixed_of(w * gs);
            if (q != 0)
                atomicAdd(a, (unsigned long long)q);
        };
        add(ap, gx * gy);
        add(ap + 1, fx * gy);
        add(ap + sy, gx * fy);
        add(ap + sy + 1, fx * fy);
    }
}

// h += acc / 2^s; acc back to zero for the next step. With maxnext, also the
// largest |h| (the next step's input) into *maxnext, as k_absmax does, so that
// step needs no pass of its own for it.
// With dest (the last step), (h + acc / 2^s) * dsc goes to dest instead, for
// every entry (the exponential's final 2^-K). Memory bound (24 bytes a value:
// acc and h read and written): four consecutive values a thread, so that 48
// bytes are in flight per thread and loads are 16 bytes.
// (256 x 256 x 160: 220 us with one value a thread and the 64-bit conversion,
// 107 us so, the rate of a copy.)
__device__ __forceinline__ float finish_one(float hv, unsigned long long a, float inv)
{
    const long long q = (long long)a;
    return q != 0 ? hv + float_of(q) * inv : hv;
}

__global__ void __launch_bounds__(kDiffeoThreads)
    k_compose_finish(float *__restrict__ h, unsigned long long *__restrict__ acc, int64_t n,
                     const unsigned int *__restrict__ maxbits, unsigned int *__restrict__ maxnext,
                     float *__restrict__ dest, float dsc)
{
    const float inv = 1.0f / fixed_scale(*maxbits);  // a power of two: exact
    float m = 0.0f;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    auto put = [&](float v) {
        const float a = fabsf(v);
        m = a > m ? a : m;  // a NaN never wins
    };
    for (int64_t e = tid; e < n / 4; e += stride) {
        ulonglong2 *ap = reinterpret_cast<ulonglong2 *>(acc) + 2 * e;
        float4 *hp = reinterpret_cast<float4 *>(h) + e;
        const ulonglong2 a0 = ap[0], a1 = ap[1];
        float4 v = *hp;
        v.x = finish_one(v.x, a0.x, inv);
        v.y = finish_one(v.y, a0.y, inv);
        v.z = finish_one(v.z, a1.x, inv);
        v.w = finish_one(v.w, a1.y, inv);
        ap[0] = make_ulonglong2(0ull, 0ull);
        ap[1] = make_ulonglong2(0ull, 0ull);
        if (dest) {
            reinterpret_cast<float4 *>(dest)[e] =
                make_float4(v.x * dsc, v.y * dsc, v.z * dsc, v.w * dsc);
        } else {
            *hp = v;
            put(v.x);
            put(v.y);
            put(v.z);
            put(v.w);
        }
    }
    for (int64_t e = n / 4 * 4 + tid; e < n; e += stride) {
        const float v = finish_one(h[e], acc[e], inv);
        acc[e] = 0ull;
        if (dest) {
            dest[e] = v * dsc;
        } else {
            h[e] = v;
            put(v);
        }
    }
    if (!maxnext)
        return;
    // one atomic per block (the grid is a few blocks per SM)
    __shared__ float wm[kDiffeoThreads / 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0)
        wm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kDiffeoThreads / 32; ++w)
            m = fmaxf(m, wm[w]);
        atomicMax(maxnext, __float_as_uint(m));
    }
}

// fixed_of in its two halves, value hi 2^21 + lo. Sums of a few stay far inside
// 32 bits each.
struct Fix {
    int hi, lo;
};

// fixed_of of the pair (w.x g, w.y g) with packed operations.
__device__ __forceinline__ void fixed_pair(float2 w, float gs, Fix &a, Fix &b)
{
    constexpr float kMagic = 12582912.0f;
    constexpr int kBits = 0x4B400000;
    const float2 m = make_float2(kMagic, kMagic);
    const float2 p = __fmul2_rn(w, make_float2(gs, gs));
    const float2 t = __ffma2_rn(p, make_float2(0x1p-21f, 0x1p-21f), m);
    const float2 d = __fadd2_rn(t, make_float2(-kMagic, -kMagic));
    const float2 l = __fadd2_rn(__ffma2_rn(d, make_float2(-0x1p21f, -0x1p21f), p), m);
    a = {__float_as_int(t.x) - kBits, __float_as_int(l.x) - kBits};
    b = {__float_as_int(t.y) - kBits, __float_as_int(l.y) - kBits};
}

__device__ __forceinline__ void add_fix(unsigned long long *a, Fix q)
{
    atomicAdd(a, (unsigned long long)((long long)q.hi * 2097152ll + q.lo));
}

// The adjoint of one squaring of a 3D field in tiles like k_compose3's: local
// terms into h, the scatter into acc. Bound by the accumulator's atomics in L2
// (a microbenchmark: 20 G warp instructions of 32 consecutive 64-bit
// reductions per second). The contributions to the far z corners of a sample
// stay in registers as exact integers and join the next slice's sample when
// its cell is the next one, which halves them where the displacement is
// smooth; exchanging x corners between lanes as well (as a version before did)
// takes more instructions than it saves atomics. 256 x 256 x 160: 428 us a step
// with 64-bit conversions and x corners merged by shuffles, 358 us with
// fixed_of, 335 us so; 467 us with one atomic per corner. Sums are of exact
// integers, so the result is the same whatever merges.
__global__ void __launch_bounds__(kDiffeoThreads, 3)
    k_compose_adjoint3(Grid g, const float *__restrict__ u, const float *__restrict__ gin,
                       float *__restrict__ h, unsigned long long *__restrict__ acc,
                       const unsigned int *__restrict__ maxbits, int ntx, int nty, int zc, int lx)
{
    const float S = fixed_scale(*maxbits);
    const int tile = blockIdx.x, tx = tile % ntx, ty = (tile / ntx) % nty, tz = tile / (ntx * nty);
    const int x = (tx << lx) + (threadIdx.x & ((1 << lx) - 1)),
              y = ty * (kDiffeoThreads >> lx) + (threadIdx.x >> lx);
    if (x >= g.X || y >= g.Y)
        return;
    // 32 bits: pointers are advanced by nv, not indexed beyond it (2,458 us for the six steps at
    // 256 x 256 x 160 on a smooth field, 2,505 with 64)
    const int nv = (int)g.nv, sy = g.X, sz = g.X * g.Y;
    const float xlo = -(float)x, xhi = (float)(g.X - 1 - x);
    const float ylo = -(float)y, yhi = (float)(g.Y - 1 - y);
    const int z1 = min((tz + 1) * zc, g.Z);
    const float *u1 = u + nv, *u2 = u1 + nv;
    const float *g1 = gin + nv, *g2 = g1 + nv;
    float *h1 = h + nv, *h2 = h1 + nv;
    int v = (tz * zc * g.Y + y) * g.X + x;
    // contributions to the corners (y, x) at the far z of the last sample's cell
    Fix carry[3][4] = {};
    int cb = -1;  // their first node
#pragma unroll 1
    for (int z = tz * zc; z < z1; ++z, v += z < z1 ? sz : 0) {  // no index past the last slice
        const float a0 = __ldg(u + v), a1 = __ldg(u1 + v), a2 = __ldg(u2 + v);
        const float gv[3] = {__ldg(gin + v), __ldg(g1 + v), __ldg(g2 + v)};
        int cx, cy, cz;
        float fx, fy, fz;
        const bool inx = field_axis(x, a0, xlo, xhi, g.X, cx, fx);
        const bool iny = field_axis(y, a1, ylo, yhi, g.Y, cy, fy);
        const bool inz = field_axis(z, a2, -(float)z, (float)(g.Z - 1 - z), g.Z, cz, fz);
        const int base = (cz * g.Y + cy) * g.X + cx;
        const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
        float loc[3] = {gv[0], gv[1], gv[2]};
        const float2 m1 = make_float2(-1.0f, -1.0f), fx2 = make_float2(fx, fx),
                     fy2 = make_float2(fy, fy);
        // derivative of the interpolant of each component at the sample, the
        // corners of the two z faces as packed pairs
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float *p = (i == 0 ? u : i == 1 ? u1 : u2) + base;
            const float *q = p + sz;
            const float2 c00 = make_float2(__ldg(p), __ldg(q));
            const float2 c01 = make_float2(__ldg(p + 1), __ldg(q + 1));
            const float2 c10 = make_float2(__ldg(p + sy), __ldg(q + sy));
            const float2 c11 = make_float2(__ldg(p + sy + 1), __ldg(q + sy + 1));
            const float2 d0 = __ffma2_rn(c00, m1, c01), d1 = __ffma2_rn(c10, m1, c11);
            const float2 dx = __ffma2_rn(fy2, __ffma2_rn(d0, m1, d1), d0);
            const float2 l0 = __ffma2_rn(fx2, d0, c00), l1 = __ffma2_rn(fx2, d1, c10);
            const float2 dy = __ffma2_rn(l0, m1, l1), b = __ffma2_rn(fy2, dy, l0);
            if (inx)
                loc[0] = fmaf(fmaf(fz, dx.y - dx.x, dx.x), gv[i], loc[0]);
            if (iny)
                loc[1] = fmaf(fmaf(fz, dy.y - dy.x, dy.x), gv[i], loc[1]);
            if (inz)
                loc[2] = fmaf(b.y - b.x, gv[i], loc[2]);
        }
        h[v] = loc[0];
        h1[v] = loc[1];
        h2[v] = loc[2];
        const float2 wy0 = make_float2(gx * gy, fx * gy), wy1 = make_float2(gx * fy, fx * fy);
        const float2 gz2 = make_float2(gz, gz), fz2 = make_float2(fz, fz);
        const float2 w00 = __fmul2_rn(wy0, gz2), w10 = __fmul2_rn(wy1, gz2);
        const float2 w01 = __fmul2_rn(wy0, fz2), w11 = __fmul2_rn(wy1, fz2);
        const bool on = cb == base;
        if (!on && cb >= 0) {
            unsigned long long *ap = acc + cb;
#pragma unroll
            for (int i = 0; i < 3; ++i, ap += nv) {
                add_fix(ap, carry[i][0]);
                add_fix(ap + 1, carry[i][1]);
                add_fix(ap + sy, carry[i][2]);
                add_fix(ap + sy + 1, carry[i][3]);
            }
        }
        unsigned long long *ap = acc + base;
#pragma unroll
        for (int i = 0; i < 3; ++i, ap += nv) {
            float gs = gv[i] * S;
            if (!(fabsf(gs) <= 0x1p42f)) {  // an infinity or a NaN
                scatter_far<3>(ap, sy, sz, fx, fy, fz, gv[i], S);
                gs = 0.0f;
            }
            Fix q[4];
            fixed_pair(w00, gs, q[0], q[1]);
            fixed_pair(w10, gs, q[2], q[3]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                q[k].hi += on ? carry[i][k].hi : 0;
                q[k].lo += on ? carry[i][k].lo : 0;
            }
            fixed_pair(w01, gs, carry[i][0], carry[i][1]);
            fixed_pair(w11, gs, carry[i][2], carry[i][3]);
            add_fix(ap, q[0]);
            add_fix(ap + 1, q[1]);
            add_fix(ap + sy, q[2]);
            add_fix(ap + sy + 1, q[3]);
        }
        cb = base + sz;
    }
    unsigned long long *ap = acc + cb;
#pragma unroll
    for (int i = 0; i < 3; ++i, ap += nv) {
        add_fix(ap, carry[i][0]);
        add_fix(ap + 1, carry[i][1]);
        add_fix(ap + sy, carry[i][2]);
        add_fix(ap + sy + 1, carry[i][3]);
    }
}

// Tiles of the marching kernels: 32 x 8 columns a block (march_lx) and zc slices, 8 of
// them or fewer while that leaves less than eight blocks per SM.
struct Tiles {
    int ntx, nty, zc, blocks, lx;
};

// scatter: up to 32 voxels a row is one tile, whose lanes' reductions then lie together
// (64 x 64 x 20: 98 us in rows of 32, 109 in rows of 8).
Tiles tiles_of(const Grid &g, bool scatter)
{
    Tiles t;
    t.lx = march_lx(g.X);
    if (scatter && g.X <= 32)
        for (t.lx = 2; (1 << t.lx) < g.X;)
            ++t.lx;
    t.ntx = (g.X + (1 << t.lx) - 1) >> t.lx;
    const int ty = kDiffeoThreads >> t.lx;
    t.nty = (g.Y + ty - 1) / ty;
    t.zc = 8;
    while (t.zc > 1 &&
           (int64_t)t.ntx * t.nty * ((g.Z + t.zc - 1) / t.zc) < 8 * (int64_t)device_sms())
        t.zc /= 2;
    t.blocks = t.ntx * t.nty * ((g.Z + t.zc - 1) / t.zc);
    return t;
}

template <int D>
cudaError_t exp_run(const Grid &g, int K, const float *v, float *u, float *traj, float *tmp,
                    cudaStream_t s)
{
    const int64_t n = (int64_t)D * g.nv;
    const float sc = ldexpf(1.0f, -K);
    // u_0 -> traj[0] (or tmp); each squaring writes the next buffer
    ProfScope ps(s, "k_exp");
    if (K == 0) {
        k_scale<<<blocks_for(n), kDiffeoThreads, 0, s>>>(v, u, sc, n);
        return cudaGetLastError();
    }
    // the first squaring reads v scaled by 2^-K (and stores u_0 = v 2^-K in
    // the trajectory); each squaring writes the next buffer. If v overlaps a
    // buffer the squarings write, u_0 is formed in a pass of its own first.
    auto overlaps = [&](const float *b, int64_t cnt) {
        return b && v < b + cnt && b < v + n;
    };
    const float *cur = v;
    float scale0 = sc;
    cudaError_t e = cudaSuccess;
    if (overlaps(u, n) || overlaps(tmp, n) || overlaps(traj, (int64_t)K * n)) {
        float *u0 = traj ? traj : ((K - 1) % 2 == 0 ? tmp : u);
        if (K == 1 && !traj)
            u0 = tmp;
        k_scale<<<blocks_for(n), kDiffeoThreads, 0, s>>>(v, u0, sc, n);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return e;
        cur = u0;
        scale0 = 1.0f;
    }
    for (int k = 0; k < K && e == cudaSuccess; ++k) {
        float *nxt;
        if (k == K - 1)
            nxt = u;
        else if (traj)
            nxt = traj + (int64_t)(k + 1) * n;
        else
            nxt = ((K - 1 - k) % 2 == 0) ? u : tmp;
        const bool scaled = k == 0 && scale0 != 1.0f;
        float *u0 = scaled ? traj : nullptr;
        if constexpr (D == 3) {
            const Tiles t = tiles_of(g, false);
            if (scaled)
                k_compose3<true><<<t.blocks, kDiffeoThreads, 0, s>>>(g, cur, nxt, scale0, u0,
                                                                     t.ntx, t.nty, t.zc, t.lx);
            else
                k_compose3<false><<<t.blocks, kDiffeoThreads, 0, s>>>(g, cur, nxt, 1.0f, u0,
                                                                      t.ntx, t.nty, t.zc, t.lx);
        } else {
            if (scaled)
                k_compose2<true><<<blocks_for(g.nv), kDiffeoThreads, 0, s>>>(g, cur, nxt, scale0,
                                                                             u0);
            else
                k_compose2<false><<<blocks_for(g.nv), kDiffeoThreads, 0, s>>>(g, cur, nxt, 1.0f,
                                                                              u0);
        }
        e = cudaGetLastError();
        cur = nxt;
    }
    return e;
}

template <int D>
cudaError_t exp_adjoint_run(const Grid &g, int K, const float *traj, const float *gu, float *gv,
                            char *ws, const unsigned int *gmax, cudaStream_t s)
{
    const int64_t n = (int64_t)D * g.nv;
    unsigned long long *acc = (unsigned long long *)ws;
    float *b0 = (float *)(ws + ((size_t)n * 8 + 255) / 256 * 256);
    float *b1 = b0 + ((size_t)n * 4 + 255) / 256 * 64;
    unsigned int *mx = (unsigned int *)(b1 + ((size_t)n * 4 + 255) / 256 * 64);
    ProfScope ps(s, "k_exp_adjoint");
    cudaError_t e = cudaMemsetAsync(acc, 0, (size_t)n * 8, s);
    const float *gin = gu;
    float *out = b0;
    // mx[0], mx[1]: the largest |g| of a step's input; the first from the caller
    // or from a pass of its own, the others from the previous step's finish
    if (e == cudaSuccess && K > 0 && !gmax) {
        e = cudaMemsetAsync(mx, 0, sizeof(unsigned int), s);
        if (e == cudaSuccess) {
            k_absmax<<<blocks_for(n) < 4 * device_sms() ? blocks_for(n) : 4 * device_sms(),
                       kDiffeoThreads, 0, s>>>(gin, n, mx);
            e = cudaGetLastError();
        }
    }
    for (int k = K - 1, j = 0; k >= 0 && e == cudaSuccess; --k, j ^= 1) {
        const float *u = traj + (int64_t)k * n;
        const unsigned int *mcur = k == K - 1 && gmax ? gmax : mx + j;
        unsigned int *mnext = k > 0 ? mx + (j ^ 1) : nullptr;
        if constexpr (D == 3) {
            const Tiles t = tiles_of(g, true);
            k_compose_adjoint3<<<t.blocks, kDiffeoThreads, 0, s>>>(g, u, gin, out, acc, mcur,
                                                                   t.ntx, t.nty, t.zc, t.lx);
        } else {
            k_compose_adjoint2<<<blocks_for(g.nv), kDiffeoThreads, 0, s>>>(g, u, gin, out, acc,
                                                                           mcur);
        }
        if (mnext && (e = cudaMemsetAsync(mnext, 0, sizeof(unsigned int), s)) != cudaSuccess)
            break;
        // the last step writes (its result) * 2^-K to gv directly
        const int fb = std::min(blocks_for((n + 3) / 4), 16 * device_sms());
        k_compose_finish<<<fb, kDiffeoThreads, 0, s>>>(out, acc, n, mcur, mnext,
                                                       k == 0 ? gv : nullptr, ldexpf(1.0f, -K));
        e = cudaGetLastError();
        gin = out;
        out = (out == b0) ? b1 : b0;
    }
    if (K > 0)
        return e;
    if (e != cudaSuccess)
        return e;
    k_scale<<<blocks_for(n), kDiffeoThreads, 0, s>>>(gin, gv, ldexpf(1.0f, -K), n);
    return cudaGetLastError();
}

}  // namespace

size_t exp_adjoint_ws(const Grid &g)
{
    const size_t n = (size_t)g.ndim * g.nv;
    return (n * 8 + 255) / 256 * 256 + 2 * ((n * 4 + 255) / 256 * 256) + 256;
}

cudaError_t launch_exp(const Grid &g, int K, const float *v, float *u, float *traj, float *tmp,
                       cudaStream_t s)
{
    return g.ndim == 3 ? exp_run<3>(g, K, v, u, traj, tmp, s) : exp_run<2>(g, K, v, u, traj, tmp, s);
}

cudaError_t launch_exp_adjoint(const Grid &g, int K, const float *traj, const float *gu, float *gv,
                               void *ws, const unsigned int *gmax, cudaStream_t s)
{
    return g.ndim == 3 ? exp_adjoint_run<3>(g, K, traj, gu, gv, (char *)ws, gmax, s)
                       : exp_adjoint_run<2>(g, K, traj, gu, gv, (char *)ws, gmax, s);
}

}  // namespace airgb
