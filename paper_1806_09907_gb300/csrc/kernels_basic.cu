// Step kernels of the unfused path: A1 B-spline expansion, A6 its adjoint,
// A2 warp, A5 warp adjoint, A4 diffusion regulariser (voxel form).
#include <algorithm>

#include "launch.h"

namespace airgb {

namespace {

constexpr int kDispTX = 128;  // x extent of a displacement tile (threads); 32 for rows up to 32
constexpr int kDispTY = 8;    // rows per tile

// Control columns a tile of n voxels can touch.
constexpr int disp_span(int n, int delta) { return (n - 1) / delta + 5; }

// A1: u_i(x) = sum_j c_{i,j} prod_k w. One CTA = one z slice, 8 rows, 128
// columns. Separable: a thread per touched control column contracts along z
// and y together, keeping the four z-contracted points that the row needs in
// registers and forming the next one every delta rows, into a row buffer in
// shared memory; then 4 x-taps per voxel. Bound by instructions: 63.6 us at
// 256 x 256 x 160, spacing 6, with a z and a y phase over elements whose
// indices were divided out and buffers sized for spacing 1 (6 CTAs per SM),
// 44.8 us so; writing u takes 18.5 us. (96 registers; held to 64, 46.6 us, to 40,
// 61.9 us.)
template <int D, int TX>
__global__ void __launch_bounds__(TX)
    k_displacement(Grid g, const __grid_constant__ Lattice L, const float *__restrict__ c,
                   float *__restrict__ u)
{
    extern __shared__ float disp_smem[];  // [D][kDispTY][njx]
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * kDispTY, z = blockIdx.z;
    const int delta = L.delta;
    const int jx0 = x0 / delta, jy0 = y0 / delta;
    const int xl = min(x0 + TX, g.X) - 1;
    const int njx = xl / delta + 4 - jx0;
    const int rows = min(kDispTY, g.Y - y0);
    const int qz = z / delta, pz = z - qz * delta, py0 = y0 - jy0 * delta;
    const float z0 = L.w[pz][0], z1 = L.w[pz][1], z2 = L.w[pz][2], z3 = L.w[pz][3];
    const int64_t nxy = (int64_t)L.nx * L.ny;
    for (int col = threadIdx.x; col < D * njx; col += TX) {
        const int i = D == 3 ? (col >= njx) + (col >= 2 * njx) : (col >= njx);
        const float *src = c + i * L.nc + (D == 3 ? qz * nxy : 0) + (int64_t)jy0 * L.nx + jx0 +
                           (col - i * njx);
        auto point = [&](int jy) {
            const float *p = src + jy * L.nx;
            if (D == 2)
                return __ldg(p);
            float acc = fmaf(z0, __ldg(p), 0.0f);
            acc = fmaf(z1, __ldg(p + nxy), acc);
            acc = fmaf(z2, __ldg(p + 2 * nxy), acc);
            return fmaf(z3, __ldg(p + 3 * nxy), acc);
        };
        float t0 = point(0), t1 = point(1), t2 = point(2), t3 = point(3);
        float *d = disp_smem + i * kDispTY * njx + (col - i * njx);
        int p = py0, jy = 3;
#pragma unroll
        for (int yr = 0; yr < kDispTY; ++yr) {
            if (yr >= rows)
                break;
            if (p == delta) {  // the same row for every column: uniform
                p = 0;
                t0 = t1, t1 = t2, t2 = t3;
                t3 = point(++jy);
            }
            float acc = fmaf(L.w[p][0], t0, 0.0f);
            acc = fmaf(L.w[p][1], t1, acc);
            acc = fmaf(L.w[p][2], t2, acc);
            d[yr * njx] = fmaf(L.w[p][3], t3, acc);
            ++p;
        }
    }
    __syncthreads();
    const int x = x0 + threadIdx.x;
    if (x >= g.X)
        return;
    const int qx = x / delta, px = x - qx * delta;
    const float w0 = L.w[px][0], w1 = L.w[px][1], w2 = L.w[px][2], w3 = L.w[px][3];
    const float *t = disp_smem + (qx - jx0);
    float *o = u + ((int64_t)z * g.Y + y0) * g.X + x;
#pragma unroll
    for (int yr = 0; yr < kDispTY; ++yr) {
        if (yr >= rows)
            break;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const float *r = t + (i * kDispTY + yr) * njx;
            float acc = w0 * r[0];
            acc = fmaf(w1, r[1], acc);
            acc = fmaf(w2, r[2], acc);
            acc = fmaf(w3, r[3], acc);
            o[(int64_t)i * g.nv] = acc;
        }
        o += g.X;
    }
}

// A6 along x and y for one z slice of one component and a band of bj control
// rows: out[o][jy][jx] = sum_y w(y, jy) sum_x w(x, jx) in[o][y][x]. A warp
// walks the rows of the band's support: a row comes in coalesced loads (the
// next one's are in flight meanwhile), is contracted along x in two steps (each
// cell's four weighted sums of its delta voxels, then per control point the
// sum over the up to four cells it supports) and kept; then the kept rows are
// contracted along y. A row's buffers belong to its warp, so only the y step
// waits for the block, and lanes stride along x, so no index is divided; a cell's
// voxels lie an odd number of words from the next cell's, so that lanes read different
// banks. Fixed order, no atomics. 256 x 256 x 160, spacing 6: 168 us for x and 31 us for y
// with one thread per output reading 4 delta values delta apart, 70 us so;
// reading the field takes 18.5 us.
constexpr int kTransThreads = 256;
constexpr int kTransWarps = kTransThreads / 32;
constexpr int kTransWidth = 320;  // voxels of a staged row at most

struct TransPlan {
    int jt, bj;         // control columns and rows of a block
    int nxt, nbands;    // blocks per slice along x and y
    int cells, pitch;   // staged cells of a row at most, and words from one to the next
    size_t smem;
};

// A block's columns: as many as need up to kTransWidth voxels of support and 48 KB (a whole row of
// most volumes); its rows: 16, so that 3/16 of the rows are read twice, or 8 or 4 when that leaves
// fewer than four blocks per SM of a 152-SM GB300. Both evened out over the blocks.
TransPlan trans_plan(const Grid &g, const Lattice &L)
{
    TransPlan t;
    const int ncx = (g.X - 1) / L.delta + 1;
    t.pitch = L.delta | 1;
    auto bytes = [&](int bj) {
        return 4 * (kMaxDelta * 4 +
                    (size_t)kTransWarps * (t.cells * t.pitch + (t.jt + 3) * 4) +
                    (size_t)(bj + 3) * L.delta * t.jt);
    };
    const int most = std::max(1, std::min(L.nx, kTransWidth));  // columns of a first guess
    t.nxt = (L.nx + most - 1) / most;
    do {
        t.jt = (L.nx + t.nxt - 1) / t.nxt;
        t.cells = std::min(ncx, t.jt + 3);
    } while ((std::min(t.cells * L.delta, g.X) > kTransWidth || bytes(16) > 48 * 1024) && ++t.nxt);
    t.nxt = (L.nx + t.jt - 1) / t.jt;
    for (t.bj = 16; t.bj > 4; t.bj /= 2)
        if ((int64_t)g.ndim * g.Z * t.nxt * ((L.ny + t.bj - 1) / t.bj) >= 4 * 152)
            break;
    t.nbands = (L.ny + t.bj - 1) / t.bj;
    t.bj = (L.ny + t.nbands - 1) / t.nbands;
    t.smem = bytes(t.bj);
    return t;
}

__global__ void __launch_bounds__(kTransThreads)
    k_transpose_xy(const float *__restrict__ in, float *__restrict__ out, int X, int Y,
                   const __grid_constant__ TransPlan t, const __grid_constant__ Lattice L)
{
    extern __shared__ __align__(16) float trans_sm[];
    const int delta = L.delta, jt = t.jt, cells = jt + 3, pitch = t.pitch;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4 *w4 = reinterpret_cast<float4 *>(trans_sm);   // [delta] weights of a phase
    float *raw = trans_sm + kMaxDelta * 4 + warp * t.cells * pitch;  // [staged cells][pitch]
    float *sums = trans_sm + kMaxDelta * 4 + kTransWarps * t.cells * pitch +
                  warp * cells * 4;  // [4][cells]
    float *t1 = trans_sm + kMaxDelta * 4 + kTransWarps * (t.cells * pitch + cells * 4);  // [rows][jt]
    if (threadIdx.x < delta)
        w4[threadIdx.x] = make_float4(L.w[threadIdx.x][0], L.w[threadIdx.x][1],
                                      L.w[threadIdx.x][2], L.w[threadIdx.x][3]);
    const int tile = blockIdx.x, tx = tile % t.nxt, band = (tile / t.nxt) % t.nbands;
    const int64_t o = tile / (t.nxt * t.nbands);
    const int jx0 = tx * jt, jy0 = band * t.bj;
    const int nj = min(jt, L.nx - jx0), nb = min(t.bj, L.ny - jy0);
    // the tile's cells inside the grid, [c0, c0 + nc), cell 0 of the tile being jx0 - 3
    const int c0 = max(jx0 - 3, 0), nc = min(jx0 + nj, (X - 1) / delta + 1) - c0;
    const int skip = c0 - (jx0 - 3);
    const int x0 = c0 * delta, width = min(nc * delta, X - x0);
    // rows of the band's support, those inside the grid
    const int y0 = (jy0 - 3) * delta, rows = (nb + 3) * delta;
    const int r0 = max(0, -y0), r1 = min(rows, Y - y0);
    const float *src = in + o * Y * X + x0;
    constexpr int PER = kTransWidth / 32;
    int place[PER];  // of this lane's voxels in raw
    const int spare = pitch - delta, inv = 65536 / delta + 1;  // i inv / 65536 = i / delta, i < 320
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = lane + 32 * k;
        place[k] = i + spare * (i * inv >> 16);
    }
    float next[PER];
    auto fetch = [&](int r) {
#pragma unroll
        for (int k = 0; k < PER; ++k)
            next[k] = r < r1 && lane + 32 * k < width
                          ? __ldg(src + (int64_t)(y0 + r) * X + lane + 32 * k) : 0.0f;
    };
    fetch(r0 + warp);
    // zero where no row or cell of the grid writes: cells before and beyond the grid's, the last
    // one's voxels beyond it, and rows
    if (skip > 0 || skip + nc < cells)
        for (int e = lane; e < cells * 4; e += 32)
            sums[e] = 0.0f;
    if (lane < nc * delta - width)
        raw[(nc - 1) * pitch + delta - 1 - lane] = 0.0f;
    for (int e = threadIdx.x; e < r0 * jt; e += kTransThreads)
        t1[e] = 0.0f;
    for (int e = r1 * jt + threadIdx.x; e < rows * jt; e += kTransThreads)
        t1[e] = 0.0f;
    __syncthreads();
    for (int r = r0 + warp; r < r1; r += kTransWarps) {
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (lane + 32 * k < width)
                raw[place[k]] = next[k];
        __syncwarp();
        fetch(r + kTransWarps);
        for (int e = lane; e < nc; e += 32) {
            const float *v = raw + e * pitch;
            float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
#pragma unroll 4
            for (int k = 0; k < delta; ++k) {
                const float a = v[k];
                const float4 w = w4[k];
                s0 = fmaf(w.x, a, s0);
                s1 = fmaf(w.y, a, s1);
                s2 = fmaf(w.z, a, s2);
                s3 = fmaf(w.w, a, s3);
            }
            float *d = sums + skip + e;
            d[0] = s0;
            d[cells] = s1;
            d[2 * cells] = s2;
            d[3 * cells] = s3;
        }
        __syncwarp();
        // control point j is fed by the cells j - 3 .. j (weights 3 .. 0)
        for (int j = lane; j < nj; j += 32) {
            const float *d = sums + j;
            t1[r * jt + j] =
                ((d[3 * cells] + d[2 * cells + 1]) + d[cells + 2]) + d[3];
        }
    }
    __syncthreads();
    for (int jb = warp; jb < nb; jb += kTransWarps)
        for (int j = lane; j < nj; j += 32) {
            const float *v = t1 + jb * delta * jt + j;
            float s3 = 0.0f, s2 = 0.0f, s1 = 0.0f, s0 = 0.0f;
#pragma unroll 4
            for (int k = 0; k < delta; ++k, v += jt) {
                const float4 w = w4[k];
                s3 = fmaf(w.w, v[0], s3);
                s2 = fmaf(w.z, v[delta * jt], s2);
                s1 = fmaf(w.y, v[2 * delta * jt], s1);
                s0 = fmaf(w.x, v[3 * delta * jt], s0);
            }
            out[(o * L.ny + jy0 + jb) * L.nx + jx0 + j] = ((s3 + s2) + s1) + s0;
        }
}

// A6 along one axis: in[o][len][inner] -> out[o][n][inner], one thread per output,
// ascending positions.
// I: the outputs' index type, 32 bits where they allow it.
template <typename I>
__global__ void __launch_bounds__(kTransThreads)
    k_transpose_axis(const float *__restrict__ in, float *__restrict__ out, I total, int len,
                     int n, I inner, const __grid_constant__ Lattice L)
{
    const int delta = L.delta;
    for (I e = blockIdx.x * (I)blockDim.x + threadIdx.x; e < total; e += (I)gridDim.x * blockDim.x) {
        const I oj = e / inner, k = e - oj * inner, o = oj / n;
        const int j = (int)(oj - o * n);
        const float *src = in + (int64_t)o * len * inner + k;
        float acc = 0.0f;
#pragma unroll
        for (int a = 3; a >= 0; --a) {
            const int t0 = (j - a) * delta;
            if (t0 < 0)
                continue;
            const int m = min(delta, len - t0);
            const float *p = src + (int64_t)t0 * inner;
#pragma unroll 4
            for (int q = 0; q < m; ++q)
                acc = fmaf(L.w[q][a], __ldg(p + (int64_t)q * inner), acc);
        }
        out[e] = acc;
    }
}

// ---- marching tiles ---------------------------------------------------------
// The point-wise kernels take 32 x 8 columns a block (a warp per row; narrower rows where
// they use more lanes, march_lx) and march
// through zc slices, so that a column's index arithmetic is done once and its
// z neighbours stay in registers. Tiles beyond the grid's blocks follow in
// order (tile += gridDim).
constexpr int kTileX = 32, kTileY = 8;  // columns of a block: kTileX * kTileY

struct March {
    int ntx, nty, ntiles, zc, lx;  // lx: log2 of a tile's columns in x
};

// Slices of a column: 8, fewer while that leaves less than eight blocks per SM.
March march_plan(const Grid &g)
{
    March m;
    m.lx = march_lx(g.X);
    m.ntx = (g.X + (1 << m.lx) - 1) >> m.lx;
    const int ty = kTileX * kTileY >> m.lx;
    m.nty = (g.Y + ty - 1) / ty;
    m.zc = 8;
    while (m.zc > 1 &&
           (int64_t)m.ntx * m.nty * ((g.Z + m.zc - 1) / m.zc) < 8 * (int64_t)device_sms())
        m.zc /= 2;
    m.ntiles = m.ntx * m.nty * ((g.Z + m.zc - 1) / m.zc);
    return m;
}

struct Column {
    int x, y, z0, z1;
    bool on;
};

__device__ __forceinline__ Column march_column(const Grid &g, const March &m, int tile)
{
    Column c;
    c.x = (tile % m.ntx << m.lx) + (threadIdx.x & ((1 << m.lx) - 1));
    c.y = tile / m.ntx % m.nty * (kTileX * kTileY >> m.lx) + (threadIdx.x >> m.lx);
    c.z0 = tile / (m.ntx * m.nty) * m.zc;
    c.z1 = min(c.z0 + m.zc, g.Z);
    c.on = c.x < g.X && c.y < g.Y;
    return c;
}

// Sample at voxel (x, y, z) displaced by (ux, uy, uz): inside, and the
// interpolant there (whatever the cell holds when outside). All axes are
// shorter than 2^22 (axis_cell).
template <int D>
__device__ __forceinline__ bool sample_at(const Grid &g, const float *__restrict__ M, int x, int y,
                                          int z, float ux, float uy, float uz, Interp &ip)
{
    AxisSample sx, sy, sz;
    bool in = axis_cell(x, ux, -(float)x, (float)(g.X - 1 - x), g.X, sx.cell, sx.f);
    in &= axis_cell(y, uy, -(float)y, (float)(g.Y - 1 - y), g.Y, sy.cell, sy.f);
    if (D == 3)
        in &= axis_cell(z, uz, -(float)z, (float)(g.Z - 1 - z), g.Z, sz.cell, sz.f);
    ip = D == 3 ? trilinear(M, g.X, g.Y, g.Z, sx, sy, sz) : bilinear(M, g.X, g.Y, sx, sy);
    return in;
}

// A2: backward warp with mask. Bound by instructions and gathers, not memory
// (256 x 256 x 160: 74 us with 64-bit index divisions and branches per voxel,
// 53 us so; its bytes take 32 us).
template <int D>
__global__ void __launch_bounds__(kTileX *kTileY)
    k_warp(Grid g, March mp, const float *__restrict__ M, const float *__restrict__ u,
           float *__restrict__ W, uint8_t *__restrict__ mask)
{
    const Column c = march_column(g, mp, blockIdx.x);
    if (!c.on)
        return;
    const int sz = g.X * g.Y, v0 = (c.z0 * g.Y + c.y) * g.X + c.x;
#pragma unroll 2
    for (int z = c.z0; z < c.z1; ++z) {
        const int v = v0 + (z - c.z0) * sz;
        Interp ip;
        const bool in = sample_at<D>(g, M, c.x, c.y, z, __ldg(u + v), __ldg(u + g.nv + v),
                                     D == 3 ? __ldg(u + 2 * (int64_t)g.nv + v) : 0.0f, ip);
        W[v] = in ? ip.v : 0.0f;
        mask[v] = in ? 1 : 0;
    }
}

// A5: grad_disp[k] = mask * grad_warped * dM~/dy_k (+ grad_disp if accumulate).
template <int D>
__global__ void __launch_bounds__(kTileX *kTileY)
    k_warp_adjoint(Grid g, March mp, const float *__restrict__ M, const float *__restrict__ u,
                   const uint8_t *__restrict__ mask, const float *__restrict__ gw,
                   float *__restrict__ gu, int accumulate)
{
    const Column c = march_column(g, mp, blockIdx.x);
    if (!c.on)
        return;
    const int sz = g.X * g.Y;
    unsigned v = (unsigned)((c.z0 * g.Y + c.y) * g.X + c.x);  // wraps after the last slice only
    for (int z = c.z0; z < c.z1; ++z, v += sz) {
        float gx = 0.0f, gy = 0.0f, gz = 0.0f;
        const float gwv = __ldg(gw + v);
        if (__ldg(mask + v) && gwv != 0.0f) {
            Interp ip;
            if (sample_at<D>(g, M, c.x, c.y, z, __ldg(u + v), __ldg(u + g.nv + v),
                             D == 3 ? __ldg(u + 2 * (int64_t)g.nv + v) : 0.0f, ip)) {
                gx = gwv * ip.gx;
                gy = gwv * ip.gy;
                gz = gwv * ip.gz;
            }
        }
        if (accumulate) {
            gu[v] += gx;
            gu[g.nv + v] += gy;
            if (D == 3)
                gu[2 * g.nv + v] += gz;
        } else {
            gu[v] = gx;
            gu[g.nv + v] = gy;
            if (D == 3)
                gu[2 * g.nv + v] = gz;
        }
    }
}

// A4: R = (1/|X|) sum_i sum_k sum_{x_k < N_k-1} (u_i(x+e_k) - u_i(x))^2 and
// grad = gscale * its derivative (+ the adjoint of the warp with
// GW != GW_NONE: mask * dS/dW * dM~/dy, dS/dW formed from the similarity's
// scalars without a pass of its own). A column's z neighbours are carried in
// registers and its x and y neighbours come from L1; one FP64 partial per
// block. 256 x 256 x 160: 139 us (one voxel a thread, an FP64 block reduction
// per 256 voxels) + 135 us (warp adjoint, reading and writing the gradient
// again) + 19 us (the scaling of dS/dW), 156 us so; its bytes take 51 us.
// maxbits (nullable): the largest |grad| as the bits of a float (a NaN never
// wins), for al_exp_field_adjoint's fixed point.
// The thread's part of R |X| as an FP64 sum, for terms that a Sum2 does not take.
template <int D>
__device__ __forceinline__ double regulariser_wide(const Grid &g, const March &mp,
                                                const float *__restrict__ u)
{
    double total = 0.0;
    for (int tile = blockIdx.x; tile < mp.ntiles; tile += gridDim.x) {
        const Column c = march_column(g, mp, tile);
        if (!c.on)
            continue;
        unsigned v = (unsigned)((c.z0 * g.Y + c.y) * g.X + c.x);
        for (int z = c.z0; z < c.z1; ++z, v += g.X * g.Y) {
            float sum = 0.0f;
            for (int i = 0; i < D; ++i) {
                const float *ui = u + i * g.nv + v;
                const float m = __ldg(ui);
                const float dx = c.x + 1 < g.X ? __ldg(ui + 1) - m : 0.0f;
                const float dy = c.y + 1 < g.Y ? __ldg(ui + g.X) - m : 0.0f;
                const float dz =
                    D == 3 && z + 1 < g.Z ? __ldg(ui + (int64_t)g.X * g.Y) - m : 0.0f;
                sum = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, sum)));
            }
            total += (double)sum;
        }
    }
    return total;
}

template <int D, int GW>
__global__ void __launch_bounds__(kTileX *kTileY, 5)
    k_regulariser(const __grid_constant__ Grid g, const __grid_constant__ March mp,
                  const float *__restrict__ u, float gscale, float *__restrict__ gu,
                  double *__restrict__ partials, AdjointArgs a,
                  unsigned int *__restrict__ maxbits)
{
    __shared__ double red[kTileX * kTileY / 32];
    __shared__ float wm[kTileX * kTileY / 32];
    Sum2 total[1];
    float big = 0.0f;
    float k0 = 0.0f, k1 = 0.0f, k2 = 0.0f, k3 = 0.0f;
    if (GW == GW_MSE || GW == GW_SCALED)
        k0 = (float)a.scal[0];
    if (GW == GW_NCC)
        k0 = (float)a.scal[0], k1 = (float)a.scal[1], k2 = (float)a.scal[3], k3 = (float)a.scal[4];
    const int sy = g.X, sz = g.X * g.Y;
    const int64_t nv = g.nv;
    for (int tile = blockIdx.x; tile < mp.ntiles; tile += gridDim.x) {
        const Column c = march_column(g, mp, tile);
        if (!c.on)
            continue;
        unsigned v = (unsigned)((c.z0 * g.Y + c.y) * g.X + c.x);
        float below[D], cur[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            cur[i] = __ldg(u + i * nv + v);
            below[i] = D == 3 && c.z0 > 0 ? __ldg(u + i * nv + v - sz) : 0.0f;
        }
        // neighbours beyond the grid are read at the voxel itself and dropped
        const bool xu = c.x + 1 < g.X, xd = c.x > 0, yu = c.y + 1 < g.Y, yd = c.y > 0;
        const int oxu = xu ? 1 : 0, oxd = xd ? -1 : 0, oyu = yu ? sy : 0, oyd = yd ? -sy : 0;
#pragma unroll 1
        for (int z = c.z0; z < c.z1; ++z, v += sz) {
            const bool zu = D == 3 && z + 1 < g.Z, zd = D == 3 && z > 0;
            float sum = 0.0f, lap[D], next[D], wxu[D], wxd[D], wyu[D], wyd[D];
#pragma unroll
            for (int i = 0; i < D; ++i) {
                const float *ui = u + i * nv;
                next[i] = D == 3 ? __ldg(ui + (unsigned)(zu ? v + sz : v)) : 0.0f;
                wxu[i] = __ldg(ui + (unsigned)(v + oxu));
                wxd[i] = __ldg(ui + (unsigned)(v + oxd));
                wyu[i] = __ldg(ui + (unsigned)(v + oyu));
                wyd[i] = __ldg(ui + (unsigned)(v + oyd));
            }
#pragma unroll
            for (int i = 0; i < D; ++i) {
                const float m = cur[i];
                float l = 0.0f;  // sum_k (u(x) - u(x-e_k)) - (u(x+e_k) - u(x))
                auto up = [&](bool ok, float w) {
                    const float d = ok ? w - m : 0.0f;
                    sum = fmaf(d, d, sum);
                    l -= d;
                };
                up(xu, wxu[i]);
                l += xd ? m - wxd[i] : 0.0f;
                up(yu, wyu[i]);
                l += yd ? m - wyd[i] : 0.0f;
                if (D == 3) {
                    up(zu, next[i]);
                    l += zd ? m - below[i] : 0.0f;
                }
                lap[i] = l;
            }
            total[0].add(sum);
            if (gu) {
                float gx = 0.0f, gy = 0.0f, gz = 0.0f;
                if (GW != GW_NONE) {
                    const bool on = __ldg(a.mask + v) != 0;
                    float gwv = 0.0f;
                    if (on) {
                        if (GW == GW_MSE)
                            gwv = k0 * (__ldg(a.W + v) - __ldg(a.F + v));
                        else if (GW == GW_NCC)
                            gwv = fmaf(k2, __ldg(a.F + v) - k0, k3 * (__ldg(a.W + v) - k1));
                        else
                            gwv = __fmul_rn(__ldg(a.gw + v), k0);
                    }
                    if (on && gwv != 0.0f) {
                        Interp ip;
                        if (sample_at<D>(g, a.M, c.x, c.y, z, cur[0], cur[1],
                                         D == 3 ? cur[D - 1] : 0.0f, ip)) {
                            gx = __fmul_rn(gwv, ip.gx);
                            gy = __fmul_rn(gwv, ip.gy);
                            gz = __fmul_rn(gwv, ip.gz);
                        }
                    }
                }
                const float add[3] = {gx, gy, gz};
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    const float r = __fadd_rn(__fmul_rn(gscale, lap[i]), add[i]);
                    gu[i * nv + v] = r;
                    const float ar = fabsf(r);
                    big = ar > big ? ar : big;
                }
            }
#pragma unroll
            for (int i = 0; i < D; ++i) {
                below[i] = cur[i];
                cur[i] = next[i];
            }
        }
    }
    double R[1];
    const bool wide = !(total[0].s <= kSum2Most);  // terms are not negative
    block_reduce_s2<1>(total, R, red);
    if (__syncthreads_or(wide)) {
        R[0] = regulariser_wide<D>(g, mp, u);
        block_reduce_d<1>(R, red);
    }
    if (threadIdx.x == 0)
        partials[blockIdx.x] = R[0];
    if (!maxbits)
        return;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, off));
    if ((threadIdx.x & 31) == 0)
        wm[threadIdx.x >> 5] = big;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kTileX * kTileY / 32; ++w)
            big = fmaxf(big, wm[w]);
        atomicMax(maxbits, __float_as_uint(big));
    }
}

// Fixed-order sum of `count` partials (one block), scaled, into out[0].
__global__ void k_sum_partials(const double *__restrict__ partials, int count, double scale,
                               double *__restrict__ out)
{
    __shared__ double red[32];
    double acc[1] = {0.0};
    for (int i = threadIdx.x; i < count; i += blockDim.x)
        acc[0] += partials[i];
    block_reduce_d<1>(acc, red);
    if (threadIdx.x == 0)
        out[0] = acc[0] * scale;
}

// {J, S, R, n_mask} of the unfused pieces; R as reg[0], or (count > 0) as the
// fixed-order sum of `count` partials times scale.
__global__ void __launch_bounds__(256)
    k_combine(const double *__restrict__ sim, const double *__restrict__ reg, int count,
              double scale, double lambda, double *__restrict__ out)
{
    __shared__ double red[8];
    double acc[1] = {0.0};
    for (int i = threadIdx.x; i < count; i += blockDim.x)
        acc[0] += reg[i];
    block_reduce_d<1>(acc, red);
    if (threadIdx.x == 0) {
        const double S = sim[0], n = sim[1], R = count > 0 ? acc[0] * scale : reg[0];
        out[0] = S + lambda * R;
        out[1] = S;
        out[2] = R;
        out[3] = n;
    }
}

int elementwise_grid(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    const int64_t most = 64 * (int64_t)device_sms();  // grid-stride loops beyond this
    return (int)(b < most ? (b < 1 ? 1 : b) : most);
}

}  // namespace

template <int TX>
static cudaError_t run_displacement(const Grid &g, const Lattice &L, const float *ctrl,
                                    float *disp, cudaStream_t s)
{
    dim3 grid((g.X + TX - 1) / TX, (g.Y + kDispTY - 1) / kDispTY, g.Z);
    const size_t smem = (size_t)g.ndim * std::min(disp_span(TX, L.delta), L.nx) * kDispTY * 4;
    if (g.ndim == 3)
        k_displacement<3, TX><<<grid, TX, smem, s>>>(g, L, ctrl, disp);
    else
        k_displacement<2, TX><<<grid, TX, smem, s>>>(g, L, ctrl, disp);
    return cudaGetLastError();
}

cudaError_t launch_displacement(const Grid &g, const Lattice &L, const float *ctrl, float *disp,
                                cudaStream_t s)
{
    return g.X <= 32 ? run_displacement<32>(g, L, ctrl, disp, s)
                     : run_displacement<kDispTX>(g, L, ctrl, disp, s);
}

size_t displacement_adjoint_ws(const Grid &g, const Lattice &L)
{
    // t1: ndim x Z x Y x nx, t2: ndim x Z x ny x nx
    size_t t1 = (size_t)g.ndim * g.Z * g.Y * L.nx;
    size_t t2 = (size_t)g.ndim * g.Z * L.ny * L.nx;
    return ((t1 * 4 + 255) / 256) * 256 + ((t2 * 4 + 255) / 256) * 256;
}

static void transpose_axis(const float *in, float *out, int64_t outer, int len, int n,
                           int64_t inner, const Lattice &L, cudaStream_t s)
{
    const int64_t total = outer * n * inner;
    const int blocks = elementwise_grid(total, kTransThreads);
    if (total < 1ll << 31)  // and a step of the grid beyond it fits 32 bits
        k_transpose_axis<unsigned><<<blocks, kTransThreads, 0, s>>>(in, out, (unsigned)total, len,
                                                                    n, (unsigned)inner, L);
    else
        k_transpose_axis<int64_t><<<blocks, kTransThreads, 0, s>>>(in, out, total, len, n, inner,
                                                                   L);
}

cudaError_t launch_displacement_adjoint(const Grid &g, const Lattice &L, const float *grad_disp,
                                        float *grad_ctrl, void *ws, cudaStream_t s)
{
    const int D = g.ndim;
    // x and y: (D*Z, Y, X) -> (D*Z, ny, nx); in 2D this is the result, in 3D the
    // second part of the workspace
    const size_t t1n = (size_t)D * g.Z * g.Y * L.nx;
    float *t2 = (float *)((char *)ws + ((t1n * 4 + 255) / 256) * 256);
    // Few cells a row leave a row's warp most lanes idle: one thread per output and axis
    // instead (three launches; from about 32 k rows on: 256 x 256 x 8 at spacing 16
    // 90 us against 32, 300 x 300 x 3 at 5 87 / 25, 128 x 256 x 16 at 6 43 / 25; 128 x 200 x 24
    // at 3 37 / 40, and 20000 x 5 at 8 20 / 31).
    if ((int64_t)D * g.Z * g.Y >= 32768 && (g.X < 24 || g.X < 5 * L.delta)) {
        const int64_t rows = (int64_t)D * g.Z * g.Y;
        float *t1 = (float *)ws, *xy = D == 3 ? t2 : grad_ctrl;
        transpose_axis(grad_disp, t1, rows, g.X, L.nx, 1, L, s);
        transpose_axis(t1, xy, (int64_t)D * g.Z, g.Y, L.ny, L.nx, L, s);
        if (D == 3)
            transpose_axis(xy, grad_ctrl, D, g.Z, L.nz, (int64_t)L.ny * L.nx, L, s);
        return cudaGetLastError();
    }
    const TransPlan t = trans_plan(g, L);
    k_transpose_xy<<<D * g.Z * t.nxt * t.nbands, kTransThreads, t.smem, s>>>(
        grad_disp, D == 3 ? t2 : grad_ctrl, g.X, g.Y, t, L);
    if (D == 3)  // z: (D, Z, ny*nx) -> (D, nz, ny*nx)
        transpose_axis(t2, grad_ctrl, D, g.Z, L.nz, (int64_t)L.ny * L.nx, L, s);
    return cudaGetLastError();
}

cudaError_t launch_warp(const Grid &g, const float *moving, const float *disp, float *warped,
                        uint8_t *mask, cudaStream_t s)
{
    const March m = march_plan(g);
    if (g.ndim == 3)
        k_warp<3><<<m.ntiles, kTileX * kTileY, 0, s>>>(g, m, moving, disp, warped, mask);
    else
        k_warp<2><<<m.ntiles, kTileX * kTileY, 0, s>>>(g, m, moving, disp, warped, mask);
    return cudaGetLastError();
}

cudaError_t launch_warp_adjoint(const Grid &g, const float *moving, const float *disp,
                                const uint8_t *mask, const float *grad_warped, float *grad_disp,
                                int accumulate, cudaStream_t s)
{
    const March m = march_plan(g);
    if (g.ndim == 3)
        k_warp_adjoint<3><<<m.ntiles, kTileX * kTileY, 0, s>>>(g, m, moving, disp, mask,
                                                               grad_warped, grad_disp, accumulate);
    else
        k_warp_adjoint<2><<<m.ntiles, kTileX * kTileY, 0, s>>>(g, m, moving, disp, mask,
                                                               grad_warped, grad_disp, accumulate);
    return cudaGetLastError();
}

size_t regulariser_ws(const Grid &g)
{
    size_t blocks = ((size_t)g.nv + 255) / 256;
    return blocks * sizeof(double);
}

// Blocks of k_regulariser: at most what its partials' workspace holds.
int regulariser_blocks(const Grid &g, const March &m)
{
    const int64_t slots = ((int64_t)g.nv + 255) / 256;
    return (int)std::min<int64_t>(std::min<int64_t>(m.ntiles, slots), 8192);
}

template <int D>
static void run_regulariser(const Grid &g, const March &m, int blocks, int gw, const float *u,
                            float gscale, float *gu, double *part, const AdjointArgs &a,
                            unsigned int *maxbits, cudaStream_t s)
{
    constexpr int T = kTileX * kTileY;
    switch (gw) {
    case GW_MSE: k_regulariser<D, GW_MSE><<<blocks, T, 0, s>>>(g, m, u, gscale, gu, part, a, maxbits); break;
    case GW_NCC: k_regulariser<D, GW_NCC><<<blocks, T, 0, s>>>(g, m, u, gscale, gu, part, a, maxbits); break;
    case GW_SCALED: k_regulariser<D, GW_SCALED><<<blocks, T, 0, s>>>(g, m, u, gscale, gu, part, a, maxbits); break;
    default: k_regulariser<D, GW_NONE><<<blocks, T, 0, s>>>(g, m, u, gscale, gu, part, a, maxbits); break;
    }
}

cudaError_t launch_regulariser_adjoint(const Grid &g, const float *disp, double weight, int gw,
                                       const AdjointArgs &a, float *grad_disp, double *partials,
                                       int *count, unsigned int *maxbits, cudaStream_t s)
{
    const March m = march_plan(g);
    *count = regulariser_blocks(g, m);
    const float gscale = (float)(2.0 * weight / (double)g.nv);
    if (g.ndim == 3)
        run_regulariser<3>(g, m, *count, gw, disp, gscale, grad_disp, partials, a, maxbits, s);
    else
        run_regulariser<2>(g, m, *count, gw, disp, gscale, grad_disp, partials, a, maxbits, s);
    return cudaGetLastError();
}

cudaError_t launch_regulariser(const Grid &g, const float *disp, double weight, double *value_dev,
                               float *grad_disp, void *ws, cudaStream_t s)
{
    double *partials = (double *)ws;
    int count = 0;
    const cudaError_t e = launch_regulariser_adjoint(g, disp, weight, GW_NONE, AdjointArgs{},
                                                     grad_disp, partials, &count, nullptr, s);
    if (e != cudaSuccess)
        return e;
    k_sum_partials<<<1, 256, 0, s>>>(partials, count, 1.0 / (double)g.nv, value_dev);
    return cudaGetLastError();
}

cudaError_t launch_combine(const double *sim_value, const double *reg, int count, double scale,
                           double lambda, double *out, cudaStream_t s)
{
    k_combine<<<1, 256, 0, s>>>(sim_value, reg, count, scale, lambda, out);
    return cudaGetLastError();
}

AL_UNIT_ERROR_READER(unit_error_basic)

}  // namespace airgb
