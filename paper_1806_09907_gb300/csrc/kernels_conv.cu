// Learned initialisation: 3x3x3 convolution layers (forward, input adjoint,
// weight adjoint) on the 5th-generation tensor cores of sm_103a.
//
// The paper names learning-based registration as planned work (Sec. I,
// Sec. V) without a network. This library trains a small encoder-decoder
// that predicts the B-spline coefficients of a pair. Its layers are dense
// contractions, and they are written here as implicit GEMMs:
//
//   forward   out[o][co]   = sum_{t, ci} in[s o + d_t][ci] * w[co][t][ci]
//             M = output voxels, N = cout, K = 27 cin (k = t cin + ci)
//   dgrad     g_in[p][ci]  = sum_{t, co} g_out[(p - d_t)/s][co] * w[co][t][ci]
//             M = input voxels,  N = cin,  K = (live taps) cout (k = tap cout + co)
//             With stride 2 only the taps whose (p - d_t)/2 is an integer
//             reach p: one per axis where p is even (d = 0), two where it
//             is odd (d = -1, +1). The input voxels are split into the 8
//             parity classes of (z, y, x), and each class runs over its own
//             1 to 8 taps instead of 27.
//   wgrad     g_w[(t,ci)][co] = sum_o in[s o + d_t][ci] * g_out[o][co]
//             M = 27 cin (+1: a row of ones gives the bias gradient),
//             N = cout, K = output voxels (split over blocks, partials
//             summed in a fixed order by k_wgrad_reduce)
//
// Activations are bf16, channels last ([b][z][y][x][c]); accumulation is
// fp32 in tensor memory. A CTA of 4 warps owns a 128-row tile of D in TMEM
// (tcgen05.alloc) and walks a stream of work items (one K slice of 64 of a
// tile each, tile after tile, the CTA's tiles strided by the grid). The
// threads gather the im2col operand of the next item with cp.async
// (16-byte copies, zero-filled at the faces) into a 2-slot shared-memory
// ring (a 3-slot ring two items ahead fitted fewer CTAs per SM and was
// slower: these gathers want resident warps more than depth); the weight
// operand of the forward and dgrad passes is stored pre-tiled in the
// shared-memory layout, so each slice of it arrives
// with one cp.async.bulk on an mbarrier. One thread issues tcgen05.mma
// (kind::f16, bf16 x bf16 -> f32, M = 128, K = 16 per instruction) on
// shared-memory descriptors and a tcgen05.commit frees the slot; after the
// last slice of a tile the threads read D back with tcgen05.ld while the
// next tile's gathers are already in flight.
//
// Shared-memory operand layout (no swizzle): 8 x 8 core matrices of 128 B
// (eight 16-byte rows). For the K-major operands (forward, dgrad) a row is 8
// consecutive K elements of one M/N index; for the MN-major operands (wgrad,
// whose K runs over voxels) a row is 8 consecutive M/N elements at one K
// index, which is exactly one 16-byte channel group of a voxel, so no
// transposition is needed. In both cases the core matrices of a tile are
// placed 128 B apart along K and 1024 B apart along M/N.
//
// Every wait on an mbarrier is bounded (about one second of %globaltimer);
// a wait that runs out records AL_ERR_TIMEOUT in the layer error word and
// the kernel carries on to its end, so no launch can hang.
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "launch.h"
#include "profile.h"

namespace airgb {

namespace {

__device__ int g_conv_error = 0;

constexpr int kThreads = 128;
constexpr int kStages = 2;                    // shared-memory ring slots
constexpr int kAhead = 1;                     // items gathered ahead of the MMA (< kStages)
constexpr int kBK = 64;                       // K elements per ring slot
constexpr int kATile = 128 * kBK * 2;         // bytes of one A slot (16 KB)
// wgrad and split-K blocks aimed at (8 per SM of a 152-SM GB300). A constant,
// not the device's SM count: the split counts size workspaces, which must not
// depend on the device the sizes are queried on.
constexpr int kTargetUnits = 1216;
constexpr int kErrTimeout = 6;                // AL_ERR_TIMEOUT
constexpr int kMaxClasses = 8;
constexpr int kMaxDynSmem = 227 * 1024;      // dynamic shared memory a CTA may have

enum { FWD = 0, DGRAD = 1, WGRAD = 2 };

struct ConvArgs {
    const __nv_bfloat16 *act;    // FWD/WGRAD: layer input; DGRAD: grad of the output
    const __nv_bfloat16 *gout;   // WGRAD: grad of the output
    const __nv_bfloat16 *wpk;    // FWD/DGRAD: weight slices in the shared-memory layout
    const float *bias;           // FWD (nullable)
    const __nv_bfloat16 *mask;   // DGRAD: ReLU factor (x_in > 0), N channels (nullable)
    const __nv_bfloat16 *addend; // DGRAD: added before the ReLU factor (nullable)
    void *out;
    int D, H, W, Do, Ho, Wo;     // input and output grid of the layer
    int cin, cout, stride;
    int N;                       // GEMM N
    int Kreal;                   // FWD 27 cin; DGRAD 27 cout (stride 1); WGRAD voxels per split
    int units, mtiles;           // work units (tiles); WGRAD: M tiles (units = mtiles x splits)
    int rows;                    // FWD: output voxels; DGRAD: input voxels; WGRAD: output voxels
    int relu, out_f32, add_stride, add_off;
    int wide;                    // out and mask lie on 32 bytes: a row's 16 columns are one access
    int64_t act_elems, gout_elems;  // elements of act and gout (checked builds)
    float *part;                 // FWD with split K: fp32 partials [class][rows][N]
    int classes;                 // DGRAD with stride 2: 8 parity classes; otherwise 1
    int cls_unit0[kMaxClasses + 1];  // first unit of each class; [classes] = units
    int cls_nst[kMaxClasses];        // K slices of a unit of each class
    int cls_slice0[kMaxClasses];     // first packed weight slice of each class
    uint32_t idesc, tmem_cols;
};

// ---- PTX wrappers ----------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase of `bar` with this parity to complete, for about one
// second at most; false (and AL_ERR_TIMEOUT recorded) if it did not.
__device__ __noinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity))
        return true;
    const uint64_t t0 = globaltimer();
    while (!mbar_try_wait(bar, parity)) {
        if (globaltimer() - t0 > 1000000000ull) {
            atomicExch(&g_conv_error, kErrTimeout);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes,
                                          uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t cols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
                 "r"(cols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols)
                 : "memory");
}

__device__ __forceinline__ void tc_before_sync()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_after_sync()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// D[tmem] (+)= A * B^T for one K = 16 slice (bf16 operands, fp32 accumulator).
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// tc_mma by the lane that has `on`, every lane of the warp calling with the same
// operands: they stay in uniform registers, which the instruction takes.
__device__ __forceinline__ void tc_mma_if(bool on, uint32_t d, uint64_t adesc, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accumulate)
{
    if (on)
        tc_mma(d, adesc, bdesc, idesc, accumulate);
}

__device__ __forceinline__ bool elect_one()
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok));
    return ok != 0;
}

// Arrive on `bar` once every tcgen05.mma issued so far by this thread is done.
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}

// 16 consecutive fp32 columns of this thread's TMEM lane (warp w reads lanes
// 32w .. 32w + 31), waiting for the load to complete.
__device__ __forceinline__ void tc_load16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i)
        v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor, no swizzle: start address, the byte
// distance between core matrices along K (leading) and along M/N (stride),
// descriptor version 1 (bits 46-47) of sm_100-class tensor cores.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo = 128, uint32_t sbo = 1024)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) |
           ((uint64_t)(sbo >> 4) << 32) | (1ull << 46);
}

// 32 bytes of a 32-byte aligned address.
__device__ __forceinline__ void store32(void *p, const uint32_t (&w)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]),
                 "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}

__device__ __forceinline__ void load32(const void *p, uint4 (&w)[2])
{
    asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(w[0].x), "=r"(w[0].y), "=r"(w[0].z), "=r"(w[0].w), "=r"(w[1].x),
                   "=r"(w[1].y), "=r"(w[1].z), "=r"(w[1].w)
                 : "l"(p));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// Byte offset of row `r` (M or N index) and 16-byte chunk `kc` in a K-major
// tile, and of K row `k` of the core matrices of M/N group `g` in an
// MN-major tile: both put core matrices 128 B apart along K, 1024 B along M/N.
__device__ __forceinline__ int kmajor_off(int r, int kc) { return (r >> 3) * 1024 + kc * 128 + (r & 7) * 16; }
__device__ __forceinline__ int mnmajor_off(int g, int k) { return g * 1024 + (k >> 3) * 128 + (k & 7) * 16; }


__device__ __forceinline__ void cp16(uint32_t dst, const void *src, bool ok)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "r"(ok ? 16 : 0)
                 : "memory");
}

// The same through L1: pieces of one 32-byte sector that go to different planes
// fetch it once.
__device__ __forceinline__ void cp16_l1(uint32_t dst, const void *src, bool ok)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "r"(ok ? 16 : 0)
                 : "memory");
}

__device__ __forceinline__ void cp4(uint32_t dst, const void *src, bool ok)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src),
                 "r"(ok ? 4 : 0)
                 : "memory");
}

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ size_t vox_index(int b, int z, int y, int x, int D, int H, int W)
{
    return (((size_t)b * D + z) * H + y) * W + x;
}

// Position of a work item: unit u (a 128-row tile; its class and index in
// the class), slice kk of the unit's nst slices.
struct Cursor {
    int u, kk, cls, tile, nst;
};

__device__ __forceinline__ void cursor_set(Cursor &c, int units, int classes, const int *unit0,
                                           const int *nst)
{
    if (c.u >= units) {
        c.nst = 0;
        return;
    }
    int k = 0;
    while (k + 1 < classes && c.u >= unit0[k + 1])
        ++k;
    c.cls = k;
    c.tile = c.u - unit0[k];
    c.nst = nst[k];
}

// Parity class geometry of the stride-2 dgrad: class bits (z, y, x), the
// number of input voxels of the class per axis, and its taps per axis.
struct ClassGeo {
    int cz, cy, cx, Qz, Qy, Qx, rows;
};

__device__ __forceinline__ ClassGeo class_geo(const ConvArgs &a, int cls)
{
    ClassGeo g;
    g.cz = (cls >> 2) & 1;
    g.cy = (cls >> 1) & 1;
    g.cx = cls & 1;
    g.Qz = (a.D - g.cz + 1) / 2;
    g.Qy = (a.H - g.cy + 1) / 2;
    g.Qx = (a.W - g.cx + 1) / 2;
    g.rows = g.Qz * g.Qy * g.Qx * (a.rows / (a.D * a.H * a.W));
    return g;
}

// ---- operand fills ---------------------------------------------------------
// Tables shared by a CTA (built once per launch, row independent):
//   tapoff[t]      element offset of tap t from the origin of a row's taps:
//                  FWD and WGRAD: input voxel s o - 1 per axis, offset
//                  ((tz H + ty) W + tx) cin; DGRAD stride 1: output voxel
//                  p + 1 per axis, offset -((tz Ho + ty) Wo + tx) cout
//   ctoff[c][ti]   DGRAD stride 2: offset ((az Ho + ay) Wo + ax) cout of
//                  tap index ti of parity class c from output voxel q
struct Tables {
    int tapoff[27];
    int ctoff[kMaxClasses][8];
};

__device__ __forceinline__ void build_tables(const ConvArgs &a, Tables &T, int tid, int mode)
{
    if (tid < 27) {
        const int tz = tid / 9, ty = (tid / 3) % 3, tx = tid % 3;
        T.tapoff[tid] = mode == DGRAD ? -((tz * a.Ho + ty) * a.Wo + tx) * a.cout
                                      : ((tz * a.H + ty) * a.W + tx) * a.cin;
    }
    if (tid < kMaxClasses * 8) {
        const int cls = tid >> 3, ti = tid & 7;
        const int cz = (cls >> 2) & 1, cy = (cls >> 1) & 1, cx = cls & 1;
        const int ix = cx ? (ti & 1) : 0;
        const int iy = cy ? ((ti >> cx) & 1) : 0;
        const int iz = ti >> (cx + cy);
        const int az = cz & (iz == 0), ay = cy & (iy == 0), ax = cx & (ix == 0);
        T.ctoff[cls][ti] = ((az * a.Ho + ay) * a.Wo + ax) * a.cout;
    }
}

// Per-thread state of the unit (tile) the producer is filling.
struct UnitState {
    int64_t rowoff;  // FWD/DGRAD: element offset of the row's tap origin (used only with a valid tap)
    uint32_t mask;   // FWD/DGRAD: valid taps (bit t, or bit ti for a parity class)
    int g0;          // WGRAD: first group of 8 M rows of the unit's M tile
    int vend;        // WGRAD: end of the unit's voxels
    int ox, oy, oz, b, vox;  // WGRAD: the thread's next voxel
};

// WGRAD: the pieces of a slice of 64 voxels are 16 bytes each, (group, voxel).
// 2^sh consecutive lanes take consecutive groups of one voxel and tap (2^sh
// divides a tap's groups, so they are contiguous bytes), the next lanes the next
// voxels: a pass of the threads covers nvox voxels, and a thread's voxels are
// nvox apart through the whole unit, so they are advanced by adding nvox in
// mixed radix (Wo, Ho, Do) instead of being divided out.
struct WLanes {
    int sh, nvox, dx, dy, dz, db;
};

__device__ __forceinline__ WLanes wgrad_lanes(const ConvArgs &a)
{
    WLanes w;
    const int nc = a.cin >> 3;
    w.sh = a.cin == 2 ? 0 : (nc & 7) == 0 ? 3 : (nc & 3) == 0 ? 2 : (nc & 1) == 0 ? 1 : 0;
    w.nvox = min(kThreads >> w.sh, kBK);
    int r = w.nvox;
    w.dx = r % a.Wo;
    r /= a.Wo;
    w.dy = r % a.Ho;
    r /= a.Ho;
    w.dz = r % a.Do;
    w.db = r / a.Do;
    return w;
}

__device__ __forceinline__ void wgrad_advance(const ConvArgs &a, const WLanes &w, UnitState &st)
{
    st.vox += w.nvox;
    st.ox += w.dx;
    st.oy += w.dy;
    st.oz += w.dz;
    st.b += w.db;
    if (st.ox >= a.Wo) {
        st.ox -= a.Wo;
        ++st.oy;
    }
    if (st.oy >= a.Ho) {
        st.oy -= a.Ho;
        ++st.oz;
    }
    if (st.oz >= a.Do) {
        st.oz -= a.Do;
        ++st.b;
    }
}

// The thread's voxel: element offset of its tap origin and the taps inside the
// grid (none beyond the unit).
__device__ __forceinline__ uint32_t wgrad_taps(const ConvArgs &a, const UnitState &st, int64_t &org)
{
    const int z = st.oz * a.stride - 1, y = st.oy * a.stride - 1, x = st.ox * a.stride - 1;
    org = ((((int64_t)st.b * a.D + z) * a.H + y) * a.W + x) * a.cin;
    // an axis's first tap is inside unless it reads -1, its last unless it reads
    // n, its middle one always; taps t = 9 tz + 3 ty + tx
    uint32_t m = (1u << 27) - 1u;
    if (x < 0)
        m &= ~0x1249249u;
    if (x + 2 >= a.W)
        m &= ~(0x1249249u << 2);
    if (y < 0)
        m &= ~0x1C0E07u;
    if (y + 2 >= a.H)
        m &= ~(0x1C0E07u << 6);
    if (z < 0)
        m &= ~0x1FFu;
    if (z + 2 >= a.D)
        m &= ~(0x1FFu << 18);
    return st.vox < st.vend ? m : 0u;
}

template <int MODE>
__device__ __forceinline__ void unit_begin(const ConvArgs &a, const Cursor &c, int tid,
                                           UnitState &st)
{
    if (MODE == FWD) {
        const int row = c.tile * 128 + tid;
        st.mask = 0;
        st.rowoff = 0;
        if (row < a.rows) {
            int r = row;
            const int ox = r % a.Wo;
            r /= a.Wo;
            const int oy = r % a.Ho;
            r /= a.Ho;
            const int oz = r % a.Do;
            const int b = r / a.Do;
            const int z0 = oz * a.stride - 1, y0 = oy * a.stride - 1, x0 = ox * a.stride - 1;
            st.rowoff = ((((int64_t)b * a.D + z0) * a.H + y0) * a.W + x0) * a.cin;
            uint32_t mz = 0, my = 0, mx = 0;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                mz |= (uint32_t)((unsigned)(z0 + d) < (unsigned)a.D) << d;
                my |= (uint32_t)((unsigned)(y0 + d) < (unsigned)a.H) << d;
                mx |= (uint32_t)((unsigned)(x0 + d) < (unsigned)a.W) << d;
            }
#pragma unroll
            for (int t = 0; t < 27; ++t)
                st.mask |= (((mz >> (t / 9)) & (my >> ((t / 3) % 3)) & (mx >> (t % 3))) & 1u) << t;
        }
    } else if (MODE == DGRAD) {
        st.mask = 0;
        st.rowoff = 0;
        if (a.classes == 1) {
            const int row = c.tile * 128 + tid;
            if (row < a.rows) {
                int r = row;
                const int x = r % a.W;
                r /= a.W;
                const int y = r % a.H;
                r /= a.H;
                const int z = r % a.D;
                const int b = r / a.D;
                // output voxel p - d = p + 1 - t per axis, t in 0..2
                st.rowoff = ((((int64_t)b * a.Do + z + 1) * a.Ho + y + 1) * a.Wo + x + 1) * a.cout;
                uint32_t mz = 0, my = 0, mx = 0;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    mz |= (uint32_t)((unsigned)(z + 1 - d) < (unsigned)a.Do) << d;
                    my |= (uint32_t)((unsigned)(y + 1 - d) < (unsigned)a.Ho) << d;
                    mx |= (uint32_t)((unsigned)(x + 1 - d) < (unsigned)a.Wo) << d;
                }
#pragma unroll
                for (int t = 0; t < 27; ++t)
                    st.mask |= (((mz >> (t / 9)) & (my >> ((t / 3) % 3)) & (mx >> (t % 3))) & 1u)
                               << t;
            }
        } else {
            const ClassGeo g = class_geo(a, c.cls);
            const int row = c.tile * 128 + tid;
            if (row < g.rows) {
                int r = row;
                const int qx = r % g.Qx;
                r /= g.Qx;
                const int qy = r % g.Qy;
                r /= g.Qy;
                const int qz = r % g.Qz;
                const int b = r / g.Qz;
                st.rowoff = ((((int64_t)b * a.Do + qz) * a.Ho + qy) * a.Wo + qx) * a.cout;
                // adjacency 1 is reachable only when q + 1 is inside
                const uint32_t okz1 = (unsigned)(qz + 1) < (unsigned)a.Do,
                               oky1 = (unsigned)(qy + 1) < (unsigned)a.Ho,
                               okx1 = (unsigned)(qx + 1) < (unsigned)a.Wo;
                const uint32_t okz0 = (unsigned)qz < (unsigned)a.Do,
                               oky0 = (unsigned)qy < (unsigned)a.Ho,
                               okx0 = (unsigned)qx < (unsigned)a.Wo;
                const int ntaps = (1 + g.cz) * (1 + g.cy) * (1 + g.cx);
                for (int ti = 0; ti < ntaps; ++ti) {
                    const int ix = g.cx ? (ti & 1) : 0;
                    const int iy = g.cy ? ((ti >> g.cx) & 1) : 0;
                    const int iz = ti >> (g.cx + g.cy);
                    // odd axis: i = 0 is tap d = -1, reading output q + 1
                    const uint32_t az = g.cz & (iz == 0), ay = g.cy & (iy == 0),
                                   ax = g.cx & (ix == 0);
                    const uint32_t ok = (az ? okz1 : okz0) & (ay ? oky1 : oky0) & (ax ? okx1 : okx0);
                    st.mask |= ok << ti;
                }
            }
        }
    } else {
        const int split = c.u / a.mtiles;
        st.g0 = (c.u - split * a.mtiles) * 16;
        st.vend = min((split + 1) * a.Kreal, a.rows);
        const WLanes w = wgrad_lanes(a);
        st.vox = split * a.Kreal + ((tid >> w.sh) & (kBK - 1));
        unsigned r = (unsigned)st.vox;  // beyond the rows only where nothing is read
        st.ox = (int)(r % (unsigned)a.Wo);
        r /= (unsigned)a.Wo;
        st.oy = (int)(r % (unsigned)a.Ho);
        r /= (unsigned)a.Ho;
        st.oz = (int)(r % (unsigned)a.Do);
        st.b = (int)(r / (unsigned)a.Do);
    }
}

// This thread's share of one work item (slot A, B).
template <int MODE>
__device__ __forceinline__ void fill_item(const ConvArgs &a, const Cursor &c, UnitState &st,
                                          uint8_t *A, uint8_t *B, int tid, const int *tapoff,
                                          const int (*ctoff)[8], int kslice0, const WLanes &wl,
                                          const int2 *gtab)
{
    const uint32_t sA = (uint32_t)__cvta_generic_to_shared(A);
    if (MODE == FWD) {
        if (a.cin == 2) {
            // K = 54: word t (2 channels) of tap t; chunk t / 4, word t % 4
            const uint32_t *src = reinterpret_cast<const uint32_t *>(a.act);
#pragma unroll
            for (int t = 0; t < 32; ++t) {
                bool ok = t < 27 && ((st.mask >> (t & 31)) & 1u);
                if (ok && !(al_index_ok(st.rowoff + tapoff[t], a.act_elems - 1)))
                    ok = false;
                cp4(sA + kmajor_off(tid, t >> 2) + (t & 3) * 4,
                    ok ? src + (st.rowoff + tapoff[t < 27 ? t : 0]) / 2 : src, ok);
            }
        } else {
            // with split K the unit's slices start at slice kslice0 of the layer
            int k = (kslice0 + c.kk) * kBK;
            int t = k / a.cin, ci = k - t * a.cin;
#pragma unroll
            for (int kc = 0; kc < 8; ++kc, k += 8) {
                bool ok = k < a.Kreal && ((st.mask >> t) & 1u);
                if (ok && !al_index_ok(st.rowoff + tapoff[t] + ci, a.act_elems - 7))
                    ok = false;
                cp16(sA + kmajor_off(tid, kc),
                     ok ? a.act + st.rowoff + tapoff[ok ? t : 0] + ci : a.act, ok);
                ci += 8;  // next group of 8 channels (cin is a multiple of 8)
                if (ci >= a.cin) {
                    ci -= a.cin;
                    ++t;
                }
            }
        }
    } else if (MODE == DGRAD) {
        const int k0 = c.kk * kBK;
        int t = k0 / a.cout, co = k0 - t * a.cout;
#pragma unroll
        for (int kc = 0; kc < 8; ++kc, co += 8) {
            if (co >= a.cout) {
                co -= a.cout;
                ++t;
            }
            bool ok = t < 27 && ((st.mask >> (t & 31)) & 1u);
            int off = 0;
            if (ok)
                off = a.classes == 1 ? tapoff[t] : ctoff[c.cls][t];
            if (ok && !al_index_ok(st.rowoff + off + co, a.act_elems - 7))
                ok = false;
            cp16(sA + kmajor_off(tid, kc), ok ? a.act + st.rowoff + off + co : a.act, ok);
        }
    } else {
        // A: rows m = (t, ci) of the M tile, K = 64 voxels
        const int v0 = st.vox - ((tid >> wl.sh) & (kBK - 1));  // first voxel of the slice
        if (a.cin == 2) {
            // Thread tid owns voxel tid % 64 of the slice and half h = tid / 64 of the
            // words: word t of the 55 rows (tap t, 2 channels; t = 27 the bias row), 14
            // words per thread; words 28..31 and the groups past them stay zero
            // (cleared once: a 2-channel layer has one M tile)
            const int k = tid & (kBK - 1), h = tid >> 6;
            int64_t org;
            const uint32_t taps = wgrad_taps(a, st, org);
            const uint32_t *src = reinterpret_cast<const uint32_t *>(a.act);
#pragma unroll
            for (int j = 0; j < 14; ++j) {
                const int t = h * 14 + j;
                const int off = mnmajor_off(t >> 2, k) + (t & 3) * 4;
                if (t == 27) {
                    *reinterpret_cast<uint32_t *>(A + off) = st.vox < st.vend ? 0x3F80u : 0u;
                } else {
                    bool ok = (taps >> t) & 1u;
                    if (ok && !al_index_ok(org + tapoff[t], a.act_elems - 1))
                        ok = false;
                    cp4(sA + off, ok ? src + (org + tapoff[t]) / 2 : src, ok);
                }
            }
            wgrad_advance(a, wl, st);
        } else {
            const int gbias = 27 * (a.cin >> 3);
            const int cl = tid & ((1 << wl.sh) - 1);
            // with one lane per voxel, the threads' second half takes the odd groups
            const int half = wl.sh == 0 ? tid >> 6 : 0;
            const int first = (half << wl.sh) + cl, gstep = wl.sh == 0 ? 2 : 1 << wl.sh;
            for (int done = 0; done < kBK; done += wl.nvox) {
                const int k = st.vox - v0;
                int64_t org;
                const uint32_t taps = wgrad_taps(a, st, org);
                const uint32_t row = sA + mnmajor_off(0, k);
#pragma unroll 4
                for (int gl = first; gl < 16; gl += gstep) {
                    const int g = st.g0 + gl;
                    if (g < gbias) {
                        const int2 e = gtab[g];
                        bool ok = (taps >> e.y) & 1u;
                        const int64_t at = org + e.x;
                        if (ok && !al_index_ok(at, a.act_elems - 7))
                            ok = false;
                        cp16(row + gl * 1024, ok ? a.act + at : a.act, ok);
                    } else if (g == gbias) {
                        *reinterpret_cast<uint4 *>(A + mnmajor_off(gl, k)) =
                            make_uint4(st.vox < st.vend ? 0x3F80u : 0u, 0, 0, 0);
                    } else if (a.mtiles > 1) {
                        *reinterpret_cast<uint4 *>(A + mnmajor_off(gl, k)) = make_uint4(0, 0, 0, 0);
                    }
                }
                wgrad_advance(a, wl, st);
            }
        }
        // B: rows n = co (N / 8 groups) x 64 voxels, contiguous in memory
        const uint32_t sB = (uint32_t)__cvta_generic_to_shared(B);
        const int ng = a.N >> 3, dv = kThreads / ng, dg = kThreads - dv * ng;
        int v = tid / ng, g = tid - v * ng;
        const __nv_bfloat16 *src = a.gout + (size_t)v0 * a.cout + tid * 8;
        for (int idx = tid; idx < ng * kBK; idx += kThreads, src += kThreads * 8) {
            bool ok = v0 + v < st.vend;
            if (ok && !al_index_ok((int64_t)v0 * a.cout + (int64_t)idx * 8, a.gout_elems - 7))
                ok = false;
            cp16(sB + mnmajor_off(g, v), ok ? src : a.gout, ok);
            v += dv;
            g += dg;
            if (g >= ng) {
                g -= ng;
                ++v;
            }
        }
    }
}

// ---- epilogue: row tid of the finished tile from TMEM lane tid -------------
template <int MODE>
__device__ __forceinline__ void epilogue_row(const ConvArgs &a, size_t orow, bool valid,
                                             uint32_t lane_addr, int cls = 0);

template <int MODE>
__device__ __forceinline__ void epilogue(const ConvArgs &a, const Cursor &c, uint32_t lane_addr,
                                         int tid)
{
    size_t orow = 0;
    bool valid = true;
    if (MODE == FWD) {
        const int row = c.tile * 128 + tid;
        valid = row < a.rows;
        orow = (size_t)row;
    } else if (MODE == DGRAD) {
        if (a.classes == 1) {
            const int row = c.tile * 128 + tid;
            valid = row < a.rows;
            orow = (size_t)row;
        } else {
            const ClassGeo g = class_geo(a, c.cls);
            const int row = c.tile * 128 + tid;
            valid = row < g.rows;
            int r = valid ? row : 0;
            const int qx = r % g.Qx;
            r /= g.Qx;
            const int qy = r % g.Qy;
            r /= g.Qy;
            const int qz = r % g.Qz;
            const int b = r / g.Qz;
            orow = vox_index(b, 2 * qz + g.cz, 2 * qy + g.cy, 2 * qx + g.cx, a.D, a.H, a.W);
        }
    } else {
        const int mt = c.u % a.mtiles, split = c.u / a.mtiles;
        orow = (size_t)split * a.mtiles * 128 + (size_t)mt * 128 + tid;
    }
    epilogue_row<MODE>(a, orow, valid, lane_addr, c.cls);
}

// Columns c0 .. c0 + 15 of output row orow. cls: K partition of a split forward
// pass. mask: the row's ReLU factors already loaded (nullable).
template <int MODE>
__device__ __forceinline__ void epilogue_chunk(const ConvArgs &a, size_t orow, float (&v)[16],
                                               int c0, int cls, const uint4 *mask = nullptr)
{
    if (MODE == FWD && a.part) {
        // split K: this K partition's partial sums, reduced by k_fwd_reduce
        float4 *o = reinterpret_cast<float4 *>(a.part + ((size_t)cls * a.rows + orow) * a.N + c0);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        return;
    }
    if (MODE == FWD) {
        if (a.bias) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                v[i] += __ldg(a.bias + c0 + i);
        }
        if (a.relu) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                v[i] = fmaxf(v[i], 0.0f);
        }
    } else if (MODE == DGRAD) {
        if (a.addend) {
            const uint4 *p =
                reinterpret_cast<const uint4 *>(a.addend + orow * a.add_stride + a.add_off + c0);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint4 w = __ldg(p + q);
                const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    v[8 * q + 2 * h] += bf16_lo(ws[h]);
                    v[8 * q + 2 * h + 1] += bf16_hi(ws[h]);
                }
            }
        }
        if (a.mask) {
            const uint4 *p = reinterpret_cast<const uint4 *>(a.mask + orow * a.N + c0);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint4 w = mask ? mask[q] : __ldg(p + q);
                const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    if (!(bf16_lo(ws[h]) > 0.0f))
                        v[8 * q + 2 * h] = 0.0f;
                    if (!(bf16_hi(ws[h]) > 0.0f))
                        v[8 * q + 2 * h + 1] = 0.0f;
                }
            }
        }
    }
    if (MODE == WGRAD || (MODE == FWD && a.out_f32)) {
        float4 *o = reinterpret_cast<float4 *>(static_cast<float *>(a.out) + orow * a.N + c0);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    } else {
        uint32_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            w[i] = pack_bf16(v[2 * i], v[2 * i + 1]);
        uint4 *o = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(a.out) + orow * a.N + c0);
        if (a.wide) {
            store32(o, w);
        } else {
            o[0] = make_uint4(w[0], w[1], w[2], w[3]);
            o[1] = make_uint4(w[4], w[5], w[6], w[7]);
        }
    }
}

// Output row orow (when valid) from N columns of this thread's TMEM lane; every
// lane of the warp calls.
template <int MODE>
__device__ __forceinline__ void epilogue_row(const ConvArgs &a, size_t orow, bool valid,
                                             uint32_t lane_addr, int cls)
{
    for (int c0 = 0; c0 < a.N; c0 += 16) {
        float v[16];
        tc_load16(lane_addr + (uint32_t)c0, v);
        if (valid)
            epilogue_chunk<MODE>(a, orow, v, c0, cls);
    }
}

// Before the last MMAs of a dgrad tile complete: pull this row's ReLU-factor
// and addend channels towards L2, so the epilogue's reads do not wait on DRAM.
__device__ __forceinline__ void dgrad_prefetch(const ConvArgs &a, const Cursor &c, int tid)
{
    size_t orow;
    if (a.classes == 1) {
        const int row = c.tile * 128 + tid;
        if (row >= a.rows)
            return;
        orow = (size_t)row;
    } else {
        const ClassGeo g = class_geo(a, c.cls);
        const int row = c.tile * 128 + tid;
        if (row >= g.rows)
            return;
        int r = row;
        const int qx = r % g.Qx;
        r /= g.Qx;
        const int qy = r % g.Qy;
        r /= g.Qy;
        const int qz = r % g.Qz;
        const int b = r / g.Qz;
        orow = vox_index(b, 2 * qz + g.cz, 2 * qy + g.cy, 2 * qx + g.cx, a.D, a.H, a.W);
    }
    if (a.mask)
        for (int c0 = 0; c0 < a.N; c0 += 64)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.mask + orow * a.N + c0));
    if (a.addend)
        for (int c0 = 0; c0 < a.N; c0 += 64)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.addend + orow * a.add_stride +
                                                          a.add_off + c0));
}

// ---- the kernel ------------------------------------------------------------
// The weight adjoint is held to 128 registers per thread so that 4 CTAs fit
// per SM (it used 150 unbounded, 3 CTAs; 847 against 915 µs per training
// step, no spills); the other passes are limited by shared memory.
template <int MODE>
__global__ void __launch_bounds__(kThreads, MODE == WGRAD ? 4 : 1) k_conv(const ConvArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = reinterpret_cast<uint8_t *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sA = sm;
    const int btile = a.N * 128;  // bytes of one B slot: N rows x 64 K
    uint8_t *sB = sA + kStages * kATile;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sB + kStages * btile);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 2 * kStages + 1);
    int *s_unit0 = reinterpret_cast<int *>(tslot + 1);
    int *s_nst = s_unit0 + kMaxClasses + 1;
    int *s_slice0 = s_nst + kMaxClasses;
    Tables &T = *reinterpret_cast<Tables *>(s_slice0 + kMaxClasses);
    // WGRAD: per group of 8 M rows, element offset from a voxel's tap origin and tap
    int2 *gtab = reinterpret_cast<int2 *>(((uintptr_t)(&T + 1) + 7) & ~(uintptr_t)7);
    const uint32_t bar_full = smem_u32(bars), bar_free = bar_full + 8 * kStages,
                   bar_done = bar_full + 16 * kStages;
    const int tid = threadIdx.x, warp = tid >> 5;

    if (tid < kMaxClasses + 1)
        s_unit0[tid] = a.cls_unit0[tid < a.classes ? tid : a.classes];
    if (tid < kMaxClasses) {
        s_nst[tid] = a.cls_nst[tid < a.classes ? tid : 0];
        s_slice0[tid] = a.cls_slice0[tid < a.classes ? tid : 0];
    }
    build_tables(a, T, tid, MODE);
    if (MODE == WGRAD && a.cin != 2) {
        const int nc = a.cin >> 3;
        for (int g = tid; g < 27 * nc; g += kThreads) {
            const int t = g / nc;
            gtab[g] = make_int2(((t / 9 * a.H + t / 3 % 3) * a.W + t % 3) * a.cin + (g - t * nc) * 8, t);
        }
    }
    const WLanes wl = MODE == WGRAD ? wgrad_lanes(a) : WLanes{};
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_free + 8 * s, 1);
        }
        mbar_init(bar_done, 1);
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tslot), a.tmem_cols);
        tmem_relinquish();
    }
    if (MODE == WGRAD && a.mtiles == 1) {
        // the A rows past the bias row never change: zero them in every slot
        for (int i = tid; i < kStages * kATile / 16; i += kThreads)
            reinterpret_cast<uint4 *>(sA)[i] = make_uint4(0, 0, 0, 0);
    }
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    const uint32_t tmem = *tslot;

    Cursor prod;
    prod.u = blockIdx.x;
    prod.kk = 0;
    cursor_set(prod, a.units, a.classes, s_unit0, s_nst);
    Cursor cons = prod;
    uint32_t pit = 0, cit = 0, nunit = 0;

    UnitState ust;
    if (prod.u < a.units)
        unit_begin<MODE>(a, prod, tid, ust);

    auto produce = [&]() {
        if (prod.u < a.units) {
            const int s = (int)(pit % kStages);
            const uint32_t use = pit / kStages;
            if (use > 0)
                mbar_wait(bar_free + 8 * s, (use - 1) & 1);
            uint8_t *B = sB + s * btile;
            if (MODE != WGRAD && tid == 0) {
                mbar_expect_tx(bar_full + 8 * s, (uint32_t)btile);
                bulk_load(smem_u32(B),
                          a.wpk + (size_t)(s_slice0[prod.cls] + prod.kk) * a.N * kBK,
                          (uint32_t)btile, bar_full + 8 * s);
            }
            fill_item<MODE>(a, prod, ust, sA + s * kATile, B, tid, T.tapoff, T.ctoff,
                            MODE == FWD ? s_slice0[prod.cls] : 0, wl, gtab);
            ++pit;
            if (++prod.kk >= prod.nst) {
                prod.kk = 0;
                prod.u += gridDim.x;
                cursor_set(prod, a.units, a.classes, s_unit0, s_nst);
                if (prod.u < a.units)
                    unit_begin<MODE>(a, prod, tid, ust);
            }
        }
        cp_commit();
    };

    // the item gathered at step i goes into the slot whose MMA was issued
    // kStages - kAhead steps earlier, so that wait seldom stalls
#pragma unroll 1
    for (int j = 0; j < kAhead; ++j)
        produce();

#pragma unroll 1
    while (cons.u < a.units) {
        produce();
        cp_wait<kAhead>();
        fence_proxy_async();
        __syncthreads();
        const int s = (int)(cit % kStages);
        const uint32_t use = cit / kStages;
        if (tid == 0) {
            if (MODE != WGRAD)
                mbar_wait(bar_full + 8 * s, use & 1);
            tc_after_sync();
            const uint32_t a0 = smem_u32(sA + s * kATile), b0 = smem_u32(sB + s * btile);
#pragma unroll
            for (int j = 0; j < kBK / 16; ++j)
                tc_mma(tmem, sdesc(a0 + 256 * j), sdesc(b0 + 256 * j), a.idesc,
                       (cons.kk | j) != 0);
            tc_commit(bar_free + 8 * s);
        }
        ++cit;
        if (cons.kk == cons.nst - 1) {
            if (MODE == DGRAD)
                dgrad_prefetch(a, cons, tid);
            if (tid == 0)
                tc_commit(bar_done);
            mbar_wait(bar_done, nunit & 1);
            tc_after_sync();
            epilogue<MODE>(a, cons, tmem + ((uint32_t)(warp * 32) << 16), tid);
            tc_before_sync();
            __syncthreads();
            ++nunit;
        }
        if (++cons.kk >= cons.nst) {
            cons.kk = 0;
            cons.u += gridDim.x;
            cursor_set(cons, a.units, a.classes, s_unit0, s_nst);
        }
    }
    cp_wait<0>();
    __syncthreads();
    if (warp == 0)
        tmem_dealloc(tmem, a.tmem_cols);
}

// ---- two input channels: forward and weight adjoint --------------------------
// A tap row (dz, dy) of an output voxel reads three x-neighbouring voxels of
// two bf16 channels: 12 consecutive bytes, which with a fourth pair make one
// 16-byte chunk (dx, ci) of 8 K elements. A 128-voxel tile is 9 planes (one
// per (dz, dy)) of 128 chunks, 16 bytes apart: as K-major rows the operand of
// the forward pass (K = 9 chunks and one of zeros, 5 MMAs of K = 16), as
// MN-major groups of 8 rows that of the weight adjoint (M = 9 groups, K = 128
// voxels; the first chunk's fourth pair holds the one that gives the bias).
// A thread gathers the 27 words of its voxel into registers by plain loads
// (with stride 2 and an even row, one 8-byte load per tap row and the third
// word from the lane before) and stores 9 chunks; k_conv filled the same tile
// with 27 4-byte asynchronous copies a row, which was bound by their number.
// One tile in shared memory: the next tile's loads are in flight in registers
// while its MMAs run, and the room left is better used by more CTAs per SM.
// 16 x 128^3 -> 64^3, stride 2: forward 205 -> 94 us, weight adjoint 280 -> 102 us
// (103 and 145 us with two slots and three loads per tap row); reading the
// input and writing or reading the output takes 40 us.
constexpr int kC2Plane = 128 * 16;  // bytes of one plane of a tile
constexpr int kC2Groups = 9;

// The 9 chunks of output voxel `row` (zero outside the grid). PAIR: stride 2
// and an even W, so that voxels 2 ox and 2 ox + 1 are one aligned 8-byte load
// and voxel 2 ox - 1 is the second of the lane before, when that lane has the
// voxel before. Every lane of the warp calls.
template <bool PAIR>
__device__ __forceinline__ void c2_gather(const ConvArgs &a, int row, bool ok,
                                          uint32_t (&w)[kC2Groups][3])
{
    unsigned r = ok ? (unsigned)row : 0u;
    const unsigned ox = r % (unsigned)a.Wo;
    r /= (unsigned)a.Wo;
    const unsigned oy = r % (unsigned)a.Ho;
    r /= (unsigned)a.Ho;
    const unsigned oz = r % (unsigned)a.Do, b = r / (unsigned)a.Do;
    const int st = PAIR ? 2 : a.stride;
    const int z0 = (int)oz * st - 1, y0 = (int)oy * st - 1, x0 = (int)ox * st - 1;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(a.act);
    const bool xl = x0 >= 0, xr = x0 + 2 < a.W;
    const bool alone = (threadIdx.x & 31) == 0 && xl;  // no lane before it
    const int64_t org = (((int64_t)b * a.D + z0) * a.H + y0) * a.W + x0;
#pragma unroll
    for (int g = 0; g < kC2Groups; ++g) {
        const int dz = g / 3, dy = g % 3;
        bool in = ok && (unsigned)(z0 + dz) < (unsigned)a.D && (unsigned)(y0 + dy) < (unsigned)a.H;
        const int64_t o = org + ((int64_t)dz * a.H + dy) * a.W;
        if (in && !al_index_ok(o + 1, a.act_elems / 2))
            in = false;
        if (PAIR) {
            const uint2 p = in ? __ldg(reinterpret_cast<const uint2 *>(src + o + 1))
                               : make_uint2(0u, 0u);
            w[g][0] = in && alone ? __ldg(src + o) : 0u;
            w[g][1] = p.x;
            w[g][2] = p.y;
        } else {
            w[g][0] = in && xl ? __ldg(src + o) : 0u;
            w[g][1] = in ? __ldg(src + o + 1) : 0u;
            w[g][2] = in && xr ? __ldg(src + o + 2) : 0u;
        }
    }
}

// Stores the chunks (every lane calls); fourth: the fourth pair of chunk 0.
template <bool PAIR>
__device__ __forceinline__ void c2_store(const ConvArgs &a, uint8_t *A, int row, bool ok,
                                         uint32_t fourth, const uint32_t (&w)[kC2Groups][3])
{
    const int tid = threadIdx.x;
    const bool left = PAIR && (tid & 31) != 0 && ok && (unsigned)row % (unsigned)a.Wo != 0;
#pragma unroll
    for (int g = 0; g < kC2Groups; ++g) {
        uint32_t w0 = w[g][0];
        if (PAIR) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, w[g][2], 1);
            w0 = left ? up : w0;
        }
        *reinterpret_cast<uint4 *>(A + g * kC2Plane + tid * 16) =
            make_uint4(w0, w[g][1], w[g][2], g == 0 ? fourth : 0u);
    }
}

// Forward: shared memory = the tile's 10 planes, the weights as 10 chunks of N
// rows, barrier.
template <int N, bool PAIR>
__global__ void __launch_bounds__(kThreads) k_conv2_fwd(const ConvArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *A = reinterpret_cast<uint8_t *>(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    uint8_t *B = A + 10 * kC2Plane;
    uint64_t *bars = reinterpret_cast<uint64_t *>(B + 10 * N * 16);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 1);
    const uint32_t bar = smem_u32(bars);
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tslot), 32);
        tmem_relinquish();
    }
    // B: chunk g, row n, element (dx, ci) = w[n][t = 3 g + dx][ci] from the packed
    // copy (k = 2 t + ci); zero for dx = 3 and chunk 9
    for (int e = tid; e < 10 * N * 8; e += kThreads) {
        const int q = e & 7, n = (e >> 3) % N, g = (e >> 3) / N;
        const int k = 2 * (3 * g + (q >> 1)) + (q & 1);
        __nv_bfloat16 v = __float2bfloat16_rn(0.0f);
        if (g < kC2Groups && q < 6)
            v = a.wpk[(n / 8) * 512 + (k / 8) * 64 + (n % 8) * 8 + (k & 7)];
        reinterpret_cast<__nv_bfloat16 *>(B)[e] = v;
    }
    *reinterpret_cast<uint4 *>(A + kC2Groups * kC2Plane + tid * 16) = make_uint4(0u, 0u, 0u, 0u);
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    const uint32_t tmem = *tslot;
    const uint32_t a0 = smem_u32(A), b0 = smem_u32(B);
    uint32_t w[kC2Groups][3];
    auto finish = [&](int tile, int it) {
        mbar_wait(bar, (uint32_t)it & 1);
        tc_after_sync();
        const int row = tile * 128 + tid;
        epilogue_row<FWD>(a, (size_t)row, row < a.rows, tmem + ((uint32_t)(warp * 32) << 16));
        tc_before_sync();
    };
    int it = 0;
    for (int tile = blockIdx.x; tile < a.units; tile += gridDim.x, ++it) {
        const int row = tile * 128 + tid;
        const bool ok = row < a.rows;
        c2_gather<PAIR>(a, row, ok, w);
        if (it > 0)
            finish(tile - gridDim.x, it - 1);
        c2_store<PAIR>(a, A, row, ok, 0u, w);
        fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
            tc_after_sync();
#pragma unroll
            for (int j = 0; j < 5; ++j)
                tc_mma(tmem, sdesc(a0 + 2 * j * kC2Plane, kC2Plane, 128),
                       sdesc(b0 + 2 * j * N * 16, N * 16, 128), a.idesc, j != 0);
            tc_commit(bar);
        }
    }
    if (it > 0)
        finish(blockIdx.x + (it - 1) * gridDim.x, it - 1);
    __syncthreads();
    if (warp == 0)
        tmem_dealloc(tmem, 32);
}

// Weight adjoint: shared memory = 16 planes (the 9 of the tile, the N / 8 of
// the output gradient, and what M = 128 reads beyond them, rows of D that are
// never used), barriers. One D per unit (a split of the voxels) in TMEM.
template <int N, bool PAIR>
__global__ void __launch_bounds__(kThreads) k_conv2_wgrad(const ConvArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *A = reinterpret_cast<uint8_t *>(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    uint8_t *G = A + kC2Groups * kC2Plane;
    uint64_t *bars = reinterpret_cast<uint64_t *>(A + 16 * kC2Plane);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 2);
    const uint32_t bar = smem_u32(bars);
    const int tid = threadIdx.x, warp = tid >> 5;
    static_assert(kC2Groups + N / 8 <= 16, "the output gradient's planes lie inside the 16");
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 8, 1);
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tslot), 32);
        tmem_relinquish();
    }
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    const uint32_t tmem = *tslot;
    const uint32_t a0 = smem_u32(A), g0 = smem_u32(G);
    uint32_t w[kC2Groups][3];
    int it = 0;
    uint32_t nunit = 0;
    for (int u = blockIdx.x; u < a.units; u += gridDim.x, ++nunit) {
        const int v0 = u * a.Kreal, v1 = min(v0 + a.Kreal, a.rows);
        for (int v = v0; v < v1; v += 128, ++it) {
            const int row = v + tid;
            const bool ok = row < v1;
            c2_gather<PAIR>(a, row, ok, w);
            uint4 gr[N / 8];
#pragma unroll
            for (int n = 0; n < N / 8; ++n) {
                bool in = ok;
                if (in && !al_index_ok((int64_t)row * N + n * 8, a.gout_elems - 7))
                    in = false;
                gr[n] = in ? __ldg(reinterpret_cast<const uint4 *>(a.gout + (size_t)row * N) + n)
                           : make_uint4(0u, 0u, 0u, 0u);
            }
            if (it > 0)
                mbar_wait(bar, (uint32_t)(it - 1) & 1);
            c2_store<PAIR>(a, A, row, ok, ok ? 0x3F80u : 0u, w);
#pragma unroll
            for (int n = 0; n < N / 8; ++n)
                *reinterpret_cast<uint4 *>(G + n * kC2Plane + tid * 16) = gr[n];
            fence_proxy_async();
            __syncthreads();
            if (tid == 0) {
                tc_after_sync();
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    tc_mma(tmem, sdesc(a0 + 256 * j, 128, kC2Plane),
                           sdesc(g0 + 256 * j, 128, kC2Plane), a.idesc, v != v0 || j != 0);
                tc_commit(bar);
            }
        }
        if (tid == 0)
            tc_commit(bar + 8);
        mbar_wait(bar + 8, nunit & 1);
        tc_after_sync();
        // row of chunk g, element (dx, ci) -> row 2 (3 g + dx) + ci of the partial
        // sums; the one (chunk 0, fourth pair) -> row 54
        const int g = tid >> 3, q = tid & 7;
        const bool keep = (g < kC2Groups && q < 6) || tid == 6;
        const int m = tid == 6 ? 54 : 6 * g + q;
        float *o = static_cast<float *>(a.out) + ((size_t)u * 128 + m) * N;
#pragma unroll
        for (int c0 = 0; c0 < N; c0 += 16) {
            float v[16];
            tc_load16(tmem + (uint32_t)c0 + ((uint32_t)(warp * 32) << 16), v);
            if (keep)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    *reinterpret_cast<float4 *>(o + c0 + 4 * k) =
                        make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
        }
        tc_before_sync();
        __syncthreads();
    }
    __syncthreads();
    if (warp == 0)
        tmem_dealloc(tmem, 32);
}

__device__ __forceinline__ int class_ntaps(int cls);

// ---- passes from a staged slab -------------------------------------------------
// k_conv gathers every row of the im2col operand tap by tap, so each input
// value passes through L2 and shared memory up to 27 times, and those copies
// bound it. Here a CTA stages the input of a band of R output rows once, as
// planes of 8 channels (16 bytes) per voxel, voxels P apart per row. With the
// no-swizzle layout a K-major operand is 16-byte rows of consecutive addresses,
// so the rows of 128 consecutive positions of the band, shifted by a tap, are
// the same memory at another start address: every tap is a descriptor, and the
// operand costs nothing beyond the staging (halo columns make a few of the 128
// rows idle). Read as MN-major groups of 8 rows, the same planes are the operand
// of the weight adjoint: the voxels are K, and 16 consecutive planes one MMA's
// 128 rows at one shift.
//
// The kinds (q: output position; for the stride-2 input adjoint q indexes voxel
// pairs, and the 8 parity classes of 2 q + c accumulate side by side in TMEM
// from the same slab):
//   FWD1   source q + d                    3 slices, rows and columns q - 1 .. q + 1
//   FWD2   source 2 q + d, split by parity: odd sources 2 q - 1 and 2 q + 1 are
//          neighbours in the odd block, 2 q is in the even block
//   DGRAD1 source q - d                    as FWD1 with the taps mirrored
//   DGRAD2 source q and q + 1              2 slices, rows q, q + 1, columns q, q + 1
//   WGRAD2 the slab of FWD2 against the output gradient of the band's positions
// Planes lie in the order (y, x parity block; z slice; 8 channels). The blocks'
// order (odd y, even x), (odd, odd), (even, odd), (even, even) makes the planes
// that a shift of WGRAD2 uses consecutive: all at (0, 0), blocks 1-2 one column
// on, 0-1 one row on, 1 both.
//
// Warps: the first 8 (16 for the input adjoints, whose epilogues read and write
// the most) take the epilogue, the warps of a TMEM quarter sharing its columns;
// one issues the MMAs; the others stage the slabs (16-byte asynchronous copies
// along rows) into a ring, two in flight. D is double buffered in TMEM (the weight
// adjoint drains once per unit; its K steps take the sets in turn), so
// staging, MMAs and epilogues of successive bands overlap. What it took, measured
// on 16 x 64^3 -> 32^3, 16 -> 32 channels, stride 2 (forward / input adjoint /
// weight adjoint):
//   k_conv                                                   124 / 332 / 178 us
//   a slab, the roles in turn, two CTAs per SM               106 / 154 us
//   roles in warps, MMAs issued by one thread from a table
//   in shared memory (its descriptors reach the uniform
//   registers one by one, over 100 cycles an MMA)            150 / 154 / 187 us
//   descriptors computed by the whole warp in uniform
//   registers, one elected lane issuing                       83 / 125 / 100 us
//   copies through L1 (two 16-byte pieces of a sector go to
//   two planes; past L1 they fetched it twice), 15 staging
//   warps, 16 epilogue warps, ReLU factors one group ahead    61 /  88 /  70 us
// The bytes take 25, 45 and 25 us; staging bounds the forward pass and the weight
// adjoint, the epilogue's loads and stores the input adjoint. The tensor core
// needs about 60 cycles per MMA here whatever N <= 64 (its A operand's 4 KB), so
// DGRAD2 joins the classes that share a shift into one MMA over their columns: the
// class order 0 1 5 4 6 7 3 2 makes most of them adjacent, 17 MMAs per 16 channels
// instead of 27.
enum { FWD1 = 0, FWD2 = 1, DGRAD1 = 2, DGRAD2 = 3, WGRAD2 = 4 };
// Epilogue and staging warps of a kind.
__host__ __device__ constexpr int slab_epi(int kind)
{
    return kind == DGRAD1 || kind == DGRAD2 ? 16 : 8;
}
__host__ __device__ constexpr int slab_prod(int kind)
{
    return kind == DGRAD1 || kind == DGRAD2 ? 7 : 15;
}
__host__ __device__ constexpr int slab_threads(int kind)
{
    return 32 * (slab_epi(kind) + 1 + slab_prod(kind));
}

struct SlabArgs {
    const __nv_bfloat16 *src;  // staged tensor, C channels
    int Sz, Sy, Sx;            // its grid
    int Qz, Qy, Qx;            // positions
    int P;                     // positions per staged row
    int R, T;                  // output rows of a band, 128-position tiles of it
    int RB;                    // staged rows of a block
    int nzb;                   // z slices
    int plane;                 // bytes of a plane (8 channels)
    int stage;                 // bytes of a ring stage
    int gplane;                // WGRAD2: bytes of an output gradient plane
    int goff;                  // WGRAD2: their offset in a stage
    int ksteps;                // WGRAD2: K steps of 16 positions that cover a band
    int krow;                  // WGRAD2: K steps of a row of outputs (a multiple of 16), else 0
    int nst;                   // ring stages
    int slack;                 // bytes behind the ring that a window may read
    int nacc;                  // accumulators in turn for tiles or units (2: double buffered)
    int nset;                  // WGRAD2: accumulator sets that a unit's K steps take in turn
    int nk;                    // MMAs of a tile or K step
    int accs;                  // TMEM columns of one accumulator set
    int bands, items;
    int upu;                   // WGRAD2: items of a unit
    int wbytes;                // weights in shared memory
    int64_t src_elems;
};

// DGRAD2: the column order of the classes, and a shift's runs of adjacent classes.
struct ShiftRun {
    int shift, pos, n, first;  // shift bits (z, y, x), first place in the class order, classes
};
constexpr int kRuns = 17;
// Shifts in descending order, so that a class sums its taps in the packed order;
// the class whose first tap a shift is starts its sum by an MMA of its own.
struct Runs {
    ShiftRun r[kRuns] = {{7, 5, 1, 1}, {6, 4, 1, 1}, {6, 5, 1, 0}, {5, 2, 1, 1}, {5, 5, 1, 0},
                         {4, 3, 1, 1}, {4, 2, 1, 0}, {4, 4, 2, 0}, {3, 6, 1, 1}, {3, 5, 1, 0},
                         {2, 7, 1, 1}, {2, 4, 3, 0}, {1, 1, 1, 1}, {1, 2, 1, 0}, {1, 5, 2, 0},
                         {0, 0, 1, 1}, {0, 1, 7, 0}};
};
__constant__ Runs c_runs = {};
__constant__ int c_cls_order[8] = {0, 1, 5, 4, 6, 7, 3, 2};

__device__ __forceinline__ int class_ntaps(int cls);

template <int C, int KIND>
__global__ void __launch_bounds__(slab_threads(KIND), 1) k_conv_slab(const ConvArgs a, const SlabArgs s)
{
    constexpr int NC = C / 8, NK16 = C / 16;
    constexpr int kSlabEpi = slab_epi(KIND), kSlabProd = slab_prod(KIND),
                  kSlabThreads = slab_threads(KIND);
    constexpr int PARTS = kSlabEpi / 4;  // warps of a TMEM quarter
    constexpr bool S2 = KIND == FWD2 || KIND == WGRAD2;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    // behind the last stage: what a window or a shifted tile reads beyond it
    uint8_t *wsm = ring + s.nst * s.stage + s.slack;
    uint64_t *bars = reinterpret_cast<uint64_t *>(wsm + ((s.wbytes + 127) & ~127));
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 12);
    // DGRAD2: class and first column in it of each 16 columns (c + 8 column)
    uint16_t *chunks = reinterpret_cast<uint16_t *>(tslot + 1);
    const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 32, bar_acc = bar_full + 64,
                   bar_free = bar_full + 80;
    const uint32_t ring0 = smem_u32(ring), w0 = smem_u32(wsm);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform to the compiler

    if (tid == 0) {
        for (int k = 0; k < s.nst; ++k) {
            mbar_init(bar_full + 8 * k, 32 * kSlabProd);
            mbar_init(bar_empty + 8 * k, 1);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(bar_acc + 8 * k, 1);
            mbar_init(bar_free + 8 * k, 32 * kSlabEpi);
        }
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tslot), a.tmem_cols);
        tmem_relinquish();
    }
    if (KIND == DGRAD2 && tid < s.accs / 16) {
        const int pos = 16 * tid / a.N;
        chunks[tid] = (uint16_t)(c_cls_order[pos] | (16 * tid - pos * a.N) << 3);
    }
    if (KIND == WGRAD2) {
        // zero the ring once: positions that no copy writes (the parity blocks' spare
        // row and column) are read as K elements
        for (int i = tid; i < (int)(wsm - ring) / 16; i += kSlabThreads)
            reinterpret_cast<uint4 *>(ring)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        // the plane of ones behind the slab's planes: its first row sums the
        // output gradient (the bias)
        const int np = 12 * NC;
        for (int i = tid; i < s.nst * (s.plane / 16); i += kSlabThreads) {
            const int st = i / (s.plane / 16), k = i - st * (s.plane / 16);
            *reinterpret_cast<uint32_t *>(ring + st * s.stage + np * s.plane + k * 16) = 0x3F80u;
        }
    } else {
        // weights: 16-byte pieces (row n, 8 of K) of the packed copy
        const uint4 *src = reinterpret_cast<const uint4 *>(a.wpk);
        if (KIND == DGRAD2) {
            // step (run, c16): rows of its classes, core matrices 128 bytes apart
            // along K, 256 along N
            const int per = a.N * 2;  // pieces of one class of one step
            for (int e = tid; e < 27 * NK16 * per; e += kSlabThreads) {
                int j = e / per, r = e - j * per;  // j: (run, c16, class of the run)
                int run = 0;
                while (j >= c_runs.r[run].n * NK16)
                    j -= c_runs.r[run++].n * NK16;
                const int c16 = j / c_runs.r[run].n, m = j - c16 * c_runs.r[run].n;
                const int cls = c_cls_order[c_runs.r[run].pos + m], sh = c_runs.r[run].shift;
                const int kc = r & 1, n = r >> 1;
                // the tap of class cls at this shift: on an odd axis the first tap
                // reads q + 1, the second q
                const int cz = cls >> 2, cy = (cls >> 1) & 1, cx = cls & 1;
                const int ix = cx & ~sh & 1, iy = cy & ~(sh >> 1) & 1, iz = cz & ~(sh >> 2) & 1;
                const int kk = ((iz * (1 + cy) + iy) * (1 + cx) + ix) * NK16 + c16;
                const int from = (a.cls_slice0[cls] + kk / 4) * a.N * 8 + (n >> 3) * 64 +
                                 ((kk & 3) * 2 + kc) * 8 + (n & 7);
                uint8_t *d = wsm + (size_t)(e / per - m) * a.N * 32;
                const int rn = m * a.N + n;
                *reinterpret_cast<uint4 *>(d + (rn >> 3) * 256 + kc * 128 + (rn & 7) * 16) =
                    __ldg(src + from);
            }
        } else {
            for (int e = tid; e < s.wbytes / 16; e += kSlabThreads)
                reinterpret_cast<uint4 *>(wsm)[e] = __ldg(src + e);
        }
    }
    fence_proxy_async();  // weights, ones and zeros were written by plain stores
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    const uint32_t tmem = *tslot;
    const uint32_t stage16 = (uint32_t)s.stage >> 4;

    // a CTA's items: strided by the grid, or (WGRAD2) upu consecutive ones per unit
    const int units = KIND == WGRAD2 ? a.units : s.items;
    const int per = KIND == WGRAD2 ? s.upu : 1;
    auto decode = [&](int item, int &b, int &qz, int &y0) {
        const int r = item / s.bands;
        y0 = (item - r * s.bands) * s.R;
        b = r / s.Qz;
        qz = r - b * s.Qz;
    };
    // WGRAD2: K steps of an item. The band's rows of outputs, row by row where a row is whole
    // steps; otherwise the steps run through the rows' spare columns and up to 15 positions
    // beyond them, whose output gradient is zero.
    auto ksteps_of = [&](int item) {
        const int rows = min(s.R, s.Qy - (item % s.bands) * s.R);
        return s.krow ? rows * s.krow : (rows * s.P + 15) / 16;
    };
    if (warp > kSlabEpi) {
        // ---- staging: a warp per source row, lanes along its 16-byte pieces
        const int pw = warp - kSlabEpi - 1;
        const int ny = S2 ? 2 * s.R + 1 : s.RB, nx = S2 ? 2 * s.Qx + 1 : s.P;
        const int o0 = KIND == DGRAD2 ? 0 : -1, mul = S2 ? 2 : 1;
        // lane: channels 8 cl .. 8 cl + 7 of voxels xl, xl + XS, ... of a row (lanes
        // beyond XS NC idle)
        constexpr int XS = 32 / NC;
        const int cl = lane % NC, xl = lane < XS * NC ? lane / NC : nx;
        // the output gradient's pieces the same way
        const int ng = a.N >> 3, gs = ng <= 32 ? 32 / ng : 1;
        const int gl = lane % ng, gx = lane < gs * ng ? lane / ng : s.P;
        uint32_t n = 0;
        for (int u = blockIdx.x; u < units; u += gridDim.x)
            for (int item = u * per; item < min((u + 1) * per, s.items); ++item, ++n) {
                const int st = (int)(n % (uint32_t)s.nst);
                const uint32_t use = n / (uint32_t)s.nst;
                if (use > 0)
                    mbar_wait(bar_empty + 8 * st, (use - 1) & 1);
                int b, qz, y0;
                decode(item, b, qz, y0);
                const uint32_t base = ring0 + st * s.stage;
                for (int row = pw; row < s.nzb * ny; row += kSlabProd) {
                    const int zi = row / ny, yi = row - zi * ny;
                    const int sz = mul * qz + o0 + zi, sy = mul * y0 + o0 + yi;
                    const bool rowok = (unsigned)sz < (unsigned)s.Sz && (unsigned)sy < (unsigned)s.Sy;
                    const int64_t at = ((((int64_t)b * s.Sz + sz) * s.Sy + sy) * s.Sx + o0) * C;
                    // S2: odd sources (yi, xi even) and even ones go to their blocks
                    const int blk_o = S2 ? ((yi & 1) ? 2 : 1) : 0, blk_e = (yi & 1) ? 3 : 0;
                    const int r0 = (S2 ? yi >> 1 : yi) * s.P;
                    const uint32_t d_o = base + (blk_o * s.nzb + zi) * NC * s.plane + r0 * 16;
                    const uint32_t d_e = base + (blk_e * s.nzb + zi) * NC * s.plane + r0 * 16;
                    // a lane keeps its 8 channels, and (32 / NC even) its x parity
                    const __nv_bfloat16 *from = s.src + at + (xl * NC + cl) * 8;
                    uint32_t to = (S2 ? ((xl & 1) ? d_e : d_o) + (xl >> 1) * 16 : d_o + xl * 16) +
                                  cl * s.plane;
                    if (!S2 || XS % 2 == 0) {
#pragma unroll 4
                        for (int xi = xl; xi < nx; xi += XS) {
                            bool ok = rowok && (unsigned)(o0 + xi) < (unsigned)s.Sx;
                            if (ok && !al_index_ok(from - s.src, s.src_elems - 7))
                                ok = false;
                            cp16_l1(to, ok ? from : s.src, ok);
                            from += XS * C;
                            to += S2 ? XS * 8 : XS * 16;
                        }
                    } else {
                        for (int xi = xl; xi < nx; xi += XS) {
                            bool ok = rowok && (unsigned)(o0 + xi) < (unsigned)s.Sx;
                            if (ok && !al_index_ok(from - s.src, s.src_elems - 7))
                                ok = false;
                            to = ((xi & 1) ? d_e : d_o) + (xi >> 1) * 16 + cl * s.plane;
                            cp16_l1(to, ok ? from : s.src, ok);
                            from += XS * C;
                        }
                    }
                }
                if (KIND == WGRAD2) {
                    // the output gradient at the band's positions, zero elsewhere
                    for (int r = pw; r * s.P < s.ksteps * 16; r += kSlabProd) {
                        const bool rowok = r < s.R && y0 + r < s.Qy;
                        const int64_t at =
                            ((((int64_t)b * s.Qz + qz) * s.Qy + y0 + r) * s.Qx) * a.N;
                        const __nv_bfloat16 *from = a.gout + at + (gx * ng + gl) * 8;
                        uint32_t to = base + s.goff + gl * s.gplane + (r * s.P + gx) * 16;
                        const int nxg = min(s.P, s.ksteps * 16 - r * s.P);
#pragma unroll 4
                        for (int x = gx; x < nxg; x += gs) {
                            bool ok = rowok && x < s.Qx;
                            if (ok && !al_index_ok(from - a.gout, a.gout_elems - 7))
                                ok = false;
                            cp16_l1(to, ok ? from : a.gout, ok);
                            from += gs * a.N;
                            to += gs * 16;
                        }
                    }
                }
                if (KIND == DGRAD2 && a.mask) {
                    // the ReLU factors of the item's voxels towards L2: the epilogue reads
                    // them one item later
                    const int line = 128 / (2 * a.N) > 0 ? 128 / (2 * a.N) : 1;  // voxels
                    for (int row = pw; row < 4 * s.R; row += kSlabProd) {
                        const int z = 2 * qz + row / (2 * s.R), y = 2 * y0 + row % (2 * s.R);
                        if (z < a.D && y < a.H)
                            for (int x = lane * line; x < a.W; x += 32 * line)
                                asm volatile("prefetch.global.L2 [%0];" ::"l"(
                                    a.mask + vox_index(b, z, y, x, a.D, a.H, a.W) * a.N));
                    }
                }
                cp_commit();
                if (n > 0) {
                    cp_wait<1>();  // the item before has landed
                    fence_proxy_async();
                    mbar_arrive(bar_full + 8 * (int)((n - 1) % (uint32_t)s.nst));
                }
            }
        if (n > 0) {
            cp_wait<0>();
            fence_proxy_async();
            mbar_arrive(bar_full + 8 * (int)((n - 1) % (uint32_t)s.nst));
        }
    } else if (warp == kSlabEpi) {
        // ---- MMAs: the whole warp computes the (uniform) operands, one lane issues
        const bool one = elect_one();
        const uint32_t pl = (uint32_t)s.plane >> 4, P = (uint32_t)s.P, N = (uint32_t)a.N;
        const uint32_t id0 = a.idesc & ~(0x3Fu << 17);  // without N
        // descriptor bits above the address
        const uint64_t ka = sdesc(0, s.plane, 128), kb = sdesc(0),
                       kbd = sdesc(0, 128, 256), ma = sdesc(0, 128, s.plane),
                       mb = sdesc(0, 128, s.gplane);
        const uint32_t w16 = w0 >> 4, r16 = ring0 >> 4;
        uint32_t n = 0, nu = 0;
        for (int u = blockIdx.x; u < units; u += gridDim.x, ++nu) {
            const uint32_t acc = nu % (uint32_t)s.nacc, use = nu / (uint32_t)s.nacc;
            if (use > 0)
                mbar_wait(bar_free + 8 * acc, (use - 1) & 1);
            const uint32_t d0 = tmem + acc * (a.tmem_cols / 2);
            const int i1 = min((u + 1) * per, s.items);
            int step = 0, set = 0;  // WGRAD2: K step of the unit, first column of its set
            for (int item = u * per; item < i1; ++item, ++n) {
                const int st = (int)(n % (uint32_t)s.nst);
                mbar_wait(bar_full + 8 * st, (n / (uint32_t)s.nst) & 1);
                tc_after_sync();
                const uint32_t base = r16 + st * stage16;
                if (KIND == WGRAD2) {
                    const int nk = ksteps_of(item);
                    // windows of 16 planes: all at shift (0, 0), blocks 1-2 one column
                    // on, 0-1 one row on, 1 both
                    constexpr int B = 3 * NC, n00 = (4 * B + 1 + 15) / 16, n2 = (2 * B + 15) / 16,
                                  n11 = (B + 15) / 16;
                    const uint32_t g0 = base + ((uint32_t)s.goff >> 4);
#pragma unroll 1
                    for (int j = 0, pos = 0, left = s.krow; j < nk; ++j, pos += 16, ++step) {
                        const uint32_t on = step >= s.nset;
                        const uint32_t dj = d0 + set;
                        set = set + s.accs == s.nset * s.accs ? 0 : set + s.accs;
                        const uint64_t b = mb + g0 + pos;
                        const uint32_t a0 = base + pos;
                        if (--left == 0) {  // krow > 0: the next row's first position
                            left = s.krow;
                            pos += s.P - s.Qx;
                        }
#pragma unroll
                        for (int k = 0; k < n00 + 2 * n2 + n11; ++k) {
                            const int sx = (k >= n00 && k < n00 + n2) || k >= n00 + 2 * n2;
                            const int sy = k >= n00 + n2;
                            const int p0 = k < n00               ? 16 * k
                                           : k < n00 + n2        ? B + 16 * (k - n00)
                                           : k < n00 + 2 * n2    ? 16 * (k - n00 - n2)
                                                                 : B + 16 * (k - n00 - 2 * n2);
                            tc_mma_if(one, dj + k * N, ma + a0 + p0 * pl + sy * P + sx, b, a.idesc,
                                      on);
                        }
                    }
                } else {
#pragma unroll 1
                    for (int m = 0; m < s.T; ++m) {
                        const uint32_t a0 = base + 128 * m, dm = d0 + m * s.accs;
                        if (KIND == DGRAD2) {
                            constexpr Runs runs{};
                            uint32_t b = w16;
#pragma unroll
                            for (int k = 0; k < kRuns; ++k) {
                                const ShiftRun r = runs.r[k];
                                const uint32_t id = id0 | ((uint32_t)r.n * (N >> 3) << 17);
                                const uint32_t sh = (r.shift >> 1 & 1) * P + (r.shift & 1);
#pragma unroll
                                for (int j = 0; j < NK16; ++j) {
                                    tc_mma_if(one, dm + r.pos * N,
                                              ka + a0 + ((r.shift >> 2) * NC + 2 * j) * pl + sh,
                                              kbd + b, id, !r.first || j != 0);
                                    b += r.n * N * 2;  // rows of 32 bytes
                                }
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < 27 * NK16; ++k) {
                                const int t = k / NK16, c16 = k % NK16;
                                int tz = t / 9, ty = t / 3 % 3, tx = t % 3, blk = 0;
                                if (KIND == DGRAD1)
                                    tz = 2 - tz, ty = 2 - ty, tx = 2 - tx;
                                if (KIND == FWD2) {
                                    // block of the tap's parities and its place in it
                                    const bool ey = ty == 1, ex = tx == 1;
                                    blk = ey ? (ex ? 3 : 2) : (ex ? 0 : 1);
                                    ty = ty == 2, tx = tx == 2;
                                }
                                tc_mma_if(one, dm,
                                          ka + a0 + ((blk * 3 + tz) * NC + 2 * c16) * pl + ty * P + tx,
                                          kb + w16 + (k / 4) * N * 8 + (k % 4) * 16, a.idesc, k != 0);
                            }
                        }
                    }
                }
                if (one)
                    tc_commit(bar_empty + 8 * st);
            }
            if (one)
                tc_commit(bar_acc + 8 * acc);
        }
        __syncwarp();
    } else {
        // ---- epilogue
        const int quarter = warp & 3, half = warp >> 2;
        const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
        // this lane's position in the two tiles
        const int l0 = quarter * 32 + lane, l1 = l0 + 128;
        const int r0 = l0 / s.P, x0 = l0 - r0 * s.P, r1 = l1 / s.P, x1 = l1 - r1 * s.P;
        const bool in0 = x0 < s.Qx && r0 < s.R, in1 = x1 < s.Qx && r1 < s.R;
        uint32_t nu = 0;
        for (int u = blockIdx.x; u < units; u += gridDim.x, ++nu) {
            const uint32_t acc = nu % (uint32_t)s.nacc;
            const uint32_t d0 = tmem + acc * (a.tmem_cols / 2) + lanes;
            if (KIND == WGRAD2) {
                mbar_wait(bar_acc + 8 * acc, (nu / (uint32_t)s.nacc) & 1);
                tc_after_sync();
                // row of window k: plane p0 + row / 8, element row % 8
                constexpr int B = 3 * NC;
                const int n00 = (4 * B + 1 + 15) / 16, n2 = (2 * B + 15) / 16;
                int sets = 0;  // that hold sums
                for (int item = u * per; item < min((u + 1) * per, s.items) && sets < s.nset; ++item)
                    sets = min(s.nset, sets + ksteps_of(item));
                for (int k = 0; k < s.nk; ++k) {
                    int sy = 0, sx = 0, p0 = 16 * k, b0 = 0, b1 = 4;
                    if (k >= n00 + 2 * n2)
                        sy = sx = 1, p0 = B + 16 * (k - n00 - 2 * n2), b0 = 1, b1 = 2;
                    else if (k >= n00 + n2)
                        sy = 1, p0 = 16 * (k - n00 - n2), b1 = 2;
                    else if (k >= n00)
                        sx = 1, p0 = B + 16 * (k - n00), b0 = 1, b1 = 3;
                    const int row = quarter * 32 + lane, p = p0 + (row >> 3);
                    const int blk = p / B, r = p - blk * B, zi = r / NC, c = r - zi * NC;
                    // blocks: (odd, even), (odd, odd), (even, odd), (even, even)
                    const int ty = blk >= 2 ? 1 : (sy ? 2 : 0);
                    const int tx = blk == 0 || blk == 3 ? 1 : (sx ? 2 : 0);
                    const bool ones = k < n00 && p == 4 * B && (row & 7) == 0;
                    const bool on = (blk >= b0 && blk < b1) || ones;
                    const int m = ones ? 27 * C : ((zi * 3 + ty) * 3 + tx) * C + c * 8 + (row & 7);
                    for (int c0 = 16 * half; c0 < a.N; c0 += 16 * PARTS) {
                        float v[16];
                        tc_load16(d0 + k * a.N + c0, v);
                        for (int q = 1; q < sets; ++q) {
                            float w[16];
                            tc_load16(d0 + q * s.accs + k * a.N + c0, w);
#pragma unroll
                            for (int e = 0; e < 16; ++e)
                                v[e] += w[e];
                        }
                        if (on)
                            epilogue_chunk<WGRAD>(a, (size_t)u * a.mtiles * 128 + m, v, c0, 0);
                    }
                }
            } else {
                int b, qz, y0;
                decode(u, b, qz, y0);
                // 16 columns at a time (this warp's chunks are PARTS apart); the ReLU factors
                // of the next chunk are loaded before the sums of this one are read
                constexpr bool BWD = KIND == DGRAD1 || KIND == DGRAD2;
                const int per_tile = (s.accs - 16 * half + 16 * PARTS - 1) / (16 * PARTS);
                struct Chunk {
                    size_t row;
                    int nn;
                    bool on;
                    uint4 mask[2];
                };
                // chunk j of this warp in tile m
                auto load = [&](int m, int j, Chunk &q) {
                    const int x = m ? x1 : x0, y = y0 + (m ? r1 : r0);
                    const int c0 = 16 * (half + PARTS * j);
                    bool on = (m ? in1 : in0) && y < s.Qy;
                    size_t row = 0;
                    int nn = c0;
                    if (KIND == DGRAD2) {
                        const int pc = on ? chunks[c0 >> 4] : 0, cls = pc & 7;
                        nn = pc >> 3;
                        const int z = 2 * qz + (cls >> 2), yy = 2 * y + ((cls >> 1) & 1),
                                  xx = 2 * x + (cls & 1);
                        on = on && z < a.D && yy < a.H && xx < a.W;
                        if (on)
                            row = vox_index(b, z, yy, xx, a.D, a.H, a.W);
                    } else if (on) {
                        row = (((size_t)b * s.Qz + qz) * s.Qy + y) * s.Qx + x;
                    }
                    q.nn = nn;
                    q.row = row;
                    q.on = on;
                    if (BWD && a.mask && on) {
                        const uint4 *p = reinterpret_cast<const uint4 *>(a.mask + row * a.N + nn);
                        if (a.wide) {
                            load32(p, q.mask);
                        } else {
                            q.mask[0] = __ldg(p);
                            q.mask[1] = __ldg(p + 1);
                        }
                    }
                };
                Chunk cur, nxt;
                if (per_tile > 0)
                    load(0, 0, cur);
                // every warp waits for the sums, also one that has no columns: the set
                // is free again when all of them have come by
                mbar_wait(bar_acc + 8 * acc, (nu / (uint32_t)s.nacc) & 1);
                tc_after_sync();
                int m = per_tile > 0 ? 0 : s.T, j = 0;
#pragma unroll 1
                while (m < s.T) {
                    int m2 = m, j2 = j + 1;
                    if (j2 >= per_tile) {
                        ++m2;
                        j2 = 0;
                    }
                    if (m2 < s.T)
                        load(m2, j2, nxt);
                    float v[16];
                    tc_load16(d0 + m * s.accs + 16 * (half + PARTS * j), v);
                    if (cur.on)
                        epilogue_chunk<BWD ? DGRAD : FWD>(a, cur.row, v, cur.nn, 0, cur.mask);
                    cur = nxt;
                    m = m2;
                    j = j2;
                }
            }
            tc_before_sync();
            mbar_arrive(bar_free + 8 * acc);
        }
    }
    __syncthreads();
    if (warp == 0)
        tmem_dealloc(tmem, a.tmem_cols);
}

// Weight slices in the shared-memory layout of the B operand: slice s holds
// rows n < N and K elements [64 s, 64 s + 64), K-major, zero beyond the real
// rows and K. mode 0 (forward): B[n = co][k = t cin + ci] = w[co][t][ci], the
// master layout's own order. mode 1 (dgrad, stride 1): B[n = ci][k = t cout
// + co] = w[co][t][ci]. mode 2 (dgrad, stride 2): the slices of the 8 parity
// classes one after the other, class c over its own taps in the order of
// class_tap.
__device__ __forceinline__ int class_ntaps(int cls)
{
    return (1 + ((cls >> 2) & 1)) * (1 + ((cls >> 1) & 1)) * (1 + (cls & 1));
}

// Tap t (0..26) of tap index ti of a parity class: per odd axis i = 0 is
// d = -1 and i = 1 is d = +1; an even axis has d = 0 only.
__device__ __forceinline__ int class_tap(int cls, int ti)
{
    const int cz = (cls >> 2) & 1, cy = (cls >> 1) & 1, cx = cls & 1;
    const int ny = 1 + cy, nx = 1 + cx;
    const int ix = ti % nx, iy = (ti / nx) % ny, iz = ti / (nx * ny);
    const int dz = cz ? 2 * iz - 1 : 0, dy = cy ? 2 * iy - 1 : 0, dx = cx ? 2 * ix - 1 : 0;
    return (dz + 1) * 9 + (dy + 1) * 3 + (dx + 1);
}

__global__ void k_pack_weights(const float *__restrict__ w, int cin, int cout, int N, int nslices,
                               int mode, __nv_bfloat16 *__restrict__ out)
{
    const int total = nslices * N * kBK;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        int s = e / (N * kBK);
        const int rem = e - s * N * kBK;
        const int g = rem / 512, r2 = rem - g * 512;
        const int kc = r2 / 64, r3 = r2 - kc * 64;
        const int n = g * 8 + r3 / 8;
        float val = 0.0f;
        if (mode == 0) {
            const int k = s * kBK + kc * 8 + (r3 & 7);
            if (n < cout && k < 27 * cin)
                val = w[(size_t)n * 27 * cin + k];
        } else if (mode == 1) {
            const int k = s * kBK + kc * 8 + (r3 & 7);
            if (n < cin && k < 27 * cout) {
                const int t = k / cout, co = k - t * cout;
                val = w[((size_t)co * 27 + t) * cin + n];
            }
        } else {
            int cls = 0;
            while (cls < 7) {
                const int ns = (class_ntaps(cls) * cout + kBK - 1) / kBK;
                if (s < ns)
                    break;
                s -= ns;
                ++cls;
            }
            const int k = s * kBK + kc * 8 + (r3 & 7);
            if (n < cin && k < class_ntaps(cls) * cout) {
                const int ti = k / cout, co = k - ti * cout;
                val = w[((size_t)co * 27 + class_tap(cls, ti)) * cin + n];
            }
        }
        out[e] = __float2bfloat16_rn(val);
    }
}

// Position of B[n][k] in a packed copy whose slices start at slice s0 and
// hold N rows: slice s0 + k / 64, group of 8 rows n / 8, chunk of 8 K
// elements (k % 64) / 8, row n % 8, element k % 8 (k_pack_weights' layout).
__device__ __forceinline__ int64_t packed_pos(int n, int k, int N, int s0)
{
    const int s = s0 + k / kBK, kk = k % kBK;
    return ((int64_t)s * N + (n / 8) * 8) * kBK + (kk / 8) * 64 + (n % 8) * 8 + (kk & 7);
}

// Adam on a network's flat parameters with k_adam_flat's update, writing each
// updated weight of the listed layers, rounded to bf16, to where
// k_pack_weights puts it: forward B[co][t cin + ci]; dgrad at stride 1
// B[ci][t cout + co]; at stride 2 B[ci][ti cout + co] in the slices of the
// tap's parity class (odd offsets on the axes of the class; ti the tap's index
// within it, x fastest). Each weight has one place per copy, so only real
// weights are written and the zero padding of the previous pack stays.
__global__ void k_adam_pack(AdamPackArgs a, const int64_t *__restrict__ step,
                            float *__restrict__ p, const float *__restrict__ g,
                            float *__restrict__ m, float *__restrict__ v)
{
    __shared__ float s_ib[2];
    if (threadIdx.x == 0) {
        const long long t = (long long)*step + 1;
        s_ib[0] = adam_inv_bias(a.adam.beta1, t);
        s_ib[1] = adam_inv_bias(a.adam.beta2, t);
    }
    __syncthreads();
    const float b1 = (float)a.adam.beta1, b2 = (float)a.adam.beta2;
    const float o1 = (float)(1.0 - a.adam.beta1), o2 = (float)(1.0 - a.adam.beta2);
    const float ib1 = s_ib[0], ib2 = s_ib[1];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.adam.n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float mm = m[i], vv = v[i];
        const float pn =
            adam_flat_update(p[i], g[i], mm, vv, b1, o1, b2, o2, a.adam.lr, a.adam.eps, ib1, ib2);
        p[i] = pn;
        m[i] = mm;
        v[i] = vv;
        for (int j = 0; j < a.nl; ++j) {
            const PackLayer &L = a.L[j];
            const int64_t r = i - L.off;
            const int K = 27 * L.cin;
            if (r < 0 || r >= (int64_t)L.cout * K)
                continue;
            const int co = (int)(r / K), k = (int)(r - (int64_t)co * K);
            const int t = k / L.cin, ci = k - t * L.cin;
            const __nv_bfloat16 b = __float2bfloat16_rn(pn);
            if (L.fwd)
                static_cast<__nv_bfloat16 *>(L.fwd)[packed_pos(co, k, L.cout, 0)] = b;
            if (L.dmode == 1) {
                static_cast<__nv_bfloat16 *>(L.dgrad)[packed_pos(ci, t * L.cout + co, L.cin, 0)] =
                    b;
            } else if (L.dmode == 2) {
                const int tz = t / 9, ty = (t / 3) % 3, tx = t % 3;
                const int cz = tz != 1, cy = ty != 1, cx = tx != 1;
                const int cls = (cz << 2) | (cy << 1) | cx;
                const int ti = ((cz ? tz / 2 : 0) * (1 + cy) + (cy ? ty / 2 : 0)) * (1 + cx) +
                               (cx ? tx / 2 : 0);
                static_cast<__nv_bfloat16 *>(L.dgrad)[packed_pos(ci, ti * L.cout + co, L.cin,
                                                                 L.cls0[cls])] = b;
            }
            break;
        }
    }
}

// g_w[co][t][ci] and g_b[co] from the wgrad partials [split][mrows][N]: one
// block of kReduceThreads per M row m = t cin + ci (m = 27 cin is the bias
// row). Thread j adds the splits j / N, j / N + G, ... of column co = j % N
// (G = kReduceThreads / N groups, coalesced reads of the N columns of a
// split), in order with compensated fp32 sums; the G group sums are then added in order
// by one thread per column, so the result does not depend on timing.
// With RECHECK the partials come from slabs whose K steps run through positions without an
// output, where a zero output gradient meets inputs that the weight does not read: an infinity
// or a NaN among those makes a sum NaN. Sums that are not finite are formed again from
// the voxels that they are of.
constexpr int kReduceThreads = 512;

// Compensated (Kahan) fp32 accumulation: the sum keeps about the precision of
// one rounding whatever the number of terms, with full-rate fp32 adds (FP64
// issues slowly on this part).
struct Kahan {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        const float y = x - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

struct RecheckArgs {
    const __nv_bfloat16 *act, *gout;
    int D, H, W, Do, Ho, Wo, stride, rows;
};

// The part of column co of M row m that voxels vox0, vox0 + step, ... give.
__device__ __forceinline__ float wgrad_voxels(const RecheckArgs &a, int m, int co, int N, int cin,
                                           int vox0, int step)
{
    const int t = m / cin, ci = m - t * cin;  // t = 27: the bias
    Kahan acc;
    for (int vox = vox0; vox < a.rows; vox += step) {
        int r = vox;
        const int x = r % a.Wo * a.stride - 1 + t % 3;
        r /= a.Wo;
        const int y = r % a.Ho * a.stride - 1 + t / 3 % 3;
        r /= a.Ho;
        const int z = r % a.Do * a.stride - 1 + t / 9;
        float in = t == 27 ? 1.0f : 0.0f;
        if (t < 27 && (unsigned)x < (unsigned)a.W && (unsigned)y < (unsigned)a.H &&
            (unsigned)z < (unsigned)a.D)
            in = __bfloat162float(a.act[vox_index(r / a.Do, z, y, x, a.D, a.H, a.W) * cin + ci]);
        acc.add(in * __bfloat162float(a.gout[(size_t)vox * N + co]));
    }
    return acc.s - acc.c;
}

// RECHECK: held to the registers of the plain form (four blocks per SM), so that the common
// case, in which every sum is finite, costs the same.
template <bool RECHECK>
__global__ void __launch_bounds__(kReduceThreads, RECHECK ? 4 : 1)
    k_wgrad_reduce(const float *__restrict__ part, int splits, int mrows, int N, int cin,
                   int cout, float *__restrict__ gw, float *__restrict__ gb,
                   const __grid_constant__ RecheckArgs a)
{
    __shared__ float red[kReduceThreads];
    const int m = blockIdx.x;
    const int groups = kReduceThreads / N;
    const int co = threadIdx.x % N, grp = threadIdx.x / N;
    Kahan acc;
    if (grp < groups) {
        const float *p = part + (size_t)m * N + co;
        const size_t step = (size_t)mrows * N;
        int sp = grp;
        // four independent loads in flight per thread, added in split order
        for (; sp + 3 * groups < splits; sp += 4 * groups) {
            const float a0 = p[(size_t)sp * step], a1 = p[(size_t)(sp + groups) * step],
                        a2 = p[(size_t)(sp + 2 * groups) * step],
                        a3 = p[(size_t)(sp + 3 * groups) * step];
            acc.add(a0);
            acc.add(a1);
            acc.add(a2);
            acc.add(a3);
        }
        for (; sp < splits; sp += groups)
            acc.add(p[(size_t)sp * step]);
    }
    red[threadIdx.x] = acc.s - acc.c;
    __syncthreads();
    const bool mine = threadIdx.x < N && co < cout;
    float v = 0.0f;
    if (mine) {
        Kahan tot;
        for (int gi = 0; gi < groups; ++gi)
            tot.add(red[gi * N + co]);
        v = tot.s - tot.c;
    }
    if constexpr (RECHECK) {
        if (__syncthreads_or(mine && !isfinite(v))) {
            red[threadIdx.x] = grp < groups ? wgrad_voxels(a, m, co, N, cin, grp, groups) : 0.0f;
            __syncthreads();
            if (mine && !isfinite(v)) {
                Kahan tot;
                for (int gi = 0; gi < groups; ++gi)
                    tot.add(red[gi * N + co]);
                v = tot.s - tot.c;
            }
        }
    }
    if (mine) {
        if (m < 27 * cin)
            gw[(size_t)co * 27 * cin + m] = v;
        else if (gb)
            gb[co] = v;
    }
}

// Split-K forward: out[row][n] = act(sum_p part[p][row][n] + bias[n]), the
// partitions added in order; bf16 or fp32 output.
__global__ void k_fwd_reduce(const float *__restrict__ part, int parts, int64_t rows, int N,
                             const float *__restrict__ bias, int relu, int out_f32,
                             void *__restrict__ out)
{
    const int64_t total = rows * N;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        float v = 0.0f;
        for (int p = 0; p < parts; ++p)
            v += part[(size_t)p * total + e];
        if (bias)
            v += __ldg(bias + (int)(e % N));
        if (relu)
            v = fmaxf(v, 0.0f);
        if (out_f32)
            static_cast<float *>(out)[e] = v;
        else
            static_cast<__nv_bfloat16 *>(out)[e] = __float2bfloat16_rn(v);
    }
}

uint32_t make_idesc(int N, bool mn_major)
{
    // kind::f16 instruction descriptor: D fp32 (bits 4-5 = 1), A and B bf16
    // (bits 7-9 = 1, 10-12 = 1), A/B major (bits 15, 16), N >> 3 (bits 17-22),
    // M >> 4 (bits 24-28), M = 128.
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)mn_major << 15) |
           ((uint32_t)mn_major << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

uint32_t tmem_cols_for(int N)
{
    uint32_t c = 32;
    while ((int)c < N)
        c <<= 1;
    return c;
}

// Dynamic shared memory: 1024-byte alignment slack, the ring's A and B
// slots, 2 kStages + 1 mbarriers, the TMEM address, the class tables, the tap
// offset tables and (WGRAD) the group table.
size_t conv_smem_bytes(int N, int groups)
{
    return 1024 + kStages * (size_t)kATile + kStages * (size_t)N * 128 + 8 * (2 * kStages + 1) +
           4 + 4 * (3 * kMaxClasses + 1) + sizeof(Tables) + 8 + groups * sizeof(int2);
}

// Parity classes of the stride-2 dgrad (host side): units, K slices and
// first packed slice of each class; returns the total number of units.
int dgrad_classes(const ConvLayer &l, int *unit0, int *nst, int *slice0, int *total_slices)
{
    int u = 0, sl = 0;
    for (int c = 0; c < kMaxClasses; ++c) {
        const int cz = (c >> 2) & 1, cy = (c >> 1) & 1, cx = c & 1;
        const int64_t rows = (int64_t)l.nb * ((l.D - cz + 1) / 2) * ((l.H - cy + 1) / 2) *
                             ((l.W - cx + 1) / 2);
        const int ntaps = (1 + cz) * (1 + cy) * (1 + cx);
        unit0[c] = u;
        nst[c] = (ntaps * l.cout + kBK - 1) / kBK;
        slice0[c] = sl;
        u += (int)((rows + 127) / 128);
        sl += nst[c];
    }
    unit0[kMaxClasses] = u;
    if (total_slices)
        *total_slices = sl;
    return u;
}

// What limits a kernel's resident CTAs on a device, found once per kernel and device.
struct KernelLimits {
    const void *fn;
    int dev, regs, fixed;  // registers of a thread; static and reserved shared memory of a CTA
    int smem_sm;
};

cudaError_t kernel_limits(const void *fn, KernelLimits *out)
{
    static std::mutex mu;
    static KernelLimits known[256];  // the kernels of this file on 8 devices
    static int n = 0;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    std::lock_guard<std::mutex> lk(mu);
    for (int k = 0; k < n; ++k)
        if (known[k].fn == fn && known[k].dev == dev) {
            *out = known[k];
            return cudaSuccess;
        }
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
    cudaFuncAttributes fa;
    if (e == cudaSuccess)
        e = cudaFuncGetAttributes(&fa, fn);
    int smem_sm = 0, resv = 0;
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&resv, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e != cudaSuccess)
        return e;
    *out = KernelLimits{fn, dev, fa.numRegs, (int)fa.sharedSizeBytes + resv, smem_sm};
    if (n < 256)
        known[n++] = *out;
    return cudaSuccess;
}

// Resident grid of a kernel of `threads` threads with `smem` bytes of dynamic shared memory and
// `cols` TMEM columns: shared memory with the largest carveout, registers, 512 TMEM columns per SM.
cudaError_t resident_grid(const void *fn, size_t smem, int cols, int threads, int units, int *grid)
{
    KernelLimits k;
    const cudaError_t e = kernel_limits(fn, &k);
    if (e != cudaSuccess)
        return e;
    const int by_smem = k.smem_sm / (int)(smem + k.fixed);
    const int by_regs = 65536 / ((k.regs * 32 + 255) / 256 * 256 * (threads / 32));
    const int occ = std::min(std::min(by_smem, by_regs), std::min(512 / cols, 16));
    if (occ < 1)
        return cudaErrorInvalidConfiguration;
    *grid = std::min(units, occ * device_sms());
    return cudaSuccess;
}

// Resident grid of k_conv<MODE>; *smem receives its dynamic shared memory.
template <int MODE>
cudaError_t conv_grid(const ConvArgs &a, int *grid, size_t *smem)
{
    *smem = conv_smem_bytes(a.N, MODE == WGRAD && a.cin != 2 ? 27 * (a.cin >> 3) : 0);
    return resident_grid((const void *)k_conv<MODE>, *smem, (int)a.tmem_cols, kThreads, a.units,
                         grid);
}

// The two-channel kernels are built for the output widths 16 and 32.
bool conv2_built(const ConvLayer &l) { return l.cin == 2 && (l.cout == 16 || l.cout == 32); }

// Host plan of a slab pass; false when no tiling of it fits (rows beyond 254
// positions, weights and two stages beyond a CTA's shared memory, TMEM columns).
bool slab_plan(int kind, int C, int N, int64_t nb, const int *S, const int *Q, SlabArgs *out,
               uint32_t *cols, size_t *smem)
{
    const bool s2 = kind == FWD2 || kind == WGRAD2;
    const int halo = kind == FWD1 || kind == DGRAD1 ? 2 : 1, nc = C / 8;
    bool found = false;
    double best_cost = 0.0;
    for (int R = std::min(Q[1], 256 / (Q[2] + halo)); R >= 1; --R) {
        SlabArgs s{};
        s.Sz = S[0], s.Sy = S[1], s.Sx = S[2];
        s.Qz = Q[0], s.Qy = Q[1], s.Qx = Q[2];
        s.P = s.Qx + halo;
        s.R = R;
        s.T = (s.R * s.P + 127) / 128;
        s.RB = s.R + halo;
        s.nzb = kind == DGRAD2 ? 2 : 3;
        s.plane = s.RB * s.P * 16;
        int sets = 1;  // accumulators of N columns
        if (kind == WGRAD2) {
            const int B = 3 * nc;
            s.nk = (4 * B + 1 + 15) / 16 + 2 * ((2 * B + 15) / 16) + (B + 15) / 16;
            s.ksteps = (s.R * s.P + 15) / 16;
            s.krow = s.Qx % 16 == 0 ? s.Qx / 16 : 0;
            s.gplane = s.ksteps * 256;
            s.goff = (4 * B + 1) * s.plane;
            s.stage = (s.goff + N / 8 * s.gplane + 127) / 128 * 128;
            sets = s.nk;
            s.T = 1;
            // the last window of 16 planes runs past the ones
            s.slack = ((4 * B + 1 + 15) / 16 * 16 - 4 * B) * s.plane;
        } else {
            s.nk = kind == DGRAD2 ? kRuns * C / 16 : 27 * C / 16;
            // a tile's rows past the band, shifted, read beyond the last plane
            s.stage = ((s2 ? 4 : 1) * s.nzb * nc * s.plane + 127) / 128 * 128;
            s.wbytes = kind == DGRAD2 ? 27 * C * N * 2 : (27 * C + 63) / 64 * 64 * N * 2;
            sets = kind == DGRAD2 ? 8 : 1;
        }
        s.accs = sets * N;
        // A weight adjoint drains its sums once per unit and needs no second buffer: its K
        // steps take what sets fit in turn, for chains of fewer roundings. (16 -> 32 channels,
        // 16 x 64^3, error against 64 bits: k_conv 1.16e-6 of the norm, one set 1.22e-6, two
        // 0.54e-6; the same time.)
        s.nacc = kind == WGRAD2 ? 1 : 2;
        s.nset = kind == WGRAD2 ? std::max(1, std::min(4, 512 / s.accs)) : 1;
        uint32_t c = 32;
        while ((int)c < s.nacc * s.nset * s.T * s.accs)
            c <<= 1;
        if (kind == DGRAD2 && 8 * N > 256)
            continue;  // the widest MMA
        const size_t fixed = 128 + (size_t)s.slack + (s.wbytes + 127) / 128 * 128 + 192;
        // reads past the last stage land in the weights and the table behind it
        const size_t past = kind == WGRAD2 ? 0 : (size_t)((halo * s.P + halo + s.T * 128) * 16);
        if (c > 512 || fixed + 2 * (size_t)s.stage > (size_t)kMaxDynSmem ||
            past > (size_t)s.RB * s.P * 16 + fixed - 192)
            continue;
        s.nst = (int)std::min<size_t>(4, ((size_t)kMaxDynSmem - fixed) / s.stage);
        // staged rows per output row, and the idle MMA rows; two stages alone leave
        // the staging's latency bare
        const double cost =
            ((double)(s2 ? 2 * s.R + 1 : s.RB) / s.R +
             (kind == WGRAD2 ? (double)s.ksteps * 16 : (double)s.T * 128) / (s.R * s.P)) *
            (s.nst > 2 ? 1.0 : 1.25);
        s.bands = (s.Qy + s.R - 1) / s.R;
        s.items = (int)(nb * s.Qz * s.bands);
        if (!found || cost < best_cost) {
            *out = s;
            *cols = c;
            *smem = fixed + (size_t)s.nst * s.stage;
            best_cost = cost;
            found = true;
        }
    }
    return found;
}

// Whether a planned slab beats k_conv, by the measured times of both (k_conv / slab in us,
// batch x size of the input). Short rows keep the staging (a warp per row) and the epilogue's
// 16-column accesses narrow; few bands do not repay the load of large weights or the zeroing of
// the ring:
//   WGRAD2 16 -> 32: 8x40x40x14 (7 outputs a row, bands of 18 and 2 rows) 23.6 / 28.9, x 20 (bands of
//          10) 29.7 / 26.8; 16x16x16x4 19.9 / 24.7, x 5 (bands of 8) 20.2 / 18.5.
//          32 -> 48: 1x32x32x32 (96 bands) 22.6 / 24.2, 16x16x16x32 33.0 / 27.5
//   DGRAD2 32 -> 16: 8x40x40x5 16.7 / 18.7, 16x16x16x5 18.7 / 13; 48 -> 32, 83 KB of weights:
//          8x40x40x12 31.0 / 34.6, 2x16x16x24 17.4 / 18.6, 16x16x16x16 20.9 / 18.5
//   DGRAD1 16 channels: 8x40x40x6 22.9 / 28.8, x 8 31.5 / 24; 48: 8x40x40x1 31.0 / 35.0
//   FWD1   16 channels: 8x40x40x3 17.1 / 18.3, x 4 18.8 / 16.5
// With two stages a band takes a latency of about 1.3 us + 0.04 us a channel, whatever its rows;
// k_conv a chain of 1.1 us a K slice or its copies at 3.75 TB/s: FWD2 48 -> 64 8x40x40x16
// 41.5 / 78.3, 16x16x16x14 31.1 / 21.3; FWD1 64 -> 48 8x40x40x20 262 / 319, x 16 209 / 179.
bool slab_pays(int kind, int C, int64_t rows, const SlabArgs &s)
{
    switch (kind) {
    case WGRAD2:
        // A single set's chains are no longer than k_conv's only without idle positions
        // (32 -> 48, 16 x 22 x 30 x 26: error 1.75e-7 of the norm, k_conv 1.49e-7)
        if (s.nset == 1 && s.krow == 0)
            return false;
        if (C == 32)
            return s.items >= 256;
        return s.Qx >= 9 || (s.Qx >= 3 && s.R <= 8);
    case DGRAD2:
        if (s.wbytes > 64 * 1024)
            return s.Qx >= 7 && s.items >= 64;
        return s.Qx >= 7 || s.items < 160;
    case DGRAD1:
        if (s.items >= 320 && s.Qx < (C == 16 ? 7 : 2))
            return false;
        break;
    case FWD1:
        if (s.items >= 320 && C == 16 && s.Qx > 1 && s.Qx < 4)
            return false;
        break;
    }
    if (s.nst > 2)
        return true;
    const double slab = 11.0 + (s.items + 151) / 152 * (1.3 + 0.0375 * C);
    return slab < std::max(8.0 + 1.1 * conv_slices(27 * C), 20.0 + 54e-6 / 3.75 * C * rows);
}

// Slab plan of a layer's weight adjoint for at most sp units; false when the layer takes k_conv.
bool wgrad_slab_plan(const ConvLayer &l, int sp, SlabArgs *s, int *units, uint32_t *cols,
                     size_t *smem)
{
    if (l.stride != 2 || (l.cin != 16 && l.cin != 32))
        return false;
    const int in[3] = {l.D, l.H, l.W};
    const int o[3] = {conv_out_size(l.D, 2), conv_out_size(l.H, 2), conv_out_size(l.W, 2)};
    if (!slab_plan(WGRAD2, l.cin, l.cout, l.nb, in, o, s, cols, smem) ||
        !slab_pays(WGRAD2, l.cin, 0, *s))
        return false;
    s->upu = (s->items + sp - 1) / sp;
    *units = (s->items + s->upu - 1) / s->upu;
    return true;
}

template <int C, int KIND>
cudaError_t run_slab(const ConvArgs &a, const SlabArgs &s, size_t smem, int units, cudaStream_t st)
{
    int grid = 0;
    const cudaError_t e = resident_grid((const void *)k_conv_slab<C, KIND>, smem,
                                        (int)a.tmem_cols, slab_threads(KIND), units, &grid);
    if (e != cudaSuccess)
        return e;
    ProfScope ps(st, KIND == WGRAD2 ? "k_conv_wgrad" : KIND == FWD1 || KIND == FWD2 ? "k_conv_fwd"
                                                                                  : "k_conv_dgrad");
    k_conv_slab<C, KIND><<<grid, slab_threads(KIND), smem, st>>>(a, s);
    return cudaGetLastError();
}

template <int C>
cudaError_t run_slab_kind(int kind, const ConvArgs &a, const SlabArgs &s, size_t smem,
                          cudaStream_t st)
{
    switch (kind) {
    case FWD1: return run_slab<C, FWD1>(a, s, smem, s.items, st);
    case FWD2: return run_slab<C, FWD2>(a, s, smem, s.items, st);
    case DGRAD1: return run_slab<C, DGRAD1>(a, s, smem, s.items, st);
    default: return run_slab<C, DGRAD2>(a, s, smem, s.items, st);
    }
}

// The weight adjoint as a slab when its plan says so (*ran), in at most *splits units. *splits
// receives the number of partial sums, which lie as k_wgrad_reduce reads them, and *recheck
// whether that has to look at sums that are not finite.
cudaError_t launch_wgrad_slab(const ConvLayer &l, ConvArgs a, cudaStream_t st, bool *ran,
                              int *splits, int *recheck)
{
    SlabArgs s;
    size_t smem = 0;
    uint32_t cols = 0;
    int units = 0;
    *ran = wgrad_slab_plan(l, *splits, &s, &units, &cols, &smem);
    if (!*ran)
        return cudaSuccess;
    s.src = a.act;
    s.src_elems = a.act_elems;
    a.tmem_cols = cols;
    a.units = *splits = units;
    *recheck = s.krow == 0;
    return l.cin == 16 ? run_slab<16, WGRAD2>(a, s, smem, a.units, st)
                       : run_slab<32, WGRAD2>(a, s, smem, a.units, st);
}

// Runs a forward pass or an input adjoint (a prepared) as a slab when it fits one; *ran says so.
cudaError_t launch_slab(int mode, const ConvLayer &l, ConvArgs a, cudaStream_t st, bool *ran)
{
    *ran = false;
    const int kind = mode == FWD ? (l.stride == 1 ? FWD1 : FWD2)
                                 : (l.stride == 1 ? DGRAD1 : DGRAD2);
    const int C = mode == DGRAD ? l.cout : l.cin;
    if (C != 16 && C != 32 && C != 48 && C != 64)
        return cudaSuccess;
    const int in[3] = {l.D, l.H, l.W}, o[3] = {a.Do, a.Ho, a.Wo};
    const int pairs[3] = {(l.D + 1) / 2, (l.H + 1) / 2, (l.W + 1) / 2};
    const int *S = mode == DGRAD ? o : in;
    const int *Q = mode == DGRAD ? (kind == DGRAD2 ? pairs : in) : o;
    SlabArgs s;
    size_t smem = 0;
    uint32_t cols = 0;
    if (!slab_plan(kind, C, a.N, l.nb, S, Q, &s, &cols, &smem) || !slab_pays(kind, C, a.rows, s))
        return cudaSuccess;
    a.tmem_cols = cols;
    s.src = a.act;
    s.src_elems = a.act_elems;
    *ran = true;
    switch (C) {
    case 16: return run_slab_kind<16>(kind, a, s, smem, st);
    case 32: return run_slab_kind<32>(kind, a, s, smem, st);
    case 48: return run_slab_kind<48>(kind, a, s, smem, st);
    default: return run_slab_kind<64>(kind, a, s, smem, st);
    }
}

template <int N, bool PAIR>
cudaError_t run_conv2(const ConvArgs &a, bool wgrad, cudaStream_t s)
{
    const size_t smem = wgrad ? 128 + 16 * kC2Plane + 32 : 128 + 10 * kC2Plane + 10 * N * 16 + 32;
    const void *fn = wgrad ? (const void *)k_conv2_wgrad<N, PAIR> : (const void *)k_conv2_fwd<N, PAIR>;
    int grid = 0;
    const cudaError_t e = resident_grid(fn, smem, 32, kThreads, a.units, &grid);
    if (e != cudaSuccess)
        return e;
    ProfScope ps(s, wgrad ? "k_conv_wgrad" : "k_conv_fwd");
    if (wgrad)
        k_conv2_wgrad<N, PAIR><<<grid, kThreads, smem, s>>>(a);
    else
        k_conv2_fwd<N, PAIR><<<grid, kThreads, smem, s>>>(a);
    return cudaGetLastError();
}

// PAIR's 8-byte loads need stride 2, an even W and an input on 8 bytes (it is on 16).
cudaError_t launch_conv2(const ConvArgs &a, bool wgrad, cudaStream_t s)
{
    const bool pair = a.stride == 2 && a.W % 2 == 0;
    if (a.N == 16)
        return pair ? run_conv2<16, true>(a, wgrad, s) : run_conv2<16, false>(a, wgrad, s);
    return pair ? run_conv2<32, true>(a, wgrad, s) : run_conv2<32, false>(a, wgrad, s);
}

int blocks_for(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    if (b > 32 * (int64_t)device_sms())  // grid-stride loops beyond this
        b = 32 * (int64_t)device_sms();
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

int conv_out_size(int n, int stride) { return (n - 1) / stride + 1; }

int conv_slices(int kreal) { return (kreal + kBK - 1) / kBK; }

size_t conv_packed_elems(const ConvLayer &l, int dgrad)
{
    if (!dgrad)
        return (size_t)conv_slices(27 * l.cin) * l.cout * kBK;
    if (l.stride == 1)
        return (size_t)conv_slices(27 * l.cout) * l.cin * kBK;
    int u0[kMaxClasses + 1], ns[kMaxClasses], s0[kMaxClasses], total = 0;
    dgrad_classes(l, u0, ns, s0, &total);
    return (size_t)total * l.cin * kBK;
}

void conv_wgrad_plan(const ConvLayer &l, int *mtiles, int *splits, int *kper)
{
    const int64_t V = (int64_t)l.nb * conv_out_size(l.D, l.stride) * conv_out_size(l.H, l.stride) *
                      conv_out_size(l.W, l.stride);
    const int mt = (27 * l.cin + 1 + 127) / 128;
    int64_t sp = (kTargetUnits + mt - 1) / mt;
    const int64_t max_sp = (V + kBK - 1) / kBK;
    if (sp > max_sp)
        sp = max_sp;
    if (sp < 1)
        sp = 1;
    int64_t kp = (V + sp - 1) / sp;
    kp = (kp + kBK - 1) / kBK * kBK;
    *mtiles = mt;
    *kper = (int)kp;
    *splits = (int)((V + kp - 1) / kp);
}

size_t conv_wgrad_ws_bytes(const ConvLayer &l)
{
    int mt, sp, kp;
    conv_wgrad_plan(l, &mt, &sp, &kp);
    return (size_t)sp * mt * 128 * l.cout * sizeof(float);
}

cudaError_t launch_conv_pack(const ConvLayer &l, const float *w, void *fwd, void *dgrad,
                             cudaStream_t s)
{
    ProfScope ps(s, "k_pack_weights");
    if (fwd) {
        const int nst = conv_slices(27 * l.cin);
        k_pack_weights<<<blocks_for((int64_t)nst * l.cout * kBK, 256), 256, 0, s>>>(
            w, l.cin, l.cout, l.cout, nst, 0, static_cast<__nv_bfloat16 *>(fwd));
    }
    if (dgrad) {
        const int nst = (int)(conv_packed_elems(l, 1) / ((size_t)l.cin * kBK));
        k_pack_weights<<<blocks_for((int64_t)nst * l.cin * kBK, 256), 256, 0, s>>>(
            w, l.cin, l.cout, l.cin, nst, l.stride == 1 ? 1 : 2,
            static_cast<__nv_bfloat16 *>(dgrad));
    }
    return cudaGetLastError();
}

void adam_pack_layer(const ConvLayer &l, int64_t off, void *fwd, void *dgrad, PackLayer *L)
{
    *L = PackLayer{};
    L->off = off;
    L->cin = l.cin;
    L->cout = l.cout;
    L->fwd = fwd;
    L->dgrad = dgrad;
    L->dmode = dgrad ? (l.stride == 1 ? 1 : 2) : 0;
    if (L->dmode == 2) {
        int u0[kMaxClasses + 1], ns[kMaxClasses];
        dgrad_classes(l, u0, ns, L->cls0, nullptr);
    }
}

cudaError_t launch_adam_pack(const AdamPackArgs &a, int64_t *step, float *p, const float *g,
                             float *m, float *v, cudaStream_t s)
{
    {
        ProfScope ps(s, "k_adam_pack");
        k_adam_pack<<<blocks_for(a.adam.n, 256), 256, 0, s>>>(a, step, p, g, m, v);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    return launch_step_tick(step, s);
}

static bool on32(const void *p) { return ((uintptr_t)p & 31u) == 0; }

static ConvArgs base_args(const ConvLayer &l)
{
    ConvArgs a = {};
    a.D = l.D;
    a.H = l.H;
    a.W = l.W;
    a.Do = conv_out_size(l.D, l.stride);
    a.Ho = conv_out_size(l.H, l.stride);
    a.Wo = conv_out_size(l.W, l.stride);
    a.cin = l.cin;
    a.cout = l.cout;
    a.stride = l.stride;
    a.classes = 1;
    return a;
}

// One class covering every unit, nst slices each.
static void single_class(ConvArgs &a, int nst)
{
    a.classes = 1;
    a.cls_unit0[0] = 0;
    a.cls_unit0[1] = a.units;
    a.cls_nst[0] = nst;
    a.cls_slice0[0] = 0;
}

// K partitions of the forward pass: split only when the tiles alone give
// fewer than two per SM of a 152-SM GB300, at least two K slices per
// partition, at most 8; a function of the shape only, so workspace sizes and
// launches agree.
int conv_fwd_splits(const ConvLayer &l)
{
    const int64_t rows = (int64_t)l.nb * conv_out_size(l.D, l.stride) *
                         conv_out_size(l.H, l.stride) * conv_out_size(l.W, l.stride);
    const int64_t tiles = (rows + 127) / 128;
    const int nst = conv_slices(27 * l.cin);
    if (tiles >= 2 * 152 || nst < 4)
        return 1;
    int64_t sp = (kTargetUnits + tiles - 1) / tiles;
    if (sp > nst / 2)
        sp = nst / 2;
    if (sp > kMaxClasses)
        sp = kMaxClasses;
    return sp < 2 ? 1 : (int)sp;
}

size_t conv_fwd_ws_bytes(const ConvLayer &l)
{
    const int sp = conv_fwd_splits(l);
    if (sp == 1)
        return 0;
    const int64_t rows = (int64_t)l.nb * conv_out_size(l.D, l.stride) *
                         conv_out_size(l.H, l.stride) * conv_out_size(l.W, l.stride);
    return (size_t)sp * rows * l.cout * sizeof(float);
}

cudaError_t launch_conv_forward(const ConvLayer &l, const void *in, const void *wpk,
                                const float *bias, int relu, int out_f32, void *out, void *ws,
                                cudaStream_t s)
{
    ConvArgs a = base_args(l);
    a.act_elems = (int64_t)l.nb * l.D * l.H * l.W * l.cin;
    a.act = static_cast<const __nv_bfloat16 *>(in);
    a.wpk = static_cast<const __nv_bfloat16 *>(wpk);
    a.bias = bias;
    a.out = out;
    a.N = l.cout;
    a.Kreal = 27 * l.cin;
    a.rows = l.nb * a.Do * a.Ho * a.Wo;
    const int tiles = (a.rows + 127) / 128;
    const int nst = conv_slices(a.Kreal);
    const int sp = ws ? conv_fwd_splits(l) : 1;
    if (sp == 1) {
        a.units = tiles;
        single_class(a, nst);
    } else {
        // K partitions as classes over the same tiles: partition p has the
        // slices [p nst / sp, (p + 1) nst / sp)
        a.part = static_cast<float *>(ws);
        a.classes = sp;
        for (int p = 0; p < sp; ++p) {
            a.cls_unit0[p] = p * tiles;
            a.cls_slice0[p] = p * nst / sp;
            a.cls_nst[p] = (p + 1) * nst / sp - p * nst / sp;
        }
        a.cls_unit0[sp] = sp * tiles;
        a.units = sp * tiles;
    }
    a.relu = relu;
    a.out_f32 = out_f32;
    a.wide = on32(out);
    a.idesc = make_idesc(a.N, false);
    a.tmem_cols = tmem_cols_for(a.N);
    if (conv2_built(l) && sp == 1)
        return launch_conv2(a, false, s);
    if (sp == 1) {
        bool ran = false;
        const cudaError_t e = launch_slab(FWD, l, a, s, &ran);
        if (ran)
            return e;
    }
    int grid = 0;
    size_t smem = 0;
    cudaError_t e = conv_grid<FWD>(a, &grid, &smem);
    if (e != cudaSuccess)
        return e;
    {
        ProfScope ps(s, "k_conv_fwd");
        k_conv<FWD><<<grid, kThreads, smem, s>>>(a);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess || sp == 1)
        return e;
    ProfScope ps(s, "k_fwd_reduce");
    k_fwd_reduce<<<blocks_for((int64_t)a.rows * a.N, 256), 256, 0, s>>>(
        a.part, sp, a.rows, a.N, bias, relu, out_f32, out);
    return cudaGetLastError();
}

cudaError_t launch_conv_dgrad(const ConvLayer &l, const void *gout, const void *wpk,
                              const void *mask, const void *addend, int add_stride, int add_off,
                              void *gin, cudaStream_t s)
{
    ConvArgs a = base_args(l);
    a.act_elems = (int64_t)l.nb * a.Do * a.Ho * a.Wo * l.cout;
    a.act = static_cast<const __nv_bfloat16 *>(gout);
    a.wpk = static_cast<const __nv_bfloat16 *>(wpk);
    a.mask = static_cast<const __nv_bfloat16 *>(mask);
    a.wide = on32(gin) && on32(mask);
    a.addend = static_cast<const __nv_bfloat16 *>(addend);
    a.add_stride = add_stride;
    a.add_off = add_off;
    a.out = gin;
    a.N = l.cin;
    a.Kreal = 27 * l.cout;
    a.rows = l.nb * l.D * l.H * l.W;
    if (l.stride == 1) {
        a.units = (a.rows + 127) / 128;
        single_class(a, conv_slices(a.Kreal));
    } else {
        a.classes = kMaxClasses;
        a.units = dgrad_classes(l, a.cls_unit0, a.cls_nst, a.cls_slice0, nullptr);
    }
    a.idesc = make_idesc(a.N, false);
    a.tmem_cols = tmem_cols_for(a.N);
    bool ran = false;
    cudaError_t e = launch_slab(DGRAD, l, a, s, &ran);
    if (ran)
        return e;
    int grid = 0;
    size_t smem = 0;
    e = conv_grid<DGRAD>(a, &grid, &smem);
    if (e != cudaSuccess)
        return e;
    ProfScope ps(s, "k_conv_dgrad");
    k_conv<DGRAD><<<grid, kThreads, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_conv_wgrad(const ConvLayer &l, const void *in, const void *gout, float *gw,
                              float *gb, void *ws, cudaStream_t s)
{
    ConvArgs a = base_args(l);
    a.act_elems = (int64_t)l.nb * l.D * l.H * l.W * l.cin;
    a.gout_elems = (int64_t)l.nb * a.Do * a.Ho * a.Wo * l.cout;
    int mt, sp, kp;
    conv_wgrad_plan(l, &mt, &sp, &kp);
    a.act = static_cast<const __nv_bfloat16 *>(in);
    a.gout = static_cast<const __nv_bfloat16 *>(gout);
    a.out = ws;
    a.N = l.cout;
    a.Kreal = kp;
    a.rows = l.nb * a.Do * a.Ho * a.Wo;
    a.mtiles = mt;
    a.units = mt * sp;
    single_class(a, kp / kBK);
    a.idesc = make_idesc(a.N, true);
    a.tmem_cols = tmem_cols_for(a.N);
    cudaError_t e;
    bool ran = false;
    int recheck = 0;
    if (conv2_built(l)) {
        e = launch_conv2(a, true, s);
    } else if ((e = launch_wgrad_slab(l, a, s, &ran, &sp, &recheck)) != cudaSuccess) {
        return e;
    } else if (!ran) {
        int grid = 0;
        size_t smem = 0;
        e = conv_grid<WGRAD>(a, &grid, &smem);
        if (e != cudaSuccess)
            return e;
        ProfScope ps(s, "k_conv_wgrad");
        k_conv<WGRAD><<<grid, kThreads, smem, s>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess)
        return e;
    ProfScope ps(s, "k_wgrad_reduce");
    // one block per M row (27 cin weights rows and the bias row)
    const RecheckArgs ra{a.act, a.gout, a.D, a.H, a.W, a.Do, a.Ho, a.Wo, a.stride, a.rows};
    auto *reduce = recheck ? k_wgrad_reduce<true> : k_wgrad_reduce<false>;
    reduce<<<27 * l.cin + 1, kReduceThreads, 0, s>>>(static_cast<const float *>(ws), sp, mt * 128,
                                                     a.N, l.cin, l.cout, gw, gb, ra);
    return cudaGetLastError();
}

int conv_device_error(bool clear)
{
    int h = 0;
    if (cudaMemcpyFromSymbol(&h, g_conv_error, sizeof(int)) != cudaSuccess)
        return -1;
    if (h != 0 && clear) {
        const int zero = 0;
        if (cudaMemcpyToSymbol(g_conv_error, &zero, sizeof(int)) != cudaSuccess)
            return -1;
    }
    return h;
}

AL_UNIT_ERROR_READER(unit_error_conv)

}  // namespace airgb
