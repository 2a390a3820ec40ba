// fmm_march.cu -- forward kernels of the restarted narrow band fast marching
// method (Yang & Stern), brick decomposition on one GB300 (sm_103a).
//
// Mapping of the paper's parallel algorithm (Sec. 4) onto the GPU:
//   subdomain Omega_p + ghost layer Theta_p  -> one 8x8x8 brick staged with its
//                                               face halo in shared memory
//   Initialize_Interface_Parallel (Alg. 8)  -> k_init_sources / k_init_reinit
//   Initialize_Heap_Parallel (Alg. 9)       -> k_march<mode 0> (one relax of
//                                               every cell next to a FIX cell)
//   local minima + AllReduce (Alg. 16)      -> k_reduce + k_control
//   March_Narrow_Band_Parallel (Alg. 12)    -> sweep_brick (fmm_sweep.cuh), run
//                                               by one of three restart
//                                               schedules (below)
//   Collect/Exchange/Integrate (Alg. 13-15) -> write-back to HBM plus the
//                                               smallest changed value and the
//                                               changed face in the neighbour's
//                                               work word; its next staging
//                                               reads the new values
//   second march of Alg. 16                 -> the neighbour is marched again
//                                               (queued, or listed as dirty)
//
// Restart schedules: continuous (k_march_queue: one launch for the whole
// solve, bricks from a device-side queue, the bound raised in the kernel when
// a restart runs out of parallel work), persistent (k_seed + k_march_queue with
// a fixed bound: one launch per restart) and phased (k_select + k_march<mode
// 1>: one launch per pass over a work list).
//
// A brick never solves cells it does not own: halo cells are read-only
// upwind data.  Every cell therefore has a single writer, and values only
// decrease, so a halo read that races with the owner's write-back can only
// return an upper bound; the owner then flags the change and the brick is
// marched again before termination can be declared.
#include "fmm_internal.h"
#include "fmm_queue.cuh"
#include "fmm_sweep.cuh"

#include <cfloat>
#include <cmath>
#include <math_constants.h>
#include <type_traits>

namespace fmmgb {
namespace {


__device__ __forceinline__ void brick_coords(const Geom &g, long long b, int &bx, int &by,
                                             int &bz)
{
    bx = (int)(b % g.nbx);
    long long r = b / g.nbx;
    by = (int)(r % g.nby);
    bz = (int)(r / g.nby);
}

// Brick across face f (0..5 = -x, +x, -y, +y, -z, +z) of brick b, or -1.  A
// batch of grids stores a neighbour table (no neighbour across the border of
// a grid); a single grid computes it from the brick coordinates.
__device__ __forceinline__ long long neighbour_brick(const Geom &g, const int *nbr, long long b,
                                                    int f)
{
    if (nbr)
        return (long long)nbr[b * kFaces + f];
    int bx, by, bz;
    brick_coords(g, b, bx, by, bz);
    const int axis = f >> 1, dir = (f & 1) ? 1 : -1;
    const int nbx = bx + (axis == 0 ? dir : 0);
    const int nby = by + (axis == 1 ? dir : 0);
    const int nbz = bz + (axis == 2 ? dir : 0);
    if (nbx < 0 || nbx >= g.nbx || nby < 0 || nby >= g.nby || nbz < 0 || nbz >= g.nbz)
        return -1;
    return ((long long)nbz * g.nby + nby) * g.nbx + nbx;
}

// ---------------------------------------------------------------------------
// Algorithm 8: interface initialisation, written directly in brick layout.
// ---------------------------------------------------------------------------

// The per-cell kernels below run one CTA of kInitThreads threads per brick
// (grid-stride over bricks), so the brick coordinates are computed once per
// brick, with 32-bit arithmetic (a grid has fewer than 2^31 bricks).
constexpr int kInitThreads = 256;

__device__ __forceinline__ void brick_xyz32(const Geom &g, int b, int &bx, int &by, int &bz)
{
    bx = b % g.nbx;
    const int r = b / g.nbx;
    by = r % g.nby;
    bz = r / g.nby;
}

template <typename real>
__global__ void __launch_bounds__(kInitThreads) k_init_sources(Geom g, real *T, uint8_t *tag)
{
    for (int b = blockIdx.x; b < (int)g.nbricks; b += gridDim.x) {
        int bx, by, bz;
        brick_xyz32(g, b, bx, by, bz);
        const long long base = (long long)b * kB3;
        for (int c = threadIdx.x; c < kB3; c += kInitThreads) {
            const int i = bx * kB + (c & 7), j = by * kB + ((c >> 3) & 7), k = bz * kB + (c >> 6);
            const bool out = i >= g.nx || j >= g.ny || k >= g.nz;
            T[base + c] = inf_v<real>();
            tag[base + c] = out ? (uint8_t)(TG_OUT | ST_FAR) : (uint8_t)ST_FAR;
        }
    }
}

template <typename real>
__global__ void k_set_sources(Geom g, const long long *src, long long n_src, real *T,
                              uint8_t *tag)
{
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n_src;
         s += (long long)gridDim.x * blockDim.x) {
        const int i = (int)src[3 * s], j = (int)src[3 * s + 1], k = (int)src[3 * s + 2];
        const long long b = ((long long)(k >> 3) * g.nby + (j >> 3)) * g.nbx + (i >> 3);
        const long long e = b * kB3 + (i & 7) + 8 * (j & 7) + 64 * (k & 7);
        T[e] = (real)0;
        tag[e] = ST_FIX;
    }
}

// Front cells of a level set: a 6-neighbour of the opposite sign marks the
// cell as adjacent to the interface; its value is sign * (sum_a d_a^-2)^-1/2
// with d_a the smaller linear-interpolation crossing distance on axis a.
__device__ __forceinline__ double rcp_sq(double d) { return __ddiv_rn(1.0, __dmul_rn(d, d)); }
__device__ __forceinline__ float rcp_sq(float d) { return 1.f / (d * d); }
__device__ __forceinline__ double inv_sqrt_exact(double v) { return __ddiv_rn(1.0, __dsqrt_rn(v)); }
__device__ __forceinline__ float inv_sqrt_exact(float v) { return 1.f / sqrtf(v); }
__device__ __forceinline__ double crossing(double fc, double fq, double h)
{
    return __dmul_rn(__ddiv_rn(fc, __dsub_rn(fc, fq)), h);
}
__device__ __forceinline__ float crossing(float fc, float fq, double h)
{
    return (fc / (fc - fq)) * (float)h;
}

__device__ __forceinline__ bool nonneg(double v)
{
    // sign bit clear, or -0, tested on the high word (and the low word for -0)
    const int hi = __double2hiint(v);
    return hi >= 0 || (hi == (int)0x80000000 && __double2loint(v) == 0);
}
__device__ __forceinline__ bool nonneg(float v)
{
    const unsigned b = __float_as_uint(v);
    return (b >> 31) == 0u || (b << 1) == 0u;
}

// Algorithm 8 for one cell (i, j, k) of an nx*ny*nz level set with cells of
// size hx * hy * hz (the crossing distance of an axis is a fraction of that
// axis's cell size).  The level set may extend zlo layers below z = 0 and zhi
// layers above z = nz - 1 (phi points at layer 0): a subdomain of a
// decomposed grid sees the layers beyond its ghost layers, so its interface
// cells are those of the whole grid.  reinit_load reads the cell and its six
// neighbours (a neighbour outside the grid reads the cell itself, which never
// changes sign), reinit_eval computes psi and the tag from them; a kernel
// issues the loads of all its cells before the first evaluation.
template <typename real>
__device__ __forceinline__ void reinit_load(const real *__restrict__ phi, int nx, int ny, int nz, int i,
                                            int j, int k, int zlo, int zhi, real &fc, real fn[6])
{
    const long long sx = 1, sy = nx, sz = (long long)nx * ny;
    const long long p = (long long)k * sz + (long long)j * sy + i;
    fc = phi[p];
    const int co[3] = {i, j, k};
    const int lo[3] = {0, 0, -zlo};
    const int ext[3] = {nx, ny, nz + zhi};
    const long long st[3] = {sx, sy, sz};
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int dir = s ? 1 : -1;
            const int q = co[a] + dir;
            const long long off = (q < lo[a] || q >= ext[a]) ? 0ll : (dir < 0 ? -st[a] : st[a]);
            fn[2 * a + s] = phi[p + off];
        }
}

template <typename real>
__device__ __forceinline__ void reinit_eval(real fc, const real fn[6], double hx, double hy, double hz,
                                            real &Tv, uint8_t &tg)
{
    const double hs[3] = {hx, hy, hz};
    // sign tests on the bit patterns (phi >= 0: sign bit clear, or -0): the
    // FP64 pipe's comparisons would bound the whole pass for double grids
    const bool pos = nonneg(fc);
    real d[3];
    bool any = false;
    bool cross[6];
#pragma unroll
    for (int n = 0; n < 6; ++n) {
        cross[n] = nonneg(fn[n]) != pos;
        any = any || cross[n];
    }
    if (!any) {
        Tv = inf_v<real>();
        tg = pos ? (uint8_t)ST_FAR : (uint8_t)(ST_FAR | TG_NEG);
        return;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        d[a] = inf_v<real>();
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (!cross[2 * a + s])
                continue;
            const real dist = crossing(fc, fn[2 * a + s], hs[a]);
            if (dist < d[a])
                d[a] = dist;
        }
    }
    real inv = (real)0;
    bool zero = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (d[a] == inf_v<real>())
            continue;
        if (d[a] == (real)0)
            zero = true;
        else
            inv = inv + rcp_sq(d[a]);
    }
    Tv = zero ? (real)0 : inv_sqrt_exact(inv);
    tg = pos ? (uint8_t)ST_FIX : (uint8_t)(ST_FIX | TG_NEG);
}

// Bits 0, 4, 8, ... of v as an 8-bit number.
__device__ __forceinline__ unsigned every_fourth(unsigned v)
{
    v &= 0x11111111u;
    v = (v | (v >> 3)) & 0x03030303u;
    v = (v | (v >> 6)) & 0x000f000fu;
    return (v | (v >> 12)) & 0xffu;
}

// Algorithm 8 takes two phases over the bricks of a CTA.  Almost no cell is at
// the interface, and telling which takes only signs: in the first phase one warp
// per brick has a lane read the 16 cells of its slots (x = lane & 7, y = lane / 8 +
// 4 (k & 1), z = k / 2) and 12 cells of the face halo, keep their signs as bits,
// and get the neighbours' signs by shifts, shuffles and ballots; the other cells
// are written at once.  The interface cells of all bricks of the CTA go to one
// list, and in the second phase the CTA's threads run reinit_load / reinit_eval on
// it: a cell takes a chain of IEEE divisions and a root (5 us in double), so a
// brick's 100 to 200 of them are spread over the CTA.
// This kernel, float / double: 33x36x40 (150 bricks, one per CTA) 6.0 / 13.3 us,
// 256^3 48 / 118 us.  With one cell a thread and seven loads for each 5.0 / 17.5 and
// 103 / 298 us; with each lane of the first phase evaluating its own interface
// cells 14.3 / 52.6 and 56 / 194 us.  Whole solves against that last form:
// 1024^3 in double 56.5 -> 55.3 ms, 256 grids of 32^3 to 192^3 in float the same.
// One brick of a level set: the caller's array with its sizes and cell sizes (a
// subdomain's layers beyond its own, see above) and the brick's coordinates.
template <typename real>
struct ReinitBrick {
    const real *phi;
    int nx, ny, nz, bx, by, bz;
    double hx, hy, hz;
    int zlo, zhi;
};

// First phase, one warp: writes the cells that are not at the interface, returns
// the slots of this lane that are.
template <typename real>
__device__ __forceinline__ unsigned reinit_signs(const ReinitBrick<real> &B, real *__restrict__ T,
                                                 uint8_t *__restrict__ tag)
{
    const real *__restrict__ phi = B.phi;
    const int nx = B.nx, ny = B.ny, nz = B.nz, bx = B.bx, by = B.by, zlo = B.zlo, zhi = B.zhi;
    constexpr unsigned kAll = 0xffffffffu, kEven = 0x5555u, kOdd = 0xaaaau;
    const int lane = threadIdx.x & 31, lx = lane & 7, lr = lane >> 3;
    const long long sy = nx, sz = (long long)nx * ny;
    const int i0 = bx * kB, j0 = by * kB, k0 = B.bz * kB;
    const int i = i0 + lx, j = j0 + lr;
    const real *col = phi + (long long)k0 * sz + (long long)j * sy + i;
    const bool in_x = i < nx, in_y0 = in_x && j < ny, in_y1 = in_x && j + 4 < ny;
    const int depth = nz + zhi - k0;   // readable layers from the brick's first one on
    real v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const bool ok = ((k & 1) ? in_y1 : in_y0) && (k >> 1) < depth;
        v[k] = ok ? col[(k >> 1) * sz + ((k & 1) ? 4 * sy : 0)] : (real)0;
    }
    // the faces: cell (u, w) = (lane & 7, lane / 8 + 4 h) of the face's plane
    real f[12];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int u = lx, w = lr + 4 * h;
        const bool yz = j0 + u < ny && w < depth, xz = i0 + u < nx && w < depth, xy = h ? in_y1 : in_y0;
        const real *px = phi + (long long)(k0 + w) * sz + (long long)(j0 + u) * sy + i0;
        const real *py = phi + (long long)(k0 + w) * sz + (long long)j0 * sy + i0 + u;
        const real *pz = col + (h ? 4 * sy : 0);
        f[h] = yz && bx > 0 ? px[-1] : (real)0;
        f[2 + h] = yz && i0 + kB < nx ? px[kB] : (real)0;
        f[4 + h] = xz && by > 0 ? py[-sy] : (real)0;
        f[6 + h] = xz && j0 + kB < ny ? py[kB * sy] : (real)0;
        f[8 + h] = xy && k0 > -zlo ? pz[-sz] : (real)0;
        f[10 + h] = xy && depth > kB ? pz[kB * sz] : (real)0;
    }
    unsigned S = 0, zm = 0, zp = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k)
        S |= (unsigned)nonneg(v[k]) << k;
    // x and y faces as 64 bits, bit u + 8 w; a lane at the face takes its
    // own row (16 slots) or column (the 8 even or odd slots)
    unsigned face[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const unsigned b0 = __ballot_sync(kAll, nonneg(f[2 * a])), b1 = __ballot_sync(kAll, nonneg(f[2 * a + 1]));
        const int sh = a < 2 ? lr : lx;
        const unsigned keep = a < 2 ? 0x11111111u : 0x01010101u;
        face[a] = every_fourth((b0 >> sh) & keep) | (every_fourth((b1 >> sh) & keep) << 8);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        zm |= (unsigned)nonneg(f[8 + h]) << h;
        zp |= (unsigned)nonneg(f[10 + h]) << (14 + h);
    }
    const unsigned xm = __shfl_up_sync(kAll, S, 1), xp = __shfl_down_sync(kAll, S, 1);
    const unsigned ym = __shfl_sync(kAll, S, (lane + 24) & 31), yp = __shfl_sync(kAll, S, (lane + 8) & 31);
    const unsigned nxm = lx == 0 ? face[0] : xm, nxp = lx == kB - 1 ? face[1] : xp;
    const unsigned nym = lr == 0 ? ((ym << 1) & kOdd) | face[2] : ym;
    const unsigned nyp = lr == 3 ? ((yp >> 1) & kEven) | (face[3] << 1) : yp;
    // slots whose neighbour is in the level set
    const int up = depth - 1 < 0 ? 0 : depth - 1 > kB ? kB : depth - 1, in_z = nz - k0 > kB ? kB : nz - k0;
    const unsigned oxm = i > 0 ? 0xffffu : 0u, oxp = i + 1 < nx ? 0xffffu : 0u;
    const unsigned oym = (j > 0 ? kEven : 0u) | kOdd;
    const unsigned oyp = (j + 1 < ny ? kEven : 0u) | (j + 5 < ny ? kOdd : 0u);
    const unsigned ozm = k0 > -zlo ? 0xffffu : 0xfffcu, ozp = (1u << (2 * up)) - 1u;
    const unsigned in = ((in_y0 ? kEven : 0u) | (in_y1 ? kOdd : 0u)) & ((1u << (2 * in_z)) - 1u);
    const unsigned cross = in & (((nxm ^ S) & oxm) | ((nxp ^ S) & oxp) | ((nym ^ S) & oym) | ((nyp ^ S) & oyp) |
                                 ((((S << 2) | zm) ^ S) & ozm) | ((((S >> 2) | zp) ^ S) & ozp));
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if ((cross >> k) & 1u)
            continue;
        T[lane + 32 * k] = inf_v<real>();
        tag[lane + 32 * k] = !((in >> k) & 1u) ? (uint8_t)(TG_OUT | ST_FAR)
                             : ((S >> k) & 1u) ? (uint8_t)ST_FAR
                                               : (uint8_t)(ST_FAR | TG_NEG);
    }
    return cross;
}

// Both phases for bricks first .. first + count - 1 (at most one per warp of the
// CTA): info(b) gives a brick, or a null phi for one without a level set, whose
// cells it has written.
struct ReinitList {
    int n;
    uint16_t cell[kInitThreads / 32 * kB3];   // warp of the brick << 9 | cell
};
template <typename real, typename Info>
__device__ __forceinline__ void reinit_bricks(int first, int count, Info &&info, real *__restrict__ T,
                                              uint8_t *__restrict__ tag, ReinitList &L)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0)
        L.n = 0;
    __syncthreads();
    if (warp < count) {
        const ReinitBrick<real> B = info(first + warp);
        const long long base = (long long)(first + warp) * kB3;
        const unsigned cross = B.phi ? reinit_signs<real>(B, T + base, tag + base) : 0u;
        const int cnt = __popc(cross);
        int pre = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, pre, o);
            if (lane >= o)
                pre += t;
        }
        int at = 0;
        if (lane == 31 && pre)
            at = atomicAdd(&L.n, pre);
        at = __shfl_sync(0xffffffffu, at, 31) + pre - cnt;
        for (unsigned m = cross; m; m &= m - 1u)
            L.cell[at++] = (uint16_t)(warp << 9 | (lane + 32 * (__ffs(m) - 1)));
    }
    __syncthreads();
    for (int l = threadIdx.x; l < L.n; l += blockDim.x) {
        const int b = first + (L.cell[l] >> 9), c = L.cell[l] & (kB3 - 1);
        const ReinitBrick<real> B = info(b);
        real fc, fn[6], Tv;
        uint8_t tg;
        reinit_load<real>(B.phi, B.nx, B.ny, B.nz, B.bx * kB + (c & 7), B.by * kB + ((c >> 3) & 7),
                          B.bz * kB + (c >> 6), B.zlo, B.zhi, fc, fn);
        reinit_eval<real>(fc, fn, B.hx, B.hy, B.hz, Tv, tg);
        T[(long long)b * kB3 + c] = Tv;
        tag[(long long)b * kB3 + c] = tg;
    }
    __syncthreads();   // the list of the next bricks
}

template <typename real>
__global__ void __launch_bounds__(kInitThreads) k_init_reinit(Geom g, double hx, double hy, double hz,
                                                              const real *__restrict__ phi, real *T,
                                                              uint8_t *tag, int zlo, int zhi, int group)
{
    __shared__ ReinitList list;
    const auto info = [&](int b) {
        ReinitBrick<real> B = {phi, g.nx, g.ny, g.nz, 0, 0, 0, hx, hy, hz, zlo, zhi};
        brick_xyz32(g, b, B.bx, B.by, B.bz);
        return B;
    };
    for (long long b = (long long)blockIdx.x * group; b < g.nbricks; b += (long long)gridDim.x * group)
        reinit_bricks<real>((int)b, (int)min((long long)group, g.nbricks - b), info, T, tag, list);
}

// Speed field to brick layout: the speed term (h/F)^2 of the shifted solve
// (h the x cell size).  Each brick also records its bucket width
// hmin * min(1/F) / sqrt(3), hmin the smallest cell size.
__device__ __forceinline__ double speed_term(double F, double h) { return (h * h) / (F * F); }
__device__ __forceinline__ float speed_term(float F, double h)
{
    const float hf = (float)h;
    return (hf * hf) / (F * F);
}

template <typename real>
__global__ void __launch_bounds__(kThreads) k_load_speed(Geom g, double h, double hmin,
                                                         const real *__restrict__ speed,
                                                         double speed_const, real *spd, real *bdelta,
                                                         Control *ctrl)
{
    __shared__ real red[kThreads / 32];
    const int t = threadIdx.x;
    for (long long b = blockIdx.x; b < g.nbricks; b += gridDim.x) {
        int bx, by, bz;
        brick_coords(g, b, bx, by, bz);
        const int i = bx * kB + (t & 7), j = by * kB + ((t >> 3) & 7), k = bz * kB + (t >> 6);
        const bool out = i >= g.nx || j >= g.ny || k >= g.nz;
        real F = (real)speed_const;
        if (speed && !out)
            F = speed[((long long)k * g.ny + j) * g.nx + i];
        if (out)
            F = (real)1;
        // F = 0: an obstacle cell, whose speed term (h/F)^2 is +inf, so no
        // solve ever gives it a finite value
        if (!(F >= (real)0) || !(F < inf_v<real>()))
            atomicOr(&ctrl->error, ERR_SPEED);
        if (spd)
            spd[b * kB3 + t] = speed_term(F, h);
        real fm = out ? (real)0 : F;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            fm = fmax(fm, __shfl_xor_sync(0xffffffffu, fm, o));
        if ((t & 31) == 0)
            red[t >> 5] = fm;
        __syncthreads();
        if (t == 0) {
            real m = red[0];
            for (int w = 1; w < kThreads / 32; ++w)
                m = fmax(m, red[w]);
            if (!(m > (real)0))
                m = (real)speed_const;
            bdelta[b] = (real)(hmin / (1.7320508075688772 * (double)m));
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// The brick march (fmm_sweep.cuh): one warp per brick, four bricks per CTA.  It
// is bound by the length of a brick's chain of steps where a grid has few
// bricks per warp, and by the ALU (float) and FP64 (double) pipes where it has
// many.  256^3 level set of 32 spheres, whole call: 2.1 ms in float, 5.0 ms in
// double (5.7 and 12.0 ms with the bucketed march this replaced); 1024^3 sphere
// in double 55 ms (236 ms).
// ---------------------------------------------------------------------------

#ifndef FMM_MARCH_BLOCKS_F32
#define FMM_MARCH_BLOCKS_F32 7
#endif
#ifndef FMM_MARCH_BLOCKS_F64
#define FMM_MARCH_BLOCKS_F64 5
#endif
#ifndef FMM_MARCH_BLOCKS_F64_TAPE
#define FMM_MARCH_BLOCKS_F64_TAPE 5
#endif
// Resident CTAs per SM the march kernels are compiled for (registers).  The warp
// tiles (5.7 / 6.2 KB in float, 9.7 / 10.2 KB in double, without / with the tape)
// and the sweep order (4 KB a CTA) allow these as well; six fp64 CTAs of 43 KB
// would not fit the 227 KB of an SM.
template <typename real, bool kTape>
constexpr int march_min_blocks()
{
    return sizeof(real) == 4 ? FMM_MARCH_BLOCKS_F32 : (kTape ? FMM_MARCH_BLOCKS_F64_TAPE : FMM_MARCH_BLOCKS_F64);
}
// Shared memory of a march CTA.
template <typename real, bool kTape>
struct MarchSmem {
    WarpTile<real, kTape> tile[kMarchWarps];
    int order[(kSweepSteps + 1) * 32];
};

__device__ __forceinline__ void flush_stats(Control *ctrl, MarchStats &st, int lane)
{
    const unsigned ex = __reduce_add_sync(FULL, (unsigned)st.exchanges);
    if (lane == 0 && st.marches) {
        atomicAdd(&ctrl->marches, st.marches);
        atomicAdd(&ctrl->rounds, st.rounds);
        atomicAdd(&ctrl->accepted, st.accepted);
        atomicAdd(&ctrl->solves, st.solves);
        atomicAdd(&ctrl->exchanges, (unsigned long long)ex);
    }
}
__device__ __forceinline__ unsigned long long vloadu(const unsigned long long *p)
{
    return *(const volatile unsigned long long *)p;
}

// Put brick b at position t of the ready queue or the waiting ring (waits,
// bounded, for a queue slot still being read; the waiting ring has a free slot
// for every append, fmm_ring.h).  own: a queue ticket this warp holds while it
// scans, or -1.  Its entry would stay unread for as long as this waits, and the
// slot waited for can be that very one (a raise that queues nearly every brick,
// and marches that queue some again meanwhile): the wait takes the entry out,
// into held.
__device__ __forceinline__ void ring_put(Control *c, unsigned long long *q, unsigned long long cap,
                                         unsigned long long t, long long b, long long own, long long &held)
{
    const unsigned long long v = ((t & 0xffffffffull) << 32) | (unsigned long long)(b + 1);
    unsigned long long *slot = q + (t % cap);
    if (atomicCAS(slot, 0ull, v) == 0ull)
        return;
    const unsigned long long ts = device_ns(), lim = vload(&c->wait_ns);
    while (atomicCAS(slot, 0ull, v) != 0ull) {
        if (own >= 0) {
            unsigned long long *mine = q + (unsigned long long)own % cap;
            const unsigned long long e = vloadu(mine);
            if (e != 0ull && (e >> 32) == ((unsigned long long)own & 0xffffffffull) && atomicCAS(mine, e, 0ull) == e)
                held = (long long)(e & 0xffffffffull) - 1;
        }
        if (device_ns() - ts > lim || (vload((const int *)&c->error) & ERR_SPIN)) {
            atomicOr(&c->error, ERR_SPIN);
            break;
        }
        __nanosleep(32);
    }
}

// ---------------------------------------------------------------------------
// The brick scheduler of the one-launch schedules.
//
// work[b] is one 64-bit word per brick: the smallest work the brick has (the
// smallest changed halo value flagged to it, or its own smallest BAND value;
// a float, rounded down) and two flags.  kWorkActive: the brick is in the
// ready queue or being marched.  kWorkWaiting: the waiting ring holds an entry
// of it.  Every transition is one atomic on that word, so a brick is queued
// once, marched by one warp, and no change is lost:
//   a march that changed a face lowers the neighbour's value and, if the
//   neighbour is not active, makes it active and queues it (value at or below
//   the bound) or leaves it in the waiting ring;
//   the warp that pops a brick takes the value (+inf in its place) before it
//   reads the halo, and at the end of the march a value that arrived
//   meanwhile keeps the brick active or sends it to the ring.
// ---------------------------------------------------------------------------
constexpr unsigned kWorkActive = 1u, kWorkWaiting = 2u, kWorkFull = 4u, kWorkFace = 8u;
constexpr unsigned kNoWork = 0x7f800000u;   // +inf

__device__ __forceinline__ unsigned long long work_word(unsigned key, unsigned flags)
{
    return ((unsigned long long)key << 32) | flags;
}
__device__ __forceinline__ unsigned work_key(float v) { return __float_as_uint(v); }
__device__ __forceinline__ unsigned work_key(double v) { return __float_as_uint(__double2float_rd(v)); }

// Take brick b from the queue: forget the work recorded so far, then read its
// halo.  Lane 0 acquires and the barrier after it orders every lane's loads
// behind that (a shuffle alone orders no memory): the word is cleared, so a load
// that missed a recorded value would lose it.  (A fence in every lane as well
// took 1 to 2% of the whole solves.)  Returns the changed faces (bit f), all ones
// for kWorkFull.
__device__ __forceinline__ unsigned take_brick(const DeviceState &s, long long b, int lane)
{
    unsigned fl = 0;
    if (lane == 0) {
        unsigned long long old = vloadu(&s.work[b]);
        for (;;) {
            const unsigned long long nw = work_word(kNoWork, (unsigned)old & (kWorkActive | kWorkWaiting));
            unsigned long long was;
            asm volatile("atom.acquire.gpu.global.cas.b64 %0, [%1], %2, %3;"
                         : "=l"(was)
                         : "l"(s.work + b), "l"(old), "l"(nw)
                         : "memory");
            if (was == old)
                break;
            old = was;
        }
        fl = (unsigned)old;
    }
    __syncwarp();
    fl = __shfl_sync(FULL, fl, 0);
    return (fl & kWorkFull) ? ~0u : fl / kWorkFace;
}

// The end of a march of brick b (written back by all lanes): lane f < 6 with a
// changed face flags the neighbour, lane kFaces ends the brick's own march,
// and the warp queues and rings what they claimed.  `bound` is the level the
// marches start at (a stale one only delays a start), kAll: no level, every
// flagged brick is queued.  `pending` changes once: the bricks queued less
// this one, after ring entries are counted and before queue slots are filled,
// so it reaches zero only with nothing queued, marching or unrecorded.
template <typename real, bool kAll>
__device__ __forceinline__ void finish_brick(const DeviceState &s, unsigned long long cap, double width, long long b,
                                             const Notify<real> &nt, int lane)
{
    Control *c = s.ctrl;
    float bound = __uint_as_float(kNoWork);
    if (!kAll)
        bound = *(const volatile float *)&c->level[(vloadu(&c->scan_word) >> 32) & 1u].bound;
    // all lanes' write-back before any lane's flags: the barrier, then each lane's
    // fence before its atomic
    __syncwarp();
    fence_acq_rel();
    long long tb = -1;        // the brick whose word this lane updates
    unsigned key = kNoWork;   // work to record
    if (nt.m) {
        tb = nt.nb;
        key = work_key(vmin(nt.v[0], nt.v[1]));
    } else if (lane == kFaces) {
        tb = b;
        const real band = vmin(nt.band[0], nt.band[1]);
        if (!kAll && (double)band <= width)
            key = work_key(band);
    }
    int act = 0;   // 1: queue tb, 2: append it to the waiting ring
    if (tb >= 0) {
        unsigned long long old = vloadu(&s.work[tb]);
        for (;;) {
            const unsigned k = umin((unsigned)(old >> 32), key);
            unsigned fl = (unsigned)old;
            act = 0;
            if (nt.m)
                fl |= kWorkFace << (lane ^ 1);
            else {
                fl &= ~kWorkActive;
                if (key < kNoWork)
                    fl |= kWorkFull;
            }
            if (!(fl & kWorkActive) && k < kNoWork) {
                if (__uint_as_float(k) <= bound) {
                    fl |= kWorkActive;
                    act = 1;
                } else if (!(fl & kWorkWaiting)) {
                    fl |= kWorkWaiting;
                    act = 2;
                }
            }
            const unsigned long long was = atomicCAS(&s.work[tb], old, work_word(k, fl));
            if (was == old)
                break;
            old = was;
        }
    }
    const unsigned bq = __ballot_sync(FULL, act == 1), bw = __ballot_sync(FULL, act == 2);
    unsigned long long tq = 0, tw = 0;
    if (lane == 0) {
        const int n = __popc(bq);
        if (bw)
            tw = atomicAdd(&c->w_tail, (unsigned long long)__popc(bw));
        if (n != 1) {
            __threadfence();   // ring entries counted, words released
            atomicAdd(&c->pending, n - 1);
        }
        if (n)
            tq = atomicAdd(&c->q_tail, (unsigned long long)n);
    }
    if (bq | bw) {
        tq = __shfl_sync(FULL, tq, 0);
        tw = __shfl_sync(FULL, tw, 0);
        const unsigned below = (1u << lane) - 1u;
        long long none = -1;   // (a warp that marches holds no ticket)
        if (act == 1)
            ring_put(c, s.queue, cap, tq + __popc(bq & below), tb, -1, none);
        else if (act == 2)
            ring_put(c, s.waiting, waiting_slots((long long)cap), tw + __popc(bw & below), tb, -1, none);
    }
    __syncwarp();
}

// Phased march: kMode 0 runs Algorithm 9 over all bricks; kMode 1 runs
// Algorithm 12 up to the restart bound over the bricks of work list `which`
// (taken one at a time from a shared counter); changes are flagged in the
// neighbours' dirty flags.
template <typename real, bool kHetero, int kMode, bool kTape, bool kAniso>
__global__ void __launch_bounds__(kMarchWarps * 32, march_min_blocks<real, kTape>())
    k_march(Geom g, DeviceState s, SolveParams p, double spd_const_term, int which)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    MarchSmem<real, kTape> &sm = *reinterpret_cast<MarchSmem<real, kTape> *>(smem_raw);
    WarpTile<real, kTape> &W = sm.tile[warp];
    Control *ctrl = s.ctrl;
    if constexpr (kMode == 0) {
        for (long long b = (long long)blockIdx.x * kMarchWarps + warp; b < g.nbricks;
             b += (long long)gridDim.x * kMarchWarps) {
            long long nbi[kFaces];
#pragma unroll
            for (int f = 0; f < kFaces; ++f)
                nbi[f] = neighbour_brick(g, s.nbr, b, f);
            // Algorithm 9 only changes cells next to a FIX cell: a brick with
            // no FIX cell in it or in its six neighbours keeps the state of
            // Algorithm 8 and has no BAND cell (one 16-byte load of tags per
            // lane and brick decides)
            bool fixnear = false;
#pragma unroll
            for (int f = -1; f < kFaces; ++f) {
                const long long q = f < 0 ? b : nbi[f < 0 ? 0 : f];
                if (q < 0)
                    continue;
                const uint4 t4 = reinterpret_cast<const uint4 *>(s.tag + q * kB3)[lane];
                const unsigned w = (t4.x & (t4.x >> 1)) | (t4.y & (t4.y >> 1)) | (t4.z & (t4.z >> 1)) |
                                   (t4.w & (t4.w >> 1));
                fixnear = fixnear || (w & 0x01010101u) != 0u;   // a byte with status ST_FIX (3)
            }
            if (!__any_sync(FULL, fixnear)) {
                if (lane < 2)
                    ((real *)s.bmin)[2 * b + lane] = inf_v<real>();
                continue;
            }
            front_brick<real, kHetero, kTape, kAniso>(s, p, spd_const_term, W, b, nbi, lane);
            __syncwarp();
        }
    } else {
        if (ctrl->done)
            return;
        load_sweep_order(sm.order);
        const long long n = (long long)ctrl->n_list[which];
        // select the list without indexing the parameter struct at run time
        // (that would copy the struct to local memory)
        const int *work_list = which ? s.list[1] : s.list[0];
        const real bound0 = (real)ctrl->bound[0], bound1 = (real)ctrl->bound[1];
        MarchStats st = {0, 0, 0, 0, 0};
        long long it = 0, next = 0;
        if (lane == 0) {
            it = (long long)atomicAdd(&ctrl->work[which], 1u);
            next = (long long)atomicAdd(&ctrl->work[which], 1u);
        }
        it = __shfl_sync(FULL, it, 0);
        next = __shfl_sync(FULL, next, 0);
        while (it < n) {
            const long long b = (long long)work_list[it];
            long long nbi[kFaces];
#pragma unroll
            for (int f = 0; f < kFaces; ++f)
                nbi[f] = neighbour_brick(g, s.nbr, b, f);
            Notify<real> nt;
            sweep_brick<real, kHetero, kTape, kAniso, true>(g, s, p, spd_const_term, sm.order, W, b, nbi, ~0u, bound0, bound1,
                                                            lane, nt, st);
            if (nt.m) {
                s.dirty[nt.nb] = 1u;
                st.exchanges += (unsigned long long)__popcll(nt.m);
            }
            __syncwarp();
            it = next;
            if (it < n && lane == 0)
                next = (long long)atomicAdd(&ctrl->work[which], 1u);
            next = __shfl_sync(FULL, next, 0);
        }
        flush_stats(ctrl, st, lane);
    }
}

// ---------------------------------------------------------------------------
// One-launch marches.  Warps take bricks from the ready queue until none is
// queued or being marched.
//
// Persistent schedule (kAll): the bound of the restart is fixed, every flagged
// brick is queued, the launch is one restart.
//
// Continuous schedule: the restarts of Algorithm 16 without the barrier
// between them, one launch for the whole solve.  The bound says which bricks
// may start; a brick marches with the bound it finds (plus the look-ahead, by
// default to its end).  Bricks whose work lies above the bound wait in a ring.
// Once fewer bricks than raise_at are queued or marching, a warp raises the
// bound to max(bound, smallest waiting value) + stride and the idle warps scan
// the ring in chunks: bricks at or below the new bound are queued, the others
// appended again.  Only bricks next to the front wait, so a raise touches a few
// per cent of the bricks (scanning the minima of all bricks took 11% of the
// 1024^3 march's warp time, and twice that waiting for the scans).  The solve
// is complete when nothing is queued, marching, waiting or being scanned.  At
// the restart limit the raises stop and the launch ends once the current
// level is drained; the work words then say what is left.
//
// Every wait is bounded (wait_ns without any progress): past the limit the
// kernel sets ERR_SPIN and returns.
// ---------------------------------------------------------------------------

// Raise the bound (one lane).  Returns true when this warp raised it.
__device__ bool try_raise(Control *c, const SolveParams &p, int pend)
{
    const unsigned long long w = vloadu(&c->scan_word);
    const int ep = (int)(w >> 32);
    const auto *lv = &c->level[ep & 1];
    if (vload(&c->scan_done) < (int)(unsigned)vloadu(&lv->chunks) || vloadu(&c->w_tail) == vloadu(&c->w_head))
        return false;
    if (atomicCAS(&c->raise_lock, ep, ep + 1) != ep)
        return false;
    __threadfence();
    const unsigned long long base = vloadu(&c->w_head), end = vloadu(&c->w_tail);
    bool ok = end != base && vload(&c->scan_done) >= (int)(unsigned)vloadu(&lv->chunks);
    if (ok && p.max_restarts > 0 && (long long)vload(&c->restart) >= p.max_restarts) {
        // the restart limit counts the raises too
        atomicOr(&c->error, ERR_RESTARTS);
        ok = false;
    }
    if (!ok) {
        __threadfence();
        atomicExch(&c->raise_lock, ep);
        return false;
    }
    const float b0 = *(const volatile float *)&lv->bound;
    const float sm = __uint_as_float(*(const volatile unsigned *)&c->scan_min);
    double v = (double)(sm < CUDART_INF_F ? fmaxf(b0, sm) : b0) + p.stride;
    if (pend > 0 && p.stride < CUDART_INF && sm < CUDART_INF_F)
        v = fmin(v, (floor((double)sm / p.stride) + p.max_lead) * p.stride);
    const float nb = fmaxf(__double2float_ru(fmin(v, p.width)), b0);
    const unsigned count = (unsigned)(end - base);
    const int warps = gridDim.x * kMarchWarps;
    int chunk = (int)((count + warps - 1) / warps);
    chunk = (chunk + 31) & ~31;
    auto *nl = &c->level[(ep + 1) & 1];
    *(volatile unsigned long long *)&nl->base = base;
    *(volatile unsigned long long *)&nl->end = end;
    *(volatile int *)&nl->chunk = chunk;
    *(volatile unsigned long long *)&nl->chunks = chunk_word((unsigned)(ep + 1), (count + chunk - 1) / chunk);
    *(volatile float *)&nl->bound = nb;
    *(volatile unsigned long long *)&c->w_head = end;
    *(volatile int *)&c->scan_done = 0;
    *(volatile unsigned *)&c->scan_min = kNoWork;
    *(volatile int *)&c->restart = vload(&c->restart) + 1;
    __threadfence();
    atomicExch(&c->scan_word, (unsigned long long)(ep + 1) << 32);
    return true;
}

// Nothing is queued, marching, waiting or being scanned (one lane; limited:
// nothing but waiting).
__device__ bool launch_done(Control *c, bool limited)
{
    const int ep = (int)(vloadu(&c->scan_word) >> 32);
    if (vload(&c->scan_done) < (int)(unsigned)vloadu(&c->level[ep & 1].chunks))
        return false;
    __threadfence();
    if (vload(&c->pending) != 0)
        return false;
    __threadfence();
    if (!limited && vloadu(&c->w_tail) != vloadu(&c->w_head))
        return false;
    __threadfence();
    return vload(&c->raise_lock) == ep && (int)(vloadu(&c->scan_word) >> 32) == ep &&
           vload(&c->scan_done) >= (int)(unsigned)vloadu(&c->level[ep & 1].chunks);
}

// One lane: the next job of the warp.  job 0: march brick arg; 1: scan chunk
// arg of raise `ep`; 2: stop.  ticket is the queue ticket the warp holds (-1:
// none).  A warp polls its own queue slot; the words every warp shares are read
// by one warp of the CTA every time and by the others every eighth time.
template <bool kAll>
__device__ void next_job(Control *c, unsigned long long *q, unsigned long long cap, const SolveParams &p, bool leader,
                         long long &ticket, int &job, long long &arg, int &ep_out)
{
    if (ticket < 0)
        ticket = (long long)atomicAdd(&c->q_head, 1ull);
    unsigned long long *slot = q + ((unsigned long long)ticket % cap);
    const unsigned long long want = (unsigned long long)ticket & 0xffffffffull;
    unsigned long long t0 = 0, seen = ~0ull;
    unsigned ns = 32, tick = leader ? 0u : (unsigned)ticket & 7u;
    for (;; ++tick) {
        const unsigned long long v = vloadu(slot);
        if (v != 0ull && (v >> 32) == want) {
            atomicExch(slot, 0ull);
            ticket = -1;
            job = 0;
            arg = (long long)(v & 0xffffffffull) - 1;
            return;
        }
        if (leader || (tick & 7u) == 7u) {
            const int err = vload(&c->error);
            if (err & ERR_SPIN) {
                job = 2;
                return;
            }
            const bool limited = (err & ERR_RESTARTS) != 0;
            const int pend = vload(&c->pending);
            unsigned long long w = vloadu(&c->scan_word);
            if (!kAll) {
                if (claimed_chunk(w, vloadu(&c->level[(w >> 32) & 1u].chunks)) >= 0) {
                    w = atomicAdd(&c->scan_word, 1ull);
                    __threadfence();   // the level this chunk belongs to
                    ep_out = (int)(w >> 32);
                    const int ch = claimed_chunk(w, vloadu(&c->level[ep_out & 1].chunks));
                    if (ch >= 0) {
                        job = 1;
                        arg = ch;
                        return;
                    }
                }
                if (!limited && pend < p.raise_at && try_raise(c, p, pend))
                    continue;
            }
            if (pend == 0 && launch_done(c, limited || kAll)) {
                job = 2;
                return;
            }
            // progress: a push, a raise or a scanned chunk
            const unsigned long long mark = vloadu(&c->q_tail) + (w << 8) + (unsigned)vload(&c->scan_done);
            const unsigned long long now = device_ns();
            if (mark != seen) {
                seen = mark;
                t0 = now;
            } else if (now - t0 > vloadu(&c->wait_ns)) {
                break;
            }
        }
        __nanosleep(ns);
        if (ns < 256)
            ns <<= 1;
    }
    atomicOr(&c->error, ERR_SPIN);
    job = 2;
}

// One warp scans a chunk of the waiting ring for the bound of raise ep.  ticket:
// the queue ticket the warp holds (or -1); returns the brick of that ticket if a
// wait had to take it from the queue, else -1.
__device__ __forceinline__ long long scan_chunk(const DeviceState &s, unsigned long long cap, int ch, int ep,
                                                long long ticket, int lane)
{
    long long held = -1;
    __syncwarp();   // every lane's loads of the level come after lane 0's claim
    Control *c = s.ctrl;
    const auto &lv = c->level[ep & 1];
    const unsigned long long end = vloadu(&lv.end), wcap = waiting_slots((long long)cap);
    const int chunk = vload(&lv.chunk);
    const float bound = *(const volatile float *)&lv.bound;
    const unsigned long long first = vloadu(&lv.base) + (unsigned long long)ch * (unsigned)chunk;
    unsigned kept = kNoWork;
    for (int i = 0; i < chunk; i += 32) {
        const unsigned long long pos = first + (unsigned)(i + lane);
        long long b = -1;
        if (pos < end) {
            // the entry may still be on its way from the warp that counted it
            unsigned long long *slot = s.waiting + pos % wcap;
            const unsigned long long want = pos & 0xffffffffull;
            unsigned long long v = vloadu(slot);
            if (v == 0ull || (v >> 32) != want) {
                const unsigned long long ts = device_ns(), lim = vloadu(&c->wait_ns);
                while (v == 0ull || (v >> 32) != want) {
                    if (device_ns() - ts > lim || (vload(&c->error) & ERR_SPIN)) {
                        atomicOr(&c->error, ERR_SPIN);
                        break;
                    }
                    __nanosleep(32);
                    v = vloadu(slot);
                }
            }
            if (v != 0ull && (v >> 32) == want) {
                v = atomicExch(slot, 0ull);
                b = (long long)(v & 0xffffffffull) - 1;
            }
        }
        int act = 0;   // 1: queue, 2: keep waiting
        if (b >= 0) {
            unsigned long long old = vloadu(&s.work[b]);
            for (;;) {
                const unsigned k = (unsigned)(old >> 32);
                unsigned fl = (unsigned)old;
                act = 0;
                if (!(fl & kWorkActive) && k < kNoWork) {
                    if (__uint_as_float(k) > bound) {
                        act = 2;
                        kept = umin(kept, k);
                        break;
                    }
                    fl |= kWorkActive;
                    act = 1;
                }
                const unsigned long long was = atomicCAS(&s.work[b], old, work_word(k, fl & ~kWorkWaiting));
                if (was == old)
                    break;
                old = was;
            }
        }
        const unsigned bq = __ballot_sync(FULL, act == 1), bw = __ballot_sync(FULL, act == 2);
        unsigned long long tq = 0, tw = 0;
        if (lane == 0) {
            if (bq) {
                atomicAdd(&c->pending, __popc(bq));
                tq = atomicAdd(&c->q_tail, (unsigned long long)__popc(bq));
            }
            if (bw)
                tw = atomicAdd(&c->w_tail, (unsigned long long)__popc(bw));
        }
        tq = __shfl_sync(FULL, tq, 0);
        tw = __shfl_sync(FULL, tw, 0);
        const unsigned below = (1u << lane) - 1u;
        long long none = -1;
        if (act == 1)
            ring_put(c, s.queue, cap, tq + __popc(bq & below), b, ticket, held);
        else if (act == 2)
            ring_put(c, s.waiting, wcap, tw + __popc(bw & below), b, -1, none);
    }
    kept = __reduce_min_sync(FULL, kept);
    if (lane == 0) {
        if (kept < kNoWork)
            atomicMin(&c->scan_min, kept);
        __threadfence();
        atomicAdd(&c->scan_done, 1);
    }
    return (long long)__reduce_max_sync(FULL, (unsigned)(held + 1)) - 1;   // a brick index has 31 bits
}

template <typename real, bool kHetero, bool kTape, bool kAniso, bool kBounded, bool kAll>
__global__ void __launch_bounds__(kMarchWarps * 32, march_min_blocks<real, kTape>())
    k_march_queue(Geom g, DeviceState s, SolveParams p, double spd_const_term)
{
    static_assert(kBounded || !kAll, "a restart with a fixed bound is a bounded march");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    MarchSmem<real, kTape> &sm = *reinterpret_cast<MarchSmem<real, kTape> *>(smem_raw);
    WarpTile<real, kTape> &W = sm.tile[warp];
    Control *ctrl = s.ctrl;
    if (ctrl->done)
        return;
    load_sweep_order(sm.order);
    const unsigned long long cap = (unsigned long long)g.nbricks;
    const real INF = inf_v<real>();
    MarchStats st = {0, 0, 0, 0, 0};
    long long ticket = -1;
    for (;;) {
        int job = 2, ep = 0;
        long long arg = 0;
        if (lane == 0)
            next_job<kAll>(ctrl, s.queue, cap, p, warp == 0, ticket, job, arg, ep);
        job = __shfl_sync(FULL, job, 0);
        arg = __shfl_sync(FULL, arg, 0);
        if (job == 2)
            break;
        if (job == 1) {
            ep = __shfl_sync(FULL, ep, 0);
            arg = scan_chunk(s, cap, (int)arg, ep, __shfl_sync(FULL, ticket, 0), lane);
            if (arg < 0)
                continue;
            ticket = -1;
        }
        const long long b = arg;
        long long nbi[kFaces];
#pragma unroll
        for (int f = 0; f < kFaces; ++f)
            nbi[f] = neighbour_brick(g, s.nbr, b, f);
        const unsigned dirty = take_brick(s, b, lane);
        real bound0 = INF, bound1 = INF;
        if (kAll) {
            bound0 = (real)ctrl->bound[0];
            bound1 = (real)ctrl->bound[1];
        } else if (kBounded) {
            // accept up to the bound plus the look-ahead, never beyond
            // width_band (cells above it stay BAND, Algorithm 12)
            const float bd = *(const volatile float *)&ctrl->level[(vloadu(&ctrl->scan_word) >> 32) & 1u].bound;
            bound0 = bound1 = (real)fmin((double)__shfl_sync(FULL, bd, 0) + p.ahead, p.width);
        }
        Notify<real> nt;
        sweep_brick<real, kHetero, kTape, kAniso, kBounded>(g, s, p, spd_const_term, sm.order, W, b, nbi, dirty,
                                                            bound0, bound1, lane, nt, st);
        st.exchanges += (unsigned long long)__popcll(nt.m);
        finish_brick<real, kAll>(s, cap, p.width, b, nt, lane);
    }
    flush_stats(ctrl, st, lane);
}

// Seed a launch: the work word of every brick from its BAND minima and the
// work a stopped launch left, queued (at or below the bound) or waiting.  A brick
// that a stopped phased solve left dirty is queued (the value is not recorded).
// all: the bound of each side is fixed and nothing waits.
template <typename real>
__global__ void k_seed(Geom g, const real *__restrict__ bmin, Control *ctrl, unsigned long long *work,
                       unsigned *dirty, unsigned long long *q, unsigned long long *waiting, double width, bool all)
{
    if (ctrl->done)
        return;
    const double bd0 = ctrl->bound[0], bd1 = ctrl->bound[1];
    const float bd = __double2float_ru(fmin(bd0, bd1));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // level 0: no scan, the bound of k_control
        ctrl->level[0].base = ctrl->level[0].end = 0ull;
        ctrl->level[0].chunks = chunk_word(0, 0);
        ctrl->level[0].chunk = 32;
        ctrl->level[0].bound = bd;
        ctrl->scan_min = __float_as_uint(bd);
        if (ctrl->hold)
            atomicAdd(&ctrl->pending, 1);   // testing: the queue never drains
    }
    const int lane = threadIdx.x & 31;
    for (long long b0 = blockIdx.x * (long long)blockDim.x; b0 < g.nbricks;
         b0 += (long long)gridDim.x * blockDim.x) {
        const long long b = b0 + threadIdx.x;
        int act = 0;
        if (b < g.nbricks) {
            const unsigned k0 = (unsigned)(work[b] >> 32);
            const real m0 = bmin[2 * b], m1 = bmin[2 * b + 1];
            unsigned key = k0 < kNoWork ? k0 : kNoWork;
            if (all) {
                // a flagged value was accepted by the neighbour: it is at or
                // below the bound of its side or of an earlier restart
                if (key < kNoWork || (lt(m0, inf_v<real>()) && (double)m0 <= bd0) ||
                    (lt(m1, inf_v<real>()) && (double)m1 <= bd1))
                    act = 1;
            } else {
                const real m = vmin(m0, m1);
                if (lt(m, inf_v<real>()) && (double)m <= width)
                    key = umin(key, work_key(m));
                if (key < kNoWork)
                    act = __uint_as_float(key) <= bd ? 1 : 2;
            }
            if (dirty[b] != 0u) {
                dirty[b] = 0u;
                act = 1;
            }
            work[b] = work_word(key, kWorkFull | (act == 1 ? kWorkActive : (act == 2 ? kWorkWaiting : 0u)));
        }
        const unsigned bq = __ballot_sync(FULL, act == 1), bw = __ballot_sync(FULL, act == 2);
        unsigned long long tq = 0, tw = 0;
        if (lane == 0) {
            if (bq) {
                atomicAdd(&ctrl->pending, __popc(bq));
                tq = atomicAdd(&ctrl->q_tail, (unsigned long long)__popc(bq));
            }
            if (bw)
                tw = atomicAdd(&ctrl->w_tail, (unsigned long long)__popc(bw));
        }
        tq = __shfl_sync(FULL, tq, 0) + __popc(bq & ((1u << lane) - 1u));
        tw = __shfl_sync(FULL, tw, 0) + __popc(bw & ((1u << lane) - 1u));
        if (act == 1)
            q[tq] = ((tq & 0xffffffffull) << 32) | (unsigned long long)(b + 1);
        else if (act == 2)
            waiting[tw] = ((tw & 0xffffffffull) << 32) | (unsigned long long)(b + 1);
    }
}

// ---------------------------------------------------------------------------
// Algorithm 16 bookkeeping: global minima of the front, exit test, bound.
// ---------------------------------------------------------------------------

template <typename real>
__global__ void k_reduce(Geom g, const real *__restrict__ bmin, const unsigned long long *__restrict__ work,
                         const unsigned *__restrict__ dirty, Control *ctrl)
{
    if (ctrl->done)
        return;
    __shared__ double r0[8], r1[8];
    __shared__ unsigned rc[8];
    double m0 = CUDART_INF, m1 = CUDART_INF;
    unsigned cnt = 0;
    for (long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x; b < g.nbricks;
         b += (long long)gridDim.x * blockDim.x) {
        m0 = fmin(m0, (double)bmin[2 * b]);
        // work a stopped launch left: its side is not recorded
        const unsigned key = (unsigned)(work[b] >> 32);
        m1 = fmin(m1, key < kNoWork ? fmin((double)__uint_as_float(key), (double)bmin[2 * b + 1])
                                    : (double)bmin[2 * b + 1]);
        cnt += dirty[b] != 0u;
    }
    m0 = warp_min(m0);
    m1 = warp_min(m1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        r0[w] = m0;
        r1[w] = m1;
        rc[w] = cnt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
            m0 = fmin(m0, r0[i]);
            m1 = fmin(m1, r1[i]);
            cnt += rc[i];
        }
        atomicMin(&ctrl->minbits[0], (unsigned long long)__double_as_longlong(m0));
        atomicMin(&ctrl->minbits[1], (unsigned long long)__double_as_longlong(m1));
        if (cnt)
            atomicAdd(&ctrl->dirty_count, cnt);
    }
}

// empty queue and waiting ring, no raise or scan under way
__device__ __forceinline__ void reset_queue(Control *c)
{
    c->q_head = c->q_tail = 0ull;
    c->w_head = c->w_tail = 0ull;
    c->pending = 0;
    c->scan_word = 0ull;
    c->scan_done = 0;
    c->raise_lock = 0;
}

__global__ void k_control(Control *c, double width, double stride, long long max_restarts)
{
    if (c->done)
        return;
    if (c->error & (ERR_SPIN | ERR_ROUNDS | ERR_RESTARTS)) {
        c->done = 1;   // a device error ends the solve (reported by the host)
        return;
    }
    const unsigned long long INF_BITS = 0x7ff0000000000000ull;
    double mv0 = fmin(__longlong_as_double((long long)c->minbits[0]), width);
    double mv1 = fmin(__longlong_as_double((long long)c->minbits[1]), width);
    c->restart += 1;
    c->host_restart += 1;
    if (mv0 >= width && mv1 >= width && c->dirty_count == 0u) {
        c->done = 1;
    } else if (max_restarts > 0 && c->restart > max_restarts) {
        c->error |= ERR_RESTARTS;
        c->done = 1;
    } else {
        c->bound[0] = fmin(mv0 + stride, width);
        c->bound[1] = fmin(mv1 + stride, width);
    }
    c->minbits[0] = INF_BITS;
    c->minbits[1] = INF_BITS;
    c->dirty_count = 0u;
    c->n_list[0] = 0u;
    c->n_list[1] = 0u;
    c->work[0] = 0u;
    c->work[1] = 0u;
    reset_queue(c);
}

// Work lists: list 0 = bricks with a BAND cell at or below the bound or with
// pending overlap changes (first march), those a stopped one-launch solve left in
// the work words among them; list 1 = bricks with pending changes
// (second march, after the exchange).  Changes flagged during the march are
// left for the next selection.
template <typename real>
__global__ void k_select(Geom g, const real *__restrict__ bmin, unsigned *dirty, unsigned long long *work,
                         Control *ctrl, int *list, int which)
{
    if (ctrl->done)
        return;
    const double bd0 = ctrl->bound[0], bd1 = ctrl->bound[1];
    const int lane = threadIdx.x & 31;
    for (long long b0 = blockIdx.x * (long long)blockDim.x; b0 < g.nbricks;
         b0 += (long long)gridDim.x * blockDim.x) {
        const long long b = b0 + threadIdx.x;
        bool sel = false, dty = false;
        if (b < g.nbricks) {
            dty = dirty[b] != 0u;
            sel = dty;
            if (which == 0) {
                // a brick takes part when it has a BAND cell at or below the
                // bound (an empty side has bound +inf, and so do the minima
                // of bricks without BAND cells)
                const double m0 = (double)bmin[2 * b], m1 = (double)bmin[2 * b + 1];
                sel = sel || (m0 < CUDART_INF && m0 <= bd0) || (m1 < CUDART_INF && m1 <= bd1);
                if ((unsigned)(work[b] >> 32) < kNoWork) {
                    sel = true;
                    work[b] = ~0ull;
                }
            }
        }
        if (dty)
            dirty[b] = 0u;
        const unsigned ball = __ballot_sync(0xffffffffu, sel);
        if (ball == 0u)
            continue;
        unsigned basepos = 0;
        if (lane == 0)
            basepos = atomicAdd(&ctrl->n_list[which], (unsigned)__popc(ball));
        basepos = __shfl_sync(0xffffffffu, basepos, 0);
        if (sel)
            list[basepos + __popc(ball & ((1u << lane) - 1u))] = (int)b;
    }
}

__global__ void k_reset_control(Control *c, unsigned long long wait_ns, int hold)
{
    c->wait_ns = wait_ns;
    c->hold = hold;
    const unsigned long long INF_BITS = 0x7ff0000000000000ull;
    c->minbits[0] = INF_BITS;
    c->minbits[1] = INF_BITS;
    c->marches = c->rounds = c->exchanges = c->accepted = c->solves = 0ull;
    c->bound[0] = c->bound[1] = 0.0;
    c->dirty_count = 0u;
    c->n_list[0] = c->n_list[1] = 0u;
    c->work[0] = c->work[1] = 0u;
    reset_queue(c);
    c->done = 0;
    c->error = 0;
    c->restart = 0;
    c->host_restart = 0;
}

template <typename real>
__device__ __forceinline__ void output_cell(real v, uint8_t tg, long long p, real *T_out, uint8_t *tags_out)
{
    const uint8_t st = tg & ST_MASK;
    // the sign as a bit (a double negation would take the FP64 pipe)
    T_out[p] = st == ST_FAR ? inf_v<real>() : ((tg & TG_NEG) ? kmark(v) : v);
    if (tags_out)
        tags_out[p] = st;
}

// Brick layout -> the caller's x-fastest arrays (signed psi, public tags);
// one CTA per brick, each warp writing rows of 8 consecutive cells.
template <typename real>
__global__ void __launch_bounds__(kInitThreads) k_output(Geom g, const real *__restrict__ T,
                                                         const uint8_t *__restrict__ tag, real *T_out,
                                                         uint8_t *tags_out)
{
    static_assert(kB3 == 2 * kInitThreads, "two cells per thread");
    for (int b = blockIdx.x; b < (int)g.nbricks; b += gridDim.x) {
        int bx, by, bz;
        brick_xyz32(g, b, bx, by, bz);
        const long long base = (long long)b * kB3;
        // cells c and c + 256 of the brick (z and z + 4), both loaded first
        const int c = threadIdx.x;
        const real v0 = T[base + c], v1 = T[base + c + kInitThreads];
        const uint8_t t0 = tag[base + c], t1 = tag[base + c + kInitThreads];
        const int i = bx * kB + (c & 7), j = by * kB + ((c >> 3) & 7), k = bz * kB + (c >> 6);
        if (i >= g.nx || j >= g.ny)
            continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int kk = k + 4 * h;
            if (kk >= g.nz)
                continue;
            output_cell<real>(h ? v1 : v0, h ? t1 : t0, ((long long)kk * g.ny + j) * g.nx + i, T_out, tags_out);
        }
    }
}

// ---------------------------------------------------------------------------
// Domain decomposition (Sec. 4.1, Algorithms 13-15): the grid of one rank is
// its slab of z layers plus the ghost layers it shares with its neighbours;
// the overlap layers are read out (signed psi, +inf for FAR cells) and the
// neighbour's copy of them is integrated.
// ---------------------------------------------------------------------------

template <typename real>
__global__ void k_layer_export(Geom g, const real *__restrict__ T, const uint8_t *__restrict__ tag,
                               int z0, int nl, real *out)
{
    const long long n = (long long)g.nx * g.ny * nl;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(p % g.nx);
        const long long r = p / g.nx;
        const int j = (int)(r % g.ny), k = z0 + (int)(r / g.ny);
        const long long b = ((long long)(k >> 3) * g.nby + (j >> 3)) * g.nbx + (i >> 3);
        const long long e = b * kB3 + (i & 7) + 8 * (j & 7) + 64 * (k & 7);
        const uint8_t tg = tag[e];
        real v = T[e];
        if ((tg & ST_MASK) == ST_FAR)
            v = inf_v<real>();
        else if (tg & TG_NEG)
            v = -v;
        out[p] = v;
    }
}

// Algorithm 15: a received value smaller in magnitude than the local one
// replaces it; the cell becomes BAND of the received value's side, so the
// next march accepts it if it is within the bound (KNOWN_OLD of Algorithm
// 15, then taken from the heap) or keeps it tentative (BAND_OLD).  FIX
// cells are never replaced.  count receives the number of replaced cells.
template <typename real>
__global__ void k_layer_integrate(Geom g, real *T, uint8_t *tag, real *bmin, int z0, int nl,
                                  const real *__restrict__ in, unsigned *count)
{
    const long long n = (long long)g.nx * g.ny * nl;
    unsigned c = 0;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(p % g.nx);
        const long long r = p / g.nx;
        const int j = (int)(r % g.ny), k = z0 + (int)(r / g.ny);
        const long long b = ((long long)(k >> 3) * g.nby + (j >> 3)) * g.nbx + (i >> 3);
        const long long e = b * kB3 + (i & 7) + 8 * (j & 7) + 64 * (k & 7);
        const real v = in[p];
        const real a = kval(v);   // |v|, -0 included
        const uint8_t tg = tag[e];
        if ((tg & ST_MASK) == ST_FIX || !(a < inf_v<real>()))
            continue;
        const bool far = (tg & ST_MASK) == ST_FAR;
        if (!far && !lt(a, T[e]))
            continue;
        const bool neg = v < (real)0 || (v == (real)0 && (tg & TG_NEG));
        T[e] = a;
        tag[e] = (uint8_t)(ST_BAND | (neg ? TG_NEG : 0));
        if constexpr (sizeof(real) == 8)
            atomicMin((unsigned long long *)&bmin[2 * b + (neg ? 0 : 1)],
                      (unsigned long long)__double_as_longlong(a));
        else
            atomicMin((unsigned *)&bmin[2 * b + (neg ? 0 : 1)], __float_as_uint(a));
        ++c;
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c)
        atomicAdd(count, c);
}

// Set the bound of a march to a given level (both sides) and empty the queue.
__global__ void k_set_bound(Control *c, double b0, double b1)
{
    c->bound[0] = b0;
    c->bound[1] = b1;
    c->done = 0;
    reset_queue(c);
    c->minbits[0] = c->minbits[1] = 0x7ff0000000000000ull;
    c->dirty_count = 0u;
}

// ---------------------------------------------------------------------------
// Batches: the bricks of many grids packed into one brick array.  bgrid[b] is
// the grid of brick b; the grid table gives its size, first brick, spacing
// and the caller's arrays.  The neighbour table (DeviceState::nbr) has no
// neighbour across the border of a grid, so the grids never exchange data.
// ---------------------------------------------------------------------------

__device__ __forceinline__ void batch_cell(const BatchGrid &G, long long b, int c, int &i, int &j,
                                           int &k)
{
    // a batch has fewer than 2^31 bricks: 32-bit arithmetic
    const int lb = (int)(b - G.brick0);
    const int bx = lb % G.nbx;
    const int r = lb / G.nbx;
    const int by = r % G.nby, bz = r / G.nby;
    i = bx * kB + (c & 7);
    j = by * kB + ((c >> 3) & 7);
    k = bz * kB + (c >> 6);
}

// Algorithm 8 for every grid of a batch: a grid with a level set gets its
// interface cells, a grid of point sources starts all FAR (k_batch_sources then
// fixes its sources).
template <typename real>
__global__ void __launch_bounds__(kInitThreads) k_batch_init(const BatchGrid *__restrict__ grids,
                                                             const int *__restrict__ bgrid, int nbricks,
                                                             real *__restrict__ T, uint8_t *__restrict__ tag,
                                                             int group)
{
    __shared__ ReinitList list;
    const auto info = [&](int b) {
        const BatchGrid &G = grids[bgrid[b]];
        int i, j, k;
        if (G.phi0) {
            batch_cell(G, b, 0, i, j, k);
            return ReinitBrick<real>{(const real *)G.phi0, G.nx, G.ny, G.nz, i / kB, j / kB, k / kB, G.h, G.h, G.h, 0, 0};
        }
        const long long base = (long long)b * kB3;
        for (int c = threadIdx.x & 31; c < kB3; c += 32) {
            batch_cell(G, b, c, i, j, k);
            T[base + c] = inf_v<real>();
            tag[base + c] = i < G.nx && j < G.ny && k < G.nz ? ST_FAR : TG_OUT | ST_FAR;
        }
        return ReinitBrick<real>{};
    };
    for (long long b = (long long)blockIdx.x * group; b < nbricks; b += (long long)gridDim.x * group)
        reinit_bricks<real>((int)b, (int)min((long long)group, nbricks - b), info, T, tag, list);
}

// The point sources of the batch: psi = 0, FIX (Algorithm 8).
template <typename real>
__global__ void k_batch_sources(const BatchGrid *__restrict__ grids, const long long *__restrict__ src,
                                long long n_src, real *T, uint8_t *tag)
{
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n_src;
         s += (long long)gridDim.x * blockDim.x) {
        const BatchGrid &G = grids[src[4 * s]];
        const int i = (int)src[4 * s + 1], j = (int)src[4 * s + 2], k = (int)src[4 * s + 3];
        const long long b = G.brick0 + ((long long)(k >> 3) * G.nby + (j >> 3)) * G.nbx + (i >> 3);
        const long long e = b * kB3 + (i & 7) + 8 * (j & 7) + 64 * (k & 7);
        T[e] = (real)0;
        tag[e] = ST_FIX;
    }
}

// Speed term (h_g/F)^2 of every cell of a batch (each grid its own h and its
// own speed field or constant) and the bucket width h_g min(1/F) / sqrt(3)
// of every brick; one CTA of 512 threads per brick, as k_load_speed.
template <typename real>
__global__ void __launch_bounds__(kThreads) k_batch_speed(const BatchGrid *__restrict__ grids,
                                                          const int *__restrict__ bgrid,
                                                          long long nbricks, real *spd, real *bdelta,
                                                          Control *ctrl)
{
    __shared__ real red[kThreads / 32];
    const int t = threadIdx.x;
    for (long long b = blockIdx.x; b < nbricks; b += gridDim.x) {
        const BatchGrid &G = grids[bgrid[b]];
        int i, j, k;
        batch_cell(G, b, t, i, j, k);
        const bool out = i >= G.nx || j >= G.ny || k >= G.nz;
        real F = (real)G.speed_const;
        if (G.speed && !out)
            F = ((const real *)G.speed)[((long long)k * G.ny + j) * G.nx + i];
        if (out)
            F = (real)1;
        if (!(F >= (real)0) || !(F < inf_v<real>()))
            atomicOr(&ctrl->error, ERR_SPEED);
        spd[b * kB3 + t] = speed_term(F, G.h);
        real fm = out ? (real)0 : F;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            fm = fmax(fm, __shfl_xor_sync(0xffffffffu, fm, o));
        if ((t & 31) == 0)
            red[t >> 5] = fm;
        __syncthreads();
        if (t == 0) {
            real mx = red[0];
            for (int w = 1; w < kThreads / 32; ++w)
                mx = fmax(mx, red[w]);
            if (!(mx > (real)0))
                mx = (real)1;
            bdelta[b] = (real)(G.h / (1.7320508075688772 * (double)mx));
        }
        __syncthreads();
    }
}

// The outputs of a batch, one CTA per brick as k_output.  256 grids of
// 32^3 to 192^3 in float: 2.0 ms as a per-cell grid-stride loop, 1.25 ms so.
template <typename real>
__global__ void __launch_bounds__(kInitThreads) k_batch_output(const BatchGrid *__restrict__ grids,
                                                               const int *__restrict__ bgrid, int nbricks,
                                                               const real *__restrict__ T,
                                                               const uint8_t *__restrict__ tag)
{
    for (int b = blockIdx.x; b < nbricks; b += gridDim.x) {
        const int c = threadIdx.x;
        const long long base = (long long)b * kB3;
        const real v0 = T[base + c], v1 = T[base + c + kInitThreads];
        const uint8_t t0 = tag[base + c], t1 = tag[base + c + kInitThreads];
        const BatchGrid &G = grids[bgrid[b]];
        const int nx = G.nx, ny = G.ny, nz = G.nz;
        real *T_out = (real *)G.T_out;
        uint8_t *tags_out = G.tags_out;
        int i, j, k;
        batch_cell(G, b, c, i, j, k);
        if (i >= nx || j >= ny)
            continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int kk = k + 4 * h;
            if (kk < nz)
                output_cell<real>(h ? v1 : v0, h ? t1 : t0, ((long long)kk * ny + j) * nx + i, T_out, tags_out);
        }
    }
}

int grid_for(long long n, int threads, int cap)
{
    long long b = (n + threads - 1) / threads;
    if (b < 1)
        b = 1;
    if (b > cap)
        b = cap;
    return (int)b;
}

// Bricks per CTA of Algorithm 8: one per warp, fewer where the bricks would
// otherwise fill only some of the 152 SMs.
int init_group(long long nbricks)
{
    const long long n = nbricks / 152;
    return (int)(n < 1 ? 1 : (n > kInitThreads / 32 ? kInitThreads / 32 : n));
}

template <typename real, bool kTape>
size_t march_smem() { return sizeof(MarchSmem<real, kTape>); }

// Deterministic mode: face f of brick b is its boundary layer on side f
// (0..5 = -x, +x, -y, +y, -z, +z), cell q = u + 8 v in the in-face
// coordinates of the halo loader of sweep_brick, holding the known value or
// +inf.  A march pass reads its neighbours' faces and the faces of the bricks
// it marched are rebuilt after the pass (which >= 0: work list `which`), so
// a pass sees the state of the previous one whatever the order of its
// marches.  which < 0: every brick.
template <typename real>
__global__ void k_faces_build(Geom g, const real *__restrict__ T, const uint8_t *__restrict__ tag,
                              const Control *ctrl, const int *list, int which, real *faces)
{
    const long long nb = which < 0 ? g.nbricks : (long long)ctrl->n_list[which];
    const long long n = nb * (kFaces * 64);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        const long long bi = e / (kFaces * 64);
        const int r = (int)(e - bi * (kFaces * 64));
        const long long b = which < 0 ? bi : (long long)list[bi];
        const int f = r >> 6, q = r & 63, u = q & 7, v = q >> 3;
        const int axis = f >> 1;
        const int edge = (f & 1) ? kB - 1 : 0;
        const int cx = axis == 0 ? edge : u;
        const int cy = axis == 1 ? edge : (axis == 0 ? u : v);
        const int cz = axis == 2 ? edge : v;
        const long long ci = b * kB3 + cx + kB * cy + kB * kB * cz;
        faces[b * (kFaces * 64) + r] = is_known(tag[ci]) ? T[ci] : inf_v<real>();
    }
}

template <typename real>
void faces_build(const Geom &g, const DeviceState &s, int which, cudaStream_t st)
{
    const int nb = grid_for(g.nbricks * (kFaces * 64), 256, 152 * 32);
    k_faces_build<real><<<nb, 256, 0, st>>>(g, (const real *)s.T, s.tag, s.ctrl,
                                            which < 0 ? nullptr : s.list[which], which, (real *)s.faces);
}

// Trace: restart, phase and list length of a march launch.
__global__ void k_trace(const Control *c, int which, int phase, int *out)
{
    out[0] = c->done ? -1 : c->restart;
    out[1] = phase;
    out[2] = c->done ? 0 : (int)c->n_list[which];
}

__global__ void k_trace_seed(const Control *c, int *out)
{
    out[0] = c->done ? -1 : c->restart;
    out[1] = 0;
    out[2] = c->done ? 0 : (int)c->q_tail;
}

__global__ void k_reset_list(Control *c, int which)
{
    if (c->done)
        return;
    c->n_list[which] = 0u;
    c->work[which] = 0u;
}

// Calls f with the speed-field, tape and unequal-cell flags as compile-time
// constants (std::true_type / std::false_type), one kernel instantiation per
// combination.
template <typename Fn>
void with_flags(bool het, bool tape, bool aniso, Fn &&f)
{
    using Y = std::true_type;
    using N = std::false_type;
    auto third = [&](auto H, auto P) {
        if (aniso)
            f(H, P, Y{});
        else
            f(H, P, N{});
    };
    if (het) {
        if (tape)
            third(Y{}, Y{});
        else
            third(Y{}, N{});
    } else if (tape) {
        third(N{}, Y{});
    } else {
        third(N{}, N{});
    }
}

// One launch of the queue march (all: a restart with a fixed bound).
template <typename real>
void queue_march(const Geom &g, const DeviceState &s, const SolveParams &p, bool all, cudaStream_t st)
{
    // with no band width and a whole-brick look-ahead no cell is ever above a
    // march's bound
    const bool bounded = std::isfinite(p.width) || std::isfinite(p.ahead);
    with_flags(s.spd != nullptr, s.tape != nullptr, p.aniso != 0, [&](auto H, auto P, auto A) {
        constexpr bool h = decltype(H)::value, t = decltype(P)::value, an = decltype(A)::value;
        const size_t sm = march_smem<real, t>();
        const int ctas = s.march_ctas, th = kMarchWarps * 32;
        if (all)
            k_march_queue<real, h, t, an, true, true><<<ctas, th, sm, st>>>(g, s, p, p.spd_term);
        else if (bounded)
            k_march_queue<real, h, t, an, true, false><<<ctas, th, sm, st>>>(g, s, p, p.spd_term);
        else
            k_march_queue<real, h, t, an, false, false><<<ctas, th, sm, st>>>(g, s, p, p.spd_term);
    });
}

template <typename real>
cudaError_t restart_impl(const Geom &g, const DeviceState &s, const SolveParams &p,
                         cudaStream_t st, cudaEvent_t *ev, int *trace)
{
    const int rb = grid_for(g.nbricks, 256, 4096);
    const bool het = s.spd != nullptr, tape = s.tape != nullptr;
    const double sct = p.spd_term;
    k_reduce<real><<<rb, 256, 0, st>>>(g, (const real *)s.bmin, s.work, s.dirty, s.ctrl);
    k_control<<<1, 1, 0, st>>>(s.ctrl, p.width, p.stride, p.max_restarts);
    if (one_launch_schedule(p.schedule)) {
        const bool all = p.schedule == kSchedulePersistent;
        k_seed<real><<<rb, 256, 0, st>>>(g, (const real *)s.bmin, s.ctrl, s.work, s.dirty, s.queue, s.waiting, p.width, all);
        if (trace)
            k_trace_seed<<<1, 1, 0, st>>>(s.ctrl, trace);
        if (ev)
            cudaEventRecord(ev[0], st);
        queue_march<real>(g, s, p, all, st);
        if (ev)
            cudaEventRecord(ev[1], st);
        return cudaGetLastError();
    }
    for (int pass = 0; pass <= p.passes; ++pass) {
        const int which = pass == 0 ? 0 : 1;
        if (pass >= 2)
            k_reset_list<<<1, 1, 0, st>>>(s.ctrl, 1);
        k_select<real><<<rb, 256, 0, st>>>(g, (const real *)s.bmin, s.dirty, s.work, s.ctrl, s.list[which], which);
        if (trace)
            k_trace<<<1, 1, 0, st>>>(s.ctrl, which, pass, trace + 3 * pass);
        if (ev)
            cudaEventRecord(ev[2 * pass], st);
        with_flags(het, tape, p.aniso != 0, [&](auto H, auto P, auto A) {
            k_march<real, decltype(H)::value, 1, decltype(P)::value, decltype(A)::value>
                <<<s.march_ctas, kMarchWarps * 32, march_smem<real, decltype(P)::value>(), st>>>(g, s, p, sct,
                                                                                                  which);
        });
        if (s.faces)
            faces_build<real>(g, s, which, st);
        if (ev)
            cudaEventRecord(ev[2 * pass + 1], st);
    }
    return cudaGetLastError();
}

template <typename real>
cudaError_t front_init_impl(const Geom &g, const DeviceState &s, const SolveParams &p,
                            cudaStream_t st)
{
    const long long need = (g.nbricks + kMarchWarps - 1) / kMarchWarps;
    const int nb = (int)(need < s.march_ctas ? need : s.march_ctas);
    with_flags(s.spd != nullptr, s.tape != nullptr, p.aniso != 0, [&](auto H, auto P, auto A) {
        k_march<real, decltype(H)::value, 0, decltype(P)::value, decltype(A)::value>
            <<<nb, kMarchWarps * 32, march_smem<real, decltype(P)::value>(), st>>>(g, s, p, p.spd_term, 0);
    });
    if (s.faces)
        faces_build<real>(g, s, -1, st);
    return cudaGetLastError();
}

// Shared-memory attributes of the march kernels with or without the tape;
// returns their resident CTAs per SM (the smallest over the kernels a solve may
// launch).
template <typename real>
int configure_march(bool tape)
{
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    int n = 1 << 20;
    for (int f = 0; f < 8; ++f)
        with_flags((f & 1) != 0, (f & 2) != 0, (f & 4) != 0, [&](auto H, auto P, auto A) {
            constexpr bool hh = decltype(H)::value, tt = decltype(P)::value, an = decltype(A)::value;
            if (tt != tape)   // (a handle launches the kernels with or without the tape, never both)
                return;
            const int sm = (int)march_smem<real, tt>();
            cudaFuncSetAttribute(k_march<real, hh, 1, tt, an>, attr, sm);
            cudaFuncSetAttribute(k_march<real, hh, 0, tt, an>, attr, sm);
            cudaFuncSetAttribute(k_march_queue<real, hh, tt, an, true, true>, attr, sm);
            cudaFuncSetAttribute(k_march_queue<real, hh, tt, an, true, false>, attr, sm);
            cudaFuncSetAttribute(k_march_queue<real, hh, tt, an, false, false>, attr, sm);
            int k = 0;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, k_march_queue<real, hh, tt, an, false, false>,
                                                          kMarchWarps * 32, sm);
            n = k < n ? k : n;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, k_march_queue<real, hh, tt, an, true, false>,
                                                          kMarchWarps * 32, sm);
            n = k < n ? k : n;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, k_march<real, hh, 1, tt, an>, kMarchWarps * 32,
                                                          sm);
            n = k < n ? k : n;
        });
    return n > 0 && n < (1 << 20) ? n : 1;
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

cudaError_t launch_init_sources(int dtype, const Geom &g, const DeviceState &s,
                                const long long *src_ijk, long long n_src, cudaStream_t st)
{
    const int nb = grid_for(g.nbricks, 1, 152 * 16);
    if (dtype == 1) {
        k_init_sources<double><<<nb, 256, 0, st>>>(g, (double *)s.T, s.tag);
        if (n_src > 0)
            k_set_sources<double><<<grid_for(n_src, 256, 1024), 256, 0, st>>>(g, src_ijk, n_src,
                                                                             (double *)s.T, s.tag);
    } else {
        k_init_sources<float><<<nb, 256, 0, st>>>(g, (float *)s.T, s.tag);
        if (n_src > 0)
            k_set_sources<float><<<grid_for(n_src, 256, 1024), 256, 0, st>>>(g, src_ijk, n_src,
                                                                            (float *)s.T, s.tag);
    }
    return cudaGetLastError();
}

cudaError_t launch_init_reinit(int dtype, const Geom &g, const DeviceState &s,
                               const SolveParams &p, const void *phi0, cudaStream_t st, int zlo,
                               int zhi)
{
    const int gr = init_group(g.nbricks), nb = grid_for(g.nbricks, gr, 152 * 16);
    const long long layer = (long long)g.nx * g.ny;
    if (dtype == 1)
        k_init_reinit<double><<<nb, kInitThreads, 0, st>>>(g, p.h, p.hy, p.hz, (const double *)phi0 + zlo * layer,
                                                  (double *)s.T, s.tag, zlo, zhi, gr);
    else
        k_init_reinit<float><<<nb, kInitThreads, 0, st>>>(g, p.h, p.hy, p.hz, (const float *)phi0 + zlo * layer,
                                                 (float *)s.T, s.tag, zlo, zhi, gr);
    return cudaGetLastError();
}

cudaError_t launch_load_speed(int dtype, const Geom &g, const DeviceState &s, double h,
                              double hmin, const void *speed, double speed_const, cudaStream_t st)
{
    const int nb = grid_for(g.nbricks, 1, 152 * 8);
    if (dtype == 1)
        k_load_speed<double><<<nb, kThreads, 0, st>>>(g, h, hmin, (const double *)speed, speed_const,
                                                      (double *)s.spd, (double *)s.bdelta, s.ctrl);
    else
        k_load_speed<float><<<nb, kThreads, 0, st>>>(g, h, hmin, (const float *)speed, speed_const,
                                                     (float *)s.spd, (float *)s.bdelta, s.ctrl);
    return cudaGetLastError();
}

cudaError_t launch_front_init(int dtype, const Geom &g, const DeviceState &s,
                              const SolveParams &p, cudaStream_t st)
{
    return dtype == 1 ? front_init_impl<double>(g, s, p, st) : front_init_impl<float>(g, s, p, st);
}

cudaError_t launch_restart(int dtype, const Geom &g, const DeviceState &s, const SolveParams &p,
                           cudaStream_t st, cudaEvent_t *ev, int *trace)
{
    return dtype == 1 ? restart_impl<double>(g, s, p, st, ev, trace)
                      : restart_impl<float>(g, s, p, st, ev, trace);
}

cudaError_t launch_reset_control(const DeviceState &s, cudaStream_t st, unsigned long long wait_ns,
                                 int hold)
{
    k_reset_control<<<1, 1, 0, st>>>(s.ctrl, wait_ns, hold);
    return cudaGetLastError();
}

cudaError_t launch_output(int dtype, const Geom &g, const DeviceState &s, void *T_out,
                          uint8_t *tags_out, cudaStream_t st)
{
    const int nb = grid_for(g.nbricks, 1, 152 * 16);
    if (dtype == 1)
        k_output<double><<<nb, kInitThreads, 0, st>>>(g, (const double *)s.T, s.tag, (double *)T_out,
                                                      tags_out);
    else
        k_output<float><<<nb, kInitThreads, 0, st>>>(g, (const float *)s.T, s.tag, (float *)T_out,
                                                     tags_out);
    return cudaGetLastError();
}

cudaError_t launch_layer_export(int dtype, const Geom &g, const DeviceState &s, int z0, int nl,
                                void *out, cudaStream_t st)
{
    const int nb = grid_for((long long)g.nx * g.ny * nl, 256, 152 * 32);
    if (dtype == 1)
        k_layer_export<double><<<nb, 256, 0, st>>>(g, (const double *)s.T, s.tag, z0, nl, (double *)out);
    else
        k_layer_export<float><<<nb, 256, 0, st>>>(g, (const float *)s.T, s.tag, z0, nl, (float *)out);
    return cudaGetLastError();
}

cudaError_t launch_layer_integrate(int dtype, const Geom &g, const DeviceState &s, int z0, int nl,
                                   const void *in, unsigned *count, cudaStream_t st)
{
    const int nb = grid_for((long long)g.nx * g.ny * nl, 256, 152 * 32);
    if (dtype == 1)
        k_layer_integrate<double><<<nb, 256, 0, st>>>(g, (double *)s.T, s.tag, (double *)s.bmin, z0, nl,
                                                      (const double *)in, count);
    else
        k_layer_integrate<float><<<nb, 256, 0, st>>>(g, (float *)s.T, s.tag, (float *)s.bmin, z0, nl,
                                                     (const float *)in, count);
    return cudaGetLastError();
}

// One march of Algorithm 12 to a given bound: every brick with a BAND cell
// at or below it marches, and bricks whose halo changed march again, until
// none is left (the persistent queue).
cudaError_t launch_march_to(int dtype, const Geom &g, const DeviceState &s, const SolveParams &p,
                            double b0, double b1, cudaStream_t st)
{
    k_set_bound<<<1, 1, 0, st>>>(s.ctrl, b0, b1);
    const int rb = grid_for(g.nbricks, 256, 4096);
    if (dtype == 1) {
        k_seed<double><<<rb, 256, 0, st>>>(g, (const double *)s.bmin, s.ctrl, s.work, s.dirty, s.queue, s.waiting, p.width,
                                           true);
        queue_march<double>(g, s, p, true, st);
    } else {
        k_seed<float><<<rb, 256, 0, st>>>(g, (const float *)s.bmin, s.ctrl, s.work, s.dirty, s.queue, s.waiting, p.width, true);
        queue_march<float>(g, s, p, true, st);
    }
    return cudaGetLastError();
}

// The per-side BAND minima of the grid (Algorithm 16's local heap tops) into
// the control block (minbits).
cudaError_t launch_minima(int dtype, const Geom &g, const DeviceState &s, cudaStream_t st)
{
    k_set_bound<<<1, 1, 0, st>>>(s.ctrl, 0.0, 0.0);
    const int rb = grid_for(g.nbricks, 256, 4096);
    if (dtype == 1)
        k_reduce<double><<<rb, 256, 0, st>>>(g, (const double *)s.bmin, s.work, s.dirty, s.ctrl);
    else
        k_reduce<float><<<rb, 256, 0, st>>>(g, (const float *)s.bmin, s.work, s.dirty, s.ctrl);
    return cudaGetLastError();
}

cudaError_t launch_select(int dtype, const Geom &g, const DeviceState &s, int which,
                          cudaStream_t st)
{
    const int rb = grid_for(g.nbricks, 256, 4096);
    if (dtype == 1)
        k_select<double><<<rb, 256, 0, st>>>(g, (const double *)s.bmin, s.dirty, s.work, s.ctrl, s.list[which], which);
    else
        k_select<float><<<rb, 256, 0, st>>>(g, (const float *)s.bmin, s.dirty, s.work, s.ctrl, s.list[which], which);
    return cudaGetLastError();
}

cudaError_t launch_reset_list(const DeviceState &s, int which, cudaStream_t st)
{
    k_reset_list<<<1, 1, 0, st>>>(s.ctrl, which);
    return cudaGetLastError();
}

cudaError_t launch_batch_init(int dtype, const BatchGrid *grids, const int *bgrid,
                              long long nbricks, const DeviceState &s, cudaStream_t st)
{
    const int gr = init_group(nbricks), nb = grid_for(nbricks, gr, 152 * 16);
    if (dtype == 1)
        k_batch_init<double><<<nb, kInitThreads, 0, st>>>(grids, bgrid, (int)nbricks, (double *)s.T, s.tag, gr);
    else
        k_batch_init<float><<<nb, kInitThreads, 0, st>>>(grids, bgrid, (int)nbricks, (float *)s.T, s.tag, gr);
    return cudaGetLastError();
}

cudaError_t launch_batch_sources(int dtype, const BatchGrid *grids, const long long *src,
                                 long long n_src, const DeviceState &s, cudaStream_t st)
{
    if (n_src <= 0)
        return cudaSuccess;
    const int nb = grid_for(n_src, 256, 1024);
    if (dtype == 1)
        k_batch_sources<double><<<nb, 256, 0, st>>>(grids, src, n_src, (double *)s.T, s.tag);
    else
        k_batch_sources<float><<<nb, 256, 0, st>>>(grids, src, n_src, (float *)s.T, s.tag);
    return cudaGetLastError();
}

cudaError_t launch_batch_speed(int dtype, const BatchGrid *grids, const int *bgrid,
                               long long nbricks, const DeviceState &s, cudaStream_t st)
{
    const int nb = grid_for(nbricks, 1, 152 * 8);
    if (dtype == 1)
        k_batch_speed<double><<<nb, kThreads, 0, st>>>(grids, bgrid, nbricks, (double *)s.spd,
                                                       (double *)s.bdelta, s.ctrl);
    else
        k_batch_speed<float><<<nb, kThreads, 0, st>>>(grids, bgrid, nbricks, (float *)s.spd,
                                                      (float *)s.bdelta, s.ctrl);
    return cudaGetLastError();
}

cudaError_t launch_batch_output(int dtype, const BatchGrid *grids, const int *bgrid,
                                long long nbricks, const DeviceState &s, cudaStream_t st)
{
    const int nb = grid_for(nbricks, 1, 152 * 64);
    if (dtype == 1)
        k_batch_output<double><<<nb, kInitThreads, 0, st>>>(grids, bgrid, (int)nbricks, (const double *)s.T, s.tag);
    else
        k_batch_output<float><<<nb, kInitThreads, 0, st>>>(grids, bgrid, (int)nbricks, (const float *)s.T, s.tag);
    return cudaGetLastError();
}

cudaError_t launch_faces_build(int dtype, const Geom &g, const DeviceState &s, cudaStream_t st)
{
    if (dtype == 1)
        faces_build<double>(g, s, -1, st);
    else
        faces_build<float>(g, s, -1, st);
    return cudaGetLastError();
}

int march_blocks_per_sm(int dtype, bool tape)
{
    return dtype == 1 ? configure_march<double>(tape) : configure_march<float>(tape);
}

}  // namespace fmmgb

