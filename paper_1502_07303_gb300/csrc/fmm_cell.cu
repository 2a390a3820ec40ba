// fmm_cell.cu -- the cell-parallel march (schedule 4) and the interface
// initialisation from given values.
//
// The cell-parallel march runs Algorithms 9-12 by buckets instead of brick
// marches and queues: one bucket step accepts, on each side, every BAND
// cell at or below min(m + delta, width_band) (m the side's smallest BAND
// value, delta the bucket width of the cell's brick), then every cell next to
// a cell accepted in this step and above it is solved again (Algorithm 10:
// Algorithm 11 from the current values, Jacobi within the step: the solves
// read the state and write a second buffer), and the improvements are applied
// (an improved cell is BAND again, so an accepted value that drops is
// corrected, as in the label-correcting brick march).  The step that finds no
// BAND cell at or below width_band on either side ends the march.  For the
// first-order scheme of Eq. (2)-(3) the result is the unique discrete solution
// the heap march of Algorithm 12 reaches (Sec. 5.2).
//
// accuracy 2 is the higher-order fast marching that Sec. 6 names as future
// work, in the textbook second-order form: on an upwind axis whose next cell
// beyond the neighbour psi1, in the same direction, is known with
// psi2 <= psi1, the one-sided difference (3 t - 4 psi1 + psi2) / (2 h)
// replaces (t - psi1) / h, i.e. Algorithm 11 runs with psi_i = (4 psi1 -
// psi2) / 3 and the axis weight (3/2)^2.  That update is not monotone in its
// operands (a larger psi2 lowers the root, and a cell keeps the smallest of
// its roots), so a second neighbour must hold its final value when it is
// read: the second-order march runs with buckets narrower than the smallest
// single-axis increment (fmm_internal.h, kSecondOrderBucket), so that a cell
// and its upwind neighbour are not accepted in the same step, as in the
// sequential march where every KNOWN value is final.  The acceptance order
// still differs from the heap's, so this march and the sequential one reach
// different second-order solutions in general (both reproduce quadratic
// solutions to rounding).
//
// The first step (Algorithm 9) streams the grid; the bucket steps run in
// cooperative launches of up to 256 steps over the bricks at the front, with
// bounded grid barriers; the host reads the termination flag between launches.
#include "fmm_internal.h"
#include "fmm_fp64.cuh"
#include "fmm_lanes.cuh"

namespace fmmgb {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kCellThreads = 256;
constexpr uint8_t TG_ACC = 16;   // accepted in the current bucket step
constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;

template <typename real>
__device__ __forceinline__ real inf_r();
template <>
__device__ __forceinline__ float inf_r<float>() { return __int_as_float(0x7f800000); }
template <>
__device__ __forceinline__ double inf_r<double>() { return __longlong_as_double(0x7ff0000000000000ll); }

// the "no new value" mark of the second buffer (all bits set: a NaN)
template <typename real>
__device__ __forceinline__ real none_r();
template <>
__device__ __forceinline__ float none_r<float>() { return __int_as_float(-1); }
template <>
__device__ __forceinline__ double none_r<double>() { return __longlong_as_double(-1ll); }

__device__ __forceinline__ float vsqrt(float v) { return sqrtf(v); }
__device__ __forceinline__ double vsqrt(double v) { return sqrt(v); }

__device__ __forceinline__ bool known(uint8_t t) { return (t & ST_MASK) >= ST_KNOWN; }

// a < b and a <= b for values >= 0 (+inf included) on their bit patterns:
// integer compares, off the FP64 pipe that runs at 1/64 of the float rate
__device__ __forceinline__ bool blt(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }
__device__ __forceinline__ bool blt(float a, float b) { return __float_as_int(a) < __float_as_int(b); }
__device__ __forceinline__ bool ble(double a, double b) { return __double_as_longlong(a) <= __double_as_longlong(b); }
__device__ __forceinline__ bool ble(float a, float b) { return __float_as_int(a) <= __float_as_int(b); }
// |v| with the sign bit cleared (-0 becomes +0, which the compares above
// need)
__device__ __forceinline__ double abs_bits(double v) { return __longlong_as_double(__double_as_longlong(v) & 0x7fffffffffffffffll); }
__device__ __forceinline__ float abs_bits(float v) { return __int_as_float(__float_as_int(v) & 0x7fffffff); }
// the "no new value" mark (all bits set)
__device__ __forceinline__ bool is_none(double v) { return __double_as_longlong(v) == -1ll; }
__device__ __forceinline__ bool is_none(float v) { return __float_as_int(v) == -1; }

// Natural coordinates of brick-layout cell e (32-bit divisions: the brick
// count of a grid of at most 2^20 cells per axis that fits in memory is far
// below 2^32).
__device__ __forceinline__ void cell_ijk(const Geom &g, long long e, int &i, int &j, int &k)
{
    const unsigned b = (unsigned)(e >> 9);
    const int c = (int)(e & 511);
    const unsigned nbx = (unsigned)g.nbx, nby = (unsigned)g.nby;
    const int bx = (int)(b % nbx);
    const unsigned r = b / nbx;
    const int by = (int)(r % nby);
    const int bz = (int)(r / nby);
    i = bx * kB + (c & 7);
    j = by * kB + ((c >> 3) & 7);
    k = bz * kB + (c >> 6);
}

// Brick-layout index of natural cell (i, j, k) (inside the grid).
__device__ __forceinline__ long long cell_at(const Geom &g, int i, int j, int k)
{
    const long long b = ((long long)(k >> 3) * g.nby + (j >> 3)) * g.nbx + (i >> 3);
    return b * kB3 + (i & 7) + 8 * (j & 7) + 64 * (k & 7);
}

// The cell `steps` cells from (i, j, k) along axis a (direction sign of
// steps), or -1 outside the grid.
__device__ __forceinline__ long long cell_along(const Geom &g, int i, int j, int k, int a, int steps)
{
    int c[3] = {i, j, k};
    const int ext[3] = {g.nx, g.ny, g.nz};
    c[a] += steps;
    if (c[a] < 0 || c[a] >= ext[a])
        return -1;
    return cell_at(g, c[0], c[1], c[2]);
}

// Algorithm 11 for the active axes (act bit a), values psi[a] and weights
// W[a] = (h / h_a)^2 (times (3/2)^2 on a second-order axis), speed term
// q = (h/F)^2: the quadratic sum_a W_a (t - psi_a)^2 = q for the unknown
// shifted by the smallest value, t = m + u, solved for the nested sets that
// drop the largest psi (ties: the higher axis) while non-empty; the smallest
// causal root (every psi_a < t), or +inf.
template <typename real>
__device__ real cell_root(const real psi[3], const real W[3], unsigned act, real q)
{
    real m = inf_r<real>();
    int nd = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if ((act >> a) & 1u) {
            ++nd;
            m = psi[a] < m ? psi[a] : m;
        }
    real best = inf_r<real>();
    for (; nd > 0; --nd) {
        real d[3], w[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const bool on = (act >> a) & 1u;
            d[a] = on ? psi[a] - m : (real)0;
            w[a] = on ? W[a] : (real)0;
        }
        const real qa = (w[0] + w[1]) + w[2];
        const real qb = (real)-2 * ((w[0] * d[0] + w[1] * d[1]) + w[2] * d[2]);
        const real qc = ((w[0] * d[0] * d[0] + w[1] * d[1] * d[1]) + w[2] * d[2] * d[2]) - q;
        const real disc = qb * qb - (real)4 * qa * qc;
        if (disc >= (real)0) {
            const real u = (-qb + vsqrt(disc)) / ((real)2 * qa);
            if (d[0] < u && d[1] < u && d[2] < u) {
                const real t = m + u;
                best = t < best ? t : best;
                // clearly above the values of the set: a subset has a larger
                // root (the dropped term (u - d)^2 is at least 1e-10 of q)
                const real lim = u * (real)0.99999;
                if (d[0] < lim && d[1] < lim && d[2] < lim)
                    return best;
            }
        }
        int j = -1;
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (((act >> a) & 1u) && (j < 0 || psi[a] >= psi[j]))
                j = a;
        act &= ~(1u << j);
    }
    return best;
}

// Interface initialisation from given values (Algorithm 8 with the values of
// the interface cells supplied): a finite T0 makes the cell FIX with |T0| on
// the side of its sign (-0 and +0 are side +1), +-inf a FAR cell of that
// side.  NaN, or a non-FIX cell next to a cell of the other side (Algorithm
// 8 puts FIX cells at both ends of every sign change), sets ERR_INPUT.
template <typename real>
__global__ void __launch_bounds__(kCellThreads) k_init_fixed(Geom g, const real *__restrict__ T0, real *T,
                                                            uint8_t *tag, Control *ctrl)
{
    const long long n = g.nbricks * kB3;
    bool bad = false;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        int i, j, k;
        cell_ijk(g, e, i, j, k);
        if (i >= g.nx || j >= g.ny || k >= g.nz) {
            T[e] = inf_r<real>();
            tag[e] = TG_OUT | ST_FAR;
            continue;
        }
        const long long p = ((long long)k * g.ny + j) * g.nx + i;
        const real v = T0[p];
        const bool neg = v < (real)0;
        if (v != v) {
            bad = true;
            T[e] = inf_r<real>();
            tag[e] = ST_FAR;
            continue;
        }
        const bool fixed = v > -inf_r<real>() && v < inf_r<real>();
        T[e] = fixed ? abs_bits(v) : inf_r<real>();
        tag[e] = (uint8_t)((fixed ? ST_FIX : ST_FAR) | (neg ? TG_NEG : 0));
        if (!fixed) {
            const int c[3] = {i, j, k};
            const int ext[3] = {g.nx, g.ny, g.nz};
            const long long st[3] = {1, g.nx, (long long)g.nx * g.ny};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (c[a] > 0 && (T0[p - st[a]] < (real)0) != neg)
                    bad = true;
                if (c[a] + 1 < ext[a] && (T0[p + st[a]] < (real)0) != neg)
                    bad = true;
            }
        }
    }
    if (__any_sync(FULL, bad) && (threadIdx.x & 31) == 0)
        atomicOr(&ctrl->error, ERR_INPUT);
}

// Start of the march: the FIX cells count as accepted (Algorithm 9 updates
// the neighbours of every FIX cell), the step minima are reset and the
// second buffer is marked empty.
template <typename real>
__global__ void __launch_bounds__(kCellThreads) k_cell_seed(Geom g, uint8_t *tag, real *next,
                                                           unsigned long long *mins)
{
    const long long n = g.nbricks * kB3;
    if (blockIdx.x == 0 && threadIdx.x < 4)
        mins[threadIdx.x] = kInfBits;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        next[e] = none_r<real>();
        const uint8_t t = tag[e];
        if ((t & ST_MASK) == ST_FIX && !(t & TG_OUT))
            tag[e] = t | TG_ACC;
    }
}

// The first step (Algorithm 9) over the whole grid: Algorithm 10 for the cells
// next to a cell accepted in it, the FIX cells: a non-FIX
// cell above an accepted neighbour is solved again from the current values
// (Algorithm 11: per axis the smaller known neighbour below the cell, the
// minus one on a tie; with kAcc = 2 the second-order difference where the
// cell beyond it is known and not above it); a smaller root goes to next.
template <typename real, int kAcc>
__global__ void __launch_bounds__(kCellThreads) k_cell_relax(Geom g, const real *__restrict__ T,
                                                            const uint8_t *__restrict__ tag,
                                                            const real *__restrict__ spd, double spd_const,
                                                            double wy, double wz, real *next, Control *ctrl)
{
    if (ctrl->done)
        return;
    const long long n = g.nbricks * kB3;
    const real wax[3] = {(real)1, (real)wy, (real)wz};
    unsigned solves = 0;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        const uint8_t t = tag[e];
        if ((t & TG_OUT) || (t & ST_MASK) == ST_FIX)
            continue;
        int i, j, k;
        cell_ijk(g, e, i, j, k);
        const real Tc = T[e];
        long long nb[6];
        bool trig = false;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            nb[q] = cell_along(g, i, j, k, q >> 1, (q & 1) ? 1 : -1);
            if (nb[q] >= 0 && (tag[nb[q]] & TG_ACC) && blt(T[nb[q]], Tc))
                trig = true;
        }
        if (!trig)
            continue;
        ++solves;
        real psi[3] = {(real)0, (real)0, (real)0}, W[3] = {(real)0, (real)0, (real)0};
        unsigned act = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const long long qm = nb[2 * a], qp = nb[2 * a + 1];
            const bool km = qm >= 0 && known(tag[qm]), kp = qp >= 0 && known(tag[qp]);
            const real vm = km ? T[qm] : inf_r<real>(), vp = kp ? T[qp] : inf_r<real>();
            int d = 0;
            if (km && blt(vm, Tc))
                d = -1;
            if (kp && blt(vp, Tc)) {
                if (d == 0)
                    d = 1;
                else if (blt(vp, vm))
                    d = 1;
            }
            if (d == 0)
                continue;
            act |= 1u << a;
            psi[a] = d < 0 ? vm : vp;
            W[a] = wax[a];
            if (kAcc == 2) {
                const long long q2 = cell_along(g, i, j, k, a, 2 * d);
                if (q2 >= 0 && known(tag[q2])) {
                    const real v2 = T[q2];
                    if (ble(v2, psi[a])) {
                        psi[a] = ((real)4 * psi[a] - v2) / (real)3;
                        W[a] = W[a] * (real)2.25;
                    }
                }
            }
        }
        const real q = spd ? spd[e] : (real)spd_const;
        const real r = cell_root<real>(psi, W, act, q);
        if (blt(r, Tc))
            next[e] = r;
    }
    solves = __reduce_add_sync(FULL, solves);
    if ((threadIdx.x & 31) == 0 && solves)
        atomicAdd(&ctrl->solves, (unsigned long long)solves);
}

// Apply the step's new values (the cell becomes BAND), clear the accepted
// marks, and reduce the smallest BAND value of each side into slot `slot`.
template <typename real>
__global__ void __launch_bounds__(kCellThreads) k_cell_apply(Geom g, real *T, uint8_t *tag, real *next,
                                                            unsigned long long *mins, int slot, Control *ctrl)
{
    if (ctrl->done)
        return;
    const long long n = g.nbricks * kB3;
    real l0 = inf_r<real>(), l1 = inf_r<real>();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        const uint8_t t = tag[e];
        if (t & TG_OUT)
            continue;
        uint8_t nt = (uint8_t)(t & ~TG_ACC);
        real v = T[e];
        const real nv = next[e];
        if (!is_none(nv)) {
            v = nv;
            T[e] = nv;
            next[e] = none_r<real>();
            nt = (uint8_t)((nt & ~ST_MASK) | ST_BAND);
        }
        if (nt != t)
            tag[e] = nt;
        if ((nt & ST_MASK) == ST_BAND) {
            if (nt & TG_NEG)
                l0 = blt(v, l0) ? v : l0;
            else
                l1 = blt(v, l1) ? v : l1;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const real a = __shfl_xor_sync(FULL, l0, o), b = __shfl_xor_sync(FULL, l1, o);
        l0 = blt(a, l0) ? a : l0;
        l1 = blt(b, l1) ? b : l1;
    }
    if ((threadIdx.x & 31) == 0) {
        if (blt(l0, inf_r<real>()))
            atomicMin(&mins[2 * slot], (unsigned long long)__double_as_longlong((double)l0));
        if (blt(l1, inf_r<real>()))
            atomicMin(&mins[2 * slot + 1], (unsigned long long)__double_as_longlong((double)l1));
    }
}

// ---------------------------------------------------------------------------
// The bucket steps after the first: one launch runs up to nsteps of them with
// a grid barrier after each of the two phases of a step.
//
// A step only changes cells at or next to the BAND cells it accepts, so it
// visits the bricks with a BAND cell at or below the step's limit and their
// face neighbours (active bricks; CTA i owns the bricks i, i + CTAs, ..., so
// neighbours lie on different SMs, its threads look at the BAND minima of
// their bricks and the neighbours).
//   relax : acceptance is evaluated, not stored (a BAND cell at or below its
//           limit counts as KNOWN).  A warp stages an active brick and lists the
//           cells next to an accepted one; the cells of all its bricks are then
//           tested and solved into `next` by the threads of the whole CTA (a
//           step has one or two active bricks a CTA, and a warp with a brick of
//           its own would test and solve its 100 cells in turn);
//   apply : accepted cells become KNOWN, new values are applied, the brick's
//           BAND minima and the global ones are renewed.
// The solves read the same state as when every step streamed the whole grid in
// three launches, so the results are the same bits.  Spheres, second order, in
// double: 128^3 (1230 steps) 98.8 ms streaming, 38.6 with a warp per brick to the
// end of the phase, 32.9 so; 32^3 (180 steps) 4.6, 5.4, 3.9 ms.  A step is the
// slowest CTA's chain (stage, list, solve, two grid barriers): 20 us on the
// smallest grids, 27 on 128^3.  (On 32^3 in float, where a streamed step took
// 18 us, it is 1.18 against 1.07 ms in first order, 59 steps.)
// ---------------------------------------------------------------------------
constexpr int kStepWarps = 16;

template <typename real>
struct StepTile {
    real T[kTile3];          // brick and face halo
    uint8_t st[kTile3];      // 0 not usable, 1 KNOWN or FIX before the step, 3 accepted in it
    alignas(16) uint8_t tg[kB3];
    unsigned sel[32];        // per lane: cells next to an accepted halo cell
};
// What the warps of a CTA share in the relax phase: a brick's tile per warp, and
// the cells of all of them (warp << 9 | cell) to test and to solve.
template <typename real>
struct StepSmem {
    StepTile<real> tile[kStepWarps];
    uint16_t test[kStepWarps * kB3], solve[kStepWarps * kB3];
};

__device__ __forceinline__ unsigned long long ldu(const unsigned long long *p)
{
    return *(const volatile unsigned long long *)p;
}

// All blocks of the launch (co-resident: a cooperative launch); false when the
// wait ran out.  count only grows within a launch.
__device__ __forceinline__ bool grid_barrier(unsigned *count, unsigned target, Control *ctrl)
{
    __shared__ bool ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = true;
        __threadfence();
        atomicAdd(count, 1u);
        unsigned long long t0 = 0;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
        for (unsigned spin = 0; (int)(*(volatile unsigned *)count - target) < 0; ++spin) {
            if ((spin & 1023u) == 1023u) {
                unsigned long long t;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (t - t0 > ldu(&ctrl->wait_ns) || (*(volatile int *)&ctrl->error & ERR_SPIN)) {
                    atomicOr(&ctrl->error, ERR_SPIN);
                    ok = false;
                    break;
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok;
}

// brick coordinates (fewer than 2^32 bricks)
__device__ __forceinline__ void brick_at(const Geom &g, long long b, int &bx, int &by, int &bz)
{
    const unsigned r = (unsigned)b / (unsigned)g.nbx;
    bx = (int)((unsigned)b - r * (unsigned)g.nbx);
    bz = (int)(r / (unsigned)g.nby);
    by = (int)(r - (unsigned)bz * (unsigned)g.nby);
}

// brick across face f, or -1
__device__ __forceinline__ long long brick_next(const Geom &g, int bx, int by, int bz, int f)
{
    const int d = (f & 1) ? 1 : -1, a = f >> 1;
    const int x = bx + (a == 0 ? d : 0), y = by + (a == 1 ? d : 0), z = bz + (a == 2 ? d : 0);
    if (x < 0 || x >= g.nbx || y < 0 || y >= g.nby || z < 0 || z >= g.nbz)
        return -1;
    return ((long long)z * g.nby + y) * g.nbx + x;
}

// cell q (0..63) of face f of a brick
__device__ __forceinline__ int face_cell(int f, int q)
{
    const int u = q & 7, v = q >> 3, edge = (f & 1) ? kB - 1 : 0;
    return f < 2 ? edge + 8 * u + 64 * v : (f < 4 ? u + 8 * edge + 64 * v : u + 8 * v + 64 * edge);
}

// The limits of a brick's sides: BAND cells at or below them are accepted
// (negative: none).  One FP64 operation a side; the comparisons with them are
// integer ones (a float cell against the limit rounded down).
template <typename real>
struct Limits {
    real lim[2];
};
__device__ __forceinline__ double limit_down(double v, double) { return v; }
__device__ __forceinline__ float limit_down(double v, float) { return __double2float_rd(v); }
template <typename real>
__device__ __forceinline__ Limits<real> brick_limits(real bd, double bucket, double width, const double m[2],
                                                     const bool has[2])
{
    Limits<real> l;
#pragma unroll
    for (int sd = 0; sd < 2; ++sd) {
        const double v = m[sd] + bucket * (double)bd;
        l.lim[sd] = has[sd] ? limit_down(blt(width, v) ? width : v, (real)0) : (real)-1;
    }
    return l;
}
template <typename real>
__device__ __forceinline__ int cell_state(uint8_t t, real v, const Limits<real> &l)
{
    if (known(t))
        return 1;
    if ((t & ST_MASK) == ST_BAND && ble(v, l.lim[(t & TG_NEG) ? 0 : 1]))
        return 3;
    return 0;
}
// A float at or above m + bucket * bd, for telling which bricks may accept a
// cell (one too many only costs a visit).
__device__ __forceinline__ float float_up(double v)
{
    const int e = __double2hiint(v) >> 20;
    return e < 900 ? 1e-36f : e >= 1150 ? __int_as_float(0x7f800000) : f32_of(v) * 1.0000003f;
}
__device__ __forceinline__ float float_up(float v) { return v * 1.0000003f; }
__device__ __forceinline__ float float_down(double v)
{
    const int e = __double2hiint(v) >> 20;
    return e < 900 || e >= 1150 ? 0.0f : f32_of(v);
}
__device__ __forceinline__ float float_down(float v) { return v; }

template <typename real, int kAcc>
__global__ void __launch_bounds__(kStepWarps * 32)
    k_cell_steps(Geom g, real *T, uint8_t *tag, const real *__restrict__ spd, double spd_const, double wy, double wz,
                 const real *__restrict__ bdelta, double bucket, double width, real *next, real *bmin,
                 unsigned *active, unsigned long long *mins, unsigned *barrier, long long step, int nsteps, Control *ctrl)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    StepSmem<real> &sm = *reinterpret_cast<StepSmem<real> *>(smem_raw);
    StepTile<real> &W = sm.tile[warp];
    __shared__ unsigned long long bm[2];
    const real INF = inf_r<real>();
    const real wax[3] = {(real)1, (real)wy, (real)wz};
    const int off[3] = {1, kTile, kTile * kTile};
    const long long first = blockIdx.x, stride = gridDim.x;
    const long long owned = first < g.nbricks ? (g.nbricks - first + stride - 1) / stride : 0;
    constexpr int kThreadsStep = kStepWarps * 32;
    __shared__ unsigned alist[kThreadsStep];   // active bricks of a chunk
    __shared__ int an, n_test, n_solve;
    const float bucket_up = (float)bucket * 1.000001f;
    unsigned target = 0;
    unsigned long long accepted = 0, solves = 0;
    long long done_steps = 0;
    bool run = *(volatile int *)&ctrl->done == 0;
    for (int it = 0; it < nsteps && run; ++it, ++step) {
        const int slot = (int)(step & 1);
        const double m[2] = {__longlong_as_double((long long)ldu(&mins[2 * slot])),
                             __longlong_as_double((long long)ldu(&mins[2 * slot + 1]))};
        const double inf = __longlong_as_double((long long)kInfBits);
        const bool has[2] = {m[0] < inf && m[0] <= width, m[1] < inf && m[1] <= width};
        if (!has[0] && !has[1]) {
            if (blockIdx.x == 0 && threadIdx.x == 0)
                ctrl->done = 1;
            break;
        }
        ++done_steps;
        const float m_up[2] = {(float)m[0] * 1.000001f + 1e-37f, (float)m[1] * 1.000001f + 1e-37f};
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            mins[2 * (slot ^ 1)] = kInfBits;
            mins[2 * (slot ^ 1) + 1] = kInfBits;
        }
        // ---- relax --------------------------------------------------------
        for (long long i0 = 0; i0 < owned; i0 += kThreadsStep) {
            if (threadIdx.x == 0)
                an = 0;
            __syncthreads();
            if (i0 + threadIdx.x < owned) {
                const long long b = first + (i0 + threadIdx.x) * stride;
                int bx, by, bz;
                brick_at(g, b, bx, by, bz);
                bool act = false;
#pragma unroll
                for (int f = -1; f < 6; ++f) {
                    const long long q = f < 0 ? b : brick_next(g, bx, by, bz, f);
                    if (q < 0)
                        continue;
                    const real q0 = __ldcg(bmin + 2 * q), q1 = __ldcg(bmin + 2 * q + 1);
                    if (!blt(q0, INF) && !blt(q1, INF))
                        continue;
                    const float up = bucket_up * float_up(bdelta[q]);
                    act = act || (has[0] && blt(q0, INF) && !(float_down(q0) > m_up[0] + up)) ||
                          (has[1] && blt(q1, INF) && !(float_down(q1) > m_up[1] + up));
                }
                active[b] = act ? 1u : 0u;
                if (act)
                    alist[atomicAdd(&an, 1)] = (unsigned)b;
            }
            __syncthreads();
            for (int a0 = 0; a0 < an; a0 += kStepWarps) {
                if (threadIdx.x == 0)
                    n_test = n_solve = 0;
                __syncthreads();
                if (a0 + warp < an) {
                    const long long b = alist[a0 + warp], base = b * kB3;
                    int bx, by, bz;
                    brick_at(g, b, bx, by, bz);
                    const Limits<real> lb = brick_limits(bdelta[b], bucket, width, m, has);
                    // the brick and its halo, with what each cell is in this step
                    __syncwarp();
                    reinterpret_cast<uint4 *>(W.tg)[lane] = __ldcg(reinterpret_cast<const uint4 *>(tag + base) + lane);
                    W.sel[lane] = 0u;
                    real v[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k)
                        v[k] = __ldcg(T + base + lane + 32 * k);
                    // (all loads first)
                    real hv[12];
                    uint8_t ht[12];
                    real hd[6];
#pragma unroll
                    for (int f = 0; f < 6; ++f) {
                        const long long nb = brick_next(g, bx, by, bz, f);
                        hd[f] = nb >= 0 ? bdelta[nb] : (real)0;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const long long e = nb * kB3 + face_cell(f ^ 1, lane + 32 * h);
                            hv[2 * f + h] = nb >= 0 ? __ldcg(T + e) : INF;
                            ht[2 * f + h] = nb >= 0 ? __ldcg(tag + e) : (uint8_t)(TG_OUT | ST_FAR);
                        }
                    }
                    __syncwarp();
                    unsigned acc = 0, open = 0;   // accepted in this step; not FIX or padding
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const int c = lane + 32 * k, ti = tile_of(c);
                        const uint8_t t = W.tg[c];
                        const int st = cell_state(t, v[k], lb);
                        open |= (unsigned)(!(t & TG_OUT) && (t & ST_MASK) != ST_FIX) << k;
                        W.T[ti] = v[k];
                        W.st[ti] = (uint8_t)st;
                        acc |= (unsigned)(st == 3) << k;
                    }
#pragma unroll
                    for (int f = 0; f < 6; ++f) {
                        const Limits<real> ln = brick_limits(hd[f], bucket, width, m, has);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int st = cell_state(ht[2 * f + h], hv[2 * f + h], ln);
                            const int hi = tile_of(face_cell(f, lane + 32 * h)) + ((f & 1) ? off[f >> 1] : -off[f >> 1]);
                            W.T[hi] = hv[2 * f + h];
                            W.st[hi] = (uint8_t)st;
                            if (st == 3) {
                                const int c = face_cell(f, lane + 32 * h);
                                atomicOr(&W.sel[c & 31], 1u << (c >> 5));
                            }
                        }
                    }
                    __syncwarp();
                    // the cells next to an accepted one
                    const unsigned cand = (neighbour_mask(acc, lane) | W.sel[lane]) & open;
                    const int cnt = __popc(cand);
                    int pre = cnt;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int t = __shfl_up_sync(FULL, pre, o);
                        if (lane >= o)
                            pre += t;
                    }
                    int at = 0;
                    if (lane == 31 && pre)
                        at = atomicAdd(&n_test, pre);
                    at = __shfl_sync(FULL, at, 31) + pre - cnt;
                    for (unsigned q = cand; q; q &= q - 1u)
                        sm.test[at++] = (uint16_t)(warp << 9 | (lane + 32 * (__ffs((int)q) - 1)));
                }
                __syncthreads();
                // of them, the cells above an accepted neighbour
                for (int j0 = 32 * warp; j0 < n_test; j0 += kThreadsStep) {
                    const int i = j0 + lane;
                    const int e = i < n_test ? sm.test[i] : 0;
                    const StepTile<real> &X = sm.tile[e >> 9];
                    const int ti = tile_of(e & (kB3 - 1));
                    const real Tc = X.T[ti];
                    bool trig = false;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        trig = trig || (X.st[ti - off[a]] == 3 && blt(X.T[ti - off[a]], Tc));
                        trig = trig || (X.st[ti + off[a]] == 3 && blt(X.T[ti + off[a]], Tc));
                    }
                    const unsigned bal = __ballot_sync(FULL, trig && i < n_test);
                    int at = 0;
                    if (lane == 0 && bal)
                        at = atomicAdd(&n_solve, __popc(bal));
                    at = __shfl_sync(FULL, at, 0) + __popc(bal & ((1u << lane) - 1u));
                    if (trig && i < n_test)
                        sm.solve[at] = (uint16_t)e;
                }
                __syncthreads();
                solves += threadIdx.x == 0 ? (unsigned)n_solve : 0u;
                for (int i = threadIdx.x; i < n_solve; i += kThreadsStep) {
                    const int e = sm.solve[i], c = e & (kB3 - 1), ti = tile_of(c);
                    const StepTile<real> &X = sm.tile[e >> 9];
                    const long long b = alist[a0 + (e >> 9)], base = b * kB3;
                    const real Tc = X.T[ti];
                    const int cc[3] = {c & 7, (c >> 3) & 7, c >> 6};
                    real psi[3] = {(real)0, (real)0, (real)0}, wt[3] = {(real)0, (real)0, (real)0};
                    unsigned axes = 0;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const bool km = X.st[ti - off[a]] != 0, kp = X.st[ti + off[a]] != 0;
                        const real vm = km ? X.T[ti - off[a]] : INF, vp = kp ? X.T[ti + off[a]] : INF;
                        int d = 0;
                        if (km && blt(vm, Tc))
                            d = -1;
                        if (kp && blt(vp, Tc)) {
                            if (d == 0)
                                d = 1;
                            else if (blt(vp, vm))
                                d = 1;
                        }
                        if (d == 0)
                            continue;
                        axes |= 1u << a;
                        psi[a] = d < 0 ? vm : vp;
                        wt[a] = wax[a];
                        if (kAcc == 2) {
                            // the cell beyond the neighbour: in the tile, or
                            // the second layer of the brick across the face
                            bool k2 = false;
                            real v2 = (real)0;
                            const int c2 = cc[a] + 2 * d;
                            if (c2 >= -1 && c2 <= kB) {
                                k2 = X.st[ti + 2 * d * off[a]] != 0;
                                v2 = X.T[ti + 2 * d * off[a]];
                            } else {
                                int bx, by, bz;
                                brick_at(g, b, bx, by, bz);
                                const long long nb = brick_next(g, bx, by, bz, 2 * a + (d > 0 ? 1 : 0));
                                if (nb >= 0) {
                                    const int step_c = a == 0 ? 1 : (a == 1 ? 8 : 64);
                                    const long long q2 = nb * kB3 + c + ((c2 & 7) - cc[a]) * step_c;
                                    v2 = __ldcg(T + q2);
                                    k2 = cell_state(__ldcg(tag + q2), v2,
                                                    brick_limits(bdelta[nb], bucket, width, m, has)) != 0;
                                }
                            }
                            if (k2 && ble(v2, psi[a])) {
                                psi[a] = ((real)4 * psi[a] - v2) / (real)3;
                                wt[a] = wt[a] * (real)2.25;
                            }
                        }
                    }
                    const real q = spd ? spd[base + c] : (real)spd_const;
                    const real r = cell_root<real>(psi, wt, axes, q);
                    if (blt(r, Tc))
                        next[base + c] = r;
                }
                __syncthreads();
            }
        }
        target += gridDim.x;
        run = grid_barrier(barrier, target, ctrl);
        // ---- apply --------------------------------------------------------
        if (threadIdx.x < 2)
            bm[threadIdx.x] = kInfBits;
        __syncthreads();
        unsigned long long w0 = kInfBits, w1 = kInfBits;
        for (long long i0 = 0; i0 < owned && run; i0 += kThreadsStep) {
            real b0 = INF, b1 = INF;
            if (threadIdx.x == 0)
                an = 0;
            __syncthreads();
            if (i0 + threadIdx.x < owned) {
                const long long b = first + (i0 + threadIdx.x) * stride;
                if (active[b] != 0u) {
                    alist[atomicAdd(&an, 1)] = (unsigned)b;
                } else {
                    b0 = __ldcg(bmin + 2 * b);
                    b1 = __ldcg(bmin + 2 * b + 1);
                }
            }
            __syncthreads();
            for (int ai = warp; ai < an; ai += kStepWarps) {
                const long long b = alist[ai], base = b * kB3;
                const Limits<real> lb = brick_limits(bdelta[b], bucket, width, m, has);
                real l0 = INF, l1 = INF;
                real v[16], nv[16];
                uint8_t tg[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    v[k] = __ldcg(T + base + lane + 32 * k);
                    nv[k] = __ldcg(next + base + lane + 32 * k);
                    tg[k] = __ldcg(tag + base + lane + 32 * k);
                }
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const long long e = base + lane + 32 * k;
                    const uint8_t t = tg[k];
                    if (t & TG_OUT)
                        continue;
                    uint8_t nt = t;
                    if (cell_state(t, v[k], lb) == 3) {
                        nt = (uint8_t)((t & ~ST_MASK) | ST_KNOWN);
                        ++accepted;
                    }
                    if (!is_none(nv[k])) {
                        v[k] = nv[k];
                        T[e] = nv[k];
                        next[e] = none_r<real>();
                        nt = (uint8_t)((nt & ~ST_MASK) | ST_BAND);
                    }
                    if (nt != t)
                        tag[e] = nt;
                    if ((nt & ST_MASK) == ST_BAND) {
                        if (nt & TG_NEG)
                            l0 = blt(v[k], l0) ? v[k] : l0;
                        else
                            l1 = blt(v[k], l1) ? v[k] : l1;
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const real x = __shfl_xor_sync(FULL, l0, o), y = __shfl_xor_sync(FULL, l1, o);
                    l0 = blt(x, l0) ? x : l0;
                    l1 = blt(y, l1) ? y : l1;
                }
                if (lane == 0) {
                    bmin[2 * b] = l0;
                    bmin[2 * b + 1] = l1;
                    b0 = blt(l0, b0) ? l0 : b0;
                    b1 = blt(l1, b1) ? l1 : b1;
                }
            }
            __syncthreads();
            const unsigned long long u0 = (unsigned long long)__double_as_longlong((double)b0),
                                     u1 = (unsigned long long)__double_as_longlong((double)b1);
            w0 = u0 < w0 ? u0 : w0;
            w1 = u1 < w1 ? u1 : w1;
        }
        if (w0 < kInfBits)
            atomicMin(&bm[0], w0);
        if (w1 < kInfBits)
            atomicMin(&bm[1], w1);
        __syncthreads();
        if (threadIdx.x < 2 && bm[threadIdx.x] < kInfBits)
            atomicMin(&mins[2 * (slot ^ 1) + threadIdx.x], bm[threadIdx.x]);
        target += gridDim.x;
        run = run && grid_barrier(barrier, target, ctrl);
    }
    solves = __shfl_sync(FULL, solves, 0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        accepted += __shfl_xor_sync(FULL, accepted, o);
    if (lane == 0) {
        if (accepted)
            atomicAdd(&ctrl->accepted, accepted);
        if (solves)
            atomicAdd(&ctrl->solves, solves);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0)
        ctrl->restart += (int)done_steps;
}

// BAND minima of every brick (the state the steps above start from).
template <typename real>
__global__ void __launch_bounds__(kCellThreads) k_cell_brick_min(Geom g, const real *__restrict__ T,
                                                                const uint8_t *__restrict__ tag, real *bmin)
{
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (kCellThreads / 32);
    for (long long b = (long long)blockIdx.x * (kCellThreads / 32) + (threadIdx.x >> 5); b < g.nbricks; b += warps) {
        real l0 = inf_r<real>(), l1 = inf_r<real>();
        for (int k = 0; k < 16; ++k) {
            const long long e = b * kB3 + lane + 32 * k;
            const uint8_t t = tag[e];
            if ((t & ST_MASK) != ST_BAND || (t & TG_OUT))
                continue;
            const real v = T[e];
            if (t & TG_NEG)
                l0 = blt(v, l0) ? v : l0;
            else
                l1 = blt(v, l1) ? v : l1;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const real x = __shfl_xor_sync(FULL, l0, o), y = __shfl_xor_sync(FULL, l1, o);
            l0 = blt(x, l0) ? x : l0;
            l1 = blt(y, l1) ? y : l1;
        }
        if (lane == 0) {
            bmin[2 * b] = l0;
            bmin[2 * b + 1] = l1;
        }
    }
}

int cell_grid(long long n)
{
    long long b = (n + kCellThreads - 1) / kCellThreads;
    const long long cap = 152LL * 16;
    if (b < 1)
        b = 1;
    return (int)(b > cap ? cap : b);
}

template <typename real>
void relax_launch(const Geom &g, const DeviceState &s, const SolveParams &p, void *next, int nb,
                  cudaStream_t st)
{
    const real *spd = (const real *)s.spd;
    if (p.accuracy == 2)
        k_cell_relax<real, 2><<<nb, kCellThreads, 0, st>>>(g, (const real *)s.T, s.tag, spd, p.spd_term,
                                                           p.wy, p.wz, (real *)next, s.ctrl);
    else
        k_cell_relax<real, 1><<<nb, kCellThreads, 0, st>>>(g, (const real *)s.T, s.tag, spd, p.spd_term,
                                                           p.wy, p.wz, (real *)next, s.ctrl);
}

template <typename real>
cudaError_t begin_t(const Geom &g, const DeviceState &s, const SolveParams &p, void *next,
                    unsigned long long *mins, cudaStream_t st)
{
    const int nb = cell_grid(g.nbricks * kB3);
    k_cell_seed<real><<<nb, kCellThreads, 0, st>>>(g, s.tag, (real *)next, mins);
    relax_launch<real>(g, s, p, next, nb, st);
    k_cell_apply<real><<<nb, kCellThreads, 0, st>>>(g, (real *)s.T, s.tag, (real *)next, mins, 0, s.ctrl);
    k_cell_brick_min<real><<<cell_grid(g.nbricks * 32), kCellThreads, 0, st>>>(g, (const real *)s.T, s.tag,
                                                                              (real *)s.bmin);
    return cudaGetLastError();
}

template <typename real, int kAcc>
cudaError_t steps_t(const Geom &g, const DeviceState &s, const SolveParams &p, void *next, unsigned long long *mins,
                    long long step, int n, cudaStream_t st)
{
    const size_t sm = sizeof(StepSmem<real>);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cell_steps<real, kAcc>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess)
        return e;
    // one CTA per SM (the barrier costs with every CTA), no more than there are bricks
    const int nb = (int)(g.nbricks < sms ? g.nbricks : sms);
    unsigned *barrier = (unsigned *)(mins + 4);
    e = cudaMemsetAsync(barrier, 0, sizeof(unsigned), st);
    if (e != cudaSuccess)
        return e;
    Geom gg = g;
    real *T = (real *)s.T, *nx = (real *)next, *bmin = (real *)s.bmin;
    uint8_t *tag = s.tag;
    const real *spd = (const real *)s.spd, *bd = (const real *)s.bdelta;
    double sc = p.spd_term, wy = p.wy, wz = p.wz, bucket = p.bucket, width = p.width;
    unsigned *active = s.dirty;
    Control *ctrl = s.ctrl;
    void *args[] = {&gg, &T, &tag, &spd, &sc, &wy, &wz, &bd, &bucket, &width, &nx, &bmin, &active, &mins, &barrier, &step,
                    &n, &ctrl};
    return cudaLaunchCooperativeKernel((const void *)k_cell_steps<real, kAcc>, dim3(nb), dim3(kStepWarps * 32), args, sm, st);
}

}  // namespace

cudaError_t launch_init_fixed(int dtype, const Geom &g, const DeviceState &s, const void *T0,
                              cudaStream_t st)
{
    const int nb = cell_grid(g.nbricks * kB3);
    if (dtype == 1)
        k_init_fixed<double><<<nb, kCellThreads, 0, st>>>(g, (const double *)T0, (double *)s.T, s.tag, s.ctrl);
    else
        k_init_fixed<float><<<nb, kCellThreads, 0, st>>>(g, (const float *)T0, (float *)s.T, s.tag, s.ctrl);
    return cudaGetLastError();
}

cudaError_t launch_cell_begin(int dtype, const Geom &g, const DeviceState &s, const SolveParams &p,
                              void *next, unsigned long long *mins, cudaStream_t st)
{
    return dtype == 1 ? begin_t<double>(g, s, p, next, mins, st) : begin_t<float>(g, s, p, next, mins, st);
}

cudaError_t launch_cell_steps(int dtype, const Geom &g, const DeviceState &s, const SolveParams &p, void *next,
                              unsigned long long *mins, long long step, int n, cudaStream_t st)
{
    if (p.accuracy == 2)
        return dtype == 1 ? steps_t<double, 2>(g, s, p, next, mins, step, n, st)
                          : steps_t<float, 2>(g, s, p, next, mins, step, n, st);
    return dtype == 1 ? steps_t<double, 1>(g, s, p, next, mins, step, n, st)
                      : steps_t<float, 1>(g, s, p, next, mins, step, n, st);
}

}  // namespace fmmgb
