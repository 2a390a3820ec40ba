// fmm_sweep.cuh -- the local march of one 8^3 brick by one warp, as ordered
// sweeps of Algorithm 11 over the brick in shared memory.
//
// The fixed point of Algorithms 10-12 inside a brick does not depend on the
// order of the updates (values only fall, every fall re-triggers the
// neighbours), so the heap of Algorithm 12 is replaced by plane-ordered
// Gauss-Seidel sweeps: a sweep visits the cells by x' + y' + z' = 0 .. 21,
// with each axis running up or down (8 octants).  All cells of one such level
// are independent, and a sweep whose octant is the direction the front
// crosses the brick in solves every cell once, from final values.  Most
// bricks need one sweep of 30 warp steps.
//
// (The bucketed march this replaced solved a cell 8.9 times and issued 226 /
// 101 warp instructions per grid point in double / float on the 512^3 sphere; a
// sweep solves it once, and with bricks marched 2.2 / 1.9 times there 42.3 / 18.4
// instructions are issued.)
//
// What tells that a sweep was enough: a cell n is solved from the level
// before it (final in this sweep) and the level after it (as it was).  It can
// need another solve only if a cell c' of the next level then fell below it,
// so when c' improves it is compared with its three neighbours of the level
// before (their values are in registers).  No such case: every cell is the
// root of its neighbours and the march is done.  Otherwise the neighbours
// found are marked and the axes on which it happened say which octant the
// next sweep runs in.  When few cells are marked, and when a brick marches
// again because halo cells changed, the cells are solved from a packed list
// instead, and each one that improves marks its neighbours above it.
//
// A step is a chain of shared-memory load, minima, sort, root, compare and store
// (75 instructions in float); in double, a double addition takes the FP64 pipe 16
// cycles a warp.  On the 512^3 sphere, where 44 / 31% of the warp slots are active,
// the march of a brick takes an SM 3000 / 5100 cycles in float / double.
#pragma once

#include "fmm_internal.h"
#include "fmm_df.cuh"
#include "fmm_fp64.cuh"

#include <cmath>

namespace fmmgb {
namespace {

constexpr unsigned FULL = 0xffffffffu;


// ---------------------------------------------------------------------------
// value helpers
// ---------------------------------------------------------------------------

template <typename real>
__device__ __forceinline__ real inf_v();
template <>
__device__ __forceinline__ float inf_v<float>() { return __int_as_float(0x7f800000); }
template <>
__device__ __forceinline__ double inf_v<double>() { return __longlong_as_double(0x7ff0000000000000ll); }

__device__ __forceinline__ bool is_known(uint8_t tg) { return (tg & ST_MASK) >= ST_KNOWN; }

// |psi| values are never negative, so double comparisons are done on the
// bit patterns (integer compares keep them off the FP64 pipe).
__device__ __forceinline__ bool lt(double a, double b)
{
    // valid for values >= 0 and +inf; a negative discriminant has the sign
    // bit set and compares below every non-negative value
    return __double_as_longlong(a) < __double_as_longlong(b);
}
__device__ __forceinline__ bool lt(float a, float b) { return a < b; }
__device__ __forceinline__ double vmin(double a, double b) { return lt(a, b) ? a : b; }
__device__ __forceinline__ float vmin(float a, float b) { return fminf(a, b); }

// Marks (bounded marches): a brick cell that no neighbour may use yet (above
// the bound and not FIX) carries the sign bit.  Compared as unsigned bit
// patterns a marked entry orders above every value including +inf.
__device__ __forceinline__ bool klt(double a, double b)
{
    return (unsigned long long)__double_as_longlong(a) < (unsigned long long)__double_as_longlong(b);
}
__device__ __forceinline__ bool klt(float a, float b) { return __float_as_uint(a) < __float_as_uint(b); }
__device__ __forceinline__ double kmin(double a, double b) { return klt(a, b) ? a : b; }
__device__ __forceinline__ float kmin(float a, float b)
{
    return __uint_as_float(umin(__float_as_uint(a), __float_as_uint(b)));
}
// mark / unmark (set / clear the sign bit, on the high word of a double)
__device__ __forceinline__ double kmark(double v)
{
    return __hiloint2double(__double2hiint(v) | (int)0x80000000, __double2loint(v));
}
__device__ __forceinline__ float kmark(float v) { return __uint_as_float(__float_as_uint(v) | 0x80000000u); }
__device__ __forceinline__ double kval(double v)
{
    return __hiloint2double(__double2hiint(v) & 0x7fffffff, __double2loint(v));
}
__device__ __forceinline__ float kval(float v) { return __uint_as_float(__float_as_uint(v) & 0x7fffffffu); }
__device__ __forceinline__ bool kmarked(double v) { return __double2hiint(v) < 0; }
__device__ __forceinline__ bool kmarked(float v) { return __float_as_int(v) < 0; }

// Warp minimum of non-negative values (or +inf): their bit patterns order
// like the values, so the integer reductions of the warp do it exactly (a
// double in two steps, high word then low word).
__device__ __forceinline__ float warp_min(float v)
{
    return __uint_as_float(__reduce_min_sync(FULL, __float_as_uint(v)));
}
__device__ __forceinline__ double warp_min(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned hi = __reduce_min_sync(FULL, (unsigned)(b >> 32));
    const unsigned lo = __reduce_min_sync(FULL, (unsigned)(b >> 32) == hi ? (unsigned)b : 0xffffffffu);
    return __longlong_as_double((long long)(((unsigned long long)hi << 32) | lo));
}
// the part of a value that orders it coarsely: the whole float, the high
// word of a double
__device__ __forceinline__ unsigned order_word(float v) { return __float_as_uint(v); }
__device__ __forceinline__ unsigned order_word(double v) { return (unsigned)__double2hiint(v); }

// Double square root without the FP64 pipe's slow conversions (fmm_fp64.cuh).
__device__ __forceinline__ double vsqrt(double v) { return sqrt_fp64(v); }
// Single precision: the hardware estimate (about one ulp; sqrt(+inf) = +inf, so
// an obstacle cell's candidate is +inf).
__device__ __forceinline__ float vsqrt(float v) { return sqrt_est(v); }
__device__ __forceinline__ float vdiv(float a, float b) { return a / b; }
__device__ __forceinline__ double vdiv(double a, double b) { return div_fp64(a, b); }

// ---------------------------------------------------------------------------
// Algorithm 11 (Solve_Quadratic_Parallel) from the per-axis upwind values
// v[a] (the smaller usable neighbour of the axis, +inf when there is none).
//
// The quadratic sum_i (t - psi_i)^2 / h^2 = 1/F^2 over the upwind set is
// solved for the unknown shifted by the smallest upwind value m: t = m + u,
// delta_i = psi_i - m, sum_i (u - delta_i)^2 = q with q = (h/F)^2.  The
// coefficients stay of order h, so rounding does not grow with psi (in psi
// itself b^2 and 4ac would cancel to ~3 (psi F/h)^2 ulp).
//
// Algorithm 11 keeps the smallest causal root over the nested sets, each time
// dropping the largest psi_i; going from the full set down, the first causal
// root already is that minimum: a causal root t_S of a nested set S satisfies
// sum over all axes of max(t_S - psi_i, 0)^2 >= (h/F)^2, so t_S is never
// below the unique solution t* of sum max(t - psi_i, 0)^2 = (h/F)^2, and t*
// is the causal root of the set {i : psi_i < t*}.  Neighbours at or above the
// cell's own value need no test of their own: a causal root that uses one is
// above it and so no improvement.
//
// The causality test psi_i < t is delta_i < u; the kernels that record the
// upwind sets for the adjoint make it on t = m + u and the values the cells
// hold (on rounded shifts delta_i < u can hold while t rounds to psi_i, and a
// recorded set must point strictly downhill).  set_out receives the upwind
// set (2 bits per axis: 1 = minus, 2 = plus neighbour).
// ---------------------------------------------------------------------------

template <typename real>
__device__ __forceinline__ void cswap(real &a, unsigned &ca, real &b, unsigned &cb)
{
    if (lt(b, a)) {
        const real t = a;
        a = b;
        b = t;
        const unsigned c = ca;
        ca = cb;
        cb = c;
    }
}

template <typename real, bool kTape>
__device__ __forceinline__ real solve_axes(const real vin[3], const unsigned cin[3], real q, uint8_t &set_out)
{
    const real INF = inf_v<real>();
    real v[3] = {vin[0], vin[1], vin[2]};
    unsigned code[3] = {cin[0], cin[1], cin[2]};
    set_out = 0;
    if constexpr (!kTape && sizeof(real) == 4) {
        // without sides to carry along: a min / max network
        const float a = fminf(v[0], v[1]), b = fmaxf(v[0], v[1]);
        const float d = fminf(b, v[2]);
        v[2] = fmaxf(b, v[2]);
        v[0] = fminf(a, d);
        v[1] = fmaxf(a, d);
    } else {
        // stable sort of three (adjacent compare-exchange, strict less-than):
        // equal values keep the lower axis first, the higher is dropped first
        cswap(v[0], code[0], v[1], code[1]);
        cswap(v[1], code[1], v[2], code[2]);
        cswap(v[0], code[0], v[1], code[1]);
    }
    const real m = v[0];
    if constexpr (sizeof(real) == 8) {
        if (!lt(m, INF))
            return INF;
        // double grids: fmm_df.cuh, unless the speed term is outside its
        // range (an obstacle's +inf)
        if (in_float_range(q)) {
            double t = 0.0;
            const int k = df_root<kTape>(m, v[1], v[2], df_speed(q), q, t);
            if (kTape)
                set_out = (uint8_t)(code[0] | (k >= 2 ? code[1] : 0u) | (k == 3 ? code[2] : 0u));
            return k ? t : INF;
        }
    }
    if constexpr (!kTape && sizeof(real) == 4) {
        // the set grows while its root exceeds the next shift, as in df_root;
        // an absent axis is +inf and its root NaN or unused, and with m = +inf
        // the result is +inf or NaN, which is below nothing
        const float d1 = v[1] - m, d2 = v[2] - m, e = d2 - d1, f1 = d1 * d1, s = vsqrt(q);
        const float u2 = 0.5f * (d1 + vsqrt(fmaf(2.0f, q, -f1)));
        const float u = d1 < s ? u2 : s;
        const float u3 = ((d1 + d2) + vsqrt(fmaf(3.0f, q, -fmaf(d2, d2, fmaf(e, e, f1))))) * (float)(1.0 / 3.0);
        return m + (d2 < u ? u3 : u);
    }
    // The set is chosen by the residual of the smaller ones (a two-value set
    // is causal when delta_1^2 < q, a three-value set when delta_2^2 +
    // (delta_2 - delta_1)^2 < q), then one root is evaluated.  Absent axes
    // are +inf and fail the tests; with m = +inf the root is +inf or NaN,
    // which is below nothing.
    const real d1 = v[1] - m, d2 = v[2] - m, e = d2 - d1;
    const real f1 = d1 * d1, f2 = fma(d2, d2, e * e);
    bool c1 = f1 < q, c2 = c1 && f2 < q;
#pragma unroll 1
    for (;;) {
        const real k = c2 ? (real)3 : (c1 ? (real)2 : (real)1);
        const real inv_k = c2 ? (real)(1.0 / 3.0) : (c1 ? (real)0.5 : (real)1);
        const real S = (c1 ? d1 : (real)0) + (c2 ? d2 : (real)0);
        const real disc = fma(k, q, -((c1 ? f1 : (real)0) + (c2 ? f2 : (real)0)));
        const real t = fma(S + vsqrt(disc), inv_k, m);
        if constexpr (kTape) {
            // the recorded set points strictly downhill
            if (c1 && !lt(c2 ? v[2] : v[1], t)) {
                c1 = c2;
                c2 = false;
                continue;
            }
            set_out = (uint8_t)(code[0] | (c1 ? code[1] : 0u) | (c2 ? code[2] : 0u));
        }
        return t;
    }
}

// Algorithm 11 with cells of size h * hy * hz: h_i^2 (t - psi_i)^2 summed
// over the set equals F^-2, i.e. sum_i w_i (u - delta_i)^2 = q with
// w_i = (h / h_i)^2 (w_x = 1), q = (h/F)^2 and the same shift t = m + u.
// The per-axis values are sorted together with their weights (and sides);
// with K = sum w_i, S = sum w_i delta_i and Q = sum w_i delta_i^2 over the
// set, disc = S^2 - K (Q - q), evaluated as K q - sum_{i<j} w_i w_j
// (delta_i - delta_j)^2, and u = (S + sqrt(disc)) / K; the largest remaining
// value is dropped while the set is not causal, as above.
template <typename real>
__device__ __forceinline__ void cswap_w(real &a, real &wa, unsigned &ca, real &b, real &wb, unsigned &cb)
{
    if (lt(b, a)) {
        const real t = a, tw = wa;
        a = b;
        b = t;
        wa = wb;
        wb = tw;
        const unsigned c = ca;
        ca = cb;
        cb = c;
    }
}

template <typename real, bool kTape>
__device__ __forceinline__ real solve_axes_w(const real vin[3], const unsigned cin[3], real q, real wy, real wz,
                                             uint8_t &set_out)
{
    const real INF = inf_v<real>();
    real v[3] = {vin[0], vin[1], vin[2]}, w[3] = {(real)1, wy, wz};
    unsigned code[3] = {cin[0], cin[1], cin[2]};
    set_out = 0;
    // stable sort of three, each weight and side with its value
    cswap_w(v[0], w[0], code[0], v[1], w[1], code[1]);
    cswap_w(v[1], w[1], code[1], v[2], w[2], code[2]);
    cswap_w(v[0], w[0], code[0], v[1], w[1], code[1]);
    const real m = v[0];
    if (!lt(m, INF))
        return INF;
    // the set by its residuals, then one root, as in solve_axes
    const real d1 = v[1] - m, d2 = v[2] - m, e = d2 - d1;
    bool c1 = w[0] * (d1 * d1) < q, c2 = c1 && fma(w[1], e * e, w[0] * (d2 * d2)) < q;
#pragma unroll 1
    for (;;) {
        const real w1 = c1 ? w[1] : (real)0, w2 = c2 ? w[2] : (real)0;
        const real x1 = c1 ? d1 : (real)0, x2 = c2 ? d2 : (real)0, x3 = c2 ? e : (real)0;
        const real K = w[0] + w1 + w2;
        const real S = fma(w1, x1, w2 * x2);
        // S^2 - K (Q - q) = K q - sum_{i<j} w_i w_j (delta_i - delta_j)^2
        // (Lagrange's identity): with unequal weights S^2 and K Q nearly
        // cancel, the pairwise form does not
        const real P = fma(w[0] * w1, x1 * x1, fma(w[0] * w2, x2 * x2, (w1 * w2) * (x3 * x3)));
        const real t = m + vdiv(S + vsqrt(fma(K, q, -P)), K);
        if constexpr (kTape) {
            if (c1 && !lt(c2 ? v[2] : v[1], t)) {
                c1 = c2;
                c2 = false;
                continue;
            }
            set_out = (uint8_t)(code[0] | (c1 ? code[1] : 0u) | (c2 ? code[2] : 0u));
        }
        return t;
    }
}

// ---------------------------------------------------------------------------
// The brick in shared memory.
// ---------------------------------------------------------------------------

// The brick and its face halo in one 10^3 tile (x fastest), shifted by one
// entry so that every row of 8 brick cells starts on a 16-byte boundary in
// double and an 8-byte boundary in float: kMT0 is the tile index of brick
// cell (0, 0, 0), kMH0 that of halo position (0, 0, 0).  A brick cell holds
// its current |psi| (with the sign bit set where a bounded march may not use
// it yet); a halo cell holds the neighbour's usable value or +inf.
constexpr int kMH0 = 1;
constexpr int kPlane = kTile * kTile;
constexpr int kMT0 = kMH0 + 1 + kTile + kPlane;
constexpr int kMTile = kMH0 + kTile * kPlane + 1;

constexpr int kListCells = 256;
template <typename real, bool kTape>
struct WarpTile {
    alignas(16) real kv[kMTile];                // brick and face halo
    alignas(16) uint8_t tg[kB3];                // tags as staged
    alignas(16) uint8_t chg[kB3];               // 1: the value fell in this march
    alignas(16) unsigned mark[32];              // per lane: cells to solve again
    alignas(16) uint16_t list[kListCells];      // those cells, packed
    alignas(16) uint8_t tp[kTape ? kB3 : 16];   // upwind sets (with a tape)
};
static_assert(sizeof(WarpTile<float, false>) % 16 == 0 && sizeof(WarpTile<double, false>) % 16 == 0 &&
                  sizeof(WarpTile<float, true>) % 16 == 0 && sizeof(WarpTile<double, true>) % 16 == 0,
              "every warp's tile starts on a 16-byte boundary");
static_assert((kMT0 * 8) % 16 == 0 && (kTile * 8) % 16 == 0 && (kMT0 * 4) % 8 == 0 && (kTile * 4) % 8 == 0 && (kPlane * 8) % 16 == 0,
              "brick rows of the tile start on 16 (double) / 8 (float) byte boundaries");

// tile index of brick cell c
__device__ __forceinline__ int mt_of(int c)
{
    return kMT0 + (c & 7) + kTile * ((c >> 3) & 7) + kPlane * (c >> 6);
}

// The q-th 16 bytes of a brick in brick order (cells c = x + 8 y + 64 z) to
// and from the tile rows: two cells per 16 bytes in double (four per row),
// four in float (two per row, stored as two 8-byte halves).  row_load clears
// the marks: the brick in global memory holds |psi|.
__device__ __forceinline__ void row_store(double *kv, int q, uint4 x)
{
    const int row = q >> 2;   // y + 8 z
    reinterpret_cast<uint4 *>(kv + kMT0 + kTile * (row & 7) + kPlane * (row >> 3))[q & 3] = x;
}
__device__ __forceinline__ void row_store(float *kv, int q, uint4 x)
{
    const int row = q >> 1;
    uint2 *d = reinterpret_cast<uint2 *>(kv + kMT0 + kTile * (row & 7) + kPlane * (row >> 3) + 4 * (q & 1));
    d[0] = make_uint2(x.x, x.y);
    d[1] = make_uint2(x.z, x.w);
}
__device__ __forceinline__ uint4 row_load(const double *kv, int q)
{
    const int row = q >> 2;
    uint4 x = reinterpret_cast<const uint4 *>(kv + kMT0 + kTile * (row & 7) + kPlane * (row >> 3))[q & 3];
    x.y &= 0x7fffffffu;   // high words
    x.w &= 0x7fffffffu;
    return x;
}
__device__ __forceinline__ uint4 row_load(const float *kv, int q)
{
    const int row = q >> 1;
    const uint2 *d =
        reinterpret_cast<const uint2 *>(kv + kMT0 + kTile * (row & 7) + kPlane * (row >> 3) + 4 * (q & 1));
    const uint2 a = d[0], b = d[1];
    return make_uint4(a.x & 0x7fffffffu, a.y & 0x7fffffffu, b.x & 0x7fffffffu, b.y & 0x7fffffffu);
}

// Brick cell and halo position of cell q (0..63) of face f: in-face
// coordinates u = q % 8, v = q / 8 over the two other axes, lower axis first.
__device__ __forceinline__ int face_cell(int f, int q, bool far_side)
{
    const int u = q & 7, v = q >> 3, axis = f >> 1;
    const int edge = ((f & 1) != 0) != far_side ? kB - 1 : 0;
    return axis == 0 ? edge + 8 * u + 64 * v : (axis == 1 ? u + 8 * edge + 64 * v : u + 8 * v + 64 * edge);
}
__device__ __forceinline__ int face_halo(int f, int q)
{
    const int axis = f >> 1;
    const int step = axis == 0 ? 1 : (axis == 1 ? kTile : kPlane);
    return mt_of(face_cell(f, q, false)) + ((f & 1) ? step : -step);
}

// ---------------------------------------------------------------------------
// Sweep order: the cells of the canonical octant (all axes up) by level
// x + y + z, at most 32 of one level per step.  Entry: bytes x, y, z and in
// the top byte bit a set when coordinate a is above 0 (the neighbour of the
// level before on that axis lies in the brick); -1: no cell.  The cell of
// another octant comes from signed strides: one byte dot product gives its
// tile index, another its cell index.
// ---------------------------------------------------------------------------
constexpr int kSweepSteps = 30;
struct SweepOrder {
    int e[(kSweepSteps + 1) * 32];
};
constexpr SweepOrder make_sweep_order()
{
    SweepOrder o{};
    int step = 0;
    for (int lev = 0; lev <= 3 * (kB - 1); ++lev) {
        int n = 0;
        for (int z = 0; z < kB; ++z)
            for (int y = 0; y < kB; ++y) {
                const int x = lev - y - z;
                if (x < 0 || x >= kB)
                    continue;
                o.e[32 * (step + n / 32) + n % 32] =
                    x | y << 8 | z << 16 | ((x > 0 ? 1 : 0) | (y > 0 ? 2 : 0) | (z > 0 ? 4 : 0)) << 24;
                ++n;
            }
        for (; n % 32 != 0; ++n)
            o.e[32 * (step + n / 32) + n % 32] = -1;
        step += n / 32;
    }
    for (int l = 0; l < 32; ++l)
        o.e[32 * kSweepSteps + l] = step == kSweepSteps ? -1 : 1 << 30;   // the row the last prefetch reads
    return o;
}
// (kept in global memory, copied to shared memory by every CTA: the fences of
// the brick queue empty the L1, and a step waits for its table entry)
constexpr SweepOrder kSweepOrderHost = make_sweep_order();
static_assert(kSweepOrderHost.e[32 * kSweepSteps] == -1, "30 steps per sweep");
__device__ const SweepOrder kSweepOrder = make_sweep_order();

__device__ __forceinline__ void load_sweep_order(int *order)
{
    for (int i = threadIdx.x; i < (kSweepSteps + 1) * 32; i += blockDim.x)
        order[i] = kSweepOrder.e[i];
    __syncthreads();
}

__device__ __forceinline__ int pack_strides(int x, int y, int z)
{
    return (x & 255) | (y & 255) << 8 | (z & 255) << 16;
}

// A brick with more cells to solve again than this is swept, one with fewer
// takes them cell by cell.  With a speed field in double a front turns inside
// the brick and bricks march again for many small corrections, which reach few
// cells at a time: 60^3 / 100^3 / 200^3 random speed, 4 sources, 6.4 / 8.6 /
// 21.1 ms at 64 cells, 4.9 / 7.4 / 17.6 at 160, 4.2 / 6.7 / 16.4 at 256.
// Without one the sweeps win: 64^3 point source 0.97 ms at 96 cells, 1.15 at
// 160; 1024^3 sphere 59 against 61; in float 4.0 / 3.9 / 4.2 / 4.6 ms at 64 /
// 96 / 160 / 256 (250^3 random speed).
template <typename real, bool kHetero>
__host__ __device__ constexpr int sweep_cells() { return kHetero && sizeof(real) == 8 ? 256 : 96; }
__device__ __forceinline__ void mark_cell(unsigned *mark, int c) { atomicOr(&mark[c & 31], 1u << (c >> 5)); }

struct MarchStats {
    unsigned long long marches, rounds, accepted, exchanges, solves;
};

// What a brick's march sends to its neighbours, in the lane of the face
// (0..5): the boundary cells that changed, the brick across the face, and the
// smallest of the changed values per side (+inf: none).  Every lane: the
// brick's BAND minima per side.
template <typename real>
struct Notify {
    unsigned long long m;
    long long nb;
    real v[2];
    real band[2];
};

// The cells to solve of a brick that marched before, to a lower bound: every cell
// is the root of what was usable then (of the FIX cells before the first march),
// so they are the cells above a neighbour that became usable (BAND, within the
// bound now) or above a halo value.  Marks them.  (Not inlined: the march has no registers left for it.)
template <typename real>
__device__ __noinline__ void reopened_cells(const real *kv, const uint8_t *tg, unsigned *mark, int lane)
{
#pragma unroll 1
    for (int k = 0; k < 16; ++k) {
        const int c = lane + 32 * k;
        const real *kp = kv + mt_of(c);
        if ((tg[c] & ST_MASK) != ST_BAND || kmarked(kp[0]))
            continue;
        const int cx = c & 7, cy = (c >> 3) & 7, cz = c >> 6;
        if (cx > 0 && lt(kp[0], kval(kp[-1])))
            mark_cell(mark, c - 1);
        if (cx < 7 && lt(kp[0], kval(kp[1])))
            mark_cell(mark, c + 1);
        if (cy > 0 && lt(kp[0], kval(kp[-kTile])))
            mark_cell(mark, c - 8);
        if (cy < 7 && lt(kp[0], kval(kp[kTile])))
            mark_cell(mark, c + 8);
        if (cz > 0 && lt(kp[0], kval(kp[-kPlane])))
            mark_cell(mark, c - 64);
        if (cz < 7 && lt(kp[0], kval(kp[kPlane])))
            mark_cell(mark, c + 64);
    }
#pragma unroll 1
    for (int q = lane; q < kFaces * 64; q += 32) {
        const int f = q >> 6, c = face_cell(f, q & 63, false);
        if (lt(kv[face_halo(f, q & 63)], kval(kv[mt_of(c)])))
            mark_cell(mark, c);
    }
}

// March brick b (Algorithms 10-12): sweep until every cell is the root of its
// neighbours.  kBounded: cells above bound0 / bound1 (sides -1 / +1) stay
// BAND and are not used as upwind values, and a halo cell counts only when
// its tag says KNOWN or FIX; otherwise there is no bound (every finite value
// ends KNOWN) and the tags of the halo are not read.  kTape: record the upwind
// set of every improvement for the adjoint.  kAniso: cells of unequal sides.
// a tile value without its sign bit (kSigned: FIX and padding cells carry it)
template <bool kSigned, typename real>
__device__ __forceinline__ real ld_val(const real *p)
{
    if constexpr (kSigned)
        return fabsf(*p);
    else
        return *p;
}

template <typename real, bool kHetero, bool kTape, bool kAniso, bool kBounded>
__device__ __forceinline__ void sweep_brick(const Geom &g, const DeviceState &s, const SolveParams &p,
                                            double spd_const_term, const int *order, WarpTile<real, kTape> &W,
                                            long long b, const long long nbi[kFaces], unsigned dirty, real bound0,
                                            real bound1, int lane, Notify<real> &out, MarchStats &st)
{
    real *T = (real *)s.T;
    const real *spd = (const real *)s.spd;
    real *bmin = (real *)s.bmin;
    const real INF = inf_v<real>();
    const long long base = b * kB3;
    constexpr int kVecs = kB3 * (int)sizeof(real) / 16 / 32;   // 16-byte pieces per lane
    // float, no bound: the sign bit marks FIX and padding cells instead (an
    // absolute value is free in float, and such a cell's entry is below every
    // candidate)
    constexpr bool kSigned = !kBounded && sizeof(real) == 4;

    // ---- stage the brick and the face layers of its neighbours ------------
    uint4 tg4;
    unsigned oct = 0;
    {
        const uint4 *gv = reinterpret_cast<const uint4 *>(T + base);
        uint4 x[kVecs];
#pragma unroll
        for (int j = 0; j < kVecs; ++j)
            x[j] = __ldcg(gv + lane + 32 * j);
        tg4 = __ldcg(reinterpret_cast<const uint4 *>(s.tag + base) + lane);
        uint4 tp4 = make_uint4(0, 0, 0, 0);
        if (kTape)
            tp4 = __ldcg(reinterpret_cast<const uint4 *>(s.tape + base) + lane);
        real hv[2 * kFaces];
#pragma unroll
        for (int f = 0; f < kFaces; ++f)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int q = lane + 32 * half;
                real v = INF;
                if (nbi[f] >= 0) {
                    if (kBounded && s.faces) {
                        // deterministic mode: the neighbour's layer as of the last pass
                        v = __ldcg((const real *)s.faces + nbi[f] * (kFaces * 64) + (f ^ 1) * 64 + q);
                    } else {
                        const long long ci = nbi[f] * kB3 + face_cell(f, q, true);
                        v = __ldcg(T + ci);
                        if (kBounded && !is_known(__ldcg(s.tag + ci)))
                            v = INF;
                    }
                }
                hv[2 * f + half] = v;
            }
#pragma unroll
        for (int j = 0; j < kVecs; ++j)
            row_store(W.kv, lane + 32 * j, x[j]);
        reinterpret_cast<uint4 *>(W.tg)[lane] = tg4;
        reinterpret_cast<uint4 *>(W.chg)[lane] = make_uint4(0, 0, 0, 0);
        if (kTape)
            reinterpret_cast<uint4 *>(W.tp)[lane] = tp4;
#pragma unroll
        for (int f = 0; f < kFaces; ++f)
#pragma unroll
            for (int half = 0; half < 2; ++half)
                W.kv[face_halo(f, lane + 32 * half)] = hv[2 * f + half];
        // the octant the first sweep runs in: away from the smaller halo
        // values of each axis
        unsigned hm[kFaces];
#pragma unroll
        for (int f = 0; f < kFaces; ++f)
            hm[f] = __reduce_min_sync(FULL, umin(order_word(hv[2 * f]), order_word(hv[2 * f + 1])));
        // (where one face of an axis changed, away from that one)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const unsigned lo = (dirty >> (2 * a)) & 1u, hi = (dirty >> (2 * a + 1)) & 1u;
            oct |= (lo == hi ? (unsigned)(hm[2 * a + 1] < hm[2 * a]) : hi) << a;
        }
    }
    // what the brick holds: cells that never change (FIX, padding), cells not
    // KNOWN yet, the side (a brick without FIX cells lies on one side), whether
    // it marched before (only a march makes a cell KNOWN)
    bool has_frozen, was_known, neg_side, marched = false;
    {
        unsigned fr = 0, kn = 0xffffffffu, ng = 0, mk = 0;
        const unsigned w[4] = {tg4.x, tg4.y, tg4.z, tg4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            fr |= (w[i] & (w[i] >> 1) & 0x01010101u) | (w[i] & 0x08080808u);
            kn &= w[i] >> 1;
            ng |= w[i] & 0x04040404u;
            mk |= (w[i] >> 1) & ~w[i] & 0x01010101u;
        }
        has_frozen = __any_sync(FULL, fr != 0u);
        was_known = __all_sync(FULL, (kn & 0x01010101u) == 0x01010101u);
        neg_side = __any_sync(FULL, ng != 0u);
        if (kBounded && kHetero && !kAniso && sizeof(real) == 8)
            marched = __any_sync(FULL, mk != 0u);
    }
    __syncwarp();
    if (kBounded) {
        // mark the cells no neighbour may use; a KNOWN cell among them (a solve
        // stopped with bricks marched far beyond its bound and resumed with a
        // lower one) is BAND again, so the brick is not KNOWN any more
        bool above = false;
#pragma unroll 4
        for (int k = 0; k < 16; ++k) {
            const int c = lane + 32 * k, ti = mt_of(c);
            const uint8_t t = W.tg[c];
            const real v = W.kv[ti];
            if ((t & ST_MASK) != ST_FIX && lt((t & TG_NEG) ? bound0 : bound1, v)) {
                W.kv[ti] = kmark(v);
                above = true;
            }
        }
        was_known = !__any_sync(FULL, above) && was_known;
        __syncwarp();
    }

    if (kSigned && has_frozen) {
#pragma unroll 4
        for (int k = 0; k < 16; ++k) {
            const int c = lane + 32 * k;
            const uint8_t t = W.tg[c];
            if ((t & TG_OUT) || (t & ST_MASK) == ST_FIX)
                W.kv[mt_of(c)] = kmark(W.kv[mt_of(c)]);
        }
        __syncwarp();
    }
    // ---- the march -----------------------------------------------------------
    // One cell of a step: Algorithm 11 from its neighbours in the tile.
    struct Cell {
        int ti, c;
        real lo[3], hi[3], cand, bnd;
        uint8_t set;
    };
    const auto solve_step = [&](int ti, int c, real q, Cell &x) {
        x.ti = ti;
        x.c = c;
        const real *kp = W.kv + x.ti;
        const real tc = kBounded ? kval(kp[0]) : kp[0];
        x.lo[0] = ld_val<kSigned>(kp - 1);
        x.hi[0] = ld_val<kSigned>(kp + 1);
        x.lo[1] = ld_val<kSigned>(kp - kTile);
        x.hi[1] = ld_val<kSigned>(kp + kTile);
        x.lo[2] = ld_val<kSigned>(kp - kPlane);
        x.hi[2] = ld_val<kSigned>(kp + kPlane);
        real w[3];
        unsigned code[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            w[a] = kBounded ? kmin(x.lo[a], x.hi[a]) : vmin(x.lo[a], x.hi[a]);
            if (kTape)
                code[a] = (klt(x.hi[a], x.lo[a]) ? 2u : 1u) << (2 * a);
            if (kBounded && kmarked(w[a]))
                w[a] = INF;
        }
        bool frozen = false;
        x.bnd = bound1;
        if (has_frozen && !kSigned) {
            const uint8_t t = W.tg[x.c];
            frozen = (t & TG_OUT) || (t & ST_MASK) == ST_FIX;
            if (kBounded)
                x.bnd = (t & TG_NEG) ? bound0 : bound1;
        } else if (kBounded) {
            x.bnd = neg_side ? bound0 : bound1;
        }
        x.cand = kAniso ? solve_axes_w<real, kTape>(w, code, q, (real)p.wy, (real)p.wz, x.set)
                        : solve_axes<real, kTape>(w, code, q, x.set);
        return lt(x.cand, tc) && !frozen;
    };
    const auto store_step = [&](const Cell &x) {
        const bool use = !kBounded || !lt(x.bnd, x.cand);
        W.kv[x.ti] = use ? x.cand : kmark(x.cand);
        W.chg[x.c] = 1;
        if (kTape)
            W.tp[x.c] = x.set;
        return use;
    };
    // marks[] collects, per owner lane, the cells to solve again (cell c: lane
    // c % 32, bit c / 32; so lane l owns x = l % 8, y = (l / 8) % 4 + 4 (k % 2),
    // z = k / 2 for bit k).
    bool improved = false;
    unsigned rounds = 0, nsolve = 0;
    unsigned cells = 0;   // this lane's cells to solve again
    int n = kB3;          // how many there are in the brick
    if (was_known && (dirty & 63u) != 0u && dirty != ~0u) {
        // a brick that marched before: the cells at the changed faces
        const unsigned lx = lane & 7u, ly = (lane >> 3) & 3u;
        if (((dirty & 1u) && lx == 0u) || ((dirty & 2u) && lx == 7u))
            cells = 0xffffu;
        if ((dirty & 4u) && ly == 0u)
            cells |= 0x5555u;
        if ((dirty & 8u) && ly == 3u)
            cells |= 0xaaaau;
        if (dirty & 16u)
            cells |= 0x0003u;
        if (dirty & 32u)
            cells |= 0xc000u;
        n = 0;
    }
    W.mark[lane] = 0u;
    __syncwarp();
    // Where a brick marches again after its bound rose, few cells change, and with
    // a speed field in double a sweep of 30 steps costs most: random speed, a
    // restart per level (schedule 2), 160^3 with 8 sources 36.2 ms when such bricks
    // are swept, 27.6 so, 24^3 with one 3.95 and 3.0 (the bucketed march: 29.8 and
    // 3.45).  Without a speed field or in float a front runs straight through and
    // sweeps win: 200^3 in double, phased, 18.2 ms swept, 20.0 so.  With unequal
    // cells as well a solve itself runs on the FP64 pipe, and every march starts so
    // (before the first one FIX cells have been used by Algorithm 9): 24^3, one
    // source, 4.0 ms when a first march sweeps, 3.6 so.
    if (kHetero && sizeof(real) == 8 && (kAniso || (kBounded && marched)) && !was_known) {
        reopened_cells<real>(W.kv, W.tg, W.mark, lane);
        __syncwarp();
        cells = W.mark[lane];
        W.mark[lane] = 0u;
        __syncwarp();
        n = (int)__reduce_add_sync(FULL, (unsigned)__popc(cells));
        if (n > sweep_cells<real, kHetero>())
            cells = 0u;
    }
    // Sweeps while many cells are left, a few cells one by one.
    for (;;) {
        if (n > sweep_cells<real, kHetero>()) {
            const int sx = (oct & 1u) ? -1 : 1, sy = (oct & 2u) ? -1 : 1, sz = (oct & 4u) ? -1 : 1;
            const int tstr = pack_strides(sx, sy * kTile, sz * kPlane);
            const int t0 = kMT0 + ((oct & 1u) ? 7 : 0) + ((oct & 2u) ? 7 * kTile : 0) + ((oct & 4u) ? 7 * kPlane : 0);
            const int cstr = pack_strides(sx, sy * 8, sz * 64);
            const int c0 = ((oct & 1u) ? 7 : 0) + ((oct & 2u) ? 56 : 0) + ((oct & 4u) ? 448 : 0);
            unsigned viol = 0;
            bool any = false;
            int e_next = order[lane];
            real q_next = (real)spd_const_term;
            if (kHetero && e_next >= 0)
                q_next = __ldg(spd + base + __dp4a(e_next, cstr, c0));
#pragma unroll 1
            for (int j = 1; j <= kSweepSteps; ++j) {
                const int e = e_next;
                const real q = q_next;
                // the next step's cell (and speed term) while this one is solved
                e_next = order[32 * j + lane];
                if (kHetero && e_next >= 0)
                    q_next = __ldg(spd + base + __dp4a(e_next, cstr, c0));
                Cell x;
                // (a lane without a cell in this step computes cell 0 and drops it)
                if (solve_step(e >= 0 ? __dp4a(e, tstr, t0) : kMT0, e >= 0 ? __dp4a(e, cstr, c0) : 0, q, x) && e >= 0) {
                    any = true;
                    if (store_step(x)) {
                        // a neighbour of the level before that is above it now
                        // needs another solve, unless the neighbour behind that
                        // one is at or below it (then it does not use this cell)
                        unsigned up = 0;
                        const real fx = (oct & 1u) ? x.hi[0] : x.lo[0], fy = (oct & 2u) ? x.hi[1] : x.lo[1],
                                   fz = (oct & 4u) ? x.hi[2] : x.lo[2];
                        if (lt(x.cand, kBounded ? kval(fx) : fx))
                            up |= 1u;
                        if (lt(x.cand, kBounded ? kval(fy) : fy))
                            up |= 2u;
                        if (lt(x.cand, kBounded ? kval(fz) : fz))
                            up |= 4u;
                        up &= (unsigned)e >> 24;
                        if (up) {
                            const real *kp = W.kv + x.ti;
                            if ((up & 1u) && !klt(x.cand, ld_val<kSigned>(kp - 2 * sx)))
                                up &= ~1u;
                            if ((up & 2u) && !klt(x.cand, ld_val<kSigned>(kp - 2 * sy * kTile)))
                                up &= ~2u;
                            if ((up & 4u) && !klt(x.cand, ld_val<kSigned>(kp - 2 * sz * kPlane)))
                                up &= ~4u;
                            if (up) {
                                if (up & 1u)
                                    mark_cell(W.mark, x.c - sx);
                                if (up & 2u)
                                    mark_cell(W.mark, x.c - 8 * sy);
                                if (up & 4u)
                                    mark_cell(W.mark, x.c - 64 * sz);
                                // the octant (relative to this sweep's) the front
                                // runs in here: against the sweep on these axes
                                // and on those whose smaller neighbour lies ahead
                                const real gx = (oct & 1u) ? x.lo[0] : x.hi[0], gy = (oct & 2u) ? x.lo[1] : x.hi[1],
                                           gz = (oct & 4u) ? x.lo[2] : x.hi[2];
                                if (klt(gx, fx) && klt(gx, x.cand))
                                    up |= 1u;
                                if (klt(gy, fy) && klt(gy, x.cand))
                                    up |= 2u;
                                if (klt(gz, fz) && klt(gz, x.cand))
                                    up |= 4u;
                                viol |= 1u << up;
                            }
                        }
                    }
                }
                __syncwarp();
            }
            ++rounds;
            nsolve += kB3;
            improved = __any_sync(FULL, any) || improved;
            cells = W.mark[lane];
            W.mark[lane] = 0u;
            // the next of the octants found, going round
            viol = __reduce_or_sync(FULL, viol);
            if (viol != 0u) {
                const unsigned at = rounds & 7u;
                oct ^= (unsigned)(__ffs((int)((viol | viol << 8) >> at)) - 1 + (int)at) & 7u;
            }
            __syncwarp();
        } else {
            // the cells to solve are packed 32 to a step, and a cell that improves
            // marks its neighbours above it
            const int cnt = __popc(cells);
            int pre = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(FULL, pre, o);
                if (lane >= o)
                    pre += t;
            }
            n = __shfl_sync(FULL, pre, 31);
            ++rounds;
            // (what does not fit the list stays for the next round)
            n = min(n, kListCells);
            nsolve += (unsigned)n;
            for (pre -= cnt; cells && pre < kListCells; cells &= cells - 1u)
                W.list[pre++] = (uint16_t)(lane + 32 * (__ffs((int)cells) - 1));
            __syncwarp();
            bool any = false;
#pragma unroll 1
            for (int i0 = 0; i0 < n; i0 += 32) {
                const bool valid = i0 + lane < n;
                const int c = valid ? W.list[i0 + lane] : 0;
                const real q = kHetero ? __ldg(spd + base + c) : (real)spd_const_term;
                Cell x;
                const bool imp = solve_step(mt_of(c), c, q, x) && valid;
                __syncwarp();   // every lane has read the tile
                if (imp) {
                    any = true;
                    if (store_step(x)) {
                        const int cx = c & 7, cy = (c >> 3) & 7, cz = c >> 6;
                        if (cx > 0 && lt(x.cand, kBounded ? kval(x.lo[0]) : x.lo[0]))
                            mark_cell(W.mark, c - 1);
                        if (cx < 7 && lt(x.cand, kBounded ? kval(x.hi[0]) : x.hi[0]))
                            mark_cell(W.mark, c + 1);
                        if (cy > 0 && lt(x.cand, kBounded ? kval(x.lo[1]) : x.lo[1]))
                            mark_cell(W.mark, c - 8);
                        if (cy < 7 && lt(x.cand, kBounded ? kval(x.hi[1]) : x.hi[1]))
                            mark_cell(W.mark, c + 8);
                        if (cz > 0 && lt(x.cand, kBounded ? kval(x.lo[2]) : x.lo[2]))
                            mark_cell(W.mark, c - 64);
                        if (cz < 7 && lt(x.cand, kBounded ? kval(x.hi[2]) : x.hi[2]))
                            mark_cell(W.mark, c + 64);
                    }
                }
                __syncwarp();
            }
            improved = __any_sync(FULL, any) || improved;
            cells |= W.mark[lane];
            W.mark[lane] = 0u;
            __syncwarp();
        }
        n = (int)__reduce_add_sync(FULL, (unsigned)__popc(cells));
        if (n == 0)
            break;
        if (rounds > (unsigned)p.max_rounds) {
            if (lane == 0)
                atomicOr(&s.ctrl->error, ERR_ROUNDS);
            break;
        }
    }
    st.solves += nsolve;
    // ---- overlap changes (Algorithm 13) -------------------------------------
    // A boundary cell that fell or became KNOWN is flagged to the neighbour
    // only if the adjacent halo cell is above it: otherwise that neighbour
    // cell can never take it as an upwind value (Algorithm 11 uses only
    // smaller neighbours, and values only decrease).
    out.m = 0;
    out.v[0] = out.v[1] = INF;
    out.nb = -1;
    if (improved || !was_known) {
#pragma unroll
        for (int f = 0; f < kFaces; ++f) {
            unsigned bits[2];
            real m0 = INF, m1 = INF;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int q = lane + 32 * half, c = face_cell(f, q, false);
                const real v = ld_val<kSigned>(W.kv + mt_of(c)), hv = W.kv[face_halo(f, q)];
                const uint8_t t = W.tg[c];
                const bool flag = nbi[f] >= 0 && (W.chg[c] || !is_known(t)) && !(kBounded && kmarked(v)) && lt(v, hv);
                bits[half] = __ballot_sync(FULL, flag);
                if (flag) {
                    if (t & TG_NEG)
                        m0 = vmin(m0, v);
                    else
                        m1 = vmin(m1, v);
                }
            }
            if (bits[0] | bits[1]) {
                m0 = warp_min(m0);
                m1 = warp_min(m1);
                if (lane == f) {
                    out.m = (unsigned long long)bits[0] | ((unsigned long long)bits[1] << 32);
                    out.nb = nbi[f];
                    out.v[0] = m0;
                    out.v[1] = m1;
                }
            }
        }
    }

    // ---- write back ----------------------------------------------------------
    real b0 = INF, b1 = INF;   // BAND minima of the two sides (Algorithm 16)
    unsigned nacc = 0;
    if (!was_known) {
        // new tags of cells 16 lane .. 16 lane + 15 (two rows of the tile)
        unsigned w[4] = {tg4.x, tg4.y, tg4.z, tg4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            unsigned nw = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned t = (w[i] >> (8 * u)) & 255u;
                const real v = W.kv[mt_of(16 * lane + 4 * i + u)];
                unsigned sv = t & ST_MASK;
                if (sv != ST_FIX && !(t & TG_OUT)) {
                    const real a = kBounded ? kval(v) : v;
                    sv = !lt(a, INF) ? ST_FAR : ((kBounded && kmarked(v)) ? ST_BAND : ST_KNOWN);
                    if (kBounded && sv == ST_BAND) {
                        if (t & TG_NEG)
                            b0 = vmin(b0, a);
                        else
                            b1 = vmin(b1, a);
                    }
                    nacc += sv == ST_KNOWN && ((t & ST_MASK) != ST_KNOWN || W.chg[16 * lane + 4 * i + u]);
                }
                nw |= ((t & ~(unsigned)ST_MASK) | sv) << (8 * u);
            }
            w[i] = nw;
        }
        reinterpret_cast<uint4 *>(s.tag + base)[lane] = make_uint4(w[0], w[1], w[2], w[3]);
        if (kBounded) {
            b0 = warp_min(b0);
            b1 = warp_min(b1);
        }
    } else if (improved) {
        const uint4 ch = reinterpret_cast<const uint4 *>(W.chg)[lane];
        nacc = __popc(ch.x) + __popc(ch.y) + __popc(ch.z) + __popc(ch.w);
    }
    if (improved) {
        uint4 *gv = reinterpret_cast<uint4 *>(T + base);
#pragma unroll
        for (int j = 0; j < kVecs; ++j)
            gv[lane + 32 * j] = row_load(W.kv, lane + 32 * j);
        if (kTape)
            reinterpret_cast<uint4 *>(s.tape + base)[lane] = reinterpret_cast<const uint4 *>(W.tp)[lane];
    }
    out.band[0] = b0;
    out.band[1] = b1;
    if (lane == 0) {
        bmin[2 * b] = b0;
        bmin[2 * b + 1] = b1;
    }
    st.accepted += __reduce_add_sync(FULL, nacc);
    st.marches += 1;
    st.rounds += rounds;
}

// Algorithm 9 on brick b: every non-FIX cell next to a FIX cell is solved
// once from the FIX cells around it (Jacobi) and becomes BAND; the brick's
// BAND minima are recorded.
template <typename real, bool kHetero, bool kTape, bool kAniso>
__device__ __forceinline__ void front_brick(const DeviceState &s, const SolveParams &p, double spd_const_term,
                                            WarpTile<real, kTape> &W, long long b, const long long nbi[kFaces],
                                            int lane)
{
    real *T = (real *)s.T;
    const real *spd = (const real *)s.spd;
    real *bmin = (real *)s.bmin;
    const real INF = inf_v<real>();
    const long long base = b * kB3;
    // the tile holds the values of the FIX cells and +inf everywhere else
#pragma unroll 4
    for (int k = 0; k < 16; ++k) {
        const int c = lane + 32 * k;
        const uint8_t t = s.tag[base + c];
        W.tg[c] = t;
        W.kv[mt_of(c)] = (t & ST_MASK) == ST_FIX ? T[base + c] : INF;
    }
#pragma unroll
    for (int f = 0; f < kFaces; ++f)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int q = lane + 32 * half;
            real v = INF;
            if (nbi[f] >= 0) {
                const long long ci = nbi[f] * kB3 + face_cell(f, q, true);
                if ((s.tag[ci] & ST_MASK) == ST_FIX)
                    v = T[ci];
            }
            W.kv[face_halo(f, q)] = v;
        }
    __syncwarp();
    real b0 = INF, b1 = INF;
#pragma unroll 1
    for (int k = 0; k < 16; ++k) {
        const int c = lane + 32 * k;
        const uint8_t t = W.tg[c];
        if ((t & TG_OUT) || (t & ST_MASK) == ST_FIX)
            continue;
        const real *kp = W.kv + mt_of(c);
        const real lo[3] = {kp[-1], kp[-kTile], kp[-kPlane]};
        const real hi[3] = {kp[1], kp[kTile], kp[kPlane]};
        real w[3];
        unsigned code[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            w[a] = vmin(lo[a], hi[a]);
            code[a] = (lt(hi[a], lo[a]) ? 2u : 1u) << (2 * a);
        }
        if (!lt(vmin(w[0], vmin(w[1], w[2])), INF))
            continue;
        const real q = kHetero ? spd[base + c] : (real)spd_const_term;
        uint8_t cset = 0;
        const real cand = kAniso ? solve_axes_w<real, kTape>(w, code, q, (real)p.wy, (real)p.wz, cset)
                                 : solve_axes<real, kTape>(w, code, q, cset);
        if (!lt(cand, INF))
            continue;
        T[base + c] = cand;
        s.tag[base + c] = (uint8_t)((t & ~ST_MASK) | ST_BAND);
        if (kTape)
            s.tape[base + c] = cset;
        if (t & TG_NEG)
            b0 = vmin(b0, cand);
        else
            b1 = vmin(b1, cand);
    }
    b0 = warp_min(b0);
    b1 = warp_min(b1);
    if (lane == 0) {
        bmin[2 * b] = b0;
        bmin[2 * b + 1] = b1;
    }
}

}  // namespace
}  // namespace fmmgb
