// mg_kernels.cu -- CUDA kernels of the variable-density pressure multigrid.
//
// Shin, Chergui & Juric, arXiv 1410.8568, Sec. 2.3.  The kernels implement
//   (1) the cell-centred operator of Eq. 10 (divided by h^2), on every level;
//   (2) the harmonic face coefficient of Eqs. 11-12 (density -> faces);
//   (3) restriction of the residual (mean of the 8 fine children);
//   (4) prolongation of the coarse error (trilinear, 27/9/3/1 over 64);
//   (5) red-black SOR relaxation;
//   (6) the exact solve on the coarsest grid (dense inverse, FP64);
// plus the FP64 outer iteration (residual, correction update, norms of the
// stopping test and of Eq. 15) and the coarse-face coefficients (mean of the
// 4 fine faces that tile a coarse face).
//
// All cell kernels are bandwidth kernels: a warp owns a contiguous x segment
// of one grid row so every load and store is coalesced; neighbours in y and z
// come through L1/L2.  Reductions are deterministic: fixed per-thread order,
// fixed shuffle tree, per-block partials summed by one block in fixed order.
#include "mg_kernels.h"
#include "mg_stencil.cuh"
#include "mg_outer.cuh"

#include <math.h>
#include <stdlib.h>

namespace gbmg {

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------

// Neighbour offsets of cell (i,j,k) with the boundary rules of the layout:
// low face of a cell is stored at the cell; at a Neumann low wall the stored
// coefficient is 0 and the neighbour index falls back to the cell itself; at a
// Neumann high wall the face is absent (coefficient 0).
template <class T, class Load>
__device__ __forceinline__ void stencil(const T *__restrict__ wx, const T *__restrict__ wy,
                                        const T *__restrict__ wz, const Load &ld, int nx, int ny,
                                        int nz, int per, int i, int j, int k, long long c, T xc,
                                        T &diag, T &flux)
{
    const long long sy = nx;
    const long long sz = (long long)nx * ny;
    T a, d, f;
    // x low / high
    a = wx[c];
    d = a;
    f = a * (ld(i > 0 ? c - 1 : ((per & 1) ? c + (nx - 1) : c)) - xc);
    if (i + 1 < nx) {
        a = wx[c + 1];
        d += a;
        f += a * (ld(c + 1) - xc);
    } else if (per & 1) {
        a = wx[c + 1 - nx];
        d += a;
        f += a * (ld(c + 1 - nx) - xc);
    }
    // y low / high
    a = wy[c];
    d += a;
    f += a * (ld(j > 0 ? c - sy : ((per & 2) ? c + sy * (ny - 1) : c)) - xc);
    if (j + 1 < ny) {
        a = wy[c + sy];
        d += a;
        f += a * (ld(c + sy) - xc);
    } else if (per & 2) {
        a = wy[c - sy * (ny - 1)];
        d += a;
        f += a * (ld(c - sy * (ny - 1)) - xc);
    }
    // z low / high
    a = wz[c];
    d += a;
    f += a * (ld(k > 0 ? c - sz : ((per & 4) ? c + sz * (nz - 1) : c)) - xc);
    if (k + 1 < nz) {
        a = wz[c + sz];
        d += a;
        f += a * (ld(c + sz) - xc);
    } else if (per & 4) {
        a = wz[c - sz * (nz - 1)];
        d += a;
        f += a * (ld(c - sz * (nz - 1)) - xc);
    }
    diag = d;
    flux = f;
}

// Sum of the coefficients of the faces of cell c (the diagonal of -A).
template <class T>
__device__ __forceinline__ T diag_of(const T *__restrict__ wx, const T *__restrict__ wy,
                                     const T *__restrict__ wz, int nx, int ny, int nz, int per,
                                     int i, int j, int k, long long c)
{
    const long long sy = nx;
    const long long sz = (long long)nx * ny;
    T d = wx[c];
    if (i + 1 < nx) d += wx[c + 1];
    else if (per & 1) d += wx[c + 1 - nx];
    d += wy[c];
    if (j + 1 < ny) d += wy[c + sy];
    else if (per & 2) d += wy[c - sy * (ny - 1)];
    d += wz[c];
    if (k + 1 < nz) d += wz[c + sz];
    else if (per & 4) d += wz[c - sz * (nz - 1)];
    return d;
}

template <class T>
struct LoadPlain {
    const T *x;
    __device__ __forceinline__ T operator()(long long q) const { return x[q]; }
};

// ---------------------------------------------------------------------------
// (5) red-black relaxation, one colour per launch
// ---------------------------------------------------------------------------
//
// Cells of one colour only read cells of the other colour, so updating them in
// place equals the textbook half-sweep whatever the order of the threads.  When
// the row length is a multiple of 4 a thread owns an aligned quad of 4 cells of
// a row (one 16-byte vector per operand for FP32, two for FP64), relaxes the 2
// cells of the launch's colour and writes the other two back unchanged;
// otherwise (small coarse levels) one cell per thread.  The FP32 cycle uses a
// 2-ulp division (relax_quot): the inner cycle is a preconditioner and only
// steers convergence; the FP64 path divides exactly.
//
// flags: kZeroGuess  (red launch) the iterate is zero on entry: red cells get
//                    omega * (-b / d), black cells 0, so no clearing pass;
//        kOuter      (finest level, last black half-sweep of a cycle) a grid
//                    whose refinement step ends with this cycle also adds the
//                    final values of every cell (both colours) to its outer
//                    iterate.
// cyc: index of the V-cycle within its refinement step (in_cycle).
template <class T, bool OUT>
__device__ __forceinline__ void half_body(const LevelView &L, int lb, int colour, T omega, bool zero,
                                          const OuterOut &po, bool go = true)
{
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2], per = L.per;
    T *__restrict__ x = (T *)L.x;
    const T *__restrict__ b = (const T *)L.b;
    const T *__restrict__ wx = (const T *)L.w[0];
    const T *__restrict__ wy = (const T *)L.w[1];
    const T *__restrict__ wz = (const T *)L.w[2];
    const long long sy = nx, sz = (long long)nx * ny;

    if ((nx & 3) != 0) {
        // one cell per thread (row tiles of 64 cells per warp, 2 per lane)
        const Tile t = fine_tile(L.n, lb, L.dxt, L.dy);
        if (!t.ok) return;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int i = t.xbase + (threadIdx.x & 31) + 32 * h;
            if (!go) return;
            if (i >= nx || ((i + t.j + t.k) & 1) != colour) {
                if (zero && i < nx) x[(long long)nx * t.row + i] = T(0);
                // the other colour's final value (the launch leaves it as it is)
                if constexpr (OUT)
                    if (i < nx) add_outer<T>(po, (int)((long long)nx * t.row + i), x[(long long)nx * t.row + i]);
                continue;
            }
            const long long c = (long long)nx * t.row + i;
            const T *di = (sizeof(T) == 8) ? (const T *)L.dinv : nullptr;
            T v;
            if (zero) {
                if (di) {
                    v = di[c] > T(0) ? omega * ((-b[c]) * di[c]) : T(0);
                } else {
                    const T d = diag_of(wx, wy, wz, nx, ny, nz, per, i, t.j, t.k, c);
                    v = omega * relax_quot(-b[c], d);
                }
            } else {
                const T xc = x[c];
                T d, f;
                stencil(wx, wy, wz, LoadPlain<T>{x}, nx, ny, nz, per, i, t.j, t.k, c, xc, d, f);
                if (di) v = di[c] > T(0) ? xc + omega * ((f - b[c]) * di[c]) : xc;  // (rows of other than whole quads)
                else v = xc + omega * relax_quot(f - b[c], d);
            }
            x[c] = v;
            if constexpr (OUT) add_outer<T>(po, (int)c, v);
        }
        return;
    }

    // an aligned quad of 4 cells per thread: a warp covers 32 quads of one row,
    // a block 8 rows
    const int nq = nx >> 2;
    const int xt_n = (nq + 31) >> 5;
    const int rb = fdiv(lb, L.dxq), tq = lb - rb * xt_n;
    const int row = rb * kRowsPerBlock + (threadIdx.x >> 5);
    if (row >= ny * nz) return;
    const int qx = (tq << 5) + (threadIdx.x & 31);
    if (qx >= nq) return;
    const int k = fdiv(row, L.dy);
    half_quad<T, OUT>(x, b, wx, wy, wz, nx, ny, nz, per, row, row - k * ny, k, qx, colour, omega, zero, po, go,
                      (const T *)L.dinv);
}

// MAYOUT: the launch carries kOuter; the test of the step's last cycle is
// per grid, so uniform over a block, and picks one of two instances of the body.
// defer (one-grid tables, whose launches the graph limits to the grid's own
// cycles): the state's load overlaps the data's and only the stores wait for
// it; with several grids a grid that sits the cycle out returns at once.
template <class T, bool MAYOUT>
__device__ __forceinline__ void half_entry(const LevelView &L, int lb, int colour, T omega, int flags, int cyc,
                                           const OuterView *__restrict__ ov, bool defer)
{
    const bool zero = flags & kZeroGuess;
    if (!MAYOUT && defer) {
        half_body<T, false>(L, lb, colour, omega, zero, OuterOut{}, in_cycle(L.st, cyc));
        return;
    }
    if (!in_cycle(L.st, cyc)) return;
    if constexpr (MAYOUT) {
        if (last_cycle(L.st, cyc)) {
            half_body<T, true>(L, lb, colour, omega, zero, outer_out(ov[L.g]));
            return;
        }
    }
    half_body<T, false>(L, lb, colour, omega, zero, OuterOut{});
}

// single: a one-grid table, its view passed by value (`one`, parameter space):
// no dependent load of the view before the grid's state and data.
template <class T, bool MAYOUT>
__global__ void __launch_bounds__(kThreads) k_half(const LevelView *__restrict__ lv,
                                                   const int *__restrict__ start, int count,
                                                   int colour, T omega, int flags, int cyc,
                                                   const OuterView *__restrict__ ov,
                                                   const __grid_constant__ LevelView one, int single)
{
    dep_entry();
    if (single) {
        half_entry<T, MAYOUT>(one, blockIdx.x, colour, omega, flags, cyc, ov, true);
        return;
    }
    const int e = find_entry(start, count);
    half_entry<T, MAYOUT>(lv[e], blockIdx.x - start[e], colour, omega, flags, cyc, ov, false);
}

// Blocks of a half-sweep launch over a level: row tiles of 32 quads (or 64
// cells) per warp, 8 rows per block.
__host__ __device__ inline int half_blocks(const int n[3])
{
    if ((n[0] & 3) != 0) return fine_blocks(n);
    const int nq = n[0] >> 2;
    return ((nq + 31) >> 5) * ((n[1] * n[2] + kRowsPerBlock - 1) / kRowsPerBlock);
}
int half_sweep_blocks(const int n[3]) { return half_blocks(n); }
int prolong_blocks(const int n[3]) { return half_blocks(n); }

// ---------------------------------------------------------------------------
// (3) residual and restriction: coarse b = mean of (b - A x) over 8 children
// ---------------------------------------------------------------------------

// defer: see half_entry
template <class T>
__device__ __forceinline__ void restrict_entry(const LevelView &L, int lb, int cyc, T omega, bool defer)
{
    const bool go = in_cycle(L.st, cyc);
    if (!defer && !go) return;
    const int ncx = L.nc[0], ncy = L.nc[1], ncz = L.nc[2];
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    const T *x = (const T *)L.x;
    const T *b = (const T *)L.b;
    const T *wx = (const T *)L.w[0], *wy = (const T *)L.w[1], *wz = (const T *)L.w[2];
    if ((nx & 3) == 0) {
        // a thread owns the coarse pair (2P, 2P+1) of a coarse row: one fine quad
        // in each of the 2 x 2 fine rows below it
        const int np = ncx >> 1;
        const int xt_n = (np + 31) >> 5;
        const int rb = fdiv(lb, L.dxp), xt = lb - rb * xt_n;
        const int crow = rb * kRowsPerBlock + (threadIdx.x >> 5);
        if (crow >= ncy * ncz) return;
        const int P = (xt << 5) + (threadIdx.x & 31);
        if (P >= np) return;
        const int K = fdiv(crow, L.dcy);
        restrict_pair<T>(L, crow, crow - K * ncy, K, P, omega, go);
        return;
    }
    if (!go) return;
    const int xt_n = coarse_xtiles(ncx);
    const int rb = fdiv(lb, L.dxc), xt = lb - rb * xt_n;
    const int crow = rb * kRowsPerBlock + (threadIdx.x >> 5);
    if (crow >= ncy * ncz) return;
    const int I = xt * kCSeg + (threadIdx.x & 31);
    if (I >= ncx) return;
    const int K = fdiv(crow, L.dcy), J = crow - K * ncy;
    T s = T(0);
#pragma unroll
    for (int dz = 0; dz < 2; dz++)
#pragma unroll
        for (int dy = 0; dy < 2; dy++)
#pragma unroll
            for (int dx = 0; dx < 2; dx++) {
                const int i = 2 * I + dx, j = 2 * J + dy, k = 2 * K + dz;
                const long long c = i + (long long)nx * (j + (long long)ny * k);
                T d, f;
                stencil(wx, wy, wz, LoadPlain<T>{x}, nx, ny, nz, L.per, i, j, k, c, x[c], d, f);
                s += b[c] - f;
            }
    const T bcv = s * T(0.125);
    ((T *)L.bc)[I + (long long)ncx * crow] = bcv;
    if (L.zr) ((T *)L.xc)[I + (long long)ncx * crow] = zero_start_red<T>(L, I, J, K, bcv, omega);
}

template <class T>
__global__ void __launch_bounds__(kThreads) k_restrict(const LevelView *__restrict__ lv,
                                                       const int *__restrict__ start, int count, int cyc,
                                                       T omega, const __grid_constant__ LevelView one,
                                                       int single)
{
    dep_entry();
    if (single) {
        restrict_entry<T>(one, blockIdx.x, cyc, omega, true);
        return;
    }
    const int e = find_entry(start, count);
    restrict_entry<T>(lv[e], blockIdx.x - start[e], cyc, omega, false);
}

// Blocks of a restriction launch over the coarse level of `n`.
int restrict_blocks(const int n[3], const int nc[3])
{
    if ((n[0] & 3) != 0) return coarse_blocks(nc);
    const int np = nc[0] >> 1;
    return ((np + 31) >> 5) * ((nc[1] * nc[2] + kRowsPerBlock - 1) / kRowsPerBlock);
}

// ---------------------------------------------------------------------------
// (4) prolongation and correction: x += P e_c.  With no post-smoothing the
// finest level's prolongation ends the cycle, so a launch with MAYOUT adds the
// result to the FP64 iterate of the grids whose step ends with this cycle
// (row tiles only: a configuration without post-smoothing is not tuned for).
// ---------------------------------------------------------------------------

template <class T, bool FLUX, bool OUT>
__device__ __forceinline__ void prolong_body(const LevelView &L, int lb, const OuterOut &po, bool go = true)
{
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    const T *ec = (const T *)L.xc;
    T *x = (T *)L.x;
    if ((nx & 3) == 0) {
        const int nq = nx >> 2;
        const int xt_n = (nq + 31) >> 5;
        const int rb = fdiv(lb, L.dxq), xt = lb - rb * xt_n;
        const int row = rb * kRowsPerBlock + (threadIdx.x >> 5);
        if (row >= ny * nz) return;
        const int qx = (xt << 5) + (threadIdx.x & 31);
        if (qx >= nq) return;
        const int k = fdiv(row, L.dy);
        if constexpr (FLUX) {
            if (!go) return;
            prolong_quad_flux<T, OUT>(L, row, row - k * ny, k, qx, po);
        } else {
            prolong_quad<T, OUT>(L, row, row - k * ny, k, qx, po, go);
        }
        return;
    }
    if (!go) return;
    const Tile t = fine_tile(L.n, lb, L.dxt, L.dy);
    if (!t.ok) return;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int i = t.xbase + (threadIdx.x & 31) + 32 * h;
        if (i >= nx) continue;
        const long long c = (long long)nx * t.row + i;
        const T xn = FLUX ? x[c] + prolong_at_flux(ec, (const T *)L.ac, L.nc, L.per, i, t.j, t.k)
                          : add_lin(x[c], prolong_at(ec, L.nc, L.per, i, t.j, t.k));
        x[c] = xn;
        if constexpr (OUT) add_outer<T>(po, (int)c, xn);
    }
}

// defer: see half_entry
template <class T, bool FLUX, bool MAYOUT>
__device__ __forceinline__ void prolong_entry(const LevelView &L, int lb, int cyc, const OuterView *__restrict__ ov,
                                              bool defer)
{
    if (!MAYOUT && defer) {
        prolong_body<T, FLUX, false>(L, lb, OuterOut{}, in_cycle(L.st, cyc));
        return;
    }
    if (!in_cycle(L.st, cyc)) return;
    if constexpr (MAYOUT) {
        if (last_cycle(L.st, cyc)) {
            prolong_body<T, FLUX, true>(L, lb, outer_out(ov[L.g]));
            return;
        }
    }
    prolong_body<T, FLUX, false>(L, lb, OuterOut{});
}

template <class T, bool FLUX, bool MAYOUT>
__global__ void __launch_bounds__(kThreads) k_prolong(const LevelView *__restrict__ lv,
                                                      const int *__restrict__ start, int count, int cyc,
                                                      const OuterView *__restrict__ ov,
                                                      const __grid_constant__ LevelView one, int single)
{
    dep_entry();
    if (single) {
        prolong_entry<T, FLUX, MAYOUT>(one, blockIdx.x, cyc, ov, true);
        return;
    }
    const int e = find_entry(start, count);
    prolong_entry<T, FLUX, MAYOUT>(lv[e], blockIdx.x - start[e], cyc, ov, false);
}

// ---------------------------------------------------------------------------
// y = A x on one level (unit checks): x in x, y in b
// ---------------------------------------------------------------------------

template <class T>
__global__ void __launch_bounds__(kThreads) k_apply(const LevelView *__restrict__ lv,
                                                    const int *__restrict__ start, int count)
{
    dep_entry();
    const int e = find_entry(start, count);
    const LevelView L = lv[e];
    const Tile t = fine_tile(L.n, blockIdx.x - start[e], L.dxt, L.dy);
    if (!t.ok) return;
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    const T *x = (const T *)L.x;
    T *y = (T *)L.b;
    const T *wx = (const T *)L.w[0], *wy = (const T *)L.w[1], *wz = (const T *)L.w[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int i = t.xbase + (threadIdx.x & 31) + 32 * h;
        if (i >= nx) continue;
        const long long c = (long long)nx * t.row + i;
        T d, f;
        stencil(wx, wy, wz, LoadPlain<T>{x}, nx, ny, nz, L.per, i, t.j, t.k, c, x[c], d, f);
        y[c] = f;
    }
}

// ---------------------------------------------------------------------------
// coefficients: density -> faces (2), caller faces -> scaled level-0 faces,
// and coarse faces
// ---------------------------------------------------------------------------

// Conversions between FP32 and FP64 by their IEEE 754 bit fields, for positive
// values whose exponent fits the FP32 normal range (the face set-up's case):
// this GPU issues the F2F conversion instructions to its narrow FP64 pipe, the
// integer forms run on the ALU.  Exponent bias 1023 (double) vs 127 (float):
// 896 between them; double mantissa 52 bits, float 23: 29 bits dropped.
//   widen_pos:   exact float -> double (normal positive f).
//   trunc_pos:   double -> float, low 29 mantissa bits dropped (a seed).
//   narrow_rn:   double -> float, round to nearest, ties to even; values
//                outside the fast range take the hardware conversion, and set
//                *tiny (if given) when they give a subnormal.
__device__ __forceinline__ double widen_pos(float f)
{
    const unsigned b = __float_as_uint(f);
    return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}
__device__ __forceinline__ float trunc_pos(unsigned hi, unsigned lo)
{
    return __uint_as_float(((hi - (896u << 20)) << 3) | (lo >> 29));
}
__device__ __forceinline__ float narrow_rn(double d, int *tiny = nullptr)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    // positive, biased exponent 897 .. 1150: a normal float (or, rounding up
    // from the largest, the overflow to infinity that the rounding rule gives)
    if ((hi >> 20) - 897u > 253u) {
        const float f = (float)d;
        if (tiny && f > 0.f && f < kTinyDiag) *tiny = 1;
        return f;
    }
    unsigned b = __float_as_uint(trunc_pos(hi, lo));
    const unsigned rem = lo & 0x1FFFFFFFu, half = 0x10000000u;
    b += (rem > half || (rem == half && (b & 1u))) ? 1u : 0u;  // a carry steps the exponent
    return __uint_as_float(b);
}

// 1 / x by Newton-Raphson iteration in FP64 from the FP32 reciprocal of x
// truncated to FP32: y <- y + y (1 - x y), the relative error squared per step
// (Markstein, IBM J. Res. Dev. 34, 1990).  Arguments that are not positive or lie
// outside [2^-125, 2^126) divide exactly.  A call, not inlined: predicated FP64
// instructions would take the pipe in every thread.
__device__ __noinline__ double recip_nr(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    if ((hi >> 20) - 898u > 250u) return 1.0 / x;  // biased exponent 898 .. 1148
    double y = widen_pos(__frcp_rn(trunc_pos(hi, lo)));
    double e = fma(-x, y, 1.0);
    y = fma(y, e, y);
    e = fma(-x, y, 1.0);
    return fma(y, e, y);
}

// 1 / x to 0.5 ulp (and 2^-17 of one) without FP64 arithmetic, whose operations
// issue at 1/64 of the FP32 rate.  x = h + m1 + m2 in 24, 23 and 6 bits; y = 1 / h
// rounded, so 1 - h y is exact in one multiply-add, and
//   1 / x = y (1 + t),  t = e + e^2 + ...,  e = (1 - h y) - m1 y - m2 y
// with e as a float pair (eh, el), |e| < 1.5 x 2^-23, and e^3 left out (2^-67).
// y t is formed as a pair and rounded to a whole number of ulps of y's binade
// (below 2^31 of them), which is added to the bits of y.  Where the sum leaves
// the binade, and for x outside [2^-60, 2^61), recip_nr.
__device__ __forceinline__ double recip(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    if ((hi >> 20) - 963u > 120u) return recip_nr(x);
    const float h = trunc_pos(hi, lo);
    const unsigned ex = __float_as_uint(h) & 0x7f800000u, e1 = ex - (23u << 23), e2 = ex - (46u << 23);
    const float m1 = __fsub_rn(__uint_as_float(e1 | (lo >> 6 & 0x7fffffu)), __uint_as_float(e1));
    const float m2 = __fsub_rn(__uint_as_float(e2 | (lo & 0x3fu) << 17), __uint_as_float(e2));
    const float y = __frcp_rn(h);
    float err;
    const float b = __fmul_rn(m1, y);
    const float eh = two_diff(__fmaf_rn(-h, y, 1.f), b, err);
    const float el = __fmaf_rn(-m2, y, __fsub_rn(err, __fmaf_rn(m1, y, -b)));
    const float n0 = __fmul_rn(y, eh);
    const float n1 = __fmaf_rn(y, __fmaf_rn(eh, eh, el), __fmaf_rn(y, eh, -n0));
    // in units of the last place of a double in y's binade
    const unsigned yb = __float_as_uint(y);
    const float ulps = __uint_as_float((306u << 23) - (yb & 0x7f800000u));
    const float f0 = __fmul_rn(n0, ulps);
    const int i0 = __float2int_rn(f0);
    const int i = i0 + __float2int_rn(__fmaf_rn(n1, ulps, __fsub_rn(f0, (float)i0)));
    const long long v = __double_as_longlong(widen_pos(y)), w = v + i;
    if ((v ^ w) >> 52) return recip_nr(x);
    return __longlong_as_double(w);
}

// Low faces of every cell, per axis.  Bound by the FP64 pipe (2 lanes per clock
// and SM) and the FP32 instructions: 512^3 with reciprocals by recip_nr (6 FP64
// operations a face) 4.40 ms, with recip (2) 1.71 ms, 128^3 78 and 36 us; HBM would
// take 44 B a cell (0.87 ms).
template <bool HARMONIC>
__global__ void __launch_bounds__(kThreads) k_faces_from_density(const __grid_constant__ FaceArgs a)
{
    dep_entry();
    const int N = a.n[0] * a.n[1] * a.n[2];  // grids have fewer than 2^31 cells
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        const int rest = fdiv(c, a.dx);
        const int i = c - rest * a.n[0];
        const int k = fdiv(rest, a.dy);
        const int j = rest - k * a.n[1];
        const int q[3] = {i, j, k};
        const int stride[3] = {1, a.n[0], a.n[0] * a.n[1]};
        const double rho_c = a.rho[c];
        // positive and finite, by the bit field
        const bool ok = (unsigned long long)__double_as_longlong(rho_c) - 1ull < 0x7fefffffffffffffull;
        double inv_c = 0.0;
        if constexpr (!HARMONIC) inv_c = recip(rho_c);
#pragma unroll
        for (int d = 0; d < 3; d++) {
            double v;
            if (q[d] == 0 && !(a.per >> d & 1)) {
                v = 0.0;  // Neumann wall
            } else {
                const int l = q[d] > 0 ? c - stride[d] : c + stride[d] * (a.n[d] - 1);
                const double rho_l = a.rho[l];
                // Eqs. 11-12 with alpha = 1/rho: 2 a_l a_c / (a_l + a_c) = 2 / (rho_l + rho_c)
                if constexpr (HARMONIC) v = (2.0 * a.scale[d]) * recip(rho_l + rho_c);
                else v = (0.5 * a.scale[d]) * (recip(rho_l) + inv_c);
            }
            if (a.out64[d]) a.out64[d][c] = v;
            if (a.out32[d]) a.out32[d][c] = narrow_rn(v, a.tiny);
            if (a.out32lo[d]) a.out32lo[d][c] = (float)(v - (double)(float)v);
        }
        if (!ok && a.err) *a.err = 1;
    }
}

__global__ void __launch_bounds__(kThreads) k_scale_faces(FaceArgs a)
{
    dep_entry();
    const int N = a.n[0] * a.n[1] * a.n[2];  // grids have fewer than 2^31 cells
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        const int i = c % a.n[0];
        const int rest = c / a.n[0];
        const int j = rest % a.n[1];
        const int k = rest / a.n[1];
        const int q[3] = {i, j, k};
        for (int d = 0; d < 3; d++) {
            double v = 0.0;
            if (!(q[d] == 0 && !(a.per >> d & 1))) {
                const double alpha = a.in[d][c];
                if (!(alpha > 0.0 && isfinite(alpha)) && a.err) *a.err = 1;
                v = alpha * a.scale[d];
            }
            a.out64[d][c] = v;
            if (a.out32[d]) a.out32[d][c] = narrow_rn(v, a.tiny);
            if (a.out32lo[d]) a.out32lo[d][c] = (float)(v - (double)(float)v);
        }
    }
}

// coarse w_d(I,J,K) = (1/16) * sum of the 4 fine w_d that tile the coarse face:
// alpha_c = mean of the 4 fine alpha, and 1/(2h)^2 = (1/4)(1/h^2).
// Cell coefficient of the flux-conserving prolongation: mean over the cell's
// non-wall faces of alpha = w h_d^2 (1 for a cell without any).
__global__ void __launch_bounds__(kThreads) k_cell_alpha(AlphaArgs a)
{
    dep_entry();
    const int N = a.n[0] * a.n[1] * a.n[2];  // grids have fewer than 2^31 cells
    const int stride[3] = {1, a.n[0], a.n[0] * a.n[1]};
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        const int rest = c / a.n[0];
        const int q[3] = {c - rest * a.n[0], rest % a.n[1], rest / a.n[1]};
        double s = 0.0;
        int m = 0;
        for (int d = 0; d < 3; d++) {
            const bool periodic = (a.per >> d) & 1;
            if (q[d] > 0 || periodic) {
                s += a.w[d][c] * a.h2[d];
                m++;
            }
            if (q[d] + 1 < a.n[d]) {
                s += a.w[d][c + stride[d]] * a.h2[d];
                m++;
            } else if (periodic) {
                s += a.w[d][c - stride[d] * (a.n[d] - 1)] * a.h2[d];
                m++;
            }
        }
        const double v = m ? s / m : 1.0;
        if (a.out64) a.out64[c] = v;
        if (a.out32) a.out32[c] = narrow_rn(v);
    }
}

// ---------------------------------------------------------------------------
// Projection step around the solve (Chorin's projection on the MAC grid).
// u[d][c] is the normal velocity on the LOW face of cell c along d; on a
// Neumann axis the low face of the first cell is a wall (zero) and the high
// wall of the last cell carries no velocity.
// ---------------------------------------------------------------------------

// S = D u / dt: sum over axes of (high face - low face) / h_d, divided by dt
__global__ void __launch_bounds__(kThreads) k_divergence(ProjArgs a)
{
    dep_entry();
    const int N = a.n[0] * a.n[1] * a.n[2];  // grids have fewer than 2^31 cells
    const int stride[3] = {1, a.n[0], a.n[0] * a.n[1]};
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        const int rest = c / a.n[0];
        const int q[3] = {c - rest * a.n[0], rest % a.n[1], rest / a.n[1]};
        double div = 0.0;
        for (int d = 0; d < 3; d++) {
            const bool periodic = (a.per >> d) & 1;
            const double lo = (q[d] > 0 || periodic) ? a.u[d][c] : 0.0;
            const double hi = q[d] + 1 < a.n[d] ? a.u[d][c + stride[d]]
                              : periodic       ? a.u[d][c - stride[d] * (a.n[d] - 1)]
                                               : 0.0;
            div += (hi - lo) / a.h[d];
        }
        a.S[c] = div / a.dt;
    }
}

// u_f -= dt alpha_f (p_c - p_low) / h_d on every face that is not a wall;
// alpha_f / h_d = w h_d with the scaled coefficient w = alpha / h_d^2.  With
// the operator of Eq. 10, D(alpha G p) = A p, so D u = dt (S - A p).
__global__ void __launch_bounds__(kThreads) k_project(ProjArgs a)
{
    dep_entry();
    const int N = a.n[0] * a.n[1] * a.n[2];
    const int stride[3] = {1, a.n[0], a.n[0] * a.n[1]};
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        const int rest = c / a.n[0];
        const int q[3] = {c - rest * a.n[0], rest % a.n[1], rest / a.n[1]};
        const double pc = a.p[c];
        for (int d = 0; d < 3; d++) {
            const bool periodic = (a.per >> d) & 1;
            if (q[d] == 0 && !periodic) continue;  // wall face
            const int m = q[d] > 0 ? c - stride[d] : c + stride[d] * (a.n[d] - 1);
            a.u[d][c] -= a.dt * (a.w[d][c] * a.h[d]) * (pc - a.p[m]);
        }
    }
}

// 1 / (sum of the cell's 6 face coefficients), summed in relax_cell's order
// (x low, x high, y low, y high, z low, z high; a wall's face is 0), so that
// relax_cell_inv relaxes against the same diagonal; 0 for a cell without faces.
__global__ void __launch_bounds__(kThreads) k_diag_inv(DiagArgs a)
{
    dep_entry();
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2], per = a.per;
    const int N = nx * ny * nz, sy = nx, sz = nx * ny;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        const int rest = fdiv(c, a.dx);
        const int i = c - rest * nx;
        const int k = fdiv(rest, a.dy);
        const int j = rest - k * ny;
        double d = a.w[0][c];
        d += i + 1 < nx ? a.w[0][c + 1] : ((per & 1) ? a.w[0][c + 1 - nx] : 0.0);
        d += a.w[1][c];
        d += j + 1 < ny ? a.w[1][c + sy] : ((per & 2) ? a.w[1][c - sy * (ny - 1)] : 0.0);
        d += a.w[2][c];
        d += k + 1 < nz ? a.w[2][c + sz] : ((per & 4) ? a.w[2][c - sz * (nz - 1)] : 0.0);
        a.out[c] = d > 0.0 ? 1.0 / d : 0.0;
    }
}

__global__ void __launch_bounds__(kThreads) k_coarsen_faces(CoarsenArgs a)
{
    dep_entry();
    const int NC = a.nc[0] * a.nc[1] * a.nc[2];
    const int nx = a.nf[0], ny = a.nf[1];
    for (int C = blockIdx.x * blockDim.x + threadIdx.x; C < NC; C += gridDim.x * blockDim.x) {
        const int rest = fdiv(C, a.dx);
        const int I = C - rest * a.nc[0];
        const int K = fdiv(rest, a.dy);
        const int J = rest - K * a.nc[1];
        const int base[3] = {2 * I, 2 * J, 2 * K};
        for (int d = 0; d < 3; d++) {
            const int e1 = (d + 1) % 3, e2 = (d + 2) % 3;
            double s = 0.0;
            for (int u = 0; u < 2; u++)
                for (int v = 0; v < 2; v++) {
                    int f[3];
                    f[d] = base[d];
                    f[e1] = base[e1] + u;
                    f[e2] = base[e2] + v;
                    s += a.wf[d][f[0] + (long long)nx * (f[1] + (long long)ny * f[2])];
                }
            const double w = s * 0.0625;
            a.wc[d][C] = w;
            if (a.wc32[d]) a.wc32[d][C] = narrow_rn(w, a.tiny);
        }
    }
}

// ---------------------------------------------------------------------------
// FP64 outer iteration
// ---------------------------------------------------------------------------

// Start of a solve: reset the state of every grid.
__global__ void k_begin(const OuterView *__restrict__ ov)
{
    dep_entry();
    if (threadIdx.x != 0) return;
    const OuterView &O = ov[blockIdx.x];
    GridState *s = O.st;
    s->tol = O.tol;
    s->max_iters = O.max_iters;
    s->iters = 0;
    s->status = 8;  // MG_EAGAIN while running
    s->active = 1;
    s->bmean = 0.0;
    s->bnorm = 0.0;
    s->r0 = 0.0;
    s->rnorm = 0.0;
    s->xmean = 0.0;
    s->cycles_next = O.inner < O.max_iters ? O.inner : O.max_iters;
    s->steps = 0;
    s->xscale = 1.0;
    s->xinv = 1.0;
    s->rprev = 0.0;
    s->pnz = 0;
    s->tiny = *O.tiny;
}

// Partial sums of the caller's right-hand side (which = 0, partial slot 3) or
// of the iterate p (which = 1, slot 1), FP64.  (The right-hand side may be
// 8-byte aligned: read by single values.)
__global__ void __launch_bounds__(kThreads) k_sum(const OuterView *__restrict__ ov,
                                                  const int *__restrict__ start, int count, int which)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView &O = ov[e];
    const int lb = blockIdx.x - start[e];
    double v[1] = {0.0};
    auto add = [&](int, double2 x, bool) { v[0] += x.x + x.y; };
    if (which == 0) {
        for_pairs(
            O, lb, [&](int c, bool both) { return make_double2(O.b[c], both ? O.b[c + 1] : 0.0); }, add);
    } else if (xp_live(O)) {
        // end of an extended-precision solve that took a step: the iterate is the
        // three-float one (summed in its internal scale)
        auto one = [&](int c) { return ((double)O.xp3[0][c] + (double)O.xp3[1][c]) + (double)O.xp3[2][c]; };
        for_pairs(
            O, lb, [&](int c, bool both) { return make_double2(one(c), both ? one(c + 1) : 0.0); }, add);
    } else {
        const bool pairs = p_pairs(O);
        for_pairs(
            O, lb, [&](int c, bool both) { return both ? ld_p(O, c, pairs) : make_double2(O.p[c], 0.0); }, add);
    }
    block_sum(v);
    if (threadIdx.x == 0) O.part[kPart * lb + (which == 0 ? 3 : 1)] = v[0];
}

// ---- extended-precision outer iteration (mixed-precision multigrid) --------
//
// The FP64 prologue reduces the right-hand side; the refinement loop itself
// runs in FP32 arithmetic on the three-float iterate (mg_xprec.cuh); the
// epilogue converts back.  Internal quantities are scaled by xscale = 2^-k,
// k chosen from the right-hand side's rms, so that the float components stay
// far from the FP32 exponent limits whatever the scale of the problem.

// Split an FP64 value into floats: v = h + m (+ z): exact for z (the 53-bit
// significand fits 72 bits), to 2^-48 |v| for the pair.
__device__ __forceinline__ void split3(double v, float &h, float &m, float &z)
{
    h = (float)v;
    const double r = v - (double)h;
    m = (float)r;
    z = (float)(r - (double)m);
}

// b0 = b - mean(b) in FP64 and the partial sums of ||b0||^2 (slot 2).  Also
// notes whether the caller's starting iterate p has a cell that is not zero
// (GridState::pnz; a NaN counts as nonzero): a cold start (p = 0) then takes
// its starting residual as b0 itself (k_residual, mode 2).
__global__ void __launch_bounds__(kThreads) k_center_rhs(const OuterView *__restrict__ ov,
                                                    const int *__restrict__ start, int count)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView &O = ov[e];
    if (!O.st->active) return;
    const int lb = blockIdx.x - start[e];
    const double m = O.st->bmean;
    double v[1] = {0.0};
    const bool pairs = p_pairs(O);
    // a nonzero p by its bits (all but the sign; a NaN's are not zero either)
    unsigned long long nz = 0;
    struct In {
        double2 b, p;
    };
    for_pairs(
        O, lb,
        [&](int c, bool both) {
            if (both) return In{make_double2(O.b[c], O.b[c + 1]), ld_p(O, c, pairs)};
            return In{make_double2(O.b[c], 0.0), make_double2(O.p[c], 0.0)};
        },
        [&](int c, const In &x, bool both) {
            const double b0 = x.b.x - m, b1 = x.b.y - m;
            v[0] = fma(b0, b0, v[0]);
            nz |= (unsigned long long)__double_as_longlong(x.p.x) << 1;
            if (both) {
                v[0] = fma(b1, b1, v[0]);
                nz |= (unsigned long long)__double_as_longlong(x.p.y) << 1;
                *reinterpret_cast<double2 *>(O.b0 + c) = make_double2(b0, b1);
            } else {
                O.b0[c] = b0;
            }
        });
    block_sum(v);
    if (__syncthreads_or(nz != 0) && threadIdx.x == 0) atomicOr(&O.st->pnz, 1);
    if (threadIdx.x == 0) O.part[kPart * lb + 2] = v[0];
}

// Scaled right-hand side and iterate in their float forms.
__global__ void __launch_bounds__(kThreads) k_xp_prepare(const OuterView *__restrict__ ov,
                                                         const int *__restrict__ start, int count)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView O = ov[e];
    if (!O.st->active) return;
    const int lb = blockIdx.x - start[e];
    const int ntiles = fine_blocks(O.n);
    const double sc = O.st->xscale;
    for (int tile = lb; tile < ntiles; tile += O.nblk) {
        const Tile t = fine_tile(O.n, tile, O.dxt, O.xy);
        if (!t.ok) continue;
        const long long rowoff = (long long)O.n[0] * t.row;
        for (int h = 0; h < 2; h++) {
            const int i = t.xbase + (threadIdx.x & 31) + 32 * h;
            if (i >= O.n[0]) continue;
            const long long c = rowoff + i;
            float z;
            split3(O.b0[c] * sc, O.xb[0][c], O.xb[1][c], z);
            split3(O.p[c] * sc, O.xp3[0][c], O.xp3[1][c], O.xp3[2][c]);
        }
    }
}

// One face of the residual: (F0, F1) += w (p_nb - p_c), w = w0 + w1
#define XP_FACE(NB, W0, W1)                                                                    \
    do {                                                                                       \
        const int nb_ = (NB);                                                                  \
        float l_;                                                                              \
        const float h_ = triple_diff(P0[nb_], P1[nb_], P2[nb_], a0, a1, a2, l_);               \
        pair_fma_acc(F0, F1, h_, l_, (W0), (W1));                                              \
    } while (0)

// r = (b - mean b) - A p in the three-float arithmetic, scaled: the V-cycle's
// FP32 right-hand side, and the partial sums of ||r||^2 (slot 0, accumulated
// from the rounded r as in the FP64 kernel).  Every cell sums its faces in the
// order of flux64 (x low, x high, y low, y high, z low, z high).  Rows of a
// multiple of 4 cells: a thread takes an aligned quad, loads every operand as
// 16-byte vectors and treats wall faces as faces of zero weight (the stored
// low wall face is 0; its neighbour index is the cell itself), so the loads
// carry no branches; the zero terms leave the sums unchanged.  Other rows: one
// cell at a time, wall faces skipped.
__global__ void __launch_bounds__(kThreads) k_residual_xp(const OuterView *__restrict__ ov,
                                                          const int *__restrict__ start, int count,
                                                          int first)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView &O = ov[e];
    if (!O.st->active) return;
    // first: the starting residual, r = b0 where the starting iterate is zero
    const bool cold = first && !O.st->pnz;
    const int lb = blockIdx.x - start[e];
    const int nx = O.n[0], ny = O.n[1], nz = O.n[2], per = O.per, nblk = O.nblk;
    const int sy = nx, sz = nx * ny;  // grids have fewer than 2^31 cells
    const float *__restrict__ P0 = O.xp3[0];
    const float *__restrict__ P1 = O.xp3[1];
    const float *__restrict__ P2 = O.xp3[2];
    const float *__restrict__ wx = O.w32[0];
    const float *__restrict__ wy = O.w32[1];
    const float *__restrict__ wz = O.w32[2];
    const float *__restrict__ lx = O.wlo[0];
    const float *__restrict__ ly = O.wlo[1];
    const float *__restrict__ lz = O.wlo[2];
    const float *__restrict__ B0 = O.xb[0];
    const float *__restrict__ B1 = O.xb[1];
    float *__restrict__ r = (float *)O.r;
    float racc = 0.f;
    if ((nx & 3) == 0) {
        const int nq = nx >> 2, items = nq * ny * nz;
        const FastDiv dq = O.xq, dy = O.xy;
        for (int g = lb * kThreads + (int)threadIdx.x; g < items; g += nblk * kThreads) {
            const int row = fdiv(g, dq);
            const int k = fdiv(row, dy), j = row - k * ny;
            const int i0 = (g - row * nq) << 2;
            const int c = row * nx + i0;
            const bool has_e = i0 + 4 < nx || (per & 1);
            const int cw = i0 > 0 ? c - 1 : ((per & 1) ? c + nx - 1 : c);
            const int ce = i0 + 4 < nx ? c + 4 : ((per & 1) ? c + 4 - nx : c + 3);
            const bool has_n = j + 1 < ny || (per & 2), has_t = k + 1 < nz || (per & 4);
            const int ds = j > 0 ? -sy : ((per & 2) ? sy * (ny - 1) : 0);
            const int dn = j + 1 < ny ? sy : ((per & 2) ? -sy * (ny - 1) : 0);
            const int db = k > 0 ? -sz : ((per & 4) ? sz * (nz - 1) : 0);
            const int dt = k + 1 < nz ? sz : ((per & 4) ? -sz * (nz - 1) : 0);
            float F0[4] = {0.f, 0.f, 0.f, 0.f}, F1[4] = {0.f, 0.f, 0.f, 0.f};
            if (!cold) {  // A p is zero: no terms
                const float4 A0 = *(const float4 *)(P0 + c), A1 = *(const float4 *)(P1 + c),
                             A2 = *(const float4 *)(P2 + c);
                const float a0[4] = {A0.x, A0.y, A0.z, A0.w}, a1[4] = {A1.x, A1.y, A1.z, A1.w},
                            a2[4] = {A2.x, A2.y, A2.z, A2.w};
                auto term = [&](int u, float n0, float n1, float n2, float w0, float w1) {
                    float l;
                    const float h = triple_diff(n0, n1, n2, a0[u], a1[u], a2[u], l);
                    pair_fma_acc(F0[u], F1[u], h, l, w0, w1);
                };
                {
                    const float4 X0 = *(const float4 *)(wx + c), X1 = *(const float4 *)(lx + c);
                    const float x0[5] = {X0.x, X0.y, X0.z, X0.w, has_e ? wx[ce] : 0.f};
                    const float x1[5] = {X1.x, X1.y, X1.z, X1.w, has_e ? lx[ce] : 0.f};
                    const float w0v = P0[cw], w1v = P1[cw], w2v = P2[cw];
                    const float e0v = P0[ce], e1v = P1[ce], e2v = P2[ce];
    #pragma unroll
                    for (int u = 0; u < 4; u++) {
                        if (u == 0) term(0, w0v, w1v, w2v, x0[0], x1[0]);
                        else term(u, a0[u - 1], a1[u - 1], a2[u - 1], x0[u], x1[u]);
                        if (u == 3) term(3, e0v, e1v, e2v, x0[4], x1[4]);
                        else term(u, a0[u + 1], a1[u + 1], a2[u + 1], x0[u + 1], x1[u + 1]);
                    }
                }
                auto axis = [&](int dlo, int dhi, bool has_hi, const float *w, const float *wl) {
                    const float4 L0 = *(const float4 *)(P0 + c + dlo), L1 = *(const float4 *)(P1 + c + dlo),
                                 L2 = *(const float4 *)(P2 + c + dlo);
                    const float4 H0 = *(const float4 *)(P0 + c + dhi), H1 = *(const float4 *)(P1 + c + dhi),
                                 H2 = *(const float4 *)(P2 + c + dhi);
                    const float4 WL0 = *(const float4 *)(w + c), WL1 = *(const float4 *)(wl + c);
                    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 WH0 = has_hi ? *(const float4 *)(w + c + dhi) : z4;
                    const float4 WH1 = has_hi ? *(const float4 *)(wl + c + dhi) : z4;
                    const float l0[4] = {L0.x, L0.y, L0.z, L0.w}, l1[4] = {L1.x, L1.y, L1.z, L1.w},
                                l2[4] = {L2.x, L2.y, L2.z, L2.w};
                    const float h0[4] = {H0.x, H0.y, H0.z, H0.w}, h1[4] = {H1.x, H1.y, H1.z, H1.w},
                                h2[4] = {H2.x, H2.y, H2.z, H2.w};
                    const float wl0[4] = {WL0.x, WL0.y, WL0.z, WL0.w}, wl1[4] = {WL1.x, WL1.y, WL1.z, WL1.w};
                    const float wh0[4] = {WH0.x, WH0.y, WH0.z, WH0.w}, wh1[4] = {WH1.x, WH1.y, WH1.z, WH1.w};
    #pragma unroll
                    for (int u = 0; u < 4; u++) {
                        term(u, l0[u], l1[u], l2[u], wl0[u], wl1[u]);
                        term(u, h0[u], h1[u], h2[u], wh0[u], wh1[u]);
                    }
                };
                axis(ds, dn, has_n, wy, ly);
                axis(db, dt, has_t, wz, lz);
            }
            const float4 Q0 = *(const float4 *)(B0 + c), Q1 = *(const float4 *)(B1 + c);
            const float q0[4] = {Q0.x, Q0.y, Q0.z, Q0.w}, q1[4] = {Q1.x, Q1.y, Q1.z, Q1.w};
            float rq[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                float tt;
                const float hh = two_diff(q0[u], F0[u], tt);
                rq[u] = __fadd_rn(hh, __fadd_rn(tt, __fsub_rn(q1[u], F1[u])));
                racc = __fmaf_rn(rq[u], rq[u], racc);
            }
            *(float4 *)(r + c) = make_float4(rq[0], rq[1], rq[2], rq[3]);
        }
    } else {
        const int n3[3] = {nx, ny, nz};
        const int ntiles = fine_blocks(n3);
        for (int tile = lb; tile < ntiles; tile += nblk) {
            const Tile t = fine_tile(n3, tile, O.dxt, O.xy);
            if (!t.ok) continue;
            const int rowoff = nx * t.row;
            const int j = t.j, k = t.k;
            for (int h = 0; h < 2; h++) {
                const int i = t.xbase + (threadIdx.x & 31) + 32 * h;
                if (i >= nx) continue;
                const int c = rowoff + i;
                const float a0 = P0[c], a1 = P1[c], a2 = P2[c];
                float F0 = 0.f, F1 = 0.f;
                if (!cold) {
                    if (i > 0) XP_FACE(c - 1, wx[c], lx[c]);
                    else if (per & 1) XP_FACE(c + nx - 1, wx[c], lx[c]);
                    if (i + 1 < nx) XP_FACE(c + 1, wx[c + 1], lx[c + 1]);
                    else if (per & 1) XP_FACE(c + 1 - nx, wx[c + 1 - nx], lx[c + 1 - nx]);
                    if (j > 0) XP_FACE(c - sy, wy[c], ly[c]);
                    else if (per & 2) XP_FACE(c + sy * (ny - 1), wy[c], ly[c]);
                    if (j + 1 < ny) XP_FACE(c + sy, wy[c + sy], ly[c + sy]);
                    else if (per & 2) XP_FACE(c - sy * (ny - 1), wy[c - sy * (ny - 1)], ly[c - sy * (ny - 1)]);
                    if (k > 0) XP_FACE(c - sz, wz[c], lz[c]);
                    else if (per & 4) XP_FACE(c + sz * (nz - 1), wz[c], lz[c]);
                    if (k + 1 < nz) XP_FACE(c + sz, wz[c + sz], lz[c + sz]);
                    else if (per & 4) XP_FACE(c - sz * (nz - 1), wz[c - sz * (nz - 1)], lz[c - sz * (nz - 1)]);
                }
                float tt;
                const float hh = two_diff(B0[c], F0, tt);
                const float rc = __fadd_rn(hh, __fadd_rn(tt, __fsub_rn(B1[c], F1)));
                r[c] = rc;
                racc = __fmaf_rn(rc, rc, racc);
            }
        }
    }
    double v[1] = {(double)racc};
    block_sum(v);
    if (threadIdx.x == 0) O.part[kPart * lb + 0] = v[0];
}
#undef XP_FACE

// r scaled by 2^k in the cycles' precision: the exponent moved and the
// significand rounded (to nearest, ties to even) in integer arithmetic, as the
// product and the F2F conversion are FP64-pipe operations; values that are not
// normal before and after take those, in a function of its own (inlined, the
// compiler predicates them and every cell issues them).
__device__ __noinline__ double scaled_slow(double r, int k) { return r * __hiloint2double((1023 + k) << 20, 0); }
__device__ __noinline__ float scaled_slow_f(double r, int k) { return (float)(r * __hiloint2double((1023 + k) << 20, 0)); }
__device__ __forceinline__ void scaled(double r, int k, float &out)
{
    const unsigned hi = (unsigned)__double2hiint(r), lo = (unsigned)__double2loint(r), mag = hi & 0x7fffffffu;
    const int ex = (int)(mag >> 20), es = ex + k - 896;  // float exponent field
    if (ex == 0 || ex == 2047 || es < 1 || es > 253) {
        // (a zero stays one)
        out = (mag | lo) == 0u ? __uint_as_float(hi) : scaled_slow_f(r, k);
        return;
    }
    unsigned b = ((unsigned)es << 23) | ((mag & 0xfffffu) << 3) | (lo >> 29);
    const unsigned rem = lo & 0x1fffffffu, half = 0x10000000u;
    b += (rem > half || (rem == half && (b & 1u))) ? 1u : 0u;
    out = __uint_as_float(b | (hi & 0x80000000u));
}
__device__ __forceinline__ void scaled(double r, int k, double &out)
{
    const int hi = __double2hiint(r), ex = (int)(((unsigned)hi & 0x7fffffffu) >> 20);
    if (ex == 0 || ex == 2047 || ex + k < 1 || ex + k > 2046) out = scaled_slow(r, k);
    else out = __hiloint2double(hi + (k << 20), __double2loint(r));
}

// Outer residual r = (b - mean b) - A p in FP64, handed to the V-cycle in its
// precision Te, scaled by xscale (a power of 2; 1 for CG).  INIT (start of a CG
// solve): also stores b0 = b - mean(b) and the partial sums of ||b0||^2 (slot 2),
// all FP64.  first (start of a multigrid iteration): a grid whose starting
// iterate is zero everywhere (GridState::pnz clear) takes r = b0 without
// evaluating A p, which is exactly zero there.  ||r||^2 goes to slot 0; after the
// first CG residual it is accumulated from the rounded, scaled r handed to the
// cycle (a norm only steers the stopping test, so its own rounding at 1e-7
// relative is immaterial, and the scale keeps FP32 squares inside the FP32 range).
//
// Bound by the FP64 pipe: 10.5 operations a cell (march_pairs) against 15 with
// each cell's six differences, b - f, the scale and the conversion for itself.
template <class Te, bool INIT>
__global__ void __launch_bounds__(kThreads, 4) k_residual(const OuterView *__restrict__ ov,
                                                          const int *__restrict__ start, int count, int first)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView &O = ov[e];
    const GridState *s = O.st;
    if (!s->active) return;
    const int lb = blockIdx.x - start[e];
    Te *r = (Te *)O.r;
    const double m = s->bmean;
    const int ksc = ((__double2hiint(s->xscale) >> 20) & 2047) - 1023;
    const bool cold = first && !s->pnz;
    double v[INIT ? 2 : 1] = {};
    Te racc = Te(0);
    if (cold) {
        for_pairs(
            O, lb, [&](int c, bool both) { return both ? ld2(O.b0 + c) : make_double2(O.b0[c], 0.0); },
            [&](int c, double2 b, bool both) {
                Te r0, r1;
                scaled(b.x, ksc, r0);
                scaled(b.y, ksc, r1);
                r[c] = r0;
                racc += r0 * r0;
                if (both) {
                    r[c + 1] = r1;
                    racc += r1 * r1;
                }
            });
    } else if (O.mitems) {  // (0 also where p is not made of aligned pairs)
        march_pairs(
            O, O.p, lb,
            [&](int c) {
                if constexpr (!INIT) return ld2(O.b0 + c);
                const double b0 = O.b[c] - m, b1 = O.b[c + 1] - m;
                *reinterpret_cast<double2 *>(O.b0 + c) = make_double2(b0, b1);
                v[INIT ? 1 : 0] = fma(b0, b0, v[INIT ? 1 : 0]);
                v[INIT ? 1 : 0] = fma(b1, b1, v[INIT ? 1 : 0]);
                return make_double2(b0, b1);
            },
            [&](int c, double s0, double s1, double2) {
                Te r0, r1;
                scaled(s0, ksc, r0);
                scaled(s1, ksc, r1);
                r[c] = r0;
                r[c + 1] = r1;
                if (O.r64) *reinterpret_cast<double2 *>(O.r64 + c) = make_double2(s0, s1);  // CG keeps the FP64 residual
                if constexpr (INIT) {
                    v[0] = fma(s0, s0, v[0]);
                    v[0] = fma(s1, s1, v[0]);
                } else {
                    racc += r0 * r0;
                    racc += r1 * r1;
                }
            });
    } else {
        for_cells(O, lb, [&](int c, int i, int j, int k) {
            double bc;
            if constexpr (INIT) {
                bc = O.b[c] - m;
                O.b0[c] = bc;
                v[INIT ? 1 : 0] += bc * bc;
            } else {
                bc = O.b0[c];
            }
            const double rc = bc - flux64(O, O.p, i, j, k, c);
            Te rt;
            scaled(rc, ksc, rt);
            r[c] = rt;
            if (O.r64) O.r64[c] = rc;
            if constexpr (INIT) v[0] += rc * rc;
            else racc += rt * rt;
        });
    }
    if (!INIT) v[0] = (double)racc;
    block_sum(v);
    if (threadIdx.x == 0) {
        O.part[kPart * lb + 0] = v[0];
        if (INIT) O.part[kPart * lb + 2] = v[INIT ? 1 : 0];
    }
}

// One block per grid: sum the block partials in a fixed order and update the
// state.  mode 0: mean of b.  mode 1: after the starting residual.  mode 2:
// after a cycle (counts it).  mode 3: mean of the final iterate.  mode 4
// (multigrid iteration): ||b - mean b|| and the scale of the cycles.  Stopping
// test: ||r|| <= tol ||b||; NaN/Inf residual = diverged; max_iters reached =
// not converged.
__global__ void __launch_bounds__(kThreads) k_finalize(const OuterView *__restrict__ ov, int mode)
{
    dep_entry();
    const OuterView &O = ov[blockIdx.x];
    GridState *s = O.st;
    if (mode != 3 && !s->active) return;
    // the mode's sum (CG's starting residual kernel also reduced b)
    const int slot = mode == 0 ? 3 : mode == 3 ? 1 : mode == 4 ? 2 : 0;
    const bool two = mode == 1 && O.r64;
    double v[2] = {0.0, 0.0};
    for (int q = threadIdx.x; q < O.nblk; q += blockDim.x) {
        v[0] += O.part[kPart * q + slot];
        if (two) v[1] += O.part[kPart * q + 2];
    }
    if (two) {
        block_sum(v);
    } else {
        double v0[1] = {v[0]};
        block_sum(v0);
        v[0] = v0[0];
    }
    if (threadIdx.x != 0) return;
    const double N = (double)O.n[0] * O.n[1] * O.n[2];
    if (mode == 0) {
        s->bmean = v[0] / N;
        return;
    }
    if (mode == 3) {
        s->xmean = v[0] / N;
        return;
    }
    if (mode == 4) {
        // extended precision: ||b - mean b|| and the internal scale 2^-k,
        // 2^k near the rms of b - mean b (k kept inside the FP32 exponent range)
        s->bnorm = sqrt(v[0]);
        const double rms = s->bnorm / sqrt(N);
        int k = (rms > 0.0 && isfinite(rms)) ? ilogb(rms) : 0;
        k = k < -100 ? -100 : (k > 100 ? 100 : k);
        s->xscale = ldexp(1.0, -k);
        s->xinv = ldexp(1.0, k);
        return;
    }
    // the partials are of the scaled residual (xscale = 1 for CG)
    const double rn = sqrt(v[0]) * s->xinv;
    int done = 0;
    if (mode == 1) {
        if (O.r64) s->bnorm = sqrt(v[1]);
        s->r0 = rn;
    } else {
        done = s->cycles_next;
        s->iters += done;
        s->steps += 1;
    }
    s->rnorm = rn;
    if (!isfinite(rn)) stop_grid(s, 5);                                      // MG_EDIVERGED
    else if (s->bnorm == 0.0 || rn <= s->tol * s->bnorm) stop_grid(s, 0);   // converged
    else if (s->iters >= s->max_iters) stop_grid(s, 4);                      // MG_ENOTCONV
    if (s->active) {
        // V-cycles of the next refinement step: inner, or (adaptive, multigrid
        // iteration) the number the last step's per-cycle reduction rate g
        // needs to reach the tolerance, taken with a 10% margin on g
        // (FP32 logarithms: the estimate only picks a cycle count, and one
        // thread's FP64 transcendentals are a long chain on the FP64 pipe)
        int c = O.inner;
        if (mode == 2 && O.adaptive && !O.r64 && s->rprev > 0.0) {
            const float lr = logf((float)(rn / s->rprev)) / (float)done;  // log g
            if (lr < 0.0f && isfinite(lr)) {
                const float lge = fminf(logf(0.95f), logf(1.1f) + lr);      // log min(0.95, 1.1 g)
                const float need = ceilf(logf((float)(s->tol * s->bnorm / rn)) / lge);
                c = need < 1.0f ? 1 : (need < (float)O.inner ? (int)need : O.inner);
            }
        }
        const int left = s->max_iters - s->iters;  // >= 1 here
        s->cycles_next = c < left ? c : left;
    }
    s->rprev = rn;
}

// End of a solve: p = p - mean(p) (a zero right-hand side gives p = 0).  After
// an extended-precision solve p = ((p0 - mean) + p1 + p2) / xscale from the
// three-float iterate: the mean leaves the leading component first, so a
// constant carried by the iterate costs no accuracy in the FP64 result.
__global__ void __launch_bounds__(kThreads) k_final(const OuterView *__restrict__ ov,
                                                    const int *__restrict__ start, int count)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView &O = ov[e];
    const GridState *s = O.st;
    const int lb = blockIdx.x - start[e];
    const double m = s->xmean;
    const bool zero = s->bnorm == 0.0;
    const bool conv = xp_live(O), pairs = p_pairs(O);
    const double inv = conv ? 1.0 / s->xscale : 1.0;  // a power of 2: exact
    auto one = [&](int c) { return ((((double)O.xp3[0][c] - m) + (double)O.xp3[1][c]) + (double)O.xp3[2][c]) * inv; };
    for_pairs(
        O, lb,
        [&](int c, bool both) {
            if (conv) return make_double2(one(c), both ? one(c + 1) : 0.0);
            return both ? ld_p(O, c, pairs) : make_double2(O.p[c], 0.0);
        },
        [&](int c, double2 p, bool both) {
            if (!conv) p = make_double2(p.x - m, p.y - m);
            if (zero) p = make_double2(0.0, 0.0);
            if (both) st_p(O, c, pairs, p);
            else O.p[c] = p.x;
        });
}

// Loop control of a graph-driven solve: keep iterating while any grid of the
// plan is still active.  Every grid stops after at most max_iters cycles, so
// the loop is bounded.
__global__ void k_loop_ctl(cudaGraphConditionalHandle h, const OuterView *__restrict__ ov, int count)
{
    dep_entry();
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    unsigned int any = 0;
    for (int g = 0; g < count; g++) any |= (unsigned int)(ov[g].st->active != 0);
    cudaGraphSetConditional(h, any);
}

// Start of a refinement step of a graph-driven solve: the step's V-cycles are
// the most any active grid of the plan asks for (switch branch c - 1).
__global__ void k_step_ctl(cudaGraphConditionalHandle h, const OuterView *__restrict__ ov, int count)
{
    dep_entry();
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int c = 1;
    for (int g = 0; g < count; g++) {
        const GridState *s = ov[g].st;
        if (s->active && s->cycles_next > c) c = s->cycles_next;
    }
    cudaGraphSetConditional(h, (unsigned int)(c - 1));
}

// Copy the state of every grid of a plan into one contiguous array (one
// device-to-host copy then serves the whole batch).
__global__ void k_gather_states(const OuterView *__restrict__ ov, int count, GridState *out)
{
    dep_entry();
    for (int g = threadIdx.x; g < count; g += blockDim.x) out[g] = *ov[g].st;
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------

thread_local int tl_dep_launch = 0;

int dep_launch_default()
{
    static const int on = [] {
        const char *e = getenv("MG_DEP_LAUNCH");
        return (e && e[0] == '0') ? 0 : 1;
    }();
    return on;
}

void launch_gather_states(const OuterTable &ot, GridState *out, cudaStream_t s)
{
    launch_k(k_gather_states, 1, 128, 0, s, ot.ov, ot.count, out);
}

void launch_step_ctl(cudaGraphConditionalHandle h, const OuterTable &ot, cudaStream_t s)
{
    launch_k(k_step_ctl, 1, 32, 0, s, h, ot.ov, ot.count);
}
void launch_loop_ctl(cudaGraphConditionalHandle h, const OuterTable &ot, cudaStream_t s)
{
    launch_k(k_loop_ctl, 1, 32, 0, s, h, ot.ov, ot.count);
}

template <class T>
void launch_half_rows(const Table &tb, int colour, double omega, int flags, const OuterView *ov, cudaStream_t s)
{
    if (flags & kOuter)
        launch_k(k_half<T, true>, tb.blocks, kThreads, 0, s, tb.lv, tb.start, tb.count, colour, (T)omega, flags,
                 tb.cyc, ov, table_view(tb), table_single(tb));
    else
        launch_k(k_half<T, false>, tb.blocks, kThreads, 0, s, tb.lv, tb.start, tb.count, colour, (T)omega, flags,
                 tb.cyc, nullptr, table_view(tb), table_single(tb));
}
template <class T>
void launch_restrict_rows(const Table &tb, double omega, cudaStream_t s)
{
    launch_k(k_restrict<T>, tb.blocks, kThreads, 0, s, tb.lv, tb.start, tb.count, tb.cyc, (T)omega,
             table_view(tb), table_single(tb));
}
template <class T>
void launch_prolong_rows(const Table &tb, const OuterView *ov, cudaStream_t s)
{
    const int c = tb.cyc;
    const LevelView one = table_view(tb);
    const int single = table_single(tb);
    const dim3 g(tb.blocks), b(kThreads);
    if (tb.flux) {
        if (ov) launch_k(k_prolong<T, true, true>, g, b, 0, s, tb.lv, tb.start, tb.count, c, ov, one, single);
        else launch_k(k_prolong<T, true, false>, g, b, 0, s, tb.lv, tb.start, tb.count, c, nullptr, one, single);
    } else {
        if (ov) launch_k(k_prolong<T, false, true>, g, b, 0, s, tb.lv, tb.start, tb.count, c, ov, one, single);
        else launch_k(k_prolong<T, false, false>, g, b, 0, s, tb.lv, tb.start, tb.count, c, nullptr, one, single);
    }
}
template <class T>
void launch_apply(const Table &tb, cudaStream_t s)
{
    launch_k(k_apply<T>, tb.blocks, kThreads, 0, s, tb.lv, tb.start, tb.count);
}
static int cells_grid(long long N)
{
    long long b = (N + kThreads - 1) / kThreads;
    if (b > 152 * 16) b = 152 * 16;
    return (int)(b < 1 ? 1 : b);
}
void launch_faces_from_density(const FaceArgs &a, cudaStream_t s)
{
    FaceArgs b = a;
    b.dx = make_fastdiv((unsigned)a.n[0]);
    b.dy = make_fastdiv((unsigned)a.n[1]);
    const int blocks = cells_grid((long long)a.n[0] * a.n[1] * a.n[2]);
    if (a.mode == 0) launch_k(k_faces_from_density<true>, blocks, kThreads, 0, s, b);
    else launch_k(k_faces_from_density<false>, blocks, kThreads, 0, s, b);
}
void launch_scale_faces(const FaceArgs &a, cudaStream_t s)
{
    launch_k(k_scale_faces, cells_grid((long long)a.n[0] * a.n[1] * a.n[2]), kThreads, 0, s, a);
}
void launch_cell_alpha(const AlphaArgs &a, cudaStream_t s)
{
    launch_k(k_cell_alpha, cells_grid((long long)a.n[0] * a.n[1] * a.n[2]), kThreads, 0, s, a);
}
void launch_divergence(const ProjArgs &a, cudaStream_t s)
{
    launch_k(k_divergence, cells_grid((long long)a.n[0] * a.n[1] * a.n[2]), kThreads, 0, s, a);
}
void launch_project(const ProjArgs &a, cudaStream_t s)
{
    launch_k(k_project, cells_grid((long long)a.n[0] * a.n[1] * a.n[2]), kThreads, 0, s, a);
}
void launch_diag_inv(const DiagArgs &a, cudaStream_t s)
{
    launch_k(k_diag_inv, cells_grid((long long)a.n[0] * a.n[1] * a.n[2]), kThreads, 0, s, a);
}
void launch_coarsen_faces(const CoarsenArgs &a, cudaStream_t s)
{
    launch_k(k_coarsen_faces, cells_grid((long long)a.nc[0] * a.nc[1] * a.nc[2]), kThreads, 0, s, a);
}
void launch_begin(const OuterView *ov, int count, cudaStream_t s) { launch_k(k_begin, count, 32, 0, s, ov); }
void launch_sum(const OuterTable &ot, int which, cudaStream_t s)
{
    launch_k(k_sum, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count, which);
}
template <class Te>
void launch_residual(const OuterTable &ot, int init, cudaStream_t s)
{
    if (init == 1) launch_k(k_residual<Te, true>, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count, 0);
    else launch_k(k_residual<Te, false>, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count, init == 2 ? 1 : 0);
}
void launch_center_rhs(const OuterTable &ot, cudaStream_t s)
{
    launch_k(k_center_rhs, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count);
}
void launch_xp_prepare(const OuterTable &ot, cudaStream_t s)
{
    launch_k(k_xp_prepare, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count);
}
void launch_residual_xp(const OuterTable &ot, int first, cudaStream_t s)
{
    launch_k(k_residual_xp, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count, first);
}
void launch_finalize(const OuterTable &ot, int mode, cudaStream_t s)
{
    launch_k(k_finalize, ot.count, kThreads, 0, s, ot.ov, mode);
}
void launch_final(const OuterTable &ot, cudaStream_t s)
{
    launch_k(k_final, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count);
}

template void launch_half_rows<float>(const Table &, int, double, int, const OuterView *, cudaStream_t);
template void launch_half_rows<double>(const Table &, int, double, int, const OuterView *, cudaStream_t);
template void launch_restrict_rows<float>(const Table &, double, cudaStream_t);
template void launch_restrict_rows<double>(const Table &, double, cudaStream_t);
template void launch_prolong_rows<float>(const Table &, const OuterView *, cudaStream_t);
template void launch_prolong_rows<double>(const Table &, const OuterView *, cudaStream_t);
template void launch_apply<float>(const Table &, cudaStream_t);
template void launch_apply<double>(const Table &, cudaStream_t);
template void launch_residual<float>(const OuterTable &, int, cudaStream_t);
template void launch_residual<double>(const OuterTable &, int, cudaStream_t);

}  // namespace gbmg
