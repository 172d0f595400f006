// mg_outer.cuh -- device helpers of the FP64 outer kernels (residual, norms,
// conjugate gradients), shared by mg_kernels.cu and mg_pcg.cu.
//
// This GPU issues FP64 at 2 lanes per clock and SM, 1/64 of FP32: what the
// outer kernels do in FP64 is counted.  Kernels without neighbours walk a grid's
// cells as pairs (for_pairs: 16-byte loads, several pairs in flight); kernels
// that apply the operator march pairs up z (march_pairs), so that a z face's
// difference serves the cells below and above it.  Sums reduce in a fixed order
// (block_sum), so every sum is deterministic.
#pragma once

#include "mg_device.cuh"

namespace gbmg {

// Deterministic block sum of N doubles; result valid in thread 0.  Only the N
// sums that a kernel needs: the shuffle tree of one sum costs a block of 8 warps
// 640 cycles of the FP64 pipe, 5 us a launch for four sums at 4 blocks per SM.
template <int N>
__device__ __forceinline__ void block_sum(double (&v)[N])
{
    __shared__ double sh[N][kThreads / 32];
#pragma unroll
    for (int q = 0; q < N; q++)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < N; q++) sh[q][w] = v[q];
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int q = 0; q < N; q++) {
            double s = lane < kThreads / 32 ? sh[q][lane] : 0.0;
#pragma unroll
            for (int o = kThreads / 64; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            v[q] = s;
        }
    }
}

__device__ __forceinline__ double2 ld2(const double *p) { return *reinterpret_cast<const double2 *>(p); }

// The caller's arrays lie at any double (mg_solve asks for a 16-byte p, a served
// request need not have one): pairs of its iterate move as vectors only where
// they are aligned (the same for every pair of a grid).
__device__ __forceinline__ bool p_pairs(const OuterView &O) { return ((size_t)O.p & 15) == 0; }
__device__ __forceinline__ double2 ld_p(const OuterView &O, int c, bool pairs)
{
    return pairs ? ld2(O.p + c) : make_double2(O.p[c], O.p[c + 1]);
}
__device__ __forceinline__ void st_p(const OuterView &O, int c, bool pairs, double2 v)
{
    if (pairs) {
        *reinterpret_cast<double2 *>(O.p + c) = v;
    } else {
        O.p[c] = v.x;
        O.p[c + 1] = v.y;
    }
}

// Every cell of a grid once, two at a time: f(c, v, both) for cells c and, if
// both, c + 1 (c even), v = load(c, both).  The pairs are dealt to the threads of
// the grid's blocks in turn; a thread has the loads of kPairs of them in flight.
constexpr int kPairs = 4;
template <class L, class F>
__device__ __forceinline__ void for_pairs(const OuterView &O, int lb, L &&load, F &&f)
{
    const int cells = O.n[0] * O.n[1] * O.n[2];  // grids have fewer than 2^31 cells
    const int pairs = cells >> 1, step = O.nblk * kThreads;
    using V = decltype(load(0, true));
    int g = lb * kThreads + (int)threadIdx.x;
    for (; (long long)g + (kPairs - 1) * step < pairs; g += kPairs * step) {
        V v[kPairs];
#pragma unroll
        for (int u = 0; u < kPairs; u++) v[u] = load(2 * (g + u * step), true);
#pragma unroll
        for (int u = 0; u < kPairs; u++) f(2 * (g + u * step), v[u], true);
    }
    for (; g < pairs; g += step) f(2 * g, load(2 * g, true), true);
    if ((cells & 1) && lb == 0 && threadIdx.x == 0) f(cells - 1, load(cells - 1, false), false);
}

// s = start - A x for the pairs of cells of a grid with rows of an even number
// of cells: f(c, s0, s1, x) at cells c, c + 1 of row pairs, start(c) = the two
// starting values, x = the two cells' values.  A thread marches a pair up O.mkz
// planes; a block's threads take 256 >> O.msub consecutive pairs of a plane (rows
// after rows: no lanes idle at a row's end) and 2^O.msub pieces of the z range.
//
// Per cell 4.5 differences (the x face inside the pair and every z face serve
// both their cells) and 6 fused multiply-adds, taken before any other rounding
// (the face difference before the product keeps the residual accurate to the
// rounding of the differences when x is smooth or carries a large constant): 10.5
// FP64 operations where a cell by itself takes 13.  Every axis is walked as if
// periodic: the face across a wall is the stored 0 of the wrapped cell.
template <class S, class F>
__device__ __forceinline__ void march_pairs(const OuterView &O, const double *__restrict__ x, int lb, S &&start, F &&f)
{
    const int nx = O.n[0], ny = O.n[1], nz = O.n[2], sz = nx * ny;
    const double *__restrict__ wx = O.w[0];
    const double *__restrict__ wy = O.w[1];
    const double *__restrict__ wz = O.w[2];
    const int tile = kThreads >> O.msub, t = (int)threadIdx.x & (tile - 1);
    const int sub = (int)threadIdx.x / tile, hx = nx >> 1, pairs = hx * ny;
    for (int it = lb; it < O.mitems; it += O.nblk) {
        const int chunk = fdiv(it, O.mdt), g = (it - chunk * O.mtiles) * tile + t;
        const int k0 = ((chunk << O.msub) + sub) * O.mkz, k1 = min(k0 + O.mkz, nz);
        if (g >= pairs || k0 >= nz) continue;
        const int j = fdiv(g, O.mdx), i = 2 * (g - j * hx), row = 2 * g;
        const int cs = j > 0 ? -nx : nx * (ny - 1), cn = j + 1 < ny ? nx : -nx * (ny - 1);
        const int cw = i > 0 ? -1 : nx - 1, ce = i + 2 < nx ? 2 : 2 - nx;
        double2 xc = ld2(x + row + sz * k0), wb = ld2(wz + row + sz * k0);
        const double2 xm = ld2(x + row + sz * (k0 > 0 ? k0 - 1 : nz - 1));
        double2 db = make_double2(xc.x - xm.x, xc.y - xm.y);  // across the low z faces
        for (int k = k0; k < k1; k++) {
            const int c = row + sz * k, ct = k + 1 < nz ? c + sz : row;
            const double2 xt2 = ld2(x + ct), wt = ld2(wz + ct);
            const double2 xs = ld2(x + c + cs), xn = ld2(x + c + cn);
            const double xw = x[c + cw], xe = x[c + ce];
            const double2 fx = ld2(wx + c), fs = ld2(wy + c), fn = ld2(wy + c + cn);
            const double fe = wx[c + ce];
            const double2 s = start(c);
            const double dm = xc.y - xc.x;
            const double2 dt = make_double2(xt2.x - xc.x, xt2.y - xc.y);
            double s0 = fma(fx.x, xc.x - xw, s.x), s1 = fma(fx.y, dm, s.y);
            s0 = fma(-fx.y, dm, s0);
            s1 = fma(-fe, xe - xc.y, s1);
            s0 = fma(fs.x, xc.x - xs.x, s0);
            s1 = fma(fs.y, xc.y - xs.y, s1);
            s0 = fma(-fn.x, xn.x - xc.x, s0);
            s1 = fma(-fn.y, xn.y - xc.y, s1);
            s0 = fma(wb.x, db.x, s0);
            s1 = fma(wb.y, db.y, s1);
            s0 = fma(-wt.x, dt.x, s0);
            s1 = fma(-wt.y, dt.y, s1);
            f(c, s0, s1, xc);
            xc = xt2;
            wb = wt;
            db = dt;
        }
    }
}

// The grid's iterate lives in the three-float form: an extended-precision
// solve that took at least one refinement step.
__device__ __forceinline__ bool xp_live(const OuterView &O) { return O.xp && O.st->steps > 0; }

// Row-tile coordinates of this thread for a fine launch (2 cells per lane).
struct Tile {
    int row, j, k, xbase;
    bool ok;
};

// (dxt divides by fine_xtiles(n[0]), dy by n[1]: multiply-shift divisions; an
// integer division by a run-time divisor goes through float conversions, which
// this GPU issues to its narrow FP64 pipe)
__device__ __forceinline__ Tile fine_tile(const int n[3], int lb, const FastDiv &dxt, const FastDiv &dy)
{
    Tile t;
    const int rb = fdiv(lb, dxt), xt = lb - rb * fine_xtiles(n[0]);
    t.row = rb * kRowsPerBlock + (threadIdx.x >> 5);
    t.ok = t.row < n[1] * n[2];
    t.k = t.ok ? fdiv(t.row, dy) : 0;
    t.j = t.ok ? t.row - t.k * n[1] : 0;
    t.xbase = xt * kSeg;
    return t;
}

// Sum over the 6 faces of w_f (x_nb - x_c), FP64 (rows of an odd number of
// cells, iterates of unaligned pairs): the face difference is taken
// before the product, which keeps the residual accurate to rounding of the
// differences when x is smooth or carries a large constant.
__device__ __forceinline__ double flux64(const OuterView &O, const double *__restrict__ x, int i,
                                         int j, int k, long long c)
{
    const int nx = O.n[0], ny = O.n[1], nz = O.n[2], per = O.per;
    const double *__restrict__ wx = O.w[0];
    const double *__restrict__ wy = O.w[1];
    const double *__restrict__ wz = O.w[2];
    const long long sy = nx, sz = (long long)nx * ny;
    const double xc = x[c];
    double f = wx[c] * (x[i > 0 ? c - 1 : ((per & 1) ? c + (nx - 1) : c)] - xc);
    if (i + 1 < nx) f += wx[c + 1] * (x[c + 1] - xc);
    else if (per & 1) f += wx[c + 1 - nx] * (x[c + 1 - nx] - xc);
    f += wy[c] * (x[j > 0 ? c - sy : ((per & 2) ? c + sy * (ny - 1) : c)] - xc);
    if (j + 1 < ny) f += wy[c + sy] * (x[c + sy] - xc);
    else if (per & 2) f += wy[c - sy * (ny - 1)] * (x[c - sy * (ny - 1)] - xc);
    f += wz[c] * (x[k > 0 ? c - sz : ((per & 4) ? c + sz * (nz - 1) : c)] - xc);
    if (k + 1 < nz) f += wz[c + sz] * (x[c + sz] - xc);
    else if (per & 4) f += wz[c - sz * (nz - 1)] * (x[c - sz * (nz - 1)] - xc);
    return f;
}

// The cells of this block's row tiles, one at a time: f(c, i, j, k) (rows of an
// odd number of cells, iterates of unaligned pairs).
template <class F>
__device__ __forceinline__ void for_cells(const OuterView &O, int lb, F &&f)
{
    const int ntiles = fine_blocks(O.n);
    for (int tile = lb; tile < ntiles; tile += O.nblk) {
        const Tile t = fine_tile(O.n, tile, O.dxt, O.xy);
        if (!t.ok) continue;
        for (int h = 0; h < 2; h++) {
            const int i = t.xbase + (threadIdx.x & 31) + 32 * h;
            if (i < O.n[0]) f(O.n[0] * t.row + i, i, t.j, t.k);
        }
    }
}

}  // namespace gbmg
