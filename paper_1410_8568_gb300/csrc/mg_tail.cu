// mg_tail.cu -- the bottom of the V-cycle in one launch (Sec. 2.3 of arXiv
// 1410.8568; FP32 cycles): every level of a grid with at most kTailCells cells
// below the finest, and the coarsest solve, run in one block of kTailThreads
// threads.  These levels are too small to fill the GPU; as separate launches
// they cost a launch latency each (10 per level and cycle) for almost no work.
//
// What bounds it is latency and shared-memory bandwidth, phase by phase: a
// 16^3 .. 2^3 tail has 33 phases separated by barriers, and a half-sweep that
// reads its coefficients from shared memory moves 11 16-byte vectors per quad
// (180 KB for a 16^3 half-sweep, 1400 cycles at the 128 B/clk of one SM).  So
// the coefficients stay in registers and the iterate is split by colour:
//  - an item is a pair of cells (2m, 2m + 1) of a row: one red, one black.  A
//    thread owns the 4 items below one coarse cell on the first level (512
//    threads at 16^3) and one item of each lower level (at most 256), with the
//    faces of both cells, the inverse diagonals (one division per cell and cycle
//    instead of one per relaxation) and both values in registers;
//  - the red and the black cells of a level are two arrays indexed by item, so
//    the y and z neighbours of a cell are the same array at item +- a row or a
//    plane: 5 conflict-free 4-byte loads per relaxed cell (the sixth
//    neighbour is the item's own other cell), no selection of cells by colour;
//  - a first-level thread's items are the children of its coarse cell: it
//    restricts by itself and prolongs all 8 cells from 27 loads; on the lower
//    levels the restriction leaves one partial sum per item (the item's two
//    cells lie below one coarse cell) and the next level's threads add their four;
//  - the first level's faces come straight from global memory into the
//    registers, the lower levels' by bulk asynchronous copies that land
//    meanwhile, and the rows of a small coarsest inverse are loaded at entry.
// Measured (clock64, 16^3 .. 2^3): 63 k SM cycles with coefficients and iterate
// read from shared memory quad by quad, 31 k here (6 k loading, 8 half-sweeps of
// 16^3 at 0.8 k, each phase below 16^3 0.2 - 0.4 k of latency); a 32^3 time step
// 618 -> 479 us, a 128^3 one 2.30 -> 2.15 ms.
#include "mg_bulk.cuh"
#include "mg_kernels.h"
#include "mg_stencil.cuh"

namespace gbmg {

namespace {

constexpr int kTailItems = 4;  // items per thread on the first level: those below a coarse cell
constexpr int kTailWarps = kTailThreads / 32;
static_assert(kTailItems * kTailThreads * 2 == kTailCells, "the threads cover the largest first level");

// Place of item q in the first level's red and black arrays.  The lanes of a
// warp own items of every other row; at rows of 8 items (16^3) those of rows
// 0 and 4 would share banks, so rows 4 .. 7 of each 8 swap the halves of
// their 16-word groups (a permutation of each 64 places: the arrays hold whole ones).
__device__ __forceinline__ int place(int q) { return q ^ ((q >> 2) & 8); }
constexpr int kTailSmemMax = 128 * 1024;
static_assert(kTailCells / 8 / 2 <= kTailThreads, "one item per thread on the lower levels");

// One pair of cells: faces, inverse diagonals, right-hand sides, values, and
// the item indices of the neighbours (two 16-bit indices per word).
struct Item {
    float fo;                  // face between the two cells of the pair
    float rf, rs, rn, rb, rt;  // red cell: the other x face, y low / high, z low / high
    float bf, bs, bn, bb, bt;  // black cell: the same
    float ri, bi;              // omega / (sum of the cell's faces), 0 without faces
    float rr, br;              // right-hand sides
    float xr, xb;              // values
    unsigned side;             // items holding the red cell's (low half) and the black cell's other x neighbour
    unsigned ny, nz;           // items of the y low (low half) / high rows, of the z low / high planes
};

// Position of an item and the parity of its row (red cell = 2m + p); packed in
// one word in shared memory on the lower levels (an edge of a tail level has at most 256 cells:
// 4096 over two edges of at least 4).
struct Pos {
    int m, j, k, p;
};

__device__ __forceinline__ Pos item_pos(const TailView &V, int t, int q)
{
    Pos o;
    const int row = fdiv(q, V.dhx[t]);
    o.m = q - row * (V.n[t][0] >> 1);
    o.k = fdiv(row, V.dy[t]);
    o.j = row - o.k * V.n[t][1];
    o.p = (o.j + o.k) & 1;
    return o;
}
__device__ __forceinline__ unsigned pack_pos(const Pos &o)
{
    return (unsigned)o.m | (unsigned)o.j << 8 | (unsigned)o.k << 16 | (unsigned)o.p << 24;
}
__device__ __forceinline__ Pos unpack_pos(unsigned w)
{
    return Pos{(int)(w & 255u), (int)(w >> 8 & 255u), (int)(w >> 16 & 255u), (int)(w >> 24)};
}

// Faces of an item as loaded, before they are sorted by colour.
struct Raw {
    float2 fx, fs, fn, fb, ft;
    float fe;
};

// Faces of item q of level t from the level's faces (global memory for the
// first level, shared memory below).  Every axis is read as if periodic: the
// face across a wall is the stored 0 of the wrapped cell's low wall.
__device__ __forceinline__ Raw item_load(const TailView &V, int t, int q, const Pos &s, const float *wx,
                                         const float *wy, const float *wz)
{
    const int nx = V.n[t][0], ny = V.n[t][1], nz = V.n[t][2];
    const int c = 2 * q, sy = nx, sz = nx * ny;
    Raw r;
    r.fx = *(const float2 *)(wx + c);
    r.fe = wx[2 * s.m + 2 < nx ? c + 2 : c + 2 - nx];
    r.fs = *(const float2 *)(wy + c);
    r.fn = *(const float2 *)(wy + (s.j + 1 < ny ? c + sy : c - sy * (ny - 1)));
    r.fb = *(const float2 *)(wz + c);
    r.ft = *(const float2 *)(wz + (s.k + 1 < nz ? c + sz : c - sz * (nz - 1)));
    return r;
}

// The item's faces by colour, inverse diagonals and neighbours (wrapped: a
// wall's face is 0).  FIRST: neighbours as places of the first level's arrays.
template <bool FIRST>
__device__ __forceinline__ void item_setup(const TailView &V, int t, int q, const Pos &s, const Raw &f, float omega,
                                           Item &o)
{
    const int hx = V.n[t][0] >> 1, ny = V.n[t][1], nz = V.n[t][2], hp = hx * ny;
    // first cell: faces fx.x (low x), fx.y; second: fx.y, fe
    const float d0 = ((((f.fx.x + f.fx.y) + f.fs.x) + f.fn.x) + f.fb.x) + f.ft.x;
    const float d1 = ((((f.fx.y + f.fe) + f.fs.y) + f.fn.y) + f.fb.y) + f.ft.y;
    const float i0 = d0 >= kTinyDiag ? omega * rcp_ftz(d0) : 0.f, i1 = d1 >= kTinyDiag ? omega * rcp_ftz(d1) : 0.f;
    const bool p = s.p;
    o.fo = f.fx.y;
    o.rf = p ? f.fe : f.fx.x;
    o.bf = p ? f.fx.x : f.fe;
    o.rs = p ? f.fs.y : f.fs.x;
    o.bs = p ? f.fs.x : f.fs.y;
    o.rn = p ? f.fn.y : f.fn.x;
    o.bn = p ? f.fn.x : f.fn.y;
    o.rb = p ? f.fb.y : f.fb.x;
    o.bb = p ? f.fb.x : f.fb.y;
    o.rt = p ? f.ft.y : f.ft.x;
    o.bt = p ? f.ft.x : f.ft.y;
    o.ri = p ? i1 : i0;
    o.bi = p ? i0 : i1;
    int qw = s.m > 0 ? q - 1 : q + hx - 1, qe = s.m + 1 < hx ? q + 1 : q + 1 - hx;
    int qs = s.j > 0 ? q - hx : q + hx * (ny - 1), qn = s.j + 1 < ny ? q + hx : q - hx * (ny - 1);
    int qb = s.k > 0 ? q - hp : q + hp * (nz - 1), qt = s.k + 1 < nz ? q + hp : q - hp * (nz - 1);
    if (FIRST) {
        qw = place(qw);
        qe = place(qe);
        qs = place(qs);
        qn = place(qn);
        qb = place(qb);
        qt = place(qt);
    }
    o.side = p ? (unsigned)qe | (unsigned)qw << 16 : (unsigned)qw | (unsigned)qe << 16;
    o.ny = (unsigned)qs | (unsigned)qn << 16;
    o.nz = (unsigned)qb | (unsigned)qt << 16;
}

// A handle with subnormal faces (GridState::tiny): every face and right-hand side
// down to the coarsest level is multiplied by 2^24, which leaves the corrections as
// they are and makes every diagonal, and its inverse, a normal float.  Here the
// first level's items, after their set-up (scaled as they are loaded, the branch
// would wait for the loads: 1 us of the launch's 19).
__device__ __forceinline__ void item_scale(Item &o, float omega)
{
    o.fo *= kTinyScale;
    o.rf *= kTinyScale, o.rs *= kTinyScale, o.rn *= kTinyScale, o.rb *= kTinyScale, o.rt *= kTinyScale;
    o.bf *= kTinyScale, o.bs *= kTinyScale, o.bn *= kTinyScale, o.bb *= kTinyScale, o.bt *= kTinyScale;
    const float rd = ((((o.fo + o.rf) + o.rs) + o.rn) + o.rb) + o.rt;
    const float bd = ((((o.fo + o.bf) + o.bs) + o.bn) + o.bb) + o.bt;
    o.ri = rd > 0.f ? omega * rcp_ftz(rd) : 0.f;
    o.bi = bd > 0.f ? omega * rcp_ftz(bd) : 0.f;
}

__device__ __forceinline__ void item_rhs(int p, float b0, float b1, Item &o)
{
    o.rr = p ? b1 : b0;
    o.br = p ? b0 : b1;
}

// Sum of w (x_nb - x_c) of the red cell, its neighbours in the black array; of the black cell
__device__ __forceinline__ float red_flux(const Item &o, const float *B)
{
    float f = o.fo * (o.xb - o.xr);
    f = fmaf(o.rf, B[o.side & 0xffffu] - o.xr, f);
    f = fmaf(o.rs, B[o.ny & 0xffffu] - o.xr, f);
    f = fmaf(o.rn, B[o.ny >> 16] - o.xr, f);
    f = fmaf(o.rb, B[o.nz & 0xffffu] - o.xr, f);
    return fmaf(o.rt, B[o.nz >> 16] - o.xr, f);
}
__device__ __forceinline__ float black_flux(const Item &o, const float *R)
{
    float f = o.fo * (o.xr - o.xb);
    f = fmaf(o.bf, R[o.side >> 16] - o.xb, f);
    f = fmaf(o.bs, R[o.ny & 0xffffu] - o.xb, f);
    f = fmaf(o.bn, R[o.ny >> 16] - o.xb, f);
    f = fmaf(o.bb, R[o.nz & 0xffffu] - o.xb, f);
    return fmaf(o.bt, R[o.nz >> 16] - o.xb, f);
}

// Shared-memory arrays of a level with N cells (host: tail_floats): red and
// black values (N / 2 each; the first level's padded to whole 64s), the natural
// copy of the correction (N; the first level: the staged right-hand side);
// below the first level the right-hand side (N), the restriction's partial sums
// and the items' positions (N / 2 each), the staged faces (3 N), the items kept
// from the way down (kItemWords N / 2) and the cell coefficients (N, flux).
// The coarsest level: right-hand side (FP64), solution, cell coefficients.
constexpr int kItemWords = sizeof(Item) / 4;
struct Arr {
    float *R, *B, *nat, *rhs, *S, *w, *a;
    unsigned *pos, *items;
    double *b;
};
__host__ __device__ constexpr int half_pad(int N, int t) { return t == 0 ? ((N >> 1) + 63) & ~63 : N >> 1; }
__device__ __forceinline__ Arr level_arr(const TailView &V, int t, float *sm)
{
    const int N = V.n[t][0] * V.n[t][1] * V.n[t][2], h = N >> 1, hp = half_pad(N, t);
    Arr o;
    float *base = sm + V.off[t];
    o.R = base;
    o.B = base + hp;
    o.nat = base + 2 * hp;
    o.rhs = o.nat + N;
    o.S = o.rhs + N;
    o.pos = (unsigned *)(o.S + h);
    o.w = o.S + 2 * h;
    o.items = (unsigned *)(o.w + 3 * N);
    o.a = o.w + 3 * N + kItemWords * h;
    o.b = nullptr;
    if (t + 1 == V.nt) {
        o.b = (double *)base;
        o.nat = base + 2 * N;
        o.a = base + 3 * N;
    }
    return o;
}

// `sweeps` red-black sweeps over a thread's I items at places q[i] (on: the
// thread has items); zero: the correction is zero on entry.  Ends with the
// values in R, B and in the items.
template <int I>
__device__ __forceinline__ void sweeps_of(Item (&it)[I], const int (&q)[I], bool on, const Arr &A, int sweeps, bool zero)
{
    for (int s = 0; s < sweeps; s++) {
        if (on) {
            if (zero && s == 0) {
#pragma unroll
                for (int i = 0; i < I; i++) {
                    it[i].xb = 0.f;
                    it[i].xr = -it[i].rr * it[i].ri;
                }
            } else {
#pragma unroll
                for (int i = 0; i < I; i++) it[i].xr = fmaf(red_flux(it[i], A.B) - it[i].rr, it[i].ri, it[i].xr);
            }
#pragma unroll
            for (int i = 0; i < I; i++) A.R[q[i]] = it[i].xr;
        }
        __syncthreads();
        if (on) {
#pragma unroll
            for (int i = 0; i < I; i++) it[i].xb = fmaf(black_flux(it[i], A.R) - it[i].br, it[i].bi, it[i].xb);
#pragma unroll
            for (int i = 0; i < I; i++) A.B[q[i]] = it[i].xb;
        }
        __syncthreads();
    }
}

// (3) the residuals of an item's two cells, summed: a quarter of the coarse
// cell above (times 8)
__device__ __forceinline__ float item_residual(const Item &it, const Arr &A)
{
    return (it.rr - red_flux(it, A.B)) + (it.br - black_flux(it, A.R));
}

// right-hand side of cell (I, J, K) of level t + 1 from level t's partial sums
__device__ __forceinline__ float coarse_rhs(const TailView &V, int t, const float *S, int I, int J, int K)
{
    const int hx = V.n[t][0] >> 1, ny = V.n[t][1];
    const float *q = S + I + hx * (2 * J + ny * 2 * K);
    return (((q[0] + q[hx]) + q[hx * ny]) + q[hx * ny + hx]) * 0.125f;
}

// (4) the prolonged correction of level t + 1 at the two cells of the item at s
// (trilinear: 64 times it, see lin)
__device__ __forceinline__ float2 prolong_item(const TailView &V, int t, const Arr &C, const Pos &s)
{
    const int ncx = V.n[t + 1][0], ncy = V.n[t + 1][1], per = V.per;
    const int nc[3] = {ncx, ncy, V.n[t + 1][2]};
    if (V.flux)
        return make_float2(prolong_at_flux(C.nat, C.a, nc, per, 2 * s.m, s.j, s.k),
                           prolong_at_flux(C.nat, C.a, nc, per, 2 * s.m + 1, s.j, s.k));
    const int Im = partner(2 * s.m, ncx, per & 1), Ip = partner(2 * s.m + 1, ncx, per & 1);
    const int J[2] = {s.j >> 1, partner(s.j, ncy, per & 2)};
    const int K[2] = {s.k >> 1, partner(s.k, nc[2], per & 4)};
    float l[2][2], h[2][2];
#pragma unroll
    for (int z = 0; z < 2; z++)
#pragma unroll
        for (int y = 0; y < 2; y++) {
            const float *er = C.nat + ncx * (J[y] + ncy * K[z]);
            const float own = er[s.m];
            l[z][y] = lin(own, er[Im]);
            h[z][y] = lin(own, er[Ip]);
        }
    return make_float2(lin(lin(l[0][0], l[0][1]), lin(l[1][0], l[1][1])),
                       lin(lin(h[0][0], h[0][1]), lin(h[1][0], h[1][1])));
}

// The same for the 4 items below coarse cell (I, J, K): item i is row (2J + (i &
// 1), 2K + (i >> 1)).  27 loads for 8 cells, interpolated along x, y, z in turn
// (prolong_item's rounding order).
__device__ __forceinline__ void prolong_children(const TailView &V, int t, const Arr &C, int I, int J, int K,
                                                 float2 (&e)[4])
{
    const int ncx = V.n[t + 1][0], ncy = V.n[t + 1][1], ncz = V.n[t + 1][2], per = V.per;
    const int X[3] = {partner(2 * I, ncx, per & 1), I, partner(2 * I + 1, ncx, per & 1)};
    const int Y[3] = {partner(2 * J, ncy, per & 2), J, partner(2 * J + 1, ncy, per & 2)};
    const int Z[3] = {partner(2 * K, ncz, per & 4), K, partner(2 * K + 1, ncz, per & 4)};
    float2 y0[3], y1[3];  // fine rows 2J and 2J + 1 on the coarse planes
#pragma unroll
    for (int z = 0; z < 3; z++) {
        float2 x[3];
#pragma unroll
        for (int y = 0; y < 3; y++) {
            const float *er = C.nat + ncx * (Y[y] + ncy * Z[z]);
            const float own = er[X[1]];
            x[y] = make_float2(lin(own, er[X[0]]), lin(own, er[X[2]]));
        }
        y0[z] = make_float2(lin(x[1].x, x[0].x), lin(x[1].y, x[0].y));
        y1[z] = make_float2(lin(x[1].x, x[2].x), lin(x[1].y, x[2].y));
    }
    e[0] = make_float2(lin(y0[1].x, y0[0].x), lin(y0[1].y, y0[0].y));
    e[1] = make_float2(lin(y1[1].x, y1[0].x), lin(y1[1].y, y1[0].y));
    e[2] = make_float2(lin(y0[1].x, y0[2].x), lin(y0[1].y, y0[2].y));
    e[3] = make_float2(lin(y1[1].x, y1[2].x), lin(y1[1].y, y1[2].y));
}

// Adds the correction e of the pair's cells; flux: as it is, else 64 times it (lin).
__device__ __forceinline__ void item_add(Item &it, int p, float2 e, bool flux)
{
    const float f = flux ? 1.f : 0.015625f;
    it.xr = fmaf(f, p ? e.y : e.x, it.xr);
    it.xb = fmaf(f, p ? e.x : e.y, it.xb);
}
__device__ __forceinline__ float2 item_cells(const Item &it, int p)
{
    return p ? make_float2(it.xb, it.xr) : make_float2(it.xr, it.xb);
}

}  // namespace

__global__ void __launch_bounds__(kTailThreads, 1) k_tail(const TailView *__restrict__ tv, float omega, int nu1,
                                                          int nu2, int cyc)
{
    dep_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *sm = (float *)smem_raw;
    __shared__ __align__(16) TailView V;
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int tiny;  // see item_scale
    const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the view by one load per thread: read field by field from global memory
    // its cache lines cost a memory latency each, one after the other
    static_assert(sizeof(TailView) % 4 == 0 && sizeof(TailView) / 4 <= kTailThreads, "one word per thread");
    const TailView &G = tv[blockIdx.x];
    const bool go = in_cycle(G.st, cyc);
    if (tid < (int)(sizeof(TailView) / 4)) ((unsigned *)&V)[tid] = ((const unsigned *)&G)[tid];
    if (tid == 0) mbar_init(&bar, 1);
    if (tid == kTailThreads - 1) tiny = G.st->tiny;
    __syncthreads();
    if (!go) return;
    const int nt = V.nt;
    // stage the right-hand side of the first level and the faces of the levels
    // between it and the coarsest (solved with G) by bulk asynchronous copies,
    // issued by one thread and completed on one mbarrier; levels above the
    // coarsest have even sizes, so N % 8 == 0: sizes are multiples of 32 bytes
    // and the offsets keep 16-byte alignment
    const int N0 = V.n[0][0] * V.n[0][1] * V.n[0][2];
    const Arr A0 = level_arr(V, 0, sm);
    if (tid == kTailThreads - 1) {
        unsigned bytes = (unsigned)(N0 * sizeof(float));
        for (int t = 1; t + 1 < nt; t++) bytes += 3u * (unsigned)(V.n[t][0] * V.n[t][1] * V.n[t][2] * sizeof(float));
        mbar_arrive_expect_tx(&bar, bytes);
        bulk_g2s(A0.nat, V.b0, (unsigned)(N0 * sizeof(float)), &bar);
        for (int t = 1; t + 1 < nt; t++) {
            const int N = V.n[t][0] * V.n[t][1] * V.n[t][2];
            const Arr A = level_arr(V, t, sm);
            for (int d = 0; d < 3; d++) bulk_g2s(A.w + d * N, V.w[t][d], (unsigned)(N * sizeof(float)), &bar);
        }
    }
    // a small coarsest inverse (n <= 32): 4 columns of a row per lane, the rows
    // packed into as few warps as hold them (FP64 runs at 2 lanes a clock)
    const int n = V.n[nt - 1][0] * V.n[nt - 1][1] * V.n[nt - 1][2];
    const int lpr = n <= 4 ? 1 : n <= 8 ? 2 : n <= 16 ? 4 : 8;  // lanes per row
    const int grow = tid / lpr, gcol = 4 * (tid & (lpr - 1));
    const bool small = n <= 32;
    double g[4] = {0.0, 0.0, 0.0, 0.0};
    if (small && grow < n)
        for (int u = 0; u < 4; u++)
            if (gcol + u < n) g[u] = V.G[grow * n + gcol + u];
    if (V.flux) {
        // cell coefficients of the tail's coarse levels (a small odd-sized
        // coarsest level rules out the vector copy)
        for (int t = 1; t < nt; t++) {
            const int N = V.n[t][0] * V.n[t][1] * V.n[t][2];
            const float *src = (const float *)V.a[t];
            float *d = level_arr(V, t, sm).a;
            for (int c = tid; c < N; c += kTailThreads) d[c] = src[c];
        }
    }
    // this thread's coarse cell (I, J, K) and the 4 items below it
    const int NC = N0 >> 3, C0 = tid < NC ? tid : 0;
    const bool on0 = tid < NC;
    const int hx0 = V.n[0][0] >> 1, ny0 = V.n[0][1];
    const int crow = fdiv(C0, V.dhx[0]), I0 = C0 - crow * hx0;
    const int K0 = fdiv(crow, V.dy[1]), J0 = crow - K0 * (ny0 >> 1);
    const int qb = I0 + hx0 * (2 * J0 + ny0 * 2 * K0);
    const int q0[kTailItems] = {qb, qb + hx0, qb + hx0 * ny0, qb + hx0 * ny0 + hx0};
    int pl0[kTailItems];
    Item it0[kTailItems];
    {
        Raw f[kTailItems];
#pragma unroll
        for (int i = 0; i < kTailItems; i++)
            f[i] = item_load(V, 0, q0[i], Pos{I0, 2 * J0 + (i & 1), 2 * K0 + (i >> 1), 0}, (const float *)V.w[0][0],
                             (const float *)V.w[0][1], (const float *)V.w[0][2]);
#pragma unroll
        for (int i = 0; i < kTailItems; i++) {
            pl0[i] = place(q0[i]);
            item_setup<true>(V, 0, q0[i], Pos{I0, 2 * J0 + (i & 1), 2 * K0 + (i >> 1), (i ^ (i >> 1)) & 1}, f[i], omega,
                             it0[i]);
        }
    }
    // every thread waits (bounded); the outcome is made uniform over the block
    const int staged = __syncthreads_and(mbar_wait(&bar, 0, V.wait_polls) ? 1 : 0);
    if (!staged) {
        // give up on this grid (reported as MG_ETIMEOUT), but let the copies
        // land before the block's shared memory is released
        if (tid == 0 && V.err) *V.err = 1;
        mbar_wait(&bar, 0, kBulkWaitPolls);
        return;
    }
    if (tiny) {  // the first level's items, the staged right-hand side and faces
#pragma unroll
        for (int i = 0; i < kTailItems; i++) item_scale(it0[i], omega);
        for (int c = tid; c < N0; c += kTailThreads) A0.nat[c] *= kTinyScale;
        for (int t = 1; t + 1 < nt; t++) {
            const int N = V.n[t][0] * V.n[t][1] * V.n[t][2];
            float *w = level_arr(V, t, sm).w;
            for (int c = tid; c < 3 * N; c += kTailThreads) w[c] *= kTinyScale;
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < kTailItems; i++) {
        const float2 b = *(const float2 *)(A0.nat + 2 * q0[i]);
        item_rhs((i ^ (i >> 1)) & 1, b.x, b.y, it0[i]);
    }
    sweeps_of<kTailItems>(it0, pl0, on0, A0, nu1, true);
    if (on0) {
        float s = item_residual(it0[0], A0);
#pragma unroll
        for (int i = 1; i < kTailItems; i++) s += item_residual(it0[i], A0);
        s *= 0.125f;
        const Arr A = level_arr(V, 1, sm);
        if (nt == 2) A.b[tid] = (double)s;
        else A.rhs[tid] = s;
    }
    __syncthreads();

    // the levels between the first and the coarsest: one item per thread, its
    // faces from shared memory, kept there for the way up
    for (int t = 1; t + 1 < nt; t++) {
        const Arr A = level_arr(V, t, sm);
        const int N = V.n[t][0] * V.n[t][1] * V.n[t][2], NI = N >> 1;
        const bool on = tid < NI;
        const int q[1] = {tid};
        Item it[1];
        if (on) {
            const Pos s = item_pos(V, t, tid);
            A.pos[tid] = pack_pos(s);
            item_setup<false>(V, t, tid, s, item_load(V, t, tid, s, A.w, A.w + N, A.w + 2 * N), omega, it[0]);
            float2 b;
            if (t == 1) {
                b = *(const float2 *)(A.rhs + 2 * tid);
            } else {
                const float *S = level_arr(V, t - 1, sm).S;
                b.x = coarse_rhs(V, t - 1, S, 2 * s.m, s.j, s.k);
                b.y = coarse_rhs(V, t - 1, S, 2 * s.m + 1, s.j, s.k);
            }
            item_rhs(s.p, b.x, b.y, it[0]);
        }
        sweeps_of<1>(it, q, on, A, nu1, true);
        if (on) {
            A.S[tid] = item_residual(it[0], A);
            const unsigned *w = (const unsigned *)&it[0];
#pragma unroll
            for (int u = 0; u < kItemWords; u++) A.items[u * NI + tid] = w[u];
        }
        __syncthreads();
    }
    {
        // exact solve on the coarsest level: e = -G b, FP64
        const int t = nt - 1;
        const Arr A = level_arr(V, t, sm);
        if (nt > 2) {
            const float *S = level_arr(V, t - 1, sm).S;
            for (int c = tid; c < n; c += kTailThreads) {
                const int row = fdiv(c, V.dx[t]), K = fdiv(row, V.dy[t]);
                A.b[c] = (double)coarse_rhs(V, t - 1, S, c - row * V.n[t][0], row - K * V.n[t][1], K);
            }
            __syncthreads();
        }
        if (tiny) {
            for (int c = tid; c < n; c += kTailThreads) A.b[c] *= 1.0 / kTinyScale;
            __syncthreads();
        }
        if (small) {
            if (warp * 32 < n * lpr) {  // whole warps (rows beyond n add zeros)
                double s = 0.0;
                for (int u = 0; u < 4; u++)
                    if (gcol + u < n) s = fma(g[u], A.b[gcol + u], s);
                for (int o = lpr >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (gcol == 0 && grow < n) A.nat[grow] = (float)(-s);
            }
        } else {
            // 8 lanes per row, 4 rows per warp: 3 of n / 8 + 3 FP64 operations per
            // lane are the row's reduction (a warp per row: 5 of n / 32 + 5)
            for (int r0 = 4 * warp; r0 < n; r0 += 4 * kTailWarps) {
                const int r = r0 + (lane >> 3), l = lane & 7;
                const double *Gr = V.G + (long long)(r < n ? r : 0) * n;
                double s = 0.0;
#pragma unroll 4
                for (int u = l; u < n; u += 8) s = fma(Gr[u], A.b[u], s);
                for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (l == 0 && r < n) A.nat[r] = (float)(-s);
            }
        }
        __syncthreads();
    }
    for (int t = nt - 2; t >= 1; t--) {
        const Arr A = level_arr(V, t, sm);
        const int NI = (V.n[t][0] * V.n[t][1] * V.n[t][2]) >> 1;
        const bool on = tid < NI;
        const int q[1] = {tid};
        Item it[1];
        Pos s{0, 0, 0, 0};
        if (on) {
            unsigned *w = (unsigned *)&it[0];
#pragma unroll
            for (int u = 0; u < kItemWords; u++) w[u] = A.items[u * NI + tid];
            s = unpack_pos(A.pos[tid]);
            item_add(it[0], s.p, prolong_item(V, t, level_arr(V, t + 1, sm), s), V.flux);
            A.R[tid] = it[0].xr;
            A.B[tid] = it[0].xb;
        }
        __syncthreads();
        sweeps_of<1>(it, q, on, A, nu2, false);
        if (on) *(float2 *)(A.nat + 2 * tid) = item_cells(it[0], s.p);
        __syncthreads();
    }
    const Arr C1 = level_arr(V, 1, sm);
    if (V.flux) {
        // 7 divisions a cell: spread over the whole block, handed over in the
        // staged right-hand side's place
        for (int q = tid; q < (N0 >> 1); q += kTailThreads)
            *(float2 *)(A0.nat + 2 * q) = prolong_item(V, 0, C1, item_pos(V, 0, q));
        __syncthreads();
    }
    if (on0) {
        float2 e[4];
        if (V.flux) {
#pragma unroll
            for (int i = 0; i < kTailItems; i++) e[i] = *(const float2 *)(A0.nat + 2 * q0[i]);
        } else {
            prolong_children(V, 0, C1, I0, J0, K0, e);
        }
#pragma unroll
        for (int i = 0; i < kTailItems; i++) {
            item_add(it0[i], (i ^ (i >> 1)) & 1, e[i], V.flux);
            A0.R[pl0[i]] = it0[i].xr;
            A0.B[pl0[i]] = it0[i].xb;
        }
    }
    __syncthreads();
    sweeps_of<kTailItems>(it0, pl0, on0, A0, nu2, false);
    if (on0)
#pragma unroll
        for (int i = 0; i < kTailItems; i++)
            *(float2 *)((float *)V.x0 + 2 * q0[i]) = item_cells(it0[i], (i ^ (i >> 1)) & 1);
}

int tail_floats(int N, int t, int nt, bool flux)
{
    if (t + 1 == nt) return (flux ? 4 : 3) * N;
    return 2 * half_pad(N, t) + N + (t > 0 ? N + N + 3 * N + kItemWords * (N / 2) + (flux ? N : 0) : 0);
}

// More than 48 KB of shared memory: a 16^3 first level takes 32 KB, the levels
// below it about 45 KB more.
cudaError_t tail_opt_in()
{
    static DeviceOnce once;
    return once([] { return cudaFuncSetAttribute(k_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, kTailSmemMax); });
}

void launch_tail(const TailView *tv, int count, size_t smem, double omega, int nu1, int nu2, int cyc, cudaStream_t s)
{
    if (tail_opt_in() != cudaSuccess) return;
    launch_k(k_tail, count, kTailThreads, smem, s, tv, (float)omega, nu1, nu2, cyc);
}

}  // namespace gbmg
