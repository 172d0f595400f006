// mg_march.cu -- one-pass red-black sweep of FP32 cycles (Sec. 2.3 item 5 of
// arXiv 1410.8568, red-black SOR) for rows of whole quads: both colours of a
// full sweep in one launch, marching up z, with the operands in registers.
//
// A sweep reads one iterate buffer and writes the other, so every value the
// red cells need is the old iterate, which no block overwrites.  A block owns
// a tile of up to 128 cells along x and R rows along y and marches up a chunk
// of planes; a thread owns one aligned quad of 4 cells of every plane.  Step k
// relaxes the red cells of plane k (own rows and one halo row on each side)
// and the black cells of plane k - 1 (own rows) and stores plane k - 1.
//
// The half-sweep pair streams every operand once per colour (46 B a cell); a
// sweep needs 24.  An earlier one-pass kernel staged whole tiles in shared
// memory and was bound by instruction issue (145 a cell, 40 % of them copies
// into shared memory, most others selections of a quad's cells by colour).
// Here
//  - a thread copies exactly its own quad of each operand into shared memory
//    (five 16-byte cp.async a plane, three planes ahead) and reads it back when
//    the march gets there: no mapping of copies to threads, no registers held
//    by loads in flight, 80 to 120 KB in flight per SM;
//  - a quad's z neighbours, faces and right-hand side stay in the thread's
//    registers from plane to plane; its x neighbours come by warp shuffle, its
//    y neighbours from the neighbouring thread's copies (old values) or from a
//    ring of the new red cells (8 bytes per thread and plane);
//  - the rows of a warp have the same parity of j, so the colour's place in
//    the quad is uniform over the warp: two instances of the step, no selects;
//  - every axis is walked as if periodic (see march_body): no tests for walls;
//  - what lies beyond the tile is copied beside it: the rows beyond the halo
//    rows by the halo rows' warps, the x neighbours and faces beyond a row's
//    ends (4 bytes per row and plane) by warp 0.
// One block barrier per step.  Measured at 512^3: 509 us, 6.3 TB/s of the 24 B a
// cell, 0.93 of the copy rate (the earlier one-pass kernel 790 us, the half-sweep
// pair 925); 235 warp instructions per quad and step.
//
// The red cells just west and east of a tile that the black cells of its edge
// need (one per row and plane: the west one where j + k is odd, else the east
// one) are relaxed by warp 0, whose own row is a halo row without a black
// phase (a 17th warp would cut the registers of every thread from 128 to 96).  Halo rows, halo cells and the planes
// below and above a chunk are computed by every block that needs them, so
// blocks never wait on one another; the block's only waits are its barriers.
//
// Every cell's new value comes from relax_cell with the same operands as in
// the red and black half-sweep launches, so the result is bitwise theirs.
#include <type_traits>

#include "mg_bulk.cuh"  // smem_u32
#include "mg_kernels.h"
#include "mg_stencil.cuh"

namespace gbmg {

namespace {

// i modulo n for i at most a few n out of range
__device__ __forceinline__ int wrapped(int i, int n)
{
    while (i < 0) i += n;
    while (i >= n) i -= n;
    return i;
}

__device__ __forceinline__ float4 ldg4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// What the black relaxation of a plane needs from the red one of the same quad.
struct Kept {
    float4 fx;
    float fe;
    float2 x, r;           // old black values, new red values
    float2 b, fs, fn, fb;  // right-hand side, y faces, low z faces at the black cells
};

// cells PAR and PAR + 2 of a quad
template <int PAR>
__device__ __forceinline__ float2 pick(const float4 &q)
{
    return PAR ? make_float2(q.y, q.w) : make_float2(q.x, q.z);
}

// Relaxation of the cells PAR, PAR + 2 of a quad: c their values, o the two
// other cells' values (offsets 1 - PAR, 3 - PAR), e the x neighbour outside
// the quad (west of cell 0 if PAR = 0, east of cell 3 if PAR = 1); omega, tiny: see relax_cell.
template <int PAR>
__device__ __forceinline__ float2 relax2(float2 c, float2 o, float e, const float4 &fx, float fe, float2 fs, float2 fn,
                                         float2 fb, float2 ft, float2 xs, float2 xn, float2 xb, float2 xt, float2 b,
                                         float omega, float tiny)
{
    float2 v;
    if (PAR == 0) {
        v.x = relax_cell(c.x, e, o.x, fx.x, fx.y, fs.x, fn.x, fb.x, ft.x, xs.x, xn.x, xb.x, xt.x, b.x, omega, tiny);
        v.y = relax_cell(c.y, o.x, o.y, fx.z, fx.w, fs.y, fn.y, fb.y, ft.y, xs.y, xn.y, xb.y, xt.y, b.y, omega, tiny);
    } else {
        v.x = relax_cell(c.x, o.x, o.y, fx.y, fx.z, fs.x, fn.x, fb.x, ft.x, xs.x, xn.x, xb.x, xt.x, b.x, omega, tiny);
        v.y = relax_cell(c.y, o.y, e, fx.w, fe, fs.y, fn.y, fb.y, ft.y, xs.y, xn.y, xb.y, xt.y, b.y, omega, tiny);
    }
    return v;
}

constexpr int W = 16;  // warps of a block: 512 threads of 128 registers, one block per SM

// Quads of a tile along x: the whole row if it fits a warp, else the row cut
// into equal tiles of at most 32 quads (the last one may be shorter).
int tile_quads(int nx)
{
    const int nq = nx >> 2, tiles = (nq + 31) / 32;
    return (nq + tiles - 1) / tiles;
}

// Shared memory of a block: the quads of the operands at four planes (x with a
// row beyond each halo row, fy with one above), the x neighbour beyond each
// row's end and the x face at its east end, and the red cells (halo cells) of
// two planes.
constexpr int kSlots = 4;
struct March {
    float4 x[kSlots][(W + 2) * 32], fx[kSlots][W * 32], fy[kSlots][(W + 1) * 32], b[kSlots][W * 32], fz[kSlots][W * 32];
    float2 red[2][W * 32];
    float xe[kSlots][W], fe[kSlots][W];
    float cell[kSlots][14][W];  // operands of the halo cells beside the own rows (relax_cell's order)
    float halo[2][W];
};

__device__ __forceinline__ void copy4(unsigned dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy16(unsigned dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// The march of one block of W warps (slot rows: W * P, P rows per warp).
//
// Every axis is walked as if it were periodic: the face across a wall is the
// low-wall entry of the wrapped cell, which the layout stores as 0, so the
// wrapped neighbour has no weight and no load, shuffle or relaxation needs a
// test for walls.  Lanes and rows beyond the tile repeat the work of a lane of
// the same parity (same values to the same places); only the stores of own
// cells are guarded.
template <bool ZERO>
__device__ __forceinline__ void march_body(const LevelView &L, int lb, int dir, float omega, float tiny, March &sh)
{
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    const float *__restrict__ xin = (const float *)(dir ? L.x2 : L.x);
    float *__restrict__ xout = (float *)(dir ? L.x : L.x2);
    const float *__restrict__ wx = (const float *)L.w[0];
    const float *__restrict__ wy = (const float *)L.w[1];
    const float *__restrict__ wz = (const float *)L.w[2];
    const float *__restrict__ bb = (const float *)L.b;
    const int t = (int)threadIdx.x, warp = t >> 5, lane = t & 31;
    // the block's tile: fS tiles per chunk (strips x x-tiles, dfq divides by the x-tiles)
    const int chunk = fdiv(lb, L.dfS), tile = lb - chunk * L.fS;
    const int nq = nx >> 2, tq = L.fT, xtiles = (nq + tq - 1) / tq;
    const int strip = fdiv(tile, L.dfq), xt_ = tile - strip * xtiles;
    const int q0 = xt_ * tq, nqt = min(tq, nq - q0);  // first quad and quads of the tile
    const int y0 = strip * L.fR, nown = min(L.fR, ny - y0);
    const int k0 = chunk * L.fKc, k1 = min(k0 + L.fKc, nz);
    const int P = 32 / tq;
    const bool tiled = xtiles > 1;
    const int sz = nx * ny;

    // slot row r of the block: row y0 - 1 + r; the rows of a warp are of one parity
    const int sub_ = lane / tq, sub = sub_ < P ? sub_ : 0, q_ = lane - sub_ * tq, q = min(q_, nqt - 1);
    int r = (warp & 1) + 2 * ((warp >> 1) * P + sub);
    const bool own = sub_ < P && q_ < nqt && r >= 1 && r <= nown;
    if (r > nown + 1) r = nown + 1 - ((r - nown - 1) & 1);  // beyond the strip: a row of the same parity
    const int jj = (y0 - 1 + (warp & 1)) & 1;               // parity of the warp's rows
    const int j = wrapped(y0 - 1 + r, ny);
    const int row = 4 * (q0 + q) + nx * j;  // the quad in plane 0
    const int rown = j + 1 < ny ? row + nx : row - nx * (ny - 1);
    // x: lanes of the neighbouring quads; a tiled row's ends
    const bool first = q == 0, last = q == nqt - 1;
    const int base = sub * tq;
    const int lw = first ? (tiled ? lane : base + nqt - 1) : base + q - 1;
    const int le = last ? (tiled ? lane : base) : base + q + 1;
    const bool ld_w = tiled && first, ld_e = tiled && last;
    const int me = r * tq + q;  // this quad in the shared rows (x: one row further)
    // a halo row's warp also copies the row beyond it (r = 0: below; above with its y faces)
    const bool lower = r == 0, upper = r == nown + 1;
    const int rowe = lower ? (j > 0 ? row - nx : row + nx * (ny - 1)) : rown;

    // the cells beyond the row's ends
    const bool halo_warp = tiled && warp == 0;
    const int i_w = wrapped(4 * q0 - 1, nx), i_e = wrapped(4 * (q0 + nqt), nx);
    // copies of the operands of the red one of them beside own row y0 + lane at
    // plane k (kk in the grid), by warp 0 of a tiled row
    auto copy_cell = [&](int k, int kk, unsigned s) {
        const int hj = y0 + lane;
        const int i = ((hj + k) & 1) ? i_w : i_e;
        const int c = i + nx * hj + sz * kk;
        const int cw = i > 0 ? c - 1 : c + nx - 1, ce = i + 1 < nx ? c + 1 : c + 1 - nx;
        const int cs = hj > 0 ? c - nx : c + nx * (ny - 1), cn = hj + 1 < ny ? c + nx : c - nx * (ny - 1);
        const int cd = kk > 0 ? c - sz : c + sz * (nz - 1), cu = kk + 1 < nz ? c + sz : c - sz * (nz - 1);
        const unsigned d = smem_u32(&sh.cell[s][0][lane]);
        constexpr unsigned w = 4u * W;
        if (!ZERO) {
            copy4(d, xin + c);
            copy4(d + w, xin + cw);
            copy4(d + 2 * w, xin + ce);
            copy4(d + 9 * w, xin + cs);
            copy4(d + 10 * w, xin + cn);
            copy4(d + 11 * w, xin + cd);
            copy4(d + 12 * w, xin + cu);
        }
        copy4(d + 3 * w, wx + c);
        copy4(d + 4 * w, wx + ce);
        copy4(d + 5 * w, wy + c);
        copy4(d + 6 * w, wy + cn);
        copy4(d + 7 * w, wz + c);
        copy4(d + 8 * w, wz + cu);
        copy4(d + 13 * w, bb + c);
    };
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float2 z2 = make_float2(0.f, 0.f);
    // copies of plane kk (in the grid) into slot s: one group
    const unsigned s_x = smem_u32(&sh.x[0][me + tq]), s_fx = smem_u32(&sh.fx[0][me]), s_fy = smem_u32(&sh.fy[0][me]),
                   s_b = smem_u32(&sh.b[0][me]), s_fz = smem_u32(&sh.fz[0][me]);
    const unsigned beyond = lower ? s_x - 16u * (unsigned)tq : s_x + 16u * (unsigned)tq;
    // warp 0 of a tiled row: lane l copies the ends of slot row l
    const bool ends = halo_warp && lane <= nown + 1;
    const int erow = nx * wrapped(y0 - 1 + (ends ? lane : 0), ny);
    auto copy_plane = [&](int k, int kk) {
        const int off = sz * kk, c = row + off;
        const unsigned s = (unsigned)(k & (kSlots - 1));
        if (!ZERO) copy16(s_x + s * (unsigned)sizeof(sh.x[0]), xin + c);
        copy16(s_fx + s * (unsigned)sizeof(sh.fx[0]), wx + c);
        copy16(s_fy + s * (unsigned)sizeof(sh.fy[0]), wy + c);
        copy16(s_b + s * (unsigned)sizeof(sh.b[0]), bb + c);
        copy16(s_fz + s * (unsigned)sizeof(sh.fz[0]), wz + c);
        if (lower || upper) {
            if (!ZERO) copy16(beyond + s * (unsigned)sizeof(sh.x[0]), xin + rowe + off);
            if (upper) copy16(s_fy + 16u * (unsigned)tq + s * (unsigned)sizeof(sh.fy[0]), wy + rowe + off);
        }
        if (ends) {
            copy4(smem_u32(&sh.fe[s][lane]), wx + erow + off + i_e);
            // the red cells of the row sit at offset (y0 - 1 + lane + k) & 1: 0 needs the west neighbour
            if (!ZERO) copy4(smem_u32(&sh.xe[s][lane]), xin + erow + off + (((y0 - 1 + lane + k) & 1) ? i_e : i_w));
        }
        if (halo_warp && lane < nown) copy_cell(k, kk, s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    float4 xk, xp;      // old iterate at planes k, k + 1
    float4 zk, zp;      // low z faces of planes k, k + 1
    Kept B;             // plane k - 1
    float2 r2 = z2;     // red cells of plane k - 2 in the black columns of plane k - 1
    float2 xm;          // old black cells of plane k - 1 in the red columns of plane k
    B.fx = z4;
    B.fe = 0.f;
    B.x = B.r = B.b = B.fs = B.fn = B.fb = z2;

    int kk3 = wrapped(k0 + 2, nz);  // plane k + 3 of the next step in the grid
    int cst = row + sz * (k0 - 2);  // the quad stored by the next step (from the third on)
    const int last_copy = k1 - 2;   // the last step whose plane k + 3 is needed: plane k1 + 1

    // one step: red of plane k, black of plane k - 1 (both at offsets PAR, PAR + 2)
    auto step = [&](auto tag, int k) {
        constexpr int PAR = decltype(tag)::value;
        const int cur = k & 1, prv = cur ^ 1, slot = k & (kSlots - 1), nslot = (k + 1) & (kSlots - 1);
        // into the slot of plane k - 1, read for the last time before the last barrier
        if (k <= last_copy) copy_plane(k + 3, kk3);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        kk3 = kk3 + 1 == nz ? 0 : kk3 + 1;
        const float4 fx = sh.fx[slot][me], fs = sh.fy[slot][me], fn = sh.fy[slot][me + tq], b = sh.b[slot][me];
        zp = sh.fz[nslot][me];
        const float2 ob = pick<1 - PAR>(xk);
        // red
        float fe = __shfl_sync(0xffffffffu, fx.x, le);
        if (ld_e) fe = sh.fe[slot][r];
        float xo = 0.f;
        float2 xs = z2, xn = z2;
        if (!ZERO) {
            xp = sh.x[nslot][me + tq];
            xo = PAR ? __shfl_sync(0xffffffffu, xk.x, le) : __shfl_sync(0xffffffffu, xk.w, lw);
            if (PAR ? ld_e : ld_w) xo = sh.xe[slot][r];
            xs = pick<PAR>(sh.x[slot][me]);
            xn = pick<PAR>(sh.x[slot][me + 2 * tq]);
        }
        const float2 red = relax2<PAR>(pick<PAR>(xk), ob, xo, fx, fe, pick<PAR>(fs), pick<PAR>(fn), pick<PAR>(zk),
                                       pick<PAR>(zp), xs, xn, xm, pick<PAR>(xp), pick<PAR>(b), omega, tiny);
        // black of plane k - 1 (the red cell beyond the tile from the halo warp)
        float ro = PAR ? __shfl_sync(0xffffffffu, B.r.x, le) : __shfl_sync(0xffffffffu, B.r.y, lw);
        if (own && k > k0) {
            if (PAR ? ld_e : ld_w) ro = sh.halo[prv][r];
            const float2 v = relax2<PAR>(B.x, B.r, ro, B.fx, B.fe, B.fs, B.fn, B.fb, pick<PAR>(zk),
                                         sh.red[prv][me - tq], sh.red[prv][me + tq], r2, red, B.b, omega, tiny);
            const int c = cst;
            Quad<float> o;
            o.v[PAR] = v.x;
            o.v[PAR + 2] = v.y;
            o.v[1 - PAR] = B.r.x;
            o.v[3 - PAR] = B.r.y;
            stq(xout + c, o);
        }
        sh.red[cur][me] = red;
        // plane k becomes plane k - 1
        r2 = B.r;
        B.fx = fx;
        B.fe = fe;
        B.x = ob;
        B.r = red;
        B.b = pick<1 - PAR>(b);
        B.fs = pick<1 - PAR>(fs);
        B.fn = pick<1 - PAR>(fn);
        B.fb = pick<1 - PAR>(zk);
        if (halo_warp && lane < nown) {
            float h[14];
#pragma unroll
            for (int u = 0; u < 14; u++) h[u] = ZERO && (u < 3 || (u > 8 && u < 13)) ? 0.f : sh.cell[slot][u][lane];
            sh.halo[cur][lane + 1] = relax_cell(h[0], h[1], h[2], h[3], h[4], h[5], h[6], h[7], h[8], h[9], h[10],
                                                h[11], h[12], h[13], omega, tiny);
        }
        cst += sz;
        xm = ob;
        xk = xp;
        zk = zp;
        // the copies of plane k + 2 (this thread's; the barrier: everyone's)
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
    };

    // the first planes: the copies of k0 - 1 .. k0 + 1 in flight, the rest of
    // what step k0 - 1 needs from below it
    const int par = (jj + k0 - 1) & 1;  // red offset of plane k0 - 1
    for (int p = k0 - 1; p <= k0 + 1; p++) copy_plane(p, wrapped(p, nz));
    xk = xp = z4;
    xm = z2;
    if (!ZERO) {
        const float4 x0 = ldg4(xin + row + sz * wrapped(k0 - 2, nz));
        xm = par ? make_float2(x0.y, x0.w) : make_float2(x0.x, x0.z);
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    if (!ZERO) xk = sh.x[(k0 - 1) & (kSlots - 1)][me + tq];
    zk = sh.fz[(k0 - 1) & (kSlots - 1)][me];
    // the colour's place alternates from plane to plane: two steps per pass;
    // which comes first is uniform over a warp
    const std::integral_constant<int, 0> even;
    const std::integral_constant<int, 1> odd;
    int k = k0 - 1;
    if (par) step(odd, k++);
    for (; k <= k1; k += 2) {
        step(even, k);
        if (k + 1 <= k1) step(odd, k + 1);
    }
}

__device__ __forceinline__ void march_entry(const LevelView &L, int lb, int dir, float omega, int flags, int cyc)
{
    extern __shared__ __align__(16) unsigned char march_smem[];
    March &sh = *(March *)march_smem;
    const float tiny = tiny_scale(L.st);
    // the whole block returns together (a grid's state is uniform)
    if (!in_cycle(L.st, cyc)) return;
    if (flags & kZeroGuess) march_body<true>(L, lb, dir, omega * tiny, tiny, sh);
    else march_body<false>(L, lb, dir, omega * tiny, tiny, sh);
}

__global__ void __launch_bounds__(32 * W, 1) k_march(const LevelView *__restrict__ lv, const int *__restrict__ start,
                                                     int count, int dir, float omega, int flags, int cyc,
                                                     const __grid_constant__ LevelView one, int single)
{
    dep_entry();
    if (single) {
        march_entry(one, blockIdx.x, dir, omega, flags, cyc);
        return;
    }
    const int e = find_entry(start, count);
    march_entry(lv[e], blockIdx.x - start[e], dir, omega, flags, cyc);
}

// p + v 2^sh (|sh| <= 500), with the conversion and the scaling on the bits of v:
// they and a multiply-add would be two FP64 operations a cell, the addition is one.
__device__ __forceinline__ double add_shifted(double p, float v, int sh)
{
    const bool small = (__float_as_uint(v) & 0x7fffffffu) < 0x00800000u;  // zero or subnormal
    const unsigned b = __float_as_uint(small ? __fmul_rn(v, 0x1p64f) : v), m = b & 0x7fffffffu;
    unsigned e = (m >> 3) + ((unsigned)(896 + sh - (small ? 64 : 0)) << 20);
    if (m >= 0x7f800000u) e = (m >> 3) + (1792u << 20);  // infinite, not a number
    if (m == 0u) e = 0u;
    return p + __hiloint2double((int)((b & 0x80000000u) | e), (int)(b << 29));
}

// The correction of the grids whose step ends with this cycle into their outer
// iterates, by the blocks of the sweep before it (block lb of nb of a grid takes
// every nb-th piece).  Bound by HBM: 20 B a cell, 432 us at 512^3 (6.2 TB/s).  With
// the update in the sweep's own stores, which left no register to ask for the
// iterate ahead of time, that sweep took 1175 us instead of 507; staging the iterate
// in shared memory as well left no L1 for what spilled, 1198 us.
__device__ __forceinline__ void outer_entry(const LevelView &L, int lb, int nb, int dir, int cyc,
                                            const OuterView *__restrict__ ov)
{
    if (!in_cycle(L.st, cyc) || !last_cycle(L.st, cyc)) return;
    const OuterOut po = outer_out(ov[L.g]);
    const float *__restrict__ x = (const float *)(dir ? L.x : L.x2);
    const int quads = L.n[0] * L.n[1] * L.n[2] >> 2, step = nb * 32 * W;
    const int hi = __double2hiint(po.inv), sh = (hi >> 20) - 1023;
    // an FP64 iterate of aligned pairs and a scale of 2^sh
    const bool shifted = po.t[0] == nullptr && ((size_t)po.p & 15) == 0 && (hi & 0xfffff) == 0 &&
                         __double2loint(po.inv) == 0 && sh >= -500 && sh <= 500;
    int q = lb * 32 * W + (int)threadIdx.x;
    if (po.t[0] != nullptr) {
        // three-float iterate: 28 B a cell.  Two quads in flight (one: a 160^3 solve 3570
        // us, 3500 with two; four take 100 registers instead of 76, and the FP64 form
        // below then loses 0.6 % of a 256^3 solve)
        constexpr int V = 2;
        for (; q < quads; q += V * step) {
            float4 v[V], t[3][V];
#pragma unroll
            for (int u = 0; u < V; u++) {
                const int c = q + u * step;
                if (c < quads) {
                    v[u] = ldg4(x + 4 * c);
                    for (int m = 0; m < 3; m++) t[m][u] = *(const float4 *)(po.t[m] + 4 * c);
                }
            }
#pragma unroll
            for (int u = 0; u < V; u++) {
                const int c = q + u * step;
                if (c < quads) {
                    triple_add(t[0][u].x, t[1][u].x, t[2][u].x, v[u].x);
                    triple_add(t[0][u].y, t[1][u].y, t[2][u].y, v[u].y);
                    triple_add(t[0][u].z, t[1][u].z, t[2][u].z, v[u].z);
                    triple_add(t[0][u].w, t[1][u].w, t[2][u].w, v[u].w);
                    for (int m = 0; m < 3; m++) *(float4 *)(po.t[m] + 4 * c) = t[m][u];
                }
            }
        }
        return;
    }
    if (!shifted) {
        for (; q < quads; q += step) {
            const float4 v = ldg4(x + 4 * q);
            const float e[4] = {v.x, v.y, v.z, v.w};
            add_outer_quad<float>(po, 4 * q, e, 0xF);
        }
        return;
    }
    double2 *__restrict__ p = (double2 *)po.p;
    constexpr int U = 4;  // quads of a thread in flight
    for (; q < quads; q += U * step) {
        float4 v[U];
        double2 a[U], d[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int c = q + u * step;
            if (c < quads) {
                v[u] = ldg4(x + 4 * c);
                a[u] = p[2 * c];
                d[u] = p[2 * c + 1];
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int c = q + u * step;
            if (c < quads) {
                p[2 * c] = make_double2(add_shifted(a[u].x, v[u].x, sh), add_shifted(a[u].y, v[u].y, sh));
                p[2 * c + 1] = make_double2(add_shifted(d[u].x, v[u].z, sh), add_shifted(d[u].y, v[u].w, sh));
            }
        }
    }
}

__global__ void __launch_bounds__(32 * W) k_outer_add(const LevelView *__restrict__ lv, const int *__restrict__ start,
                                                      int count, int dir, int cyc, const OuterView *__restrict__ ov,
                                                      const __grid_constant__ LevelView one, int single)
{
    dep_entry();
    if (single) {
        outer_entry(one, blockIdx.x, gridDim.x, dir, cyc, ov);
        return;
    }
    const int e = find_entry(start, count);
    outer_entry(lv[e], blockIdx.x - start[e], start[e + 1] - start[e], dir, cyc, ov);
}


// A step of the march costs about this at full rows of a tile: 1792 cells x 24 B
// a block at the measured copy rate of 152 of them (0.96 us; 0.85 out of L2).
constexpr double kStepUs = 0.95;
constexpr int kSms = 152;

}  // namespace

bool march_fits(const int n[3], int per)
{
    // rows of whole quads, and an even number of cells along every periodic
    // axis (else the colours do not alternate across the wrap)
    return (n[0] & 3) == 0 && n[1] >= 2 && n[2] >= 2 && !((per & 2) && (n[1] & 1)) && !((per & 4) && (n[2] & 1));
}

bool tiled_fits(const int n[3], int per) { return n[0] % 128 == 0 && march_fits(n, per); }

// tiles of a plane: strips of rows x tiles of quads
static int march_tiles(const int n[3], int *strips)
{
    const int tq = tile_quads(n[0]), nq = n[0] >> 2, rmax = W * (32 / tq) - 2;
    *strips = (n[1] + rmax - 1) / rmax;
    return *strips * ((nq + tq - 1) / tq);
}

// Planes per block for a level swept alone, or 0 where the two half-sweep
// launches are faster.  The chunks are as many as make the fewest steps over
// the waves of blocks (a chunk of kc planes takes kc + 2); the sweep is then
// estimated at 2 us + 0.95 us a step, the half-sweep pair at 2 us + 6 us per
// million cells out of L2, 6.9 beyond (46 B a cell at the copy rate).  Measured
// (us a sweep, pair -> march): 512^3 925 -> 509, 256^3 117 -> 67, 192^3 52.6 ->
// 39.3, 128^3 14.1 -> 11.5; and where the rule keeps the pair: 200 x 100^2 13.7
// -> 18.8, 100^3 8.3 -> 10.9, 96^3 7.0 -> 8.2, 64^3 3.9 -> 6.
int march_chunk(const int n[3], int per)
{
    if (!march_fits(n, per)) return 0;
    int strips;
    const int tiles = march_tiles(n, &strips), nz = n[2];
    int best = 0, best_steps = 0;
    for (int c = 1; c <= nz && c <= 64; c++) {
        const int kc = (nz + c - 1) / c;
        const int blocks = tiles * ((nz + kc - 1) / kc);
        const int steps = (blocks + kSms - 1) / kSms * (kc + 2);
        // fewer chunks unless more of them save 3 %
        if (best == 0 || steps * 100 < best_steps * 97) {
            best = kc;
            best_steps = steps;
        }
    }
    const double cells = (double)n[0] * n[1] * n[2] * 1e-6;
    const double pair = cells * (cells <= 3.0 ? 6.0 : 6.9);
    return best_steps * kStepUs < pair ? best : 0;
}

int march_layout(LevelView &v, int kc)
{
    const int ny = v.n[1], nz = v.n[2], nq = v.n[0] >> 2;
    int strips;
    v.fS = march_tiles(v.n, &strips);
    v.fT = tile_quads(v.n[0]);
    v.fR = (ny + strips - 1) / strips;
    const int chunks = (nz + kc - 1) / kc;
    v.fKc = (nz + chunks - 1) / chunks;
    v.dfS = make_fastdiv((unsigned)v.fS);
    v.dfq = make_fastdiv((unsigned)((nq + v.fT - 1) / v.fT));
    return v.fS * ((nz + v.fKc - 1) / v.fKc);
}

cudaError_t march_opt_in()
{
    static DeviceOnce once;
    return once(
        [] { return cudaFuncSetAttribute(k_march, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(March)); });
}

void launch_march(const Table &tb, int dir, double omega, int flags, const OuterView *ov, cudaStream_t s)
{
    if (tb.blocks == 0 || march_opt_in() != cudaSuccess) return;
    launch_k(k_march, tb.blocks, 32 * W, sizeof(March), s, tb.lv, tb.start, tb.count, dir, (float)omega, flags, tb.cyc,
             table_view(tb), table_single(tb));
    if (flags & kOuter)
        launch_k(k_outer_add, tb.blocks, 32 * W, 0, s, tb.lv, tb.start, tb.count, dir, tb.cyc, ov, table_view(tb),
                 table_single(tb));
}

}  // namespace gbmg
