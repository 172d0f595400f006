// mg_coarse.cu -- the coarsest grid's dense inverse (Sec. 2.3 item 6 of arXiv
// 1410.8568: the error on the coarsest grid is solved exactly), for coarsest
// grids of at most kMaxCoarse cells: set-up and solve.
#include "mg_kernels.h"
#include "mg_cluster.cuh"
#include "mg_stencil.cuh"

namespace gbmg {

// ---------------------------------------------------------------------------
// (6) coarsest grid: exact solve e = -G b with G = (-A + c 1 1^T)^{-1}
// ---------------------------------------------------------------------------

// For sum(b) = 0 this is the zero-mean solution of A e = b; for sum(b) != 0 it
// solves A e = b - mean(b) and adds a constant, which the cycle ignores
// (A 1 = 0) and the final mean removal takes out.  One warp per row of G
// (rows are contiguous, G is symmetric), lanes split the dot product, fixed
// shuffle tree.  A grid whose finest level is its coarsest (C.outer) adds e
// to its FP64 iterate in the last cycle of a refinement step (ov non-null).
//
// Bound by the FP64 pipe (n^2 multiply-adds, 2 lanes per clock and SM): the rows
// of a grid are split over gridDim.y blocks, one row per warp.
template <class T>
__global__ void __launch_bounds__(kThreads) k_coarse_solve(const CoarseView *__restrict__ cv, int cyc,
                                                           const OuterView *__restrict__ ov)
{
    dep_entry();
    const CoarseView &C = cv[blockIdx.x];
    if (C.gmres || !in_cycle(C.st, cyc)) return;  // GMRES grids: k_coarse_gmres
    __shared__ double rb[kMaxCoarse];
    const int n = C.nc, warps = (int)(blockDim.x >> 5), first = (int)blockIdx.y * warps;
    if (first >= n) return;
    const T *b = (const T *)C.b;
    for (int t = threadIdx.x; t < n; t += blockDim.x) rb[t] = (double)b[t];
    __syncthreads();
    T *x = (T *)C.x;
    const bool out = ov != nullptr && C.outer && last_cycle(C.st, cyc);
    const OuterOut po = out ? outer_out(ov[C.g]) : OuterOut{};
    const int lane = threadIdx.x & 31;
    for (int t = first + (int)(threadIdx.x >> 5); t < n; t += warps * (int)gridDim.y) {
        const double *Gt = C.G + (long long)t * n;
        double s = 0.0;
        for (int u = lane; u < n; u += 32) s += Gt[u] * rb[u];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            const T xn = (T)(-s);
            x[t] = xn;
            if (out) add_outer<T>(po, t, xn);
        }
    }
}

// ---------------------------------------------------------------------------
// set-up: S = -A + c 1 1^T of the coarsest level and its inverse
// ---------------------------------------------------------------------------

namespace {

constexpr int kSetupThreads = 512;
constexpr int kSetupCluster = 16;  // blocks of a larger grid

// The lower triangle's element e = r (r + 1) / 2 + c lies in register t of a
// lane: e = 32 ((t * warps + warp) * CB + block) + lane.
__device__ __forceinline__ int triangle(int r, int c) { return r * (r + 1) / 2 + c; }
__device__ __forceinline__ int triangle_row(int e)
{
    int r = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while (triangle(r + 1, 0) <= e) r++;
    while (triangle(r, 0) > e) r--;
    return r;
}

// 1 / x to within an ulp: from the FP32 reciprocal y of x (relative error e of
// about 2^-23), 1 / x = y (1 + e + e^2 + ...), cut off at e^3.  A pivot waits for
// this: 228 cycles here, 392 by __drcp_rn.  Values that FP32 does not hold (and
// what is not positive) take that.
__device__ __forceinline__ double pivot_recip(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x);
    if ((hi >> 20) - 898u > 250u) return __drcp_rn(x);  // biased exponent 898 .. 1148
    float y32;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y32) : "f"((float)x));
    const double y = (double)y32, e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// Sum of cell c's faces, and of those towards cell `nb` (a neighbour across
// both faces of a two-cell periodic axis counts twice, the cell itself, on a
// one-cell axis, not at all).
__device__ __forceinline__ double faces_of_cell(const CoarseView &C, int c, int nb, double &towards)
{
    const int nn[3] = {C.n[0], C.n[1], C.n[2]}, st[3] = {1, nn[0], nn[0] * nn[1]};
    const int q[3] = {c % nn[0], (c / nn[0]) % nn[1], c / (nn[0] * nn[1])};
    double a[6];
    int to[6];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const bool per = (C.per >> d) & 1;
        // low face: stored at the cell; high face: at the neighbour
        const int lo = q[d] > 0 ? c - st[d] : per ? c + st[d] * (nn[d] - 1) : c;
        const int hi = q[d] + 1 < nn[d] ? c + st[d] : per ? c - st[d] * (nn[d] - 1) : c;
        to[2 * d] = lo;
        to[2 * d + 1] = hi;
        a[2 * d] = lo != c ? C.w[d][c] : 0.0;
        a[2 * d + 1] = hi != c ? C.w[d][hi] : 0.0;
    }
    double sum = 0.0;
    towards = 0.0;
#pragma unroll
    for (int f = 0; f < 6; f++) {
        sum += a[f];
        if (to[f] == nb) towards += a[f];
    }
    return sum;
}

}  // namespace

// Assemble S = -A + c 1 1^T (c = mean diagonal / n, so the constant vector
// becomes an eigenvector with a mid-spectrum eigenvalue) and invert it by
// sweeps (Goodnight, Am. Stat. 33, 1979): the sweep of pivot k replaces, for
// i, j != k,
//   S_ij by S_ij - S_ik S_kj / S_kk,  S_ik by S_ik / S_kk,  S_kk by -1 / S_kk,
// stays symmetric, and after all of them S holds -S^{-1}.  S is symmetric
// positive definite, so no pivoting is needed; a non-positive pivot means the
// grid is cut into pieces by zero coefficients and raises *err.
//
// Bound by the latency of a pivot (multiply, multiply-add, reciprocal, barrier)
// and, for larger grids, by the FP64 pipe (n^3 / 2 multiply-adds: only the lower
// triangle is kept).  The elements stay in registers; a pivot's column is all
// that goes through shared memory.  CB = 1: one block, one barrier per pivot.
// CB > 1: each block first works out its elements of the next pivot's column,
// arrives at the cluster barrier and updates the rest while the others arrive;
// the column is then gathered from their owners.  Two buffers each of published
// and gathered columns: what a block overwrites was read before the barrier
// that it has waited for.
// Per set-up, against Gauss-Jordan elimination of the full matrix by one block
// through L2: 8 cells 17 us -> 8 us, 27 cells 47 us -> 27 us, 72 cells 210 us ->
// 88 us, 125 cells 1.04 ms -> 0.16 ms, 385 cells 16.6 ms -> 0.97 ms; the
// inverse's error against extended precision is the same (1e-14 of the largest entry
// at 441 cells and a density ratio of 1000).
template <int CB, int EP>
__global__ void __launch_bounds__(kSetupThreads, 1) k_coarse_setup(const __grid_constant__ CoarseView C, double inv_n2)
{
    dep_entry();
    __shared__ double pub[2][kMaxCoarse + 2];                   // published entries of a pivot column; [n]: 1 / pivot
    __shared__ double2 got[CB > 1 ? 2 : 1][CB > 1 ? kMaxCoarse + 2 : 1];  // gathered column, and divided by the pivot
    __shared__ double red[kSetupThreads / 32], mid;
    const int n = C.nc, tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31, warps = (int)blockDim.x >> 5;
    const int rank = CB > 1 ? (int)cluster_rank() : 0;
    const int total = triangle(n, 0);

    double diag = 0.0, none;
    for (int c = tid; c < n; c += (int)blockDim.x) diag += faces_of_cell(C, c, -1, none);
    // the same sum in every block, in a fixed order
    if (32 * warp < n)
        for (int o = 16; o > 0; o >>= 1) diag += __shfl_xor_sync(0xffffffffu, diag, o);
    if (lane == 0) red[warp] = diag;
    if (tid < 2) {  // what elements beyond the triangle read
        pub[tid][n + 1] = 0.0;
        if constexpr (CB > 1) got[tid][n + 1] = make_double2(0.0, 0.0);
    }
    __syncthreads();
    if (warp == 0) {
        double s = lane < warps ? red[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) mid = s * inv_n2;
    }
    __syncthreads();
    const double c0 = mid;

    double S[EP];
    int at[EP];  // row << 16 | column
#pragma unroll
    for (int t = 0; t < EP; t++) {
        const int e = 32 * ((t * warps + warp) * CB + rank) + lane;
        S[t] = 0.0;
        at[t] = (n + 1) << 16 | (n + 1);
        if (e < total) {
            const int r = triangle_row(e), c = e - triangle(r, 0);
            at[t] = r << 16 | c;
            double towards;
            const double sum = faces_of_cell(C, r, c, towards);
            S[t] = (r == c ? sum : -towards) + c0;
            if (c == 0) {
                pub[0][r] = S[t];
                if (r == 0) pub[0][n] = pivot_recip(S[t]);
            }
        }
    }
    if constexpr (CB > 1) cluster_sync();
    else __syncthreads();

    bool bad = false;
    for (int k = 0; k < n; k++) {
        const int next = k + 1;
        double rd;
        if constexpr (CB > 1) {
            const unsigned p = smem_u32(&pub[k & 1][0]);
            const unsigned own_k = (unsigned)(triangle(k, k) >> 5) % CB;
            rd = ld_cluster(map_rank(p + 8u * (unsigned)n, own_k));
            if (tid < n) {
                const unsigned own = (unsigned)(triangle(max(tid, k), min(tid, k)) >> 5) % CB;
                const double v = ld_cluster(map_rank(p + 8u * (unsigned)tid, own));
                got[k & 1][tid] = make_double2(v, v * rd);
            }
            __syncthreads();
        } else {
            rd = pub[k & 1][n];
        }
        // not a positive pivot (the same in every block): 1 / pivot is negative,
        // infinite or not a number
        if ((unsigned)__double2hiint(rd) >= 0x7ff00000u) {
            bad = true;
            break;
        }
        const double *v1 = pub[k & 1];
        const double2 *v2 = got[CB > 1 ? k & 1 : 0];
        // element (r, c) after the sweep of pivot k
        auto swept = [&](int r, int c, double s) {
            double u, v;
            if constexpr (CB > 1) {
                u = v2[r].y;
                v = v2[c].x;
            } else {
                u = v1[r] * rd;
                v = v1[c];
            }
            double x = fma(-u, v, s);
            if (r == k || c == k) x = r == c ? -rd : r != k ? u : CB > 1 ? v2[c].y : v * rd;
            return x;
        };
        auto publish = [&](int r, int c, double x) {
            pub[next & 1][r == next ? c : r] = x;
            if (r == c) pub[next & 1][n] = pivot_recip(x);
        };
        if constexpr (CB > 1) {
            if (next < n) {
#pragma unroll
                for (int t = 0; t < EP; t++) {
                    const int r = at[t] >> 16, c = at[t] & 0xffff;
                    if (r == next || c == next) publish(r, c, swept(r, c, S[t]));
                }
            }
            cluster_arrive();
        }
#pragma unroll
        for (int t = 0; t < EP; t++) {
            const int r = at[t] >> 16, c = at[t] & 0xffff;
            if (32 * (t * warps + warp) * CB < total) S[t] = swept(r, c, S[t]);
            if (CB == 1 && next < n && (r == next || c == next)) publish(r, c, S[t]);
        }
        if constexpr (CB > 1) cluster_wait();
        else __syncthreads();
    }
    if constexpr (CB > 1) cluster_sync();  // no block leaves while its column is gathered
    if (bad && rank == 0 && tid == 0) *C.err = 1;
#pragma unroll
    for (int t = 0; t < EP; t++) {
        const int r = at[t] >> 16, c = at[t] & 0xffff;
        if (r < n) {
            C.G[(long long)r * n + c] = -S[t];
            C.G[(long long)c * n + r] = -S[t];
        }
    }
}

template <class T>
void launch_coarse_solve(const CoarseView *cv, int count, int most, int cyc, const OuterView *ov, cudaStream_t s)
{
    const int warps = kThreads / 32;
    launch_k(k_coarse_solve<T>, dim3((unsigned)count, (unsigned)((most + warps - 1) / warps)), kThreads, 0, s, cv, cyc,
             ov);
}

// 16 blocks per cluster are beyond the portable 8: the kernel opts in.
template <int EP>
static cudaError_t setup_opt_in()
{
    static DeviceOnce once;
    return once([] {
        return cudaFuncSetAttribute(k_coarse_setup<kSetupCluster, EP>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    });
}

template <int EP>
static void setup_cluster(const CoarseView &v, double inv_n2, cudaStream_t s)
{
    if (setup_opt_in<EP>() != cudaSuccess) return;
    ClusterLaunch l(kSetupCluster, kSetupCluster, kSetupThreads, 0, s);
    cudaLaunchKernelEx(&l.c, k_coarse_setup<kSetupCluster, EP>, v, inv_n2);
}

template <int EP>
static cudaError_t setup_supported()
{
    const cudaError_t e = setup_opt_in<EP>();
    if (e != cudaSuccess) return e;
    static DeviceOnce once;
    return once([] {
        ClusterLaunch l(kSetupCluster, kSetupCluster, kSetupThreads, 0, nullptr);
        return l.placeable(k_coarse_setup<kSetupCluster, EP>);
    });
}

// elements of a lane of the cluster for a coarsest grid of n cells (0: one block)
static int setup_elements(int n)
{
    const int total = n * (n + 1) / 2;
    return total <= kSetupThreads ? 0 : total <= 5 * kSetupCluster * kSetupThreads ? 5 : 17;
}

cudaError_t coarse_setup_opt_in(int n)
{
    const int ep = setup_elements(n);
    return ep == 0 ? cudaSuccess : ep == 5 ? setup_supported<5>() : setup_supported<17>();
}

// One element per thread as long as one block holds them (n <= 31): without the
// cluster barrier a pivot takes 0.8 us there, against 1.2 us.
void launch_coarse_setup(const CoarseView &v, cudaStream_t s)
{
    const int n = v.nc, total = n * (n + 1) / 2;
    const double inv_n2 = 1.0 / ((double)n * n);
    static_assert(kMaxCoarse <= kSetupThreads, "a thread per entry of a gathered column");
    static_assert(kMaxCoarse * (kMaxCoarse + 1) / 2 <= 17 * kSetupCluster * kSetupThreads, "elements in registers");
    const int ep = setup_elements(n);
    if (ep == 0) launch_k(k_coarse_setup<1, 1>, 1, (total + 31) & ~31, 0, s, v, inv_n2);
    else if (ep == 5) setup_cluster<5>(v, inv_n2, s);
    else setup_cluster<17>(v, inv_n2, s);
}

template void launch_coarse_solve<float>(const CoarseView *, int, int, int, const OuterView *, cudaStream_t);
template void launch_coarse_solve<double>(const CoarseView *, int, int, int, const OuterView *, cudaStream_t);

}  // namespace gbmg
