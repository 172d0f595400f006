// mg_gmres.cu -- GMRES on the coarsest grid (Sec. 2.3 item 6 of arXiv
// 1410.8568: the error on the coarsest grid is solved by GMRES).
//
// Used for coarsest grids above the dense inverse's kMaxCoarse cells (sizes
// with a large odd factor) or on request.  Solves A e = b - mean(b) in FP64
// (the coarsest solve stays FP64 in every precision) until the residual is
// below gm_tol ||b - mean b|| or after gm_max Krylov steps; e is returned with
// zero mean.
//
// The operator is symmetric (and -A positive semidefinite), so the Arnoldi
// basis of GMRES reduces to a short recurrence: the minimal-residual iterate
// over the Krylov space without a stored basis, without restarts, in two
// updates per vector instead of an orthogonalisation against every basis vector (conjugate
// residuals: Stiefel 1955; equivalent to GMRES for such operators, Eisenstat,
// Elman & Schultz 1983).  The system is scaled by its diagonal on both sides,
//   B = I - D^-1/2 (off-diagonal part) D^-1/2,  r^ = D^-1/2 r,  e = D^-1/2 y,
// which takes the density ratio out of the step count; the stopping test is on
// the unscaled residual (r = D^1/2 r^), and a claimed convergence is checked
// with the residual evaluated from e (face differences first), from which the
// recurrence starts again if rounding kept it above the tolerance.
//
// What bounds it: the FP64 pipe (2 lanes per clock and SM) and the latency of
// the reductions.  One grid runs on a cluster of up to 16 blocks, each holding
// its cells' vectors and coefficients in shared memory and reading its
// neighbours' residual through distributed shared memory: 15 FP64 operations
// per cell and step, one reduction (3 sums) and two cluster barriers per step.
// A 100^3 time step (25^3 coarsest grid): 1287 ms with one 1024-thread block,
// Arnoldi and modified Gram-Schmidt through L2; 12.5 ms here, the same errors.  Every sum runs in a fixed
// order, so the result is deterministic.
#include "mg_kernels.h"
#include "mg_stencil.cuh"
#include "mg_cluster.cuh"

#include <math.h>

namespace gbmg {

namespace {

constexpr int kGmThreads = 256, kGmWarps = kGmThreads / 32;
constexpr int kGmCluster = 16;                                  // blocks per grid
constexpr int kGmCells = kMaxCoarseGmres / kGmCluster;          // most cells of a block
constexpr int kGmPer = kGmCells / kGmThreads;                   // most cells of a thread
constexpr int kGmSmem = kGmCells * (10 * 8 + 6 * 4);            // r, p, q, d, 6 coefficients; 6 addresses
constexpr int kGmRestarts = 8;
static_assert(kGmPer * kGmThreads == kGmCells, "whole threads");
static_assert(kGmSmem + 3 * kGmThreads * 8 + 1024 <= 232448, "shared memory of one block");

struct GmScratch {
    double part[3][kGmThreads];       // one value per thread
    double all[2][3][kGmCluster];     // one total per block of the cluster (alternating sums)
    double tot[3];
};

// Sums over the cluster of `count` values per thread, in a fixed order; every
// thread gets them in v.  Two block barriers and one cluster barrier.  A warp
// per sum adds the threads' values (8 per lane, then a shuffle tree): the sum
// over all warps' lanes would cost as much FP64 time as a step.
__device__ __forceinline__ void cluster_sum(double v[3], int count, GmScratch &S, unsigned &turn, unsigned rank,
                                            unsigned size)
{
    // two sets of totals: a block may start the next sum while another still
    // reads this one, but not the one after it (the next sum's barrier)
    turn ^= 1u;
    const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int q = 0; q < count; q++) S.part[q][tid] = v[q];
    __syncthreads();
    if (warp < count) {
        double s = S.part[warp][lane];
        for (int u = 1; u < kGmWarps; u++) s += S.part[warp][lane + 32 * u];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane < (int)size) st_cluster(map_rank(smem_u32(&S.all[turn][warp][rank]), (unsigned)lane), s);
    }
    cluster_sync();
    if (warp < count) {
        double s = lane < (int)size ? S.all[turn][warp][lane] : 0.0;
        for (int o = kGmCluster / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) S.tot[warp] = s;
    }
    __syncthreads();
    for (int q = 0; q < count; q++) v[q] = S.tot[q];
}

// Neighbour cells of cell c in the order x low, x high, y low, ...: their index
// and the scaled face between (0 and the cell itself at a wall).
__device__ __forceinline__ void faces_of(const CoarseView &C, int c, int nb[6], double w[6])
{
    const int nx = C.n[0], ny = C.n[1], nz = C.n[2], per = C.per;
    const int rest = c / nx;
    const int i = c - rest * nx, j = rest % ny, k = rest / ny;
    const int pos[3] = {i, j, k}, n[3] = {nx, ny, nz}, st[3] = {1, nx, nx * ny};
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const bool p = (per >> d) & 1;
        const int lo = pos[d] > 0 ? c - st[d] : p ? c + st[d] * (n[d] - 1) : c;
        const int hi = pos[d] + 1 < n[d] ? c + st[d] : p ? c - st[d] * (n[d] - 1) : c;
        nb[2 * d] = lo;
        nb[2 * d + 1] = hi;
        w[2 * d] = lo != c ? C.w[d][c] : 0.0;
        w[2 * d + 1] = hi != c ? C.w[d][hi] : 0.0;
    }
}

}  // namespace

template <class T>
__global__ void __launch_bounds__(kGmThreads, 1) k_coarse_gmres(const CoarseView *__restrict__ cv, int cyc,
                                                                const OuterView *__restrict__ ov, int size)
{
    dep_entry();
    const CoarseView &C = cv[blockIdx.x / (unsigned)size];
    if (!C.gmres || !in_cycle(C.st, cyc)) return;  // uniform over the cluster
    cluster_arrive();  // this block has started (waited for before the first remote access)
    extern __shared__ __align__(16) unsigned char gm_smem[];
    __shared__ GmScratch S;
    unsigned turn = 0;
    const unsigned rank = cluster_rank();
    const int n = C.nc, tid = (int)threadIdx.x;
    const int per = (n + size - 1) / size;  // cells of a block (the last ones may hold fewer)
    const int c0 = min((int)rank * per, n), cells = min(per, n - c0);
    double *r = (double *)gm_smem, *p = r + per, *q = p + per, *d = q + per, *a = d + per;
    double y[kGmPer];  // the solution at the thread's cells u = tid + m kGmThreads
    unsigned *ad = (unsigned *)(a + 6 * per);
    const T *bt = (const T *)C.b;

    // diagonal, its inverse root (exchanged through r), scaled off-diagonals
    // and the neighbours' addresses; mean of b
    double v[3] = {0.0, 0.0, 0.0};
    for (int u = tid; u < cells; u += kGmThreads) {
        int nb[6];
        double w[6], s = 0.0;
        faces_of(C, c0 + u, nb, w);
        for (int f = 0; f < 6; f++) s += w[f];
        d[u] = s;
        r[u] = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
        for (int f = 0; f < 6; f++) {
            const int o = nb[f] / per;
            ad[6 * u + f] = map_rank(smem_u32(r + (nb[f] - o * per)), (unsigned)o);
            a[6 * u + f] = w[f];
        }
        v[0] += (double)bt[c0 + u];
    }
    cluster_wait();  // every block has started: its shared memory may be written
    cluster_sum(v, 1, S, turn, rank, (unsigned)size);  // (its cluster barrier publishes r)
    const double mean = v[0] / n;
    for (int u = tid; u < cells; u += kGmThreads) {
        const double s = r[u];
        for (int f = 0; f < 6; f++) a[6 * u + f] *= s * ld_cluster(ad[6 * u + f]);
    }
    v[0] = 0.0;
    for (int u = tid; u < cells; u += kGmThreads) {
        const double b = (double)bt[c0 + u] - mean;
        v[0] += b * b;
    }
#pragma unroll
    for (int m = 0; m < kGmPer; m++) y[m] = 0.0;
    cluster_sum(v, 1, S, turn, rank, (unsigned)size);  // (its cluster barrier: the neighbours' roots are read)
    const double goal = C.gm_tol * C.gm_tol * v[0];
    double best = INFINITY;
    int it = 0;
    for (int start = 0; v[0] > 0.0 && it < C.gm_max && start <= kGmRestarts; start++) {
        // r^ = D^-1/2 (b - A e), e = D^-1/2 y: from zero, or evaluated with face
        // differences from the exchanged e
        if (start > 0) {
#pragma unroll
            for (int m = 0; m < kGmPer; m++) {
                const int u = tid + m * kGmThreads;
                if (u < cells) r[u] = d[u] > 0.0 ? y[m] / sqrt(d[u]) : 0.0;
            }
            cluster_sync();
            double keep[kGmPer];
            v[0] = 0.0;
#pragma unroll
            for (int m = 0; m < kGmPer; m++) {
                const int u = tid + m * kGmThreads;
                keep[m] = 0.0;
                if (u >= cells) continue;
                int nb[6];
                double w[6], s = (double)bt[c0 + u] - mean;
                faces_of(C, c0 + u, nb, w);
                for (int f = 0; f < 6; f++) s -= w[f] * (ld_cluster(ad[6 * u + f]) - r[u]);
                keep[m] = s;
                v[0] += s * s;
            }
            cluster_sum(v, 1, S, turn, rank, (unsigned)size);  // every read of e is done
#pragma unroll
            for (int m = 0; m < kGmPer; m++) {
                const int u = tid + m * kGmThreads;
                if (u < cells) r[u] = d[u] > 0.0 ? keep[m] / sqrt(d[u]) : 0.0;
            }
            // converged, or no further gain from starting again (or NaN)
            if (!(v[0] > goal) || !(v[0] < 0.25 * best)) break;
            best = v[0];
        } else {
            for (int u = tid; u < cells; u += kGmThreads)
                r[u] = d[u] > 0.0 ? ((double)bt[c0 + u] - mean) / sqrt(d[u]) : 0.0;
        }
        for (int u = tid; u < cells; u += kGmThreads) p[u] = q[u] = 0.0;
        cluster_sync();
        // conjugate residuals on B: with s = B r, rho = (r, s):
        //   beta = rho / rho_old, p = r + beta p, q = B p = s + beta q,
        //   alpha = rho / (q, q), y += alpha p, r -= alpha q
        // and (q, q) = (s, s) - beta^2 (q, q)_old, q being orthogonal to its predecessor.
        // With A = -D^1/2 B D^1/2 on e, the correction enters y with a minus sign.
        double rho_old = 0.0, qq = 0.0;
        bool done = false;
        while (it < C.gm_max && !done) {
            double s[kGmPer];
            v[0] = v[1] = v[2] = 0.0;
#pragma unroll
            for (int m = 0; m < kGmPer; m++) {
                const int u = tid + m * kGmThreads;
                s[m] = 0.0;
                if (u >= cells) continue;
                const double ru = r[u];
                double f = ru;
                for (int g = 0; g < 6; g++) f = fma(-a[6 * u + g], ld_cluster(ad[6 * u + g]), f);
                s[m] = f;
                v[0] = fma(ru, f, v[0]);
                v[1] = fma(f, f, v[1]);
                v[2] = fma(ru * ru, d[u], v[2]);
            }
            cluster_sum(v, 3, S, turn, rank, (unsigned)size);
            const double beta = rho_old > 0.0 ? v[0] / rho_old : 0.0;
            qq = v[1] - beta * beta * qq;
            rho_old = v[0];
            // converged by the recurrence, or broken down (rounding, NaN): the
            // residual evaluated from e decides
            done = !(v[2] > goal) || !(qq > 0.0) || !(v[0] > 0.0);
            if (!done) {
                const double alpha = v[0] / qq;
#pragma unroll
                for (int m = 0; m < kGmPer; m++) {
                    const int u = tid + m * kGmThreads;
                    if (u >= cells) continue;
                    const double pu = fma(beta, p[u], r[u]), qu = fma(beta, q[u], s[m]);
                    p[u] = pu;
                    q[u] = qu;
                    y[m] = fma(-alpha, pu, y[m]);
                    r[u] = fma(-alpha, qu, r[u]);
                }
                it++;
            }
            cluster_sync();
        }
        v[0] = 1.0;  // (go round again to check)
    }
    // e = D^-1/2 y with zero mean
    v[0] = 0.0;
#pragma unroll
    for (int m = 0; m < kGmPer; m++) {
        const int u = tid + m * kGmThreads;
        if (u >= cells) continue;
        y[m] = d[u] > 0.0 ? y[m] / sqrt(d[u]) : 0.0;
        v[0] += y[m];
    }
    cluster_sum(v, 1, S, turn, rank, (unsigned)size);
    const double em = v[0] / n;
    T *x = (T *)C.x;
    // single-level grid: the last cycle of a refinement step also updates p
    const bool out = ov != nullptr && C.outer && last_cycle(C.st, cyc);
    const OuterOut po = out ? outer_out(ov[C.g]) : OuterOut{};
#pragma unroll
    for (int m = 0; m < kGmPer; m++) {
        const int u = tid + m * kGmThreads;
        if (u >= cells) continue;
        const T xn = (T)(y[m] - em);
        x[c0 + u] = xn;
        if (out) add_outer<T>(po, c0 + u, xn);
    }
    cluster_sync();  // no block leaves while another may still write its sums
}

// 16 blocks per cluster are beyond the portable 8: the kernel opts in.
template <class T>
static cudaError_t gm_opt_in()
{
    static DeviceOnce once;
    return once([] {
        const cudaError_t e =
            cudaFuncSetAttribute(k_coarse_gmres<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGmSmem);
        if (e != cudaSuccess) return e;
        return cudaFuncSetAttribute(k_coarse_gmres<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    });
}

template <class T>
void launch_coarse_gmres(const CoarseView *cv, int count, int cyc, const OuterView *ov, cudaStream_t s)
{
    if (gm_opt_in<T>() != cudaSuccess) return;
    ClusterLaunch l(kGmCluster, count * kGmCluster, kGmThreads, kGmSmem, s);
    cudaLaunchKernelEx(&l.c, k_coarse_gmres<T>, cv, cyc, ov, kGmCluster);
}

template <class T>
static cudaError_t gm_supported()
{
    const cudaError_t e = gm_opt_in<T>();
    if (e != cudaSuccess) return e;
    static DeviceOnce once;
    return once([] {
        ClusterLaunch l(kGmCluster, kGmCluster, kGmThreads, kGmSmem, nullptr);
        return l.placeable(k_coarse_gmres<T>);
    });
}

// (a mixed handle solves its coarsest grid in FP64 on request: mg_coarse_solve)
cudaError_t coarse_gmres_opt_in()
{
    const cudaError_t e = gm_supported<float>();
    return e != cudaSuccess ? e : gm_supported<double>();
}

template void launch_coarse_gmres<float>(const CoarseView *, int, int, const OuterView *, cudaStream_t);
template void launch_coarse_gmres<double>(const CoarseView *, int, int, const OuterView *, cudaStream_t);

}  // namespace gbmg
