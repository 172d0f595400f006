// mg_pcg.cu -- conjugate gradients preconditioned by V-cycles (MG_SOLVER_PCG).
//
// The pressure operator A of Eq. 10 (arXiv 1410.8568) is symmetric negative
// semidefinite with the constants as its null space; CG runs on the SPD
// operator -A on the zero-mean subspace.  The residual keeps the sign of the
// multigrid iteration, r = b0 - A p, and q = A d, so that
//   alpha = (r.z) / (d.q),  p += alpha d,  r -= alpha q,
//   beta = -alpha (z_new.q) / (r.z)_old  (Polak-Ribiere form: equal to the
//   classical one for a fixed symmetric preconditioner, and tolerant of the
//   FP32 V-cycle being a slightly variable one),
//   d = (z_new - mean z_new) + beta d,
// with z = M r the correction of inner_cycles V-cycles from zero.  Every
// vector of the outer iteration is FP64; the V-cycle runs in its own
// precision.  All sums are block partials reduced in a fixed order by one
// block per grid (deterministic, the same alone and in a batch).
#include "mg_kernels.h"
#include "mg_outer.cuh"
#include "mg_stencil.cuh"

#include <math.h>

namespace gbmg {

// q = A d (FP64, face differences first) and partial d.q (slot 0)
__global__ void __launch_bounds__(kThreads, 4) k_pcg_matvec(const OuterView *__restrict__ ov,
                                                            const int *__restrict__ start, int count)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView &O = ov[e];
    if (!O.st->active) return;
    const int lb = blockIdx.x - start[e];
    double v[1] = {0.0};
    if (O.mitems) {
        march_pairs(O, O.d, lb, [](int) { return make_double2(0.0, 0.0); },
                    [&](int c, double s0, double s1, double2 d) {
                        *reinterpret_cast<double2 *>(O.q + c) = make_double2(-s0, -s1);
                        v[0] = fma(-s0, d.x, v[0]);
                        v[0] = fma(-s1, d.y, v[0]);
                    });
    } else {
        for_cells(O, lb, [&](int c, int i, int j, int k) {
            const double qc = flux64(O, O.d, i, j, k, c);
            O.q[c] = qc;
            v[0] += O.d[c] * qc;
        });
    }
    block_sum(v);
    if (threadIdx.x == 0) O.part[kPart * lb + 0] = v[0];
}

// p += alpha d, r -= alpha q, the V-cycle's right-hand side = r in its
// precision Te, partial ||r||^2 (slot 0, FP64)
template <class Te>
__global__ void __launch_bounds__(kThreads) k_pcg_update(const OuterView *__restrict__ ov,
                                                         const int *__restrict__ start, int count)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView &O = ov[e];
    const GridState *s = O.st;
    if (!s->active) return;
    const int lb = blockIdx.x - start[e];
    const double a = s->alpha;
    const bool pairs = p_pairs(O);
    Te *rv = (Te *)O.r;
    double v[1] = {0.0};
    struct In {
        double2 p, d, r, q;
    };
    for_pairs(
        O, lb,
        [&](int c, bool both) {
            if (both) return In{ld_p(O, c, pairs), ld2(O.d + c), ld2(O.r64 + c), ld2(O.q + c)};
            const double2 z = make_double2(0.0, 0.0);
            In x{z, z, z, z};
            x.p.x = O.p[c];
            x.d.x = O.d[c];
            x.r.x = O.r64[c];
            x.q.x = O.q[c];
            return x;
        },
        [&](int c, const In &x, bool both) {
            const double2 p = make_double2(fma(a, x.d.x, x.p.x), fma(a, x.d.y, x.p.y));
            const double2 r = make_double2(fma(-a, x.q.x, x.r.x), fma(-a, x.q.y, x.r.y));
            v[0] = fma(r.x, r.x, v[0]);
            v[0] = fma(r.y, r.y, v[0]);
            O.p[c] = p.x;
            O.r64[c] = r.x;
            rv[c] = (Te)r.x;
            if (both) {
                O.p[c + 1] = p.y;
                O.r64[c + 1] = r.y;
                rv[c + 1] = (Te)r.y;
            }
        });
    block_sum(v);
    if (threadIdx.x == 0) O.part[kPart * lb + 0] = v[0];
}

// z = the V-cycle correction (FP64); partials z.q (slot 0), r.z (slot 1),
// sum z (slot 2)
template <class Te>
__global__ void __launch_bounds__(kThreads) k_pcg_z(const OuterView *__restrict__ ov,
                                                    const int *__restrict__ start, int count)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView &O = ov[e];
    if (!O.st->active) return;
    const int lb = blockIdx.x - start[e];
    const Te *ev = (const Te *)O.e;
    double v[3] = {0.0, 0.0, 0.0};
    struct In {
        double2 q, r;
        Te z0, z1;
    };
    for_pairs(
        O, lb,
        [&](int c, bool both) {
            if (both) return In{ld2(O.q + c), ld2(O.r64 + c), ev[c], ev[c + 1]};
            return In{make_double2(O.q[c], 0.0), make_double2(O.r64[c], 0.0), ev[c], Te(0)};
        },
        [&](int c, const In &x, bool both) {
            const double z0 = (double)x.z0, z1 = (double)x.z1;
            v[0] = fma(z0, x.q.x, v[0]);
            v[1] = fma(x.r.x, z0, v[1]);
            v[2] += z0;
            O.z[c] = z0;
            if (both) {
                v[0] = fma(z1, x.q.y, v[0]);
                v[1] = fma(x.r.y, z1, v[1]);
                v[2] += z1;
                O.z[c + 1] = z1;
            }
        });
    block_sum(v);
    if (threadIdx.x == 0)
        for (int f = 0; f < 3; f++) O.part[kPart * lb + f] = v[f];
}

// d = (z - mean z) + beta d (first: d = z - mean z)
__global__ void __launch_bounds__(kThreads) k_pcg_dir(const OuterView *__restrict__ ov,
                                                      const int *__restrict__ start, int count, int first)
{
    dep_entry();
    const int e = find_entry(start, count);
    const OuterView &O = ov[e];
    const GridState *s = O.st;
    if (!s->active) return;
    const int lb = blockIdx.x - start[e];
    const double m = s->zmean, b = s->beta;
    struct In {
        double2 z, d;
    };
    for_pairs(
        O, lb,
        [&](int c, bool both) {
            const double2 z2 = make_double2(0.0, 0.0);
            if (both) return In{ld2(O.z + c), first ? z2 : ld2(O.d + c)};
            return In{make_double2(O.z[c], 0.0), first ? z2 : make_double2(O.d[c], 0.0)};
        },
        [&](int c, const In &x, bool both) {
            O.d[c] = first ? x.z.x - m : fma(b, x.d.x, x.z.x - m);
            if (both) O.d[c + 1] = first ? x.z.y - m : fma(b, x.d.y, x.z.y - m);
        });
}

// One block per grid: reduce the partials in a fixed order and update the
// scalars.  mode 0: after the first preconditioning (rz, mean z, beta = 0);
// mode 1: after the product A d (alpha; d.q must be negative, else the
// iteration broke down and the grid stops as diverged); mode 2: after a
// later preconditioning (beta, rz, mean z).
__global__ void __launch_bounds__(kThreads) k_pcg_finalize(const OuterView *__restrict__ ov, int mode)
{
    dep_entry();
    const OuterView &O = ov[blockIdx.x];
    GridState *s = O.st;
    if (!s->active) return;
    const double N = (double)O.n[0] * O.n[1] * O.n[2];
    if (mode == 1) {
        double dq[1] = {0.0};
        for (int q = threadIdx.x; q < O.nblk; q += blockDim.x) dq[0] += O.part[kPart * q];
        block_sum(dq);
        if (threadIdx.x != 0) return;
        const double a = s->rz / dq[0];
        if (!(dq[0] < 0.0) || !isfinite(a)) {
            stop_grid(s, 5);  // MG_EDIVERGED
            return;
        }
        s->alpha = a;
        return;
    }
    double v[3] = {0.0, 0.0, 0.0};
    for (int q = threadIdx.x; q < O.nblk; q += blockDim.x)
        for (int f = 0; f < 3; f++) v[f] += O.part[kPart * q + f];
    block_sum(v);
    if (threadIdx.x != 0) return;
    s->beta = mode == 0 ? 0.0 : -s->alpha * v[0] / s->rz;
    s->rz = v[1];
    s->zmean = v[2] / N;
    if (!isfinite(s->beta) || !isfinite(s->rz)) stop_grid(s, 5);
}

void launch_pcg_matvec(const OuterTable &ot, cudaStream_t s)
{
    launch_k(k_pcg_matvec, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count);
}
template <class Te>
void launch_pcg_update(const OuterTable &ot, cudaStream_t s)
{
    launch_k(k_pcg_update<Te>, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count);
}
template <class Te>
void launch_pcg_z(const OuterTable &ot, cudaStream_t s)
{
    launch_k(k_pcg_z<Te>, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count);
}
void launch_pcg_dir(const OuterTable &ot, int first, cudaStream_t s)
{
    launch_k(k_pcg_dir, ot.blocks, kThreads, 0, s, ot.ov, ot.start, ot.count, first);
}
void launch_pcg_finalize(const OuterTable &ot, int mode, cudaStream_t s)
{
    launch_k(k_pcg_finalize, ot.count, kThreads, 0, s, ot.ov, mode);
}

template void launch_pcg_update<float>(const OuterTable &, cudaStream_t);
template void launch_pcg_update<double>(const OuterTable &, cudaStream_t);
template void launch_pcg_z<float>(const OuterTable &, cudaStream_t);
template void launch_pcg_z<double>(const OuterTable &, cudaStream_t);

}  // namespace gbmg
