// The whole CGP step of many independent instances in ONE persistent launch (a form beyond
// the paper).  Every thread-block cluster of the launch takes instances from a queue (the
// host orders them by an estimate of their step, longest first) and advances each by one complete step of Eqs. 21-26;
// the cluster's CTAs share the rows, reduce through distributed shared memory, and
// synchronise with the hardware cluster barrier between phases; clusters never wait on one
// another.
//
//   Eq. 21     the rows of the momentum system (step_rows.cuh), then BiCGStab with Jacobi
//              for both velocity components (three cluster sums per iteration; restarted from
//              the true residual after a breakdown): FP64, or for a mixed instance FP32 inner
//              solves inside FP64 refinement, then FP64 only if the sweeps fell short
//   Eqs. 22-23 the injected coarse right-hand side (with the range projection of a
//              pure-Neumann problem and the lifted phi data of a traction boundary), then the
//              instance's one-launch coarse PCG (coarse_pcg_body: FP64, or FP32 inner / FP64
//              outer, as the instance is assembled)
//   Eq. 24     prolongation, level by level
//   Eq. 25     the correction's right-hand side and, with the consistent mass, Chebyshev
//              semi-iteration on M0 with Jacobi: the eigenvalues of D^-1 M of P1 triangles lie
//              in [1/2, 2] (every element matrix D_e^-1 M_e has eigenvalues 1/2, 1/2, 2), so the
//              steps need no inner products and their number follows from the tolerance
//              (error <= 4 * 3^-n of the initial one in the energy norm)
//   Eq. 26     the rotational term (D U~, and the same Chebyshev solve on M) and the update
// In a mixed instance the momentum BiCGStab's inner iterations and the Chebyshev steps run in
// FP32: on this GPU the narrow FP64 pipe is the busiest unit of the cluster's FP64 iterations.
// Clocks of a 66k-row instance's step on 8 CTAs (iterations in
// brackets): momentum 5.5M (20 iterations), coarse solve at 4,225 rows 7.5M (450; 10.4M with
// its vectors in memory), the two mass solves 4.3M (5.8M in FP64), assembly 1.0M.
#pragma once

#include <cooperative_groups.h>

#include "coarse_pcg.cuh"
#include "solver.cuh"
#include "step_rows.cuh"

namespace cgp {

namespace cgrp_bs = cooperative_groups;

// everything one instance's step reads and writes (device pointers into its solver)
struct BatchStepArgs {
    // fine level
    int nf;
    SellView Af;
    const int32_t *rowptr, *col, *sell_ptr, *vt_ptr, *vt_list, *tri, *vtslot;
    const double *geo, *xy, *S, *M, *M0, *CxT, *CyT, *Cx, *Cy, *dinvM0, *dinvM, *mlumpF;
    const uint8_t* tag;
    double *U, *Uprev, *P, *Ut, *w, *h, *A, *dinvA, *b, *g, *delta, *div, *qrot, *phi;
    BicgVecs bv;
    double *c0, *c1, *c2;   // Chebyshev work: residual, two directions (2 nf each)
    // mixed instances (null otherwise): FP32 copies of A (refreshed each step) and its Jacobi
    // diagonal, FP32 work vectors (2 nf each); the momentum solve then runs FP32 inner solves
    // inside FP64 refinement
    int64_t nnz;
    float *A32, *dinvA32;
    float* fv[10];
    const float *M0f, *Mf, *dinvM0f, *dinvMf;   // FP32 mass matrices and Jacobi diagonals
    double tol_mass2;
    // coarse level and its solve
    SellView Ac;
    const double *Cxc, *Cyc, *Kc, *cxy;
    const uint8_t* ctag;
    CoarsePcgArgs coarse;
    int pure_neumann;
    // prolongation: levels lc .. lf
    int nlev;
    int nv[5];
    const int32_t* parents[5];   // parents[l]: end points of the vertices added at level lc + l + 1
    // parameters
    BcParams bc;
    double dt, inv_re, tol_mom2;
    int chi, lumped, max_it_mom, cheb_steps;
    double* tdev;
    DeviceStats* stats;
    KrylovState* ks;
};

// number of Chebyshev steps for a relative energy-norm error tol with eigenvalue bounds
// [1/2, 2] (condition 4): 4 * 3^-n <= tol
__host__ __device__ inline int cheb_steps_for(double tol) {
    int n = 1;
    double bound = 4.0 / 3.0;
    while (bound > tol && n < 200) {
        bound /= 3.0;
        ++n;
    }
    return n;
}

// The step's coefficients of the semi-iteration with these bounds (theta = 1.25, delta = 0.75):
// d' = c1 d + c2 D^-1 r.  A table: the recurrence's two FP64 divides in every thread cost 7k
// clocks a step.
struct ChebTable {
    double c1[200], c2[200];
    constexpr ChebTable() : c1(), c2() {
        const double delta = 0.75, sigma = 1.25 / 0.75;
        double rho = 1.0 / sigma;
        for (int k = 0; k < 200; ++k) {
            const double next = 1.0 / (2.0 * sigma - rho);
            c1[k] = next * rho;
            c2[k] = 2.0 * next / delta;
            rho = next;
        }
    }
};
static __constant__ ChebTable kChebTable = ChebTable();

// Mixed instances: the momentum system runs up to kBatchIrSweeps FP64-residual sweeps around
// an FP32 BiCGStab (each asked for kBatchInnerTol of its right-hand side, or what is left to
// the tolerance) while they gain at least a decade each, then the FP64 BiCGStab unless a
// sweep's residual already met the tolerance.  (With three sweeps, two of 32 cavities at a
// tolerance of 1e-12 were left just above it and spent 15M clocks in the FP64 iteration.)
constexpr int kBatchIrSweeps = 8;
constexpr double kBatchInnerTol = 1e-4;
constexpr int kBatchInnerMaxit = 200;

// rows sl[0 .. U-1] (slices; one past the end: none) of the two- or one-component product A u,
// the pattern and value loads of all U slices in flight together
template <int U, int NC, class T>
__device__ __forceinline__ void spmv_slices(const SellView& A, const T* __restrict__ val, const T* __restrict__ u,
                                            const int (&sl)[U], int lane, T (&ax)[U][NC]) {
    int base[U], w[U], wmax = 0;
#pragma unroll
    for (int q = 0; q < U; ++q) {
        base[q] = w[q] = 0;
        if (sl[q] < A.nslices) {
            base[q] = __ldg(A.ptr + sl[q]);
            w[q] = (__ldg(A.ptr + sl[q] + 1) - base[q]) >> 5;
        }
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
        wmax = max(wmax, w[q]);
#pragma unroll
        for (int c = 0; c < NC; ++c) ax[q][c] = T(0);
    }
    for (int k0 = 0; k0 < wmax; k0 += 8) {
        int cj[U][8];
        T av[U][8];
#pragma unroll
        for (int q = 0; q < U; ++q)
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                cj[q][k] = 0;
                av[q][k] = T(0);
                if (k0 + k < w[q]) {
                    const int e = base[q] + 32 * (k0 + k) + lane;
                    cj[q][k] = __ldg(A.col + e);
                    av[q][k] = __ldg(val + e);
                }
            }
#pragma unroll
        for (int q = 0; q < U; ++q)
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k0 + k < w[q]) {
                    T xv[NC];
                    ldv<NC>(u, cj[q][k], xv);
#pragma unroll
                    for (int c = 0; c < NC; ++c) ax[q][c] += av[q][k] * xv[c];
                }
    }
}

// `steps` Chebyshev steps on B e = r (NC interleaved components) from e = 0, with Jacobi and the
// bounds [1/2, 2] of D^-1 B; one cluster barrier per step.  r is overwritten.
template <int NC, class T>
__device__ void cluster_cheb_steps(const SellView& B, const T* __restrict__ val, const T* __restrict__ dinv, T* r, T* e,
                                   T* d0, T* d1, int steps, int crank, int csize, cgrp_bs::cluster_group& cl) {
    constexpr int U = sizeof(T) == 4 ? 2 : 1;   // slices in flight per warp (registers)
    const int n = B.n, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5, wid = threadIdx.x >> 5;
    const int stride = csize * nwarp;
    for (int i = crank * blockDim.x + threadIdx.x; i < n; i += csize * blockDim.x) {
        T rv[NC], dv[NC], zero[NC];
        ldv<NC>(r, i, rv);
        const T di = dinv[i] * T(0.8);   // 1 / theta
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            dv[c] = di * rv[c];
            zero[c] = T(0);
        }
        stv<NC>(d0, i, dv);
        stv<NC>(e, i, zero);
    }
    cl.sync();
    T* dc = d0;
    T* dn = d1;
    for (int k = 0; k < steps; ++k) {
        const T c1 = (T)kChebTable.c1[k], c2 = (T)kChebTable.c2[k];
        for (int s0 = crank * nwarp + wid; s0 < B.nslices; s0 += U * stride) {
            int sl[U];
#pragma unroll
            for (int q = 0; q < U; ++q) sl[q] = s0 + q * stride;
            T dv[U][NC], rv[U][NC], ev[U][NC], di[U], wv[U][NC];
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const int i = sl[q] * 32 + lane;
                if (i < n) {
                    ldv<NC>(dc, i, dv[q]);
                    ldv<NC>(r, i, rv[q]);
                    ldv<NC>(e, i, ev[q]);
                    di[q] = dinv[i];
                }
            }
            spmv_slices<U, NC>(B, val, dc, sl, lane, wv);
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const int i = sl[q] * 32 + lane;
                if (i < n) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        ev[q][c] += dv[q][c];
                        rv[q][c] -= wv[q][c];
                        dv[q][c] = c1 * dv[q][c] + c2 * di[q] * rv[q][c];
                    }
                    stv<NC>(e, i, ev[q]);
                    stv<NC>(r, i, rv[q]);
                    stv<NC>(dn, i, dv[q]);
                }
            }
        }
        cl.sync();
        T* t = dc;
        dc = dn;
        dn = t;
    }
}

// B x = rhs in FP64 by one run of the semi-iteration
template <int NC>
__device__ __noinline__ void cluster_chebyshev(const SellView& B, const double* __restrict__ val, const double* __restrict__ dinv,
                                  const double* __restrict__ rhs, double* x, double* r, double* d0, double* d1,
                                  int steps, int crank, int csize, cgrp_bs::cluster_group& cl) {
    // (each thread copies the rows that it initialises in cluster_cheb_steps)
    for (int i = crank * blockDim.x + threadIdx.x; i < B.n; i += csize * blockDim.x) {
        double v[NC];
        ldv<NC>(rhs, i, v);
        stv<NC>(r, i, v);
    }
    cluster_cheb_steps<NC, double>(B, val, dinv, r, x, d0, d1, steps, crank, csize, cl);
}

// B x = rhs of a mixed instance: sweeps of the FP64 residual and kBatchChebSteps FP32 steps
// (each reduces the error to below 1e-5) until the residual meets the tolerance; false when
// kBatchChebSweeps did not get there (the caller then runs the FP64 semi-iteration).  A step of
// a 66k-row instance on 8 CTAs is bound by the FP64 pipe in FP64 (130k clocks), by latency in
// FP32.
constexpr int kBatchChebSteps = 12, kBatchChebSweeps = 6;

template <int NC>
__device__ __noinline__ bool cluster_cheb_mixed(const SellView& B, const double* __restrict__ val, const float* __restrict__ val32,
                                   const float* __restrict__ dinv32, const double* __restrict__ rhs, double* x,
                                   float* r32, float* e, float* d0, float* d1, double tol2, ClusterSync& cs, int crank,
                                   int csize, cgrp_bs::cluster_group& cl, int& steps) {
    const int n = B.n, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5, wid = threadIdx.x >> 5;
    double bb[NC];
    steps = 0;
    for (int sw = 0; sw <= kBatchChebSweeps; ++sw) {
        double acc[2 * NC];
#pragma unroll
        for (int c = 0; c < 2 * NC; ++c) acc[c] = 0.0;
        for (int sl = crank * nwarp + wid; sl < B.nslices; sl += csize * nwarp) {
            const int i = sl * 32 + lane;
            double ax[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) ax[c] = 0.0;
            if (sw) sell_accum<NC>(B, val, sl, lane, [&](int j, double (&o)[NC]) { ldv<NC>(x, j, o); }, ax);
            if (i < n) {
                double bv[NC], zero[NC];
                float rf[NC];
                ldv<NC>(rhs, i, bv);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const double rv = bv[c] - ax[c];
                    rf[c] = (float)rv;
                    zero[c] = 0.0;
                    acc[c] += rv * rv;
                    acc[NC + c] += bv[c] * bv[c];
                }
                stv<NC>(r32, i, rf);
                if (!sw) stv<NC>(x, i, zero);
            }
        }
        double tot[2 * NC];
        cs.sum(acc, tot);   // (r32 is complete: a cluster barrier)
        bool all = true, finite_all = true;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if (!sw) bb[c] = tot[NC + c];
            all = all && tot[c] <= tol2 * bb[c];
            finite_all = finite_all && isfinite(tot[c]);
        }
        if (all) return true;
        if (!finite_all || sw == kBatchChebSweeps) return false;
        cluster_cheb_steps<NC, float>(B, val32, dinv32, r32, e, d0, d1, kBatchChebSteps, crank, csize, cl);
        steps += kBatchChebSteps;
        for (int sl = crank * nwarp + wid; sl < B.nslices; sl += csize * nwarp) {
            const int i = sl * 32 + lane;
            if (i < n) {
                double xv[NC];
                float ev[NC];
                ldv<NC>(x, i, xv);
                ldv<NC>(e, i, ev);
#pragma unroll
                for (int c = 0; c < NC; ++c) xv[c] += (double)ev[c];
                stv<NC>(x, i, xv);
            }
        }
        cl.sync();
    }
    return false;
}

// BiCGStab with Jacobi for the two velocity components of one instance, on its cluster.  T:
// FP64, or FP32 for the inner solve of a refinement sweep (its per-thread partial sums are then
// FP32, the cluster sums FP64).  x starts from V.x, or from 0 with zero_x.  A breakdown (rho or
// omega vanishing before convergence) restarts from the true residual, at most `restarts`
// times.  Converged when <r, r> <= tol2 <b, b> for each component.  Returns the iterations;
// status, the last <r, r> and <b, b> go out.
template <class T>
__device__ __noinline__ int cluster_bicgstab(const SellView& A, const T* __restrict__ val, const T* __restrict__ dinv,
                                const T* __restrict__ b, const BicgVecsT<T>& V, double tol2, int maxit, int restarts,
                                bool zero_x, ClusterSync& cs, cgrp_bs::cluster_group& cl, int crank, int csize,
                                int& status, double (&rr)[2], double (&bb)[2]) {
    const int n = A.n, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int tid = crank * blockDim.x + threadIdx.x, nthr = csize * blockDim.x;
    // rows (vector passes) and slices (products) in flight per thread: the passes are bound by
    // latency, a thread walking 16 rows of a 66k-row instance one after the other
    constexpr int U = sizeof(T) == 4 ? 2 : 1, R = sizeof(T) == 4 ? 4 : 1, R2 = sizeof(T) == 4 ? 2 : 1;
    double rho[2] = {0.0, 0.0}, alpha[2] = {0.0, 0.0}, omega[2] = {0.0, 0.0}, beta[2] = {0.0, 0.0};
    int done[2] = {0, 0}, it = 0;
    status = 0;
    for (int restart = 0; restart <= restarts; ++restart) {
        {   // r = b - A x, rhat = r, p = v = 0
            const bool zx = zero_x && restart == 0;
            T acc[4] = {T(0), T(0), T(0), T(0)};
            for (int sl = crank * nwarp + wid; sl < A.nslices; sl += csize * nwarp) {
                const int i = sl * 32 + lane;
                T ax[2] = {T(0), T(0)};
                if (!zx) spmv2_row(A, val, V.x, sl, lane, ax);
                if (i < n) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const T bv = b[2 * i + c], rv = bv - ax[c];
                        if (zx) V.x[2 * i + c] = T(0);
                        V.r[2 * i + c] = rv;
                        V.rhat[2 * i + c] = rv;
                        V.p[2 * i + c] = T(0);
                        V.v[2 * i + c] = T(0);
                        acc[c] += rv * rv;
                        acc[2 + c] += bv * bv;
                    }
                }
            }
            const double accd[4] = {(double)acc[0], (double)acc[1], (double)acc[2], (double)acc[3]};
            double tot[4];
            cs.sum(accd, tot);
            for (int c = 0; c < 2; ++c) {
                rho[c] = tot[c];
                rr[c] = tot[c];
                if (restart == 0) bb[c] = tot[2 + c];
                done[c] = !(rr[c] > tol2 * bb[c]);
                alpha[c] = omega[c] = beta[c] = 0.0;
            }
        }
        bool broke = false;
        while (!(done[0] && done[1]) && it < maxit && !broke) {
            // p = r + beta (p - omega v), y = D^-1 p.  (Vectors of a component that is done
            // may hold anything from here on; only its x is kept.)
            for (int i0 = tid; i0 < n; i0 += R * nthr) {
                T rv[R][2], pv[R][2], vv[R][2], di[R];
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    const int i = i0 + q * nthr;
                    if (i < n) {
                        ldv<2>(V.r, i, rv[q]);
                        ldv<2>(V.p, i, pv[q]);
                        ldv<2>(V.v, i, vv[q]);
                        di[q] = dinv[i];
                    }
                }
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    const int i = i0 + q * nthr;
                    if (i < n) {
                        T yv[2];
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            pv[q][c] = rv[q][c] + (T)beta[c] * (pv[q][c] - (T)omega[c] * vv[q][c]);
                            yv[c] = di[q] * pv[q][c];
                        }
                        stv<2>(V.p, i, pv[q]);
                        stv<2>(V.y, i, yv);
                    }
                }
            }
            cl.sync();
            {   // v = A y, alpha = rho / <rhat, v>
                T acc[2] = {T(0), T(0)};
                for (int s0 = crank * nwarp + wid; s0 < A.nslices; s0 += U * csize * nwarp) {
                    int sl[U];
#pragma unroll
                    for (int q = 0; q < U; ++q) sl[q] = s0 + q * csize * nwarp;
                    T ax[U][2];
                    spmv_slices<U, 2>(A, val, V.y, sl, lane, ax);
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        const int i = sl[q] * 32 + lane;
                        if (i < n) {
                            T rh[2];
                            ldv<2>(V.rhat, i, rh);
                            stv<2>(V.v, i, ax[q]);
#pragma unroll
                            for (int c = 0; c < 2; ++c) acc[c] += rh[c] * ax[q][c];
                        }
                    }
                }
                const double accd[2] = {(double)acc[0], (double)acc[1]};
                double q[2];
                int flag;   // bit c: not finite, bit 2 + c: breakdown
                cs.sum_to(accd, q, flag, [&](const double (&t)[2], double (&o)[2]) -> int {
                    int f = 0;
                    for (int c = 0; c < 2; ++c) {
                        o[c] = rho[c] / t[c];
                        if (!isfinite(t[c])) f |= 1 << c;
                        else if (t[c] == 0.0) f |= 4 << c;
                    }
                    return f;
                });
                for (int c = 0; c < 2; ++c) {
                    if (done[c]) continue;
                    if (flag >> c & 1) {
                        done[c] = 1;
                        status = CGP_ENONFINITE;
                    } else if (flag >> (2 + c) & 1) {
                        broke = true;
                    } else {
                        alpha[c] = q[c];
                    }
                }
            }
            if (broke) break;
            // s = r - alpha v, z = D^-1 s
            for (int i0 = tid; i0 < n; i0 += R * nthr) {
                T rv[R][2], vv[R][2], di[R];
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    const int i = i0 + q * nthr;
                    if (i < n) {
                        ldv<2>(V.r, i, rv[q]);
                        ldv<2>(V.v, i, vv[q]);
                        di[q] = dinv[i];
                    }
                }
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    const int i = i0 + q * nthr;
                    if (i < n) {
                        T zv[2];
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            rv[q][c] -= (T)alpha[c] * vv[q][c];
                            zv[c] = di[q] * rv[q][c];
                        }
                        stv<2>(V.s, i, rv[q]);
                        stv<2>(V.z, i, zv);
                    }
                }
            }
            cl.sync();
            {   // t = A z, omega = <t, s> / <t, t>
                T acc[4] = {T(0), T(0), T(0), T(0)};
                for (int s0 = crank * nwarp + wid; s0 < A.nslices; s0 += U * csize * nwarp) {
                    int sl[U];
#pragma unroll
                    for (int q = 0; q < U; ++q) sl[q] = s0 + q * csize * nwarp;
                    T ax[U][2];
                    spmv_slices<U, 2>(A, val, V.z, sl, lane, ax);
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        const int i = sl[q] * 32 + lane;
                        if (i < n) {
                            T sv[2];
                            ldv<2>(V.s, i, sv);
                            stv<2>(V.t, i, ax[q]);
#pragma unroll
                            for (int c = 0; c < 2; ++c) {
                                acc[c] += ax[q][c] * sv[c];
                                acc[2 + c] += ax[q][c] * ax[q][c];
                            }
                        }
                    }
                }
                const double accd[4] = {(double)acc[0], (double)acc[1], (double)acc[2], (double)acc[3]};
                double q[2];
                int flag;
                cs.sum_to(accd, q, flag, [](const double (&t)[4], double (&o)[2]) -> int {
                    for (int c = 0; c < 2; ++c) o[c] = (t[2 + c] > 0.0 && isfinite(t[2 + c])) ? t[c] / t[2 + c] : 0.0;
                    return 0;
                });
                for (int c = 0; c < 2; ++c) omega[c] = done[c] ? 0.0 : q[c];
            }
            {   // x += alpha y + omega z, r = s - omega t, <rhat, r>, <r, r>
                T acc[4] = {T(0), T(0), T(0), T(0)};
                for (int i0 = tid; i0 < n; i0 += R2 * nthr) {
                    T xv[R2][2], yv[R2][2], zv[R2][2], sv[R2][2], tv[R2][2], rh[R2][2];
#pragma unroll
                    for (int q = 0; q < R2; ++q) {
                        const int i = i0 + q * nthr;
                        if (i < n) {
                            ldv<2>(V.x, i, xv[q]);
                            ldv<2>(V.y, i, yv[q]);
                            ldv<2>(V.z, i, zv[q]);
                            ldv<2>(V.s, i, sv[q]);
                            ldv<2>(V.t, i, tv[q]);
                            ldv<2>(V.rhat, i, rh[q]);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < R2; ++q) {
                        const int i = i0 + q * nthr;
                        if (i < n) {
#pragma unroll
                            for (int c = 0; c < 2; ++c) {
                                if (!done[c]) xv[q][c] += (T)alpha[c] * yv[q][c] + (T)omega[c] * zv[q][c];
                                sv[q][c] -= (T)omega[c] * tv[q][c];
                                acc[c] += rh[q][c] * sv[q][c];
                                acc[2 + c] += sv[q][c] * sv[q][c];
                            }
                            stv<2>(V.x, i, xv[q]);
                            stv<2>(V.r, i, sv[q]);
                        }
                    }
                }
                const double accd[4] = {(double)acc[0], (double)acc[1], (double)acc[2], (double)acc[3]};
                double q[6];   // <r, r>, the next rho, the next beta
                int flag;      // bit c: not finite, bit 2 + c: converged, bit 4 + c: breakdown
                cs.sum_to(accd, q, flag, [&](const double (&t)[4], double (&o)[6]) -> int {
                    int f = 0;
                    for (int c = 0; c < 2; ++c) {
                        o[c] = t[2 + c];
                        o[2 + c] = t[c];
                        o[4 + c] = (t[c] / rho[c]) * (alpha[c] / omega[c]);
                        if (!isfinite(t[c]) || !isfinite(t[2 + c])) f |= 1 << c;
                        else if (t[2 + c] <= tol2 * bb[c]) f |= 4 << c;
                        else if (omega[c] == 0.0 || t[c] == 0.0) f |= 16 << c;
                    }
                    return f;
                });
                for (int c = 0; c < 2; ++c) {
                    if (done[c]) continue;
                    if (flag >> c & 1) {
                        status = CGP_ENONFINITE;
                        done[c] = 1;
                        continue;
                    }
                    rr[c] = q[c];
                    if (flag >> (2 + c) & 1) {
                        done[c] = 1;
                    } else if (flag >> (4 + c) & 1) {
                        broke = true;
                    } else {
                        beta[c] = q[4 + c];
                        rho[c] = q[2 + c];
                    }
                }
            }
            ++it;
        }
        if (!broke) break;
        if (restart == restarts) status = CGP_EBREAKDOWN;
    }
    if (!(done[0] && done[1]) && !status) status = CGP_ENOTCONV;
    return it;
}

// (the phases are calls: inlined side by side they spilled 1.6 KB a thread)
static __device__ __noinline__ void coarse_pcg_call(const CoarsePcgArgs& a, ClusterSync& sy) { coarse_pcg_body(a, sy); }

static __global__ void __launch_bounds__(512, 1) k_batch_step(const BatchStepArgs* __restrict__ args, int ninst,
                                                              unsigned int* queue, int dyn_floats) {
    extern __shared__ float dyn[];   // the coarse CG's vectors (inner_cg_shared)
    __shared__ ClusterShared<512> sm;
    __shared__ int job;
    ClusterSync sy(sm, dyn_floats ? dyn : nullptr, dyn_floats);
    ClusterSync& cs = sy;
    cgrp_bs::cluster_group& cl = sy.cluster;
    const int crank = (int)cl.block_rank(), csize = (int)cl.num_blocks();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int tid = crank * blockDim.x + threadIdx.x, nthr = csize * blockDim.x;
    for (;;) {
        if (crank == 0 && threadIdx.x == 0) job = (int)atomicAdd(queue, 1u);
        cl.sync();
        const int jb = *cl.map_shared_rank(&job, 0);
        cl.sync();   // every CTA has read rank 0's job before it can change
        if (jb >= ninst) break;
        const BatchStepArgs& a = args[jb];
        const int nf = a.nf;
        const double dt = a.dt, tn = *a.tdev + dt;
        const BcParams bc = a.bc;
        // ---- Eq. 21: w = 2 U^n - U^{n-1}, h = dt F + 2 U^n - 1/2 U^{n-1}
        for (int i = tid; i < nf; i += nthr) {
            const double2 u = reinterpret_cast<const double2*>(a.U)[i];
            const double2 up = reinterpret_cast<const double2*>(a.Uprev)[i];
            double fx = 0.0, fy = 0.0;
            body_force(bc, i, a.xy[2 * i], a.xy[2 * i + 1], tn, fx, fy);
            reinterpret_cast<double2*>(a.w)[i] = make_double2(2.0 * u.x - up.x, 2.0 * u.y - up.y);
            reinterpret_cast<double2*>(a.h)[i] =
                make_double2(dt * fx + (2.0 * u.x - 0.5 * up.x), dt * fy + (2.0 * u.y - 0.5 * up.y));
        }
        cl.sync();
        for (int i = tid; i < nf; i += nthr)
            mom_assemble_row<false>(i, a.rowptr, a.col, a.sell_ptr, a.vt_ptr, a.vt_list, a.tri, a.geo, a.vtslot, a.S,
                                    a.M, a.CxT, a.CyT, a.P, a.w, a.h, a.tag, a.xy, bc, tn, dt, a.A, a.dinvA, a.b,
                                    a.Ut, nullptr);
        cl.sync();
        // ---- the momentum solve (two components), x = U~ from w.  Mixed instances: FP64
        // residual sweeps around an FP32 BiCGStab on the FP32 copy of A, then the FP64
        // BiCGStab unless a sweep's residual met the tolerance; FP64 instances: the FP64
        // BiCGStab alone (a breakdown restarts it from the true residual, at most 4 times).
        const BicgVecs V = a.bv;
        double rr[2] = {0.0, 0.0}, bb[2] = {0.0, 0.0};
        int it = 0, status = 0;
        bool polish = true;
        if (a.A32) {
            for (int64_t e = tid; e < a.nnz; e += nthr) a.A32[e] = (float)a.A[e];
            for (int i = tid; i < nf; i += nthr) a.dinvA32[i] = (float)a.dinvA[i];
            cl.sync();
            const BicgVecsT<float> W{a.fv[0], a.fv[1], a.fv[2], a.fv[3], a.fv[4], a.fv[5], a.fv[6], a.fv[7], a.fv[8]};
            float* r32 = a.fv[9];
            double far_last = INFINITY;
            for (int sw = 0; sw < kBatchIrSweeps; ++sw) {
                double acc[4] = {0.0, 0.0, 0.0, 0.0};
                for (int sl = crank * nwarp + wid; sl < a.Af.nslices; sl += csize * nwarp) {
                    const int i = sl * 32 + lane;
                    double ax[2];
                    spmv2_row(a.Af, a.A, V.x, sl, lane, ax);
                    if (i < nf) {
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const double bv = a.b[2 * i + c], rv = bv - ax[c];
                            r32[2 * i + c] = (float)rv;
                            acc[c] += rv * rv;
                            acc[2 + c] += bv * bv;
                        }
                    }
                }
                double tot[4];
                cs.sum(acc, tot);
                if (sw == 0) {
                    bb[0] = tot[2];
                    bb[1] = tot[3];
                }
                rr[0] = tot[0];
                rr[1] = tot[1];
                if (!isfinite(tot[0]) || !isfinite(tot[1])) break;   // the FP64 solve reports it
                if (rr[0] <= a.tol_mom2 * bb[0] && rr[1] <= a.tol_mom2 * bb[1]) {
                    polish = false;
                    break;
                }
                // a sweep that gained less than a decade is the last (components of one matrix:
                // the larger residual relative to its target decides)
                const double far = fmax(bb[0] > 0.0 ? rr[0] / bb[0] : 0.0, bb[1] > 0.0 ? rr[1] / bb[1] : 0.0);
                if (far > 0.01 * far_last) break;
                far_last = far;
                // the inner solve aims at kBatchInnerTol, or at what is left to the tolerance
                // (a factor 2 of margin in the norm) when that is less
                double t2 = kBatchInnerTol * kBatchInnerTol, need = 1.0;
                for (int c = 0; c < 2; ++c)
                    if (rr[c] > a.tol_mom2 * bb[c]) need = fmin(need, 0.25 * a.tol_mom2 * bb[c] / rr[c]);
                t2 = fmax(t2, need);
                int st_in = 0;
                double rr_in[2], bb_in[2];
                it += cluster_bicgstab<float>(a.Af, a.A32, a.dinvA32, r32, W, t2, kBatchInnerMaxit, 0, true, cs, cl,
                                              crank, csize, st_in, rr_in, bb_in);
                if (st_in == CGP_ENONFINITE) break;
                for (int i = tid; i < nf; i += nthr) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) V.x[2 * i + c] += (double)W.x[2 * i + c];
                }
                cl.sync();
            }
        }
        if (polish) {
            double bb64[2];
            it += cluster_bicgstab<double>(a.Af, a.A, a.dinvA, a.b, V, a.tol_mom2, a.max_it_mom, 4, false, cs, cl, crank,
                                           csize, status, rr, bb64);
            bb[0] = bb64[0];
            bb[1] = bb64[1];
        }
        // ---- Eqs. 22-23: r = -3/(2 dt) (Cx_c u~ + Cy_c v~) at the coarse vertices (the fine
        // prefix); phi data on PHI_ZERO vertices (zero, or lifted for a traction boundary)
        {
            const bool lift = has_natural_data(bc);
            double acc[1] = {0.0};
            for (int sl = crank * nwarp + wid; sl < a.Ac.nslices; sl += csize * nwarp) {
                const int i = sl * 32 + lane;
                double sx[1] = {0.0}, syv[1] = {0.0}, sk[1] = {0.0};
                sell_accum<1>(a.Ac, a.Cxc, sl, lane, [&](int j, double (&o)[1]) { o[0] = a.Ut[2 * j]; }, sx);
                sell_accum<1>(a.Ac, a.Cyc, sl, lane, [&](int j, double (&o)[1]) { o[0] = a.Ut[2 * j + 1]; }, syv);
                auto gN = [&](int j) { return natural_pressure(bc, a.cxy[2 * j], a.cxy[2 * j + 1], tn) - a.P[j]; };
                if (lift)
                    sell_accum<1>(a.Ac, a.Kc, sl, lane,
                                  [&](int j, double (&o)[1]) { o[0] = (a.ctag[j] & CGP_PHI_ZERO) ? gN(j) : 0.0; }, sk);
                if (i < a.Ac.n) {
                    double r;
                    if (a.ctag[i] & CGP_PHI_ZERO) r = lift ? gN(i) : 0.0;
                    else r = -1.5 / dt * (sx[0] + syv[0]) - sk[0];
                    a.coarse.b[i] = r;
                    acc[0] += r;
                }
            }
            double tot[1];
            cs.sum(acc, tot);
            if (crank == 0 && threadIdx.x == 0) a.ks[KS_POIS].mean = a.pure_neumann ? tot[0] / a.Ac.n : 0.0;
            cl.sync();
        }
        coarse_pcg_call(a.coarse, sy);   // ends with a cluster barrier
        // ---- Eq. 24: prolongation, one level after the other
        for (int l = 0; l + 1 < a.nlev; ++l) {
            const int nc_l = a.nv[l], n_new = a.nv[l + 1] - a.nv[l];
            const int2* pr = reinterpret_cast<const int2*>(a.parents[l]);
            for (int e = tid; e < n_new; e += nthr) {
                const int2 p2 = pr[e];
                a.phi[nc_l + e] = 0.5 * (a.phi[p2.x] + a.phi[p2.y]);
            }
            cl.sync();
        }
        // ---- Eq. 25: g = -2/3 dt (Cx phi, Cy phi) off the Dirichlet rows; the correction
        for (int sl = crank * nwarp + wid; sl < a.Af.nslices; sl += csize * nwarp) {
            const int i = sl * 32 + lane;
            double ax[1] = {0.0}, ay[1] = {0.0};
            sell_accum<1>(a.Af, a.Cx, sl, lane, [&](int j, double (&o)[1]) { o[0] = a.phi[j]; }, ax);
            sell_accum<1>(a.Af, a.Cy, sl, lane, [&](int j, double (&o)[1]) { o[0] = a.phi[j]; }, ay);
            if (i < nf) {
                const double c = -2.0 / 3.0 * dt;
                const double2 gv = (a.tag[i] & CGP_VEL_DIR) ? make_double2(0.0, 0.0) : make_double2(c * ax[0], c * ay[0]);
                reinterpret_cast<double2*>(a.g)[i] = gv;
                if (a.lumped) reinterpret_cast<double2*>(a.delta)[i] = make_double2(gv.x / a.mlumpF[i], gv.y / a.mlumpF[i]);
            }
        }
        cl.sync();
        int it_corr = 0, it_mass = 0;   // Chebyshev steps
        if (!a.lumped) {
            if (!(a.A32 && cluster_cheb_mixed<2>(a.Af, a.M0, a.M0f, a.dinvM0f, a.g, a.delta, a.fv[0], a.fv[1], a.fv[2],
                                                 a.fv[3], a.tol_mass2, cs, crank, csize, cl, it_corr))) {
                cluster_chebyshev<2>(a.Af, a.M0, a.dinvM0, a.g, a.delta, a.c0, a.c1, a.c2, a.cheb_steps, crank, csize,
                                     cl);
                it_corr += a.cheb_steps;
            }
        }
        // ---- Eq. 26: the rotational term q with M q = D U~ (or its lumped form)
        if (a.chi) {
            for (int sl = crank * nwarp + wid; sl < a.Af.nslices; sl += csize * nwarp) {
                const int i = sl * 32 + lane;
                double sx[1] = {0.0}, syv[1] = {0.0};
                sell_accum<1>(a.Af, a.Cx, sl, lane, [&](int j, double (&o)[1]) { o[0] = a.Ut[2 * j]; }, sx);
                sell_accum<1>(a.Af, a.Cy, sl, lane, [&](int j, double (&o)[1]) { o[0] = a.Ut[2 * j + 1]; }, syv);
                if (i < nf) {
                    const double s = sx[0] + syv[0];
                    a.div[i] = s;
                    if (a.lumped) a.qrot[i] = s / a.mlumpF[i];
                }
            }
            cl.sync();
            if (!a.lumped) {
                if (!(a.A32 && cluster_cheb_mixed<1>(a.Af, a.M, a.Mf, a.dinvMf, a.div, a.qrot, a.fv[0], a.fv[1], a.fv[2],
                                                     a.fv[3], a.tol_mass2, cs, crank, csize, cl, it_mass))) {
                    cluster_chebyshev<1>(a.Af, a.M, a.dinvM, a.div, a.qrot, a.c0, a.c1, a.c2, a.cheb_steps, crank, csize,
                                         cl);
                    it_mass += a.cheb_steps;
                }
            }
        }
        // ---- end of the step
        for (int i = tid; i < nf; i += nthr) {
            const double2 u = reinterpret_cast<const double2*>(a.U)[i];
            const double2 ut = reinterpret_cast<const double2*>(a.Ut)[i];
            const double2 d = reinterpret_cast<const double2*>(a.delta)[i];
            reinterpret_cast<double2*>(a.Uprev)[i] = u;
            reinterpret_cast<double2*>(a.U)[i] = make_double2(ut.x + d.x, ut.y + d.y);
            double p = a.P[i] + a.phi[i];
            if (a.chi) p -= a.inv_re * a.qrot[i];
            a.P[i] = p;
        }
        if (crank == 0 && threadIdx.x == 0) {
            *a.tdev = tn;
            KrylovState* ks = a.ks;
            ks[KS_MOM].iter = it;
            ks[KS_MOM].rr[0] = rr[0];
            ks[KS_MOM].rr[1] = rr[1];
            ks[KS_MOM].bb[0] = bb[0];
            ks[KS_MOM].bb[1] = bb[1];
            ks[KS_MOM].status = status;
            DeviceStats* st = a.stats;
            st->steps += 1;
            st->sum_outer += ks[KS_POIS].pad[0];
            const int its[KS_COUNT] = {it, ks[KS_POIS].iter, it_corr, it_mass};
            for (int k = 0; k < KS_COUNT; ++k) {
                st->last_it[k] = its[k];
                st->sum_it[k] += its[k];
            }
            st->res[KS_MOM] = fmax(bb[0] > 0.0 ? sqrt(rr[0] / bb[0]) : 0.0, bb[1] > 0.0 ? sqrt(rr[1] / bb[1]) : 0.0);
            st->res[KS_POIS] = ks[KS_POIS].bb[0] > 0.0 ? sqrt(ks[KS_POIS].rr[0] / ks[KS_POIS].bb[0]) : 0.0;
            if (!st->status && status) st->status = status;
            if (!st->status && ks[KS_POIS].status) st->status = ks[KS_POIS].status;
        }
        cl.sync();   // the instance's vectors are complete before the cluster takes the next one
    }
}

}  // namespace cgp
