// FP64 coarse solve of a small system with the inverse of its matrix (Eq. 23): iterative
// refinement x += K^+ (b - A x) in one cooperative launch, K^+ made once at assembly
// (k_ml_inverse in coarse_ml.cuh).
//
// At most kDirectMaxRows rows, so K^+ (20 MB at that size) stays in L2.  A sweep: the residual and
// its norm, a slice per CTA; a grid barrier; every CTA adds the slices' sums and decides alike; a
// warp per row of K^+ r; a grid barrier.  The residual falls by about 1e12 a sweep, so two true
// residuals and one product are usual: bound by the launch, the barriers and one pass over K^+.
// Measured (GB300), cgp_poisson_solve to 1e-10: 80 us for 1,089 rows, 89 for 1,600, of which the
// call's copies and its synchronisation take most (169 rows: 76); register-resident PCG of 1,681
// rows 750.  Cavity 64^2 in FP64 (4 steps): 4.48 -> 2.39 ms.
#pragma once

#include "coarse_ml.cuh"

namespace cgp {

constexpr int kDirectThreads = 512;

struct DirectShared {
    double r[kDirectMaxRows];
    double part[kDirectThreads / 32][2];
    double tot[2];
};

// e = K0 (+ shift everywhere) as a dense matrix that was zeroed; a thread per row
__global__ void k_direct_dense(SellView A, const double* __restrict__ val, const int32_t* __restrict__ rowptr, double shift,
                               double* __restrict__ e) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.n) return;
    double* row = e + (size_t)i * A.n;
    if (shift != 0.0)
        for (int j = 0; j < A.n; ++j) row[j] = shift;
    const int base = A.ptr[i >> 5] + (i & 31), len = rowptr[i + 1] - rowptr[i];
    for (int k = 0; k < len; ++k) row[A.col[base + 32 * k]] += val[base + 32 * k];
}

static __global__ void __launch_bounds__(kDirectThreads, 1) k_direct_solve(CoarsePcgArgs a, const double* __restrict__ inv) {
    __shared__ DirectShared sm;
    GridBarrier bar(a.bar_count, a.bar_err, a.wait_test);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = kDirectThreads / 32;
    const int G = (int)gridDim.x, cta = (int)blockIdx.x;
    const SellView& A = a.A;
    const int n = A.n, ns = A.nslices;
    double *x = a.x, *r = a.w64;
    const double mean = a.project ? a.st->mean : 0.0;
    int iters = 0, status = 0;
    double bb = 0.0, rr = 0.0;
    bool converged = false;
    for (;;) {
        // ---- r = b - A x: slice s on warp 0 of CTA s mod G
        double* part = a.partials + (size_t)(iters & 1) * 2 * ns;
        if (wid == 0)
            for (int s = cta; s < ns; s += G) {
                const int i = 32 * s + lane;
                double ax[1] = {0.0}, bi = 0.0, ri = 0.0;
                const bool zero = a.zero_x && iters == 0;
                if (!zero) sell_accum<1>(A, a.val, s, lane, [&](int j, double (&g)[1]) { g[0] = ldcg(x + j); }, ax);
                if (i < n) {
                    bi = a.b[i];
                    if (a.project && iters == 0) a.b[i] = bi -= mean;
                    ri = bi - ax[0];
                    __stcg(r + i, ri);
                }
                const double v[2] = {ri * ri, bi * bi};
                warp_sums_to(v, &sm.tot[0]);
                __syncwarp();
                if (lane < 2) __stcg(part + 2 * s + lane, sm.tot[lane]);
                __syncwarp();
            }
        if (!bar.sync()) {
            status = CGP_ETIMEOUT;
            break;
        }
        for (int j = tid; j < n; j += kDirectThreads) sm.r[j] = ldcg(r + j);
        if (wid < 2) {
            double s = 0.0;
            for (int k = lane; k < ns; k += 32) s += ldcg(part + 2 * k + wid);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) sm.part[0][wid] = s;
        }
        __syncthreads();
        rr = sm.part[0][0];
        if (iters == 0) bb = sm.part[0][1];
        if (!isfinite(rr) || !isfinite(bb)) {
            status = CGP_ENONFINITE;
            break;
        }
        if (rr <= a.tol2 * bb) {
            converged = true;
            break;
        }
        if (iters >= a.max_outer || iters >= a.maxit) break;
        // ---- x += K^+ r: row i on a warp of CTA i mod G
        for (int i = wid * G + cta; i < n; i += nw * G) {
            const double* row = inv + (size_t)i * n;
            double q[4] = {0.0, 0.0, 0.0, 0.0};
            for (int j0 = lane; j0 < n; j0 += 32 * 16) {
                double c[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) c[k] = j0 + 32 * k < n ? __ldg(row + j0 + 32 * k) : 0.0;
#pragma unroll
                for (int k = 0; k < 16; ++k)
                    if (j0 + 32 * k < n) q[k & 3] = fma(c[k], sm.r[j0 + 32 * k], q[k & 3]);
            }
            double s = (q[0] + q[1]) + (q[2] + q[3]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) __stcg(x + i, a.zero_x && iters == 0 ? s : ldcg(x + i) + s);
        }
        ++iters;
        if (!bar.sync()) {
            status = CGP_ETIMEOUT;
            break;
        }
    }
    if (cta != 0) return;
    if (iters == 0 && a.zero_x)
        for (int i = tid; i < n; i += kDirectThreads) x[i] = 0.0;
    // ---- pure-Neumann mean fix, by one CTA (x is complete)
    if (a.mlump && status != CGP_ETIMEOUT) {
        __syncthreads();
        double v[2] = {0.0, 0.0};
        for (int i = tid; i < n; i += kDirectThreads) {
            const double m = __ldg(a.mlump + i);
            v[0] += m * ldcg(x + i);
            v[1] += m;
        }
        warp_sums_to(v, sm.part[wid]);
        __syncthreads();
        double t0 = 0.0, t1 = 0.0;
        for (int k = 0; k < nw; ++k) {
            t0 += sm.part[k][0];
            t1 += sm.part[k][1];
        }
        const double shift = t0 / t1;
        for (int i = tid; i < n; i += kDirectThreads) x[i] = ldcg(x + i) - shift;
    }
    if (tid == 0) {
        KrylovState* st = a.st;
        st->iter = iters;
        st->bb[0] = bb;
        st->rr[0] = rr;
        st->bb[1] = 0.0;
        st->rr[1] = 0.0;
        st->status = status ? status : (converged ? 0 : CGP_ENOTCONV);
        st->done = 1;
        st->pad[0] = iters;
        st->pad[1] = 0;
    }
}

}  // namespace cgp
