// Memory-resident FP64 coarse solve over compact subdomains (Eq. 23), for systems that the
// register-resident solve (coarse_rr.cuh) cannot hold and whose level is the base mesh (the others
// are coarse_ml.cuh's): the same iteration, Chronopoulos and Gear's PCG with M^{-1} = D^{-1} +
// Z E^+ Z^T, with its vectors in global memory.
//
// The host plan (gp_plan in rr_plan.cuh) sorts the rows into compact subdomains of whole
// 32-row slices, kGridCtasPerSm CTAs each, and the solve runs on a copy of the matrix in that
// order: a CTA's rows lie in one subdomain, so its sum of w is one more column of the reduction,
// and the gathers of neighbouring rows share lines.  The solution and the right-hand side stay
// in the solver's order and are read and written through the permutation, a few times a solve.
// Per iteration: w = A u with the sums, one grid-wide reduction after which every CTA adds the
// partials of all subdomains and forms alpha, beta, s = Z^T r and its own mu = E^+ s, then the
// vector updates and a plain barrier (u complete before its gather).
//
// Bound by memory and by the FP64 pipe alike: about 110 bytes and 16 FP64 operations per row
// and iteration beside the matrix.  1,050,625 rows to 1e-10: 1,516 iterations of 54 us in 81 ms
// (Jacobi alone, rows in refinement order: about 4,650 of 50 us in 234 ms).
#pragma once

#include "coarse_pcg.cuh"
#include "rr_plan.cuh"

namespace cgp {

struct GpPlan {
    int nslots = 0, nslices = 0;     // rows with padding (whole slices), slices
    int nsub = 0, ctas = 0;          // 0: no plan
    const int32_t* perm = nullptr;   // slot -> row, or -1
    const int32_t* ptr = nullptr;    // the permuted matrix (SELL-32, columns are slots)
    const int32_t* col = nullptr;
    const double* val = nullptr;
    const double* dinv = nullptr;    // 1 / a_ii, negative for a row outside the coarse space, 0 padding
    const int32_t* first = nullptr;  // ctas + 1: first slice of every CTA
    const double* einv = nullptr;    // nsub x nsub
    double* vec = nullptr;           // 6 vectors of nslots: x, r, u, w, p, s
};

struct GpShared {
    double part[4][kGridThreads];
    double tot[3], out[4], mu;
    double zt[kRRMaxSub], zs[kRRMaxSub], zq[kRRMaxSub], einv[kRRMaxSub];
    int flag;
};

// the copy of the matrix in slot order, its diagonal's inverse (sign: outside the coarse space)
__global__ void k_gp_matrix(int nslots, const int32_t* __restrict__ perm, const int32_t* __restrict__ slot_of,
                            const int32_t* __restrict__ rowptr, const int32_t* __restrict__ sell_ptr,
                            const int32_t* __restrict__ sell_col, const double* __restrict__ val,
                            const double* __restrict__ dinv, const uint8_t* __restrict__ tag,
                            const int32_t* __restrict__ ptr, int32_t* __restrict__ pcol, double* __restrict__ pval,
                            double* __restrict__ pdinv) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nslots) return;
    const int i = perm[t], base = ptr[t >> 5] + (t & 31), w = (ptr[(t >> 5) + 1] - ptr[t >> 5]) >> 5;
    int len = 0, src = 0;
    double d = 0.0;
    if (i >= 0) {
        len = rowptr[i + 1] - rowptr[i];
        src = sell_ptr[i >> 5] + (i & 31);
        d = (tag[i] & CGP_PHI_ZERO) ? -dinv[i] : dinv[i];
    }
    pdinv[t] = d;
    for (int k = 0; k < w; ++k) {
        pcol[base + 32 * k] = k < len ? slot_of[sell_col[src + 32 * k]] : t;
        pval[base + 32 * k] = k < len ? val[src + 32 * k] : 0.0;
    }
}

struct GpSync : GridSync {
    GpShared& g;
    const GpPlan& pl;
    int sub, per;   // this CTA's subdomain; CTAs per subdomain
    __device__ GpSync(unsigned* c, int* e, double* p, GridShared& s, GpShared& gs, const GpPlan& plan, int wait_test)
        : GridSync(c, e, p, s, wait_test), g(gs), pl(plan) {
        per = (int)gridDim.x / plan.nsub;
        sub = (int)blockIdx.x / per;
    }
    // Grid-wide sums of v[0..2] handed to f (warp 0 of every CTA) and the subdomains' sums of
    // v[3]: start takes them as s, otherwise s -= out[0] (sums + out[1] zq).  mu: this
    // subdomain's entry of E^+ s.
    template <class F>
    __device__ bool reduce(const double (&v)[4], bool start, double (&out)[4], int& flag, double& mu, F f) {
        const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, G = (int)gridDim.x;
#pragma unroll
        for (int k = 0; k < 4; ++k) g.part[k][tid] = v[k];
        __syncthreads();
        double* mine = partials + (size_t)slot * 4 * G;
        if (wid < 4) {
            const double s = column_sum(g.part[wid]);
            if (lane == 0) __stcg(mine + (size_t)wid * G + blockIdx.x, s);
        }
        if (!sync()) return false;
        if (wid < 3) {
            double s = 0.0;
            for (int b0 = lane; b0 < G; b0 += 32 * 8) {
                double q[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) q[j] = b0 + 32 * j < G ? __ldcg(mine + (size_t)wid * G + b0 + 32 * j) : 0.0;
                s += ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) g.tot[wid] = s;
        } else {
            // warps 3 .. 7: a thread per subdomain
            for (int j = tid - 96; j < pl.nsub; j += kGridThreads - 96) {
                double s = 0.0;
                for (int c = 0; c < per; ++c) s += __ldcg(mine + (size_t)3 * G + j * per + c);
                g.zt[j] = s;
            }
        }
        __syncthreads();
        if (wid == 0) {
            const double t[3] = {g.tot[0], g.tot[1], g.tot[2]};
            double o[4] = {0.0, 0.0, 0.0, 0.0};
            const int fl = f(t, o);
            double m = 0.0;
            for (int j = lane; j < pl.nsub; j += 32) {
                double q = 0.0, s = g.zt[j];
                if (!start) {
                    q = fma(o[1], g.zq[j], s);
                    s = fma(-o[0], q, g.zs[j]);
                }
                g.zq[j] = q;
                g.zs[j] = s;
                m = fma(g.einv[j], s, m);
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) m += __shfl_xor_sync(0xffffffffu, m, d);
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < 4; ++k) g.out[k] = o[k];
                g.mu = m;
                g.flag = fl;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k] = g.out[k];
        flag = g.flag;
        mu = g.mu;
        slot ^= 1;
        return true;
    }
};

static __global__ void __launch_bounds__(kGridThreads, kGridCtasPerSm) k_pcg_grid_plan(CoarsePcgArgs a, GpPlan pl) {
    __shared__ GridShared gsm;
    __shared__ GpShared sm;
    GpSync sy(a.bar_count, a.bar_err, a.partials, gsm, sm, pl, a.wait_test);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = kGridThreads / 32;
    for (int j = threadIdx.x; j < pl.nsub; j += kGridThreads) sm.einv[j] = __ldg(pl.einv + (size_t)sy.sub * pl.nsub + j);
    const SellView A{pl.nslots, pl.nslices, pl.ptr, pl.col};
    const int s_begin = __ldg(pl.first + blockIdx.x), s_end = __ldg(pl.first + blockIdx.x + 1);
    const size_t n = (size_t)pl.nslots;
    double *x = pl.vec, *r = x + n, *u = r + n, *w = u + n, *p = w + n, *s = p + n;
    const double mean = a.project ? a.st->mean : 0.0;
    for (int sl = s_begin + wid; sl < s_end; sl += nw) {
        const int t = sl * 32 + lane, i = __ldg(pl.perm + t);
        if (i >= 0 && a.project) a.b[i] -= mean;
        __stcg(x + t, i >= 0 && !a.zero_x ? a.x[i] : 0.0);
    }
    int iters = 0, status = sy.sync() ? 0 : CGP_ETIMEOUT, outer = 0;
    double bb = 0.0, rr_final = 0.0;
    bool converged = false;
    auto plain = [](const double (&t)[3], double (&q)[4]) -> int {
        q[0] = t[0];
        q[1] = t[1];
        return 0;
    };
    while (status == 0) {
        // ---- outer: r = b - A x, then u = M^{-1} r
        double v[4] = {0.0, 0.0, 0.0, 0.0}, o[4], mu;
        int flag;
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int t = sl * 32 + lane, i = __ldg(pl.perm + t);
            double ax[1] = {0.0};
            if (!(a.zero_x && outer == 0))
                sell_accum<1>(A, pl.val, sl, lane, [&](int j, double (&g)[1]) { g[0] = ldcg(x + j); }, ax);
            const double bi = i >= 0 ? a.b[i] : 0.0, ri = bi - ax[0];
            __stcg(r + t, ri);
            v[0] += ri * ri;
            v[1] += bi * bi;
            if (__ldg(pl.dinv + t) > 0.0) v[3] += ri;
        }
        if (!sy.reduce(v, true, o, flag, mu, plain)) {
            status = CGP_ETIMEOUT;
            break;
        }
        if (outer == 0) bb = o[1];
        rr_final = o[0];
        if (!isfinite(o[0])) {
            status = CGP_ENONFINITE;
            break;
        }
        if (o[0] <= a.tol2 * bb) {
            converged = true;
            break;
        }
        if (outer >= a.max_outer || iters >= a.maxit) {
            status = CGP_ENOTCONV;
            break;
        }
        // the sums of <r, u> and <r, r> of the coming reduction, from the pass that makes u
        v[0] = v[2] = 0.0;
        auto make_u = [&](int t, double ri) {
            const double d = __ldg(pl.dinv + t), ui = fma(fabs(d), ri, d > 0.0 ? mu : 0.0);
            __stcg(u + t, ui);
            v[0] += ri * ui;
            v[2] += ri * ri;
        };
        for (int sl = s_begin + wid; sl < s_end; sl += nw) make_u(sl * 32 + lane, ldcg(r + sl * 32 + lane));
        if (!sy.sync()) {
            status = CGP_ETIMEOUT;
            break;
        }
        const double stop2 = 0.25 * a.tol2 * bb;
        double gamma = 0.0, d = 0.0, rr_best = INFINITY;
        int best_k = 0, leave = 0;
        for (int k = 0;; ++k) {
            v[1] = v[3] = 0.0;
            for (int sl = s_begin + wid; sl < s_end; sl += nw) {
                const int t = sl * 32 + lane;
                const double wv = row_spmv<double>(A, pl.val, nullptr, sl, lane, [&](int j) { return ldcg(u + j); });
                __stcg(w + t, wv);
                v[1] += wv * ldcg(u + t);
                if (__ldg(pl.dinv + t) > 0.0) v[3] += wv;
            }
            // out: alpha, beta, gamma, d; flag as in inner_pcg
            if (!sy.reduce(v, false, o, flag, mu, [&](const double (&t)[3], double (&q)[4]) -> int {
                    const double tg = t[0], trr = t[2];
                    const double beta = k ? tg / gamma : 0.0;
                    q[3] = k ? t[1] - beta * beta * d : t[1];
                    q[2] = tg;
                    q[1] = beta;
                    q[0] = tg / q[3];
                    if (k && !(isfinite(tg) && isfinite(t[1]) && isfinite(trr))) return 3;
                    if (k && (tg == 0.0 || trr <= stop2)) return 1;
                    if (trr < 0.5 * rr_best) {
                        rr_best = trr;
                        best_k = k;
                    }
                    if (!isfinite(q[0]) || q[0] == 0.0) return 2;
                    return k - best_k > stagnation_window(k, rr_best <= 1e4 * stop2) || iters >= a.maxit ? 1 : 0;
                })) {
                status = CGP_ETIMEOUT;
                break;
            }
            if (flag) {
                leave = flag;
                break;
            }
            gamma = o[2];
            d = o[3];
            v[0] = v[2] = 0.0;
            for (int sl = s_begin + wid; sl < s_end; sl += nw) {
                const int t = sl * 32 + lane;
                double p_i = ldcg(u + t), s_i = ldcg(w + t);
                if (k) {
                    p_i = fma(o[1], ldcg(p + t), p_i);
                    s_i = fma(o[1], ldcg(s + t), s_i);
                }
                const double r_i = fma(-o[0], s_i, ldcg(r + t));
                __stcg(p + t, p_i);
                __stcg(s + t, s_i);
                __stcg(x + t, fma(o[0], p_i, ldcg(x + t)));
                __stcg(r + t, r_i);
                make_u(t, r_i);
            }
            ++iters;
            if (!sy.sync()) {   // u is complete before it is gathered
                status = CGP_ETIMEOUT;
                break;
            }
        }
        if (status) break;
        if (leave == 3) {
            status = CGP_ENONFINITE;
            break;
        }
        ++outer;   // (x was complete at the barrier before the last gather)
    }
    // ---- pure-Neumann mean fix, and x back in the solver's order
    double shift = 0.0;
    if (a.mlump && status != CGP_ETIMEOUT) {
        double acc[2] = {0.0, 0.0}, tot[2];
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int t = sl * 32 + lane, i = __ldg(pl.perm + t);
            if (i >= 0) {
                acc[0] += __ldg(a.mlump + i) * ldcg(x + t);
                acc[1] += __ldg(a.mlump + i);
            }
        }
        if (sy.sum(acc, tot)) shift = tot[0] / tot[1];
        else status = CGP_ETIMEOUT;
    }
    for (int sl = s_begin + wid; sl < s_end; sl += nw) {
        const int t = sl * 32 + lane, i = __ldg(pl.perm + t);
        if (i >= 0) a.x[i] = ldcg(x + t) - shift;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        KrylovState* st = a.st;
        st->iter = iters;
        st->bb[0] = bb;
        st->rr[0] = rr_final;
        st->bb[1] = 0.0;
        st->rr[1] = 0.0;
        st->status = status ? status : (converged ? 0 : CGP_ENOTCONV);
        st->done = 1;
        st->pad[0] = outer;
        st->pad[1] = 0;
    }
}

}  // namespace cgp
