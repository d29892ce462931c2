// Memory-resident FP64 coarse solve with an additive multilevel preconditioner (Eq. 23) over the
// coarse level and the mesh levels below it, if any.
//
// Chronopoulos and Gear's PCG as in coarse_pcg.cuh, with the preconditioner of Bramble, Pasciak
// and Xu (Math. Comp. 55, 1990) over the nested levels 0 .. L (L: the coarse level):
//     M^{-1} = sum_l P_l D_l^{-1} P_l^T + P_0 Z E^+ Z^T P_0^T,
// P_l the linear interpolation from level l to L, D_l the diagonal of level l's stiffness matrix,
// Z the indicator vectors of up to kMlMaxSub compact subdomains of the base mesh's vertices and
// E = Z^T K_0 Z (phi = 0 vertices are in no P_l and in no subdomain).  All in FP64.
//
// The vertices of a level are the first ones of the next, a new vertex is the midpoint of its two
// parents, and after a refinement every neighbour of an old vertex is a midpoint on one of its
// edges.  So the restriction of row i is r_i plus half the sum over i's neighbours, read from the
// pattern of the upper level, and the prolongation a copy or a mean of two: no stored P.
//
// An iteration: w = A u with <w, u>; w's restrictions, level by level, and on the base mesh the
// subdomains' sums (a CTA or a warp each); the reduction; x, r, p, s and, by the recurrence of r
// itself, the restricted residuals of all levels, mu = E^+ Z^T P_0^T r and z on the base mesh; u from
// the prolonged z, with <r, u> and <r, r>.  L + 3 grid barriers (one more with z stored).
//
// One CTA per SM (152 arrivals at a barrier: 1.7 us; with four per SM 5.5), E^+ in shared memory.
// Small levels are bound by the barriers and by chains of FP64 operations (about 100 clocks each,
// also between the shuffles of a sum), large ones by the FP64 pipe and the gathers.  Measured
// (GB300), to 1e-10, against the same solve with subdomains alone:
//        rows  levels below   iterations       us an iteration     ms
//      16,641  2               52  (272)       20  (9.2)           1.04  (2.51)
//      32,489  1, channel      88  (279)       19  (10.9)          1.70  (3.03)
//      66,049  2               74  (403)       23  (10.8)          1.71  (4.35)
//     491,401  2              152  (1,034)     55  (30)            8.3   (31)
//   1,050,625  3              127  (1,516)    100  (54)           12.8   (81)
//      16,641  none            96  (242)       14  (8.8)           1.38  (2.12)
//     263,169  none           347  (669)       33  (23)           11.3   (15.3)
// (in brackets up to 66,049 rows the register-resident solve, beyond a memory-resident one on rows
// sorted into 152 subdomains.)  Without a level below, M^{-1} = D^{-1} + Z E^+ Z^T on the level itself.
#pragma once

#include "coarse_pcg.cuh"
#include "rr_plan.cuh"

namespace cgp {

// 1 / diagonal of a level's stiffness matrix: the sum over a vertex's triangles of
// |opposite edge|^2 / (4 area)
__global__ void k_ml_diag(int n, const double* __restrict__ xy, const int32_t* __restrict__ tri,
                          const int32_t* __restrict__ vt_ptr, const int32_t* __restrict__ vt_list,
                          const uint8_t* __restrict__ tag, double* __restrict__ dinv) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double d = 0.0;
    for (int q = vt_ptr[i]; q < vt_ptr[i + 1]; ++q) {
        const int32_t* v = tri + 3 * (size_t)vt_list[q];
        const int a = v[0] == i ? v[1] : v[0], b = v[2] == i ? v[1] : v[2];
        const double xi = xy[2 * (size_t)i], yi = xy[2 * (size_t)i + 1];
        const double ax = xy[2 * (size_t)a] - xi, ay = xy[2 * (size_t)a + 1] - yi;
        const double bx = xy[2 * (size_t)b] - xi, by = xy[2 * (size_t)b + 1] - yi;
        const double ex = ax - bx, ey = ay - by;
        d += (ex * ex + ey * ey) / (2.0 * fabs(ax * by - ay * bx));
    }
    dinv[i] = (tag[i] & CGP_PHI_ZERO) || !(d > 0.0) ? 0.0 : 1.0 / d;
}

// In place, the inverse of the symmetric positive definite m x m matrix e by Gauss and Jordan's
// elimination without pivoting, a cooperative launch of one CTA per SM that holds its rows (every
// G-th) in shared memory; the owner of a pivot row hands it on through `row` (2 x m), one grid
// barrier a step.  *bad: a pivot is not safely positive, or a wait ran out.
constexpr int kInverseThreads = 512, kInverseRows = 32;   // rows of a CTA at most
__global__ void __launch_bounds__(kInverseThreads) k_ml_inverse(int m, double* __restrict__ e, double* __restrict__ row,
                                                    unsigned* count, int* err, int* bad) {
    extern __shared__ double mine[];
    GridBarrier bar(count, err, 0);
    const int G = (int)gridDim.x, cta = (int)blockIdx.x, own = cta < m ? (m - cta + G - 1) / G : 0;
    __shared__ double diag, f[kInverseRows];
    for (int q = 0; q < own; ++q)
        for (int j = threadIdx.x; j < m; j += blockDim.x) mine[(size_t)q * m + j] = e[(size_t)(cta + q * G) * m + j];
    __syncthreads();
    for (int p = 0; p < m; ++p) {
        double* pass = row + (size_t)(p & 1) * m;
        if (p % G == cta) {
            double* r = mine + (size_t)(p / G) * m;
            if (threadIdx.x == 0) {
                if (!(r[p] > 1e-10 * e[(size_t)p * m + p])) *bad = 1;
                diag = 1.0 / r[p];
                r[p] = 1.0;
            }
            __syncthreads();
            for (int j = threadIdx.x; j < m; j += blockDim.x) {
                const double v = r[j] * diag;
                r[j] = v;
                __stcg(pass + j, v);
            }
        }
        if (!bar.sync()) {
            if (threadIdx.x == 0) *bad = 1;
            return;
        }
        // column p of the other rows, then their update, each entry of the pivot row read once
        if (threadIdx.x < own) f[threadIdx.x] = cta + threadIdx.x * G == p ? 0.0 : mine[(size_t)threadIdx.x * m + p];
        __syncthreads();
        for (int j = threadIdx.x; j < m; j += blockDim.x) {
            const double v = __ldcg(pass + j);
            for (int q = 0; q < own; ++q) {
                double& r = mine[(size_t)q * m + j];
                if (j != p) r = fma(-f[q], v, r);
                else if (cta + q * G != p) r = -f[q] * v;
            }
        }
        __syncthreads();
    }
    for (int q = 0; q < own; ++q)
        for (int j = threadIdx.x; j < m; j += blockDim.x) e[(size_t)(cta + q * G) * m + j] = mine[(size_t)q * m + j];
}
// symmetric again (e is the inverse to rounding), and the constants taken out
__global__ void k_ml_symmetric(int m, double* __restrict__ e, double shift) {
    const int j = blockIdx.x, k0 = threadIdx.x;
    for (int k = k0; k <= j; k += blockDim.x) {
        const double v = 0.5 * (e[(size_t)j * m + k] + e[(size_t)k * m + j]) - shift;
        e[(size_t)j * m + k] = e[(size_t)k * m + j] = v;
    }
}

constexpr int kMlThreads = 1024;   // most threads per CTA (one CTA per SM)
constexpr int kMlPerCta = 4;       // most subdomains per CTA

struct MlShared {
    double part[3][kMlThreads];
    double tot[3], out[4], group[kMlThreads / 32];
    int flag;
};
// dynamic shared memory: the CTA's rows of E^+
inline size_t ml_shared_bytes(int nsub) { return sizeof(double) * kMlPerCta * (size_t)nsub; }

// the sum of a group's values, in every thread of it: a warp, or 8 warps on a named barrier
__device__ __forceinline__ double ml_group_sum(MlShared& sm, int gs, double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (gs == 32) return v;
    const int wid = threadIdx.x >> 5, w0 = wid & ~7, id = 1 + (wid >> 3);
    asm volatile("bar.sync %0, 256;" ::"r"(id) : "memory");   // the last sum has been read
    if ((threadIdx.x & 31) == 0) sm.group[wid] = v;
    asm volatile("bar.sync %0, 256;" ::"r"(id) : "memory");
    v = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) v += sm.group[w0 + k];
    return v;
}

struct MlSync : GridBarrier {
    MlShared& sm;
    const MlPlan& pl;
    double* partials;
    const double* einv;   // this group's row of E^+
    int gs, gt, slot = 0;
    bool has;             // this group has a subdomain
    __device__ MlSync(const CoarsePcgArgs& a, MlShared& s, const MlPlan& p) : GridBarrier(a.bar_count, a.bar_err, a.wait_test), sm(s), pl(p), partials(a.partials) {}

    // Grid-wide sums of v[0..2], handed to f on warp 0, whose out[] and flag every thread gets;
    // t: this group's entry of E^+ times the subdomains' sums (complete at the same barrier).
    template <class F>
    __device__ bool reduce(const double (&v)[3], double (&out)[4], int& flag, double& t, F f) {
        const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, G = (int)gridDim.x;
#pragma unroll
        for (int k = 0; k < 3; ++k) sm.part[k][tid] = v[k];
        __syncthreads();
        double* mine = partials + ((size_t)slot * 3 + wid) * G;
        if (wid < 3) {
            const double s = column_sum(sm.part[wid]);
            if (lane == 0) __stcg(mine + blockIdx.x, s);
        }
        if (!sync()) return false;
        t = 0.0;
        if (has) {
            // four chains, their loads in flight together
            double q[4] = {0.0, 0.0, 0.0, 0.0};
            for (int j0 = gt; j0 < pl.nsub; j0 += 8 * gs) {
                double z[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) z[k] = j0 + k * gs < pl.nsub ? ldcg(pl.zs + j0 + k * gs) : 0.0;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (j0 + k * gs < pl.nsub) q[k & 3] = fma(einv[j0 + k * gs], z[k], q[k & 3]);
            }
            t = ml_group_sum(sm, gs, (q[0] + q[1]) + (q[2] + q[3]));
        }
        if (wid < 3) {
            double s = 0.0;
            for (int b0 = lane; b0 < G; b0 += 32 * 8) {
                double q[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) q[j] = b0 + 32 * j < G ? __ldcg(mine + b0 + 32 * j) : 0.0;
                s += ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) sm.tot[wid] = s;
        }
        __syncthreads();
        if (wid == 0) {
            const double tot[3] = {sm.tot[0], sm.tot[1], sm.tot[2]};
            double o[4] = {0.0, 0.0, 0.0, 0.0};
            const int fl = f(tot, o);
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < 4; ++k) sm.out[k] = o[k];
                sm.flag = fl;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k] = sm.out[k];
        flag = sm.flag;
        slot ^= 1;
        return true;
    }
};

// restriction of `from` (level above) to row i
__device__ __forceinline__ double ml_restrict(const MlLevel& v, const double* from, int i) {
    const int base = __ldg(v.ptr + (i >> 5)) + (i & 31), len = __ldg(v.rowptr + i + 1) - __ldg(v.rowptr + i);
    double s = ldcg(from + i);
    for (int k0 = 0; k0 < len; k0 += 8) {
        int c[8];
        double g[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) c[k] = k0 + k < len ? __ldg(v.col + base + 32 * (k0 + k)) : -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) g[k] = c[k] >= 0 ? ldcg(from + c[k]) : 0.0;
        s += ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7]));
    }
    return 0.5 * s;   // (the row holds i itself too)
}

// z of vertex i of level L, all levels up to it: stored on the base mesh, formed from the residuals
// on the others
template <int L>
__device__ __forceinline__ double ml_z(const MlPlan& pl, int i) {
    if constexpr (L == 0) {
        return ldcg(pl.lev[0].z + i);
    } else {
        const MlLevel &v = pl.lev[L], &b = pl.lev[L - 1];
        const double own = __ldg(v.dinv + i) * ldcg(v.rs + i);
        if (i < b.n) return own + ml_z<L - 1>(pl, i);
        const int2 e = __ldg(b.parents + (i - b.n));
        return fma(0.5, ml_z<L - 1>(pl, e.x) + ml_z<L - 1>(pl, e.y), own);
    }
}
// prolongation of level L's z to vertex i of the level above
template <int L>
__device__ __forceinline__ double ml_prolong(const MlPlan& pl, int i) {
    const MlLevel& v = pl.lev[L];
    if (i < v.n) return ml_z<L>(pl, i);
    const int2 e = __ldg(v.parents + (i - v.n));
    return 0.5 * (ml_z<L>(pl, e.x) + ml_z<L>(pl, e.y));
}
// the same where level L's z is stored
__device__ __forceinline__ double ml_prolong_stored(const MlLevel& v, int i) {
    if (i < v.n) return ldcg(v.z + i);
    const int2 e = __ldg(v.parents + (i - v.n));
    return 0.5 * (ldcg(v.z + e.x) + ldcg(v.z + e.y));
}

// kT: most threads per CTA of the instance (512: 128 registers a thread, no spills)
template <int kT>
static __global__ void __launch_bounds__(kT, 1) k_pcg_grid_ml(CoarsePcgArgs a, MlPlan pl) {
    __shared__ MlShared sm;
    extern __shared__ double ml_dyn[];
    MlSync sy(a, sm, pl);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    const int G = (int)gridDim.x, cta = (int)blockIdx.x;
    const SellView& A = a.A;
    const int s_begin = (int)((int64_t)A.nslices * cta / G), s_end = (int)((int64_t)A.nslices * (cta + 1) / G);
    const size_t n = (size_t)A.n;
    double *x = a.x, *r = a.w64, *u = r + n, *w = u + n, *p = w + n, *s = p + n;
    const int top = pl.levels - 1;   // the level below the coarse one
    const bool flat = top < 0;       // the coarse level is the base mesh: M^{-1} = D^{-1} + Z E^+ Z^T
    // this group's subdomain of the base mesh; kMlPerCta groups of a CTA have one each (as warps,
    // those after the ones that add up the sums)
    const int gs = pl.group, gt = tid & (gs - 1), gi = gs == 32 ? wid - 4 : tid / gs;
    const int sub = gi >= 0 && gi < kMlPerCta ? gi * G + cta : pl.nsub;
    const bool has = sub < pl.nsub;
    int k0 = 0, k1 = 0;
    if (has) {
        k0 = __ldg(pl.first + sub);
        k1 = __ldg(pl.first + sub + 1);
        double* row = ml_dyn + (size_t)gi * pl.nsub;
        for (int j = gt; j < pl.nsub; j += gs) row[j] = __ldg(pl.einv + (size_t)sub * pl.nsub + j);
    }
    sy.gs = gs;
    sy.gt = gt;
    sy.has = has;
    sy.einv = ml_dyn + (size_t)(has ? gi : 0) * pl.nsub;
    const double mean = a.project ? a.st->mean : 0.0;
    int iters = 0, status = 0, outer = 0;
    double bb = 0.0, rr_final = 0.0, v[3] = {0.0, 0.0, 0.0};
    bool converged = false;
    for (int sl = s_begin + wid; sl < s_end; sl += nw) {
        const int i = sl * 32 + lane;
        if (i >= A.n) continue;
        if (a.project) a.b[i] -= mean;
        // a row with phi = 0 is the identity's: solved at once, its residual stays zero
        if (__ldg(pl.tag + i) & CGP_PHI_ZERO) __stcg(x + i, a.b[i]);
        else if (a.zero_x) __stcg(x + i, 0.0);
    }
    if (!sy.sync()) status = CGP_ETIMEOUT;
    double mu = 0.0, mq = 0.0;       // this group's entries of E^+ Z^T P_0^T r and of the same of s
    auto rows_of = [&](int count, auto&& f) {   // this thread's rows of a level
        for (int i = (wid * G + cta) * 32 + lane; i < count; i += 32 * nw * G) f(i);
    };
    auto base_rows = [&](auto&& f) {            // and of the base mesh
        for (int k = k0 + gt; k < k1; k += gs) f(__ldg(pl.perm + k));
    };
    // P_l^T of a complete vector on the coarse level into ws of all levels, then the subdomains'
    // sums into zs; the caller's barrier completes both
    auto restrict_all = [&](const double* from) -> bool {
        for (int l = top; l > 0; --l) {
            const MlLevel& q = pl.lev[l];
            rows_of(q.n, [&](int i) { __stcg(q.ws + i, __ldg(q.dinv + i) != 0.0 ? ml_restrict(q, from, i) : 0.0); });
            from = q.ws;
            if (!sy.sync()) return false;
        }
        if (has) {
            double t = 0.0;
            base_rows([&](int i) {
                if (i < 0) return;
                if (flat) {
                    t += ldcg(from + i);
                    return;
                }
                const double q = ml_restrict(pl.lev[0], from, i);
                __stcg(pl.lev[0].ws + i, q);
                t += q;
            });
            t = ml_group_sum(sm, gs, t);
            if (gt == 0) __stcg(pl.zs + sub, t);
        }
        return true;
    };
    // the levels' residuals: rs = ws, or ss = ws + beta ss and rs -= alpha ss; on the base mesh mu
    // and z as well (both are linear in the residual and follow the same recurrence)
    auto advance = [&](bool start, double alpha, double beta, bool first, double t) {
        auto step = [&](const MlLevel& q, int i) -> double {
            double c = ldcg(q.ws + i);
            if (!start) {
                const double rs = ldcg(q.rs + i);
                if (!first) c = fma(beta, ldcg(q.ss + i), c);
                __stcg(q.ss + i, c);
                c = fma(-alpha, c, rs);
            }
            __stcg(q.rs + i, c);
            return c;
        };
        if (has) {
            if (start) {
                mu = t;
            } else {
                mq = first ? t : fma(beta, mq, t);
                mu = fma(-alpha, mq, mu);
            }
            base_rows([&](int i) {
                if (i >= 0 && flat) __stcg(pl.lev[0].z + i, mu);
                else if (i >= 0) __stcg(pl.lev[0].z + i, fma(__ldg(pl.lev[0].dinv + i), step(pl.lev[0], i), mu));
                else __stcg(pl.lev[0].z - 2 - i, 0.0);
            });
        }
        for (int l = 1; l <= top; ++l) rows_of(pl.lev[l].n, [&](int i) { step(pl.lev[l], i); });
    };
    // u = D^{-1} r + the prolonged z; v[0] = <r, u>, v[2] = <r, r> of this thread's rows
    auto make_u = [&]() -> bool {
        auto rows = [&](auto&& z) {
            v[0] = v[2] = 0.0;
            for (int sl = s_begin + wid; sl < s_end; sl += nw) {
                const int i = sl * 32 + lane;
                if (i >= A.n) continue;
                const double ri = ldcg(r + i), ui = fma(__ldg(a.dinv + i), ri, z(i));
                __stcg(u + i, ui);
                v[0] += ri * ui;
                v[2] += ri * ri;
            }
            return sy.sync();
        };
        if (flat) return rows([&](int i) { return ldcg(pl.lev[0].z + i); });
        if (pl.stored && top > 0) {
            const MlLevel& q = pl.lev[top];
            rows_of(q.n, [&](int i) {
                __stcg(q.z + i, top == 1 ? ml_z<1>(pl, i) : top == 2 ? ml_z<2>(pl, i) : ml_z<3>(pl, i));
            });
            if (!sy.sync()) return false;
            return rows([&](int i) { return ml_prolong_stored(q, i); });
        }
        if (top == 0) return rows([&](int i) { return ml_prolong<0>(pl, i); });
        if (top == 1) return rows([&](int i) { return ml_prolong<1>(pl, i); });
        if (top == 2) return rows([&](int i) { return ml_prolong<2>(pl, i); });
        return rows([&](int i) { return ml_prolong<3>(pl, i); });
    };
    auto plain = [](const double (&s)[3], double (&q)[4]) -> int {
        q[0] = s[0];
        q[1] = s[1];
        return 0;
    };
    while (status == 0) {
        // ---- outer: r = b - A x and its restrictions, then u = M^{-1} r
        double o[4], t;
        int flag;
        v[0] = v[1] = v[2] = 0.0;
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane;
            double ax[1] = {0.0};
            if (!(a.zero_x && outer == 0))
                sell_accum<1>(A, a.val, sl, lane, [&](int j, double (&g)[1]) { g[0] = ldcg(x + j); }, ax);
            if (i >= A.n) continue;
            const double bi = a.b[i], ri = __ldg(pl.tag + i) & CGP_PHI_ZERO ? 0.0 : bi - ax[0];
            __stcg(r + i, ri);
            v[0] += ri * ri;
            v[1] += bi * bi;
        }
        if (!sy.sync() || !restrict_all(r) || !sy.reduce(v, o, flag, t, plain)) {
            status = CGP_ETIMEOUT;
            break;
        }
        if (outer == 0) bb = o[1];
        rr_final = o[0];
        if (!isfinite(o[0]) || !isfinite(bb)) {
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
        advance(true, 0.0, 0.0, true, t);
        if (!sy.sync() || !make_u()) {
            status = CGP_ETIMEOUT;
            break;
        }
        const double stop2 = 0.25 * a.tol2 * bb, stall = stall_level(rr_final, stop2);
        double gamma = 0.0, d = 0.0, rr_best = INFINITY;
        int best_k = 0, leave = 0;
        for (int k = 0;; ++k) {
            // 1 / gamma', off the reduction's chain
            const double rg = k && wid == 0 ? newton_quotient(1.0, gamma) : 0.0;
            v[1] = 0.0;
            for (int sl = s_begin + wid; sl < s_end; sl += nw) {
                const int i = sl * 32 + lane;
                const double wv = row_spmv<double>(A, a.val, nullptr, sl, lane, [&](int j) { return ldcg(u + j); });
                if (i >= A.n) continue;
                __stcg(w + i, wv);
                v[1] += wv * ldcg(u + i);
            }
            if (!sy.sync() || !restrict_all(w)) {
                status = CGP_ETIMEOUT;
                break;
            }
            // out: alpha, beta, gamma, d; flag as in inner_pcg
            if (!sy.reduce(v, o, flag, t, [&](const double (&s)[3], double (&q)[4]) -> int {
                    const double beta = s[0] * rg;
                    q[3] = k ? fma(-beta * beta, d, s[1]) : s[1];
                    q[2] = s[0];
                    q[1] = beta;
                    q[0] = newton_quotient(s[0], q[3]);
                    if (k && !(finite_bits(s[0]) && finite_bits(s[1]) && finite_bits(s[2]))) return 3;
                    if (k && (s[0] == 0.0 || s[2] <= stop2)) return 1;
                    if (s[2] < 0.5 * rr_best) {
                        rr_best = s[2];
                        best_k = k;
                    }
                    if (!finite_bits(q[0]) || q[0] == 0.0) return 2;
                    return k - best_k > stagnation_window(k, rr_best <= stall) || iters >= a.maxit ? 1 : 0;
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
            for (int sl = s_begin + wid; sl < s_end; sl += nw) {
                const int i = sl * 32 + lane;
                if (i >= A.n) continue;
                double p_i = ldcg(u + i), s_i = ldcg(w + i);
                if (k) {
                    p_i = fma(o[1], ldcg(p + i), p_i);
                    s_i = fma(o[1], ldcg(s + i), s_i);
                }
                __stcg(p + i, p_i);
                __stcg(s + i, s_i);
                __stcg(x + i, fma(o[0], p_i, ldcg(x + i)));
                __stcg(r + i, fma(-o[0], s_i, ldcg(r + i)));
            }
            advance(false, o[0], o[1], k == 0, t);
            ++iters;
            if (!sy.sync() || !make_u()) {
                status = CGP_ETIMEOUT;
                break;
            }
        }
        if (status) break;
        if (leave == 3) {
            status = CGP_ENONFINITE;
            break;
        }
        ++outer;   // (x was complete at the barriers of the last preconditioning)
    }
    // ---- pure-Neumann mean fix
    if (a.mlump && status != CGP_ETIMEOUT) {
        double o[4], t;
        int flag;
        v[0] = v[1] = v[2] = 0.0;
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane;
            if (i >= A.n) continue;
            v[0] += __ldg(a.mlump + i) * ldcg(x + i);
            v[1] += __ldg(a.mlump + i);
        }
        if (sy.reduce(v, o, flag, t, plain)) {
            const double shift = o[0] / o[1];
            for (int sl = s_begin + wid; sl < s_end; sl += nw)
                if (sl * 32 + lane < A.n) __stcg(x + sl * 32 + lane, ldcg(x + sl * 32 + lane) - shift);
        } else {
            status = CGP_ETIMEOUT;
        }
    }
    if (blockIdx.x == 0 && tid == 0) {
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

inline auto ml_kernel(int threads) -> void (*)(CoarsePcgArgs, MlPlan) {
    return threads <= 512 ? k_pcg_grid_ml<512> : k_pcg_grid_ml<kMlThreads>;
}

}  // namespace cgp
