// Whole coarse-Poisson solve (Eq. 23) in ONE kernel launch.
//
// The coarse system of a CGP step is small (tens of thousands of rows, a few MB, L2
// resident): a PCG with two kernel launches per iteration is bound by launch and
// grid-synchronisation latency.  This kernel keeps every iteration on the device and
// synchronises in one of two ways (the Sync policy):
//
//  * GridSync: a cooperative launch over the whole GPU (every CTA co-resident); the
//    reductions go through per-CTA partial sums in global memory and a software grid
//    barrier (one atomic arrive per CTA, a bounded acquire-spin; on timeout every CTA
//    leaves with CGP_ETIMEOUT instead of hanging).
//  * ClusterSync: one thread-block cluster (up to 16 CTAs); the reductions go through
//    distributed shared memory after a hardware cluster barrier.
//
// Either way every CTA adds the per-CTA sums in the same fixed order, so all CTAs hold
// bit-identical scalars and take identical branches (the barrier counts always match).
// Vectors written inside the kernel are read with ld.global.cg (L2), never through the
// incoherent L1; read-only data (pattern, values, Jacobi diagonal) goes through the
// read-only path.
//
// The FP64 PCG recurrence is Chronopoulos and Gear's with w = A u formed every iteration: one
// reduction and one plain barrier (u complete before its gather) per iteration.
//
// Mixed precision (iterative refinement, CGP_MIXED): the outer residual r = b - A x, its
// norm and the convergence test are FP64; each inner PCG runs its SpMV and vector updates
// in FP32 on an FP32 copy of the matrix, with FP64 accumulation of the dot products.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "krylov.cuh"

namespace cgp {

namespace cgrp = cooperative_groups;

constexpr int kClusterThreads = 1024;
constexpr int kGridThreads = 256;
// CTAs per SM of the memory-resident grid solve: the passes stream, so bytes in flight count.
// 1,050,625 rows to 1e-10 (about 4,650 iterations): 331 / 257 / 233 ms with 2 / 3 / 4 (64
// registers a thread); the update pass with two slices in flight was slower (242 ms)
constexpr int kGridCtasPerSm = 4;
constexpr unsigned kSpinLimit = 1u << 24;   // polls of one grid barrier before giving up (~seconds)
constexpr unsigned kSpinLimitTest = 1u << 14;   // the same under the wait test hook (milliseconds)
constexpr int kStagnation = 2000;           // FP64 inner iterations without halving the best residual
// ... unless this run of the recurrence has itself brought <r, r> down by 1e12 and to within 1e4 of
// its target (norms: 1e6 and 100).  A run of an eighth of the iterations' usual 33 halvings, k / 4,
// is then a stall at the recurrence's attainable accuracy, and a restart from the true residual has
// little left to do.  (One of three seeded loads on 1025^2 rows stalled just above 1e-10 and waited
// out the 2000: 3,572 iterations instead of 1,920.)  A run that starts near its target is not
// stalled when it is slow: with the second condition alone, warm starts with a smooth residual were
// restarted again and again (1025^2 rows, Jacobi, smooth residuals 20 and 50 times the target away:
// 5,132 and 6,783 iterations instead of 1,417 and 1,428).
__device__ __forceinline__ double stall_level(double rr_start, double stop2) { return fmin(1e-12 * rr_start, 1e4 * stop2); }
__device__ __forceinline__ int stagnation_window(int k, bool may_stall) {
    return !may_stall ? kStagnation : (k / 4 < 200 ? 200 : (k / 4 < kStagnation ? k / 4 : kStagnation));
}
constexpr int kStagnation32 = 300;          // the same for the FP32 inner solve of the mixed form

struct CoarsePcgArgs {
    SellView A;
    const double* val;      // FP64 matrix (SELL values)
    const float* valf;      // FP32 copy (mixed precision) or nullptr
    const double* dinv;
    const float* dinvf;
    double* b;              // rhs (projected in place when `project`)
    double* x;              // solution / initial guess
    const double* x_alt;    // optional second initial guess: used instead of x when its FP64 residual is smaller
    double* w64;            // FP64 work: 5 vectors of n (r, u, w, s, p), or rr_work_doubles
    float* w32;             // FP32 work: 7 vectors of n (r, u, z, q, s, p, e)
    const double* mlump;    // non-null: fix sum m_i x_i = 0 after the solve (pure Neumann)
    KrylovState* st;        // out: iter (inner iterations), rr, bb, status, done; in: mean when project
    double tol2;
    double inner_tol;       // mixed: relative reduction asked of each inner solve
    int maxit;
    int zero_x, project, mixed;
    int max_outer;
    // GridSync only
    unsigned int* bar_count;   // zeroed before the launch
    int* bar_err;              // zeroed before the launch; set on a barrier timeout
    double* partials;          // 2 slots x gridDim x 4 doubles
    // test hook (cgp_set_wait_test; 0 otherwise): every bounded wait also waits for one
    // signal that nothing sends, under a limit of milliseconds, so the solve ends with
    // CGP_ETIMEOUT without a fault or a hang
    int wait_test;
    // the learned guess's judge (on-chip solve only; null otherwise): gate[0] = steps left in
    // which the network is not evaluated, gate[1] = consecutive steps in which its direction
    // lowered the starting residual by less than 5 %
    int* gate;
    // plan of the register-resident FP64 solve (rr_plan.cuh), or null and 0
    const int32_t* perm;
    const int32_t* rowptr;
    const double* einv;
    int nsub;
};

template <class T>
__device__ __forceinline__ T ldcg(const T* p) { return __ldcg(p); }

// ------------------------------------------------------------------ sync policies
// Both policies reduce the same way inside a CTA: every thread leaves its values in shared
// memory and warp r adds the column of value r (blockDim / 32 loads and 5 shuffles), so a
// reduction costs the narrow FP64 pipe one warp's chain per value instead of 5 NR additions
// in every warp (a warp-wide FP64 addition holds an SM's pipe for 16 clocks).  And both hand
// the totals to f(tot, out) on warp 0 alone, which forms the iteration's scalars: an FP64
// divide in every thread of a 256-thread CTA holds the pipe for about 1,800 clocks.
// f returns a flag that every thread receives with out.
constexpr int kSumMax = 4;   // values of one reduction; every CTA has at least as many warps

struct SumShared {
    double out[2 * kSumMax];
    int flag;
};

// (after the caller's values are in part[r][thread]) the CTA's total of value r, in every lane
// of the calling warp; part has at least blockDim.x columns
__device__ __forceinline__ double column_sum(const double* __restrict__ part) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    double t[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (j < nw) t[j] = part[32 * j + lane];
    for (int k = 4; k < nw; k += 4)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (k + j < nw) t[j] += part[32 * (k + j) + lane];
    double s = (t[0] + t[1]) + (t[2] + t[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

struct PassTotals {
    template <int NR, int NO>
    __device__ int operator()(const double (&tot)[NR], double (&out)[NO]) const {
#pragma unroll
        for (int k = 0; k < NR; ++k) out[k] = tot[k];
        return 0;
    }
};

constexpr int kMaxClusterCtas = 16;

// shared memory of a ClusterSync whose CTA has at most T threads
template <int T>
struct ClusterShared {
    double part[kSumMax][T];
    double slots[2][kSumMax][kMaxClusterCtas];   // [set][value][CTA of the cluster]
    SumShared res;
};

struct ClusterSync {
    cgrp::cluster_group cluster;
    double* part;
    int cols;                                    // columns of part
    double (*slots)[kSumMax][kMaxClusterCtas];
    SumShared* res;
    float* dyn;        // dynamic shared memory for inner_cg_shared (null: none), and its floats
    int dyn_floats;
    int slot = 0;
    template <int T>
    __device__ explicit ClusterSync(ClusterShared<T>& sm, float* d = nullptr, int nd = 0)
        : cluster(cgrp::this_cluster()), part(&sm.part[0][0]), cols(T), slots(sm.slots), res(&sm.res), dyn(d),
          dyn_floats(nd) {}
    __device__ int rank() const { return (int)cluster.block_rank(); }
    __device__ int ranks() const { return (int)cluster.num_blocks(); }
    __device__ bool sync() {
        cluster.sync();
        return true;
    }
    // every CTA's partial goes into every CTA's slots before the one cluster barrier; two slot
    // sets alternate, so a set is rewritten only after every CTA has read it (it arrived at the
    // barrier between)
    template <int NR, int NO, class F>
    __device__ bool sum_to(const double (&v)[NR], double (&out)[NO], int& flag, F f) {
        static_assert(NR <= kSumMax && NO <= 2 * kSumMax, "SumShared sizes");
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, ncl = ranks();
#pragma unroll
        for (int k = 0; k < NR; ++k) part[k * cols + threadIdx.x] = v[k];
        __syncthreads();
        if (wid < NR) {
            const double s = column_sum(part + wid * cols);
            if (lane < ncl) *cluster.map_shared_rank(&slots[slot][wid][rank()], lane) = s;
        }
        cluster.sync();
        if (wid == 0) {
            double tot[NR], o[NO];
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                tot[k] = lane < ncl ? slots[slot][k][lane] : 0.0;
#pragma unroll
                for (int d = kMaxClusterCtas / 2; d > 0; d >>= 1) tot[k] += __shfl_xor_sync(0xffffffffu, tot[k], d);
                tot[k] = __shfl_sync(0xffffffffu, tot[k], lane & (kMaxClusterCtas - 1));
            }
            const int fl = f(tot, o);
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < NO; ++k) res->out[k] = o[k];
                res->flag = fl;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NO; ++k) out[k] = res->out[k];
        flag = res->flag;
        slot ^= 1;
        return true;
    }
    template <int NR>
    __device__ bool sum(const double (&v)[NR], double (&tot)[NR]) {
        int flag;
        return sum_to(v, tot, flag, PassTotals{});
    }
    __device__ void finish() { cluster.sync(); }   // no CTA leaves while its shared memory may be written
};

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// n / d by Newton's iteration for 1 / d from the 20-bit approximation (two steps: 80 bits, so
// the quotient is within rounding of the exact one); not finite where d is 0 or not finite.  The
// approximation takes subnormal d for 0 and has 0 for 1 / d from 2^1022 on: there a division (a
// call, or its chain takes part in every quotient).
static __device__ __noinline__ double divided(double n, double d) { return n / d; }
__device__ __forceinline__ double newton_quotient(double n, double d) {
    const unsigned ex = (unsigned)__double2hiint(d) >> 20 & 0x7ffu;
    if (ex - 1u >= 0x7fcu && ex != 0x7ffu) return divided(n, d);
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    r = fma(r, fma(-d, r, 1.0), r);
    const double e = fma(-d, r, 1.0), q = n * r;
    return fma(q, e, q);
}
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

struct GridShared {
    double part[kSumMax][kGridThreads];
    double tot[kSumMax];
    SumShared res;
};

struct GridBarrier {
    unsigned* count;
    int* err;
    unsigned gen = 0;
    unsigned extra = 0;            // arrivals awaited beyond the grid's (1 under the wait test hook)
    unsigned limit = kSpinLimit;
    __device__ GridBarrier(unsigned* c, int* e, int wait_test)
        : count(c), err(e), extra(wait_test ? 1u : 0u), limit(wait_test ? kSpinLimitTest : kSpinLimit) {}
    __device__ bool sync() {
        __shared__ int ok;
        __syncthreads();
        ++gen;
        if (threadIdx.x == 0) {
            int good = 1;
            // arrive: a release-ordered add publishes this CTA's writes (cumulative over the
            // CTA through the barrier above); wait: acquire-spin on the counter
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
            const unsigned target = gen * gridDim.x + extra;
            unsigned spins = 0;
            for (;;) {
                const unsigned v = ld_acquire_gpu(count);
                if ((int)(v - target) >= 0) break;
                if (++spins > limit) {
                    atomicExch(err, 1);
                    good = 0;
                    break;
                }
                if ((spins & 63) == 0 && *(volatile int*)err) {
                    good = 0;
                    break;
                }
            }
            ok = good;
        }
        __syncthreads();
        return ok != 0;
    }
};

struct GridSync : GridBarrier {
    double* partials;
    GridShared& sm;
    int slot = 0;
    __device__ GridSync(unsigned* c, int* e, double* p, GridShared& s, int wait_test = 0)
        : GridBarrier(c, e, wait_test), partials(p), sm(s) {}
    __device__ int rank() const { return (int)blockIdx.x; }
    __device__ int ranks() const { return (int)gridDim.x; }
    // per-CTA partials [set][value][CTA]; after the grid barrier warp r of every CTA adds the
    // partials of value r in the same order (lane l takes l, l + 32, ...)
    template <int NR, int NO, class F>
    __device__ bool sum_to(const double (&v)[NR], double (&out)[NO], int& flag, F f) {
        static_assert(NR <= kSumMax && NO <= 2 * kSumMax, "SumShared sizes");
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, G = (int)gridDim.x;
#pragma unroll
        for (int k = 0; k < NR; ++k) sm.part[k][threadIdx.x] = v[k];
        __syncthreads();
        double* mine = partials + ((size_t)slot * kSumMax + wid) * G;
        if (wid < NR) {
            const double s = column_sum(sm.part[wid]);
            if (lane == 0) __stcg(mine + blockIdx.x, s);
        }
        if (!sync()) return false;
        if (wid < NR) {
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
            double tot[NR], o[NO];
#pragma unroll
            for (int k = 0; k < NR; ++k) tot[k] = sm.tot[k];
            const int fl = f(tot, o);
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < NO; ++k) sm.res.out[k] = o[k];
                sm.res.flag = fl;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NO; ++k) out[k] = sm.res.out[k];
        flag = sm.res.flag;
        slot ^= 1;
        return true;
    }
    template <int NR>
    __device__ bool sum(const double (&v)[NR], double (&tot)[NR]) {
        int flag;
        return sum_to(v, tot, flag, PassTotals{});
    }
    __device__ void finish() {}
};

// FP32 counterpart of sell_accum (FP32 values, FP32 gathered vector, FP32 sum)
template <class Gather>
__device__ __forceinline__ float sell_accum_f(const SellView& A, const float* __restrict__ val, int sl, int lane,
                                              Gather&& g) {
    const int base = __ldg(A.ptr + sl), w = (__ldg(A.ptr + sl + 1) - base) >> 5;
    float s = 0.0f;
    for (int k0 = 0; k0 < w; k0 += 8) {
        int cj[8];
        float av[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            cj[u] = 0;
            av[u] = 0.0f;
            if (k0 + u < w) {
                const int e = base + 32 * (k0 + u) + lane;
                cj[u] = __ldg(A.col + e);
                av[u] = __ldg(val + e);
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (k0 + u < w) s += av[u] * g(cj[u]);
    }
    return s;
}

// ------------------------------------------------------------------ the solve
template <class T>
struct InnerVecs {
    T *r, *u, *w, *z, *q, *s, *p, *e;
};

// sum_k val(row,k) * g(col(row,k)) in precision T (FP32 values for T = float)
template <class T, class Gather>
__device__ __forceinline__ T row_spmv(const SellView& A, const double* __restrict__ v64, const float* __restrict__ v32,
                                      int sl, int lane, Gather&& g) {
    if constexpr (sizeof(T) == 4) {
        return sell_accum_f(A, v32, sl, lane, g);
    } else {
        double acc[1] = {0.0};
        sell_accum<1>(A, v64, sl, lane, [&](int j, double (&o)[1]) { o[0] = g(j); }, acc);
        return acc[0];
    }
}

// Inner FP64 PCG (Chronopoulos-Gear, w = A u formed every iteration as in coarse_rr.cuh) on
// A x = b from the residual r and u = D^{-1} r in V (written before the last barrier), with
// gamma = <r, u> and rr_start = <r, r>; x itself is V.e.  Two passes over the rows per iteration: w = A u with the
// reduction, then the vector updates.  Returns false on a barrier timeout.  iters counts
// iterations across calls.  outcome: 0 = ended normally (target met, or stagnation),
// 1 = breakdown before an update (the iterate is intact), 2 = a non-finite value after an
// update (the iterate is not).
template <class Sync>
__device__ bool inner_pcg(const CoarsePcgArgs& a, Sync& sy, const InnerVecs<double>& V, const double* __restrict__ dinv,
                          int s_begin, int s_end, double gamma, double rr_start, double stop2, int& iters, int& outcome) {
    outcome = 0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const SellView& A = a.A;
    double d = 0.0, rr_best = INFINITY, part[3] = {0.0, 0.0, 0.0};
    const double stall = stall_level(rr_start, stop2);
    int best_k = 0;
    for (int k = 0;; ++k) {
        // w = A u, <w, u> (u is complete)
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane;
            const double wv = row_spmv<double>(A, a.val, a.valf, sl, lane, [&](int j) { return ldcg(V.u + j); });
            if (i < A.n) {
                __stcg(V.w + i, wv);
                part[1] += wv * ldcg(V.u + i);
            }
        }
        // out: alpha, beta, gamma, d; flag: 0 go on, else 1 + outcome
        double o[4];
        int flag;
        if (!sy.sum_to(part, o, flag, [&](const double (&t)[3], double (&q)[4]) -> int {
                const double tg = k ? t[0] : gamma, trr = k ? t[2] : INFINITY;
                const double beta = k ? tg / gamma : 0.0;
                q[3] = k ? t[1] - beta * beta * d : t[1];
                q[2] = tg;
                q[1] = beta;
                q[0] = tg / q[3];
                if (k && !(isfinite(t[0]) && isfinite(t[1]) && isfinite(t[2]))) return 3;
                if (k && (t[0] == 0.0 || trr <= stop2)) return 1;
                // CG residual norms are not monotone: only a long run without halving the
                // smallest counts as stagnation, and hands back to the true residual
                if (trr < 0.5 * rr_best) {
                    rr_best = trr;
                    best_k = k;
                }
                if (!isfinite(q[0]) || q[0] == 0.0) return 2;
                return k - best_k > stagnation_window(k, rr_best <= stall) || iters >= a.maxit ? 1 : 0;
            }))
            return false;
        if (flag) {
            outcome = flag - 1;
            return true;
        }
        gamma = o[2];
        d = o[3];
        part[0] = part[1] = part[2] = 0.0;
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane;
            if (i >= A.n) continue;
            double p_i = ldcg(V.u + i), s_i = ldcg(V.w + i);
            if (k) {
                p_i = fma(o[1], ldcg(V.p + i), p_i);
                s_i = fma(o[1], ldcg(V.s + i), s_i);
            }
            const double r_i = fma(-o[0], s_i, ldcg(V.r + i)), u_i = __ldg(dinv + i) * r_i;
            __stcg(V.p + i, p_i);
            __stcg(V.s + i, s_i);
            __stcg(V.e + i, fma(o[0], p_i, ldcg(V.e + i)));
            __stcg(V.r + i, r_i);
            __stcg(V.u + i, u_i);
            part[0] += r_i * u_i;
            part[2] += r_i * r_i;
        }
        ++iters;
        if (!sy.sync()) return false;   // u is complete before it is gathered
    }
}

// Inner PCG in its classical form (two reductions per iteration) on A e = r0 in precision
// T, from e = 0 and r = r0, u = D^{-1} r0 in V; p and q use V.p/V.s (p double-buffered
// with V.q because the SpMV gathers p at neighbouring rows while rows are rewritten).
// Used for the FP32 inner solves of the mixed form, where the longer recurrence of the
// one-reduction form drifts.  Same outcome codes as inner_pcg.
template <class T, class Sync>
__device__ bool inner_pcg_classic(const CoarsePcgArgs& a, Sync& sy, const InnerVecs<T>& V,
                                  const T* __restrict__ dinv, int s_begin, int s_end, double rz, double stop2,
                                  int& iters, int& outcome) {
    outcome = 0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const SellView& A = a.A;
    T* p_old = V.u;   // the first direction is z = u itself
    T* p_new = V.p;
    T* z = V.u;       // u holds D^{-1} r
    T* q = V.q;
    double beta = 0.0, rr_best = INFINITY;
    int best_k = 0;
    for (int k = 0; iters < a.maxit; ++k) {
        // phase A: p_new = z + beta p_old (p_old = z at k = 0), q = A p_new, <p_new, q>
        const T be = (T)beta;
        double pq_acc[1] = {0.0};
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane;
            const T qi = row_spmv<T>(A, a.val, a.valf, sl, lane,
                                     [&](int j) { return k ? ldcg(z + j) + be * ldcg(p_old + j) : ldcg(z + j); });
            if (i < A.n) {
                const T pv = k ? ldcg(z + i) + be * ldcg(p_old + i) : ldcg(z + i);
                __stcg(p_new + i, pv);
                __stcg(q + i, qi);
                pq_acc[0] += (double)pv * (double)qi;
            }
        }
        double o1[1];
        int flag;
        if (!sy.sum_to(pq_acc, o1, flag, [&](const double (&t)[1], double (&q)[1]) -> int {
                q[0] = rz / t[0];   // alpha
                return !(t[0] != 0.0) || !isfinite(t[0]);
            }))
            return false;
        if (flag) {
            outcome = 1;
            return true;
        }
        const T al = (T)o1[0];
        // phase B: e += alpha p, r -= alpha q, z = D^{-1} r; <r,z>, <r,r>
        double acc2[2] = {0.0, 0.0};
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane;
            if (i >= A.n) continue;
            __stcg(V.e + i, ldcg(V.e + i) + al * ldcg(p_new + i));
            const T rv = ldcg(V.r + i) - al * ldcg(q + i);
            const T zv = __ldg(dinv + i) * rv;
            __stcg(V.r + i, rv);
            __stcg(V.z + i, zv);
            acc2[0] += (double)rv * (double)zv;
            acc2[1] += (double)rv * (double)rv;
        }
        // flag: 1 = not finite, 2 = target met (or exact), 3 = the FP32 recurrence is drifting
        // away (its iterate is not to be used), 4 = stagnating
        double t2[2];
        if (!sy.sum_to(acc2, t2, flag, [&](const double (&t)[2], double (&q)[2]) -> int {
                q[0] = t[0];
                q[1] = t[0] / rz;   // beta
                if (!isfinite(t[0]) || !isfinite(t[1])) return 1;
                if (t[0] == 0.0 || t[1] == 0.0 || t[1] <= stop2) return 2;
                if (t[1] < 0.5 * rr_best) {
                    rr_best = t[1];
                    best_k = k;
                    return 0;
                }
                return t[1] > 1e4 * rr_best ? 3 : (k - best_k > kStagnation32 ? 4 : 0);
            }))
            return false;
        ++iters;
        if (flag) {
            outcome = flag == 1 || flag == 3 ? 2 : 0;
            return true;
        }
        rz = t2[0];
        beta = t2[1];
        // from now on z lives in V.z, and the directions alternate between V.p and V.s
        z = V.z;
        p_old = p_new;
        p_new = (p_new == V.p) ? V.s : V.p;
    }
    return true;
}

// Floats of shared memory inner_cg_shared needs per CTA: u of all rows, and r, w, p, s, e of
// the CTA's own.
__host__ __device__ inline int shared_cg_floats(int nslices, int ctas) {
    return 32 * nslices + 5 * 32 * ((nslices + ctas - 1) / ctas);
}

// Inner FP32 CG of one cluster with its vectors in shared memory, in Chronopoulos and Gear's
// form with w = A u formed every iteration: every CTA holds u of all rows, and a row's owner
// stores its new u into every CTA (distributed shared memory), so the SpMV gathers locally;
// r, w, p, s, e of the own rows stay in the CTA, the matrix streams through L1.  One reduction
// and one plain cluster barrier per iteration.  (inner_pcg_classic, with its vectors in global
// memory and two reductions, took 16k clocks an iteration on at most 1,089 rows and 22k on
// 4,225, on 8 CTAs.)  Dot products are accumulated in FP64 as there; same outcome codes.
__device__ inline void inner_cg_shared(const CoarsePcgArgs& a, ClusterSync& sy, const InnerVecs<float>& V, int s_begin,
                                       int s_end, double gamma, double stop2, int& iters, int& outcome) {
    outcome = 0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5, ncl = sy.ranks();
    const SellView& A = a.A;
    const int own = 32 * ((A.nslices + ncl - 1) / ncl);
    float* const u = sy.dyn;
    float* const r = u + 32 * A.nslices;
    float *const w = r + own, *const p = w + own, *const s = p + own, *const e = s + own;
    auto publish = [&](int i, float v) {
        for (int c = 0; c < ncl; ++c) sy.cluster.map_shared_rank(u, c)[i] = v;
    };
    for (int sl = s_begin + wid; sl < s_end; sl += nw) {
        const int i = sl * 32 + lane, l = i - 32 * s_begin;
        const bool in = i < A.n;
        r[l] = in ? ldcg(V.r + i) : 0.0f;
        p[l] = s[l] = e[l] = 0.0f;
        publish(i, in ? ldcg(V.u + i) : 0.0f);
    }
    sy.sync();
    double d = 0.0, rg = 0.0, c = 0.0, rr_best = INFINITY, part[3] = {0.0, 0.0, 0.0};
    int best_k = 0;
    for (int k = 0;; ++k) {
        if (wid == 0 && k) {   // 1 / gamma' and d' / gamma'^2, off the reduction's chain
            rg = 1.0 / gamma;
            c = d * rg * rg;
        }
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane, l = i - 32 * s_begin;
            const float wv = sell_accum_f(A, a.valf, sl, lane, [&](int j) { return u[j]; });
            w[l] = wv;
            if (i < A.n) part[1] += (double)wv * (double)u[i];
        }
        // out: alpha, beta, gamma, d; flag: 0 go on, else 1 + outcome
        double o[4];
        int flag;
        const double gamma0 = gamma;
        sy.sum_to(part, o, flag, [&](const double (&t)[3], double (&q)[4]) -> int {
            const double tg = k ? t[0] : gamma0, trr = k ? t[2] : INFINITY;
            q[3] = t[1] - tg * tg * c;
            q[2] = tg;
            q[1] = tg * rg;
            q[0] = tg / q[3];
            if (k && !(isfinite(t[0]) && isfinite(t[1]) && isfinite(t[2]))) return 3;
            if (k && (t[0] == 0.0 || trr <= stop2)) return 1;
            if (trr < 0.5 * rr_best) {
                rr_best = trr;
                best_k = k;
            } else if (trr > 1e4 * rr_best) {
                return 3;   // the FP32 recurrence is drifting away: its iterate is not to be used
            }
            if (!isfinite(q[0]) || q[0] == 0.0) return 2;
            return k - best_k > kStagnation32 || iters >= a.maxit ? 1 : 0;
        });
        if (flag) {
            outcome = flag - 1;
            break;
        }
        gamma = o[2];
        d = o[3];
        const float al = (float)o[0], be = (float)o[1];
        part[0] = part[1] = part[2] = 0.0;
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane, l = i - 32 * s_begin;
            const float pv = fmaf(be, p[l], u[i]), sv = fmaf(be, s[l], w[l]);
            const float rv = fmaf(-al, sv, r[l]), uv = i < A.n ? __ldg(a.dinvf + i) * rv : 0.0f;
            p[l] = pv;
            s[l] = sv;
            e[l] = fmaf(al, pv, e[l]);
            r[l] = rv;
            publish(i, uv);
            part[0] += (double)rv * (double)uv;
            part[2] += (double)rv * (double)rv;
        }
        ++iters;
        sy.sync();   // u is complete before it is gathered
    }
    for (int sl = s_begin + wid; sl < s_end; sl += nw) {
        const int i = sl * 32 + lane;
        if (i < A.n) __stcg(V.e + i, e[i - 32 * s_begin]);
    }
}

template <class Sync>
__device__ void coarse_pcg_body(const CoarsePcgArgs& a, Sync& sy) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const SellView& A = a.A;
    const int part = sy.rank(), parts = sy.ranks();
    const int s_begin = (int)(((int64_t)A.nslices * part) / parts);
    const int s_end = (int)(((int64_t)A.nslices * (part + 1)) / parts);
    const double mean = a.project ? a.st->mean : 0.0;
    const double tol2 = a.tol2;
    const size_t n = (size_t)A.n;
    double* xv = a.x;
    InnerVecs<double> V64{a.w64, a.w64 + n, a.w64 + 2 * n, nullptr, nullptr, a.w64 + 3 * n, a.w64 + 4 * n, xv};
    InnerVecs<float> V32{a.w32, a.w32 + n, nullptr, a.w32 + 2 * n, a.w32 + 3 * n, a.w32 + 4 * n, a.w32 + 5 * n,
                         a.w32 + 6 * n};
    double bb = 0.0, rr_final = 0.0;
    int iters = 0, status = 0, outer = 0, used_alt = 0;
    bool mixed_now = a.mixed != 0;   // cleared if an FP32 inner solve ever produces a non-finite value
    bool converged = false;
    if (a.x_alt && !a.zero_x) {
        // the judge of the learned guess: keep whichever start has the smaller FP64 residual
        double acc[2] = {0.0, 0.0};
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane;
            double ax[1] = {0.0}, aa[1] = {0.0};
            sell_accum<1>(A, a.val, sl, lane, [&](int j, double (&o)[1]) { o[0] = ldcg(xv + j); }, ax);
            sell_accum<1>(A, a.val, sl, lane, [&](int j, double (&o)[1]) { o[0] = __ldg(a.x_alt + j); }, aa);
            if (i < A.n) {
                const double bi = a.b[i] - mean;
                acc[0] += (bi - ax[0]) * (bi - ax[0]);
                acc[1] += (bi - aa[0]) * (bi - aa[0]);
            }
        }
        double tot[2];
        bool ok = sy.template sum<2>(acc, tot);
        if (ok && tot[1] < tot[0]) {
            used_alt = 1;
            for (int sl = s_begin + wid; sl < s_end; sl += nw) {
                const int i = sl * 32 + lane;
                if (i < A.n) __stcg(xv + i, __ldg(a.x_alt + i));
            }
            ok = sy.sync();
        }
        if (!ok) status = CGP_ETIMEOUT;
    }
    for (; status == 0;) {
        // ---- outer residual r = b - A x (FP64), ||r||^2, ||b||^2, inner start r, u = D^{-1} r
        double acc[3] = {0.0, 0.0, 0.0};
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane;
            double axv[1] = {0.0};
            if (!(a.zero_x && outer == 0))
                sell_accum<1>(A, a.val, sl, lane, [&](int j, double (&o)[1]) { o[0] = ldcg(xv + j); }, axv);
            if (i < A.n) {
                double bi = a.b[i];
                if (a.project && outer == 0) {
                    bi -= mean;
                    a.b[i] = bi;
                }
                if (a.zero_x && outer == 0) __stcg(xv + i, 0.0);
                const double ri = bi - axv[0];
                if (mixed_now) {
                    const float rf = (float)ri;
                    const float uf = __ldg(a.dinvf + i) * rf;
                    __stcg(V32.r + i, rf);
                    __stcg(V32.u + i, uf);
                    __stcg(V32.e + i, 0.0f);
                    acc[2] += (double)rf * (double)uf;
                } else {
                    const double ui = __ldg(a.dinv + i) * ri;
                    __stcg(V64.r + i, ri);
                    __stcg(V64.u + i, ui);
                    acc[2] += ri * ui;
                }
                acc[0] += ri * ri;
                acc[1] += bi * bi;
            }
        }
        double tot[3];
        if (!sy.template sum<3>(acc, tot)) {
            status = CGP_ETIMEOUT;
            break;
        }
        if (outer == 0) bb = tot[1];
        const double rr0 = tot[0];
        rr_final = rr0;
        if (!isfinite(rr0)) {
            status = CGP_ENONFINITE;
            break;
        }
        if (rr0 <= tol2 * bb) {
            converged = true;
            break;
        }
        if (outer >= a.max_outer || iters >= a.maxit) {
            status = CGP_ENOTCONV;
            break;
        }
        bool ok;
        int outcome = 0;
        if (mixed_now) {
            const double stop2 = fmax(a.inner_tol * a.inner_tol * rr0, 0.25 * tol2 * bb);
            bool shared = false;
            if constexpr (std::is_same<Sync, ClusterSync>::value)
                shared = sy.dyn && shared_cg_floats(A.nslices, parts) <= sy.dyn_floats;
            if (shared) {
                if constexpr (std::is_same<Sync, ClusterSync>::value)
                    inner_cg_shared(a, sy, V32, s_begin, s_end, tot[2], stop2, iters, outcome);
                ok = true;
            } else {
                ok = inner_pcg_classic<float>(a, sy, V32, a.dinvf, s_begin, s_end, tot[2], stop2, iters, outcome);
            }
        } else {
            // FP64: the inner recurrence updates x itself; the next outer pass re-checks the true residual
            ok = inner_pcg(a, sy, V64, a.dinv, s_begin, s_end, tot[2], rr0, 0.25 * tol2 * bb, iters, outcome);
        }
        if (!ok) {
            status = CGP_ETIMEOUT;
            break;
        }
        if (outcome == 2 && !mixed_now) {
            status = CGP_ENONFINITE;   // x itself is no longer finite
            break;
        }
        if (outcome == 2) {
            // the FP32 correction blew up: drop it and finish this solve with FP64 inner solves
            mixed_now = false;
        } else if (mixed_now) {
            for (int sl = s_begin + wid; sl < s_end; sl += nw) {
                const int i = sl * 32 + lane;
                if (i < A.n) __stcg(xv + i, ldcg(xv + i) + (double)ldcg(V32.e + i));
            }
        }
        // x is complete before any CTA forms the next outer residual
        if (!sy.sync()) {
            status = CGP_ETIMEOUT;
            break;
        }
        ++outer;
    }
    // ---- pure-Neumann mean fix: x -= sum(m x) / sum(m)
    if (a.mlump && status != CGP_ETIMEOUT) {
        bool ok = sy.sync();
        double acc[2] = {0.0, 0.0};
        for (int sl = s_begin + wid; sl < s_end; sl += nw) {
            const int i = sl * 32 + lane;
            if (i < A.n) {
                acc[0] += __ldg(a.mlump + i) * ldcg(xv + i);
                acc[1] += __ldg(a.mlump + i);
            }
        }
        double tot[2];
        ok = ok && sy.template sum<2>(acc, tot);
        if (ok) {
            const double mu = tot[0] / tot[1];
            for (int sl = s_begin + wid; sl < s_end; sl += nw) {
                const int i = sl * 32 + lane;
                if (i < A.n) __stcg(xv + i, ldcg(xv + i) - mu);
            }
        } else {
            status = CGP_ETIMEOUT;
        }
    }
    if (part == 0 && threadIdx.x == 0) {
        KrylovState* st = a.st;
        st->iter = iters;
        st->bb[0] = bb;
        st->rr[0] = rr_final;
        st->bb[1] = 0.0;
        st->rr[1] = 0.0;
        st->status = status ? status : (converged ? 0 : CGP_ENOTCONV);
        st->done = 1;
        st->pad[0] = outer;
        st->pad[1] = used_alt;
    }
    sy.finish();
}

static __global__ void __launch_bounds__(kClusterThreads, 1) k_pcg_cluster(CoarsePcgArgs a) {
    __shared__ ClusterShared<kClusterThreads> sm;
    ClusterSync sy(sm);
    sy.sync();   // every CTA runs before its shared memory is written
    coarse_pcg_body(a, sy);
}

// Coarse solves of many independent CGP instances in ONE persistent launch: every cluster
// of the launch takes instances from a queue (the host orders them longest step first) and
// solves each with the ClusterSync body; clusters never wait on one another.
static __global__ void __launch_bounds__(kClusterThreads, 1) k_pcg_batch(const CoarsePcgArgs* __restrict__ args, int ninst,
                                                                  unsigned int* queue) {
    __shared__ ClusterShared<kClusterThreads> sm;
    __shared__ int job;
    ClusterSync sy(sm);
    for (;;) {
        if (sy.rank() == 0 && threadIdx.x == 0) job = (int)atomicAdd(queue, 1u);
        sy.cluster.sync();
        const int j = *sy.cluster.map_shared_rank(&job, 0);
        sy.cluster.sync();   // every CTA has read rank 0's job before it can change
        if (j >= ninst) break;
        const CoarsePcgArgs a = args[j];
        coarse_pcg_body(a, sy);
    }
}

static __global__ void __launch_bounds__(kGridThreads, kGridCtasPerSm) k_pcg_grid(CoarsePcgArgs a) {
    __shared__ GridShared sm;
    GridSync sy(a.bar_count, a.bar_err, a.partials, sm, a.wait_test);
    coarse_pcg_body(a, sy);
}

}  // namespace cgp
