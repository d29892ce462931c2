// Register-resident variant of the one-launch FP64 coarse solve (Eq. 23).
//
// A cooperative launch of at most one CTA per SM; every warp owns at most one SELL-32 slice
// (32 rows), and every thread keeps its row's first kRRWidth entries (column and value) and
// its PCG vectors (x, r, u, p, s, w) in registers for the whole solve; longer rows re-read
// their remaining entries.  Same outer loop as coarse_pcg_body (FP64 true residual, restart on
// stagnation, optional second initial guess, pure-Neumann mean fix).
//
// Inner iteration: Chronopoulos and Gear's PCG with w = A u formed anew every iteration,
//     p = u + beta p, s = w + beta s, x += alpha p, r -= alpha s, u = D^{-1} r, w = A u,
//     gamma = <r, u>, delta = <w, u>;  beta = gamma / gamma', d = delta - beta^2 d', alpha = gamma / d
// (a prime marks the previous iteration).
// (The pipelined form, which advances w by a recurrence as well, needs one meeting of the CTAs
// per iteration instead of two, but its recursive residual stalls near 1e-9 and then waits out
// the stagnation window: 10,272 iterations to 1e-10 on the channel's 32,489-row system where
// this form takes 1,243, and 2,878 against 580 on 129^2 vertices.)
//
// What bounds an iteration is latency: two round trips through L2 and the narrow FP64 pipe
// (a warp-wide FP64 operation holds an SM's pipe for 16 clocks).  Hence:
//  * u travels without a barrier: a row's owner stores the 16-byte word {u, generation} (one
//    single-copy atomic access) and a reader polls the words of its columns until they carry
//    the generation it needs.  The reductions keep the buffer safe to overwrite: a row's next
//    word is stored only after every CTA has published its sums, and those depend on the words
//    read.
//  * a reduction is one exchange: each CTA stores {partial sum, generation} words and every
//    CTA polls all of them, so data and arrival travel together; two slot sets alternate.
//  * the CTA's sums go through shared memory to three warps (one per sum; 16 + 5 dependent
//    additions) instead of shuffles in every warp, and alpha and beta are formed by one warp:
//    FP64 divides in every thread cost more than the SpMV.
// Measured (GB300), 129^2 rows to 1e-10: 7.8 us an iteration and 4.5 ms a solve (the pipelined
// kernel with a counting barrier, shuffles and divides in every thread: 15.7-25.0 ms);
// 66,049 rows, 14 warps a CTA: 11 us an iteration (vectors in memory: 17.4 us).
// Every CTA adds the partials in the same order, so all hold identical scalars.
// Every poll is bounded: after a limit the reader marks its sums as failed, sets the error
// word, and all CTAs leave with CGP_ETIMEOUT.
#pragma once

#include "coarse_pcg.cuh"

namespace cgp {

constexpr int kRRWidth = 8;          // entries of a row held in registers
constexpr int kRRMaxWarps = 16;      // warps (slices) per CTA: 512 threads of up to 128 registers
constexpr int kRRMinWarps = 8;       // fewer CTAs to poll: 4 warps took 9.4 us an iteration on 129^2 rows, 8 take 7.9
constexpr int kRRPoll = 5;           // words a lane of the polling warps loads at a time (5 x 32 CTAs)

// Shape of the launch for nslices slices on `sms` SMs: as few warps per CTA as keep one CTA
// per SM, at least kRRMinWarps.  Returns false when the system does not fit.
inline bool rr_shape(int nslices, int sms, int* ctas, int* warps) {
    int w = (nslices + sms - 1) / sms;
    if (w < kRRMinWarps) w = kRRMinWarps;
    *warps = w;
    *ctas = (nslices + w - 1) / w;
    return w <= kRRMaxWarps;
}

// Work area (doubles): slots [2][3][ctas + 1] words, the error word (2 doubles), u words [n].
// Zeroed before every launch: generation 0 is never awaited.
inline size_t rr_work_doubles(int n, int ctas) { return 12 * (size_t)(ctas + 1) + 2 + 2 * (size_t)n; }

// one 16-byte {value, tag} word, single-copy atomic, at L2
__device__ __forceinline__ void st_word(double* p, double v, unsigned long long tag) {
    asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p), "d"(v), "l"(tag)
                 : "memory");
}
__device__ __forceinline__ void ld_word(const double* p, double& v, unsigned long long& tag) {
    asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
                 : "=d"(v), "=l"(tag)
                 : "l"(p)
                 : "memory");
}

constexpr unsigned long long kRRFail = 1ull << 63;   // tag bit: the CTA's sums are not valid

struct RRShared {
    double part[3][kRRMaxWarps * 32];
    double tot[3];
    double out[4];
    int ok[3];
    int good;
};

struct RRSync {
    RRShared& sm;
    double* slots;
    int* err;
    unsigned long long gen = 0, ugen = 0;   // generations of the sums and of the u words
    unsigned limit;
    int extra;                              // slots awaited beyond the grid's (1 under the wait test hook)

    __device__ RRSync(RRShared& s, double* sl, int* e, int wait_test)
        : sm(s), slots(sl), err(e), limit(wait_test ? kSpinLimitTest : kSpinLimit), extra(wait_test ? 1 : 0) {}

    // true when a waiting thread has to give up (its own limit, or another's failure)
    __device__ bool expired(unsigned spins) const {
        if (spins > limit) {
            atomicExch(err, 1);
            return true;
        }
        return (spins & 63) == 0 && *(volatile int*)err;
    }

    // Grid-wide sums of (v0, v1, v2), which warp 0 hands to f(t0, t1, t2, out); every thread
    // gets out[0..3].  `bad`: this thread's values are not valid.  False: some wait ran out.
    template <class F>
    __device__ bool reduce(double v0, double v1, double v2, int bad, double (&out)[4], F f) {
        const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5, G = (int)gridDim.x;
        sm.part[0][tid] = v0;
        sm.part[1][tid] = v1;
        sm.part[2][tid] = v2;
        const int anybad = __syncthreads_or(bad);
        ++gen;
        if (wid < 3) {
            // entries beyond the CTA's threads are zero (cleared at the start)
            double t[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) t[j] = sm.part[wid][32 * j + lane];
            for (int k = 4; k < nw; k += 4)
#pragma unroll
                for (int j = 0; j < 4; ++j) t[j] += sm.part[wid][32 * (k + j) + lane];
            double s = (t[0] + t[1]) + (t[2] + t[3]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            // the words of one sum lie side by side, so a warp's poll reads whole lines
            double* base = slots + 2 * (size_t)(G + 1) * (3 * (gen & 1) + wid);
            if (lane == 0) st_word(base + 2 * (size_t)blockIdx.x, s, anybad ? gen | kRRFail : gen);
            double a = 0.0;
            bool ok = true;
            for (int b0 = lane; b0 < G + extra; b0 += 32 * kRRPoll) {
                double v[kRRPoll];
                unsigned long long tg[kRRPoll];
#pragma unroll
                for (int j = 0; j < kRRPoll; ++j) {
                    v[j] = 0.0;
                    tg[j] = gen;
                    if (b0 + 32 * j < G + extra) ld_word(base + 2 * (size_t)(b0 + 32 * j), v[j], tg[j]);
                }
                unsigned spins = 0;
                for (;;) {
                    bool wait = false;
#pragma unroll
                    for (int j = 0; j < kRRPoll; ++j)
                        if ((tg[j] & ~kRRFail) != gen) {
                            ld_word(base + 2 * (size_t)(b0 + 32 * j), v[j], tg[j]);
                            wait |= (tg[j] & ~kRRFail) != gen;
                        }
                    if (!wait) break;
                    if (expired(++spins)) {
                        ok = false;
                        break;
                    }
                }
#pragma unroll
                for (int j = 0; j < kRRPoll; ++j) ok = ok && !(tg[j] & kRRFail);
                // a tree over the words of this lane; one that this CTA count does not have is 0
                if (G > 32) a += ((v[0] + v[1]) + (v[2] + v[3])) + v[4];
                else a = v[0];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            ok = __all_sync(0xffffffffu, ok);
            if (lane == 0) {
                sm.tot[wid] = a;
                sm.ok[wid] = ok;
            }
            asm volatile("bar.sync 1, 96;" ::: "memory");   // the three reducing warps
            if (wid == 0) {
                double o[4] = {0.0, 0.0, 0.0, 0.0};
                f(sm.tot[0], sm.tot[1], sm.tot[2], o);
                if (lane < 4) sm.out[lane] = lane == 0 ? o[0] : (lane == 1 ? o[1] : (lane == 2 ? o[2] : o[3]));
                if (lane == 0) sm.good = sm.ok[0] && sm.ok[1] && sm.ok[2];
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k] = sm.out[k];
        return sm.good != 0;
    }
};

// kWarps: most warps per CTA of the instance (8: no spills; 16: 128 registers a thread)
template <int kWarps>
static __global__ void __launch_bounds__(kWarps * 32, 1) k_pcg_grid_rr(CoarsePcgArgs a) {
    __shared__ RRShared sm;
    double* const slots = a.w64;
    int* const err = reinterpret_cast<int*>(a.w64 + 12 * (size_t)(gridDim.x + 1));
    double* const ubuf = a.w64 + 12 * (size_t)(gridDim.x + 1) + 2;
    for (int k = threadIdx.x; k < 3 * kRRMaxWarps * 32; k += blockDim.x) (&sm.part[0][0])[k] = 0.0;
    __syncthreads();
    RRSync sy(sm, slots, err, a.wait_test);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const SellView& A = a.A;
    const int sl = (int)blockIdx.x * nw + wid;              // this warp's slice (one at most)
    const bool has = sl < A.nslices;
    const int i = sl * 32 + lane;
    const bool row = has && i < A.n;
    // ---- row data, loaded once
    int col[kRRWidth];
    double av[kRRWidth];
    int w_ = 0;
    double dinv_i = 0.0;
#pragma unroll
    for (int k = 0; k < kRRWidth; ++k) {
        col[k] = 0;
        av[k] = 0.0;
    }
    if (has) {
        const int base = __ldg(A.ptr + sl);
        w_ = (__ldg(A.ptr + sl + 1) - base) >> 5;
#pragma unroll
        for (int k = 0; k < kRRWidth; ++k)
            if (k < w_) {
                col[k] = __ldg(A.col + base + 32 * k + lane);
                av[k] = __ldg(a.val + base + 32 * k + lane);
            }
    }
    if (row) {
        dinv_i = __ldg(a.dinv + i);
        if (a.project) a.b[i] -= a.st->mean;   // read again at every outer residual
    }
    int bad = 0;
    // this row's word of the vector being multiplied, then (A v)_i from the rows' words
    auto nothing = [] {};
    auto multiply = [&](double v_i, auto&& meanwhile) -> double {
        const unsigned long long want = ++sy.ugen;
        if (row) st_word(ubuf + 2 * (size_t)i, v_i, want);
        meanwhile();
        double v[kRRWidth];
        unsigned pend = 0;
#pragma unroll
        for (int k = 0; k < kRRWidth; ++k) {
            v[k] = 0.0;
            if (k < w_) {
                unsigned long long tg;
                ld_word(ubuf + 2 * (size_t)col[k], v[k], tg);
                if (tg != want) pend |= 1u << k;
            }
        }
        unsigned spins = 0;
        while (pend) {
#pragma unroll
            for (int k = 0; k < kRRWidth; ++k)
                if (pend >> k & 1) {
                    unsigned long long tg;
                    ld_word(ubuf + 2 * (size_t)col[k], v[k], tg);
                    if (tg == want) pend &= ~(1u << k);
                }
            if (pend && sy.expired(++spins)) {
                bad = 1;
                break;
            }
        }
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int k = 0; k < kRRWidth; k += 2)
            if (k < w_) {
                s0 += av[k] * v[k];
                s1 += av[k + 1] * v[k + 1];
            }
        for (int k = kRRWidth; k < w_ && !bad; ++k) {   // entries beyond the registers
            const int e = __ldg(A.ptr + sl) + 32 * k + lane;
            const int c = __ldg(A.col + e);
            double x;
            unsigned long long tg;
            ld_word(ubuf + 2 * (size_t)c, x, tg);
            for (spins = 0; tg != want;) {
                if (sy.expired(++spins)) {
                    bad = 1;
                    break;
                }
                ld_word(ubuf + 2 * (size_t)c, x, tg);
            }
            s0 += __ldg(a.val + e) * x;
        }
        return s0 + s1;
    };
    auto plain = [](double t0, double t1, double t2, double (&o)[4]) {
        o[0] = t0;
        o[1] = t1;
        o[2] = t2;
    };
    double x_i = (row && !a.zero_x) ? a.x[i] : 0.0;
    int iters = 0, status = 0, outer = 0, used_alt = 0;
    double bb = 0.0, rr_final = 0.0, o[4];
    bool converged = false;
    // ---- the judge of a second initial guess compares FP64 residuals
    if (a.x_alt && !a.zero_x) {
        const double ax = multiply(x_i, nothing);
        double aa = 0.0, y = 0.0;
        if (has)
            for (int k = 0; k < w_; ++k) {
                const int e = __ldg(A.ptr + sl) + 32 * k + lane;
                aa += __ldg(a.val + e) * __ldg(a.x_alt + __ldg(A.col + e));
            }
        if (row) y = __ldg(a.x_alt + i);
        const double b_i = row ? a.b[i] : 0.0;
        const double e0 = row ? (b_i - ax) * (b_i - ax) : 0.0, e1 = row ? (b_i - aa) * (b_i - aa) : 0.0;
        if (!sy.reduce(e0, e1, 0.0, bad, o, plain)) {
            status = CGP_ETIMEOUT;
        } else if (o[1] < o[0]) {
            used_alt = 1;
            x_i = y;
        }
    }
    while (status == 0) {
        // ---- outer: r = b - A x, u = D^{-1} r
        double r_i = 0.0;
        const double ax = (a.zero_x && outer == 0) ? 0.0 : multiply(x_i, nothing);
        const double b_i = row ? a.b[i] : 0.0;
        if (row) r_i = b_i - ax;
        double u_i = dinv_i * r_i;
        if (!sy.reduce(r_i * r_i, b_i * b_i, 0.0, bad, o, plain)) {
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
        // ---- inner iterations; o = (alpha, beta, gamma, d) of the coming update, and why to
        // leave in the shared flag: 1 = target met or restart, 2 = not finite
        const double stop2 = 0.25 * a.tol2 * bb;
        double p_i = 0.0, s_i = 0.0, rg = 0.0, c = 0.0, rr_best = INFINITY;
        double gd[2] = {0.0, 0.0};   // gamma and d of the last update
        int best_k = 0, leave = 0;
        for (int k = 0;; ++k) {
            // warp 0 prepares the next scalars while the words travel: 1 / gamma' and d' / gamma'^2
            const double w_i = multiply(u_i, [&] {
                if (wid == 0 && k) {
                    rg = 1.0 / gd[0];
                    c = gd[1] * rg * rg;
                }
            });
            const bool ok = sy.reduce(
                r_i * u_i, w_i * u_i, r_i * r_i, bad, o, [&](double tg, double td, double trr, double (&q)[4]) {
                    const double beta = tg * rg;
                    const double dn = td - tg * tg * c;
                    q[0] = tg / dn;
                    q[1] = beta;
                    q[2] = tg;
                    q[3] = dn;
                    if (k && !(isfinite(tg) && isfinite(td) && isfinite(trr))) {
                        q[0] = 0.0;
                        q[1] = 2.0;     // not finite after an update
                    } else if (k && (trr <= stop2 || tg == 0.0 || trr == 0.0)) {
                        q[0] = 0.0;
                        q[1] = 1.0;
                    } else {
                        // a long run without halving the smallest residual, or a breakdown
                        // before the update: back to the true residual
                        if (trr < 0.5 * rr_best) {
                            rr_best = trr;
                            best_k = k;
                        }
                        if (!isfinite(q[0]) || k - best_k > kStagnation || iters >= a.maxit) {
                            q[0] = 0.0;
                            q[1] = 1.0;
                        }
                    }
                });
            if (!ok) {
                status = CGP_ETIMEOUT;
                break;
            }
            if (o[0] == 0.0) {          // alpha = 0 carries the reason to leave
                leave = o[1] == 2.0 ? 2 : 1;
                break;
            }
            if (row) {
                p_i = fma(o[1], p_i, u_i);
                s_i = fma(o[1], s_i, w_i);
                x_i = fma(o[0], p_i, x_i);
                r_i = fma(-o[0], s_i, r_i);
                u_i = dinv_i * r_i;
            }
            ++iters;
            gd[0] = o[2];
            gd[1] = o[3];
        }
        if (status) break;
        if (leave == 2) {
            status = CGP_ENONFINITE;
            break;
        }
        ++outer;
    }
    // ---- pure-Neumann mean fix
    if (a.mlump && status != CGP_ETIMEOUT) {
        const double m = row ? __ldg(a.mlump + i) : 0.0;
        if (sy.reduce(m * x_i, m, 0.0, bad, o, [](double t0, double t1, double, double (&q)[4]) { q[0] = t0 / t1; }))
            x_i -= o[0];
        else
            status = CGP_ETIMEOUT;
    }
    if (row) a.x[i] = x_i;
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
        st->pad[1] = used_alt;
    }
}

inline auto rr_kernel(int warps) -> void (*)(CoarsePcgArgs) {
    return warps <= 8 ? k_pcg_grid_rr<8> : k_pcg_grid_rr<kRRMaxWarps>;
}

// zero the work area (a.w64), then the solve
inline cudaError_t rr_launch(const CoarsePcgArgs& a, int ctas, int warps, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(a.w64, 0, rr_work_doubles(a.A.n, ctas) * sizeof(double), st);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas, 1, 1);
    cfg.blockDim = dim3(32 * warps, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, rr_kernel(warps), a);
}

}  // namespace cgp
