// Register-resident variant of the one-launch FP64 coarse solve (Eq. 23).
//
// A cooperative launch of thread-block clusters, at most one CTA per SM; every warp owns at most
// one SELL-32 slice (32 rows), and every thread keeps its row's first kRRWidth entries (column and value) and
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
// With a plan (rr_plan.cuh; the default with the learned guess, whose second start coarse_ml.cuh
// does not take) the rows go to the CTAs as compact subdomains
// and the preconditioner is Jacobi plus an additive coarse correction, as in the on-chip solve:
// M^{-1} = D^{-1} + Z E^+ Z^T with Z the CTAs' indicator vectors and E = Z^T K Z, all in FP64.
// A CTA's sum of w joins the exchange of the other sums; from them s = Z^T r follows by the
// recurrence of r itself (s -= alpha (Z^T w + beta Z^T s')), every first CTA forms mu = E^+ s
// for its cluster and sends it down with alpha and beta, and u = D^{-1} r + mu.  Iterations to
// 1e-10 fall from 580 to 250 (129^2 rows, 72 subdomains), 1,243 to 251 (the channel's 32,489
// rows, 128), 1,162 to 348 (257^2, 144).
//
// What bounds an iteration is latency: two round trips through L2 and the narrow FP64 pipe
// (a warp-wide FP64 operation holds an SM's pipe for 16 clocks).  Hence:
//  * u travels without a barrier: a row's owner stores the 16-byte word {u, generation} (one
//    single-copy atomic access) and a reader polls the words of its columns until they carry
//    the generation it needs.  The reductions keep the buffer safe to overwrite: a row's next
//    word is stored only after every CTA has published its sums, and those depend on the words
//    read.
//  * a reduction climbs: the CTA's sums go through shared memory to three warps (one per sum)
//    and from there to the first CTA of the cluster (st.async on its mbarrier); with several
//    clusters the first CTAs exchange {sum, generation} words through L2, each polling one
//    word per cluster; the first CTA's warp 0 forms alpha and beta and sends them down to its
//    cluster.  (Every CTA polling every CTA's words took 6.5k clocks with 66 CTAs and 8.8k
//    with 148: the polls delay the stores they wait for.)  Two sets of slots alternate.
//  * one warp per cluster forms the scalars: FP64 divides in every thread cost more than the
//    SpMV.  Their divides come down to one reciprocal with two Newton steps, and the checks
//    (finite, converged, stagnating) compare bit patterns on the integer pipe.
// Measured (GB300): 3,872 rows, one cluster of 16, Jacobi: 4.6 us an iteration (every CTA
// polling all: 7.4).  129^2 rows, 9 clusters of 8, to 1e-10: 2.4 ms with the plan, 4.1 ms with
// Jacobi alone, 7.0 us an iteration (14-25 ms: the pipelined kernel with a counting barrier,
// shuffles and divides in every thread).  66,049 rows, 37 clusters of 4: 348 iterations of
// 13 us (1,217 of 10 us in memory with Jacobi, 17 us in the pipelined form).  Of the 14k
// clocks of the 129^2 case with Jacobi the gather takes 3.4k, the words between clusters 4.6k,
// the sums and scalars 4k.
// Every cluster adds the partials in the same order, so all CTAs hold identical scalars.
// Every poll is bounded: after a limit the reader marks its sums as failed, sets the error
// word, and all CTAs leave with CGP_ETIMEOUT.
#pragma once

#include "coarse_pcg.cuh"
#include "rr_plan.cuh"

namespace cgp {

constexpr int kRRWidth = 8;          // entries of a row held in registers
constexpr int kRRMaxWarps = 16;      // warps (slices) per CTA: 512 threads of up to 128 registers
constexpr int kRRMinWarps = 4;       // the reductions use three warps
constexpr int kRRCluster = 8;        // CTAs per cluster of a launch of several clusters: 8, or 4
constexpr int kRRSingle = 16;        // CTAs of a launch of one cluster (small systems)

struct RRShape {
    int ctas = 0, cluster = 0, warps = 0;   // ctas = 0: the system does not fit
};

// co-resident clusters of the largest CTAs: one of kRRSingle CTAs or none; of 8; of 4
struct RRCapacity {
    int single = 0, eight = 0, four = 0;
};

// Launch for nslices slices: one cluster up to 8 slices per CTA (no exchange through L2 in the
// sums); else clusters of 8 with as few warps per CTA as they allow, at least 8 (fewer CTAs,
// fewer words); where 16 warps per CTA do not do (fewer clusters of 8 than SMs / 8 fit the
// GPCs), clusters of 4.
inline RRShape rr_shape(int nslices, const RRCapacity& cap) {
    RRShape s;
    if (cap.single > 0 && nslices <= 8 * kRRSingle) {
        s.cluster = s.ctas = kRRSingle;
        s.warps = (nslices + kRRSingle - 1) / kRRSingle;
        if (s.warps < kRRMinWarps) s.warps = kRRMinWarps;
        return s;
    }
    for (int size : {kRRCluster, kRRCluster / 2}) {
        int fit = size == kRRCluster ? cap.eight : cap.four;
        if (fit > kRRMaxClusters) fit = kRRMaxClusters;
        if (fit > kRRMaxSub / size) fit = kRRMaxSub / size;
        if (fit < 1) continue;
        int w = (nslices + size * fit - 1) / (size * fit);
        if (w < 8) w = 8;
        if (w > kRRMaxWarps) continue;
        const int need = (nslices + w - 1) / w;
        s.warps = w;
        s.cluster = size;
        s.ctas = (need + size - 1) / size * size;
        return s;
    }
    return s;
}

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

constexpr unsigned long long kRRFail = 1ull << 63;   // tag bit: the sums are not valid

// 16 bytes into another CTA's shared memory, completing 16 bytes on its mbarrier
__device__ __forceinline__ void st_async16(uint32_t addr, double a, unsigned long long b, uint32_t mbar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(addr),
                 "l"(__double_as_longlong(a)), "l"(b), "r"(mbar)
                 : "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void mbar_init1(uint64_t* mb) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(mb)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* mb, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(mb)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* mb, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"((uint32_t)__cvta_generic_to_shared(mb)), "r"(parity)
        : "memory");
    return ok != 0;
}

constexpr long long kRRWaitCycles = 4000000000LL;    // ~2 s: a wait this long means a lost signal
constexpr long long kRRWaitCyclesTest = 20000000LL;  // ~10 ms, under the wait test hook
constexpr long long kRRDrainCycles = 100000LL;       // ~50 us, after a wait that ran out

constexpr int kRREinvMax = kRRCluster * kRRMaxSub;   // and kRRSingle^2 is less
static_assert(kRRSingle * kRRSingle <= kRREinvMax, "rows of E^+ of one cluster");

enum RRCorrection { kRRNone, kRRStart, kRRAdvance };   // reduce: what becomes of s = Z^T r

struct RRWord {
    double v;
    unsigned long long tag;
};

struct RRShared {
    double part[4][kRRMaxWarps * 32];
    RRWord up[2][4][kRRSingle];     // first CTA of the cluster: the CTAs' sums {sum, 1 if not valid}
    RRWord down[2][3];              // {out0, out1 as bits}, {out2, out3}, {mu, 1 if valid}
    double tot[3], ab[2];
    int ok[4], valid;
    // first CTA of the cluster, with a plan: Z^T w as received, s = Z^T r and Z^T s' (alternating),
    // and the rows of E^+ of the cluster's CTAs
    double zt[kRRMaxSub], zs[2][kRRMaxSub], zq[2][kRRMaxSub], einv[kRREinvMax];
    uint64_t up_bar[2], down_bar[2];
};

struct RRSync {
    RRShared& sm;
    double* words;
    int* err;
    unsigned long long ugen = 0;            // generation of the u words
    unsigned long long gen = 0;             // generation of the sums
    unsigned limit;
    long long cycles;
    int test;                               // 1 under the wait test hook: the first CTA of every
                                            // cluster also awaits 16 bytes that nothing sends
    int rank, ncl, nclusters, cluster_id, nsub, zpar = 0;
    uint32_t up_remote, up_bar_remote;      // the first CTA's up[0][0][rank] and up_bar[0]

    __device__ RRSync(RRShared& s, double* w, int* e, int wait_test, int nsub_)
        : sm(s), words(w), err(e), nsub(nsub_), limit(wait_test ? kSpinLimitTest : kSpinLimit),
          cycles(wait_test ? kRRWaitCyclesTest : kRRWaitCycles), test(wait_test ? 1 : 0) {
        cgrp::cluster_group c = cgrp::this_cluster();
        rank = (int)c.block_rank();
        ncl = (int)c.num_blocks();
        nclusters = (int)gridDim.x / ncl;
        cluster_id = (int)blockIdx.x / ncl;
        up_remote = cluster_addr(&sm.up[0][0][rank], 0);
        up_bar_remote = cluster_addr(&sm.up_bar[0], 0);
        if (threadIdx.x == 0) {
            for (int k = 0; k < 2; ++k) {
                mbar_init1(&sm.up_bar[k]);
                mbar_init1(&sm.down_bar[k]);
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        c.sync();
    }

    // true when a thread polling memory has to give up (its own limit, or another's failure)
    __device__ bool expired(unsigned spins) const {
        if (spins > limit) {
            atomicExch(err, 1);
            return true;
        }
        return (spins & 63) == 0 && *(volatile int*)err;
    }
    __device__ bool wait(uint64_t* mb, uint32_t parity) const {
        const long long t0 = clock64();
        while (!mbar_try(mb, parity))
            if (clock64() - t0 > cycles) {
                atomicExch(err, 1);
                return false;
            }
        return true;
    }

    // the word's value once it carries this generation (tag: kRRFail set when it never does, or
    // when its writer's sums are not valid)
    __device__ double poll_word(const double* w, unsigned long long& tag) const {
        double v;
        ld_word(w, v, tag);
        for (unsigned spins = 0; (tag & ~kRRFail) != gen;) {
            if (expired(++spins)) {
                tag = kRRFail;
                break;
            }
            ld_word(w, v, tag);
        }
        return v;
    }
    // warp 3 of a first CTA: lanes < ncl hold the CTAs' z sums; all nsub of them into sm.zt
    __device__ void exchange_z(double a, bool ok, int par) {
        const int lane = threadIdx.x & 31;
        if (nclusters == 1) {
            if (lane < ncl) sm.zt[lane] = a;
        } else {
            double* base = words + kRRZWords + 2 * (size_t)kRRMaxSub * par;
            if (lane < ncl) st_word(base + 2 * (cluster_id * ncl + lane), a, ok ? gen : gen | kRRFail);
            double v[kRRMaxSub / 32];
            unsigned long long tag[kRRMaxSub / 32];
#pragma unroll
            for (int j = 0; j < kRRMaxSub / 32; ++j) {   // all five in flight before the first is awaited
                tag[j] = gen;
                v[j] = 0.0;
                if (lane + 32 * j < nsub) ld_word(base + 2 * (lane + 32 * j), v[j], tag[j]);
            }
#pragma unroll
            for (int j = 0; j < kRRMaxSub / 32; ++j) {
                if ((tag[j] & ~kRRFail) != gen) v[j] = poll_word(base + 2 * (lane + 32 * j), tag[j]);
                if (lane + 32 * j < nsub) sm.zt[lane + 32 * j] = v[j];
                ok = ok && !(tag[j] & kRRFail);
            }
            ok = __all_sync(0xffffffffu, ok);
        }
        if (lane == 0) sm.ok[3] = ok;
    }

    // Grid-wide sums of (v0, v1, v2), which warp 0 of every cluster's first CTA hands to
    // f(t0, t1, t2, out); every thread gets out[0..3].  `bad`: this thread's values are not
    // valid.  False (in all threads of the CTA): some wait ran out.  With a plan, z of all
    // threads of a CTA is added up too: kRRStart takes the sums as s, kRRAdvance as Z^T w of the
    // coming update s -= alpha (Z^T w + beta Z^T s') (alpha, beta = out[0], out[1]), and mu is
    // this CTA's entry of E^+ s.
    // A set of slots is rewritten two reductions later, and a CTA gets there only after its
    // first CTA has sent the reduction between, that is, after all contributed to it and so
    // had read what the set held.
    template <class F>
    __device__ bool reduce(double v0, double v1, double v2, double z, RRCorrection corr, int bad, double (&out)[4],
                           double& mu, F f) {
        const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
        const int par = (int)(gen & 1);
        const uint32_t phase = (uint32_t)(gen >> 1) & 1u;
        ++gen;
        sm.part[0][tid] = v0;
        sm.part[1][tid] = v1;
        sm.part[2][tid] = v2;
        const int nv = nsub ? 4 : 3;
        if (nsub) sm.part[3][tid] = z;
        const int anybad = __syncthreads_or(bad);
        if (wid < nv) {
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
            if (lane == 0)
                st_async16(up_remote + (uint32_t)(sizeof(RRWord) * kRRSingle * (4 * par + wid)), s, anybad ? 1ull : 0ull,
                           up_bar_remote + 8 * par);
            if (tid == 0) mbar_expect(&sm.down_bar[par], 3 * sizeof(RRWord));
            if (rank == 0) {
                if (tid == 0) mbar_expect(&sm.up_bar[par], (uint32_t)sizeof(RRWord) * (nv * ncl + test));
                bool ok = wait(&sm.up_bar[par], phase);
                double a = 0.0;
                if (lane < ncl) {
                    a = sm.up[par][wid][lane].v;
                    ok = ok && sm.up[par][wid][lane].tag == 0;
                }
                ok = __all_sync(0xffffffffu, ok);
                if (wid == 3) {
                    exchange_z(a, ok, par);
                } else {
#pragma unroll
                    for (int o = kRRSingle / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                    if (nclusters > 1) {
                        double* base = words + 2 * (size_t)kRRMaxClusters * (3 * par + wid);
                        if (lane == 0) st_word(base + 2 * cluster_id, a, ok ? gen : gen | kRRFail);
                        unsigned long long t0 = gen, t1 = gen;
                        a = 0.0;
                        if (lane < nclusters) a = poll_word(base + 2 * lane, t0);
                        if (lane + 32 < nclusters) a += poll_word(base + 2 * (lane + 32), t1);
                        ok = __all_sync(0xffffffffu, !((t0 | t1) & kRRFail));
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                    }
                    if (lane == 0) {
                        sm.tot[wid] = a;
                        sm.ok[wid] = ok;
                    }
                }
                asm volatile("bar.sync 1, %0;" ::"r"(32 * nv) : "memory");   // the reducing warps
                if (wid == 0) {
                    double o[4] = {0.0, 0.0, 0.0, 0.0};
                    f(sm.tot[0], sm.tot[1], sm.tot[2], o);
                    const bool valid = sm.ok[0] && sm.ok[1] && sm.ok[2] && (!nsub || sm.ok[3]);
                    if (lane < ncl) {
                        const uint32_t dst = cluster_addr(&sm.down[par][0], lane), mb = cluster_addr(&sm.down_bar[par], lane);
                        st_async16(dst, o[0], (unsigned long long)__double_as_longlong(o[1]), mb);
                        st_async16(dst + 16, o[2], (unsigned long long)__double_as_longlong(o[3]), mb);
                        if (!nsub) st_async16(dst + 32, 0.0, valid ? 1ull : 0ull, mb);
                    }
                    if (lane == 0) {
                        sm.ab[0] = o[0];
                        sm.ab[1] = o[1];
                        sm.valid = valid;
                    }
                }
            }
        }
        // the correction, on up to eight warps of the first CTA
        if (nsub && rank == 0 && wid < 8) {
            const int nb = nw < 8 ? nw : 8;
            asm volatile("bar.sync 2, %0;" ::"r"(32 * nb) : "memory");   // zt, ab and valid are there
            double sv[kRRMaxSub / 32];
#pragma unroll
            for (int j = 0; j < kRRMaxSub / 32; ++j) {
                const int k = lane + 32 * j;
                sv[j] = 0.0;
                if (k < nsub && corr != kRRNone) {
                    double q = 0.0;
                    if (corr == kRRStart) {
                        sv[j] = sm.zt[k];
                    } else {
                        q = fma(sm.ab[1], sm.zq[zpar][k], sm.zt[k]);
                        sv[j] = fma(-sm.ab[0], q, sm.zs[zpar][k]);
                    }
                    if (wid == 0) {
                        sm.zq[zpar ^ 1][k] = q;
                        sm.zs[zpar ^ 1][k] = sv[j];
                    }
                }
            }
            for (int c = wid; c < ncl; c += nb) {
                double m = 0.0;
                if (corr != kRRNone) {
#pragma unroll
                    for (int j = 0; j < kRRMaxSub / 32; ++j)
                        if (lane + 32 * j < nsub) m = fma(sm.einv[c * nsub + lane + 32 * j], sv[j], m);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
                }
                if (lane == 0)
                    st_async16(cluster_addr(&sm.down[par][2], c), m, sm.valid ? 1ull : 0ull,
                               cluster_addr(&sm.down_bar[par], c));
            }
            if (corr != kRRNone) zpar ^= 1;
        }
        const bool got = wait(&sm.down_bar[par], phase);
        out[0] = sm.down[par][0].v;
        out[1] = __longlong_as_double((long long)sm.down[par][0].tag);
        out[2] = sm.down[par][1].v;
        out[3] = __longlong_as_double((long long)sm.down[par][1].tag);
        mu = sm.down[par][2].v;
        const bool valid = sm.down[par][2].tag != 0;
        return __syncthreads_and(got && valid) != 0;
    }
};

// kWarps: most warps per CTA of the instance (8: no spills; 16: 128 registers a thread)
template <int kWarps>
static __global__ void __launch_bounds__(kWarps * 32, 1) k_pcg_grid_rr(CoarsePcgArgs a) {
    __shared__ RRShared sm;
    int* const err = reinterpret_cast<int*>(a.w64 + kRRHead - 2);
    double* const ubuf = a.w64 + kRRHead;
    for (int k = threadIdx.x; k < 4 * kRRMaxWarps * 32; k += blockDim.x) (&sm.part[0][0])[k] = 0.0;
    if (a.nsub) {
        const cgrp::cluster_group c = cgrp::this_cluster();
        if (c.block_rank() == 0)
            for (int k = threadIdx.x; k < (int)c.num_blocks() * a.nsub; k += blockDim.x)
                sm.einv[k] = __ldg(a.einv + (size_t)blockIdx.x * a.nsub + k);
    }
    RRSync sy(sm, a.w64, err, a.wait_test, a.nsub);   // (ends with a cluster barrier)
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const SellView& A = a.A;
    // ---- this thread's row: from the plan, or one slice per warp; its entry k is at base + 32 k
    int i, base = 0, w_ = 0;
    bool row, in_space = false;
    if (a.perm) {
        const int g = __ldg(a.perm + blockIdx.x * blockDim.x + threadIdx.x);
        row = g != -1;
        in_space = g >= 0;
        i = g >= 0 ? g : -2 - g;
        if (row) {
            base = __ldg(A.ptr + (i >> 5)) + (i & 31);
            w_ = __ldg(a.rowptr + i + 1) - __ldg(a.rowptr + i);
        }
    } else {
        const int sl = (int)blockIdx.x * nw + wid;
        i = sl * 32 + lane;
        row = i < A.n;
        if (row) {
            // up to the last entry that is not 0, so that no word is awaited for padding, whose
            // column may be no row's (and none for the lanes beyond the last row)
            base = __ldg(A.ptr + sl) + lane;
            const int width = (__ldg(A.ptr + sl + 1) - base + lane) >> 5;
#pragma unroll 8
            for (int k = 0; k < width; ++k)
                if (__ldg(a.val + base + 32 * k) != 0.0) w_ = k + 1;
        }
    }
    // ---- row data, loaded once
    int col[kRRWidth];
    double av[kRRWidth];
    double dinv_i = 0.0;
#pragma unroll
    for (int k = 0; k < kRRWidth; ++k) {
        col[k] = 0;
        av[k] = 0.0;
        if (k < w_) {
            col[k] = __ldg(A.col + base + 32 * k);
            av[k] = __ldg(a.val + base + 32 * k);
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
            const int e = base + 32 * k;
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
    double bb = 0.0, rr_final = 0.0, mu = 0.0, o[4];
    bool converged = false;
    // ---- the judge of a second initial guess compares FP64 residuals
    if (a.x_alt && !a.zero_x) {
        const double ax = multiply(x_i, nothing);
        double aa = 0.0, y = 0.0;
        for (int k = 0; k < w_; ++k) aa += __ldg(a.val + base + 32 * k) * __ldg(a.x_alt + __ldg(A.col + base + 32 * k));
        if (row) y = __ldg(a.x_alt + i);
        const double b_i = row ? a.b[i] : 0.0;
        const double e0 = row ? (b_i - ax) * (b_i - ax) : 0.0, e1 = row ? (b_i - aa) * (b_i - aa) : 0.0;
        if (!sy.reduce(e0, e1, 0.0, 0.0, kRRNone, bad, o, mu, plain)) {
            status = CGP_ETIMEOUT;
        } else if (o[1] < o[0]) {
            used_alt = 1;
            x_i = y;
        }
    }
    while (status == 0) {
        // ---- outer: r = b - A x, u = M^{-1} r
        double r_i = 0.0;
        const double ax = (a.zero_x && outer == 0) ? 0.0 : multiply(x_i, nothing);
        const double b_i = row ? a.b[i] : 0.0;
        if (row) r_i = b_i - ax;
        if (!sy.reduce(r_i * r_i, b_i * b_i, 0.0, in_space ? r_i : 0.0, kRRStart, bad, o, mu, plain)) {
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
        double u_i = fma(dinv_i, r_i, in_space ? mu : 0.0);   // M^{-1} r
        // ---- inner iterations; o = (alpha, beta, gamma, d) of the coming update, and why to
        // leave in the shared flag: 1 = target met or restart, 2 = not finite
        const double stop2 = 0.25 * a.tol2 * bb;
        double p_i = 0.0, s_i = 0.0, rg = 0.0, c = 0.0;
        const long long stall_bits = __double_as_longlong(stall_level(rr_final, stop2));
        long long half_best = 0x7fe0000000000000ll;   // bits of half the smallest <r, r> so far
        double gd[2] = {0.0, 0.0};   // gamma and d of the last update
        int best_k = 0, leave = 0;
        for (int k = 0;; ++k) {
            // the scalars' warp prepares 1 / gamma' and d' / gamma'^2 while the words travel
            const double w_i = multiply(u_i, [&] {
                if (wid == 0 && sy.rank == 0 && k) {
                    rg = 1.0 / gd[0];
                    c = gd[1] * rg * rg;
                }
            });
            const bool ok = sy.reduce(
                r_i * u_i, w_i * u_i, r_i * r_i, in_space ? w_i : 0.0, kRRAdvance, bad, o, mu, [&](double tg, double td, double trr, double (&q)[4]) {
                    const double dn = td - tg * (tg * c);   // (tg^2 alone leaves the range of FP64)
                    q[0] = newton_quotient(tg, dn);
                    q[1] = tg * rg;
                    q[2] = tg;
                    q[3] = dn;
                    // (trr is a sum of squares: for such values the bit patterns order as the
                    // numbers do, and one exponent less is half)
                    const long long rb = __double_as_longlong(trr);
                    if (k && !(finite_bits(tg) && finite_bits(td) && finite_bits(trr))) {
                        q[0] = 0.0;
                        q[1] = 2.0;     // not finite after an update
                    } else if (k && (rb <= __double_as_longlong(stop2) || (__double_as_longlong(tg) << 1) == 0)) {
                        q[0] = 0.0;
                        q[1] = 1.0;
                    } else {
                        // a long run without halving the smallest residual, or a breakdown
                        // before the update: back to the true residual
                        if (rb < half_best) {
                            half_best = rb - (1ll << 52);
                            best_k = k;
                        }
                        const bool may_stall = half_best + (1ll << 52) <= stall_bits;
                        if (!finite_bits(q[0]) || k - best_k > stagnation_window(k, may_stall) || iters >= a.maxit) {
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
                u_i = fma(dinv_i, r_i, in_space ? mu : 0.0);
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
        if (sy.reduce(m * x_i, m, 0.0, 0.0, kRRNone, bad, o, mu, [](double t0, double t1, double, double (&q)[4]) { q[0] = t0 / t1; }))
            x_i -= o[0];
        else
            status = CGP_ETIMEOUT;
    }
    if (row) a.x[i] = x_i;
    cgrp::this_cluster().sync();   // no CTA leaves while its shared memory may be written
    if (status == CGP_ETIMEOUT) {
        // a CTA whose wait ran out has not seen every store that was sent to it: all are on their way
        // now, and 50 us outlast the latest of them (no further meeting: the others may be gone)
        const long long t0 = clock64();
        while (clock64() - t0 < kRRDrainCycles) {
        }
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
        st->pad[1] = used_alt;
    }
}

inline auto rr_kernel(int warps) -> void (*)(CoarsePcgArgs) {
    return warps <= 8 ? k_pcg_grid_rr<8> : k_pcg_grid_rr<kRRMaxWarps>;
}

// attributes: clusters of `cluster` CTAs, all CTAs co-resident
inline void rr_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int ctas, int cluster, int warps,
                      cudaStream_t st) {
    cfg = {};
    cfg.gridDim = dim3(ctas, 1, 1);
    cfg.blockDim = dim3(32 * warps, 1, 1);
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
}

inline cudaError_t rr_capacity(RRCapacity* cap) {
    *cap = RRCapacity{};
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    for (int w : {8, kRRMaxWarps}) {
        const cudaError_t e = cudaFuncSetAttribute(rr_kernel(w), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    auto count = [&](int cluster, int warps) {
        int n = 0;
        rr_config(cfg, attr, cluster, cluster, warps, nullptr);
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, rr_kernel(warps), &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        return n;
    };
    cap->single = count(kRRSingle, 8);
    cap->eight = count(kRRCluster, kRRMaxWarps);
    cap->four = count(kRRCluster / 2, kRRMaxWarps);
    return cudaSuccess;
}

// zero the work area (a.w64), then the solve
inline cudaError_t rr_launch(const CoarsePcgArgs& a, const RRShape& sh, cudaStream_t st) {
    const cudaError_t e = cudaMemsetAsync(a.w64, 0, rr_work_doubles(a.A.n) * sizeof(double), st);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    rr_config(cfg, attr, sh.ctas, sh.cluster, sh.warps, st);
    return cudaLaunchKernelEx(&cfg, rr_kernel(sh.warps), a);
}

}  // namespace cgp
