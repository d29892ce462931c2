// Host plans of the FP64 coarse solves over compact subdomains: the register-resident one
// (coarse_rr.cuh: which row every thread holds) and the multilevel one (coarse_ml.cuh), with the
// coarse space of their preconditioner.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <vector>

namespace cgp {

constexpr int kRRMaxSub = 160;   // subdomains (one per CTA): five per lane of a warp
constexpr int kRRMaxClusters = 64;   // clusters of a launch: two polled words per lane

// Work area (doubles): words [2][3][kRRMaxClusters], words of the CTAs' Z^T w [2][kRRMaxSub], the
// error word (2 doubles), u words [n].  Zeroed before every launch: generation 0 is never awaited.
constexpr size_t kRRZWords = 12 * (size_t)kRRMaxClusters;
constexpr size_t kRRHead = kRRZWords + 4 * (size_t)kRRMaxSub + 2;
inline size_t rr_work_doubles(int n) { return kRRHead + 2 * (size_t)n; }

struct RRHostPlan {
    int nsub = 0;                  // 0: no plan (the slices in order, Jacobi alone)
    std::vector<int32_t> perm;     // per thread of the launch: row i, -2 - i (a row outside the
                                   // coarse space: phi = 0 there), or -1
    std::vector<double> einv;      // nsub x nsub: pseudo-inverse of E = Z^T K Z
};

// Splits the n rows (vertices xy) by recursive coordinate bisection into `ctas` compact
// subdomains of at most `threads` rows, one per CTA, and inverts the Galerkin matrix of their
// indicator vectors.  neumann: constants are K's null space.  False (P.nsub = 0) when E is
// not safely invertible, e.g. for a mesh of several parts.
bool rr_plan(int n, const std::vector<int32_t>& rowptr, const std::vector<int32_t>& sell_ptr,
             const std::vector<int32_t>& sell_col, const std::vector<double>& val, const std::vector<double>& xy,
             const std::vector<uint8_t>& in_space, int ctas, int threads, bool neumann, RRHostPlan& P);

// Systems solved with the inverse of their matrix (coarse_direct.cuh).  Making it takes 6 ms at
// assembly for 1,089 rows and 12 ms for 1,600, and grows with the cube; the solve saves 0.7 ms each
// time.  A caller's iteration cap below kDirectMinCap is one on PCG iterations.
constexpr int kDirectMaxRows = 1600, kDirectMinCap = 64;

// Plan of the multilevel solve (coarse_ml.cuh): the base mesh's vertices in nsub compact
// subdomains, and their Galerkin matrix (made regular), which the device inverts.
constexpr int kMlMaxSub = 608;
// Every system too large for the inverse of its matrix.  Measured against the register-resident
// solve, to 1e-10: 1,681 rows 0.54 ms with a level below, 0.73 without (0.76), the channel's 2,181
// 0.66 and 0.73 (1.50), 4,225 rows 0.73-0.94 (1.42-1.58), 66,049 rows without a level below 3.2 (3.8).
inline bool ml_wanted(int nslices) { return 32 * nslices > kDirectMaxRows; }
struct MlHostPlan {
    int nsub = 0;
    std::vector<int32_t> perm;      // vertices by subdomain: i, or -2 - i (outside the space)
    std::vector<int32_t> first;     // nsub + 1
    std::vector<double> e;          // nsub x nsub
    double shift = 0.0;             // E^+ = e^{-1} - shift
};

// False (P.nsub = 0) when there is nothing to invert.
bool ml_plan(int n, const std::vector<double>& xy, const std::vector<int32_t>& tri, const std::vector<uint8_t>& in_space,
             int nsub, bool neumann, MlHostPlan& P);

// device views of the multilevel solve
constexpr int kMlMaxLevels = 4;   // levels below the coarse one

struct MlLevel {
    int n = 0;                          // its vertices
    const int32_t* rowptr = nullptr;    // the pattern of the level ABOVE: its rows 0 .. n - 1 restrict
    const int32_t* ptr = nullptr;
    const int32_t* col = nullptr;
    const int2* parents = nullptr;      // of the vertices that the level above adds
    const double* dinv = nullptr;       // 1 / diagonal, 0 where phi = 0
    double* rs = nullptr;               // restricted residual
    double* ws = nullptr;               // restricted w = A u
    double* ss = nullptr;               // restricted s
    double* z = nullptr;                // preconditioned, all levels up to this one (base; uppermost if stored)
};

struct MlPlan {
    int levels = 0, nsub = 0;           // 0: no plan
    MlLevel lev[kMlMaxLevels];
    const int32_t* perm = nullptr;      // base vertices by subdomain (those with phi = 0: -2 - i)
    const int32_t* first = nullptr;     // nsub + 1
    const double* einv = nullptr;       // nsub x nsub
    double* zs = nullptr;               // the subdomains' sums
    bool stored = false;                // the uppermost of the levels stores its z
    int group = 256;           // threads per subdomain: a CTA or a warp
    const uint8_t* tag = nullptr;       // of the coarse level
};

}  // namespace cgp
