// Host plans of the FP64 coarse solves over compact subdomains: the register-resident one
// (coarse_rr.cuh: which row every thread holds), the memory-resident one (coarse_gp.cuh: the
// order of the rows) and, where the coarse level has levels below it, the multilevel one
// (coarse_ml.cuh), with the coarse space of their preconditioner.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

namespace cgp {

constexpr int kRRMaxSub = 160;   // subdomains (one per CTA): five per lane of a warp

// The memory-resident solve has a plan for systems of more slices than any launch of the
// register-resident one holds by design (16 per SM of about 150), up to a size whose host plan
// (about 0.1 s per million rows, once per solver) is soon earned back.
constexpr int kGpMinSlices = 2048, kGpMaxSlices = 1 << 17;
inline bool gp_wanted(int nslices) { return nslices > kGpMinSlices && nslices <= kGpMaxSlices; }
inline size_t gp_slots(int64_t n) { return (size_t)n + 32 * (size_t)kRRMaxSub; }
inline size_t gp_entries(int64_t nnz_sell) { return (size_t)nnz_sell + (size_t)nnz_sell / 4 + 32 * 64 * (size_t)kRRMaxSub; }

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

// Plan of the memory-resident solve: nsub compact subdomains of whole 32-row slices, `per` CTAs
// each, and the slices' widths in the new order.
struct GpHostPlan {
    int nsub = 0, per = 0, nslices = 0;
    std::vector<int32_t> perm;      // slot -> row, or -1 (padding)
    std::vector<int32_t> slot_of;   // row -> slot
    std::vector<int32_t> ptr;       // nslices + 1: first entry of every slice
    std::vector<int32_t> first;     // nsub per + 1: first slice of every CTA
    std::vector<double> einv;
};

// False (P.nsub = 0) when E is not safely invertible.
bool gp_plan(int n, const std::vector<int32_t>& rowptr, const std::vector<int32_t>& sell_ptr,
             const std::vector<int32_t>& sell_col, const std::vector<double>& val, const std::vector<double>& xy,
             const std::vector<uint8_t>& in_space, int nsub, int max_per, bool neumann, GpHostPlan& P);

// Systems solved with the inverse of their matrix (coarse_direct.cuh).  Making it takes 6 ms at
// assembly for 1,089 rows and 12 ms for 1,600, and grows with the cube; the solve saves 0.7 ms each
// time.  A caller's iteration cap below kDirectMinCap is one on PCG iterations.
constexpr int kDirectMaxRows = 1600, kDirectMinCap = 64;

// Plan of the multilevel solve (coarse_ml.cuh): the base mesh's vertices in nsub compact
// subdomains, and their Galerkin matrix (made regular), which the device inverts.
constexpr int kMlMaxSub = 608;
// Every system too large for the inverse of its matrix.  Measured against the register-resident
// solve, to 1e-10: 1,681 rows 0.54 ms (0.75), the channel's 2,181 0.66 (1.50), 4,225 rows with one
// to three levels below 0.73-0.94 (1.52-1.58).
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
