// Host plan of the register-resident FP64 coarse solve (coarse_rr.cuh): which row every thread
// holds, and the coarse space of its preconditioner.
#pragma once

#include <cstdint>
#include <vector>

namespace cgp {

constexpr int kRRMaxSub = 160;   // subdomains (one per CTA): five per lane of a warp

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

}  // namespace cgp
