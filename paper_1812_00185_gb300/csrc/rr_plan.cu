// Host plan of the register-resident FP64 coarse solve (see rr_plan.cuh).
#include <algorithm>
#include <cmath>
#include <numeric>

#include "rr_plan.cuh"

namespace cgp {

namespace {

// assigns idx[lo, hi) to the parts p0 .. p1 - 1, at most `cap` each
void bisect(std::vector<int32_t>& idx, const std::vector<double>& xy, int lo, int hi, int p0, int p1, int cap,
            std::vector<int32_t>& first) {
    if (p1 - p0 == 1) {
        first[p0] = lo;
        return;
    }
    double mn[2] = {INFINITY, INFINITY}, mx[2] = {-INFINITY, -INFINITY};
    for (int k = lo; k < hi; ++k)
        for (int d = 0; d < 2; ++d) {
            const double v = xy[2 * (size_t)idx[k] + d];
            mn[d] = std::min(mn[d], v);
            mx[d] = std::max(mx[d], v);
        }
    const int axis = mx[1] - mn[1] > mx[0] - mn[0] ? 1 : 0;
    const int parts = p1 - p0, left = parts / 2, here = hi - lo;
    int64_t take = ((int64_t)here * left + parts / 2) / parts;
    take = std::max<int64_t>(take, here - (int64_t)cap * (parts - left));
    take = std::min<int64_t>(take, (int64_t)cap * left);
    const int mid = lo + (int)take;
    std::nth_element(idx.begin() + lo, idx.begin() + mid, idx.begin() + hi, [&](int32_t a, int32_t b) {
        const double x = xy[2 * (size_t)a + axis], y = xy[2 * (size_t)b + axis];
        return x < y || (x == y && a < b);
    });
    bisect(idx, xy, lo, mid, p0, p0 + left, cap, first);
    bisect(idx, xy, mid, hi, p0 + left, p1, cap, first);
}

}  // namespace

bool rr_plan(int n, const std::vector<int32_t>& rowptr, const std::vector<int32_t>& sell_ptr,
             const std::vector<int32_t>& sell_col, const std::vector<double>& val, const std::vector<double>& xy,
             const std::vector<uint8_t>& in_space, int ctas, int threads, bool neumann, RRHostPlan& P) {
    P = RRHostPlan{};
    const int m = ctas;
    if (m < 2 || m > kRRMaxSub || (int64_t)m * threads < n) return false;
    std::vector<int32_t> idx(n), first(m + 1, n), sub(n);
    std::iota(idx.begin(), idx.end(), 0);
    bisect(idx, xy, 0, n, 0, m, threads, first);
    std::vector<int32_t> perm((size_t)m * threads, -1);
    for (int c = 0; c < m; ++c) {
        // rows of one length side by side, so that a warp's lanes have the same entry count
        std::sort(idx.begin() + first[c], idx.begin() + first[c + 1], [&](int32_t a, int32_t b) {
            const int la = rowptr[a + 1] - rowptr[a], lb = rowptr[b + 1] - rowptr[b];
            return la > lb || (la == lb && a < b);
        });
        for (int k = first[c]; k < first[c + 1]; ++k) {
            const int i = idx[k];
            sub[i] = in_space[i] ? c : -1;
            perm[(size_t)c * threads + (k - first[c])] = in_space[i] ? i : -2 - i;
        }
    }
    std::vector<double> E((size_t)m * m, 0.0);
    for (int i = 0; i < n; ++i) {
        if (sub[i] < 0) continue;
        for (int k = 0; k < rowptr[i + 1] - rowptr[i]; ++k) {
            const int64_t e = (int64_t)sell_ptr[i >> 5] + 32 * k + (i & 31);
            const int j = sub[sell_col[e]];
            if (j >= 0) E[(size_t)sub[i] * m + j] += val[e];
        }
    }
    double trace = 0.0;
    for (int j = 0; j < m; ++j) trace += E[(size_t)j * m + j];
    if (!(trace > 0.0) || !std::isfinite(trace)) return false;
    // constants made regular: E + sigma v v^T with v = 1 / sqrt(m), whose inverse is
    // E^+ + v v^T / sigma.  A subdomain without rows of the space only meets zeros.
    const double sigma = trace / m, shift = neumann ? sigma / m : 0.0;
    for (int j = 0; j < m; ++j) {
        for (int k = 0; k < j; ++k) {
            const double s = 0.5 * (E[(size_t)j * m + k] + E[(size_t)k * m + j]) + shift;
            E[(size_t)j * m + k] = E[(size_t)k * m + j] = s;
        }
        double& d = E[(size_t)j * m + j];
        d = d == 0.0 && !neumann ? sigma : d + shift;
    }
    // Cholesky, then the inverse column by column
    std::vector<double> L(E);
    for (int j = 0; j < m; ++j) {
        for (int k = 0; k <= j; ++k) {
            double s = L[(size_t)j * m + k];
            for (int q = 0; q < k; ++q) s -= L[(size_t)j * m + q] * L[(size_t)k * m + q];
            if (k < j) {
                L[(size_t)j * m + k] = s / L[(size_t)k * m + k];
            } else {
                if (!(s > 1e-10 * E[(size_t)j * m + j])) return false;
                L[(size_t)j * m + j] = std::sqrt(s);
            }
        }
    }
    std::vector<double> inv((size_t)m * m), y(m);
    for (int c = 0; c < m; ++c) {
        for (int j = 0; j < m; ++j) {
            double s = j == c ? 1.0 : 0.0;
            for (int q = c; q < j; ++q) s -= L[(size_t)j * m + q] * y[q];
            y[j] = j < c ? 0.0 : s / L[(size_t)j * m + j];
        }
        for (int j = m - 1; j >= 0; --j) {
            double s = y[j];
            for (int q = j + 1; q < m; ++q) s -= L[(size_t)q * m + j] * y[q];
            y[j] = s / L[(size_t)j * m + j];
        }
        for (int j = 0; j < m; ++j) inv[(size_t)j * m + c] = y[j] - (neumann ? 1.0 / (sigma * m) : 0.0);
    }
    for (int j = 0; j < m; ++j)
        for (int k = 0; k < j; ++k)
            inv[(size_t)j * m + k] = inv[(size_t)k * m + j] =
                0.5 * (inv[(size_t)j * m + k] + inv[(size_t)k * m + j]);
    for (double x : inv)
        if (!std::isfinite(x)) return false;
    P.nsub = m;
    P.perm.swap(perm);
    P.einv.swap(inv);
    return true;
}

}  // namespace cgp
