// Host plans of the FP64 coarse solves over compact subdomains (see rr_plan.cuh).
#include <algorithm>
#include <cmath>
#include <exception>
#include <thread>
#include <utility>

#include "rr_plan.cuh"

namespace cgp {

namespace {

struct Point {
    double x[2];
    int32_t id;
};

// p[lo, hi) into the parts p0 .. p1 - 1 of at most `cap` points, halving the longer side of the
// bounding box.  The two halves of a large piece go to two threads.
void bisect(Point* p, int lo, int hi, int p0, int p1, int cap, int32_t* first) {
    if (p1 - p0 == 1) {
        first[p0] = lo;
        return;
    }
    double mn[2] = {INFINITY, INFINITY}, mx[2] = {-INFINITY, -INFINITY};
    for (int k = lo; k < hi; ++k)
        for (int d = 0; d < 2; ++d) {
            mn[d] = std::min(mn[d], p[k].x[d]);
            mx[d] = std::max(mx[d], p[k].x[d]);
        }
    const int axis = mx[1] - mn[1] > mx[0] - mn[0] ? 1 : 0;
    const int parts = p1 - p0, left = parts / 2, here = hi - lo;
    int64_t take = ((int64_t)here * left + parts / 2) / parts;
    take = std::max<int64_t>(take, here - (int64_t)cap * (parts - left));
    take = std::min<int64_t>(take, (int64_t)cap * left);
    const int mid = lo + (int)take;
    std::nth_element(p + lo, p + mid, p + hi, [axis](const Point& a, const Point& b) {
        return a.x[axis] < b.x[axis] || (a.x[axis] == b.x[axis] && a.id < b.id);
    });
    std::thread other;
    if (here > 100000) {
        try {
            other = std::thread(bisect, p, lo, mid, p0, p0 + left, cap, first);
        } catch (const std::exception&) {   // no thread or no memory for one: one after the other
        }
    }
    if (!other.joinable()) bisect(p, lo, mid, p0, p0 + left, cap, first);
    bisect(p, mid, hi, p0 + left, p1, cap, first);
    if (other.joinable()) other.join();
}

std::vector<Point> points(int n, const std::vector<double>& xy) {
    std::vector<Point> p(n);
    for (int i = 0; i < n; ++i) p[i] = {{xy[2 * (size_t)i], xy[2 * (size_t)i + 1]}, i};
    return p;
}

// E = Z^T K Z of the subdomains sub[i] (-1: outside the space)
std::vector<double> galerkin(int n, int m, const std::vector<int32_t>& rowptr, const std::vector<int32_t>& sell_ptr,
                             const std::vector<int32_t>& sell_col, const std::vector<double>& val,
                             const std::vector<int32_t>& sub) {
    std::vector<double> E((size_t)m * m, 0.0);
    for (int i = 0; i < n; ++i) {
        if (sub[i] < 0) continue;
        double* row = E.data() + (size_t)sub[i] * m;
        for (int k = 0; k < rowptr[i + 1] - rowptr[i]; ++k) {
            const int64_t e = (int64_t)sell_ptr[i >> 5] + 32 * k + (i & 31);
            const int j = sub[sell_col[e]];
            if (j >= 0) row[j] += val[e];
        }
    }
    return E;
}

// Constants made regular: E + sigma v v^T with v = 1 / sqrt(m), whose inverse is E^+ + v v^T / sigma
// (neumann: constants are E's null space).  A subdomain without rows of the space only meets
// zeros.  Returns sigma, 0 when E is no matrix to invert.
double regular(int m, std::vector<double>& E, bool neumann) {
    double trace = 0.0;
    for (int j = 0; j < m; ++j) trace += E[(size_t)j * m + j];
    if (!(trace > 0.0) || !std::isfinite(trace)) return 0.0;
    const double sigma = trace / m, shift = neumann ? sigma / m : 0.0;
    for (int j = 0; j < m; ++j) {
        for (int k = 0; k < j; ++k) {
            const double s = 0.5 * (E[(size_t)j * m + k] + E[(size_t)k * m + j]) + shift;
            E[(size_t)j * m + k] = E[(size_t)k * m + j] = s;
        }
        double& d = E[(size_t)j * m + j];
        d = d == 0.0 && !neumann ? sigma : d + shift;
    }
    return sigma;
}

// pseudo-inverse of the Galerkin matrix E (neumann: constants are its null space); false when a
// pivot is not safely positive
bool inverse(int m, std::vector<double> E, bool neumann, std::vector<double>& inv) {
    const double sigma = regular(m, E, neumann);
    if (!(sigma > 0.0)) return false;
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
    inv.assign((size_t)m * m, 0.0);
    std::vector<double> y(m);
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
    return true;
}

}  // namespace

bool rr_plan(int n, const std::vector<int32_t>& rowptr, const std::vector<int32_t>& sell_ptr,
             const std::vector<int32_t>& sell_col, const std::vector<double>& val, const std::vector<double>& xy,
             const std::vector<uint8_t>& in_space, int ctas, int threads, bool neumann, RRHostPlan& P) {
    P = RRHostPlan{};
    const int m = ctas;
    if (m < 2 || m > kRRMaxSub || (int64_t)m * threads < n) return false;
    std::vector<Point> pts = points(n, xy);
    std::vector<int32_t> first(m + 1, n), sub(n);
    bisect(pts.data(), 0, n, 0, m, threads, first.data());
    std::vector<int32_t> perm((size_t)m * threads, -1);
    for (int c = 0; c < m; ++c) {
        // rows of one length side by side, so that a warp's lanes have the same entry count
        std::sort(pts.begin() + first[c], pts.begin() + first[c + 1], [&](const Point& a, const Point& b) {
            const int la = rowptr[a.id + 1] - rowptr[a.id], lb = rowptr[b.id + 1] - rowptr[b.id];
            return la > lb || (la == lb && a.id < b.id);
        });
        for (int k = first[c]; k < first[c + 1]; ++k) {
            const int i = pts[k].id;
            sub[i] = in_space[i] ? c : -1;
            perm[(size_t)c * threads + (k - first[c])] = in_space[i] ? i : -2 - i;
        }
    }
    std::vector<double> inv;
    if (!inverse(m, galerkin(n, m, rowptr, sell_ptr, sell_col, val, sub), neumann, inv)) return false;
    P.nsub = m;
    P.perm.swap(perm);
    P.einv.swap(inv);
    return true;
}

bool ml_plan(int n, const std::vector<double>& xy, const std::vector<int32_t>& tri, const std::vector<uint8_t>& in_space,
             int nsub, bool neumann, MlHostPlan& P) {
    P = MlHostPlan{};
    const int m = std::min(std::min(nsub, kMlMaxSub), n);
    if (m < 2) return false;
    std::vector<Point> pts = points(n, xy);
    std::vector<int32_t> first(m + 1, n), sub(n), perm(n);
    bisect(pts.data(), 0, n, 0, m, (n + m - 1) / m + 1, first.data());
    for (int c = 0; c < m; ++c)
        for (int k = first[c]; k < first[c + 1]; ++k) {
            const int i = pts[k].id;
            sub[i] = in_space[i] ? c : -1;
            perm[k] = in_space[i] ? i : -2 - i;
        }
    // E from the triangles' element matrices: |T| g_a g_b with g the gradients of the hats
    std::vector<double> E((size_t)m * m, 0.0);
    for (size_t t = 0; 3 * t < tri.size(); ++t) {
        const int32_t* v = &tri[3 * t];
        double ex[3], ey[3];   // edge opposite to each corner
        for (int a = 0; a < 3; ++a) {
            const size_t b = v[(a + 1) % 3], c = v[(a + 2) % 3];
            ex[a] = xy[2 * c] - xy[2 * b];
            ey[a] = xy[2 * c + 1] - xy[2 * b + 1];
        }
        const double area4 = 2.0 * std::fabs(ex[0] * ey[1] - ey[0] * ex[1]);
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b)
                if (sub[v[a]] >= 0 && sub[v[b]] >= 0)
                    E[(size_t)sub[v[a]] * m + sub[v[b]]] += (ex[a] * ex[b] + ey[a] * ey[b]) / area4;
    }
    const double sigma = regular(m, E, neumann);
    if (!(sigma > 0.0)) return false;
    P.nsub = m;
    P.shift = neumann ? 1.0 / (sigma * m) : 0.0;
    P.perm.swap(perm);
    P.first.swap(first);
    P.e.swap(E);
    return true;
}

}  // namespace cgp
