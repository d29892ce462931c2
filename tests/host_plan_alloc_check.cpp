// Driver of tests/test_host_memory.py: the multilevel plan of many points, the k-th host allocation
// failing for k = 1, 2, ...: every run ends with the plan or with std::bad_alloc.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>

#include "../paper_1812_00185_gb300/csrc/rr_plan.cuh"

static std::atomic<long> left{0};   // 0: not armed

void* operator new(size_t n) {
    if (left.load() > 0 && left.fetch_sub(1) == 1) throw std::bad_alloc();
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }

int main() {
    const int n = 450000, side = 671;
    std::vector<double> xy(2 * (size_t)n);
    for (int i = 0; i < n; ++i) {
        xy[2 * (size_t)i] = (double)(i % side);
        xy[2 * (size_t)i + 1] = (double)(i / side);
    }
    const std::vector<int32_t> tri = {0, side - 1, n - 1};   // (across subdomains)
    const std::vector<uint8_t> in_space(n, 1);
    int failed = 0, made = 0;
    for (long k = 1; k <= 24; ++k) {
        cgp::MlHostPlan P;
        left = k;
        try {
            if (cgp::ml_plan(n, xy, tri, in_space, cgp::kMlMaxSub, true, P)) ++made;
        } catch (const std::bad_alloc&) {
            ++failed;
        }
        left = 0;
    }
    std::printf("failed %d made %d\n", failed, made);
    return failed > 0 && made > 0 ? 0 : 1;
}
