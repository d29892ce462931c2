// Driver of tests/test_gpu_scaled_loads.py: newton_quotient(n, d) of pairs read from a file.
#include <cstdio>
#include <vector>

#include "../paper_1812_00185_gb300/csrc/coarse_pcg.cuh"

__global__ void quotients(int count, const double* n, const double* d, double* q) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        q[i] = cgp::newton_quotient(n[i], d[i]);
}

int main(int argc, char** argv) {
    if (argc != 4) return 2;
    const int count = atoi(argv[1]);
    const size_t bytes = sizeof(double) * count;
    std::vector<double> h(2 * (size_t)count);
    FILE* f = fopen(argv[2], "rb");
    if (!f || fread(h.data(), sizeof(double), h.size(), f) != h.size()) return 2;
    fclose(f);
    double* dev = nullptr;
    if (cudaMalloc(&dev, 3 * bytes) != cudaSuccess) return 1;
    if (cudaMemcpy(dev, h.data(), 2 * bytes, cudaMemcpyHostToDevice) != cudaSuccess) return 1;
    quotients<<<64, 128>>>(count, dev, dev + count, dev + 2 * (size_t)count);
    if (cudaMemcpy(h.data(), dev + 2 * (size_t)count, bytes, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    f = fopen(argv[3], "wb");
    if (!f || fwrite(h.data(), 1, bytes, f) != bytes) return 2;
    return fclose(f) ? 2 : 0;
}
