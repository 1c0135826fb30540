// Sums the terms a (b r - c) of the nodes in a binary file as the adjoint of an FP32 state
// does, in one warp, and prints the sum exactly (run by tests/test_gpu_adjoint_sums.py).
// File: count, then per node six a, six b, r, six c (float).
#include <cstdio>
#include <vector>

#include "adjoint_terms.cuh"

__global__ void k_sum(const float* p, int n, double* out) {
    llb::Wide<float> s;
    for (int i = threadIdx.x; i < n; i += 32) s.add_node(p + 19 * i, p + 19 * i + 6, p[19 * i + 12], p + 19 * i + 13);
    const double v = s.warp_sum();
    if (threadIdx.x == 0) *out = v;
}

int main(int argc, char** argv) {
    std::FILE* f = argc > 1 ? std::fopen(argv[1], "rb") : nullptr;
    int n = 0;
    if (!f || std::fread(&n, sizeof(n), 1, f) != 1 || n < 1 || n > (1 << 20)) return 2;
    std::vector<float> h(19 * (size_t)n);
    if (std::fread(h.data(), sizeof(float), h.size(), f) != h.size()) return 2;
    float* d = nullptr;
    double *o = nullptr, v = 0.0;
    if (cudaMalloc(&d, h.size() * sizeof(float)) != cudaSuccess || cudaMalloc(&o, sizeof(double)) != cudaSuccess) return 3;
    cudaMemcpy(d, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice);
    k_sum<<<1, 32>>>(d, n, o);
    if (cudaMemcpy(&v, o, sizeof(v), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    std::printf("%a\n", v);
    return 0;
}
