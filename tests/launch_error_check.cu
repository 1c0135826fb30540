// Check of launch_overlapped (compiled and run by tests/test_gpu_launch_error.py): a launch
// that the runtime refuses (more threads than a block can have) returns its error, and
// the next launch does not find it again.
#include <cstdio>

#include "overlap.cuh"

__global__ void k_set(int* p, int v) {
    llb::dep_wait();
    *p = v;
}

int main() {
    int *d = nullptr, h = 0;
    if (cudaMalloc(&d, sizeof(int)) != cudaSuccess) return 2;
    const cudaError_t refused = llb::launch_overlapped(k_set, 1, 4096, 0, nullptr, d, 7);
    const cudaError_t left = cudaPeekAtLastError();
    const cudaError_t next = llb::launch_overlapped(k_set, 1, 32, 0, nullptr, d, 5);
    const cudaError_t copy = cudaMemcpy(&h, d, sizeof(int), cudaMemcpyDeviceToHost);
    const bool ok = refused != cudaSuccess && left == cudaSuccess && next == cudaSuccess &&
                    copy == cudaSuccess && h == 5;
    std::printf(ok ? "launch error check ok\n" : "refused %d left %d next %d copy %d value %d\n", refused, left, next, copy, h);
    return ok ? 0 : 1;
}
