// Step kernels launched one after the other on a stream, each set up while the CTAs of
// the one before it end (programmatic dependent launch).  It saves the launch between
// two short steps: 50 steps with their conversions, launched by llb_step, of 131 x 97 x
// 75 D3Q27 1269 to 1161 us, of two components at 128^3 D3Q19 with diagnostics 4512 to
// 4400; the replayed graph of 200 steps of 32^3 955 to 917.
//
// A kernel launched with launch_overlapped may start once every CTA of the kernel
// before it has called dep_launch (or has ended); it touches no global memory before
// dep_wait, which returns when the kernel before it has ended and its writes are
// visible.  dep_launch comes when a CTA has no item left: called at the start, the
// waiting CTAs of the next step take the place of running ones (graph steps of 48^3
// 6.4 us, so 5.6, without overlap 5.8; 32^3 5.05, 4.6, 4.8).  After a kernel that never
// calls dep_launch, or a copy, the launch is an ordinary one.
//
// What the kernel before wrote is read with load_dep and through pointers that are not
// __restrict__.  The non-coherent load (__ldg, or what the compiler makes of a const
// __restrict__ pointer) is for data that is read-only for the whole life of a kernel, and
// the life of these begins while the kernel before still writes.  It was faster (256^3 D3Q19
// 1 %, 200 steps of 32^3 in a graph 884 us against 917).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace llb {

__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class T>
__device__ __forceinline__ T load_dep(const T* p) { return *p; }

template <class... P, class... A>
cudaError_t launch_overlapped(void (*kern)(P...), int grid, int block, size_t smem, cudaStream_t stream, A&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // reported here: the next launch must not find it again
    return e;
}

}  // namespace llb
