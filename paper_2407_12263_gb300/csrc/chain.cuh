// chain.cuh -- launches of kernels that follow one another on a stream without the gap between them.
//
// A kernel launched by launch_chained may be brought up while the kernel before it on its stream is
// still running (programmatic stream serialization). It calls chain_begin() before it touches memory,
// which waits until everything before it has completed and is visible, and chain_next() when its work is
// all but done: once every block has said so (or left), the kernel after it is brought up. Order and
// results are those of plain launches, in streams and in captured graphs; what is gained is part of a
// launch, 0.2 to 0.7 us per step (304^2 FP32 3.15 -> 2.71 us; the other sizes of 184^2 to 600^2 and 24^3
// to 80^3 in both schemes, FP32 and FP16, 1.01 to 1.21 times faster). chain_next() stands before a step's
// stores: said at the start of a block, the next grid's first blocks take what slots are free and the
// rest come unevenly to the SMs (304^2 15% slower than plain launches).
//
// Such a kernel is alive while the one before it still writes what it will read. It therefore loads with
// ordinary loads through pointers without __restrict__, which the wait orders: __ldg, and the loads of a
// `const T* __restrict__` parameter that the compiler turns into it, are for data that nobody writes in
// the kernel's lifetime, may be moved above the wait, and go through a cache that need not see the
// writes. (The same holds for a __restrict__ pointer of a kernel that only reads through it.) Ordinary
// loads cost nothing: 128^3 FP32 92.9 us a step, FP16 59.3, 256^3 FP16 453.6 with either.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace lbm {

__device__ __forceinline__ void chain_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;"); }

template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
    if (e != cudaSuccess) (void)cudaGetLastError();  // reported here: the next plain launch must not find it
    return e;
}

}  // namespace lbm
