// Launches that may begin while the kernel before them on the stream still runs
// (programmatic dependent launch): the next kernel's launch, and whatever it does before
// await_previous(), overlap the previous kernel.
//
// Every thread of such a kernel calls await_previous() before it touches memory that an
// earlier kernel reads or writes: it returns once the previous kernel has finished and its
// writes are visible.  Only after that is the next kernel let in (admit_next(), else when the
// grid ends), so at most two kernels of a stream overlap and everything before the previous
// one has finished by the time a kernel runs its prologue.  Without a dependent launch on
// either side both calls do nothing; with early false the launch is an ordinary one.
//
// A kernel that lives on L1 is not admitted early beside one that occupies every SM: it runs to
// its end with the L1 that the SM had then (k_to_fixed in fixed_point.cu, k_oz_contract, k_oz_gemm).
//
// What it is for: a split sigma of a small space is three or four kernels of 5 to 15 us, and
// their launches and set-up (the operator's digits into shared memory) stood between them.
// us per sigma of FCI, calls issued back to back, ordinary / dependent launches:
//   determinants      4,900       14,400      63,504      853,776     2,944,656
//   s = 3             28.7/20.7   32.8/26.7   52.5/46.6   450/442     1,631/1,627
//   s = 6             32.8/23.6   39.0/32.9   71.0/65.2   671/663     2,534/2,530
#pragma once

#include <cuda_runtime.h>

__device__ __forceinline__ void await_previous() { cudaGridDependencySynchronize(); }
__device__ __forceinline__ void admit_next() { cudaTriggerProgrammaticLaunchCompletion(); }  // after await_previous()

template <class... P, class... A>
cudaError_t launch_dependent(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = early;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
