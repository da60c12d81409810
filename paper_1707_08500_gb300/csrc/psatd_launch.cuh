#pragma once
// Launches that overlap at their ends.
#include <cuda_runtime.h>

#include "psatd_internal.h"

namespace psatd {

// Launches of one stream overlap at their ends: every kernel lets the next
// one start its blocks as soon as slots free up (launch_dependents), and none
// reads or writes global memory, the ticket counter included, before the
// kernels ahead of it have finished and their writes are visible (wait).  Both
// do nothing in a launch without the attribute.  A block is alive while the
// kernel ahead still writes, so what that kernel may write (fields, spectra,
// partial sums, global arrays) is not constant for this one: it is read with
// ordinary loads, __ldcg, __ldcs or asynchronous copies, never through the non-coherent path
// (__ldg, or const __restrict__ pointers, which allow it).  That path is for
// what only set-up copies write: descriptors, tables, twiddles.
__device__ __forceinline__ void wait_for_previous_launch() {
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

// Whether a launch of this many blocks gains by overlapping: its early blocks go
// to the SMs that are free first, so a few still get an SM each and enough of
// them fill every SM, but a number between crowds some SMs while others idle.
constexpr bool overlap_pays(int64_t blocks) { return blocks <= kSms / 4 || blocks >= 8 * int64_t(kSms); }

// Launch that may start before the kernels ahead of it on the stream have
// finished (see wait_for_previous_launch): a push is three to six dependent
// launches, and their gaps and block start-up are what small problems wait for.
// Eight boxes of 48^3: 97 to 86 us a step, one box of 32^3 63.5 to 60.9.
// overlap = false: an ordinary launch.
template <class K, class... A>
static cudaError_t launch_maybe_overlapped(bool overlap, K k, dim3 grid, int threads, int smem, cudaStream_t st,
                                           const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(unsigned(threads));
    cfg.dynamicSmemBytes = size_t(smem);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = overlap ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, args...);
    return e != cudaSuccess ? e : cudaPeekAtLastError();
}
template <class K, class... A>
static cudaError_t launch_overlapped(K k, dim3 grid, int threads, int smem, cudaStream_t st, const A&... args) {
    return launch_maybe_overlapped(true, k, grid, threads, smem, st, args...);
}

}  // namespace psatd
