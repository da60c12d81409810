// FP32 plane stages with thread-private transforms of compile-time length
// (passes A and C) and their launcher.
// rows: the largest local y length.
#include "psatd_regfft.cuh"

namespace psatd {

// stage 0: pass A, stage 2: pass C (see stage_item)
cudaError_t launch_stage_reg(int stage, int rows, const LaunchCommon& c, int64_t item0, int64_t nitems, int smem, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    const Args<float> a = make_args<float>(c, item0, nitems);
    // pass A: a thread per row, up to 64 rows or up to kRegRows
    if (rows > kRegRows) return cudaErrorInvalidValue;
    if (stage == 0) return rows <= 64 ? launch_kernel<float>(k_pass_a_reg<64>, a, smem, st, 64)
                                      : launch_kernel<float>(k_pass_a_reg<kRegRows>, a, smem, st, kRegRows);
    if (stage == 2) return launch_kernel<float>(k_pass_c_reg, a, smem, st, kRegThreads, true);
    return cudaErrorInvalidValue;
}

}  // namespace psatd
