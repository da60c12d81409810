// Launcher of the FP32 z stage and its instantiations (see psatd_zpass.cuh).
#include "psatd_zpass.cuh"

namespace psatd {

// Eq. 1 of boxes one cell deep along z.
cudaError_t launch_stage_flat(bool stag, const LaunchCommon& c, int64_t item0, int64_t nitems, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    const Args<float> a = make_args<float>(c, item0, nitems);
    return stag ? launch_kernel<float>(k_pass_b_flat<true>, a, 0, st) : launch_kernel<float>(k_pass_b_flat<false>, a, 0, st);
}

cudaError_t launch_stage_z(int zlen, int modes, bool heat, bool stag, const LaunchCommon& c, int64_t item0, int64_t nitems,
                           int smem, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    const Args<float> a = make_args<float>(c, item0, nitems);
    // warps a CTA and CTAs per SM: a thread per (first-factor output, mode) and
    // 12 warps per SM at 168 registers; the heat equation's small items fit more
    if (heat) return launch_kernel<float>(k_pass_z<0, kZModesHeat, true, false, 4, 4>, a, smem, st, 4 * 32);
    if (modes == kZModesAsked)
        return stag ? launch_kernel<float>(k_pass_z<0, kZModesAsked, false, true, 6, 2>, a, smem, st, 6 * 32)
                    : launch_kernel<float>(k_pass_z<0, kZModesAsked, false, false, 6, 2>, a, smem, st, 6 * 32);
    if (stag) return launch_kernel<float>(k_pass_z<0, kZModes, false, true, 6, 2>, a, smem, st, 6 * 32);
    switch (zlen) {
        case 96: return launch_kernel<float>(k_pass_z<24, kZModes, false, false, 6, 2>, a, smem, st, 6 * 32);
        case 80: return launch_kernel<float>(k_pass_z<20, kZModes, false, false, 5, 2>, a, smem, st, 5 * 32);
        case 64: return launch_kernel<float>(k_pass_z<16, kZModes, false, false, 4, 3>, a, smem, st, 4 * 32);
        case 48: return launch_kernel<float>(k_pass_z<12, kZModes, false, false, 3, 4>, a, smem, st, 3 * 32);
        case 32: return launch_kernel<float>(k_pass_z<8, kZModes, false, false, 2, 6>, a, smem, st, 2 * 32);
        default: return launch_kernel<float>(k_pass_z<0, kZModes, false, false, 6, 2>, a, smem, st, 6 * 32);
    }
}

}  // namespace psatd
