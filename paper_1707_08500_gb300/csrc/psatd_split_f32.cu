// FP32 stages with one axis length compiled in: the row and column launches of
// the split-plane schedule and the z stage of long axes (one box over the grid,
// the global solver).
#include "psatd_kernels.cuh"

namespace psatd {

// f(integral_constant) for v among the lengths of `list`
template <const auto& list, int I = 0, class F>
static bool with_length(int v, F&& f) {
    if constexpr (I < int(sizeof(list) / sizeof(list[0]))) {
        if (v == list[I]) { f(std::integral_constant<int, list[I]>{}); return true; }
        return with_length<list, I + 1>(v, f);
    }
    return false;
}

// Stages 1 and 4 to 7 (see stage_item); false when the plan's length is not
// compiled in.
bool launch_stage_length(int stage, const LaunchCommon& c, int64_t item0, int64_t nitems, int smem, cudaStream_t st,
                         cudaError_t* err) {
    *err = cudaSuccess;
    const Args<float> a = make_args<float>(c, item0, nitems);
    auto go = [&](auto k) { if (nitems > 0) *err = launch_kernel<float>(k, a, smem, st, kThreads, stage >= 6); };
    if (stage == 1) {
        static_assert(sizeof(kLongZ) / sizeof(ZChunk) == 3, "one line per entry of kLongZ");
        if (c.longZ == kLongZ[0].L) go(k_pass_b<float, GeoZ<kLongZ[0].L, kLongZ[0].M>>);
        else if (c.longZ == kLongZ[1].L) go(k_pass_b<float, GeoZ<kLongZ[1].L, kLongZ[1].M>>);
        else if (c.longZ == kLongZ[2].L) go(k_pass_b<float, GeoZ<kLongZ[2].L, kLongZ[2].M>>);
        else return false;
        return true;
    }
    switch (stage) {
        case 4: return with_length<kSplitX>(c.splitX, [&](auto l) { go(k_rows_fwd<float, decltype(l)::value>); });
        case 5: return with_length<kSplitY>(c.splitY, [&](auto l) { go(k_cols<float, false, decltype(l)::value>); });
        case 6: return with_length<kSplitY>(c.splitY, [&](auto l) { go(k_cols<float, true, decltype(l)::value>); });
        case 7: return with_length<kSplitX>(c.splitX, [&](auto l) { go(k_rows_inv<float, decltype(l)::value>); });
        default: return false;
    }
}

}  // namespace psatd
