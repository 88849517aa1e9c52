// pz_line_bwd.cu -- instantiations of the far-wing reverse pass: strength and van der Waals sums, or
// (pz_line_bwd4.cu, PZ_BWD_FOUR) the radiative and Stark damping sums as well.
#include "pz_far.cuh"

#ifndef PZ_BWD_FOUR
#define PZ_BWD_FOUR false
#define PZ_BWD_LAUNCH launch_far_bwd
#endif

namespace pz {

template <int J, int DS, int MINB>
static cudaError_t launch_bwd_t(pz_ctx *c, const LineArgs &g, int LC, size_t smem, cudaStream_t s) {
    const Tiling &t = c->tiling;
    auto kern = k_line_bwd<J, DS, MINB, PZ_BWD_FOUR>;
    static std::atomic<bool> attr_set[kMaxDevices];
    if (!attr_set[c->device].load(std::memory_order_acquire)) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFarSmemMax);
        attr_set[c->device].store(true, std::memory_order_release);
    }
    const int grid = persistent_grid(c, kern, 32 * t.GW, smem, g.n_items);
    kern<<<grid, 32 * t.GW, smem, s>>>(g, t.GW, LC);
    c->launches++;
    return cudaGetLastError();
}

#define PZ_TILE_BWD(A, B, M) \
    if (c->tiling.J == A && c->tiling.DS == B && c->tiling.minb == M) return launch_bwd_t<A, B, M>(c, g, LC, smem, s);
cudaError_t PZ_BWD_LAUNCH(pz_ctx *c, const LineArgs &g, int LC, size_t smem, cudaStream_t s) {
    PZ_TILE_LIST(PZ_TILE_BWD)
    return cudaErrorInvalidConfiguration;
}

}  // namespace pz
