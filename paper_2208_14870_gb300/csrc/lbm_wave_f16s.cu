// Strip kernels (k_strip, three or four steps per launch) and register tiles for
// the LBM_F16S population storage.
#include "lbm_ops.cuh"

namespace lbm {
cudaError_t strip_f16s(const StepParams& a, const Coef<float>& c, bool gen, int T, bool check, int seg, int* warps,
                       cudaStream_t st) {
    if (check) return T == 4 ? launch_strip_t<S_F16S, 4, true>(a, c, gen, seg, warps, st) : cudaErrorInvalidValue;
    switch (T) {
        case 3: return launch_strip_t<S_F16S, 3, false>(a, c, gen, seg, warps, st);
        case 4: return launch_strip_t<S_F16S, 4, false>(a, c, gen, seg, warps, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t tile_f16s(const StepParams& a, const Coef<float>& c, bool gen, const TileShape& t, bool check,
                      unsigned rounds, cudaStream_t st) {
    return launch_tile<S_F16S>(a, c, gen, t, check, rounds, st);
}
}  // namespace lbm
