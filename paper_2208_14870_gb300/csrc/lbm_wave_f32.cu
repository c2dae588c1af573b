// Strip kernels (k_strip, two to six steps per launch) for the LBM_F32
// population storage.
#include "lbm_ops.cuh"

namespace lbm {
cudaError_t strip_f32(const StepParams& a, const Coef<float>& c, bool gen, int T, bool check, int seg, int* warps,
                      cudaStream_t st) {
    if (check) {
        if (T == 5) return launch_strip_t<S_F32, 5, true>(a, c, gen, seg, warps, st);
        return T == 4 ? launch_strip_t<S_F32, 4, true>(a, c, gen, seg, warps, st) : cudaErrorInvalidValue;
    }
    switch (T) {
        case 2: return launch_strip_t<S_F32, 2, false>(a, c, gen, seg, warps, st);
        case 3: return launch_strip_t<S_F32, 3, false>(a, c, gen, seg, warps, st);
        case 4: return launch_strip_t<S_F32, 4, false>(a, c, gen, seg, warps, st);
        case 5: return launch_strip_t<S_F32, 5, false>(a, c, gen, seg, warps, st);
        case 6: return launch_strip_t<S_F32, 6, false>(a, c, gen, seg, warps, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t tile_f32(const StepParams& a, const Coef<float>& c, bool gen, const TileShape& t, bool check,
                     cudaStream_t st) {
    return launch_tile<S_F32>(a, c, gen, t, check, 0, st);
}
}  // namespace lbm
