// Strip kernels (k_strip, two to seven steps per launch) for the LBM_F32
// population storage.
#include "lbm_ops.cuh"

namespace lbm {
cudaError_t strip_f32(const StepParams& a, const Coef<float>& c, bool gen, int T, bool check, int seg, int* warps,
                      cudaStream_t st) {
    if (check) return T == 4 ? launch_strip_t<S_F32, 4, true>(a, c, gen, seg, warps, st) : cudaErrorInvalidValue;
    switch (T) {
        case 2: return launch_strip_t<S_F32, 2, false>(a, c, gen, seg, warps, st);
        case 3: return launch_strip_t<S_F32, 3, false>(a, c, gen, seg, warps, st);
        case 4: return launch_strip_t<S_F32, 4, false>(a, c, gen, seg, warps, st);
        case 5: return launch_strip_t<S_F32, 5, false>(a, c, gen, seg, warps, st);
        case 6: return launch_strip_t<S_F32, 6, false>(a, c, gen, seg, warps, st);
        case 7: return launch_strip_t<S_F32, 7, false>(a, c, gen, seg, warps, st);
        default: return cudaErrorInvalidValue;
    }
}
}  // namespace lbm
