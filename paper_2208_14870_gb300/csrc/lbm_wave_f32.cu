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

template <int RR, bool GEN, bool CHECK>
static cudaError_t launch_tile_k(const StepParams& a, const Coef<float>& c, const TileShape& t, cudaStream_t st) {
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const auto kernel = k_tile<RR, GEN, CHECK>;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!done[dev]) {
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tile_smem(16));
            if (e != cudaSuccess) return e;
            done[dev] = true;
        }
    }
    const int ox = kStSlots - 2 * (t.T - 1);
    const int64_t blocks = tile_count(t, a.nx, a.ny);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    return launch_after(kernel, dim3((unsigned)blocks), dim3(32 * t.NW), tile_smem(t.NW), st, a, pair_coef(c), t.T,
                        (a.nx + ox - 1) / ox);
}

template <int RR>
static cudaError_t launch_tile(const StepParams& a, const Coef<float>& c, bool gen, const TileShape& t, bool check,
                               cudaStream_t st) {
    if (gen) return check ? launch_tile_k<RR, true, true>(a, c, t, st) : launch_tile_k<RR, true, false>(a, c, t, st);
    return check ? launch_tile_k<RR, false, true>(a, c, t, st) : launch_tile_k<RR, false, false>(a, c, t, st);
}

cudaError_t tile_f32(const StepParams& a, const Coef<float>& c, bool gen, const TileShape& t, bool check,
                     cudaStream_t st) {
    if (t.T < 1 || t.NW < 1 || t.NW > 16 || t.NW * t.RR - 2 * (t.T - 1) < 1 || t.T > 16) return cudaErrorInvalidValue;
    return t.RR == 2 ? launch_tile<2>(a, c, gen, t, check, st) : launch_tile<4>(a, c, gen, t, check, st);
}
}  // namespace lbm
