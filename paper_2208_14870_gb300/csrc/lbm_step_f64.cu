// Kernels and launchers for the LBM_F64 population storage.
#include "lbm_ops.cuh"

namespace lbm {
template struct Ops<S_F64>;

// check: at most max_blocks blocks (partial sets)
cudaError_t tile_f64(const StepParams& a, const Coef<double>& c, bool gen, const Tile64Shape& t, bool check,
                     int64_t max_blocks, cudaStream_t st) {
    const int64_t tiles = tile64_count(t, a.nx, a.ny);
    const int64_t blocks = check && tiles > max_blocks ? max_blocks : tiles;
    if (t.T < 1 || tile64_smem(t) > 48 * 1024 || blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    const int ntx = (a.nx + t.bx - 1) / t.bx;
    // whole warps for the slots of the first step, at most four
    const int slots = (t.bx + 2 * (t.T - 1)) * (t.by + 2 * (t.T - 1)), warps = (slots + 31) / 32;
    const dim3 grid((unsigned)blocks), block(32 * (warps < 4 ? warps : 4));
    const size_t sm = tile64_smem(t);
    if (gen)
        return check ? launch_after(k_tile64<true, true>, grid, block, sm, st, a, c, t.T, t.bx, t.by, ntx, tiles)
                     : launch_after(k_tile64<true, false>, grid, block, sm, st, a, c, t.T, t.bx, t.by, ntx, tiles);
    return check ? launch_after(k_tile64<false, true>, grid, block, sm, st, a, c, t.T, t.bx, t.by, ntx, tiles)
                 : launch_after(k_tile64<false, false>, grid, block, sm, st, a, c, t.T, t.bx, t.by, ntx, tiles);
}
}  // namespace lbm
