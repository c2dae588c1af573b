// Kernels and launchers for the LBM_F64 population storage.
#include "lbm_ops.cuh"

namespace lbm {
// (steps: tile_f64)
template cudaError_t Ops<S_F64>::fields(const StepParams&, const Coef<double>&, double, const FieldOut&, cudaStream_t);
template cudaError_t Ops<S_F64>::export_pop(const StepParams&, double, double*, cudaStream_t);
template cudaError_t Ops<S_F64>::import_pop(const StepParams&, double, const double*, cudaStream_t);

// blocks: of the launch (partial sets of a checked one)
cudaError_t tile_f64(const StepParams& a, const Coef<double>& c, bool gen, const Tile64Shape& t, bool check,
                     int64_t* blocks, cudaStream_t st) {
    const dim3 grid = tile64_grid(t, a.nx, a.ny, check ? kMaxCheckBlocks : (int64_t)1 << 40);
    *blocks = (int64_t)grid.x * grid.y;
    if (t.T < 1 || t.T > kT64Max || tile64_smem(t) > kT64Smem || a.plane > 0x7fffffffLL) return cudaErrorInvalidValue;
    const int nty = (a.ny + t.by - 1) / t.by;
    if (t.T == 1) {
        const dim3 block(32, kOne64Rows);
        if (gen)
            return check ? launch_after(k_one64<true, true>, grid, block, 0, st, a, c, nty)
                         : launch_after(k_one64<true, false>, grid, block, 0, st, a, c, nty);
        return check ? launch_after(k_one64<false, true>, grid, block, 0, st, a, c, nty)
                     : launch_after(k_one64<false, false>, grid, block, 0, st, a, c, nty);
    }
    // whole warps for the slots of the first step (two lanes each), at most sixteen
    const int slots = (t.bx + 2 * (t.T - 1)) * (t.by + 2 * (t.T - 1)), warps = (2 * slots + 31) / 32;
    const dim3 block(32 * (warps < 16 ? warps : 16));
    const size_t sm = tile64_smem(t);
    if (gen)
        return check ? launch_after(k_tile64<true, true>, grid, block, sm, st, a, c, t, nty)
                     : launch_after(k_tile64<true, false>, grid, block, sm, st, a, c, t, nty);
    return check ? launch_after(k_tile64<false, true>, grid, block, sm, st, a, c, t, nty)
                 : launch_after(k_tile64<false, false>, grid, block, sm, st, a, c, t, nty);
}
}  // namespace lbm
