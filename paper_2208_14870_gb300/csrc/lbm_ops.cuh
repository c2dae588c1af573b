// lbm_ops.cuh -- launchers of the per-storage kernels; included by exactly one
// translation unit per storage type (lbm_step_f64.cu, lbm_step_f32.cu,
// lbm_step_f16s.cu), which instantiates Ops<S> for its type (FP64: without step).
#pragma once

#include <mutex>

#include "lbm_kernels.cuh"

namespace lbm {

// The two-step kernels use more than 48 KB of dynamic shared memory, which
// each device must allow once per kernel.
template <int S>
static cudaError_t t2_allow_smem() {
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return cudaSuccess;
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    e = cudaFuncSetAttribute(k_step2<S, false, false, false>, at, kT2Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step2<S, false, true, false>, at, kT2Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step2<S, true, false, false>, at, kT2Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step2<S, true, true, false>, at, kT2Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step2<S, false, false, true>, at, kT2Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step2<S, false, true, true>, at, kT2Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step2<S, true, false, true>, at, kT2Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step2<S, true, true, true>, at, kT2Smem);
    if (e == cudaSuccess) done[dev] = true;
    return e;
}

template <int S>
static cudaError_t t3_allow_smem() {
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return cudaSuccess;
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    e = cudaFuncSetAttribute(k_step3<S, false, false, false>, at, kT3Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step3<S, true, false, false>, at, kT3Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step3<S, false, false, true>, at, kT3Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step3<S, true, false, true>, at, kT3Smem);
    if (e == cudaSuccess) done[dev] = true;
    return e;
}

// Three fused plain steps, one block per tile.  (The library puts residual
// checks on two-step launches; a checked three-step launch is not offered.)
template <int S>
static cudaError_t launch_step3(const StepParams& a, const Coef<float>& c, bool gen, bool check,
                                int check_blocks, cudaStream_t st) {
    (void)check_blocks;
    if (check) return cudaErrorNotSupported;
    cudaError_t e = t3_allow_smem<S>();
    if (e != cudaSuccess) return e;
    const unsigned int grid = (unsigned int)step3_tiles(a.nx, a.ny);
    const dim3 block(kT2Threads);
    const bool any = !step3_fits(a.nx, a.ny);   // lattice smaller than the slot array
    if (any)
        return gen ? launch_after(k_step3<S, true, false, true>, grid, block, kT3Smem, st, a, c)
                   : launch_after(k_step3<S, false, false, true>, grid, block, kT3Smem, st, a, c);
    return gen ? launch_after(k_step3<S, true, false, false>, grid, block, kT3Smem, st, a, c)
               : launch_after(k_step3<S, false, false, false>, grid, block, kT3Smem, st, a, c);
}

// One strip kernel: its dynamic shared memory (above 48 KB) is allowed once
// per device; warps: resident warps per multiprocessor (no launch).
template <int S, bool GEN, int T, bool CHECK>
static cudaError_t launch_strip_k(const StepParams& a, const Coef<float>& c, int seg, int* warps, cudaStream_t st) {
    static std::mutex mu;
    static int resident[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const auto kernel = k_strip<S, GEN, T, CHECK>;
    constexpr int NW = kStNW, SM = st_smem<S, T, CHECK>();
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!resident[dev]) {
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SM);
            if (e != cudaSuccess) return e;
            int b = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, 32 * NW, SM);
            if (e != cudaSuccess) return e;
            resident[dev] = b > 0 ? b * NW : NW;
        }
        if (warps) {
            *warps = resident[dev];
            return cudaSuccess;
        }
    }
    const int64_t ns = strip_count(S, T, a.nx), items = ns * ((a.ny + seg - 1) / seg);
    if (items > 0x7fffffffLL - 64) return cudaErrorInvalidValue;
    return launch_after(kernel, dim3((unsigned)((items + NW - 1) / NW)), dim3(32 * NW), SM, st, a, pair_coef(c), seg,
                        (int)ns, (int)items);
}

template <int S, int T, bool CHECK>
static cudaError_t launch_strip_t(const StepParams& a, const Coef<float>& c, bool gen, int seg, int* warps,
                                  cudaStream_t st) {
    return gen ? launch_strip_k<S, true, T, CHECK>(a, c, seg, warps, st)
               : launch_strip_k<S, false, T, CHECK>(a, c, seg, warps, st);
}

// Register tiles (k_tile).
template <int S, int RR, bool GEN, bool CHECK>
static cudaError_t launch_tile_k(const StepParams& a, const Coef<float>& c, const TileShape& t, unsigned rounds,
                                 cudaStream_t st) {
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const auto kernel = k_tile<S, RR, GEN, CHECK>;
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
                        (a.nx + ox - 1) / ox, rounds);
}

template <int S, int RR>
static cudaError_t launch_tile_r(const StepParams& a, const Coef<float>& c, bool gen, const TileShape& t, bool check,
                                 unsigned rounds, cudaStream_t st) {
    if (gen)
        return check ? launch_tile_k<S, RR, true, true>(a, c, t, rounds, st)
                     : launch_tile_k<S, RR, true, false>(a, c, t, rounds, st);
    return check ? launch_tile_k<S, RR, false, true>(a, c, t, rounds, st)
                 : launch_tile_k<S, RR, false, false>(a, c, t, rounds, st);
}

template <int S>
static cudaError_t launch_tile(const StepParams& a, const Coef<float>& c, bool gen, const TileShape& t, bool check,
                               unsigned rounds, cudaStream_t st) {
    if (t.T < 1 || t.NW < 1 || t.NW > 16 || t.NW * t.RR - 2 * (t.T - 1) < 1 || t.T > 16) return cudaErrorInvalidValue;
    return t.RR == 2 ? launch_tile_r<S, 2>(a, c, gen, t, check, rounds, st)
                     : launch_tile_r<S, 4>(a, c, gen, t, check, rounds, st);
}

// Two fused steps: one block per tile (check: up to check_blocks blocks).
template <int S>
static cudaError_t launch_step2(const StepParams& a, const Coef<float>& c, bool gen, bool check,
                                int check_blocks, cudaStream_t st) {
    cudaError_t e = t2_allow_smem<S>();
    if (e != cudaSuccess) return e;
    const int64_t tiles = step2_tiles(a.nx, a.ny);
    const unsigned int grid = (unsigned int)(check ? (tiles < check_blocks ? tiles : check_blocks) : tiles);
    const dim3 block(kT2Threads);
    const auto go = [&](auto any) {              // any: lattice smaller than the slot array
        constexpr bool ANY = decltype(any)::value;
        if (gen)
            return check ? launch_after(k_step2<S, true, true, ANY>, grid, block, kT2Smem, st, a, c)
                         : launch_after(k_step2<S, true, false, ANY>, grid, block, kT2Smem, st, a, c);
        return check ? launch_after(k_step2<S, false, true, ANY>, grid, block, kT2Smem, st, a, c)
                     : launch_after(k_step2<S, false, false, ANY>, grid, block, kT2Smem, st, a, c);
    };
    return step2_fits(a.nx, a.ny) ? go(std::false_type()) : go(std::true_type());
}

template <int S, int V>
static cudaError_t launch_step_v(const StepParams& a, const Coef<typename StoreT<S>::T>& c, bool gen, bool check,
                                 int check_blocks, cudaStream_t st) {
    const dim3 block(32, BY);
    const int64_t tiles = step_tiles(a.nx, a.ny, V);
    const unsigned int grid = (unsigned int)(check ? (tiles < check_blocks ? tiles : check_blocks) : tiles);
    if (gen)
        return check ? launch_after(k_step<S, V, true, true>, grid, block, 0, st, a, c)
                     : launch_after(k_step<S, V, true, false>, grid, block, 0, st, a, c);
    return check ? launch_after(k_step<S, V, false, true>, grid, block, 0, st, a, c)
                 : launch_after(k_step<S, V, false, false>, grid, block, 0, st, a, c);
}

template <int S>
cudaError_t Ops<S>::step(const StepParams& a, const Coef<T>& c, int V, bool gen, bool check,
                         int check_blocks, cudaStream_t st) {
    return V == 1 ? launch_step_v<S, 1>(a, c, gen, check, check_blocks, st)
                  : launch_step_v<S, max_vec<S>()>(a, c, gen, check, check_blocks, st);
}

template <int S>
cudaError_t Ops<S>::fields(const StepParams& a, const Coef<double>& c, T theta, const FieldOut& out,
                           cudaStream_t st) {
    return launch_after(k_fields<S>, step_grid(a.nx, a.ny, 1), dim3(32, BY), 0, st, a, c, theta, out);
}

template <int S>
cudaError_t Ops<S>::export_pop(const StepParams& a, T theta, double* out, cudaStream_t st) {
    k_export<S><<<step_grid(a.nx, a.ny, 1), dim3(32, BY), 0, st>>>(a, theta, out);
    return cudaGetLastError();
}

template <int S>
cudaError_t Ops<S>::import_pop(const StepParams& a, T theta, const double* in, cudaStream_t st) {
    k_import<S><<<step_grid(a.nx, a.ny, 1), dim3(32, BY), 0, st>>>(a, theta, in);
    return cudaGetLastError();
}

}  // namespace lbm
