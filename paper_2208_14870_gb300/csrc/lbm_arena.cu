// lbm_arena.cu -- the kernels of the packed lattice arena (see lbm_arena.cuh):
// strip items, and the persistent chunk kernels, one instantiation per storage
// type (FP32, FP16-shifted) and tile width.
#include <mutex>

#include "lbm_arena.cuh"

namespace lbm {

namespace cg = cooperative_groups;

constexpr int kArenaNW = 4;   // warps per block of the strip items

// The step parameters and rates of problem P, whose state lies in buffer src.
template <int S>
__device__ __forceinline__ StepParams prob_params(const BatchArgs& A, const BatchProb& P, int src) {
    StepParams a{};
    a.nx = P.nx;
    a.ny = P.ny;
    a.pitch = P.pitch;
    a.plane = P.plane;
    a.src = (src ? A.pop1 : A.pop0) + P.pop_off;
    a.dst = (src ? A.pop0 : A.pop1) + P.pop_off;
    if (S == S_F16S) {
        a.csrc = reinterpret_cast<const float*>((src ? A.car1 : A.car0) + P.car_off);
        a.cdst = reinterpret_cast<float*>((src ? A.car0 : A.car1) + P.car_off);
        a.hscale = P.hscale;
        a.hinv = P.hinv;
    }
    const float* force = reinterpret_cast<const float*>(A.fs + P.fs_off);
    a.gx = force;
    a.gy = force + P.plane;
    a.snap = A.fs + P.snap_off;
    return a;
}

__device__ __forceinline__ Coef<float> prob_coef(const BatchProb& P) {
    Coef<float> c{};
    c.q11 = P.q11;
    c.qs = P.qs;
    c.qd = P.qd;
    c.qtheta = P.qtheta;
    c.theta = P.theta;
    return c;
}

template <int S, int V, bool CHECK>
__device__ __forceinline__ void arena_tile(const BatchArgs& A, const BatchProb& P, int tile,
                                           int s, ResAcc<S>& acc) {
    const int ntx = (P.nx + 32 * V - 1) / (32 * V);
    const int ty = tile / ntx, tx = tile - ty * ntx;
    step_tile<S, V, false, CHECK>(prob_params<S>(A, P, (P.parity + s) & 1), prob_coef(P), tx, ty, acc);
}

// A problem's residual partials (maxima through the bit patterns of
// non-negative doubles).
__device__ __forceinline__ void add_to_problem(double* dst, const double w[kRes]) {
    unsigned long long* d = reinterpret_cast<unsigned long long*>(dst);
    atomicMax(d + 0, (unsigned long long)__double_as_longlong(w[0]));
    atomicMax(d + 1, (unsigned long long)__double_as_longlong(w[1]));
    atomicAdd(dst + 2, w[2]);
    atomicAdd(dst + 3, w[3]);
    atomicMax(d + 4, (unsigned long long)__double_as_longlong(w[4]));
}

// Block reduction of one tile's residual partials (converted to FP64 per
// thread) into the problem's FP64 accumulator.
template <int S>
__device__ __forceinline__ void tile_to_problem(const ResAcc<S>& acc, double* dst,
                                                double (*red)[32]) {
    const int tid = threadIdx.y * 32 + threadIdx.x;
    double v[kRes];
    acc.to_double(v);
    warp_reduce_res(v);
    block_reduce_res(v, red, tid, kThreads / 32);
    if (tid == 0) add_to_problem(dst, v);
    __syncthreads();
}

template <int S, int V>
__global__ void __launch_bounds__(kThreads, 2) k_arena_chunk(const BatchArgs A) {
    cg::grid_group grid = cg::this_grid();
    __shared__ double red[kRes][32];
    const int ntiles = *A.ntiles;
    for (int s = 0; s < A.nsteps; ++s) {
        const bool last = (s == A.nsteps - 1);
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
            const uint2 tl = A.tiles[t];
            const BatchProb P = A.probs[tl.x];
            const bool check = last && P.check;  // uniform over the block
            ResAcc<S> acc;
            if (!check) {
                arena_tile<S, V, false>(A, P, (int)tl.y, s, acc);
            } else {
                arena_tile<S, V, true>(A, P, (int)tl.y, s, acc);
                tile_to_problem<S>(acc, A.acc + (int64_t)tl.x * kRes, red);
            }
        }
        if (s + 1 < A.nsteps) grid.sync();
    }
}

// One tile of two steps (k_step2's tile) of problem P; s counts step pairs.
template <int S, bool CHECK>
__device__ __forceinline__ void arena_tile2(const BatchArgs& A, const BatchProb& P, int tile, int s,
                                            float* sm, ResAcc<S>& acc) {
    const int ntx = (P.nx + kT2OX - 1) / kT2OX;
    const int ty = tile / ntx, tx = tile - ty * ntx;
    step2_tile<S, false, CHECK, true>(prob_params<S>(A, P, (P.parity + s) & 1), prob_coef(P), sm, tx, ty, acc);
}

// The chunk with two steps per tile visit and one grid barrier per pair of
// steps (nsteps even); the residual check rides on the second step of the
// chunk's last pair.
template <int S>
__global__ void __launch_bounds__(kT2Threads, 2) k_arena_chunk2(const BatchArgs A) {
    cg::grid_group grid = cg::this_grid();
    extern __shared__ float t2_smem[];
    __shared__ double red[kRes][32];
    const int ntiles = *A.ntiles;
    const int npairs = A.nsteps / 2;
    for (int s = 0; s < npairs; ++s) {
        const bool last = (s == npairs - 1);
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
            const uint2 tl = A.tiles[t];
            const BatchProb P = A.probs[tl.x];
            const bool check = last && P.check;  // uniform over the block
            ResAcc<S> acc;
            if (!check) {
                arena_tile2<S, false>(A, P, (int)tl.y, s, t2_smem, acc);
            } else {
                arena_tile2<S, true>(A, P, (int)tl.y, s, t2_smem, acc);
                tile_to_problem<S>(acc, A.acc + (int64_t)tl.x * kRes, red);
            }
            __syncthreads();   // the slots are reused by the block's next tile
        }
        if (s + 1 < npairs) grid.sync();
    }
}

// T steps of the listed strip items, one warp each: item (problem, i) is strip
// i mod strips, segment i / strips of P.seg rows.
template <int S, int T, bool CHECK>
__global__ void __launch_bounds__(32 * kArenaNW, 3)
k_arena_strips(const BatchArgs A, const uint2* items, int count, int group) {
    extern __shared__ float4 strip_mem[];
    const int warp = threadIdx.x >> 5, item = (int)blockIdx.x * kArenaNW + warp;
    if (item >= count) return;
    // (items and problems are written by copies, which no launch overtakes)
    const uint2 tl = items[item];
    const BatchProb P = A.probs[tl.x];
    const StepParams a = prob_params<S>(A, P, (P.parity + group) & 1);
    const PairCoef c = pair_coef(prob_coef(P));
    const int ns = (P.nx + kArenaOX - 1) / kArenaOX;
    const int strip = (int)tl.y % ns, y0 = (int)tl.y / ns * P.seg, rows = min(P.seg, P.ny - y0);
    const uint32_t sm = (uint32_t)__cvta_generic_to_shared(strip_mem) + warp * st_warp_smem<S, T, CHECK>();
    ResAcc2 acc;
    if (CHECK && P.check) {
        strip_walk<S, false, T, true, kArenaOX>(a, c, sm, strip, y0, rows, acc, P.half != 0);
        double w[kRes];
        acc.to_double(w);
        warp_reduce_res(w);
        if ((threadIdx.x & 31) == 0) add_to_problem(A.acc + (int64_t)tl.x * kRes, w);
    } else {
        strip_walk<S, false, T, false, kArenaOX>(a, c, sm, strip, y0, rows, acc, P.half != 0);
    }
}

// Ghost columns of the listed problems' current states, one block each.
template <int S>
__global__ void __launch_bounds__(256) k_arena_ghosts(const BatchArgs A, const uint2* items) {
    after_predecessor();
    const BatchProb P = A.probs[items[blockIdx.x].x];
    fill_ghosts<S>(prob_params<S>(A, P, P.parity ^ 1), threadIdx.x, blockDim.x);   // (dst: the current state)
}

__global__ void __launch_bounds__(256) k_arena_force(const ForceIn f) {
    double m = 0.0;
    unsigned int bad = 0;
    const int64_t n = (int64_t)f.nx * f.ny;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t y = i / f.nx;
        const int x = (int)(i - y * f.nx);
        const int64_t h = f.tr ? (int64_t)x * f.hx + y : y * f.hx + x;
        const double u = f.gx[h], v = f.gy[h];
        if (!(isfinite(u) && isfinite(v))) bad = 1;
        m = fmax(m, fmax(fabs(u), fabs(v)));
        float* o = f.out + y * f.pitch + f.ghost + x;
        const float gx = (float)(f.tr ? v : u) * f.scale, gy = (float)(f.tr ? u : v) * f.scale;
        o[0] = gx;
        o[f.plane] = gy;
        if (x < f.ghost) {
            o[f.nx] = gx;
            o[f.plane + f.nx] = gy;
        }
        if (x >= f.nx - f.ghost) {
            o[-f.nx] = gx;
            o[f.plane - f.nx] = gy;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(f.stat, (unsigned long long)__double_as_longlong(m));
        if (bad) atomicOr(f.stat + 1, 1ULL);
    }
}

cudaError_t launch_arena_force(const ForceIn& f, cudaStream_t st) {
    const int64_t n = (int64_t)f.nx * f.ny, blocks = (n + 1023) / 1024;
    k_arena_force<<<(unsigned)(blocks < 2048 ? blocks : 2048), 256, 0, st>>>(f);
    return cudaGetLastError();
}

// A kernel's dynamic shared memory above 48 KB, allowed once per device.
template <auto* KERNEL>
static cudaError_t allow_smem_once(int bytes) {
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    done[dev] = e == cudaSuccess;
    return e;
}

template <int S, int T, bool CHECK>
static cudaError_t launch_strips_k(const BatchArgs& a, const uint2* items, int count, int group, cudaStream_t st) {
    constexpr int SM = kArenaNW * st_warp_smem<S, T, CHECK>();
    const auto kernel = k_arena_strips<S, T, CHECK>;
    const cudaError_t e = allow_smem_once<k_arena_strips<S, T, CHECK>>(SM);
    if (e != cudaSuccess) return e;
    return launch_after(kernel, dim3((unsigned)((count + kArenaNW - 1) / kArenaNW)), dim3(32 * kArenaNW), SM, st, a, items,
                        count, group);
}

cudaError_t launch_arena_strips(int dtype, int T, bool check, const BatchArgs& a, const uint2* items, int count,
                                int group, cudaStream_t st) {
    if (dtype == S_F16S) {
        if (T == 4)
            return check ? launch_strips_k<S_F16S, 4, true>(a, items, count, group, st)
                         : launch_strips_k<S_F16S, 4, false>(a, items, count, group, st);
        return cudaErrorInvalidValue;
    }
    if (check) {
        if (T == 5) return launch_strips_k<S_F32, 5, true>(a, items, count, group, st);
        return T == 4 ? launch_strips_k<S_F32, 4, true>(a, items, count, group, st) : cudaErrorInvalidValue;
    }
    switch (T) {
        case 2: return launch_strips_k<S_F32, 2, false>(a, items, count, group, st);
        case 3: return launch_strips_k<S_F32, 3, false>(a, items, count, group, st);
        case 5: return launch_strips_k<S_F32, 5, false>(a, items, count, group, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_arena_ghosts(int dtype, const BatchArgs& a, const uint2* items, int count, cudaStream_t st) {
    return dtype == S_F16S ? launch_after(k_arena_ghosts<S_F16S>, dim3((unsigned)count), dim3(256), 0, st, a, items)
                           : launch_after(k_arena_ghosts<S_F32>, dim3((unsigned)count), dim3(256), 0, st, a, items);
}

template <int S>
static cudaError_t t2_arena_allow_smem() {
    return cudaFuncSetAttribute(k_arena_chunk2<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, kT2Smem);
}

template <int S>
static cudaError_t launch_two_step(const BatchArgs& a, int grid, cudaStream_t st) {
    if (a.nsteps % 2) return cudaErrorInvalidValue;
    cudaError_t e = t2_arena_allow_smem<S>();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kT2Threads);
    cfg.dynamicSmemBytes = kT2Smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_arena_chunk2<S>, a);
}

template <int S, int V>
static cudaError_t launch_v(const BatchArgs& a, int grid, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(32, BY);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_arena_chunk<S, V>, a);
}

cudaError_t launch_arena_chunk(int dtype, int V, const BatchArgs& a, int grid, cudaStream_t st) {
    if (V == kTileTwoStep)
        return dtype == S_F16S ? launch_two_step<S_F16S>(a, grid, st) : launch_two_step<S_F32>(a, grid, st);
    if (dtype == S_F16S) {
        switch (V) {
            case 1: return launch_v<S_F16S, 1>(a, grid, st);
            case 2: return launch_v<S_F16S, 2>(a, grid, st);
            case 4: return launch_v<S_F16S, 4>(a, grid, st);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (V) {
        case 1: return launch_v<S_F32, 1>(a, grid, st);
        case 2: return launch_v<S_F32, 2>(a, grid, st);
        case 4: return launch_v<S_F32, 4>(a, grid, st);
        default: return cudaErrorInvalidValue;
    }
}

template <int S, int V>
static int occ() {
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_arena_chunk<S, V>, kThreads, 0);
    return b;
}

template <int S>
static int occ2() {
    if (t2_arena_allow_smem<S>() != cudaSuccess) return 0;
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_arena_chunk2<S>, kT2Threads, kT2Smem);
    return b;
}

int arena_occupancy(int dtype, int V) {
    if (V == kTileTwoStep) return dtype == S_F16S ? occ2<S_F16S>() : occ2<S_F32>();
    if (dtype == S_F16S) return V == 1 ? occ<S_F16S, 1>() : V == 2 ? occ<S_F16S, 2>() : occ<S_F16S, 4>();
    return V == 1 ? occ<S_F32, 1>() : V == 2 ? occ<S_F32, 2>() : occ<S_F32, 4>();
}

}  // namespace lbm
