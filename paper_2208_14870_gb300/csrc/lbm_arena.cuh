// lbm_arena.cuh -- packed lattice arena for many independent periodic
// problems of uneven sizes and material parameters, advanced together in
// chunks of k steps.
//
// Every problem p owns, in three device buffers,
//   pop[0], pop[1] : its 8 population planes (ping-pong; FP32 or FP16),
//   car[0], car[1] : FP16-shifted only: the two FP32 carriers, one float2 per node,
//   fs             : force (2 FP32 planes) then residual snapshot (2 planes of
//                    (hi, lo) FP32 pairs),
// placed by a first-fit allocator (256-byte aligned).  Rows carry ghost columns
// (row_ghost) where the strips run; a problem that fits the arena only without
// them is laid out plainly.
//
// The strip chunk (kTileWave) launches one kernel per group of steps over the
// (problem, strip, segment) items of all running problems, one warp per item;
// the other tile codes, and the problems too narrow for strips, run a chunk in one persistent cooperative kernel that
// walks the (problem, tile) list grid-stride and synchronises the grid between
// steps.  The last step of a chunk carries the residual check for the problems
// flagged in their descriptor (a problem checks every `check_period` chunks of
// its own steps); its per-problem partial sums go to per-problem FP64
// accumulators with atomics.  The host reads them after the chunk, retires
// converged problems, admits new ones and rebuilds the item lists between
// chunks.
#pragma once

#include <cooperative_groups.h>

#include <map>
#include <string>
#include <vector>

#include "lbm_kernels.cuh"

namespace lbm {

struct BatchProb {
    int64_t pop_off;   // bytes into each population buffer, of column 0
    int64_t car_off;   // bytes into each carrier buffer (F16S)
    int64_t fs_off;    // bytes into the force/snapshot buffer: force planes
    int64_t snap_off;  // ... and snapshot planes
    int64_t plane;     // elements between planes
    int nx, ny, pitch, check, dtype, parity;   // check: this chunk's last step checks
    int seg;                            // strip chunk: rows per item
    int half;                           // ... FP16S: the state is rounded after every second step
    float q11, qs, qd, qtheta, theta, hscale, hinv;   // rates in the quarter form of collide
};

struct BatchArgs {
    const BatchProb* probs;
    const uint2* tiles;        // (problem, tile)
    const int* ntiles;         // device scalar: number of valid tiles
    char* pop0;
    char* pop1;
    char* car0;
    char* car1;
    char* fs;
    double* acc;               // kRes doubles per problem
    int nsteps;
};

constexpr int kArenaAlign = 256;

// First-fit allocator over [0, capacity) with coalescing of free ranges.
class RangeAllocator {
public:
    void reset(int64_t capacity) {
        free_.clear();
        if (capacity > 0) free_[0] = capacity;
        cap_ = capacity;
    }
    int64_t capacity() const { return cap_; }
    // returns offset or -1
    int64_t alloc(int64_t bytes) {
        bytes = (bytes + kArenaAlign - 1) / kArenaAlign * kArenaAlign;
        for (auto it = free_.begin(); it != free_.end(); ++it) {
            if (it->second >= bytes) {
                const int64_t off = it->first, rest = it->second - bytes;
                free_.erase(it);
                if (rest > 0) free_[off + bytes] = rest;
                return off;
            }
        }
        return -1;
    }
    void release(int64_t off, int64_t bytes) {
        bytes = (bytes + kArenaAlign - 1) / kArenaAlign * kArenaAlign;
        auto it = free_.emplace(off, bytes).first;
        auto nx = std::next(it);
        if (nx != free_.end() && it->first + it->second == nx->first) {
            it->second += nx->second;
            free_.erase(nx);
        }
        if (it != free_.begin()) {
            auto pv = std::prev(it);
            if (pv->first + pv->second == it->first) {
                pv->second += it->second;
                free_.erase(it);
            }
        }
    }
    int64_t largest_free() const {
        int64_t m = 0;
        for (auto& kv : free_) m = kv.second > m ? kv.second : m;
        return m;
    }

private:
    std::map<int64_t, int64_t> free_;
    int64_t cap_ = 0;
};

// Tile code of two-step tiles: the 62 x 22-node tiles of k_step2, two steps
// per tile visit and one grid barrier per pair of steps (chunk length even).
constexpr int kTileTwoStep = 3;

// Tile code of the strip chunk: every launch advances the listed items by a
// group of steps (FP32 five; FP16S four, of which lattices below 256 x 8 round
// their state after the second one too: in launches of their own, two steps each,
// 12 small problems of a server took 1.08 ms per 100 steps instead of 0.94).  Strips have
// kArenaOX output columns whatever the group, so that one item list serves a
// chunk; problems without ghost columns take pairs of steps on two-step tiles, all of a
// chunk's in one cooperative launch beside the strips (a launch per pair: 100
// problems of sides 8 to 64 1.13 against 0.89 ms per 400 steps, FP16S 1.51 against 1.21; 50 of
// sides 4 to 15 alone 0.73 against 0.78).
// Chunk lengths: multiples of 4.
constexpr int kTileWave = 5;
constexpr int kArenaOX = 56;
inline int64_t arena_strips(int nx) { return (nx + kArenaOX - 1) / kArenaOX; }

inline bool arena_wide(int nx, int ny) { return wave_fits(nx, ny) && (int64_t)nx * ny < (int64_t(1) << 31); }
// Problems the strips run on: ghost columns (images of distinct columns).
inline bool arena_padded(int nx) { return nx >= 2 * kGhost; }
inline int arena_pitch(int nx) { return (nx + 2 * kGhost + 7) / 8 * 8; }

// Weight of solving an nx x ny problem as given against its transpose: columns
// of 256-column strips with 250 outputs for lattices from 256 x 8 on, slots of
// two-step tiles at about half that rate for smaller ones.  A fixed rule: the
// choice decides the rounding order of the solution and is reported with it.
inline double arena_cost(int nx, int ny) {
    if (arena_wide(nx, ny)) return double((nx + 249) / 250) * 256 / nx;
    return 1.94 * (double((nx + kT2OX - 1) / kT2OX) * kT2W / nx) * (double((ny + kT2OY - 1) / kT2OY) * kT2H / ny);
}

// Solve a problem on its transpose (x and y exchanged) where that is clearly
// cheaper.  The scheme is symmetric under the exchange (velocities (c_x, c_y)
// -> (c_y, c_x) map the moments 10 <-> 01, 12 <-> 21, s -> s, d -> -d, 11 ->
// 11, 22 -> 22 onto each other; Table 1 and the rates with w_12 = w_21 follow),
// so the transposed problem's solution is the solution's transpose with u_x
// <-> u_y and sigma_xx <-> sigma_yy; only the rounding order differs.
inline bool arena_transpose(int nx, int ny) { return arena_cost(ny, nx) < 0.95 * arena_cost(nx, ny); }

// Number of tiles of an nx x ny problem for the persistent kernels' tile codes.
inline int64_t arena_tiles(int nx, int ny, int V) {
    return V == kTileTwoStep ? step2_tiles(nx, ny) : step_tiles(nx, ny, V);
}

// Launch one chunk of a persistent kernel: nsteps steps of every listed tile
// (all of storage type dtype: S_F32 or S_F16S), residual check fused into the
// last step.  Tile code V: width 32*V for V in {1, 2, 4}, or kTileTwoStep.
// Cooperative launch: grid must not exceed arena_occupancy(dtype, V) x SM
// count.
cudaError_t launch_arena_chunk(int dtype, int V, const BatchArgs& a, int grid, cudaStream_t st);
// Resident blocks per SM of the chunk kernel.
int arena_occupancy(int dtype, int V);

// The strip chunk's launches.  T steps of `count` strip items (check: the last
// step checks the flagged problems); the ghost columns of `count` problems (items:
// problem numbers).  group: how many groups of steps of its problems ran before in
// this chunk (buffer parity).
cudaError_t launch_arena_strips(int dtype, int T, bool check, const BatchArgs& a, const uint2* items, int count,
                                int group, cudaStream_t st);
// A problem's force from the caller's FP64 arrays (device memory, hx columns per
// row) into its FP32 planes of `plane` elements: rows of nx columns with their
// ghost columns, transposed with the components exchanged for a problem solved
// on its transpose.  stat[0]: max |g| (bit pattern of a non-negative double),
// stat[1]: non-zero for a non-finite entry; both zero before.
struct ForceIn {
    const double *gx, *gy;
    int hx, tr;
    float* out;                // row 0, first ghost column
    int nx, ny, pitch, ghost;
    int64_t plane;
    float scale;               // of the converted force (a power of two)
    unsigned long long* stat;
};
cudaError_t launch_arena_force(const ForceIn& f, cudaStream_t st);
cudaError_t launch_arena_ghosts(int dtype, const BatchArgs& a, const uint2* items, int count, cudaStream_t st);

}  // namespace lbm
