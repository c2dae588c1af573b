// lbm_engine.cuh -- host side of the packed lattice arena: admission of
// problems into arena slots, chunks (strip launches, or a CUDA graph around the
// cooperative kernel of the other tile codes), per-problem residual bookkeeping, retirement and
// solution recovery.  Shared by lbm_batch_solve and the serving loop.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <string>
#include <vector>

#include "lbm_arena.cuh"

namespace lbm {

enum ProbState { P_FREE = 0, P_RUNNING = 1, P_DONE = 2 };

// Strip chunk: strips (FP32 five steps per launch, FP16S four), or two-step tiles
// (problems without ghost columns).
enum ProbClass { C_STRIPS = 0, C_PAIRS = 1, kClasses = 2 };

struct HostProb {
    int state = P_FREE;
    int nx = 0, ny = 0;            // the arena lattice (the caller's, or its transpose)
    bool tr = false;               // solved transposed (arena_transpose)
    int64_t n = 0;
    int pitch = 0, ghost = 0;      // row layout (ghost columns at either end, or none)
    int64_t plane = 0;             // elements between planes
    int cls = 0;                   // strip chunk: which launches advance it (ProbClass)
    bool ghosts_ok = true;         // the current state's ghost columns hold its images
    double lambda = 0.0, mu = 0.0;
    int64_t pop_off = -1, car_off = -1, fs_off = -1;
    int64_t pop_bytes = 0, car_bytes = 0, fs_bytes = 0;
    int parity = 0;
    int hexp = 0;
    float q11 = 0, qs = 0, qd = 0, qtheta = 0, theta = 0;   // rates in the quarter form of collide
    int64_t steps = 0;
    int64_t max_iters = 0;
    double tol = 0.0;
    bool snap_valid = false;
    bool check_now = false;    // the coming chunk checks this problem
    int period = 1;            // residual window = period chunks (adapt_period)
    int64_t last_check = 0;    // steps at the previous check
    double r_prev = 0.0;       // residual of the previous check
    int status = 0;            // lbm status when done
    double residual = 0.0;
    int64_t lups = 0;          // nodes x steps
};

class ArenaEngine {
public:
    ~ArenaEngine();
    // dtype: S_F32 or S_F16S.  Capacities in nodes (population / carrier /
    // force+snapshot bytes follow from the storage type); a problem with ghost
    // columns takes slots_for nodes, one laid out plainly its own.
    int init(int dtype, int64_t node_capacity, int max_probs, int check_every, cudaStream_t st,
             std::string* err);
    // Lay every problem out without ghost columns (before init).
    void set_plain() { plain_ = true; }
    int dtype() const { return dtype_; }
    int check_every() const { return k_; }
    // Bytes of device memory a problem of n nodes needs in this arena.
    int64_t bytes_for(int64_t n) const;
    // Nodes a problem takes with ghost columns (in the orientation it is solved in).
    static int64_t slots_for(int nx, int ny);
    // Admit a problem; returns slot >= 0, kNoRoom if it does not fit now, or a
    // negative lbm status on error.  gx, gy: host FP64, nx*ny each, read until
    // the stream has been waited for.  FP32: the force of a large problem is checked
    // later, by check_forces.
    static constexpr int kNoRoom = INT_MIN;
    int admit(int nx, int ny, double lambda, double mu, const double* gx, const double* gy,
              double tol, int64_t max_iters, std::string* err);
    // LBM_ERR_ARG if a problem admitted since init has a non-finite force entry
    // (small and FP16S problems are refused by admit already).
    int check_forces(std::string* err);
    // One chunk of check_every steps for every running problem, launched on the
    // engine's streams, and the wait for it; afterwards finished problems are in
    // state P_DONE (not yet released).  No other call between the two.
    int start_chunk(int V, std::string* err);
    int finish_chunk(int V, float* device_ms, std::string* err);
    int run_chunk(int V, float* device_ms, std::string* err) {
        if (device_ms) *device_ms = 0.0f;
        const int rc = start_chunk(V, err);
        return rc ? rc : finish_chunk(V, device_ms, err);
    }
    // Solution fields of count finished (or running) problems into host arrays,
    // FP64, lattice units; outs holds 5 nullable host arrays (ux, uy, sxx, syy,
    // sxy) per problem.
    int recover_many(int count, const int* slots, double* const* outs, std::string* err);
    void release(int slot);
    // Staging (doubles) that admissions of `most` nodes and a recovery of `fields` field
    // values in all (0: none), at most 5 * most of one problem, will not have to grow.
    int reserve_staging(int64_t most, int64_t fields, std::string* err) {
        return ensure_fields_buffer(std::max(2 * most, fields ? std::max(5 * most, std::min(fields, kRecoverBlock)) : 0), err);
    }
    const HostProb& prob(int slot) const { return probs_[slot]; }
    int running() const { return nrunning_; }
    int64_t running_tiles(int V) const;
    int64_t running_nodes() const;
    // Arena bytes held by admitted problems (running or finished, not released).
    int64_t resident_bytes() const;
    int max_probs() const { return (int)probs_.size(); }
    // Blocks of a chunk's launches (strip chunk: of the largest launch so far).
    int grid_blocks(int V) const;
    int64_t free_nodes_hint() const;
    int64_t device_bytes() const { return dev_bytes_; }
    cudaStream_t stream() const { return st_; }

private:
    template <typename T>
    cudaError_t device_alloc(T** p, int64_t bytes) {
        const cudaError_t e = cudaMalloc(p, bytes);
        if (e == cudaSuccess) dev_bytes_ += bytes;
        else *p = nullptr;
        return e;
    }
    template <typename T>
    void device_free(T** p, int64_t bytes) {
        cudaFree(*p);
        dev_bytes_ -= bytes;
        *p = nullptr;
    }
    // Problems are recovered in blocks of so many doubles (32 MB; a larger problem is a
    // block of its own).
    static constexpr int64_t kRecoverBlock = int64_t(4) << 20;
    int upload_tiles(int V, std::string* err);
    int choose_seg() const;
    int launch_strip_chunk(std::string* err);
    bool place(HostProb& p);
    void unplace(const HostProb& p);
    int admit_small(HostProb& p, int hx, const double* gx, const double* gy, std::string* err);
    int admit_large(HostProb& p, int hx, const double* gx, const double* gy, int slot, std::string* err);
    BatchArgs chunk_args() const;
    cudaError_t launch_fields(int slot, double* dst);
    int ensure_fields_buffer(int64_t len, std::string* err);
    int ensure_graph(int V, std::string* err);

    int dtype_ = S_F32;
    bool plain_ = false;
    int k_ = 100;
    cudaStream_t st_ = nullptr;
    int sms_ = 1;
    char* pop_[2] = {nullptr, nullptr};
    char* car_[2] = {nullptr, nullptr};
    char* fs_ = nullptr;
    RangeAllocator apop_, acar_, afs_;
    std::vector<HostProb> probs_;
    BatchProb* d_probs_ = nullptr;
    double* d_acc_ = nullptr;
    double* h_acc_ = nullptr;         // pinned
    uint2* d_tiles_ = nullptr;
    int64_t tiles_cap_ = 0;
    int* d_ntiles_ = nullptr;
    int class_begin_[kClasses + 1] = {};   // strip chunk: item ranges of the classes
    int pairs_grid_ = 0;                              // most blocks of the pairs' launch
    int strip_blocks_ = 0;                            // largest launch so far
    int ghosts_begin_ = 0, ghosts_end_ = 0;           // ... and of the problems whose ghost columns are stale
    cudaStream_t side_[kClasses - 1] = {};   // strips and narrow problems run side by side
    cudaEvent_t fork_ = nullptr, join_[kClasses - 1] = {};
    uint2* h_tiles_ = nullptr;        // pinned
    int64_t h_tiles_cap_ = 0;
    int tiles_V_ = 0;                 // V the device tile list was built for
    int wave_seg_ = 0;                // rows per strip item of the current list
    bool tiles_dirty_ = true;
    bool desc_dirty_ = true;
    float* h_force_ = nullptr;        // pinned: converted forces of small problems
    int64_t h_force_used_ = 0;        // ... since the stream was last waited for (floats)
    unsigned long long* d_stat_ = nullptr;   // per problem: max |g|, non-finite flag (ForceIn)
    double* d_fields_ = nullptr;      // FP64 staging: the caller's force, recovered fields
    int64_t d_fields_cap_ = 0;
    double* h_fields_ = nullptr;      // pinned: recovered fields of small problems
    int64_t h_fields_cap_ = 0;
    cudaGraphExec_t graph_[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    bool graph_failed_[6] = {false, false, false, false, false, false};
    cudaEvent_t ev0_ = nullptr, ev1_ = nullptr;
    int nrunning_ = 0;
    std::atomic<int64_t> dev_bytes_{0};   // (a server's statistics read it while the worker runs)
};

// Message for lbm_last_error() on this host thread; returns code.
int set_last_error(int code, const std::string& msg);

// Autotuner cache: tile width chosen for a workload signature.
int autotune_lookup(const std::string& key);
void autotune_store(const std::string& key, int V);

}  // namespace lbm
