// lbm_engine.cu -- host side of the packed lattice arena (lbm_engine.cuh).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <memory>
#include <mutex>
#include <new>
#include <sstream>
#include <sys/stat.h>

#include "../../include/lbm.h"
#include "lbm_engine.cuh"

static_assert(lbm::kTileTwoStep == LBM_TILE_TWO_STEP, "tile code of two-step tiles");
static_assert(lbm::kTileWave == LBM_TILE_WAVE, "tile code of the strip chunk");

namespace lbm {

namespace {

int cuerr(cudaError_t e, const char* what, std::string* err) {
    if (err) *err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
}

#define ECK(call)                                                 \
    do {                                                          \
        cudaError_t e_ = (call);                                  \
        if (e_ != cudaSuccess) return cuerr(e_, #call, err);      \
    } while (0)

int64_t pop_bytes_per_node(int dtype) { return dtype == S_F16S ? 8 * 2 : 8 * 4; }
int64_t car_bytes_per_node(int dtype) { return dtype == S_F16S ? 2 * 4 : 0; }
// Copies between the caller's arrays and the device.  The runtime refuses host
// ranges that are pinned in part, or in several parts (arrays that follow one
// another, pinned each by itself): these go through memory of our own.
constexpr size_t kBounce = size_t(16) << 20;
cudaError_t copy_in(void* dst, const void* src, size_t bytes, cudaStream_t st) {
    cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
    if (e != cudaErrorInvalidValue) return e;
    cudaGetLastError();
    const std::unique_ptr<char[]> own(new (std::nothrow) char[std::min(bytes, kBounce)]);
    if (!own) return cudaErrorMemoryAllocation;
    e = cudaSuccess;
    for (size_t at = 0; at < bytes && e == cudaSuccess; at += kBounce) {
        const size_t len = std::min(bytes - at, kBounce);
        std::memcpy(own.get(), static_cast<const char*>(src) + at, len);
        e = cudaMemcpyAsync(static_cast<char*>(dst) + at, own.get(), len, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    return e;
}
cudaError_t copy_out(void* dst, const void* src, size_t bytes, cudaStream_t st) {
    cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, st);
    if (e != cudaErrorInvalidValue) return e;
    cudaGetLastError();
    const std::unique_ptr<char[]> own(new (std::nothrow) char[std::min(bytes, kBounce)]);
    if (!own) return cudaErrorMemoryAllocation;
    e = cudaSuccess;
    for (size_t at = 0; at < bytes && e == cudaSuccess; at += kBounce) {
        const size_t len = std::min(bytes - at, kBounce);
        e = cudaMemcpyAsync(own.get(), static_cast<const char*>(src) + at, len, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e == cudaSuccess) std::memcpy(static_cast<char*>(dst) + at, own.get(), len);
    }
    return e;
}
// force (2 FP32 planes) + residual snapshot (2 planes of (hi, lo) FP32 pairs)
constexpr int64_t kFsBytesPerNode = 2 * 4 + 2 * 8;

}  // namespace

ArenaEngine::~ArenaEngine() {
    if (st_) cudaStreamSynchronize(st_);
    for (auto& g : graph_)
        if (g) cudaGraphExecDestroy(g);
    for (int i = 0; i < 2; ++i) {
        if (pop_[i]) cudaFree(pop_[i]);
        if (car_[i]) cudaFree(car_[i]);
    }
    if (fs_) cudaFree(fs_);
    if (d_probs_) cudaFree(d_probs_);
    if (d_acc_) cudaFree(d_acc_);
    if (d_tiles_) cudaFree(d_tiles_);
    if (d_ntiles_) cudaFree(d_ntiles_);
    if (d_fields_) cudaFree(d_fields_);
    if (d_stat_) cudaFree(d_stat_);
    if (h_acc_) cudaFreeHost(h_acc_);
    if (h_tiles_) cudaFreeHost(h_tiles_);
    if (h_force_) cudaFreeHost(h_force_);
    if (h_fields_) cudaFreeHost(h_fields_);
    for (int i = 0; i < kClasses - 1; ++i) {
        if (side_[i]) cudaStreamDestroy(side_[i]);
        if (join_[i]) cudaEventDestroy(join_[i]);
    }
    if (fork_) cudaEventDestroy(fork_);
    if (ev0_) cudaEventDestroy(ev0_);
    if (ev1_) cudaEventDestroy(ev1_);
}

int64_t ArenaEngine::slots_for(int nx, int ny) {
    if (arena_transpose(nx, ny)) std::swap(nx, ny);
    return arena_padded(nx) ? (int64_t)arena_pitch(nx) * ny : (int64_t)nx * ny;
}

int64_t ArenaEngine::bytes_for(int64_t n) const {
    auto al = [](int64_t b) { return (b + kArenaAlign - 1) / kArenaAlign * kArenaAlign; };
    return 2 * al(pop_bytes_per_node(dtype_) * n) + 2 * al(car_bytes_per_node(dtype_) * n) +
           al(kFsBytesPerNode * n);
}

int ArenaEngine::init(int dtype, int64_t node_capacity, int max_probs, int check_every,
                      cudaStream_t st, std::string* err) {
    if (dtype != S_F32 && dtype != S_F16S) {
        if (err) *err = "arena: storage must be LBM_F32 or LBM_F16S";
        return LBM_ERR_ARG;
    }
    dtype_ = dtype;
    k_ = check_every;
    st_ = st;
    int dev = 0;
    ECK(cudaGetDevice(&dev));
    ECK(cudaDeviceGetAttribute(&sms_, cudaDevAttrMultiProcessorCount, dev));
    // a strip of the last problem reads past its last row: that much of every
    // buffer is not given out
    const int64_t over = kRowSlack * 8, slack = (int64_t)max_probs * kArenaAlign + over;
    const int64_t pb = pop_bytes_per_node(dtype) * node_capacity + slack;
    const int64_t cb = car_bytes_per_node(dtype) * node_capacity + slack;
    const int64_t fb = kFsBytesPerNode * node_capacity + slack;
    for (int i = 0; i < 2; ++i) {
        ECK(device_alloc(&pop_[i], pb));
        if (dtype == S_F16S) ECK(device_alloc(&car_[i], cb));
    }
    ECK(device_alloc(&fs_, fb));
    apop_.reset(pb - over);
    acar_.reset(dtype == S_F16S ? cb - over : 0);
    afs_.reset(fb - over);
    probs_.assign(max_probs, HostProb());
    ECK(device_alloc(&d_probs_, sizeof(BatchProb) * max_probs));
    ECK(device_alloc(&d_acc_, sizeof(double) * kRes * max_probs));
    ECK(cudaMallocHost(&h_acc_, sizeof(double) * kRes * max_probs));
    ECK(device_alloc(&d_stat_, 2 * sizeof(unsigned long long) * max_probs));
    ECK(cudaMemsetAsync(d_stat_, 0, 2 * sizeof(unsigned long long) * max_probs, st_));
    ECK(device_alloc(&d_ntiles_, 2 * sizeof(int)));
    ECK(cudaMemsetAsync(d_ntiles_, 0, 2 * sizeof(int), st_));
    for (int i = 0; i < kClasses - 1; ++i) {
        ECK(cudaStreamCreateWithFlags(&side_[i], cudaStreamNonBlocking));
        ECK(cudaEventCreateWithFlags(&join_[i], cudaEventDisableTiming));
    }
    ECK(cudaEventCreateWithFlags(&fork_, cudaEventDisableTiming));
    ECK(cudaEventCreate(&ev0_));
    ECK(cudaEventCreate(&ev1_));
    return LBM_OK;
}

// Arena memory for p (its lattice set), with ghost columns where the strips run,
// or without them if the arena could never hold it with them.
bool ArenaEngine::place(HostProb& p) {
    for (int plain = arena_padded(p.nx) && !plain_ ? 0 : 1; plain < 2; ++plain) {
        p.ghost = plain ? 0 : kGhost;
        p.pitch = plain ? p.nx : arena_pitch(p.nx);
        p.plane = (int64_t)p.pitch * p.ny;
        p.pop_bytes = pop_bytes_per_node(dtype_) * p.plane;
        p.car_bytes = car_bytes_per_node(dtype_) * p.plane;
        p.fs_bytes = kFsBytesPerNode * p.plane;
        if (!plain && (p.pop_bytes > apop_.capacity() || p.car_bytes > acar_.capacity() || p.fs_bytes > afs_.capacity()))
            continue;
        p.pop_off = apop_.alloc(p.pop_bytes);
        if (p.pop_off < 0) return false;
        p.car_off = dtype_ == S_F16S ? acar_.alloc(p.car_bytes) : 0;
        if (p.car_off < 0) {
            apop_.release(p.pop_off, p.pop_bytes);
            return false;
        }
        p.fs_off = afs_.alloc(p.fs_bytes);
        if (p.fs_off < 0) {
            apop_.release(p.pop_off, p.pop_bytes);
            if (dtype_ == S_F16S) acar_.release(p.car_off, p.car_bytes);
            return false;
        }
        return true;
    }
    return false;
}

void ArenaEngine::unplace(const HostProb& p) {
    apop_.release(p.pop_off, p.pop_bytes);
    if (dtype_ == S_F16S) acar_.release(p.car_off, p.car_bytes);
    afs_.release(p.fs_off, p.fs_bytes);
}

// A small problem, of at most so many nodes: its force is converted on the host, into
// pinned memory: three calls of the runtime per admission (FP16S four) instead of
// six.  200 problems of sides 4 to 31 on a server, 400 steps: 10.9 -> 10.0 ms; 100 of
// sides 16 to 64 7.50 -> 7.11 (up to 1024 nodes 7.35, up to 16384 7.02).
constexpr int64_t kSmall = 4096;
constexpr int64_t kForceStage = int64_t(1) << 18;      // floats (a problem of 4096 nodes takes at most 2 * 2 * 4096)
// Problems of at most so many nodes are recovered many to a copy (recover_many).
constexpr int64_t kSmallFields = 2048;
constexpr int64_t kFieldStage = int64_t(1) << 18;      // doubles
// Up to so many nodes the host looks for max |g| (FP16S): 16 bytes per node to read,
// against some 15 us for the device's answer.
constexpr int64_t kHostMax = 16384;

// Max |g| of both components, infinite or NaN if an entry is not finite (of the bit
// patterns of |g|, which order like the values).
static double force_max(const double* gx, const double* gy, int64_t n) {
    uint64_t m = 0;
    for (const double* g : {gx, gy})
        for (int64_t i = 0; i < n; ++i) {
            uint64_t b;
            std::memcpy(&b, g + i, sizeof b);
            m = std::max<uint64_t>(m, b & 0x7fffffffffffffffULL);
        }
    double gmax;
    std::memcpy(&gmax, &m, sizeof gmax);
    return gmax;
}

// The force planes of a placed problem, whose snapshot is cleared; converted on the
// host (finite, hexp set).  hx: columns of the caller's arrays.
int ArenaEngine::admit_small(HostProb& p, int hx, const double* gx, const double* gy, std::string* err) {
    const int64_t len = 2 * p.plane;
    if (!h_force_) ECK(cudaMallocHost(&h_force_, sizeof(float) * kForceStage));
    if (h_force_used_ + len > kForceStage) {
        ECK(cudaStreamSynchronize(st_));
        h_force_used_ = 0;
    }
    float* h = h_force_ + h_force_used_;
    h_force_used_ += len;
    std::memset(h, 0, sizeof(float) * len);
    const float scale = std::ldexp(1.0f, p.hexp);
    for (int c = 0; c < 2; ++c) {
        const double* g = (c == 0) == p.tr ? gy : gx;      // (transposed: components exchanged)
        for (int y = 0; y < p.ny; ++y) {
            float* row = h + c * p.plane + (int64_t)y * p.pitch + p.ghost;
            if (p.tr)
                for (int x = 0; x < p.nx; ++x) row[x] = (float)g[(int64_t)x * hx + y] * scale;
            else
                for (int x = 0; x < p.nx; ++x) row[x] = (float)g[(int64_t)y * hx + x] * scale;
            for (int x = 0; x < p.ghost; ++x) {
                row[p.nx + x] = row[x];
                row[x - p.ghost] = row[p.nx + x - p.ghost];
            }
        }
    }
    ECK(cudaMemcpyAsync(fs_ + p.fs_off, h, sizeof(float) * len, cudaMemcpyHostToDevice, st_));
    ECK(cudaMemsetAsync(fs_ + p.fs_off + sizeof(float) * len, 0, p.fs_bytes - sizeof(float) * len, st_));
    return LBM_OK;
}

// The same on the device, from a copy of the caller's arrays (in the caller's units
// and unchecked, but for FP16S up to kHostMax nodes).
int ArenaEngine::admit_large(HostProb& p, int hx, const double* gx, const double* gy, int slot, std::string* err) {
    const int64_t n = p.n, len = 2 * p.plane;
    // (staged where the fields are)
    const int rc = ensure_fields_buffer(std::max<int64_t>(2 * n, int64_t(1) << 20), err);
    if (rc) return rc;
    unsigned long long* stat = d_stat_ + 2 * slot;
    float* force = reinterpret_cast<float*>(fs_ + p.fs_off);
    ECK(copy_in(d_fields_, gx, sizeof(double) * n, st_));
    ECK(copy_in(d_fields_ + n, gy, sizeof(double) * n, st_));
    ECK(cudaMemsetAsync(stat, 0, 2 * sizeof(unsigned long long), st_));
    ECK(cudaMemsetAsync(force, 0, p.fs_bytes, st_));
    ForceIn f{};
    f.gx = d_fields_;
    f.gy = d_fields_ + n;
    f.hx = hx;
    f.tr = p.tr ? 1 : 0;
    f.out = force;
    f.nx = p.nx;
    f.ny = p.ny;
    f.pitch = p.pitch;
    f.ghost = p.ghost;
    f.plane = p.plane;
    f.stat = stat;
    f.scale = std::ldexp(1.0f, p.hexp);
    ECK(launch_arena_force(f, st_));
    if (dtype_ != S_F16S || n <= kHostMax) return LBM_OK;
    unsigned long long got[2];
    ECK(cudaMemcpyAsync(got, stat, sizeof(got), cudaMemcpyDeviceToHost, st_));
    ECK(cudaStreamSynchronize(st_));
    double gmax;
    std::memcpy(&gmax, &got[0], sizeof(double));
    if (got[1]) {
        if (err) *err = "admit: non-finite force";
        return LBM_ERR_ARG;
    }
    p.hexp = f16s_exponent(gmax, p.nx, p.ny);
    if (p.hexp != 0) {
        k_scale_float<<<256, 256, 0, st_>>>(force, len, std::ldexp(1.0f, p.hexp));
        ECK(cudaGetLastError());
    }
    return LBM_OK;
}

int ArenaEngine::admit(int nx, int ny, double lambda, double mu, const double* gx, const double* gy,
                       double tol, int64_t max_iters, std::string* err) {
    if (nx < 1 || ny < 1 || !gx || !gy || !(mu > 0.0) || !(lambda + mu > 0.0) ||
        !std::isfinite(lambda) || !std::isfinite(mu)) {
        if (err) *err = "admit: bad problem (sizes, moduli or null force)";
        return LBM_ERR_ARG;
    }
    int slot = -1;
    for (int i = 0; i < (int)probs_.size(); ++i)
        if (probs_[i].state == P_FREE) {
            slot = i;
            break;
        }
    if (slot < 0) return kNoRoom;
    const int64_t n = (int64_t)nx * ny;
    // a problem that is cheaper on its transpose is solved there: lattice
    // ny x nx, force components exchanged, node (x, y) at x * ny + y
    const bool tr = arena_transpose(nx, ny);
    HostProb p;
    p.nx = tr ? ny : nx;
    p.ny = tr ? nx : ny;
    p.tr = tr;
    p.n = n;
    if (!place(p)) return kNoRoom;
    // FP16S keeps its state, the force included, in units scaled by 2^hexp from
    // max |g| (store_f16s)
    if (n <= (dtype_ == S_F16S ? kHostMax : kSmall)) {
        const double gmax = force_max(gx, gy, n);
        if (!std::isfinite(gmax)) {
            unplace(p);
            if (err) *err = "admit: non-finite force";
            return LBM_ERR_ARG;
        }
        if (dtype_ == S_F16S) p.hexp = f16s_exponent(gmax, p.nx, p.ny);
    }
    const int rc = n <= kSmall ? admit_small(p, nx, gx, gy, err) : admit_large(p, nx, gx, gy, slot, err);
    if (rc) {
        unplace(p);
        return rc;
    }
    ECK(cudaMemsetAsync(pop_[0] + p.pop_off, 0, p.pop_bytes, st_));
    if (dtype_ == S_F16S) ECK(cudaMemsetAsync(car_[0] + p.car_off, 0, p.car_bytes, st_));
    p.parity = 0;
    p.cls = p.ghost ? C_STRIPS : C_PAIRS;
    p.lambda = lambda;
    p.mu = mu;
    // Table 1 / Eq. relaxation_rate with theta = 1/3, w_12 = w_21 = w_22 = 1
    const double theta = 1.0 / 3.0, K = lambda + mu;
    p.theta = (float)theta;
    p.qtheta = (float)(0.25 * theta);   // quarter form of collide
    p.q11 = (float)(0.25 * (1.0 - 1.0 / (mu / theta + 0.5)));
    p.qs = (float)(0.25 * (1.0 - 1.0 / (2.0 * K / (1.0 + theta) + 0.5)));
    p.qd = (float)(0.25 * (1.0 - 1.0 / (2.0 * mu / (1.0 - theta) + 0.5)));
    p.tol = tol;
    p.max_iters = max_iters;
    p.period = check_period(dtype_, tol, k_, std::min(nx, ny));
    p.r_prev = INFINITY;
    p.last_check = 0;
    p.state = P_RUNNING;
    probs_[slot] = p;
    ++nrunning_;
    tiles_dirty_ = true;
    desc_dirty_ = true;
    return slot;
}

int64_t ArenaEngine::running_tiles(int V) const {
    int64_t t = 0;
    for (const auto& p : probs_)
        if (p.state == P_RUNNING) {
            if (V != kTileWave) t += arena_tiles(p.nx, p.ny, V);
            else if (p.cls == C_PAIRS) t += step2_tiles(p.nx, p.ny);
            else t += arena_strips(p.nx) * ((p.ny + wave_seg_ - 1) / wave_seg_);
        }
    return t;
}

int ArenaEngine::check_forces(std::string* err) {
    std::vector<unsigned long long> got(2 * probs_.size());
    ECK(cudaMemcpyAsync(got.data(), d_stat_, sizeof(unsigned long long) * got.size(), cudaMemcpyDeviceToHost, st_));
    ECK(cudaStreamSynchronize(st_));
    for (size_t i = 0; i < probs_.size(); ++i)
        if (got[2 * i + 1]) {
            if (err) *err = "admit: non-finite force";
            return LBM_ERR_ARG;
        }
    return LBM_OK;
}

// Rows per strip item of the running problems, by strip_shape's model: the
// segments whose warps take the fewest cycles over all problems (a few large
// problems get short segments, many get long ones).
int ArenaEngine::choose_seg() const {
    const int64_t slots = 12LL * sms_;
    int best = 16;
    double cost = 0.0;
    for (int seg = 8; seg <= 512; seg += seg < 32 ? 4 : (seg < 128 ? 16 : 64)) {
        int64_t items = 0;
        int rows = 0;
        for (const auto& p : probs_)
            if (p.state == P_RUNNING && p.cls != C_PAIRS) {
                items += arena_strips(p.nx) * ((p.ny + seg - 1) / seg);
                rows = std::max(rows, std::min(p.ny, seg));
            }
        if (items == 0) break;
        double c = 0.0;
        const double full = (double)(rows + 8) * (5 * (70.0 + 115.0 * 3) + 150.0);
        const int64_t waves = (items - 1) / slots, rest = items - waves * slots;
        c = waves * full + (double)(rows + 8) * (5 * (70.0 + 115.0 * ((rest + 4 * sms_ - 1) / (4 * sms_))) + 150.0);
        if (cost == 0.0 || c < cost) {
            cost = c;
            best = seg;
        }
    }
    return best;
}

int64_t ArenaEngine::running_nodes() const {
    int64_t t = 0;
    for (const auto& p : probs_)
        if (p.state == P_RUNNING) t += p.n;
    return t;
}

int64_t ArenaEngine::resident_bytes() const {
    int64_t b = 0;
    for (const auto& p : probs_)
        if (p.state != P_FREE) b += bytes_for(p.plane);
    return b;
}

int ArenaEngine::grid_blocks(int V) const {
    return V == kTileWave ? strip_blocks_ : arena_occupancy(dtype_, V) * sms_;
}

int64_t ArenaEngine::free_nodes_hint() const {
    return apop_.largest_free() / pop_bytes_per_node(dtype_);
}

int ArenaEngine::upload_tiles(int V, std::string* err) {
    if (V == kTileWave) {
        wave_seg_ = choose_seg();
        desc_dirty_ = true;
    }
    // (strip chunk: one more item per problem, for the ghost columns)
    const int64_t nt = running_tiles(V) + (V == kTileWave ? nrunning_ : 0);
    if (nt > (int64_t)INT32_MAX) {
        if (err) *err = "arena: too many tiles";
        return LBM_ERR_ARG;
    }
    if (h_tiles_cap_ < nt) {
        if (h_tiles_) {
            ECK(cudaStreamSynchronize(st_));
            cudaFreeHost(h_tiles_);
            h_tiles_ = nullptr;
            h_tiles_cap_ = 0;
        }
        const int64_t cap = nt + nt / 4 + 1024;
        ECK(cudaMallocHost(&h_tiles_, sizeof(uint2) * cap));
        h_tiles_cap_ = cap;
    }
    if (tiles_cap_ < nt) {
        if (d_tiles_) {
            ECK(cudaStreamSynchronize(st_));
            device_free(&d_tiles_, sizeof(uint2) * tiles_cap_);
            tiles_cap_ = 0;
        }
        const int64_t cap = nt + nt / 4 + 1024;
        ECK(device_alloc(&d_tiles_, sizeof(uint2) * cap));
        tiles_cap_ = cap;
        for (auto& g : graph_)  // the graphs hold the old tile pointer
            if (g) {
                cudaGraphExecDestroy(g);
                g = nullptr;
            }
    }
    ECK(cudaStreamSynchronize(st_));  // the pinned list may feed a previous copy
    int64_t t = 0;
    if (V == kTileWave) {
        for (int cls = 0; cls < kClasses; ++cls) {
            class_begin_[cls] = (int)t;
            for (int s = 0; s < (int)probs_.size(); ++s) {
                const HostProb& p = probs_[s];
                if (p.state != P_RUNNING || p.cls != cls) continue;
                const int64_t m = cls == C_PAIRS ? step2_tiles(p.nx, p.ny)
                                                 : arena_strips(p.nx) * ((p.ny + wave_seg_ - 1) / wave_seg_);
                for (int64_t i = 0; i < m; ++i) h_tiles_[t++] = make_uint2((unsigned)s, (unsigned)i);
            }
        }
        class_begin_[kClasses] = (int)t;
        ghosts_begin_ = (int)t;
        for (int s = 0; s < (int)probs_.size(); ++s)
            if (probs_[s].state == P_RUNNING && probs_[s].ghost && !probs_[s].ghosts_ok)
                h_tiles_[t++] = make_uint2((unsigned)s, 0u);
        ghosts_end_ = (int)t;
    } else {
        for (int s = 0; s < (int)probs_.size(); ++s) {
            const HostProb& p = probs_[s];
            if (p.state != P_RUNNING) continue;
            const int64_t m = arena_tiles(p.nx, p.ny, V);
            for (int64_t i = 0; i < m; ++i) h_tiles_[t++] = make_uint2((unsigned)s, (unsigned)i);
        }
    }
    static thread_local int nt_host[2];
    nt_host[0] = (int)t;
    nt_host[1] = V == kTileWave ? class_begin_[C_PAIRS + 1] - class_begin_[C_PAIRS] : 0;
    if (t > 0) ECK(cudaMemcpyAsync(d_tiles_, h_tiles_, sizeof(uint2) * t, cudaMemcpyHostToDevice, st_));
    ECK(cudaMemcpyAsync(d_ntiles_, nt_host, sizeof(nt_host), cudaMemcpyHostToDevice, st_));
    ECK(cudaStreamSynchronize(st_));
    tiles_V_ = V;
    tiles_dirty_ = false;
    return LBM_OK;
}

BatchArgs ArenaEngine::chunk_args() const {
    BatchArgs a{};
    a.probs = d_probs_;
    a.tiles = d_tiles_;
    a.ntiles = d_ntiles_;
    a.pop0 = pop_[0];
    a.pop1 = pop_[1];
    a.car0 = car_[0];
    a.car1 = car_[1];
    a.fs = fs_;
    a.acc = d_acc_;
    a.nsteps = k_;
    return a;
}

int ArenaEngine::ensure_graph(int V, std::string* err) {
    if (graph_[V] || graph_failed_[V]) return LBM_OK;
    const BatchArgs a = chunk_args();
    const int grid = grid_blocks(V);
    if (grid < 1) {
        if (err) *err = "arena: chunk kernel cannot be resident";
        return LBM_ERR_CUDA;
    }
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(st_, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaMemsetAsync(d_acc_, 0, sizeof(double) * kRes * probs_.size(), st_);
        launch_arena_chunk(dtype_, V, a, grid, st_);
        cudaMemcpyAsync(h_acc_, d_acc_, sizeof(double) * kRes * probs_.size(), cudaMemcpyDeviceToHost, st_);
        e = cudaStreamEndCapture(st_, &g);
    }
    if (e == cudaSuccess && g) e = cudaGraphInstantiate(&graph_[V], g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        cudaGetLastError();  // clear; fall back to direct launches
        graph_[V] = nullptr;
        graph_failed_[V] = true;
    }
    return LBM_OK;
}

// Steps of the launches that advance strip items by a chunk of k steps (k a multiple
// of 4); the last one carries the check.
static std::vector<int> chunk_groups(int dtype, int k) {
    if (dtype == S_F16S || k < 5) return std::vector<int>(k / 4, 4);
    // fives after the rest (two threes where it would be one step)
    std::vector<int> g;
    const int r = k % 5;
    if (r == 1) g = {3, 3};
    else if (r == 4) g = {2, 2};
    else if (r) g = {r};
    g.resize(g.size() + (k - (r == 1 ? 6 : r)) / 5, 5);
    return g;
}

// One chunk: strips in a sequence of launches, and beside them the problems too narrow
// for strips in one.
int ArenaEngine::launch_strip_chunk(std::string* err) {
    const BatchArgs a = chunk_args();
    ECK(cudaMemsetAsync(d_acc_, 0, sizeof(double) * kRes * probs_.size(), st_));
    if (ghosts_end_ > ghosts_begin_)
        ECK(launch_arena_ghosts(dtype_, a, d_tiles_ + ghosts_begin_, ghosts_end_ - ghosts_begin_, st_));
    int busy[kClasses], nb = 0;
    for (int c = 0; c < kClasses; ++c)
        if (class_begin_[c + 1] > class_begin_[c]) busy[nb++] = c;
    if (nb > 1) ECK(cudaEventRecord(fork_, st_));
    for (int b = nb - 1; b >= 0; --b) {          // the first class last, on the engine's own stream
        const int c = busy[b], count = class_begin_[c + 1] - class_begin_[c];
        const cudaStream_t st = b == 0 ? st_ : side_[b - 1];
        if (b > 0) ECK(cudaStreamWaitEvent(st, fork_, 0));
        const uint2* items = d_tiles_ + class_begin_[c];
        if (c == C_PAIRS && pairs_grid_ == 0) pairs_grid_ = std::max(1, arena_occupancy(dtype_, kTileTwoStep) * sms_);
        const int blocks = c == C_PAIRS ? std::min(count, pairs_grid_) : (count + 3) / 4;
        strip_blocks_ = std::max(strip_blocks_, blocks);
        if (c == C_PAIRS) {
            BatchArgs p = a;
            p.tiles = items;
            p.ntiles = d_ntiles_ + 1;
            ECK(launch_arena_chunk(dtype_, kTileTwoStep, p, blocks, st));
        } else {
            const std::vector<int> groups = chunk_groups(dtype_, k_);
            for (int g = 0; g < (int)groups.size(); ++g)
                ECK(launch_arena_strips(dtype_, groups[g], g + 1 == (int)groups.size(), a, items, count, g, st));
        }
        if (b > 0) ECK(cudaEventRecord(join_[b - 1], st));
    }
    for (int b = 1; b < nb; ++b) ECK(cudaStreamWaitEvent(st_, join_[b - 1], 0));
    ECK(cudaMemcpyAsync(h_acc_, d_acc_, sizeof(double) * kRes * probs_.size(), cudaMemcpyDeviceToHost, st_));
    return LBM_OK;
}

int ArenaEngine::start_chunk(int V, std::string* err) {
    if (V != 1 && V != 2 && V != 4 && !(V == kTileTwoStep && k_ % 2 == 0) && !(V == kTileWave && k_ % 4 == 0)) {
        if (err) *err = "arena: tile code must be 1, 2 or 4 warps of 32, two-step tiles with an even chunk, "
                        "or the wavefront chunk with a chunk of a multiple of 4 steps";
        return LBM_ERR_ARG;
    }
    if (nrunning_ == 0) return LBM_OK;
    if (tiles_dirty_ || tiles_V_ != V) {
        int rc = upload_tiles(V, err);
        if (rc) return rc;
    }
    for (auto& p : probs_) {
        if (p.state != P_RUNNING) continue;
        const bool now = ((p.steps + k_) % ((int64_t)k_ * p.period)) == 0;
        if (now != p.check_now) {
            p.check_now = now;
            desc_dirty_ = true;
        }
    }
    if (desc_dirty_) {
        std::vector<BatchProb> d(probs_.size());
        for (size_t i = 0; i < probs_.size(); ++i) {
            const HostProb& p = probs_[i];
            BatchProb& b = d[i];
            // (of column 0)
            b.pop_off = p.pop_off + p.ghost * pop_bytes_per_node(dtype_) / 8;
            b.car_off = p.car_off + p.ghost * car_bytes_per_node(dtype_);
            b.fs_off = p.fs_off + p.ghost * (int64_t)sizeof(float);
            b.snap_off = p.fs_off + 2 * p.plane * (int64_t)sizeof(float);
            b.plane = p.plane;
            b.nx = p.nx;
            b.ny = p.ny;
            b.pitch = p.pitch;
            b.check = p.check_now ? 1 : 0;
            b.dtype = dtype_;
            b.parity = p.parity;
            b.seg = wave_seg_;
            b.half = dtype_ == S_F16S && !arena_wide(p.nx, p.ny) ? 1 : 0;
            b.q11 = p.q11;
            b.qs = p.qs;
            b.qd = p.qd;
            b.qtheta = p.qtheta;
            b.theta = p.theta;
            b.hscale = std::ldexp(1.0f, p.hexp);
            b.hinv = std::ldexp(1.0f, -p.hexp);
        }
        ECK(cudaMemcpyAsync(d_probs_, d.data(), sizeof(BatchProb) * d.size(), cudaMemcpyHostToDevice, st_));
        ECK(cudaStreamSynchronize(st_));
        desc_dirty_ = false;
    }
    int rc = V == kTileWave ? LBM_OK : ensure_graph(V, err);
    if (rc) return rc;
    ECK(cudaEventRecord(ev0_, st_));
    if (V == kTileWave) {
        rc = launch_strip_chunk(err);
        if (rc) return rc;
    } else if (graph_[V]) {
        ECK(cudaGraphLaunch(graph_[V], st_));
    } else {
        const BatchArgs a = chunk_args();
        ECK(cudaMemsetAsync(d_acc_, 0, sizeof(double) * kRes * probs_.size(), st_));
        ECK(launch_arena_chunk(dtype_, V, a, grid_blocks(V), st_));
        ECK(cudaMemcpyAsync(h_acc_, d_acc_, sizeof(double) * kRes * probs_.size(), cudaMemcpyDeviceToHost, st_));
    }
    ECK(cudaEventRecord(ev1_, st_));
    return LBM_OK;
}

int ArenaEngine::finish_chunk(int V, float* device_ms, std::string* err) {
    if (device_ms) *device_ms = 0.0f;
    if (nrunning_ == 0) return LBM_OK;
    ECK(cudaStreamSynchronize(st_));
    h_force_used_ = 0;
    if (device_ms) ECK(cudaEventElapsedTime(device_ms, ev0_, ev1_));
    for (int s = 0; s < (int)probs_.size(); ++s) {
        HostProb& p = probs_[s];
        if (p.state != P_RUNNING) continue;
        p.steps += k_;
        p.lups += p.n * k_;
        // the buffers swap once per group of steps: k steps, k/2 pairs, or a strip
        // chunk's groups
        const int64_t swaps = V == kTileWave && p.cls == C_STRIPS ? (int64_t)chunk_groups(dtype_, k_).size()
                                                                  : (V == kTileWave || V == kTileTwoStep ? k_ / 2 : k_);
        if (V != kTileWave) p.ghosts_ok = false;
        else if (!p.ghosts_ok) {
            p.ghosts_ok = true;
            tiles_dirty_ = true;      // (the list of stale ghost columns)
        }
        if (swaps & 1) {
            p.parity ^= 1;
            desc_dirty_ = true;
        }
        const double* raw = h_acc_ + (int64_t)s * kRes;
        bool done = false;
        if (!p.check_now) {
            // no residual this chunk
        } else if (raw[4] != 0.0 || !std::isfinite(raw[0]) || !std::isfinite(raw[1])) {
            p.status = LBM_ERR_DIVERGED;
            p.residual = INFINITY;
            done = true;
        } else if (!p.snap_valid) {
            p.snap_valid = true;
            p.residual = INFINITY;
            p.last_check = p.steps;
        } else {
            const double window = (double)(p.steps - p.last_check);
            p.last_check = p.steps;
            p.residual = raw[1] > 0.0 ? raw[0] / (window * raw[1]) : 0.0;
            if (p.residual < p.tol) {
                p.status = LBM_OK;
                done = true;
            } else {
                p.period = adapt_period(p.period, p.residual, p.r_prev);
                p.r_prev = p.residual;
            }
        }
        if (!done && p.steps >= p.max_iters) {
            p.status = LBM_ERR_NOT_CONVERGED;
            done = true;
        }
        if (done) {
            p.state = P_DONE;
            --nrunning_;
            tiles_dirty_ = true;
        }
    }
    return LBM_OK;
}

// FP64 fields of problem `slot` into device memory dst (5 planes of n).
cudaError_t ArenaEngine::launch_fields(int slot, double* dst) {
    const HostProb& p = probs_[slot];
    StepParams a{};
    a.nx = p.nx;
    a.ny = p.ny;
    a.pitch = p.pitch;
    a.plane = p.plane;
    const int64_t po = p.pop_off + p.ghost * pop_bytes_per_node(dtype_) / 8;
    a.src = pop_[p.parity] + po;
    a.dst = pop_[p.parity ^ 1] + po;
    if (dtype_ == S_F16S) {
        const int64_t co = p.car_off + p.ghost * car_bytes_per_node(dtype_);
        a.csrc = reinterpret_cast<const float*>(car_[p.parity] + co);
        a.cdst = reinterpret_cast<float*>(car_[p.parity ^ 1] + co);
        a.hscale = std::ldexp(1.0f, p.hexp);
        a.hinv = std::ldexp(1.0f, -p.hexp);
    }
    a.gx = fs_ + p.fs_off + p.ghost * sizeof(float);
    a.gy = fs_ + p.fs_off + (p.ghost + p.plane) * sizeof(float);
    const double theta = 1.0 / 3.0, K = p.lambda + p.mu;
    const double w11 = 1.0 / (p.mu / theta + 0.5), ws = 1.0 / (2.0 * K / (1.0 + theta) + 0.5),
                 wd = 1.0 / (2.0 * p.mu / (1.0 - theta) + 0.5);
    Coef<double> c{};
    c.b11 = 1.0 - 0.5 * w11;
    c.bs = 1.0 - 0.5 * ws;
    c.bd = 1.0 - 0.5 * wd;
    c.theta = theta;
    set_factors(c);
    FieldOut o = field_planes(dst, p.n);
    if (p.tr) {
        // back to the caller's lattice: u_x <-> u_y, sigma_xx <-> sigma_yy,
        // node (x, y) of the transpose at x * ny + y
        std::swap(o.p[0], o.p[1]);
        std::swap(o.p[2], o.p[3]);
        o.tr = 1;
    }
    return dtype_ == S_F16S ? Ops<S_F16S>::fields(a, c, (float)theta, o, st_)
                            : Ops<S_F32>::fields(a, c, (float)theta, o, st_);
}

int ArenaEngine::ensure_fields_buffer(int64_t len, std::string* err) {
    if (d_fields_cap_ >= len) return LBM_OK;
    if (d_fields_) {
        ECK(cudaStreamSynchronize(st_));
        device_free(&d_fields_, sizeof(double) * d_fields_cap_);
        d_fields_cap_ = 0;
    }
    ECK(device_alloc(&d_fields_, sizeof(double) * len));
    d_fields_cap_ = len;
    return LBM_OK;
}

int ArenaEngine::recover_many(int count, const int* slots, double* const* outs, std::string* err) {
    // Problems are packed into blocks of kRecoverBlock doubles: one field launch per
    // problem into a device block, then copies straight into the callers' arrays,
    // one per problem where its five arrays lie one after the other.  Small problems
    // come in one copy per block and are handed out by the host: a copy each into pageable
    // arrays costs a wait of some 8 us (200 problems of sides 4 to 31 on a server, 400
    // steps: 10.0 -> 7.7 ms; eight of 64 x 64, which are not small, 1.49 ms a batch, as
    // small ones 1.64).
    int64_t need = 0, all = 0;
    for (int i = 0; i < count; ++i) {
        const HostProb& p = probs_[slots[i]];
        if (p.state == P_FREE) {
            if (err) *err = "recover: empty slot";
            return LBM_ERR_STATE;
        }
        need = std::max(need, 5 * p.n);
        all += 5 * p.n;
    }
    if (count == 0) return LBM_OK;
    int rc = ensure_fields_buffer(std::max(need, std::min(all, kRecoverBlock)), err);
    if (rc) return rc;
    // small problems first, many to a copy
    std::vector<int> small, large;
    for (int i = 0; i < count; ++i) (probs_[slots[i]].n <= kSmallFields ? small : large).push_back(i);
    for (size_t i = 0; i < small.size();) {
        size_t j = i;
        int64_t used = 0;
        for (; j < small.size() && used + 5 * probs_[slots[small[j]]].n <= std::min(kFieldStage, d_fields_cap_); ++j) {
            ECK(launch_fields(slots[small[j]], d_fields_ + used));
            used += 5 * probs_[slots[small[j]]].n;
        }
        if (h_fields_cap_ < used) {
            if (h_fields_) cudaFreeHost(h_fields_);
            h_fields_ = nullptr;
            h_fields_cap_ = 0;
            const int64_t cap = small.size() == j ? used : kFieldStage;
            ECK(cudaMallocHost(&h_fields_, sizeof(double) * cap));
            h_fields_cap_ = cap;
        }
        ECK(cudaMemcpyAsync(h_fields_, d_fields_, sizeof(double) * used, cudaMemcpyDeviceToHost, st_));
        ECK(cudaStreamSynchronize(st_));
        const double* from = h_fields_;
        for (; i < j; ++i) {
            const int64_t n = probs_[slots[small[i]]].n;
            for (int f = 0; f < 5; ++f, from += n)
                if (double* to = outs[5 * (int64_t)small[i] + f]) std::memcpy(to, from, sizeof(double) * n);
        }
    }
    for (size_t i = 0; i < large.size();) {
        size_t j = i;
        int64_t used = 0;
        for (; j < large.size() && (j == i || used + 5 * probs_[slots[large[j]]].n <= d_fields_cap_); ++j) {
            ECK(launch_fields(slots[large[j]], d_fields_ + used));
            used += 5 * probs_[slots[large[j]]].n;
        }
        int64_t off = 0;
        for (size_t q = i; q < j; ++q) {
            const int64_t n = probs_[slots[large[q]]].n;
            double* const* o = outs + 5 * (int64_t)large[q];
            for (int f = 0; f < 5;) {
                int g = f + 1;
                while (o[f] && g < 5 && o[g] == o[f] + (g - f) * n) ++g;
                if (o[f])
                    ECK(copy_out(o[f], d_fields_ + off + f * n, sizeof(double) * n * (g - f), st_));
                f = g;
            }
            off += 5 * n;
        }
        ECK(cudaStreamSynchronize(st_));
        i = j;
    }
    return LBM_OK;
}

void ArenaEngine::release(int slot) {
    HostProb& p = probs_[slot];
    if (p.state == P_FREE) return;
    if (p.state == P_RUNNING) {
        --nrunning_;
        tiles_dirty_ = true;
    }
    unplace(p);
    p = HostProb();
}

// ---------------------------------------------------------------------------
// Autotuner cache: "key V" lines in $LBM_AUTOTUNE_CACHE (default
// $HOME/.cache/lbm_gb300/autotune.txt).  LBM_AUTOTUNE=0 disables lookups.
// ---------------------------------------------------------------------------

namespace {
std::mutex g_tune_mutex;

std::string cache_path() {
    const char* p = std::getenv("LBM_AUTOTUNE_CACHE");
    if (p && *p) return p;
    const char* h = std::getenv("HOME");
    std::string dir = std::string(h && *h ? h : "/tmp") + "/.cache";
    mkdir(dir.c_str(), 0755);
    dir += "/lbm_gb300";
    mkdir(dir.c_str(), 0755);
    return dir + "/autotune.txt";
}
}  // namespace

int autotune_lookup(const std::string& key) {
    const char* off = std::getenv("LBM_AUTOTUNE");
    if (off && std::string(off) == "0") return 0;
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    std::ifstream in(cache_path());
    std::string k;
    int v = 0, found = 0;
    while (in >> k >> v)
        if (k == key) found = v;
    return found;
}

void autotune_store(const std::string& key, int V) {
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    std::ofstream out(cache_path(), std::ios::app);
    if (out) out << key << " " << V << "\n";
}

}  // namespace lbm
