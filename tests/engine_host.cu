// The host code of the arena and the server (lbm_engine.cu, lbm_server.cu) on a
// stand-in for the CUDA runtime, without a GPU: device memory is host memory,
// kernels advance the clock of their stream by a millisecond (the recovery fills
// field k with k + 1, the others do nothing else), and
// copies and fills run, in order, when the stream is waited for -- as late as the
// runtime allows.  Freeing the source of a copy that has not run is recorded.
// usage: engine_host SCENARIO; prints "ok" or what is wrong.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <new>
#include <set>
#include <string>
#include <vector>

#include "lbm_engine.cu"
#include "lbm_server.cu"

namespace fake {

// Sources of copies that have not run (no allocation: read from operator delete).
constexpr int kMost = 1 << 12;
struct Source {
    const char* p;
    size_t n;
};
Source sources[kMost];
int nsources = 0;
std::atomic_flag lock = ATOMIC_FLAG_INIT;
std::atomic<int> freed_in_flight{0};

struct Hold {
    Hold() {
        while (lock.test_and_set()) {}
    }
    ~Hold() { lock.clear(); }
};

void check_free(const void* p) {
    if (!p) return;
    Hold h;
    for (int i = 0; i < nsources; ++i)
        if (sources[i].p == p) ++freed_in_flight;
}

std::mutex mu;
std::vector<std::function<void()>> work;      // of all streams (each wait runs all of it)
std::map<char*, size_t> device, pinned;       // allocations
std::map<void*, double> clocks;               // of the streams, ms
std::map<void*, double> events;
std::vector<size_t> sizes;                    // of the device allocations, in turn
std::vector<char*> bases;
int calls = 0;                                // copies, fills, launches and waits
size_t device_bytes = 0, device_peak = 0;
int launches = 0, fail_launch = -1;           // the launch of this number fails

bool within(const std::map<char*, size_t>& m, const void* p, size_t n) {
    auto it = m.upper_bound((char*)p);
    if (it == m.begin()) return false;
    --it;
    return (char*)p >= it->first && (char*)p + n <= it->first + it->second;
}

void run_all() {
    std::vector<std::function<void()>> now;
    {
        std::lock_guard<std::mutex> l(mu);
        now.swap(work);
    }
    for (auto& f : now) f();
    Hold h;
    nsources = 0;
}

cudaError_t launch(void* stream) {
    std::lock_guard<std::mutex> l(mu);
    ++calls;
    if (launches++ == fail_launch) return cudaErrorLaunchFailure;
    clocks[stream] += 1.0;
    return cudaSuccess;
}

}  // namespace fake

#ifndef __CUDA_ARCH__      // (host only)
void* operator new(size_t n) {
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void* operator new[](size_t n) { return operator new(n); }
void operator delete(void* p) noexcept {
    fake::check_free(p);
    std::free(p);
}
void operator delete[](void* p) noexcept { operator delete(p); }
void operator delete(void* p, size_t) noexcept { operator delete(p); }
void operator delete[](void* p, size_t) noexcept { operator delete(p); }

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
    std::lock_guard<std::mutex> l(fake::mu);
    *p = std::calloc(1, n);
    fake::device[(char*)*p] = n;
    fake::sizes.push_back(n);
    fake::bases.push_back((char*)*p);
    fake::device_bytes += n;
    fake::device_peak = std::max(fake::device_peak, fake::device_bytes);
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    fake::run_all();
    std::lock_guard<std::mutex> l(fake::mu);
    fake::device_bytes -= fake::device[(char*)p];
    fake::device.erase((char*)p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
    std::lock_guard<std::mutex> l(fake::mu);
    *p = std::calloc(1, n);
    fake::pinned[(char*)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void* p) {
    fake::run_all();
    std::lock_guard<std::mutex> l(fake::mu);
    fake::pinned.erase((char*)p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind kind, cudaStream_t) {
    std::lock_guard<std::mutex> l(fake::mu);
    // (as the runtime does: host ranges that are pinned in part, or in two parts, are refused)
    const char* h0 = kind == cudaMemcpyDeviceToHost ? (const char*)d : (const char*)s;
    for (auto& r : fake::pinned)
        if (h0 < r.first + r.second && h0 + n > r.first && !fake::within(fake::pinned, h0, n)) return cudaErrorInvalidValue;
    ++fake::calls;
    fake::work.push_back([=] { std::memcpy(d, s, n); });
    fake::Hold h;
    if (fake::nsources < fake::kMost) fake::sources[fake::nsources++] = {(const char*)s, n};
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    std::lock_guard<std::mutex> l(fake::mu);
    ++fake::calls;
    fake::work.push_back([=] { std::memset(d, v, n); });
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes* a, const void* p) {
    std::lock_guard<std::mutex> l(fake::mu);
    std::memset(a, 0, sizeof(*a));
    a->type = fake::within(fake::pinned, p, 1) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = (cudaStream_t)std::malloc(1);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    std::free(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    ++fake::calls;
    fake::run_all();
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    std::lock_guard<std::mutex> l(fake::mu);
    fake::clocks[s] = std::max(fake::clocks[s], fake::events[e]);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t)std::malloc(1);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    std::free(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    std::lock_guard<std::mutex> l(fake::mu);
    fake::events[e] = fake::clocks[s];
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
    std::lock_guard<std::mutex> l(fake::mu);
    *ms = (float)(fake::events[b] - fake::events[a]);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "stand-in"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, enum cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t s) { return fake::launch(s); }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) {
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
char __cudaInitModule(void**) { return 0; }
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t s) { return fake::launch(s); }
}

#endif

// What the engine launches (lbm_arena.cu, lbm_step_f32.cu, lbm_step_f16s.cu).
namespace lbm {
int set_last_error(int code, const std::string&) { return code; }
cudaError_t launch_arena_chunk(int, int, const BatchArgs&, int, cudaStream_t st) { return fake::launch(st); }
int arena_occupancy(int, int) { return 1; }
cudaError_t launch_arena_strips(int, int, bool, const BatchArgs&, const uint2*, int, int, cudaStream_t st) {
    return fake::launch(st);
}
cudaError_t launch_arena_ghosts(int, const BatchArgs&, const uint2*, int, cudaStream_t st) { return fake::launch(st); }
cudaError_t launch_arena_force(const ForceIn&, cudaStream_t st) { return fake::launch(st); }
template <int S>
cudaError_t Ops<S>::fields(const StepParams& a, const Coef<double>&, T, const FieldOut& o, cudaStream_t st) {
    const int64_t n = (int64_t)a.nx * a.ny;
    {
        std::lock_guard<std::mutex> l(fake::mu);
        fake::work.push_back([=] {
            for (int k = 0; k < 5; ++k) std::fill(o.p[k], o.p[k] + n, 1.0 + k);
        });
    }
    return fake::launch(st);
}
__global__ void k_scale_float(float*, int64_t, float) {}
}  // namespace lbm

namespace {

#define EXPECT(x)                                                          \
    do {                                                                   \
        if (!(x)) {                                                        \
            std::printf("line %d: not so: %s\n", __LINE__, #x);            \
            std::exit(1);                                                  \
        }                                                                  \
    } while (0)

struct Problem {
    int nx, ny;
    std::vector<double> gx, gy, out[5];
    lbm_result r{};
    Problem(int nx, int ny) : nx(nx), ny(ny), gx((size_t)nx * ny, 1.0), gy(gx) {
        double** o[5] = {&r.ux, &r.uy, &r.sxx, &r.syy, &r.sxy};
        for (int k = 0; k < 5; ++k) {
            out[k].assign(gx.size(), -7.0);
            *o[k] = out[k].data();
        }
    }
    lbm_problem in() { return {nx, ny, 0.3, 0.4, gx.data(), gy.data()}; }
};

// The force of an admitted request outlives its copy to the device, also when the
// chunk after the admission fails and the request is taken back at once.
void server_force(bool fail) {
    lbm_server* s = nullptr;
    EXPECT(lbm_server_create(size_t(64) << 20, 100, &s) == LBM_OK);
    if (fail) fake::fail_launch = 12;
    std::vector<Problem> p;
    for (int i = 0; i < 6; ++i) p.emplace_back(40 + i, i < 4 ? 120 : 30);      // (large and small)
    std::vector<uint64_t> t;
    for (int i = 0; i < 6; ++i) {
        const lbm_problem in = p[i].in();
        uint64_t ticket = 0;
        if (lbm_server_submit(s, &in, i % 2 ? LBM_F16S : LBM_F32, 0.0, 300, &ticket) == LBM_OK) t.push_back(ticket);
        else EXPECT(fail);
    }
    for (size_t i = 0; i < t.size(); ++i) {
        EXPECT(lbm_server_wait(s, t[i], 60.0, &p[i].r) == LBM_OK);
        EXPECT(fail || p[i].r.iters == 300);
    }
    lbm_server_destroy(s);
    EXPECT(fake::freed_in_flight == 0);
}

// The device time a server reports is the time its kernels took: one millisecond
// each here, all of a chunk's on one stream.
void server_device_ms() {
    lbm_server* s = nullptr;
    EXPECT(lbm_server_create(size_t(64) << 20, 100, &s) == LBM_OK);
    const int before = fake::launches;
    Problem a(300, 40), b(310, 50);
    lbm_problem in[2] = {a.in(), b.in()};
    uint64_t t[2];
    EXPECT(lbm_server_submit(s, &in[0], LBM_F32, 0.0, 200, &t[0]) == LBM_OK);
    EXPECT(lbm_server_submit(s, &in[1], LBM_F16S, 0.0, 200, &t[1]) == LBM_OK);
    EXPECT(lbm_server_wait(s, t[0], 60.0, &a.r) == LBM_OK && lbm_server_wait(s, t[1], 60.0, &b.r) == LBM_OK);
    lbm_stats st{};
    EXPECT(lbm_server_stats(s, &st) == LBM_OK);
    // (two forces and two recoveries are no part of a chunk)
    EXPECT(st.device_ms == fake::launches - before - 4);
    lbm_server_destroy(s);
}

// A request whose fields could not be recovered says so, and leaves the caller's
// arrays alone.
void server_recovery_fails() {
    lbm_server* s = nullptr;
    EXPECT(lbm_server_create(size_t(64) << 20, 100, &s) == LBM_OK);
    Problem p(300, 40);
    const lbm_problem in = p.in();
    fake::fail_launch = fake::launches + 1 + 20;       // the force, twenty launches of five steps
    uint64_t t;
    EXPECT(lbm_server_submit(s, &in, LBM_F32, 0.0, 100, &t) == LBM_OK);
    EXPECT(lbm_server_wait(s, t, 60.0, &p.r) == LBM_OK && p.r.status == LBM_ERR_CUDA && p.r.iters == 100);
    for (auto& o : p.out)
        for (double v : o) EXPECT(v == -7.0);
    lbm_server_destroy(s);
}

// Problems too narrow for strips take one launch per chunk, however many steps.
void narrow_launches(int dtype) {
    ArenaEngine e;
    std::string err;
    EXPECT(e.init(dtype, 20000, 4, 100, (cudaStream_t)&e, &err) == LBM_OK);
    std::vector<double> g(100, 1.0);
    const int s = e.admit(10, 10, 0.3, 0.4, g.data(), g.data(), 0.0, 300, &err);
    EXPECT(s >= 0 && !e.prob(s).ghost);
    for (int chunk = 0; chunk < 3; ++chunk) {
        const int before = fake::launches, parity = e.prob(s).parity;
        EXPECT(e.run_chunk(kTileWave, nullptr, &err) == LBM_OK);
        EXPECT(fake::launches == before + 1 && e.prob(s).parity == parity);      // (fifty pairs of steps)
    }
    EXPECT(e.prob(s).state == P_DONE && e.prob(s).steps == 300);
}

// Small problems: at most four calls of the runtime per admission, whose force planes
// hold the caller's values (scaled), transposed where the problem is, with their
// periodic images and zeros around them; an entry that is not finite is refused as a
// bad argument.
void small_forces(int dtype) {
    ArenaEngine e;
    std::string err;
    EXPECT(e.init(dtype, 300000, 128, 100, (cudaStream_t)&e, &err) == LBM_OK);
    const size_t fs = dtype == S_F16S ? 4 : 2;         // (the force buffer: full_arena)
    for (auto wh : {std::pair<int, int>{1, 1}, {5, 9}, {16, 16}, {17, 40}, {57, 3}, {16, 250}, {250, 16}, {64, 64}}) {
        const int nx = wh.first, ny = wh.second;
        std::vector<double> g[2];
        for (int c = 0; c < 2; ++c)
            for (int i = 0; i < nx * ny; ++i) g[c].push_back((c ? -0.375 : 0.25) + i * 0.125);
        fake::run_all();
        fake::calls = 0;
        const int s = e.admit(nx, ny, 0.3, 0.4, g[0].data(), g[1].data(), 0.0, 100, &err);
        EXPECT(s >= 0 && fake::calls <= (dtype == S_F16S ? 4 : 3) + 1);      // (a reset of the staging at most)
        fake::run_all();
        const HostProb& p = e.prob(s);
        const float* f = (const float*)(fake::bases[fs] + p.fs_off);
        for (int c = 0; c < 2; ++c)
            for (int y = 0; y < p.ny; ++y)
                for (int x = -p.ghost; x < p.pitch - p.ghost; ++x) {
                    const int xw = (x + p.nx) % p.nx;
                    const double v = p.tr ? g[1 - c][xw * nx + y] : g[c][y * nx + xw];
                    const bool in = x < p.nx + p.ghost;
                    EXPECT(f[c * p.plane + y * p.pitch + p.ghost + x] == (in ? std::ldexp(v, p.hexp) : 0.0));
                }
        const float* snap = f + 2 * p.plane;
        for (int64_t i = 0; i < 4 * p.plane; ++i) EXPECT(snap[i] == 0.0f);
        g[1].back() = -INFINITY;
        EXPECT(e.admit(nx, ny, 0.3, 0.4, g[0].data(), g[1].data(), 0.0, 100, &err) == LBM_ERR_ARG);
        g[1].back() = NAN;
        EXPECT(e.admit(nx, ny, 0.3, 0.4, g[0].data(), g[1].data(), 0.0, 100, &err) == LBM_ERR_ARG);
        EXPECT(e.running() == s + 1);
    }
}

// Fields of many small problems come in few copies; each goes where its caller wants
// it, and fields that nobody wants nowhere.
void small_fields(int dtype) {
    ArenaEngine e;
    std::string err;
    EXPECT(e.init(dtype, 400000, 128, 100, (cudaStream_t)&e, &err) == LBM_OK);
    std::vector<int> slots;
    std::vector<std::vector<double>> mem;
    std::vector<double*> outs;
    for (int i = 0; i < 100; ++i) {
        const int nx = i == 50 ? 90 : 8 + i % 38, ny = i == 50 ? 80 : 45 - i % 37;
        const std::vector<double> g((size_t)nx * ny, 1.0);
        slots.push_back(e.admit(nx, ny, 0.3, 0.4, g.data(), g.data(), 0.0, 100, &err));
        EXPECT(slots.back() >= 0);
        mem.emplace_back(5 * g.size(), -7.0);
        for (int f = 0; f < 5; ++f) outs.push_back((i + f) % 7 ? &mem.back()[f * g.size()] : nullptr);
    }
    EXPECT(e.run_chunk(kTileWave, nullptr, &err) == LBM_OK);
    fake::calls = 0;
    EXPECT(e.recover_many(100, slots.data(), outs.data(), &err) == LBM_OK);
    EXPECT(fake::calls <= 100 + 2 * 2 + 6);        // (two blocks of small ones, the large one's fields)
    for (int i = 0; i < 100; ++i) {
        const int64_t n = e.prob(slots[i]).n;
        for (int f = 0; f < 5; ++f) {
            const int from = !e.prob(slots[i]).tr || f == 4 ? f : f ^ 1;      // (the transpose's field)
            for (int64_t k = 0; k < n; ++k) EXPECT(mem[i][f * n + k] == (outs[5 * i + f] ? 1.0 + from : -7.0));
        }
    }
}

// The arena says what it holds on the device, and its forces and fields are staged in
// one buffer.
void staging(int dtype) {
    const int nx = 600, ny = 500, n = nx * ny;
    std::vector<double> g(n, 1.0), out(5 * n);
    std::string err;
    const size_t none = fake::device_bytes;
    ArenaEngine e;
    EXPECT(e.init(dtype, 620 * 500, 4, 100, (cudaStream_t)&e, &err) == LBM_OK);
    const size_t empty = fake::device_bytes;
    EXPECT(e.device_bytes() == (int64_t)(empty - none));
    const int s = e.admit(nx, ny, 0.3, 0.4, g.data(), g.data(), 0.0, 100, &err);
    EXPECT(s >= 0 && e.device_bytes() == (int64_t)(fake::device_bytes - none));
    EXPECT(e.run_chunk(kTileWave, nullptr, &err) == LBM_OK && e.prob(s).state == P_DONE);
    const size_t ran = e.device_bytes();
    EXPECT(ran == fake::device_bytes - none);
    double* outs[5];
    for (int k = 0; k < 5; ++k) outs[k] = &out[k * n];
    EXPECT(e.recover_many(1, &s, outs, &err) == LBM_OK);
    EXPECT(e.device_bytes() == (int64_t)(fake::device_bytes - none));
    EXPECT(fake::device_peak <= empty + 5 * n * sizeof(double) + (size_t(1) << 20));   // (a megabyte for tables)
}

// A full arena: what a strip reads beyond the rows of the last problem (at most 72
// columns from eight before its first one) lies within the arena's buffers.
void full_arena(int dtype) {
    for (int nx : {16, 57, 64, 113, 200}) {
        ArenaEngine e;
        std::string err;
        const int most = 256;
        fake::sizes.clear();
        EXPECT(e.init(dtype, 20000, most, 100, (cudaStream_t)&e, &err) == LBM_OK);
        int64_t over = 0, pops = 0, cars = 0, fs = 0;
        std::vector<double> g;
        for (int ny = 64; ny >= 1;) {
            g.assign((size_t)nx * ny, 1.0);
            const int s = e.admit(nx, ny, 0.3, 0.4, g.data(), g.data(), 0.0, 100, &err);
            if (s < 0) {
                EXPECT(s == ArenaEngine::kNoRoom);
                --ny;
                continue;
            }
            const HostProb& p = e.prob(s);
            if (!p.ghost) continue;
            // from the first column of a problem to the last column its last strip's copies take
            const int64_t last = (arena_strips(p.nx) - 1) * kArenaOX - st_left<S_F32, 5>() + kStCols;
            const int64_t extent = (int64_t)p.pitch * (p.ny - 1) + p.ghost + last;
            const int64_t b = dtype == S_F16S ? 2 : 4;
            over = std::max(over, extent - p.plane);
            pops = std::max(pops, p.pop_off + b * (7 * p.plane + extent));
            if (dtype == S_F16S) cars = std::max(cars, p.car_off + 8 * extent);
            fs = std::max(fs, p.fs_off + 4 * (p.plane + extent));
        }
        EXPECT(over > 0 && over <= kRowSlack);
        const bool car = dtype == S_F16S;      // (allocated in turn: populations, carriers, both again, forces)
        EXPECT(pops <= (int64_t)fake::sizes[0] && fs <= (int64_t)fake::sizes[car ? 4 : 2]);
        EXPECT(!car || cars <= (int64_t)fake::sizes[1]);
    }
}

// Forces and results in host memory that is pinned in parts: arrays that follow
// one another, pinned each by itself, and arrays across the end of a pinned range.
void pinned_parts(int dtype) {
    const int nx = 80, ny = 80, n = nx * ny;
    std::vector<double> mem(7 * n, -7.0);
    for (int k = 2; k < 7; ++k) fake::pinned[(char*)&mem[k * n]] = n * sizeof(double);
    fake::pinned[(char*)mem.data()] = n / 2 * sizeof(double);          // half of g_x
    for (int i = 0; i < 2 * n; ++i) mem[i] = 1.0;
    ArenaEngine e;
    std::string err;
    EXPECT(e.init(dtype, 20000, 4, 100, (cudaStream_t)&e, &err) == LBM_OK);
    const int s = e.admit(nx, ny, 0.3, 0.4, &mem[0], &mem[n], 0.0, 100, &err);
    EXPECT(s >= 0);
    EXPECT(e.run_chunk(kTileWave, nullptr, &err) == LBM_OK && e.prob(s).state == P_DONE);
    double* outs[5];
    for (int k = 0; k < 5; ++k) outs[k] = &mem[(2 + k) * n];
    EXPECT(e.recover_many(1, &s, outs, &err) == LBM_OK);
    for (int i = 2 * n; i < 7 * n; ++i) EXPECT(mem[i] == i / n - 1);
    // pinned in part only
    fake::pinned.erase((char*)&mem[4 * n]);
    fake::pinned[(char*)&mem[4 * n]] = 100;
    std::fill(mem.begin() + 2 * n, mem.end(), -7.0);
    EXPECT(e.recover_many(1, &s, outs, &err) == LBM_OK);
    for (int i = 2 * n; i < 7 * n; ++i) EXPECT(mem[i] == i / n - 1);
    for (int k = 2; k < 7; ++k) fake::pinned.erase((char*)&mem[k * n]);
    fake::pinned.erase((char*)mem.data());
}

}  // namespace

int main(int argc, char** argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "server_force") server_force(false);
    else if (what == "server_force_failing") server_force(true);
    else if (what == "server_device_ms") server_device_ms();
    else if (what == "server_recovery_fails") server_recovery_fails();
    else if (what == "narrow_launches_f32") narrow_launches(S_F32);
    else if (what == "narrow_launches_f16s") narrow_launches(S_F16S);
    else if (what == "small_forces_f32") small_forces(S_F32);
    else if (what == "small_forces_f16s") small_forces(S_F16S);
    else if (what == "small_fields_f32") small_fields(S_F32);
    else if (what == "small_fields_f16s") small_fields(S_F16S);
    else if (what == "staging_f32") staging(S_F32);
    else if (what == "staging_f16s") staging(S_F16S);
    else if (what == "full_arena_f32") full_arena(S_F32);
    else if (what == "full_arena_f16s") full_arena(S_F16S);
    else if (what == "pinned_parts_f32") pinned_parts(S_F32);
    else if (what == "pinned_parts_f16s") pinned_parts(S_F16S);
    else return 2;
    std::printf("ok\n");
    std::fflush(stdout);
    std::_Exit(0);      // (the stand-in's maps go last)
}
