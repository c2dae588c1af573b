// lbm_kernels.cuh -- CUDA kernels of the periodic lattice Boltzmann scheme for
// linear elasticity (arXiv 2208.14870): fused stream-collide step (Algorithm 1)
// with an optional fused steady-state residual, solution recovery (Table 2),
// population import/export and force upload.  Instantiated once per storage
// type by lbm_step_f64.cu, lbm_step_f32.cu and lbm_step_f16s.cu.
//
// Memory layout (structure of arrays): population p of node (x, y) lives at
// base + p*plane + y*pitch + x (`plane` >= pitch*ny is padded to 256 bytes;
// rows may hold ghost columns, see row_ghost).  The
// stored state between steps is the post-collision population f*_p(x) of the
// previous step ("pull" scheme): a step gathers f_p(x) = f*_p(x - c_p) with the
// periodic wrap done by index arithmetic (Sec. 5.1), collides, and writes
// f*_p(x) to the other buffer of a ping-pong pair.
//
// Thread mapping: a block of 32 x BY threads covers a tile of 32*V columns by
// BY rows; a thread handles V nodes of one row spaced 32 apart, so each warp
// load or store instruction touches 32 consecutive nodes of one plane.
#pragma once

#include <type_traits>

#include "lbm_core.cuh"

namespace lbm {

// Launch shape (compile-time): rows per block, resident blocks per SM the
// plain step is compiled for, and nodes per thread of the FP16-shifted wide
// variant. The defaults are the fastest of a sweep at 16384^2 on GB300
// (FP32: BY 8, 4 blocks, 4 nodes; FP16S: 4 blocks of 2 nodes beat 3 of 4).
#ifndef LBM_BY
#define LBM_BY 8
#endif
#ifndef LBM_MINB_F32
#define LBM_MINB_F32 4
#endif
#ifndef LBM_MINB_F16S
#define LBM_MINB_F16S 4
#endif
#ifndef LBM_F16S_V
#define LBM_F16S_V 2
#endif
constexpr int BY = LBM_BY;         // rows per block (block = 32 x BY threads)

enum Storage { S_F64 = 0, S_F32 = 1, S_F16S = 2 };

// Nodes per thread (spaced 32 apart) of the wide step variant per storage.
template <int S>
constexpr int max_vec() {
    return S == S_F64 ? 2 : (S == S_F16S ? LBM_F16S_V : 4);
}
constexpr int kThreads = 32 * BY;

template <int S> struct StoreT;
// T: collision arithmetic, P: stored population, G: stored force.
template <> struct StoreT<S_F64> { using T = double; using P = double; using G = double; };
template <> struct StoreT<S_F32> { using T = float; using P = float; using G = float; };
template <> struct StoreT<S_F16S> { using T = float; using P = __half; using G = float; };

// Residual partial sums of one block: max|du|, max|u|, sum du^2, sum u^2,
// non-finite flag.
constexpr int kRes = 5;

struct StepParams {
    int nx, ny;
    int pitch;              // elements between rows
    int64_t plane;          // elements between planes
    const void* src;        // 8 population planes (storage type)
    void* dst;
    const float* csrc;      // F16S: carriers (m*_10, m*_01) interleaved per node (float2)
    float* cdst;
    const void* gx;         // force planes (G)
    const void* gy;
    float hscale;           // F16S: the state's scale 2^e (see store_f16s)
    float hinv;             // 1 / hscale
    void* snap;             // residual: u_x, u_y snapshot, 2 planes (ResSnap)
    double* partials;       // residual: kRes doubles per block
    unsigned int* counter;  // residual: blocks finished, reset by the last block; null:
                            // blocks only write partials (k_residual_finish combines them)
    double* result;         // residual: kRes doubles
};

template <typename T>
__device__ __forceinline__ T ldg(const T* p) { return __ldg(p); }

// ---------------------------------------------------------------------------
// Steady-state residual (Sec. 2.1's stopping test; reading: max and L2 norms
// of u^t - u^(t-w) over a window of w steps).  Each thread keeps partials over
// its nodes -- max|du|, max|u| (over nodes and both components), sum du^2,
// sum u^2 and a non-finite flag -- and the snapshot holds u of the previous
// check, two planes laid out as the populations':
//   FP64 storage: u from the FP64 collision, FP64 snapshot and partials;
//   FP32 / FP16S: u as an exact FP32 pair from exact_displacement, the
//   snapshot as (hi, lo) pairs (16 bytes per node, like two FP64 planes), and
//   pair partials (about 2^-44 relative); the sums are converted to FP64 per thread.
// Warps, blocks and the grid combine the sums in FP64 (ResPart: the maxima as pairs
// within a block).
template <int S> struct ResSnap { float2 u, v; };          // (hi, lo) per component
template <> struct ResSnap<S_F64> { double u, v; };

// A thread's partial as FP64 (a NaN among the maxima -- an infinite difference --
// is left to the flag).
__device__ __forceinline__ double pair_to_double(float h, float l) { return (double)h + (double)l; }
__device__ __forceinline__ double max_to_double(float h, float l) {
    const double v = pair_to_double(h, l);
    return v >= 0.0 ? v : 0.0;
}

template <int S> struct ResAcc {
    float dh = 0.f, dl = 0.f, uh = 0.f, ul = 0.f, d2h = 0.f, d2l = 0.f, u2h = 0.f, u2l = 0.f, bad = 0.f;
    // [max|du|, max|u|, sum du^2, sum u^2, flag]
    __device__ __forceinline__ void to_double(double w[kRes]) const {
        w[0] = max_to_double(dh, dl);
        w[1] = max_to_double(uh, ul);
        w[2] = pair_to_double(d2h, d2l);
        w[3] = pair_to_double(u2h, u2l);
        w[4] = bad;
    }
};
// Combination of kRes partials across a warp's lanes (result in every lane).
// The maxima and the flag are non-negative doubles, which order like their bit
// patterns: they are combined as integers (an FP64 instruction takes 64 cycles
// of a scheduler), the sums in FP64.
__device__ __forceinline__ double max_bits(double a, double b) {
    const unsigned long long x = (unsigned long long)__double_as_longlong(a), y = (unsigned long long)__double_as_longlong(b);
    return __longlong_as_double((long long)(x > y ? x : y));
}
template <> struct ResAcc<S_F64> {
    double d = 0.0, u = 0.0, d2 = 0.0, u2 = 0.0, bad = 0.0;
    __device__ __forceinline__ void to_double(double w[kRes]) const {
        w[0] = d >= 0.0 ? d : 0.0;
        w[1] = u >= 0.0 ? u : 0.0;
        w[2] = d2;
        w[3] = u2;
        w[4] = bad;
    }
};

// max(m, |h + l|) on normalised pairs (|l| <= ulp(h) / 2), lexicographically.
// Once a thread's running maximum is established few nodes reach it, so the
// full comparison sits behind one test of the hi part.
__device__ __forceinline__ void pair_max_abs(float& mh, float& ml, float h, float l) {
    if (fabsf(h) >= mh) {
        if (h < 0.0f) {
            h = -h;
            l = -l;
        }
        if (h > mh || l > ml) {
            mh = h;
            ml = l;
        }
    }
}

// s += (h + l)^2 in pair arithmetic: h*h with its exact FMA error, plus
// 2 h l (l^2 is below 2^-48 h^2 and dropped); the sum stays normalised.
__device__ __forceinline__ void pair_add_square(float& sh, float& sl, float h, float l) {
    const float p = __fmul_rn(h, h);
    const float e = fmaf(2.0f * h, l, fmaf(h, h, -p));
    float t;
    const float s = two_sum(sh, p, t);
    sh = fast_two_sum(s, __fadd_rn(sl, __fadd_rn(t, e)), sl);
}

template <int S>
__device__ __forceinline__ ResSnap<S> snap_load(const StepParams& a, int64_t n, int64_t idx) {
    ResSnap<S> o;
    if constexpr (S == S_F64) {
        const double* sp = static_cast<const double*>(a.snap);
        o.u = sp[idx];
        o.v = sp[n + idx];
    } else {
        const float2* sp = static_cast<const float2*>(a.snap);
        o.u = sp[idx];
        o.v = sp[n + idx];
    }
    return o;
}

// Residual check of one node: compare u^t of the step's input state (pulled
// populations f, force g; FP64 storage: the collision's u, v) with the
// snapshot entry `old` loaded before, store u^t as the new snapshot entry and
// update the thread's partials.
template <int S>
__device__ __forceinline__ void check_node(const StepParams& a, int64_t n, int64_t idx, ResAcc<S>& acc,
                                           const ResSnap<S>& old, const typename StoreT<S>::T f[8],
                                           typename StoreT<S>::T gx, typename StoreT<S>::T gy,
                                           typename StoreT<S>::T u, typename StoreT<S>::T v) {
    if constexpr (S == S_F64) {
        (void)f;
        (void)gx;
        (void)gy;
        double* sp = static_cast<double*>(a.snap);
        sp[idx] = u;
        sp[n + idx] = v;
        const double du = u - old.u, dv = v - old.v;
        // (maxima by the ALU; a NaN among them is left to the flag)
        acc.d = max_bits(acc.d, max_bits(fabs(du), fabs(dv)));
        acc.u = max_bits(acc.u, max_bits(fabs(u), fabs(v)));
        acc.d2 += du * du + dv * dv;
        acc.u2 += u * u + v * v;
        if (!(isfinite(u) && isfinite(v))) acc.bad = 1.0;
    } else {
        (void)u;
        (void)v;
        const float4 w = exact_displacement(f, gx, gy);
        float2* sp = static_cast<float2*>(a.snap);
        sp[idx] = make_float2(w.x, w.y);
        sp[n + idx] = make_float2(w.z, w.w);
        float e, dl;
        // du = u^t - u^(t-w) as a pair: the hi parts' difference exactly,
        // then the lo parts' (both below an ulp of u)
        float dh = two_sum(w.x, -old.u.x, e);
        dh = two_sum(dh, __fadd_rn(e, __fsub_rn(w.y, old.u.y)), dl);
        pair_max_abs(acc.dh, acc.dl, dh, dl);
        pair_add_square(acc.d2h, acc.d2l, dh, dl);
        dh = two_sum(w.z, -old.v.x, e);
        dh = two_sum(dh, __fadd_rn(e, __fsub_rn(w.w, old.v.y)), dl);
        pair_max_abs(acc.dh, acc.dl, dh, dl);
        pair_add_square(acc.d2h, acc.d2l, dh, dl);
        pair_max_abs(acc.uh, acc.ul, w.x, w.y);
        pair_max_abs(acc.uh, acc.ul, w.z, w.w);
        pair_add_square(acc.u2h, acc.u2l, w.x, w.y);
        pair_add_square(acc.u2h, acc.u2l, w.z, w.w);
        if (!(isfinite(w.x) && isfinite(w.z))) acc.bad = 1.0f;
    }
}
__device__ __forceinline__ void combine_res(double w[kRes], const double v[kRes]) {
    w[0] = max_bits(w[0], v[0]);
    w[1] = max_bits(w[1], v[1]);
    w[2] += v[2];
    w[3] += v[3];
    w[4] = max_bits(w[4], v[4]);
}
__device__ __forceinline__ void warp_reduce_res(double w[kRes]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        double v[kRes];
#pragma unroll
        for (int k = 0; k < kRes; ++k) v[k] = __shfl_xor_sync(0xffffffffu, w[k], o);
        combine_res(w, v);
    }
}
// The same across the block's warps (at most 32): every lane of every warp
// brings its warp's partials, thread 0's w receives the block's.
__device__ __forceinline__ void block_reduce_res(double w[kRes], double (*sh)[32], int tid, int nwarps) {
    const int lane = tid & 31, warp = tid >> 5;
    if (lane == 0)
        for (int k = 0; k < kRes; ++k) sh[k][warp] = w[k];
    __syncthreads();
    if (warp == 0) {
        for (int k = 0; k < kRes; ++k) w[k] = lane < nwarps ? sh[k][lane] : 0.0;
        warp_reduce_res(w);
    }
}

// The residual check of two nodes at a time, in packed instructions: the
// partials of the low and the high node of a lane's pairs are kept apart until
// the end, where the halves a lane owns count (own0, own1).
struct ResAcc2 {
    float dh[2] = {0.f, 0.f}, dl[2] = {0.f, 0.f}, uh[2] = {0.f, 0.f}, ul[2] = {0.f, 0.f};
    pair_t d2h = 0, d2l = 0, u2h = 0, u2l = 0, fin = 0;   // fin: 0 until a displacement is not finite
    bool own0 = false, own1 = false;
    __device__ __forceinline__ void to_double(double w[kRes]) const {
        const bool own[2] = {own0, own1};
        float a[2], b[2], c[2], d[2], f[2];
        unpk(fin, f[0], f[1]);
        unpk(d2h, a[0], a[1]);
        unpk(d2l, b[0], b[1]);
        unpk(u2h, c[0], c[1]);
        unpk(u2l, d[0], d[1]);
        for (int k = 0; k < kRes; ++k) w[k] = 0.0;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (own[h]) {
                const double v[kRes] = {max_to_double(dh[h], dl[h]), max_to_double(uh[h], ul[h]),
                                        pair_to_double(a[h], b[h]), pair_to_double(c[h], d[h]), f[h] == 0.0f ? 0.0 : 1.0};
                combine_res(w, v);
            }
    }
};

// (h, l) += (g, m), pairs (about 2^-45 relative).
__device__ __forceinline__ void pair_add(float& h, float& l, float g, float m) {
    float e;
    const float s = two_sum(h, g, e), x = __fadd_rn(__fadd_rn(l, m), e), r = __fadd_rn(s, x);
    l = __fsub_rn(x, __fsub_rn(r, s));
    h = r;
}

// The partials of a thread's, warp's or block's nodes: the maxima as pairs, which
// lose nothing when they are combined, the sums in FP64 from the thread on (their
// pairs have FP32's range, which a block's sum may leave).  An FP64 instruction
// takes 64 cycles of a scheduler: maxima converted in every thread and two
// sums that cross the warp side by side were 38 of them, 5 us of a checked launch of
// k_tile.
struct ResPart {
    float dh, dl, uh, ul;
    double d2, u2;
    bool bad;
    __device__ __forceinline__ void add_maxima(float odh, float odl, float ouh, float oul) {
        pair_max_abs(dh, dl, odh, odl);
        pair_max_abs(uh, ul, ouh, oul);
    }
    // over the warp (in every lane); the sums share their four last steps, d2 in the lower half-warp and u2 in the upper
    __device__ __forceinline__ void add_warp() {
        constexpr unsigned ALL = 0xffffffffu;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            auto get = [&](float v) { return __shfl_xor_sync(ALL, v, o); };
            add_maxima(get(dh), get(dl), get(uh), get(ul));
        }
        const bool upper = threadIdx.x & 16;
        double s = (upper ? u2 : d2) + __shfl_xor_sync(ALL, upper ? d2 : u2, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(ALL, s, o);
        d2 = __shfl_sync(ALL, s, 0);
        u2 = __shfl_sync(ALL, s, 16);
        bad = __any_sync(ALL, bad);
    }
    __device__ __forceinline__ void to_double(double w[kRes]) const {
        w[0] = max_to_double(dh, dl);
        w[1] = max_to_double(uh, ul);
        w[2] = d2;
        w[3] = u2;
        w[4] = bad ? 1.0 : 0.0;
    }
};
__device__ __forceinline__ ResPart res_part(const ResAcc2& r) {
    float a[2], b[2], c[2], d[2], f[2];
    unpk(r.fin, f[0], f[1]);
    unpk(r.d2h, a[0], a[1]);
    unpk(r.d2l, b[0], b[1]);
    unpk(r.u2h, c[0], c[1]);
    unpk(r.u2l, d[0], d[1]);
    ResPart p{0.f, 0.f, 0.f, 0.f, 0.0, 0.0, false};
    float ah = 0.f, al = 0.f, ch = 0.f, cl = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (h ? r.own1 : r.own0) {
            p.add_maxima(r.dh[h], r.dl[h], r.uh[h], r.ul[h]);
            pair_add(ah, al, a[h], b[h]);
            pair_add(ch, cl, c[h], d[h]);
            p.bad |= f[h] != 0.0f;
        }
    p.d2 = pair_to_double(ah, al);
    p.u2 = pair_to_double(ch, cl);
    return p;
}

// two_sum (lbm_core.cuh) on pairs.
__device__ __forceinline__ pair_t two_sum2(pair_t a, pair_t b, pair_t& e) {
    const pair_t s = add2(a, b), bb = sub2(s, a);
    e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
    return s;
}
__device__ __forceinline__ pair_t two_diff2(pair_t a, pair_t b, pair_t& e) {      // a - b
    const pair_t s = sub2(a, b), bb = sub2(s, a);
    e = sub2(sub2(a, sub2(s, bb)), add2(b, bb));
    return s;
}
// s += a^2 + b^2, a and b in two parts each (pair_add_square's terms of both
// squares, joined before they meet the sum).
__device__ __forceinline__ void pair_add_squares2(pair_t& sh, pair_t& sl, pair_t ah, pair_t al, pair_t bh, pair_t bl) {
    float a0, a1, b0, b1;
    unpk(ah, a0, a1);
    unpk(bh, b0, b1);
    const pair_t p = pk(__fmul_rn(a0, a0), __fmul_rn(a1, a1)), q = pk(__fmul_rn(b0, b0), __fmul_rn(b1, b1));
    const pair_t np = pk(__fmul_rn(-a0, a0), __fmul_rn(-a1, a1)), nq = pk(__fmul_rn(-b0, b0), __fmul_rn(-b1, b1));
    const pair_t ea = fma2(add2(ah, ah), al, fma2(ah, ah, np)), eb = fma2(add2(bh, bh), bl, fma2(bh, bh, nq));
    pair_t t, t2;
    const pair_t w = two_sum2(p, q, t), s = two_sum2(sh, w, t2);
    const pair_t x = add2(add2(sl, t2), add2(t, add2(ea, eb))), r = add2(s, x);
    sl = sub2(x, sub2(r, s));
    sh = r;
}
// max over both of |h + l| into (mh, ml): one test for two candidates, which
// few nodes pass once a thread's maximum is established.
__device__ __forceinline__ void pair_max_abs2(float& mh, float& ml, float h, float l, float g, float m) {
    if (fmaxf(fabsf(h), fabsf(g)) >= mh) {
        pair_max_abs(mh, ml, h, l);
        pair_max_abs(mh, ml, g, m);
    }
}

// Residual check of a lane's two nodes (pulled populations f, force gx, gy):
// check_node's arithmetic for FP32 and FP16-shifted storage.  o0, o1: their
// snapshot entries; store(u0, v0, u1, v1) writes the new ones.
template <int S, typename STORE>
__device__ __forceinline__ void check_pair(ResAcc2& acc, const ResSnap<S>& o0, const ResSnap<S>& o1, const pair_t f[8],
                                           pair_t gx, pair_t gy, STORE&& store) {
    const pair_t half = splat(0.5f);
    pair_t er, es, e12, e21, ea, eb, e10, e01, eu, ev;
    const pair_t r = two_diff2(f[4], f[6], er), s = two_diff2(f[5], f[7], es);
    const pair_t m12 = two_diff2(r, s, e12), m21 = two_sum2(r, s, e21);
    const pair_t a = two_diff2(f[0], f[2], ea), b = two_diff2(f[1], f[3], eb);
    const pair_t m10 = two_sum2(a, m12, e10), m01 = two_sum2(b, m21, e01);
    const pair_t u = two_sum2(m10, fma2(half, gx, 0), eu), v = two_sum2(m01, fma2(half, gy, 0), ev);
    const pair_t ulo = add2(add2(add2(eu, e10), add2(ea, e12)), sub2(er, es));
    const pair_t vlo = add2(add2(add2(ev, e01), add2(eb, e21)), add2(er, es));
    pair_t ul, vl;
    const pair_t uh = two_sum2(u, ulo, ul), vh = two_sum2(v, vlo, vl);
    float4 n0, n1;                                // (u hi, u lo, v hi, v lo) of either node
    unpk(uh, n0.x, n1.x);
    unpk(ul, n0.y, n1.y);
    unpk(vh, n0.z, n1.z);
    unpk(vl, n0.w, n1.w);
    store(make_float2(n0.x, n0.y), make_float2(n0.z, n0.w), make_float2(n1.x, n1.y), make_float2(n1.z, n1.w));
    pair_t e, ul2, vl2;
    pair_t du = two_diff2(uh, pk(o0.u.x, o1.u.x), e);
    du = two_sum2(du, add2(e, sub2(ul, pk(o0.u.y, o1.u.y))), ul2);
    pair_t dv = two_diff2(vh, pk(o0.v.x, o1.v.x), e);
    dv = two_sum2(dv, add2(e, sub2(vl, pk(o0.v.y, o1.v.y))), vl2);
    pair_add_squares2(acc.d2h, acc.d2l, du, ul2, dv, vl2);
    pair_add_squares2(acc.u2h, acc.u2l, uh, ul, vh, vl);
    acc.fin = fma2(uh, 0, fma2(vh, 0, acc.fin));
    float x[2], y[2], p[2], q[2];
    unpk(du, x[0], x[1]);
    unpk(ul2, y[0], y[1]);
    unpk(dv, p[0], p[1]);
    unpk(vl2, q[0], q[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float4 n = h ? n1 : n0;
        pair_max_abs2(acc.dh[h], acc.dl[h], x[h], y[h], p[h], q[h]);
        pair_max_abs2(acc.uh[h], acc.ul[h], n.x, n.y, n.z, n.w);
    }
}

// Stored values that the pull of one node reads: the 8 populations f*_p(x - c_p)
// as stored (and, FP16S, the carriers of the 8 source nodes).
template <int S> struct Pulled { typename StoreT<S>::P p[8]; };
template <> struct Pulled<S_F16S> { __half p[8]; float2 c[8]; };

// Load the stored values of the pull of node (x, y) (loads only).
// r0, rm, rp: offsets of rows y, y-1, y+1 (wrapped); xm, xp: columns x-1, x+1.
// I: in-plane offset type (int where a plane has fewer than 2^31 nodes).
template <int S, typename I = int64_t>
__device__ __forceinline__ void pull_load(const StepParams& a, I r0, I rm, I rp,
                                          int x, int xm, int xp, Pulled<S>& q) {
    using P = typename StoreT<S>::P;
    const P* s = static_cast<const P*>(a.src);
    const int64_t pl = a.plane;
    const I i0 = r0 + xm, i1 = rm + x, i2 = r0 + xp, i3 = rp + x;
    const I i4 = rm + xm, i5 = rm + xp, i6 = rp + xp, i7 = rp + xm;
    if constexpr (S == S_F16S) {
        // carriers interleaved per node: (m*_10, m*_01) as one float2
        const float2* c = reinterpret_cast<const float2*>(a.csrc);
        q.c[0] = ldg(c + i0);
        q.c[1] = ldg(c + i1);
        q.c[2] = ldg(c + i2);
        q.c[3] = ldg(c + i3);
        q.c[4] = ldg(c + i4);
        q.c[5] = ldg(c + i5);
        q.c[6] = ldg(c + i6);
        q.c[7] = ldg(c + i7);
    }
    q.p[0] = ldg(s + 0 * pl + i0);
    q.p[1] = ldg(s + 1 * pl + i1);
    q.p[2] = ldg(s + 2 * pl + i2);
    q.p[3] = ldg(s + 3 * pl + i3);
    q.p[4] = ldg(s + 4 * pl + i4);
    q.p[5] = ldg(s + 5 * pl + i5);
    q.p[6] = ldg(s + 6 * pl + i6);
    q.p[7] = ldg(s + 7 * pl + i7);
}

// The pre-collision populations f_p(x) from the pulled stored values
// (FP16S: the stored deviation + the equilibrium part of the source carrier,
// both in the state's scaled units; see store_f16s).
template <int S>
__device__ __forceinline__ void pull_decode(const StepParams& a, const Pulled<S>& q,
                                            typename StoreT<S>::T f[8], typename StoreT<S>::T theta) {
    using T = typename StoreT<S>::T;
    if constexpr (S == S_F16S) {
        (void)a;
        const float k1 = 0.5f * (1.0f - theta), k5 = 0.25f * theta;
        f[0] = fmad(k1, q.c[0].x, __half2float(q.p[0]));
        f[1] = fmad(k1, q.c[1].y, __half2float(q.p[1]));
        f[2] = fmad(-k1, q.c[2].x, __half2float(q.p[2]));
        f[3] = fmad(-k1, q.c[3].y, __half2float(q.p[3]));
        f[4] = fmad(k5, q.c[4].x + q.c[4].y, __half2float(q.p[4]));
        f[5] = fmad(k5, q.c[5].y - q.c[5].x, __half2float(q.p[5]));
        f[6] = fmad(-k5, q.c[6].x + q.c[6].y, __half2float(q.p[6]));
        f[7] = fmad(k5, q.c[7].x - q.c[7].y, __half2float(q.p[7]));
    } else {
        (void)a;
        (void)theta;
#pragma unroll
        for (int p = 0; p < 8; ++p) f[p] = T(q.p[p]);
    }
}

// Gather the pre-collision populations of node (x, y): f_p(x) = f*_p(x - c_p).
template <int S>
__device__ __forceinline__ void gather(const StepParams& a, int64_t r0, int64_t rm, int64_t rp,
                                       int x, int xm, int xp, typename StoreT<S>::T f[8],
                                       typename StoreT<S>::T theta) {
    Pulled<S> q;
    pull_load<S>(a, r0, rm, rp, x, xm, xp, q);
    pull_decode<S>(a, q, f, theta);
}

// FP16-shifted store of one node: the deviations N (FP32) are rounded to
// FP16, and the FP32 carriers absorb the first moments of the ROUNDED
// deviations, c10 = m*_10 - m_10(N_rounded), so that the stored state
// N_rounded + E(c) keeps the first moments m*_10, m*_01 exactly (E(c) has
// first moments c, no second moments).  Without this, the rounding of N would
// feed the conserved mean-displacement mode every step and u would drift.
// Scaled units: an FP16S lattice keeps its whole FP32 state -- carriers,
// force, intermediate populations, residual snapshot -- multiplied by its
// power-of-two scale 2^e (StepParams::hscale), chosen so that the deviations
// sit well inside FP16's normal range.  The scale commutes with every
// rounding, so this is the same arithmetic as unscaled values with the FP16
// rounding done on N 2^e, without a multiplication per population in the
// decode and two here; only the recovery, the export, the import and the
// reported norms of u convert.
__device__ __forceinline__ void store_f16s(const StepParams& a, int64_t idx, const float n[8],
                                           float m10s, float m01s) {
    __half* d = static_cast<__half*>(a.dst);
    const int64_t pl = a.plane;
    float r[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        const __half h = __float2half_rn(n[p]);
        d[p * pl + idx] = h;
        r[p] = __half2float(h);
    }
    const float e10 = (r[0] - r[2]) + ((r[4] - r[6]) - (r[5] - r[7]));
    const float e01 = (r[1] - r[3]) + ((r[4] - r[6]) + (r[5] - r[7]));
    reinterpret_cast<float2*>(a.cdst)[idx] = make_float2(m10s - e10, m01s - e01);
}

// The values a node stores after its collision (raw moments m, force g; GEN
// as for collide): the eight post-collision populations, or for FP16S the
// eight deviations N and the carriers (c10, c01) = (m*_10, m*_01); u, v
// receive the displacement.  Computed apart from the stores so that kernels
// can run it on every thread and predicate only the stores.
template <int S, bool GEN>
__device__ __forceinline__ void post_state(const Mom<typename StoreT<S>::T>& m, typename StoreT<S>::T gx,
                                           typename StoreT<S>::T gy, const Coef<typename StoreT<S>::T>& c,
                                           typename StoreT<S>::T& u, typename StoreT<S>::T& v,
                                           typename StoreT<S>::T f[8], float& c10, float& c01) {
    using T = typename StoreT<S>::T;
    if constexpr (S == S_F16S) {
        const Mom<T> s = collide<T, GEN>(m, gx, gy, c, u, v);
        populations<!GEN>(deviation_moments(s, c.qtheta), f);
        c10 = s.m10;
        c01 = s.m01;
    } else {
        collide_populations<GEN>(m, gx, gy, c, u, v, f);
        c10 = c01 = 0.0f;
    }
}

// Store the post_state values of node idx.
template <int S>
__device__ __forceinline__ void store_state(const StepParams& a, int64_t idx, const typename StoreT<S>::T f[8],
                                            float c10, float c01) {
    using P = typename StoreT<S>::P;
    if constexpr (S == S_F16S) {
        store_f16s(a, idx, f, c10, c01);
    } else {
        P* d = static_cast<P*>(a.dst);
        const int64_t pl = a.plane;
#pragma unroll
        for (int p = 0; p < 8; ++p) d[p * pl + idx] = P(f[p]);
    }
}

// Collide node idx (raw moments m, force g) and store its post-collision
// state.
template <int S, bool GEN>
__device__ __forceinline__ void scatter_local(const StepParams& a, int64_t idx,
                                              const Mom<typename StoreT<S>::T>& m,
                                              typename StoreT<S>::T gx, typename StoreT<S>::T gy,
                                              const Coef<typename StoreT<S>::T>& c) {
    typename StoreT<S>::T f[8], u, v;
    float c10, c01;
    post_state<S, GEN>(m, gx, gy, c, u, v, f, c10, c01);
    store_state<S>(a, idx, f, c10, c01);
}

// Residual reduction of a block.  Each thread's partials (ResAcc) are
// converted to FP64 and combined across the warp, the block and the grid in
// FP64.  With a counter, the grid-level pass is done by the last block to
// finish (counted with an atomic), which also resets the counter for the next
// check; without one (the library's own check launches) the blocks stop after
// writing their partials and k_residual_finish combines them in a separate
// launch.
// Paired partials (no counter): the block's partial set.
__device__ __forceinline__ void residual_reduce_pairs(const StepParams& a, const ResAcc2& acc) {
    __shared__ ResPart sh[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    ResPart p = res_part(acc);
    p.add_warp();
    if (lane == 0) sh[warp] = p;
    __syncthreads();
    if (warp != 0) return;
    if (lane < (int)(blockDim.x >> 5)) p = sh[lane];
    else p = ResPart{0.f, 0.f, 0.f, 0.f, 0.0, 0.0, false};
    p.add_warp();
    if (lane != 0) return;
    double w[kRes];
    p.to_double(w);
    for (int k = 0; k < kRes; ++k) a.partials[(int64_t)blockIdx.x * kRes + k] = w[k];
}
template <typename ACC>
__device__ __forceinline__ void residual_reduce(const StepParams& a, const ACC& acc) {
    __shared__ double sh[kRes][32];
    __shared__ bool is_last;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nthr = blockDim.x * blockDim.y, nwarps = nthr >> 5;
    double v[kRes];
    acc.to_double(v);
    warp_reduce_res(v);
    block_reduce_res(v, sh, tid, nwarps);
    const unsigned int nblocks = gridDim.x * gridDim.y;
    const unsigned int bid = blockIdx.y * gridDim.x + blockIdx.x;
    if (tid == 0) {
        for (int k = 0; k < kRes; ++k) a.partials[(int64_t)bid * kRes + k] = v[k];
        if (a.counter != nullptr) {
            __threadfence();
            const unsigned int done = atomicAdd(a.counter, 1u);
            is_last = (done == nblocks - 1);
        }
    }
    // Partials only: a later k_residual_finish launch combines them, so the
    // block ends here without a memory fence or a grid counter.
    if (a.counter == nullptr) return;
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    double w[kRes] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (unsigned int b = tid; b < nblocks; b += nthr) {
        double q[kRes];
#pragma unroll
        for (int k = 0; k < kRes; ++k) q[k] = __ldcg(a.partials + (int64_t)b * kRes + k);
        combine_res(w, q);
    }
    warp_reduce_res(w);
    block_reduce_res(w, sh, tid, nwarps);
    if (tid == 0) {
        for (int k = 0; k < kRes; ++k) a.result[k] = w[k];
        *a.counter = 0u;
        __threadfence();
    }
}

// One pseudo-time step (Algorithm 1) over the whole lattice.
//
// The lattice is cut into tiles of 32*V columns by BY rows; block b handles
// tiles b, b + gridDim.x, ...  The plain step is launched with one block per
// tile.  CHECK adds the steady-state residual: u^t (the displacement of this
// step's input state) is compared with the snapshot taken at the previous
// check, the snapshot is overwritten with u^t, and each block reduces its
// partials once, after all of its tiles (FP64 across warps, blocks and the
// grid).  The library launches it with one block per tile up to
// kMaxCheckBlocks blocks (more tiles per block beyond that).
// One tile of one step: tile (tx, ty) covers columns tx*32V .. tx*32V+32V-1
// and rows ty*BY .. ty*BY+BY-1.  With CHECK the thread's residual partials
// are accumulated into acc.
template <int S, int V, bool GEN, bool CHECK>
__device__ __forceinline__ void step_tile(const StepParams& a,
                                          const Coef<typename StoreT<S>::T>& c, int tx, int ty,
                                          ResAcc<S>& acc) {
    using T = typename StoreT<S>::T;
    using G = typename StoreT<S>::G;
    const int nx = a.nx, ny = a.ny;
    const int y = ty * BY + threadIdx.y;
    const int xb = tx * (32 * V) + threadIdx.x;
    if (y >= ny) return;
    const G* __restrict__ gxp = static_cast<const G*>(a.gx);
    const G* __restrict__ gyp = static_cast<const G*>(a.gy);
    const int64_t n = a.plane;
    const int ym = wrap_dec(y, ny), yp = wrap_inc(y, ny);
    const int64_t r0 = (int64_t)y * a.pitch, rm = (int64_t)ym * a.pitch, rp = (int64_t)yp * a.pitch;
    // Phase 1: issue every load of the thread's V nodes before any store,
    // so that up to V*10 (V*12 with the snapshot) loads are in flight.
    T f[V][8], gx[V], gy[V];
    ResSnap<S> so[V];
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const int x = xb + 32 * j;
        if (x < nx) {
            gather<S>(a, r0, rm, rp, x, wrap_dec(x, nx), wrap_inc(x, nx), f[j], c.theta);
            gx[j] = T(ldg(gxp + r0 + x));
            gy[j] = T(ldg(gyp + r0 + x));
            if (CHECK) so[j] = snap_load<S>(a, n, r0 + x);
        }
    }
    // Phase 2: collide and store.
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const int x = xb + 32 * j;
        if (x < nx) {
            const int64_t idx = r0 + x;
            if constexpr (S == S_F64) {
                T u, v, fs[8];
                step_f64<GEN>(f[j], gx[j], gy[j], c, u, v, fs);
                store_state<S>(a, idx, fs, 0.0f, 0.0f);
                if (CHECK) check_node<S>(a, n, idx, acc, so[j], f[j], gx[j], gy[j], u, v);
            } else {
                const Mom<T> m = moments(f[j]);
                scatter_local<S, GEN>(a, idx, m, gx[j], gy[j], c);
                if (CHECK) {
                    T u, v;
                    displacement(m, gx[j], gy[j], u, v);
                    check_node<S>(a, n, idx, acc, so[j], f[j], gx[j], gy[j], u, v);
                }
            }
        }
    }
}

template <int S, int V, bool GEN, bool CHECK>
__global__ void __launch_bounds__(kThreads, CHECK ? 2 : (S == S_F32 ? LBM_MINB_F32 : LBM_MINB_F16S))
k_step(const StepParams a, const Coef<typename StoreT<S>::T> c) {
    after_predecessor();
    const int ntx = (a.nx + 32 * V - 1) / (32 * V);
    const int64_t ntiles = (int64_t)ntx * ((a.ny + BY - 1) / BY);
    ResAcc<S> acc;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int ty = (int)(t / ntx), tx = (int)(t - (int64_t)ty * ntx);
        step_tile<S, V, GEN, CHECK>(a, c, tx, ty, acc);
    }
    if (CHECK) residual_reduce(a, acc);
}

// Periodic image in [0, n) of a slot coordinate v >= -1.  ANY = false
// needs n at least the slot span (one conditional subtraction); ANY = true
// serves any n (a lattice smaller than the slot array appears in it more
// than once).  The two are separate kernels because the general form costs
// the large-lattice kernel 4-6 % even where it never takes the long path.
template <bool ANY>
__device__ __forceinline__ int wrap_slot(int v, int n) {
    if (v < 0) v += n;
    if (ANY && v < 0) v = v % n + n;   // v >= -2 on a lattice of one node
    if (v >= n) v = (!ANY || v < 2 * n) ? v - n : v % n;
    return v;
}

// Pulled populations and stored ones of FP64 storage, by node indices of 31 bits
// (a state of 2^31 nodes is larger than the device's memory).
__device__ __forceinline__ void pull64(const StepParams& a, int r0, int rm, int rp, int x, int xm, int xp, double f[8]) {
    const double* s = static_cast<const double*>(a.src);
    const int64_t pl = a.plane;
    f[0] = ldg(s + 0 * pl + (r0 + xm));                       // f_p(x) = f*_p(x - c_p)
    f[1] = ldg(s + 1 * pl + (rm + x));
    f[2] = ldg(s + 2 * pl + (r0 + xp));
    f[3] = ldg(s + 3 * pl + (rp + x));
    f[4] = ldg(s + 4 * pl + (rm + xm));
    f[5] = ldg(s + 5 * pl + (rm + xp));
    f[6] = ldg(s + 6 * pl + (rp + xp));
    f[7] = ldg(s + 7 * pl + (rp + xm));
}
__device__ __forceinline__ void push64(const StepParams& a, int idx, const double f[8]) {
    double* d = static_cast<double*>(a.dst);
#pragma unroll
    for (int p = 0; p < 8; ++p) (d + p * a.plane)[idx] = f[p];
}

// A launch of FP64 storage: T steps; T > 1: blocks of bx x by nodes (k_tile64),
// T = 1: k_one64.
constexpr int kT64Max = 4;        // most steps per launch
constexpr int kT64Smem = 48 * 1024;
struct Tile64Shape {
    int T = 0, bx = 0, by = 0;
    int inv[kT64Max] = {};        // step t: 2^16 / (width of its slots), rounded up
    double cost = 0.0;            // modelled cycles of one launch
};

// ---------------------------------------------------------------------------
// T pseudo-time steps per launch of FP64 storage (T >= 1, a run-time count).
//
// A step of a node is some 600 instructions in a row (step_f64), so a small
// lattice is spread over all SMs, and every node over two lanes (step_f64_half): a
// block owns bx x by nodes, holds the states between its steps in shared memory
// over a halo that shrinks by one node per step, and its threads take the slots
// of a step in linear order.  The periodic images of the slots' columns and rows
// come from a table that is made before the wait for the predecessor.  Several
// steps per launch recompute the halos but save launches; tile64_shape weighs
// the two.  64 x 64: 1.11 us per step (one lane per node 1.39, two without the
// table 1.21; on the FP64 pipe 2.05, one step of 64 x 8 tiles per launch 8.3).
// What is left is latency: of a launch's 2 us, and of about 0.5 us per step.
template <bool GEN, bool CHECK>
__global__ void __launch_bounds__(512)
k_tile64(const StepParams a, const Coef<double> c, const __grid_constant__ Tile64Shape sh, int nty) {
    extern __shared__ double tile64_mem[];
    const int nx = a.nx, ny = a.ny, H = sh.T - 1, sw = sh.bx + 2 * H, sr = sh.by + 2 * H, area = sw * sr;
    ResAcc<S_F64> acc;
    const int x0 = (int)blockIdx.x * sh.bx - H;               // node of slot (0, 0)
    // the lane's half of a node: populations h, h + 2, h + 4, h + 6 and the force's
    // component h; f_p(x) = f*_p(x - c_p)
    const int h = threadIdx.x & 1, d1 = h ? 1 : -1;
    const int64_t pl = a.plane;
    const double *src = static_cast<const double*>(a.src) + h * pl, *force = static_cast<const double*>(h ? a.gy : a.gx);
    double* dst = static_cast<double*>(a.dst) + h * pl;
    const int off0 = h * area + (h ? -sw : -1), off1 = (2 + h) * area + (h ? sw : 1), off2 = (4 + h) * area - sw + d1,
              off3 = (6 + h) * area + sw - d1;
    // lattice column, and first node of the lattice row, of the slots -1 .. sw, -1 .. sr
    int* col = reinterpret_cast<int*>(tile64_mem + 16 * area) + 1;
    int* row = col + sw + 2;
    for (int ty = blockIdx.y; ty < nty; ty += gridDim.y) {
        const int y0 = ty * sh.by - H;
        for (int i = threadIdx.x; i < sw + sr + 4; i += blockDim.x) {
            const bool c = i < sw + 2;
            const int n = c ? nx : ny, v = (c ? x0 + i : y0 + i - (sw + 2)) - 1, m = v % n;
            col[i - 1] = (m < 0 ? m + n : m) * (c ? 1 : (int)a.pitch);
        }
        __syncthreads();
        after_predecessor();
        for (int t = 0; t <= H; ++t) {
            const bool last = t == H;
            const int aw = sw - 2 * t, count = aw * (sh.by + 2 * (H - t)), inv = sh.inv[t];
            const double* from = tile64_mem + (t & 1) * 8 * area;
            double* to = tile64_mem + ((t + 1) & 1) * 8 * area;
            // two lanes per slot; whole warps go round, past the last slot too
            for (int i = threadIdx.x; (i & ~31) < 2 * count; i += blockDim.x) {
                const int slot = min(i >> 1, count - 1);
                const int q = (slot * inv) >> 16, sx = t + slot - q * aw, sy = t + q;   // q = slot / aw
                const bool own = (i >> 1) < count && (!last || (x0 + sx < nx && y0 + sy < ny));
                const int x = col[sx], y = row[sy], idx = y + x, at = sy * sw + sx;
                double f[4];
                if (t == 0) {
                    const int rm = row[sy - 1], rp = row[sy + 1], xl = col[sx + d1], xr = col[sx - d1];
                    f[0] = ldg(src + (h ? rm + x : y + xl));
                    f[1] = ldg(src + 2 * pl + (h ? rp + x : y + xr));
                    f[2] = ldg(src + 4 * pl + (rm + xl));
                    f[3] = ldg(src + 6 * pl + (rp + xr));
                } else {
                    f[0] = from[at + off0];
                    f[1] = from[at + off1];
                    f[2] = from[at + off2];
                    f[3] = from[at + off3];
                }
                const double g = ldg(force + idx);
                double w, fs[4];
                step_f64_half<GEN>(f, g, h, c, w, fs);
                if (!last) {
                    if (own) {
#pragma unroll
                        for (int p = 0; p < 4; ++p) to[at + (2 * p + h) * area] = fs[p];
                    }
                    continue;
                }
                if (CHECK) {
                    const double v = __shfl_xor_sync(0xffffffffu, w, 1);
                    const double zero[8] = {};
                    if (own && h == 0)
                        check_node<S_F64>(a, pl, idx, acc, snap_load<S_F64>(a, pl, idx), zero, 0.0, 0.0, w, v);
                }
                if (own) {
#pragma unroll
                    for (int p = 0; p < 4; ++p) (dst + 2 * p * pl)[idx] = fs[p];
                }
            }
            if (H) __syncthreads();
        }
    }
    if (CHECK) residual_reduce(a, acc);
}

// One step per launch of FP64 storage (lattices of some 200 x 200 nodes and more):
// blocks of 32 x 4 nodes.  1500 x 1100: 37.8 us per step, 238 MB of populations
// and force at 6.3 TB/s (with 64-bit tile divisions and
// addresses 47; on the FP64 pipe 116, with tiles of 64 x 8 137).
constexpr int kOne64Rows = 4;
template <bool GEN, bool CHECK>
__global__ void __launch_bounds__(32 * kOne64Rows)
k_one64(const StepParams a, const Coef<double> c, int nty) {
    const int nx = a.nx, ny = a.ny, pitch = (int)a.pitch;
    ResAcc<S_F64> acc;
    after_predecessor();
    const int x = (int)blockIdx.x * 32 + threadIdx.x;
    for (int ty = blockIdx.y; ty < nty; ty += gridDim.y) {
        const int y = ty * kOne64Rows + threadIdx.y;
        if (x >= nx || y >= ny) continue;
        const int row = y * pitch, idx = row + x;
        double f[8];
        pull64(a, row, wrap_dec(y, ny) * pitch, wrap_inc(y, ny) * pitch, x, wrap_dec(x, nx), wrap_inc(x, nx), f);
        const double gx = ldg(static_cast<const double*>(a.gx) + idx), gy = ldg(static_cast<const double*>(a.gy) + idx);
        double u, v, fs[8];
        step_f64<GEN>(f, gx, gy, c, u, v, fs);
        if (CHECK) check_node<S_F64>(a, a.plane, idx, acc, snap_load<S_F64>(a, a.plane, idx), f, gx, gy, u, v);
        push64(a, idx, fs);
    }
    if (CHECK) residual_reduce(a, acc);
}

// ---------------------------------------------------------------------------
// Two pseudo-time steps per launch, FP32 or FP16-shifted storage (temporal
// blocking).
//
// A block of 256 threads (8 warps) owns one output tile of kT2OX x kT2OY
// nodes (62 x 22) and a slot array of kT2W x kT2H nodes (64 x 24, 48 KB of
// FP32 populations): the tile grown by one node on every side.  Step 1 pulls the stored f*(t) from global memory exactly as
// the single step does, collides every slot and keeps f*(t+1) of all slots in
// shared memory; step 2 pulls f*(t+1) of the tile's nodes from shared memory
// (their pull neighbours are the halo slots), collides again and stores
// f*(t+2) of the tile.  The state crosses HBM once per two steps: per node and
// launch 32 bytes read, 32 written and 8 of force read, i.e. 36 bytes per
// lattice update instead of 72 (FP16-shifted: 28 instead of 56).  Thread
// (lane, warp) owns slot columns lane and lane + 32 and slot rows warp + 8k in
// both steps, so the force it loaded in step 1 serves step 2 from registers.
// The per-node arithmetic is the single step's (gather, collide, populations),
// so with FP32 storage a launch reproduces two single-step launches exactly.
// With FP16-shifted storage the intermediate state f*(t+1) stays in FP32
// (only the state written back is rounded to the storage format), so results
// differ from one step per launch by less than the storage rounding.
//
// Any lattice size works: slot coordinates wrap periodically, and a lattice
// smaller than the slot array appears in it more than once (ANY = true, the
// general wrap; the batched arena uses it for every problem).  A lattice of
// at least kT2W x kT2H (step2_fits) takes the ANY = false kernel, whose wrap
// is one conditional subtraction.  CHECK makes the second step the
// residual-check step of k_step<..., CHECK> (snapshot compared with u^{t+1},
// the second step's input state); its snapshot loads are issued before the
// barrier between the steps.
#ifndef LBM_T2_RPW
#define LBM_T2_RPW 3
#endif
#ifndef LBM_MINB_T2
#define LBM_MINB_T2 3
#endif
#ifndef LBM_MINB_T2_F16S
#define LBM_MINB_T2_F16S 4
#endif
#ifndef LBM_T2_B
#define LBM_T2_B 1
#endif
constexpr int kT2Rows = LBM_T2_RPW;             // slot rows per warp
constexpr int kT2B = LBM_T2_B;                  // slot rows gathered together in step 1
static_assert(kT2Rows % kT2B == 0, "rows per warp must be a multiple of the gather batch");
constexpr int kT2W = 64;                        // slot columns (two per lane)
constexpr int kT2H = 8 * kT2Rows;               // slot rows
constexpr int kT2OX = kT2W - 2, kT2OY = kT2H - 2;
constexpr int kT2Threads = 256;
constexpr int kT2Smem = 8 * kT2H * kT2W * (int)sizeof(float);
static_assert(kT2Threads == kThreads, "residual_reduce sizes its scratch by kThreads");

template <int S, bool GEN, bool CHECK, bool ANY>
__device__ __forceinline__ void step2_tile(const StepParams& a, const Coef<float>& c, float* sm,
                                           int tx, int ty, ResAcc<S>& acc) {
    constexpr int PL = kT2H * kT2W;             // shared-memory plane
    const int nx = a.nx, ny = a.ny;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x0 = tx * kT2OX - 1, y0 = ty * kT2OY - 1;   // node of slot (0, 0)
    const float* __restrict__ gxp = static_cast<const float*>(a.gx);
    const float* __restrict__ gyp = static_cast<const float*>(a.gy);
    int X[2], XM[2], XP[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int x = wrap_slot<ANY>(x0 + lane + 32 * j, nx);
        X[j] = x;
        XM[j] = wrap_dec(x, nx);
        XP[j] = wrap_inc(x, nx);
    }
    float gx[kT2Rows][2], gy[kT2Rows][2];   // force of the thread's slots
    // Step 1: f*(t+1) of every slot into shared memory.
#pragma unroll
    for (int kb = 0; kb < kT2Rows; kb += kT2B) {
        float f[kT2B][2][8];
#pragma unroll
        for (int b = 0; b < kT2B; ++b) {
            const int k = kb + b;
            const int y = wrap_slot<ANY>(y0 + warp + 8 * k, ny);
            const int64_t r0 = (int64_t)y * a.pitch;
            const int64_t rm = (int64_t)wrap_dec(y, ny) * a.pitch, rp = (int64_t)wrap_inc(y, ny) * a.pitch;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                gather<S>(a, r0, rm, rp, X[j], XM[j], XP[j], f[b][j], c.theta);
                gx[k][j] = ldg(gxp + r0 + X[j]);
                gy[k][j] = ldg(gyp + r0 + X[j]);
            }
        }
#pragma unroll
        for (int b = 0; b < kT2B; ++b) {
            const int k = kb + b, r = warp + 8 * k;
            float* s = sm + r * kT2W + lane;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float u, v, fs[8];
                collide_populations<GEN>(moments(f[b][j]), gx[k][j], gy[k][j], c, u, v, fs);
#pragma unroll
                for (int p = 0; p < 8; ++p) s[p * PL + 32 * j] = fs[p];
            }
        }
    }
    const int64_t n = a.plane;
    ResSnap<S> so[kT2Rows][2];
    if (CHECK) {
#pragma unroll
        for (int k = 0; k < kT2Rows; ++k) {
            const int r = warp + 8 * k, y = y0 + r;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int col = lane + 32 * j, x = x0 + col;
                if (r >= 1 && r <= kT2H - 2 && y < ny && col >= 1 && col <= kT2W - 2 && x < nx)
                    so[k][j] = snap_load<S>(a, n, (int64_t)y * a.pitch + x);
            }
        }
    }
    __syncthreads();
    // Step 2: the tile's nodes pull f*(t+1) from shared memory.
#pragma unroll
    for (int k = 0; k < kT2Rows; ++k) {
        const int r = warp + 8 * k;
        const int y = y0 + r;
        if (r < 1 || r > kT2H - 2 || y >= ny) continue;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int col = lane + 32 * j;
            const int x = x0 + col;
            if (col < 1 || col > kT2W - 2 || x >= nx) continue;
            const int64_t idx = (int64_t)y * a.pitch + x;
            const float* s = sm + r * kT2W + col;
            float f[8];
            f[0] = s[0 * PL - 1];               // f_p(x) = f*_p(x - c_p)
            f[1] = s[1 * PL - kT2W];
            f[2] = s[2 * PL + 1];
            f[3] = s[3 * PL + kT2W];
            f[4] = s[4 * PL - kT2W - 1];
            f[5] = s[5 * PL - kT2W + 1];
            f[6] = s[6 * PL + kT2W + 1];
            f[7] = s[7 * PL + kT2W - 1];
            const Mom<float> m = moments(f);
            scatter_local<S, GEN>(a, idx, m, gx[k][j], gy[k][j], c);
            if (CHECK) {
                float u, v;
                displacement(m, gx[k][j], gy[k][j], u, v);
                check_node<S>(a, n, idx, acc, so[k][j], f, gx[k][j], gy[k][j], u, v);
            }
        }
    }
}

#ifndef LBM_MINB_T2_CHECK
#define LBM_MINB_T2_CHECK 3
#endif
template <int S, bool GEN, bool CHECK, bool ANY>
__global__ void __launch_bounds__(kT2Threads,
                                  CHECK ? LBM_MINB_T2_CHECK : (S == S_F16S ? LBM_MINB_T2_F16S : LBM_MINB_T2))
k_step2(const StepParams a, const Coef<float> c) {
    after_predecessor();
    extern __shared__ float t2_smem[];
    const int ntx = (a.nx + kT2OX - 1) / kT2OX;
    const int64_t ntiles = (int64_t)ntx * ((a.ny + kT2OY - 1) / kT2OY);
    ResAcc<S> acc;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int ty = (int)(t / ntx), tx = (int)(t - (int64_t)ty * ntx);
        step2_tile<S, GEN, CHECK, ANY>(a, c, t2_smem, tx, ty, acc);
        if (t + gridDim.x < ntiles) __syncthreads();   // slots are reused by the next tile
    }
    if (CHECK) residual_reduce(a, acc);
}

// ---------------------------------------------------------------------------
// Three pseudo-time steps per launch (FP32 or FP16-shifted storage).
//
// The two-step scheme carried one step further: a block of 256 threads owns an
// output tile of kT3OX x kT3OY nodes (60 x 12) and two shared-memory slot
// arrays A and B of kT3W x kT3H slots (64 x 16, 32 KB each): the tile grown
// by two nodes on every side.  Step 1 pulls f*(t) from global memory and
// writes f*(t+1) of every slot to A; step 2 pulls from A and writes f*(t+2)
// of the slots one node inside the edge to B; step 3 pulls from B and stores
// f*(t+3) of the tile.  Per node and launch the state crosses HBM once: 72 B
// (FP32) or 56 B (FP16S) for three lattice updates.  Thread (lane, warp) owns
// slot columns lane and lane + 32 and rows warp + 8k in all three steps; the
// per-node arithmetic is the single step's, so FP32 results equal three
// single-step launches bit for bit (FP16S keeps the two intermediate states
// in FP32).  CHECK would make the third step the residual-check step; the
// library puts its checks on two-step launches instead, which cost less
// relative to their plain form.  ANY as for k_step2; the library uses the
// ANY = false kernel from kT3W x kT3H nodes up.
#ifndef LBM_T3_RPW
#define LBM_T3_RPW 2
#endif
#ifndef LBM_MINB_T3
#define LBM_MINB_T3 3
#endif
constexpr int kT3Rows = LBM_T3_RPW;             // slot rows per warp
constexpr int kT3W = 64;                        // slot columns (two per lane)
constexpr int kT3H = 8 * kT3Rows;               // slot rows
constexpr int kT3OX = kT3W - 4, kT3OY = kT3H - 4;
constexpr int kT3Smem = 2 * 8 * kT3H * kT3W * (int)sizeof(float);

template <int S, bool GEN, bool CHECK, bool ANY>
__device__ __forceinline__ void step3_tile(const StepParams& a, const Coef<float>& c, float* smA,
                                           int tx, int ty, ResAcc<S>& acc) {
    constexpr int PL = kT3H * kT3W;             // shared-memory plane
    float* smB = smA + 8 * PL;
    const int nx = a.nx, ny = a.ny;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x0 = tx * kT3OX - 2, y0 = ty * kT3OY - 2;   // node of slot (0, 0)
    const float* __restrict__ gxp = static_cast<const float*>(a.gx);
    const float* __restrict__ gyp = static_cast<const float*>(a.gy);
    int X[2], XM[2], XP[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int x = wrap_slot<ANY>(x0 + lane + 32 * j, nx);
        X[j] = x;
        XM[j] = wrap_dec(x, nx);
        XP[j] = wrap_inc(x, nx);
    }
    float gx[kT3Rows][2], gy[kT3Rows][2];
    // Step 1: f*(t+1) of every slot into A.
#pragma unroll
    for (int k = 0; k < kT3Rows; ++k) {
        const int r = warp + 8 * k;
        const int y = wrap_slot<ANY>(y0 + r, ny);
        const int64_t r0 = (int64_t)y * a.pitch;
        const int64_t rm = (int64_t)wrap_dec(y, ny) * a.pitch, rp = (int64_t)wrap_inc(y, ny) * a.pitch;
        float f[2][8];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            gather<S>(a, r0, rm, rp, X[j], XM[j], XP[j], f[j], c.theta);
            gx[k][j] = ldg(gxp + r0 + X[j]);
            gy[k][j] = ldg(gyp + r0 + X[j]);
        }
        float* s = smA + r * kT3W + lane;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float u, v, fs[8];
            collide_populations<GEN>(moments(f[j]), gx[k][j], gy[k][j], c, u, v, fs);
#pragma unroll
            for (int p = 0; p < 8; ++p) s[p * PL + 32 * j] = fs[p];
        }
    }
    __syncthreads();
    // Step 2: f*(t+2) of the slots one node inside the edge, from A into B.
#pragma unroll
    for (int k = 0; k < kT3Rows; ++k) {
        const int r = warp + 8 * k;
        if (r < 1 || r > kT3H - 2) continue;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int col = lane + 32 * j;
            if (col < 1 || col > kT3W - 2) continue;
            const float* s = smA + r * kT3W + col;
            float f[8];
            f[0] = s[0 * PL - 1];               // f_p(x) = f*_p(x - c_p)
            f[1] = s[1 * PL - kT3W];
            f[2] = s[2 * PL + 1];
            f[3] = s[3 * PL + kT3W];
            f[4] = s[4 * PL - kT3W - 1];
            f[5] = s[5 * PL - kT3W + 1];
            f[6] = s[6 * PL + kT3W + 1];
            f[7] = s[7 * PL + kT3W - 1];
            float u, v, fs[8];
            collide_populations<GEN>(moments(f), gx[k][j], gy[k][j], c, u, v, fs);
            float* d = smB + r * kT3W + col;
#pragma unroll
            for (int p = 0; p < 8; ++p) d[p * PL] = fs[p];
        }
    }
    const int64_t n = a.plane;
    ResSnap<S> so[kT3Rows][2];
    if (CHECK) {
#pragma unroll
        for (int k = 0; k < kT3Rows; ++k) {
            const int r = warp + 8 * k, y = y0 + r;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int col = lane + 32 * j, x = x0 + col;
                if (r >= 2 && r <= kT3H - 3 && y < ny && col >= 2 && col <= kT3W - 3 && x < nx)
                    so[k][j] = snap_load<S>(a, n, (int64_t)y * a.pitch + x);
            }
        }
    }
    __syncthreads();
    // Step 3: the tile's nodes pull f*(t+2) from B and store f*(t+3).
#pragma unroll
    for (int k = 0; k < kT3Rows; ++k) {
        const int r = warp + 8 * k;
        const int y = y0 + r;
        if (r < 2 || r > kT3H - 3 || y >= ny) continue;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int col = lane + 32 * j;
            const int x = x0 + col;
            if (col < 2 || col > kT3W - 3 || x >= nx) continue;
            const int64_t idx = (int64_t)y * a.pitch + x;
            const float* s = smB + r * kT3W + col;
            float f[8];
            f[0] = s[0 * PL - 1];
            f[1] = s[1 * PL - kT3W];
            f[2] = s[2 * PL + 1];
            f[3] = s[3 * PL + kT3W];
            f[4] = s[4 * PL - kT3W - 1];
            f[5] = s[5 * PL - kT3W + 1];
            f[6] = s[6 * PL + kT3W + 1];
            f[7] = s[7 * PL + kT3W - 1];
            const Mom<float> m = moments(f);
            scatter_local<S, GEN>(a, idx, m, gx[k][j], gy[k][j], c);
            if (CHECK) {
                float u, v;
                displacement(m, gx[k][j], gy[k][j], u, v);
                check_node<S>(a, n, idx, acc, so[k][j], f, gx[k][j], gy[k][j], u, v);
            }
        }
    }
}

template <int S, bool GEN, bool CHECK, bool ANY>
__global__ void __launch_bounds__(kT2Threads, LBM_MINB_T3)
k_step3(const StepParams a, const Coef<float> c) {
    after_predecessor();
    extern __shared__ float t3_smem[];
    const int ntx = (a.nx + kT3OX - 1) / kT3OX;
    const int64_t ntiles = (int64_t)ntx * ((a.ny + kT3OY - 1) / kT3OY);
    ResAcc<S> acc;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int ty = (int)(t / ntx), tx = (int)(t - (int64_t)ty * ntx);
        step3_tile<S, GEN, CHECK, ANY>(a, c, t3_smem, tx, ty, acc);
        if (t + gridDim.x < ntiles) __syncthreads();   // slots are reused by the next tile
    }
    if (CHECK) residual_reduce(a, acc);
}

// ---------------------------------------------------------------------------
// T pseudo-time steps per launch, one warp per strip of the
// lattice (FP32 or FP16-shifted storage).
//
// A warp owns a strip of 64 slot columns (lane l holds columns 2l and 2l + 1
// as FP32 pairs, pair_t) and a segment of `rows` output rows, and walks
// down the segment one row per iteration at all T step levels at once: in
// iteration i level j updates local row i - (j - 1), one row behind level
// j - 1.  What a level still needs of the level above it stays in registers:
//   populations with c_y = +1 (2, 5, 6) of the last two rows it produced,
//   those with c_y = 0 (1, 3) of the last one, those with c_y = -1 (4, 7, 8)
//   of the row it produced in this iteration,
// i.e. eight values per column and level boundary, and the horizontal movers
// pass between lanes by shuffles.  A warp shares nothing, so there is no
// barrier: its shared memory holds the rows on their way from global memory
// (asynchronous copies LA rows ahead, which need no registers) and the force of
// the last rows, which the levels read one after the other.  The halo is T - 1 columns per
// side and T - 1 rows per end.
//
// FP16-shifted storage decodes the stored deviations and carriers of the
// lane's own columns (one carrier per node instead of the eight a pulled node
// needs) one row ahead of level 1, which costs one more halo row and column.
//
// The per-node operations are lbm_core.cuh's, so FP32 results equal T
// single-step launches bit for bit.
//
// What bounds it: the five-step FP32 launch moves 72 bytes per node at 6.15 TB/s,
// 0.90 of the measured copy peak (16384^2, 3.14 ms; the block-wide wavefront
// kernel before it took 3.31 ms for four steps); six steps (3.67 ms, 0.611 per step)
// are bound by latency and the FMA pipe (issue 60 %, FMA pipe 58 %, DRAM 64 % of
// the time, three warps per scheduler).  An update issues 56 instructions (that
// kernel: 90), 27 of them packed arithmetic, two operations each; FP16S four-step
// launches, 69 instructions, run at 0.79 of the copy peak (0.63), bound alike.
// One code copy serves the first iterations too (each level's test is one
// uniform branch): with a copy of its own for them the code left the
// instruction cache and the compiler took 202 registers instead of 150.
constexpr int kGhost = 8;                        // ghost columns per row end (at least kStTMax + 1)
constexpr int kStSlots = 64;                     // slot columns of a strip (two per lane)
constexpr int kStTMax = 6;                       // most steps per launch (seven: 0.627 ms per step at 16384^2, six 0.611)

template <int S> __host__ __device__ constexpr int st_lag() { return S == S_F16S ? 1 : 0; }
// halo rows per end, and halo columns: at least as many per side, even on the
// left so that pairs start on even columns
template <int S, int T> __host__ __device__ constexpr int st_halo() { return T - 1 + st_lag<S>(); }
template <int S, int T> __host__ __device__ constexpr int st_left() { return (st_halo<S, T>() + 1) & ~1; }
template <int S, int T> __host__ __device__ constexpr int st_ox() {
    return (kStSlots - st_left<S, T>() - st_halo<S, T>()) & ~1;
}
// warps per block; the kernel is compiled for three resident blocks, twelve
// warps per SM (168 registers a thread; at 16384^2 with registers for eight warps
// 87.6 ms per 100 steps against 79.8).  With the check for two: at 168 registers
// it spilled, and every thread's partials were converted (T = 5 at 16384^2 6.20 ms,
// at 1024^2 39.8 us; with two blocks 5.72 and 35.6).  As ResPart combines them, and
// with k_residual_finish: 5.52 ms and 35.9 us (sums as pairs 5.46 and 35.5); FP16S
// 1000 x 700 28.8 us, 8192^2 1.40 ms
constexpr int kStNW = 4;
// rows copied ahead of the rows in use, and population rows held: FP32 has the
// rows above, at and below level 1 in use, FP16S the decoded row
template <int S> __host__ __device__ constexpr int st_la() { return S == S_F16S ? 3 : 1; }
constexpr int kWvD = 4;
// force rows held: those the levels still read and the rows ahead (a power of two)
template <int S, int T> __host__ __device__ constexpr int st_ring() {
    return T + 1 + st_la<S>() <= 4 ? 4 : (T + 1 + st_la<S>() <= 8 ? 8 : 16);
}
// One row in shared memory, in 16-byte chunks.  FP32: 72 columns (the strip's
// and one on either side, from a multiple of four on) of eight planes; FP16S:
// 72 columns (from a multiple of eight on) of eight planes and the carriers.
// The force: two planes of 72 columns, in a ring of its own.
constexpr int kStCols = 72;
template <int S> __host__ __device__ constexpr int st_row() { return S == S_F16S ? kStCols * (8 * 2 + 8) : kStCols * 8 * 4; }
constexpr int kStFRow = 2 * kStCols * 4;
// Rows of residual snapshot entries held (CHECK, 1024 bytes each): the row being
// checked and the st_la rows on their way, each in the group of copies that the
// wait of its own iteration is the first to cover (a power of two).
template <int S> __host__ __device__ constexpr int st_snaps() { return S == S_F16S ? 4 : 2; }
template <int S, int T, bool CHECK> __host__ __device__ constexpr int st_warp_smem() {
    return kWvD * st_row<S>() + st_ring<S, T>() * kStFRow + (CHECK ? 1024 * st_snaps<S>() : 0);
}
template <int S, int T, bool CHECK> __host__ __device__ constexpr int st_smem() {
    return kStNW * st_warp_smem<S, T, CHECK>();
}

template <int B>
__device__ __forceinline__ void copy_async(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(B) : "memory");
}
__device__ __forceinline__ pair_t lds_pair(uint32_t a) {
    pair_t d;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(d) : "r"(a) : "memory");
    return d;
}
__device__ __forceinline__ void lds_pairs(uint32_t a, pair_t& x, pair_t& y) {
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "r"(a) : "memory");
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
    uint32_t d;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(d) : "r"(a) : "memory");
    return d;
}
__device__ __forceinline__ void sts_pair(uint32_t a, pair_t p) {
    asm volatile("st.shared.b64 [%0], %1;" ::"r"(a), "l"(p) : "memory");
}
__device__ __forceinline__ float lds_float(uint32_t a) {
    float d;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(d) : "r"(a) : "memory");
    return d;
}
// A register pair the assembler cannot rebuild from a constant (it would, at
// each use, with two moves): a round trip through shared memory.
__device__ __forceinline__ pair_t opaque(pair_t p, uint32_t a) {
    asm volatile("st.shared.b64 [%0], %1;" ::"r"(a), "l"(p) : "memory");
    return lds_pair(a);
}

// FP16S: the deviations of the state after a collision, rounded to FP16 (h, and
// widened again in r), and the carriers that absorb the first moments of the
// rounding (store_f16s).
template <bool GEN>
__device__ __forceinline__ void round_state(const Post2& m, const PairCoef& c, __half2 h[8], pair_t r[8], pair_t& c10,
                                            pair_t& c01) {
    Post2 w = m;
    w.m10 = w.m01 = 0;
    w.m12 = fma2(splat(-c.qtheta), m.m10, m.m12);
    w.m21 = fma2(splat(-c.qtheta), m.m01, m.m21);
    pair_t fs[8];
    Pop2<!GEN>(w, c).all(c, fs);
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        float lo, hi;
        unpk(fs[p], lo, hi);
        h[p] = __floats2half2_rn(lo, hi);
        const float2 b = __half22float2(h[p]);
        r[p] = pk(b.x, b.y);
    }
    const pair_t r46 = sub2(r[4], r[6]), r57 = sub2(r[5], r[7]);
    c10 = sub2(m.m10, add2(sub2(r[0], r[2]), sub2(r46, r57)));
    c01 = sub2(m.m01, add2(sub2(r[1], r[3]), add2(r46, r57)));
}

// One strip and segment.  sm: the warp's shared memory (shared-space address).
// The lattice's rows carry ghost columns (row_ghost): the kGhost columns
// beyond either end hold the periodic images, so that a strip's rows are
// contiguous and its copies aligned wherever it lies; the strips that own the
// outermost kGhost columns store their images too.
// half (FP16S): the state is rounded after every second step, as by launches of two.
// OX: output columns of a strip (at most st_ox).  Waits for the previous launch
// (after_predecessor) just before the first copy: 1024^2 1.684 -> 1.669 ms per 400
// steps, FP16S 1000 x 700 1.664 -> 1.637.
template <int S, bool GEN, int T, bool CHECK, int OX = st_ox<S, T>()>
__device__ __forceinline__ void strip_walk(const StepParams& a, const PairCoef& ca, uint32_t sm, int strip, int y0,
                                           int rows, ResAcc2& acc, bool half = false) {
    static_assert(OX % 2 == 0 && OX <= st_ox<S, T>(), "pairs, within the slots");
    constexpr int LAG = st_lag<S>(), H = st_halo<S, T>(), HL = st_left<S, T>(),
                  LA = st_la<S>(), R = st_ring<S, T>(), ROW = st_row<S>(), SN = st_snaps<S>();
    static_assert(SN > LA && (!CHECK || LA <= 2 * H), "a snapshot entry has a slot until it is read, and is copied in time");
    constexpr int OFF = 1 - LAG;                             // copied row of local row i: i + OFF
    constexpr int AHEAD = 2 * OFF + LA;                      // rows copied ahead of iteration i
    constexpr int CA = S == S_F16S ? 8 : 4;                  // columns of a chunk of populations
    using P = typename StoreT<S>::P;
    const int nx = a.nx, ny = a.ny, pitch = a.pitch;
    const int lane = threadIdx.x & 31;
    PairCoef c = ca;
    c.half = opaque(ca.half, sm + 8 * lane);
    c.nhalf = opaque(ca.nhalf, sm + 8 * lane);
    c.nfour = opaque(ca.nfour, sm + 8 * lane);
    __syncwarp();
    const int xs0 = strip * OX - HL;                         // lattice column of slot 0
    // first column of a row in shared memory (rounded down, also below zero)
    const int xa0 = ((xs0 - OFF + (1 << 20)) & ~(CA - 1)) - (1 << 20);
    const int xs = xs0 + 2 * lane;                           // the lane's first column
    const bool ok = 2 * lane >= HL && 2 * lane < HL + OX && xs < nx;
    const bool two = ok && xs + 1 < nx;                      // (an odd lattice's last column stands alone)
    const int64_t n = a.plane;
    const int nit = rows + 2 * H;
    const uint32_t frc = sm + kWvD * ROW;                   // force ring
    const uint32_t snp = frc + R * kStFRow + lane * 32;      // snapshot entries of SN rows (CHECK)
    const uint32_t own = (uint32_t)(xs - xa0);               // the lane's first column within a row
    // Copies of a row: 16-byte chunks, chunk q = lane + 32 m (FP32: 18 per
    // plane, eight populations, then the force; FP16S: 9 per plane, eight
    // populations, then 36 of the carriers, then the force).
    constexpr int NP = S == S_F16S ? 108 : 144, NQ = NP + 36, NM = (NQ + 31) / 32;
    const char* base[NM];
    unsigned stride[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        const int q = min(lane + 32 * m, NQ - 1);
        if (q >= NP) {
            const int k = q - NP, p = k / 18;
            base[m] = reinterpret_cast<const char*>(static_cast<const float*>(p == 0 ? a.gx : a.gy) + xa0 + 4 * (k - 18 * p));
            stride[m] = 4 * pitch;
        } else if (S == S_F16S && q >= 72) {
            base[m] = reinterpret_cast<const char*>(reinterpret_cast<const float2*>(a.csrc) + xa0 + 2 * (q - 72));
            stride[m] = 8 * pitch;
        } else {
            constexpr int PC = kStCols / CA;                 // chunks of a plane
            const int p = q / PC;
            base[m] = reinterpret_cast<const char*>(static_cast<const P*>(a.src) + p * a.plane + xa0 + CA * (q - PC * p));
            stride[m] = (unsigned)sizeof(P) * pitch;
        }
    }
    int ly = (y0 - H - OFF) % ny;                            // lattice row of the next copy
    if (ly < 0) ly += ny;
    auto copy_row = [&](int i) {
        const uint32_t d = sm + (i & (kWvD - 1)) * ROW + lane * 16, g = frc + (i & (R - 1)) * kStFRow + lane * 16;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const uint32_t dp = d + m * 512, df = g + m * 512 - NP * 16;
            const uint32_t e = 32 * m + 31 < NP ? dp : (32 * m >= NP ? df : (lane + 32 * m < NP ? dp : df));
            if (32 * m + 31 < NQ || lane + 32 * m < NQ) copy_async<16>(e, base[m] + (uint64_t)ly * stride[m]);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ly = wrap_inc(ly, ny);
    };
    // level boundaries (FP16S: the first one below the decoded rows)
    constexpr int NB = T - 1 + LAG;
    pair_t up[NB > 0 ? NB : 1][2][3], mid[NB > 0 ? NB : 1][2];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
#pragma unroll
        for (int k = 0; k < 3; ++k) up[b][0][k] = up[b][1][k] = 0;
        mid[b][0] = mid[b][1] = 0;
    }
    int64_t so = (int64_t)y0 * pitch + xs;                   // the lane's first column of the next output row

    // The lane's stores besides its pair in place: the odd last column, and the
    // periodic images of columns near either end (off: from a column to its
    // image, 0 without one); one(dx, k) stores column k of the pair at the
    // pair's place + dx.
    auto image = [&](bool own, int x) { return !own ? 0 : (x < kGhost ? nx : (x >= nx - kGhost ? -nx : 0)); };
    if (CHECK) {
        acc.own0 = ok;
        acc.own1 = two;
    }
    const int off0 = image(ok, xs), off1 = image(two, xs + 1);
    const bool edge = __any_sync(0xffffffffu, off0 != 0 || off1 != 0 || ok != two);
    auto images = [&](auto&& one) {
        if (ok != two) one(0, 0);
        if (off0) one(off0, 0);
        if (off1) one(off1 + 1, 1);
    };

    // one iteration; K = i mod 2
    auto iter = [&](int i, auto k_c) {
        constexpr int K = decltype(k_c)::value;
        pair_t f[8];
        __syncwarp();                             // every lane is done with the rows this copy replaces
        if (CHECK && ok && i + LA >= 2 * H && i + LA < nit) {
            // snapshot entries of the output row of iteration i + LA, in this row's
            // group of copies, which is complete then (the entry after an odd
            // lattice's last column is in the plane, too): as loads into registers
            // the assembler moved them down to their use
            const float2* sp = static_cast<const float2*>(a.snap) + (so + (int64_t)min(LA, i + LA - 2 * H) * pitch);
            const uint32_t d = snp + ((i + LA) & (SN - 1)) * 1024;
            copy_async<16>(d, sp);
            copy_async<16>(d + 16, sp + n);
        }
        copy_row(i + AHEAD);                      // (rows past the last are copied too: any row is in range)
        asm volatile("cp.async.wait_group %0;" ::"n"(LA) : "memory");
        __syncwarp();                             // the rows of this iteration have arrived for every lane
        // Over boundary b: the pulled populations of the next level meet their
        // opposites, and only then the boundary's registers take the new row.
        // Populations 6 and 8 cross negated (Opp2).
        Opp2 o;
        auto cross = [&](int b, auto&& g) {
            const pair_t d4 = g(4), d7 = from_right(g(7)), d8 = from_left(g(8));
            if (CHECK && b == NB - 1) {
                f[0] = mid[b][0];
                f[1] = up[b][K][0];
                f[2] = mid[b][1];
                f[3] = d4;
                f[4] = up[b][K][1];
                f[5] = neg2(up[b][K][2]);
                f[6] = d7;
                f[7] = neg2(d8);
            }
            o = opposites2(mid[b][0], up[b][K][0], mid[b][1], d4, up[b][K][1], up[b][K][2], d7, d8);
            up[b][K][0] = g(2);
            up[b][K][1] = from_left(g(5));
            up[b][K][2] = from_right(g(6));
            mid[b][0] = from_left(g(1));
            mid[b][1] = from_right(g(3));
        };
        // Over boundary b: the state of rounded deviations (6 and 8 negated) and
        // carriers, decoded (pull_decode).
        auto cross_rounded = [&](int b, pair_t c10, pair_t c01, auto&& stored) {
            const float k1 = 0.5f * (1.0f - c.theta), k5 = 0.25f * c.theta;
            const pair_t sum = add2(c10, c01), dif = sub2(c10, c01);
            cross(b, [&](int p) {
                switch (p) {
                    case 1: return fma2(splat(k1), c10, stored(0));
                    case 2: return fma2(splat(k1), c01, stored(1));
                    case 3: return fma2(splat(-k1), c10, stored(2));
                    case 4: return fma2(splat(-k1), c01, stored(3));
                    case 5: return fma2(splat(k5), sum, stored(4));
                    case 6: return fma2(splat(k5), dif, stored(5));
                    case 7: return fma2(splat(-k5), sum, stored(6));
                    default: return fma2(splat(-k5), dif, stored(7));
                }
            });
        };
        if constexpr (S == S_F32) {
            // f_p(x) = f*_p(x - c_p), from rows i - 1, i and i + 1 (local rows
            // of the copies start one above the strip's, hence the + 1)
            constexpr int PL = kStCols * 4;
            const uint32_t o4 = own * 4, rm = sm + (i & (kWvD - 1)) * ROW + o4,
                           r0 = sm + ((i + 1) & (kWvD - 1)) * ROW + o4, rp = sm + ((i + 2) & (kWvD - 1)) * ROW + o4;
            auto left = [&](uint32_t r) { return pk(lds_float(r - 4), lds_float(r)); };
            auto right = [&](uint32_t r) { return pk(lds_float(r + 4), lds_float(r + 8)); };
            pair_t w[8];
            w[0] = left(r0);
            w[1] = lds_pair(rm + PL);
            w[2] = right(r0 + 2 * PL);
            w[3] = lds_pair(rp + 3 * PL);
            w[4] = left(rm + 4 * PL);
            w[5] = right(rm + 5 * PL);
            w[6] = right(rp + 6 * PL);
            w[7] = left(rp + 7 * PL);
            o = opposites2(w);
            if (CHECK && T == 1)
#pragma unroll
                for (int p = 0; p < 8; ++p) f[p] = w[p];
        } else {
            // the populations of the lane's columns in row i
            const uint32_t r = sm + (i & (kWvD - 1)) * ROW;
            pair_t e0, e1;                        // (m*_10, m*_01) of either column
            lds_pairs(r + kStCols * 16 + own * 8, e0, e1);
            cross_rounded(0, pk(pk_lo(e0), pk_lo(e1)), pk(pk_hi(e0), pk_hi(e1)), [&](int p) {
                uint32_t h = lds_u32(r + (p * kStCols + own) * 2);
                if (p == 5 || p == 7) h ^= 0x80008000u;
                const float2 v = __half22float2(*reinterpret_cast<__half2*>(&h));
                return pk(v.x, v.y);
            });
        }
#pragma unroll
        for (int j = 1; j <= T; ++j) {
            if (i < 2 * (j - 1 + LAG)) break;         // level j starts two rows after level j - 1
            const uint32_t fr = frc + ((i + OFF - LAG - (j - 1)) & (R - 1)) * kStFRow + own * 4;
            const pair_t gx = lds_pair(fr), gy = lds_pair(fr + kStCols * 4);
            const Post2 m = collide2<GEN>(moments2(o, c), gx, gy, c);
            if (S == S_F16S && j < T && j % 2 == 0 && half) {
                __half2 h[8];
                pair_t w[8], c10, c01;
                round_state<GEN>(m, c, h, w, c10, c01);
                cross_rounded(j - 1 + LAG, c10, c01, [&](int p) { return p == 5 || p == 7 ? neg2(w[p]) : w[p]; });
                continue;
            }
            if (j < T) {
                const Pop2<!GEN> w(m, c);
                cross(j - 1 + LAG, [&](int p) {
                    switch (p) {
                        case 1: return w.f1(c);
                        case 2: return w.f2(c);
                        case 3: return w.f3(c);
                        case 4: return w.f4(c);
                        case 5: return w.f5();
                        case 6: return w.nf6();
                        case 7: return w.f7();
                        default: return w.nf8();
                    }
                });
                continue;
            }
            // level T: the output row
            pair_t fs[8];
            if (CHECK) {
                ResSnap<S> sn0, sn1;
                pair_t e0, e1;
                lds_pairs(snp + (i & (SN - 1)) * 1024, e0, e1);
                unpk(e0, sn0.u.x, sn0.u.y);
                unpk(e1, sn1.u.x, sn1.u.y);
                lds_pairs(snp + (i & (SN - 1)) * 1024 + 16, e0, e1);
                unpk(e0, sn0.v.x, sn0.v.y);
                unpk(e1, sn1.v.x, sn1.v.y);
                check_pair<S>(acc, sn0, sn1, f, gx, gy, [&](float2 u0, float2 v0, float2 u1, float2 v1) {
                    float2* sp = static_cast<float2*>(a.snap) + so;
                    if (two) {
                        *reinterpret_cast<float4*>(sp) = make_float4(u0.x, u0.y, u1.x, u1.y);
                        *reinterpret_cast<float4*>(sp + n) = make_float4(v0.x, v0.y, v1.x, v1.y);
                    } else if (ok) {
                        sp[0] = u0;
                        sp[n] = v0;
                    }
                });
            }
            if constexpr (S == S_F32) {
                Pop2<!GEN>(m, c).all(c, fs);
                float* d = static_cast<float*>(a.dst) + so;
                if (two) {
#pragma unroll
                    for (int p = 0; p < 8; ++p) *reinterpret_cast<pair_t*>(d + p * a.plane) = fs[p];
                }
                if (edge) {
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        float lo, hi;
                        unpk(fs[p], lo, hi);
                        images([&](int dx, int k) { d[p * a.plane + dx] = k ? hi : lo; });
                    }
                }
            } else {
                __half* d = static_cast<__half*>(a.dst) + so;
                __half2 hs[8];
                pair_t c10, c01;
                round_state<GEN>(m, c, hs, fs, c10, c01);
                if (two) {
#pragma unroll
                    for (int p = 0; p < 8; ++p) *reinterpret_cast<__half2*>(d + p * a.plane) = hs[p];
                }
                float4 v;
                unpk(c10, v.x, v.z);
                unpk(c01, v.y, v.w);
                float2* cd = reinterpret_cast<float2*>(a.cdst) + so;
                if (two) *reinterpret_cast<float4*>(cd) = v;
                if (edge) {
#pragma unroll
                    for (int p = 0; p < 8; ++p)
                        images([&](int dx, int k) { d[p * a.plane + dx] = k ? __high2half(hs[p]) : __low2half(hs[p]); });
                    images([&](int dx, int k) { cd[dx] = k ? make_float2(v.z, v.w) : make_float2(v.x, v.y); });
                }
            }
            so += pitch;
        }
    };

    using K0 = std::integral_constant<int, 0>;
    using K1 = std::integral_constant<int, 1>;
    after_predecessor();
#pragma unroll
    for (int r = 0; r < AHEAD; ++r) copy_row(r);
    int i = 0;
    for (;;) {                                    // (one copy of each phase: the code fits the instruction cache)
        iter(i, K0{});
        if (++i >= nit) break;
        iter(i, K1{});
        if (++i >= nit) break;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");     // no copy outlives the strip
}

template <int S, bool GEN, int T, bool CHECK>
__global__ void __launch_bounds__(32 * kStNW, CHECK ? 2 : 3)
k_strip(const StepParams a, const PairCoef c, int seg, int nstrips, int items) {
    extern __shared__ float4 st_mem[];
    const int warp = threadIdx.x >> 5;
    const int item = (int)blockIdx.x * kStNW + warp;
    ResAcc2 acc;
    if (item < items) {
        const int strip = item % nstrips, y0 = (item / nstrips) * seg;
        const uint32_t sm = (uint32_t)__cvta_generic_to_shared(st_mem) + warp * st_warp_smem<S, T, CHECK>();
        strip_walk<S, GEN, T, CHECK>(a, c, sm, strip, y0, min(seg, a.ny - y0), acc);
    }
    if (CHECK) residual_reduce_pairs(a, acc);
}

// ---------------------------------------------------------------------------
// Several steps per launch of a small lattice (FP32 storage): a block holds
// one tile in registers.
//
// A launch of a small lattice is bound by latency, not by traffic or
// arithmetic: the strips of k_strip are too few to fill the GPU and each
// walks its rows one after the other.  Here a block of NW warps owns a tile of
// 64 slot columns by NW * RR slot rows, warp w rows w * RR .. w * RR + RR - 1
// with two columns per lane, and keeps every population in registers for all
// T steps of the launch (T is a run-time count).  A slot's state is held as
// the pulls of its neighbours will want it: after the collision the horizontal
// movers are shifted by shuffle, so that a row's next populations are its own
// (1, 3), those with c_y = +1 (2, 5, 6) of the row below it in memory order and
// those with c_y = -1 (4, 7, 8) of the row after it -- registers of the same
// lane, except at the edge of a warp's rows, where six values per column pass
// through shared memory (double-buffered: one block barrier per step).
// Tiles overlap by T - 1 slots per side.
//
// Any lattice size works: slots wrap periodically, and a lattice smaller than
// a tile appears in it more than once.
//
// Measured (GB300, launches back to back, against what ran before at these
// sizes): 100 x 75 0.59 us per step (three-step tiles 2.07), 333 x 517 1.13
// (wavefront 4.0).  A launch of T steps takes 2.8 us (start, loads, stores) and
// 0.24 us per step (8 warps of two rows) to 0.67 us (12 warps of four): FMA-pipe
// and latency bound, 2 to 3 warps per scheduler.
template <int S, int RR, bool GEN, bool CHECK>
__global__ void __launch_bounds__(512, 1)
k_tile(const StepParams a, const PairCoef ca, int T, int ntx, unsigned rounds) {
    extern __shared__ float4 tile_mem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nx = a.nx, ny = a.ny, H = T - 1;
    const int ox = kStSlots - 2 * H, oy = nw * RR - 2 * H;
    const int tx = blockIdx.x % ntx, ty = blockIdx.x / ntx;
    // the lane's pair in the rows the warps exchange: [parity][warp + 1][up, down][3]
    const uint32_t sm = (uint32_t)__cvta_generic_to_shared(tile_mem) + lane * 8;
    const uint32_t par_bytes = (uint32_t)(nw + 2) * 6 * 256;
    PairCoef c = ca;
    c.half = opaque(ca.half, sm + warp * 256);
    c.nhalf = opaque(ca.nhalf, sm + warp * 256);
    c.nfour = opaque(ca.nfour, sm + warp * 256);
    __syncthreads();
    after_predecessor();
    const int xs = tx * ox - H + 2 * lane, ys = ty * oy - H + warp * RR;   // the first slot's node
    auto wrapped = [](int v, int n) {
        v %= n;
        return v < 0 ? v + n : v;
    };
    const int xa = wrapped(xs - 1, nx), xb = wrapped(xs, nx), xc = wrapped(xs + 1, nx), xd = wrapped(xs + 2, nx);
    using P = typename StoreT<S>::P;
    const P* src = static_cast<const P*>(a.src);
    const int64_t pl = a.plane;
    const float k1 = 0.5f * (1.0f - c.theta), k5 = 0.25f * c.theta;   // (FP16S: pull_decode)
    struct Row {
        pair_t m1, m3, u2, u5, nu6, d4, d7, nd8;
    } s[RR];
    pair_t gx[RR], gy[RR];
    auto ld2 = [&](const float* p, int x0, int x1) { return pk(ldg(p + x0), ldg(p + x1)); };
    // The populations pulled from memory row y; parts: 1 those with c_y = +1, 2
    // those with c_y = 0, 4 those with c_y = -1 (6 and 8 negated).
    auto pull = [&](int64_t y, int parts, Row& q) {
        const int64_t row = y * a.pitch;
        const P* p = src + row;
        if constexpr (S == S_F32) {
            if (parts & 2) {
                q.m1 = ld2(p, xa, xb);
                q.m3 = ld2(p + 2 * pl, xc, xd);
            }
            if (parts & 1) {
                q.u2 = ld2(p + pl, xb, xc);
                q.u5 = ld2(p + 4 * pl, xa, xb);
                q.nu6 = ld2(p + 5 * pl, xc, xd);
            }
            if (parts & 4) {
                q.d4 = ld2(p + 3 * pl, xb, xc);
                q.d7 = ld2(p + 6 * pl, xc, xd);
                q.nd8 = ld2(p + 7 * pl, xa, xb);
            }
        } else {
            auto h2 = [&](int k, int x0, int x1) {
                return pk(__half2float(ldg(p + k * pl + x0)), __half2float(ldg(p + k * pl + x1)));
            };
            const float2* cr = reinterpret_cast<const float2*>(a.csrc) + row;
            const float2 ca_ = ldg(cr + xa), cb = ldg(cr + xb), cc = ldg(cr + xc), cd = ldg(cr + xd);
            const pair_t l0 = pk(ca_.x, cb.x), l1 = pk(ca_.y, cb.y), r0 = pk(cc.x, cd.x), r1 = pk(cc.y, cd.y);
            const pair_t m1 = pk(cb.y, cc.y);
            if (parts & 2) {
                q.m1 = fma2(splat(k1), l0, h2(0, xa, xb));
                q.m3 = fma2(splat(-k1), r0, h2(2, xc, xd));
            }
            if (parts & 1) {
                q.u2 = fma2(splat(k1), m1, h2(1, xb, xc));
                q.u5 = fma2(splat(k5), add2(l0, l1), h2(4, xa, xb));
                q.nu6 = fma2(splat(-k5), sub2(r0, r1), h2(5, xc, xd));
            }
            if (parts & 4) {
                q.d4 = fma2(splat(-k1), m1, h2(3, xb, xc));
                q.d7 = fma2(splat(-k5), add2(r0, r1), h2(6, xc, xd));
                q.nd8 = fma2(splat(k5), sub2(l0, l1), h2(7, xa, xb));
            }
        }
    };
#pragma unroll
    for (int r = 0; r < RR; ++r) {
        const int y = wrapped(ys + r, ny);
        pull(y, 7, s[r]);
        gx[r] = ld2(static_cast<const float*>(a.gx) + (int64_t)y * a.pitch, xb, xc);
        gy[r] = ld2(static_cast<const float*>(a.gy) + (int64_t)y * a.pitch, xb, xc);
    }
#pragma unroll
    for (int r = 0; r < RR; ++r) {
        s[r].nu6 = neg2(s[r].nu6);
        s[r].nd8 = neg2(s[r].nd8);
    }
    auto put = [&](uint32_t e, pair_t x, pair_t y, pair_t z) {
        sts_pair(e, x);
        sts_pair(e + 256, y);
        sts_pair(e + 512, z);
    };
    auto slot = [&](int w) { return sm + (uint32_t)(w + 1) * (6 * 256); };
    put(slot(warp), s[RR - 1].u2, s[RR - 1].u5, s[RR - 1].nu6);
    put(slot(warp) + 768, s[0].d4, s[0].d7, s[0].nd8);
    if (warp == 0) {               // the row before the tile, whose upward movers step 1 pulls
        Row q;
        pull(wrapped(ys - 1, ny), 1, q);
        put(slot(-1), q.u2, q.u5, neg2(q.nu6));
    }
    if (warp == nw - 1) {          // the row after it
        Row q;
        pull(wrapped(ys + RR, ny), 4, q);
        put(slot(nw) + 768, q.d4, q.d7, neg2(q.nd8));
    }
    __syncthreads();
    const int s0 = 2 * lane;
    const bool ok0 = s0 >= H && s0 < kStSlots - H && xs < nx, ok1 = s0 + 1 >= H && s0 + 1 < kStSlots - H && xs + 1 < nx;
    ResAcc2 acc;
    acc.own0 = ok0;
    acc.own1 = ok1;
    // the check's snapshot entries of the coming row, loaded one row ahead
    ResSnap<S> sn[2];
    auto owned_row = [&](int r) {
        const int q = warp * RR + r;
        return q >= H && q < nw * RR - H && ys + r < ny;
    };
    auto snap_row = [&](int r) {
        if (!owned_row(r)) return;
        const int64_t idx = (int64_t)(ys + r) * a.pitch + xs;
        if (ok0) sn[0] = snap_load<S>(a, pl, idx);
        if (ok1) sn[1] = snap_load<S>(a, pl, idx + 1);
    };
    for (int t = 0; t < T; ++t) {
        const bool last = t == T - 1;
        if (CHECK && last) snap_row(0);
        const uint32_t par = (t & 1) ? par_bytes : 0;
        const uint32_t above = slot(warp - 1) + par, below = slot(warp + 1) + par + 768;
        pair_t u2 = lds_pair(above), u5 = lds_pair(above + 256), nu6 = lds_pair(above + 512);
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            pair_t d4, d7, nd8;
            if (r + 1 < RR) {
                d4 = s[r + 1 < RR ? r + 1 : r].d4;
                d7 = s[r + 1 < RR ? r + 1 : r].d7;
                nd8 = s[r + 1 < RR ? r + 1 : r].nd8;
            } else {
                d4 = lds_pair(below);
                d7 = lds_pair(below + 256);
                nd8 = lds_pair(below + 512);
            }
            const Opp2 o = opposites2(s[r].m1, u2, s[r].m3, d4, u5, nu6, d7, nd8);
            const Post2 m = collide2<GEN>(moments2(o, c), gx[r], gy[r], c);
            // the populations after the collision, or (FP16S, where the state is
            // rounded: after the steps of `rounds`, and the last) the rounded
            // deviations and the carriers
            pair_t w[8], c10 = 0, c01 = 0;
            const bool round = S == S_F16S && (last || (rounds >> t & 1));
            if (!round) {
                const Pop2<!GEN> q(m, c);
                w[0] = q.f1(c);
                w[1] = q.f2(c);
                w[2] = q.f3(c);
                w[3] = q.f4(c);
                w[4] = q.f5();
                w[5] = q.nf6();
                w[6] = q.f7();
                w[7] = q.nf8();
            } else {
                __half2 h[8];
                round_state<GEN>(m, c, h, w, c10, c01);
                if (!last) {
                    const pair_t sum = add2(c10, c01), dif = sub2(c10, c01);
                    w[0] = fma2(splat(k1), c10, w[0]);
                    w[1] = fma2(splat(k1), c01, w[1]);
                    w[2] = fma2(splat(-k1), c10, w[2]);
                    w[3] = fma2(splat(-k1), c01, w[3]);
                    w[4] = fma2(splat(k5), sum, w[4]);
                    w[5] = fma2(splat(k5), dif, neg2(w[5]));
                    w[6] = fma2(splat(-k5), sum, w[6]);
                    w[7] = fma2(splat(-k5), dif, neg2(w[7]));
                }
            }
            if (last) {
                ResSnap<S> now[2];
                if (CHECK) {
                    now[0] = sn[0];
                    now[1] = sn[1];
                    if (r + 1 < RR) snap_row(r + 1);
                }
                if (owned_row(r)) {
                    const int y = ys + r;
                    const int64_t idx = (int64_t)y * a.pitch + xs;
                    P* d = static_cast<P*>(a.dst) + idx;
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        float lo, hi;
                        unpk(S == S_F32 && (p == 5 || p == 7) ? neg2(w[p]) : w[p], lo, hi);
                        if (ok0) d[p * pl] = P(lo);            // (FP16S: exact)
                        if (ok1) d[p * pl + 1] = P(hi);
                    }
                    if constexpr (S == S_F16S) {
                        float4 v;
                        unpk(c10, v.x, v.z);
                        unpk(c01, v.y, v.w);
                        float2* cd = reinterpret_cast<float2*>(a.cdst) + idx;
                        if (ok0) cd[0] = make_float2(v.x, v.y);
                        if (ok1) cd[1] = make_float2(v.z, v.w);
                    }
                    if (CHECK) {
                        const pair_t f[8] = {s[r].m1, u2, s[r].m3, d4, u5, neg2(nu6), d7, neg2(nd8)};
                        check_pair<S>(acc, now[0], now[1], f, gx[r], gy[r],
                                          [&](float2 u0, float2 v0, float2 u1, float2 v1) {
                                              float2* sp = static_cast<float2*>(a.snap) + idx;
                                              if (ok0) {
                                                  sp[0] = u0;
                                                  sp[pl] = v0;
                                              }
                                              if (ok1) {
                                                  sp[1] = u1;
                                                  sp[pl + 1] = v1;
                                              }
                                          });
                    }
                }
            }
            u2 = s[r].u2;
            u5 = s[r].u5;
            nu6 = s[r].nu6;
            s[r].u2 = w[1];
            s[r].d4 = w[3];
            s[r].m1 = from_left(w[0]);
            s[r].m3 = from_right(w[2]);
            s[r].u5 = from_left(w[4]);
            s[r].nu6 = from_right(w[5]);
            s[r].d7 = from_right(w[6]);
            s[r].nd8 = from_left(w[7]);
        }
        if (last) break;
        const uint32_t next = slot(warp) + (par_bytes - par);
        put(next, s[RR - 1].u2, s[RR - 1].u5, s[RR - 1].nu6);
        put(next + 768, s[0].d4, s[0].d7, s[0].nd8);
        __syncthreads();
    }
    if (CHECK) residual_reduce_pairs(a, acc);
}

// Destinations of the five solution fields u_x, u_y, sigma_xx, sigma_yy,
// sigma_xy (nx*ny doubles each; a null entry is not written).  Device memory,
// or pinned host memory the device can address (the recovery then writes the
// caller's arrays over the host link directly).
// tr: the lattice is the transpose of the caller's (x and y exchanged), so
// node (x, y) goes to entry x * ny + y of each destination.
struct FieldOut {
    double* p[5];
    int tr;
};

inline FieldOut field_planes(double* out, int64_t n) {
    FieldOut o;
    for (int k = 0; k < 5; ++k) o.p[k] = out + k * n;
    o.tr = 0;
    return o;
}

// log2 of a power of two.
__device__ __forceinline__ int ilogb2(float p) { return (int)(__float_as_uint(p) >> 23) - 127; }

// Solution fields of the current state (Table 2, Eq. compute_bared), FP64.
template <int S>
__global__ void __launch_bounds__(kThreads)
k_fields(const StepParams a, const Coef<double> c, typename StoreT<S>::T theta, const FieldOut out) {
    using T = typename StoreT<S>::T;
    using G = typename StoreT<S>::G;
    after_predecessor();
    const int nx = a.nx, ny = a.ny;
    const int y = blockIdx.y * BY + threadIdx.y;
    const int x = blockIdx.x * 32 + threadIdx.x;
    if (y >= ny || x >= nx) return;
    const int ym = wrap_dec(y, ny), yp = wrap_inc(y, ny);
    const int64_t r0 = (int64_t)y * a.pitch, rm = (int64_t)ym * a.pitch, rp = (int64_t)yp * a.pitch;
    T f[8];
    gather<S>(a, r0, rm, rp, x, wrap_dec(x, nx), wrap_inc(x, nx), f, theta);
    const int64_t idx = r0 + x;
    const G gxs = static_cast<const G*>(a.gx)[idx], gys = static_cast<const G*>(a.gy)[idx];
    // In integers, as the FP64 collision (step_f64): FP64 arithmetic, 64 cycles of a
    // scheduler per warp instruction, would bound the recovery.  The unit is 2^-58
    // of the power of two above the node's largest value, so every sum of FP32
    // values is exact to a unit (pairs of FP32 sums were to 2^-44); sxx, syy, sxy
    // are Eq. compute_bared with Table 2's factors.  Three of the five results leave
    // through the FP64 pipe (16384^2 FP32: none 4.63 ms, two 4.48, three 4.26, four
    // 4.64; five with nine FP64 instructions per node 5.57, all in FP64 10.3).
    uint32_t e = 0;
    auto top = [&](auto v) {
        if constexpr (S == S_F64) e = max(e, (uint32_t)__double2hiint(v) & 0x7ff00000u);
        else e = max(e, __float_as_uint(v) & 0x7f800000u);
    };
#pragma unroll
    for (int p = 0; p < 8; ++p) top(f[p]);
    top(gxs);
    top(gys);
    double u, v, sxx, syy, mb11;
    const bool fixed = c.fields_fixed && (S == S_F64 ? e - (100u << 20) <= (1900u << 20) : e - (64u << 23) < (191u << 23));
    if (fixed) {
        auto fix = [&](auto w, int h) {
            if constexpr (S == S_F64) return to_fixed<true>(w, e, h);
            else return to_fixed(w, e, h);
        };
        int64_t F[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) F[p] = fix(f[p], 0);
        const int64_t hx = fix(gxs, 1), hy = fix(gys, 1);
        const int64_t p = F[4] + F[6], q = F[5] + F[7], r = F[4] - F[6], s = F[5] - F[7];
        const int64_t U = (F[0] - F[2]) + (r - s) + hx, V = (F[1] - F[3]) + (r + s) + hy;
        const int64_t s13 = F[0] + F[2], s24 = F[1] + F[3];
        const int64_t X = mul_fixed(c.h11, p - q), P = mul_fixed(c.hs, s13 + s24 + 2 * (p + q)), D = mul_fixed(c.hd, s13 - s24);
        // exponent field of the same power of two in FP64 (FP16S: out of the state's scaled units)
        const uint32_t e64 = S == S_F64 ? e : (e >> 3) + ((uint32_t)(896 - (S == S_F16S ? ilogb2(a.hscale) : 0)) << 20);
        u = from_fixed_fp64(U, e64);
        v = from_fixed_fp64(V, e64);
        sxx = from_fixed_fp64(P + D, e64);
        syy = from_fixed<true>(P - D, e64);
        mb11 = from_fixed<true>(-2 * X, e64);
    } else {
        uint32_t any = nonzero(gxs) | nonzero(gys);
#pragma unroll
        for (int p = 0; p < 8; ++p) any |= nonzero(f[p]);
        u = v = sxx = syy = mb11 = 0.0;                  // a node of zeros (as in step_f64)
        if (any) {
            double w[8];
            const double scale = S == S_F16S ? (double)a.hinv : 1.0;
#pragma unroll
            for (int p = 0; p < 8; ++p) w[p] = (double)f[p] * scale;
            const Mom<double> m = moments(w);
            u = m.m10 + 0.5 * ((double)gxs * scale);
            v = m.m01 + 0.5 * ((double)gys * scale);
            sxx = -0.5 * (c.bs * m.ms + c.bd * m.md);
            syy = -0.5 * (c.bs * m.ms - c.bd * m.md);
            mb11 = c.b11 * m.m11;
        }
    }
    const double un = 1.0;         // (the fields' own unit)
    const int64_t o = out.tr ? (int64_t)x * ny + y : (int64_t)y * nx + x;
    if (out.p[0]) out.p[0][o] = u;
    if (out.p[1]) out.p[1][o] = v;
    if (out.p[2]) out.p[2][o] = sxx;
    if (out.p[3]) out.p[3][o] = syy;
    if (out.p[4]) out.p[4][o] = -mb11 * un;
}

// Pre-collision populations of the current state into 8 FP64 planes.
template <int S>
__global__ void __launch_bounds__(kThreads)
k_export(const StepParams a, typename StoreT<S>::T theta, double* out) {
    using T = typename StoreT<S>::T;
    const int nx = a.nx, ny = a.ny;
    const int y = blockIdx.y * BY + threadIdx.y;
    const int x = blockIdx.x * 32 + threadIdx.x;
    if (y >= ny || x >= nx) return;
    const int ym = wrap_dec(y, ny), yp = wrap_inc(y, ny);
    const int64_t r0 = (int64_t)y * a.pitch, rm = (int64_t)ym * a.pitch, rp = (int64_t)yp * a.pitch;
    T f[8];
    gather<S>(a, r0, rm, rp, x, wrap_dec(x, nx), wrap_inc(x, nx), f, theta);
    const int64_t idx = (int64_t)y * nx + x, n = (int64_t)nx * ny;
    // (FP16S: back from the state's scaled units; a power of two, exact)
    const double unscale = S == S_F16S ? (double)a.hinv : 1.0;
#pragma unroll
    for (int p = 0; p < 8; ++p) out[p * n + idx] = double(f[p]) * unscale;
}

// Load pre-collision populations f (8 FP64 planes): the stored post-collision
// value at x is f*_p(x) = f_p(x + c_p) (inverse of the pull gather).
template <int S>
__global__ void __launch_bounds__(kThreads)
k_import(const StepParams a, typename StoreT<S>::T theta, const double* in) {
    using T = typename StoreT<S>::T;
    using P = typename StoreT<S>::P;
    const int nx = a.nx, ny = a.ny;
    const int y = blockIdx.y * BY + threadIdx.y;
    const int x = blockIdx.x * 32 + threadIdx.x;
    if (y >= ny || x >= nx) return;
    const int xm = wrap_dec(x, nx), xp = wrap_inc(x, nx);
    const int ym = wrap_dec(y, ny), yp = wrap_inc(y, ny);
    const int64_t n = (int64_t)nx * ny;
    const int64_t r0 = (int64_t)y * nx, rm = (int64_t)ym * nx, rp = (int64_t)yp * nx;
    // f*_p(x) = f_p(x + c_p); FP16S: in the state's scaled units (the power
    // of two commutes with the rounding to FP32)
    const T sc = S == S_F16S ? T(a.hscale) : T(1);
    T fs[8];
    fs[0] = T(in[0 * n + r0 + xp]) * sc;
    fs[1] = T(in[1 * n + rp + x]) * sc;
    fs[2] = T(in[2 * n + r0 + xm]) * sc;
    fs[3] = T(in[3 * n + rm + x]) * sc;
    fs[4] = T(in[4 * n + rp + xp]) * sc;
    fs[5] = T(in[5 * n + rp + xm]) * sc;
    fs[6] = T(in[6 * n + rm + xm]) * sc;
    fs[7] = T(in[7 * n + rm + xp]) * sc;
    const int64_t idx = (int64_t)y * a.pitch + x;
    P* d = static_cast<P*>(a.dst);
    if constexpr (S == S_F16S) {
        const Mom<T> s = moments(fs);
        T nf[8];
        populations(deviation_moments(quarter(s), T(0.25) * theta), nf);
        (void)d;
        store_f16s(a, idx, nf, s.m10, s.m01);
    } else {
        (void)theta;
        for (int p = 0; p < 8; ++p) d[p * a.plane + idx] = P(fs[p]);
    }
}

// Force upload in one pass over the FP64 input (device memory, or pinned host
// memory the device can address): the force in the storage force type G, its
// max |g| over both components (non-negative doubles order like their bit
// patterns, so an unsigned 64-bit atomicMax suffices) and `bad` set by a
// non-finite entry.
template <typename G>
__global__ void k_force_ingest(const double* gx, const double* gy, G* ox, G* oy, int64_t n, int nx, int pitch,
                               unsigned long long* absmax, unsigned int* bad) {
    double m = 0.0;
    unsigned int b = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double u = gx[i], v = gy[i];
        const int64_t y = i / nx, o = i + y * (pitch - nx);   // rows of nx values, pitch apart
        ox[o] = G(u);
        oy[o] = G(v);
        if (pitch > nx) {                                      // periodic images (row_ghost)
            const int x = (int)(i - y * nx);
            if (x < kGhost) {
                ox[o + nx] = G(u);
                oy[o + nx] = G(v);
            }
            if (x >= nx - kGhost) {
                ox[o - nx] = G(u);
                oy[o - nx] = G(v);
            }
        }
        if (!(isfinite(u) && isfinite(v))) b = 1;
        m = fmax(m, fmax(fabs(u), fabs(v)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        b |= __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(absmax, (unsigned long long)__double_as_longlong(m));
        if (b) atomicOr(bad, 1u);
    }
}

// The ghost columns of the state in a.dst (row_ghost), after a kernel that
// writes only the lattice's own columns: thread `i` of `step` takes rows, ghost
// columns and planes (and, FP16S, carriers) in turn.
template <int S>
__device__ __forceinline__ void fill_ghosts(const StepParams& a, int64_t i, int64_t step) {
    using P = typename StoreT<S>::P;
    const int64_t per = (int64_t)a.ny * 2 * kGhost, total = per * (S == S_F16S ? 9 : 8);
    for (; i < total; i += step) {
        const int p = (int)(i / per), g = (int)(i % (2 * kGhost));
        const int64_t row = (i % per) / (2 * kGhost) * a.pitch;
        const int64_t to = row + (g < kGhost ? g - kGhost : a.nx + g - kGhost), from = to + (g < kGhost ? a.nx : -a.nx);
        if (S == S_F16S && p == 8) {
            float2* c = reinterpret_cast<float2*>(a.cdst);
            c[to] = c[from];
        } else {
            P* d = static_cast<P*>(a.dst) + p * a.plane;
            d[to] = d[from];
        }
    }
}

template <int S>
__global__ void k_fill_ghosts(const StepParams a) {
    after_predecessor();
    fill_ghosts<S>(a, blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
}

// F16S: multiply every stored deviation by `factor` (a power of two).
__global__ void k_rescale_half(__half* h, int64_t count, float factor);
// Multiply `count` floats by `factor` (a power of two: exact unless the result
// leaves FP32's normal range).
__global__ void k_scale_float(float* v, int64_t count, float factor);

// Grid-level pass of the residual when the check launch wrote per-block
// partials only (StepParams::counter == nullptr): one block combines the
// nblocks partial sets (FP64) into result.
__global__ void k_residual_finish(const double* partials, int64_t nblocks, double* result);
constexpr int kFinishThreads = 1024;

// Higher-order force correction with periodic central differences (FP64).
__global__ void k_force_correct(const double* gx, const double* gy, double* ox, double* oy, int nx,
                                int ny, double d1, double d2, double d3);

// Launchers (defined per storage type).
template <int S>
struct Ops {
    using T = typename StoreT<S>::T;
    // check_blocks: grid cap of the CHECK launch (<= partials slots); one
    // block per tile below it
    static cudaError_t step(const StepParams& a, const Coef<T>& c, int V, bool gen, bool check,
                            int check_blocks, cudaStream_t st);
    static cudaError_t fields(const StepParams& a, const Coef<double>& c, T theta, const FieldOut& out,
                              cudaStream_t st);
    static cudaError_t export_pop(const StepParams& a, T theta, double* out, cudaStream_t st);
    static cudaError_t import_pop(const StepParams& a, T theta, const double* in, cudaStream_t st);
};

// FP16-shifted storage scale: stored deviation = deviation * 2^e.  At steady
// state the deviations are second moments ~ tau * grad u ~ |g| * L / (2 pi);
// e maps max|g| * max(nx, ny) to 2^8, leaving 2^7 of headroom below FP16's
// maximum and keeping values far above its smallest normal.
inline int f16s_exponent(double gmax, int nx, int ny) {
    if (!(gmax > 0.0)) return 0;
    const double L = double(nx > ny ? nx : ny);
    int e = 8 - (int)ceil(log2(gmax * L));
    return e < -60 ? -60 : (e > 60 ? 60 : e);
}

// Residual windows per check interval k: rounding keeps a converged stored
// state jittering by about J |u|, which floors a w-step residual near J / w.
// Measured (max|u^t - u^(t-w)| / max|u| long after convergence): FP64 ~3e-15;
// FP32 1.3e-7 .. 4.3e-7 on every shape and nu tried; FP16-shifted storage
// 2.5e-7 .. 1e-5, larger for a shorter lattice side (its stored deviations are
// of size ~ |grad u| ~ u / min(nx, ny)) and for larger nu.  A solve asking for
// tol starts with windows of min(64, max(1, ceil(2 J / (tol k)))) intervals of
// k steps, J = 4e-7 (FP32) or 6e-4 / min(nx, ny) (FP16S), and adapt_period
// stretches them while the residual stagnates, so a floor above the estimate
// cannot stall the solve.  The cap keeps divergence detection (made at
// checks) within 64 intervals; a tol that would need more is below what the
// storage type can resolve.
inline int check_period(int dtype, double tol, int k, int nmin) {
    const double J = dtype == S_F16S ? 6e-4 / (double)(nmin > 1 ? nmin : 1)
                                     : (dtype == S_F32 ? 4e-7 : 3e-15);
    if (!(tol > 0.0) || k < 1) return 64;
    const double p = ceil(2.0 * J / (tol * (double)k));
    return p < 1.0 ? 1 : (p > 64.0 ? 64 : (int)p);
}

// The next window length (in intervals of k steps) after a check above tol:
// doubled (up to 64) when the residual r did not fall below 0.95 of the
// previous check's r_prev.  Decay faster than 5 % per window keeps the window;
// a residual held up by the rounding floor J / w, or decaying very slowly, gets
// longer windows (which lower the floor and cost fewer checks; the stopping
// step moves by at most one window).
inline int adapt_period(int period, double r, double r_prev) {
    return (r > 0.95 * r_prev && period < 64) ? (period * 2 > 64 ? 64 : period * 2) : period;
}

// Rows of a lattice the library lays out itself.  FP32 and FP16S rows from 64
// columns on (what the strip kernel runs on) hold kGhost ghost columns at
// either end, the periodic images of the columns at the other one, and start
// on 16-byte boundaries; column 0 is kGhost elements into the row.
constexpr int kRowSlack = 128;    // elements a buffer holds beyond its planes: a strip reads past a row's end
inline int row_ghost(int dtype, int nx) { return dtype != S_F64 && nx >= 64 && nx < (1 << 30) ? kGhost : 0; }
inline int row_pitch(int dtype, int nx) { return row_ghost(dtype, nx) ? (nx + 2 * kGhost + 7) / 8 * 8 : nx; }

inline int64_t step_tiles(int nx, int ny, int V) {
    return (int64_t)((nx + 32 * V - 1) / (32 * V)) * ((ny + BY - 1) / BY);
}

// Grid cap of the residual-check launches: one FP64 partial set per block.
constexpr int64_t kMaxCheckBlocks = int64_t(1) << 19;

// Two-step launches of a single lattice: from one full slot array up (smaller
// lattices would mostly compute duplicate slots).
inline bool step2_fits(int nx, int ny) { return nx >= kT2W && ny >= kT2H; }

inline int64_t step2_tiles(int nx, int ny) {
    return (int64_t)((nx + kT2OX - 1) / kT2OX) * ((ny + kT2OY - 1) / kT2OY);
}

// Three-step launches of a single lattice: from one full slot array up.
inline bool step3_fits(int nx, int ny) { return nx >= kT3W && ny >= kT3H; }

inline int64_t step3_tiles(int nx, int ny) {
    return (int64_t)((nx + kT3OX - 1) / kT3OX) * ((ny + kT3OY - 1) / kT3OY);
}

// The wavefront schedule's lattices (the documented limit of
// lbm_set_wavefront; FP16S: four steps per launch from here on).
#define LBM_WV_NW 8   // in warps of 32 columns
inline bool wave_fits(int nx, int ny) { return nx >= 32 * LBM_WV_NW && ny >= 8; }

// Strips of a strip launch of T steps.
inline int64_t strip_count(int dtype, int T, int nx) {
    const int halo = T - 1 + (dtype == S_F16S ? 1 : 0), left = (halo + 1) & ~1, ox = (kStSlots - left - halo) & ~1;
    return (nx + ox - 1) / ox;
}

struct StripShape {
    int T = 0, seg = 0;
    double cost = 0.0;            // modelled cycles of one launch
};

// Rows per segment of a launch of T steps that takes the fewest cycles on
// `nsm` multiprocessors of `warps` resident warps each, and its cost.  Fitted on
// GB300 (300 x 2000 to 16384^2, T = 2 .. 6; within 10 %): a warp's iteration costs
// 70 + 115 w cycles per level with w warps on its scheduler, and a segment of seg
// rows takes seg + 2 (halo rows) iterations, so the best segments are those whose
// warps just fill a whole number of waves (4096 x 3000, T = 5: 213 to 229 us with
// 32 to 256 rows chosen by halving, 155 us with the 125 rows that fill one
// wave); a checked row costs 1250 cycles (FP16S 1600) more; the state moves at 3.0 kB per
// cycle (6.2 TB/s).  rows > 0 fixes the segment.
inline StripShape strip_shape(int dtype, int T, bool check, int nx, int ny, int nsm, int warps, int rows) {
    const int64_t ns = strip_count(dtype, T, nx);
    const int halo = T - 1 + (dtype == S_F16S ? 1 : 0);
    // (short launches wait longer for their rows)
    const double slow = T == 2 ? 1.6 : (T == 3 ? 1.3 : (T == 4 ? 1.08 : 1.0));
    const double mem = (double)nx * ny * ((dtype == S_F16S ? 56 : 72) + (check ? 32 : 0)) / 3040.0;
    StripShape best;
    auto consider = [&](int64_t seg) {
        if (seg < 1) seg = 1;
        if (seg > ny) seg = ny;
        const int64_t items = ns * ((ny + seg - 1) / seg), slots = (int64_t)nsm * warps;
        auto wave = [&](double w) {
            return slow * (double)(seg + 2 * halo) * (T * (70.0 + 115.0 * w) + 150.0) + (check ? (dtype == S_F32 ? 1250.0 : 1600.0) * seg : 0.0);
        };
        // full waves (many run into one another), then what is left
        const int64_t full = (items - 1) / slots, rest = items - full * slots;
        const double part = full < 8 ? wave((double)((rest + 4 * nsm - 1) / (4 * nsm)))
                                     : wave(warps / 4.0) * (double)rest / (double)slots;
        const double busy = full * wave(warps / 4.0) + part;
        const double cost = 3000.0 + pow(pow(busy, 6.0) + pow(mem, 6.0), 1.0 / 6.0);
        if (best.seg == 0 || cost < best.cost) {
            best.T = T;
            best.seg = (int)seg;
            best.cost = cost;
        }
    };
    if (rows > 0) {
        consider(rows);
        return best;
    }
    for (int w = 1; w <= 24 * warps / 4; ++w) {     // w warps per scheduler in all
        const int64_t nseg = (int64_t)4 * nsm * w / ns;
        if (nseg < 1) continue;
        const int64_t seg = (ny + nseg - 1) / nseg;
        if (seg < 4 && best.seg) break;
        consider(seg < 4 ? 4 : seg);
    }
    if (best.seg == 0) consider(256);
    return best;
}

inline int tile64_smem(const Tile64Shape& t) {
    const int w = t.bx + 2 * (t.T - 1), h = t.by + 2 * (t.T - 1);
    return t.T > 1 ? 2 * 8 * 8 * w * h + 4 * (w + h + 4) : 0;
}
// Blocks of bx x by nodes in two dimensions, at most `most` of them in all if
// the width allows it (each then takes several, one below the other).
inline dim3 tile64_grid(const Tile64Shape& t, int nx, int ny, int64_t most) {
    const int64_t w = (nx + t.bx - 1) / t.bx, h = (ny + t.by - 1) / t.by;
    const int64_t cap = std::max<int64_t>(1, std::min<int64_t>(65535, most / w));
    return dim3((unsigned)w, (unsigned)std::min(h, cap));
}
inline Tile64Shape tile64(int T, int bx, int by) {
    Tile64Shape t;
    t.T = T;
    t.bx = T > 1 ? bx : 32;
    t.by = T > 1 ? by : kOne64Rows;
    for (int s = 0; s < T; ++s) {
        const int aw = t.bx + 2 * (T - 1 - s);
        t.inv[s] = (65536 + aw - 1) / aw;
    }
    return t;
}

// The FP64 launch with the fewest modelled cycles per step.  Fitted on GB300 (1 x 1
// to 1500 x 1100, T = 1 .. 4; within 4 %, the choice within 2 % of the best): W
// warps on an SM's scheduler take 660 W cycles in a tile (780 W in k_one64), a step
// of a tile 320 and a launch 2830 (3290) besides.  64 x 64: T = 3 on 8 x 4 nodes,
// 1.11 us per step (T = 1 2.1); 256 x 256: T = 1, 3.3 us (T = 2 on 16 x 16 3.9).
inline Tile64Shape tile64_shape(int nx, int ny, int nsm) {
    const int tiles[9][2] = {{4, 4}, {8, 2}, {16, 2}, {8, 4}, {16, 4}, {8, 8}, {16, 8}, {32, 4}, {16, 16}};
    Tile64Shape best;
    for (int T = 1; T <= kT64Max; ++T)
        for (const auto& b : tiles) {
            Tile64Shape t = tile64(T, b[0], b[1]);
            if (tile64_smem(t) > kT64Smem) continue;
            const dim3 g = tile64_grid(t, nx, ny, (int64_t)1 << 40);
            const int64_t here = ((int64_t)g.x * ((ny + t.by - 1) / t.by) + nsm - 1) / nsm;   // tiles per SM
            t.cost = T > 1 ? 2830.0 : 3290.0;
            for (int s = 0; s < T; ++s) {
                const int slots = (t.bx + 2 * (T - 1 - s)) * (t.by + 2 * (T - 1 - s));
                const int64_t warps = here * (T > 1 ? (slots + 15) / 16 : (slots + 31) / 32);
                t.cost += T > 1 ? 320.0 + 660.0 * (double)((warps + 3) / 4) : 780.0 * (double)((warps + 3) / 4);
            }
            if (best.T == 0 || t.cost * best.T < 0.999 * best.cost * t.T) best = t;
        }
    return best;
}

cudaError_t tile_f64(const StepParams& a, const Coef<double>& c, bool gen, const Tile64Shape& t, bool check,
                     int64_t* blocks, cudaStream_t st);

// A tile launch: T steps, blocks of NW warps of RR rows.
struct TileShape {
    int T = 0, RR = 0, NW = 0;
    double cost = 0.0;            // modelled cycles of one launch
};
inline int64_t tile_count(const TileShape& t, int nx, int ny) {
    const int ox = kStSlots - 2 * (t.T - 1), oy = t.NW * t.RR - 2 * (t.T - 1);
    return (int64_t)((nx + ox - 1) / ox) * ((ny + oy - 1) / oy);
}
inline int tile_smem(int NW) { return 2 * (NW + 2) * 6 * 256; }

// The tile launch with the fewest modelled cycles per step.  Fitted to
// launches back to back on GB300 (2 .. 12 steps, 4 .. 16 warps, one block per
// multiprocessor): an FP32 step costs a warp about 50 + 97 w cycles per row with w
// warps on its scheduler; start, loads and stores together 3500 cycles and 145
// per slot row of a multiprocessor.  16 warps are resident.  FP16S (1 x 1 to
// 1400 x 1400, 95 % of the launches within 20 %, the choice within 4 % of the best): 303 + 61 w cycles
// per row and step, 49 w more where the state is rounded, which is every `group`
// steps; a launch takes whole groups.
inline TileShape tile_shape(int dtype, int group, int nx, int ny, int nsm) {
    TileShape best;
    for (int T = 2; T <= 12; ++T)
        for (int RR = 2; RR <= 4 && T % group == 0; RR += 2)
            for (int NW = 2; NW <= 16; ++NW) {
                TileShape t;
                t.T = T;
                t.RR = RR;
                t.NW = NW;
                if (NW * RR - 2 * (T - 1) < 1) continue;
                const int64_t blocks = tile_count(t, nx, ny), slots = (int64_t)nsm * (16 / NW);
                const int64_t waves = (blocks + slots - 1) / slots;
                const int64_t here = ((blocks < slots ? blocks : slots) + nsm - 1) / nsm * NW;   // warps
                const double w = (double)((here + 3) / 4);
                if (dtype == S_F32)
                    t.cost = 3500.0 + (double)waves * (145.0 * RR * here + T * RR * (50.0 + 97.0 * w));
                else
                    t.cost = 2000.0 + (double)waves * RR * (177.0 * here + T * (303.0 + 61.0 * w) + T / group * 49.0 * w);
                if (best.T == 0 || t.cost * best.T < best.cost * t.T) best = t;
            }
    return best;
}

// T fused steps of FP32 storage on register tiles (k_tile); check: the last
// step is the residual-check step (one partial set per block).
cudaError_t tile_f32(const StepParams& a, const Coef<float>& c, bool gen, const TileShape& t, bool check,
                     cudaStream_t st);
// The same of FP16-shifted storage; bit t of rounds: the state is rounded after
// step t (as by a launch that ends there).
cudaError_t tile_f16s(const StepParams& a, const Coef<float>& c, bool gen, const TileShape& t, bool check,
                      unsigned rounds, cudaStream_t st);

// T fused steps on the wavefront schedule (k_strip; FP32: T = 2 .. 6, FP16S:
// T = 3, 4; check: T = 4, FP32 also 5, with the residual on the last step), segments of seg
// rows.  warps non-null: only the resident warps per multiprocessor of that
// kernel.  Defined with each storage type's kernels.
cudaError_t strip_f32(const StepParams& a, const Coef<float>& c, bool gen, int T, bool check, int seg, int* warps,
                      cudaStream_t st);
cudaError_t strip_f16s(const StepParams& a, const Coef<float>& c, bool gen, int T, bool check, int seg, int* warps,
                       cudaStream_t st);

// Three fused steps (k_step3); defined with each storage type's kernels.
cudaError_t step3_f32(const StepParams& a, const Coef<float>& c, bool gen, bool check,
                      int check_blocks, cudaStream_t st);
cudaError_t step3_f16s(const StepParams& a, const Coef<float>& c, bool gen, bool check,
                       int check_blocks, cudaStream_t st);

// Two fused steps (k_step2) of FP32 or FP16-shifted storage; defined with
// each storage type's kernels.
cudaError_t step2_f32(const StepParams& a, const Coef<float>& c, bool gen, bool check,
                      int check_blocks, cudaStream_t st);
cudaError_t step2_f16s(const StepParams& a, const Coef<float>& c, bool gen, bool check,
                       int check_blocks, cudaStream_t st);

inline dim3 step_grid(int nx, int ny, int V) {
    return dim3((unsigned)((nx + 32 * V - 1) / (32 * V)), (unsigned)((ny + BY - 1) / BY));
}

}  // namespace lbm
