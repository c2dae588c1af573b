// lbm_core.cuh -- per-node arithmetic of the periodic lattice Boltzmann scheme
// for linear elasticity (Boolakee, Geier, De Lorenzis, arXiv 2208.14870),
// shared by every kernel of the library.
//
// Populations are kept in the paper's one-index order (Sec. 4, population
// table): c_1..c_8 = (1,0) (0,1) (-1,0) (0,-1) (1,1) (-1,1) (-1,-1) (1,-1),
// stored here as f[0..7].  Moments use the paper's moment order
// 10, 01, 11, s, d, 12, 21, 22 (Sec. 4, moment table).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace lbm {

// Rounding is spelled out wherever it could depend on the compiler: a
// product that is not exact is either rounded on its own (rmul, never fused
// into a later add) or fused on purpose (fmad).  Products with 1/2, 1/4 and 2
// are exact, so fusing them or not gives the same bits.  Every kernel that
// runs this arithmetic (one step per launch, two steps per launch, the
// batched arena) therefore computes the same bits for the same inputs.
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fmad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmad(double a, double b, double c) { return fma(a, b, c); }

// Moments of the collision basis.
template <typename T>
struct Mom {
    T m10, m01, m11, ms, md, m12, m21, m22;
};

// A factor in [-1/2, 1/2) as a multiple of 2^-64: its upper and lower halves, the
// lower one without its last bit (step_fixed).
struct Factor {
    int hi, lo;
};
inline Factor factor(double v) {
    const int64_t b = llrint(ldexp(v, 64));
    return {(int)(b >> 32), (int)((uint32_t)b >> 1)};
}
// The same constants as factors (FP64 storage); fixed, fields_fixed: all of them
// are in range.
template <typename T>
struct CoefFixed {};
template <>
struct CoefFixed<double> {
    Factor k11, ks, kd, kw12t, k12, kw21t, k21, k22;
    Factor h11, hs, hd;            // -b / 2 of the bared moments (recovery of the fields)
    int fixed, fields_fixed;
};

// Per-lattice constants of the collision in compute precision, in the
// quarter form collide returns (every factor of a second-order moment
// divided by 4; see collide):
//   q11 = (1 - w11)/4, qs = (1 - ws)/4, qd = (1 - wd)/4     (Eq. collision, m^eq = 0)
//   qw12t = w12 theta / 4, q12 = (1 - w12)/4, ...          (m^eq_12 = theta mbar_10)
//   qtheta = theta / 4; theta itself for the FP16-shifted store
template <typename T>
struct Coef : CoefFixed<T> {
    T q11, qs, qd;
    T qw12t, q12, qw21t, q21, q22;
    T qtheta, theta;
    T b11, bs, bd;   // 1 - w/2 (bared moments, Eq. compute_bared)
};
inline void set_factors(Coef<float>&) {}
inline void set_factors(Coef<double>& c) {
    const double q[8] = {c.q11, c.qs, c.qd, c.qw12t, c.q12, c.qw21t, c.q21, c.q22};
    Factor* k[8] = {&c.k11, &c.ks, &c.kd, &c.kw12t, &c.k12, &c.kw21t, &c.k21, &c.k22};
    c.fixed = 1;
    for (int i = 0; i < 8; ++i) {
        if (fabs(q[i]) < 0.499) *k[i] = factor(q[i]);
        else c.fixed = 0;
    }
    const double b[3] = {-0.5 * c.b11, -0.5 * c.bs, -0.5 * c.bd};
    Factor* h[3] = {&c.h11, &c.hs, &c.hd};
    c.fields_fixed = 1;
    for (int i = 0; i < 3; ++i) {
        if (fabs(b[i]) < 0.499) *h[i] = factor(b[i]);
        else c.fields_fixed = 0;
    }
}

// Raw moments of eight populations, Eq. moments and Eq. replace_raw, written
// as a butterfly: with p = f5 + f7, q = f6 + f8, r = f5 - f7, s = f6 - f8,
//   m11 = p - q, m22 = p + q, m12 = r - s, m21 = r + s,
//   m10 = (f1 - f3) + m12, m01 = (f2 - f4) + m21,
//   ms = (f1 + f3) + (f2 + f4) + 2 m22, md = (f1 + f3) - (f2 + f4).
template <typename T>
__device__ __forceinline__ Mom<T> moments(const T f[8]) {
    Mom<T> m;
    const T p = f[4] + f[6], q = f[5] + f[7];
    const T r = f[4] - f[6], s = f[5] - f[7];
    m.m11 = p - q;
    m.m22 = p + q;
    m.m12 = r - s;
    m.m21 = r + s;
    m.m10 = (f[0] - f[2]) + m.m12;
    m.m01 = (f[1] - f[3]) + m.m21;
    const T s13 = f[0] + f[2], s24 = f[1] + f[3];
    m.ms = (s13 + s24) + T(2) * m.m22;
    m.md = s13 - s24;
    return m;
}

// Collision in moment space (Algorithm 1, collision block):
//   mbar_10 = m_10 + g_x/2, mbar_01 = m_01 + g_y/2          (Eqs. coll10, coll01)
//   m*_a = w_a m^eq_a + (1 - w_a) m_a, Table 1 equilibria  (Eq. collision)
//   m*_10 = mbar_10 + g_x/2, m*_01 = mbar_01 + g_y/2       (Eqs. coll10post, coll01post)
// GEN = false is the standard case w_12 = w_21 = w_22 = 1 (Sec. 3.3.2),
// where m*_12 = theta u, m*_21 = theta v, m*_22 = 0.
// u, v receive the displacement mbar_10, mbar_01 (Table 2).
//
// Returned in the form the back-transform consumes ("quarter form"): m*_10
// and m*_01 as they are, the moments of order two and higher (11, s, d, 12,
// 21, 22) divided by 4.  The 1/4 rides on the coefficients (Coef), and since
// 4 is a power of two, (c/4) * m rounds to exactly (c * m)/4: the stored
// populations are the same bits as without it, at six fewer multiplications
// per node.
// The displacement u = mbar_10, v = mbar_01 of raw moments m (Eqs. coll10,
// coll01; Table 2).
template <typename T>
__device__ __forceinline__ void displacement(const Mom<T>& m, T gx, T gy, T& u, T& v) {
    u = m.m10 + T(0.5) * gx;
    v = m.m01 + T(0.5) * gy;
}

template <typename T, bool GEN>
__device__ __forceinline__ Mom<T> collide(const Mom<T>& m, T gx, T gy, const Coef<T>& c,
                                          T& u, T& v) {
    Mom<T> s;
    displacement(m, gx, gy, u, v);
    s.m10 = m.m10 + gx;
    s.m01 = m.m01 + gy;
    s.m11 = rmul(c.q11, m.m11);
    s.ms = rmul(c.qs, m.ms);
    s.md = rmul(c.qd, m.md);
    if (GEN) {
        s.m12 = fmad(c.qw12t, u, rmul(c.q12, m.m12));
        s.m21 = fmad(c.qw21t, v, rmul(c.q21, m.m21));
        s.m22 = rmul(c.q22, m.m22);
    } else {
        s.m12 = rmul(c.qtheta, u);
        s.m21 = rmul(c.qtheta, v);
        s.m22 = T(0);
    }
    return s;
}

// Raw moments in quarter form (for states that did not come from collide).
template <typename T>
__device__ __forceinline__ Mom<T> quarter(Mom<T> m) {
    const T q = T(0.25);
    m.m11 = q * m.m11;
    m.ms = q * m.ms;
    m.md = q * m.md;
    m.m12 = q * m.m12;
    m.m21 = q * m.m21;
    m.m22 = q * m.m22;
    return m;
}

// Back-transformation f = M^-1 m (Eq. moments_post solved in closed form),
// from the quarter form (m11 ... m22 below are the moments divided by 4):
//   A = m10 - 4 m12, B = m01 - 4 m21, P = ms - 2 m22 + md, Q = ms - 2 m22 - md
//   f1 = P + A/2, f3 = P - A/2, f2 = Q + B/2, f4 = Q - B/2
//   f5 = m22 + m11 + m12 + m21, f6 = m22 - m11 - m12 + m21,
//   f7 = m22 + m11 - m12 - m21, f8 = m22 - m11 + m12 - m21.
// ZERO22: the standard rates (w_22 = 1, so m*_22 = m^eq_22 = 0) drop m22
// from the sums; that changes at most the sign of a zero population, so every
// kernel running the standard rates uses this form.
template <bool ZERO22 = false, typename T>
__device__ __forceinline__ void populations(const Mom<T>& s, T f[8]) {
    const T A = fmad(T(-4), s.m12, s.m10), B = fmad(T(-4), s.m21, s.m01);
    if (ZERO22) {
        const T P = s.ms + s.md, Q = s.ms - s.md;
        f[0] = fmad(T(0.5), A, P);
        f[2] = fmad(T(-0.5), A, P);
        f[1] = fmad(T(0.5), B, Q);
        f[3] = fmad(T(-0.5), B, Q);
        const T h3 = s.m12 + s.m21, h4 = s.m21 - s.m12;
        f[4] = s.m11 + h3;
        f[6] = s.m11 - h3;
        f[5] = h4 - s.m11;
        f[7] = -s.m11 - h4;
        return;
    }
    const T t = fmad(T(-2), s.m22, s.ms);
    const T P = t + s.md, Q = t - s.md;
    f[0] = fmad(T(0.5), A, P);
    f[2] = fmad(T(-0.5), A, P);
    f[1] = fmad(T(0.5), B, Q);
    f[3] = fmad(T(-0.5), B, Q);
    const T h1 = s.m22 + s.m11, h2 = s.m22 - s.m11;
    const T h3 = s.m12 + s.m21, h4 = s.m21 - s.m12;
    f[4] = h1 + h3;
    f[6] = h1 - h3;
    f[5] = h2 + h4;
    f[7] = h2 - h4;
}

// Post-collision populations straight from the raw moments: collide, then
// populations (the standard rates drop m*_22).  (Merging the two into fused
// multiply-adds on the raw moments saves two operations per node but measured
// slower in the four-step wavefront kernel.)
template <bool GEN, typename T>
__device__ __forceinline__ void collide_populations(const Mom<T>& m, T gx, T gy, const Coef<T>& c, T& u, T& v,
                                                    T f[8]) {
    populations<!GEN>(collide<T, GEN>(m, gx, gy, c, u, v), f);
}

// The same step of FP64 storage.  GB300's FP64 pipe takes 64 cycles of a
// scheduler per warp instruction, an integer instruction one or two, so the step
// runs in integers: the node's populations and half forces become multiples of
// one unit, 2^-58 of the power of two above the largest of them (at least five
// bits more than FP64 holds of that one), their sums are exact, its five
// products (eight at general rates) are good to two and a half units, and the results
// are rounded to FP64 once.  So the error is bounded relative to the node's largest
// value: before the last rounding a population is within 20 units of the exact
// result (34 at general rates; each input loses less than a unit), 2^-53.7 (2^-52.9) of
// that power of two, where FP64 arithmetic rounds at 2^-53 of each of its partial
// sums.  A value far below the node's largest one has fewer bits than
// FP64 would keep of it until it meets the others in a sum, and none from 2^-58
// on.  The first moments of the result are mbar + g / 2 up to the last rounding.
// About 600 integer instructions, two cycles of the ALU for 360 of them, against 34
// FP64 ones (2176 cycles): 1500 x 1100 116 -> 44 us per step; with the signs on the FMA
// pipe 43.0, and with two, three, four, five, six of the results on the FP64 pipe
// 40.2, 39.9, 37.8, 37.8, 41.6 us.  Nodes of infinities, NaN or values near the ends of the exponent range, and
// rates with a factor of 1/2 or more, take FP64 arithmetic.
// m (below 2^63) with the sign of the word w.  FMA: most of the work on the FMA pipe
// (a multiplication by the sign) instead of the ALU, which bounds the step where many warps share a scheduler; slower
// where one warp runs alone.
template <bool FMA>
__device__ __forceinline__ int64_t signed_as(uint64_t m, int w) {
    const int t = w >> 31;
    if (!FMA) return ((int64_t)m ^ (int64_t)t) - (int64_t)t;
    const uint32_t s = (uint32_t)(t | 1), ml = (uint32_t)m, mh = (uint32_t)(m >> 32);
    uint32_t lo, hi;
    // (-m = m (2^32 - 1) - m 2^32 in 64 bits)
    asm("{\n\t.reg .b64 r;\n\tmul.wide.u32 r, %2, %4;\n\tmov.b64 {%0, %1}, r;\n\tmad.lo.s32 %1, %3, %4, %1;\n\t"
        "mad.lo.s32 %1, %2, %5, %1;\n\t}" : "=&r"(lo), "=&r"(hi) : "r"(ml), "r"(mh), "r"(s), "r"(t));
    return (int64_t)((uint64_t)hi << 32 | lo);
}
// x as a multiple of the unit; h: one more halving.
template <bool FMA>
__device__ __forceinline__ int64_t to_fixed(double x, uint32_t e, int h) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t d = (e - (hi & 0x7ff00000u)) >> 20;
    uint64_t m = ((uint64_t)((hi & 0x000fffffu) | 0x00100000u) << 32 | lo) << (5 - h);
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(d));                 // (64 and more: zero)
    return signed_as<FMA>(m, (int)hi);
}
// An FP32 x as a multiple of 2^-58 of the power of two above the largest value of
// exponent field e.
__device__ __forceinline__ int64_t to_fixed(float x, uint32_t e, int h) {
    const uint32_t b = __float_as_uint(x), d = (e - (b & 0x7f800000u)) >> 23;
    uint64_t m = (uint64_t)((b & 0x007fffffu) | 0x00800000u) << (34 - h);
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(d));
    return signed_as<true>(m, (int)b);
}
// v units (|v| < 2^63), rounded to FP64 (ties to even).
template <bool FMA>
__device__ __forceinline__ double from_fixed(int64_t v, uint32_t e) {
    const int vh = (int)(v >> 32);
    const uint64_t a = (uint64_t)signed_as<FMA>((uint64_t)v, vh);
    const uint32_t ah = (uint32_t)(a >> 32), x = ah ? ah : (uint32_t)a;
    int t;                                                         // the highest set bit, 0 .. 62 (-1: none)
    asm("bfind.u32 %0, %1;" : "=r"(t) : "r"(x));
    if (ah) t += 32;
    const uint64_t b = a << (62 - t), m = (b + 511 + (((uint32_t)b >> 10) & 1)) >> 10;   // [2^52, 2^53], or 0
    uint32_t hi = (uint32_t)(m >> 32);
    if (x) hi += ((uint32_t)t << 20) + (e - (58u << 20));
    return __hiloint2double((int)(hi | (vh & 0x80000000)), (int)(uint32_t)m);
}
// The same by two FP64 additions: v's upper word above 2^84 + 2^63
// units, its lower word above 2^52; the first difference is exact.
__device__ __forceinline__ double from_fixed_fp64(int64_t v, uint32_t e) {
    const int k = (int)(e + (27u << 20));
    const double d1 = __hiloint2double(k, (int)((uint32_t)(v >> 32) ^ 0x80000000u));
    const double d2 = __hiloint2double((int)(e - (5u << 20)), (int)(uint32_t)v);
    return (d1 - __hiloint2double(k, (int)0x80100000u)) + d2;      // 2^84 + 2^63 + 2^52
}
// a times a factor, within about a unit (|a| < 2^62).
__device__ __forceinline__ int64_t mul_fixed(Factor k, int64_t a) {
    const int ah = (int)(a >> 32), al = (int)((uint32_t)a >> 1);
    const int64_t t = (int64_t)ah * k.lo + (int64_t)al * k.hi;
    return (int64_t)ah * k.hi + (t >> 31);
}

// Not zero if x is neither of the zeros.
__device__ __forceinline__ uint32_t nonzero(double x) {
    return (uint32_t)__double2hiint(x) << 1 | (uint32_t)__double2loint(x);
}
__device__ __forceinline__ uint32_t nonzero(float x) { return __float_as_uint(x) << 1; }

template <bool GEN>
__device__ __forceinline__ void step_f64(const double f[8], double gx, double gy, const Coef<double>& c, double& u,
                                         double& v, double o[8]) {
    uint32_t e = 0;
#pragma unroll
    for (int p = 0; p < 8; ++p) e = max(e, (uint32_t)__double2hiint(f[p]) & 0x7ff00000u);
    e = max(e, (uint32_t)__double2hiint(gx) & 0x7ff00000u);
    e = max(e, (uint32_t)__double2hiint(gy) & 0x7ff00000u);
    if (!c.fixed || e - (100u << 20) > (1900u << 20)) {
        // A node of zeros (no force has reached it yet) keeps them: with FP64 arithmetic
        // a lattice of one force among zeros took 1569 us instead of 473 for twelve steps
        // (1500 x 1100), and warps of zeros and others ran both paths (1875 us).
        uint32_t any = nonzero(gx) | nonzero(gy);
#pragma unroll
        for (int p = 0; p < 8; ++p) any |= nonzero(f[p]);
        if (any == 0) {
            u = v = 0.0;
#pragma unroll
            for (int p = 0; p < 8; ++p) o[p] = 0.0;
            return;
        }
        collide_populations<GEN>(moments(f), gx, gy, c, u, v, o);
        return;
    }
    int64_t F[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) F[p] = to_fixed<true>(f[p], e, 0);
    const int64_t hx = to_fixed<true>(gx, e, 1), hy = to_fixed<true>(gy, e, 1);
    const int64_t p = F[4] + F[6], q = F[5] + F[7], r = F[4] - F[6], s = F[5] - F[7];
    const int64_t m11 = p - q, m22 = p + q, m12 = r - s, m21 = r + s;
    const int64_t U = (F[0] - F[2]) + m12 + hx, V = (F[1] - F[3]) + m21 + hy;
    const int64_t s13 = F[0] + F[2], s24 = F[1] + F[3];
    const int64_t X = mul_fixed(c.k11, m11), S = mul_fixed(c.ks, s13 + s24 + 2 * m22), D = mul_fixed(c.kd, s13 - s24);
    int64_t Tu = mul_fixed(c.kw12t, U), Tv = mul_fixed(c.kw21t, V), W = 0;
    if (GEN) {
        Tu += mul_fixed(c.k12, m12);
        Tv += mul_fixed(c.k21, m21);
        W = mul_fixed(c.k22, m22);
    }
    // m*_10 - m*_12 and m*_01 - m*_21, halved without a loss
    const int64_t A = U + hx - 4 * Tu, B = V + hy - 4 * Tv, Ah = A >> 1, Bh = B >> 1;
    const int64_t P = S + D - 2 * W, Q = S - D - 2 * W;
    o[0] = from_fixed_fp64(P + Ah, e);
    o[2] = from_fixed_fp64(P - (A - Ah), e);
    o[1] = from_fixed_fp64(Q + Bh, e);
    o[3] = from_fixed_fp64(Q - (B - Bh), e);
    o[4] = from_fixed<true>(W + X + (Tu + Tv), e);
    o[6] = from_fixed<true>(W + X - (Tu + Tv), e);
    o[5] = from_fixed<true>(W - X + (Tv - Tu), e);
    o[7] = from_fixed<true>(W - X - (Tv - Tu), e);
    u = from_fixed<false>(U, e);
    v = from_fixed<false>(V, e);
}

// step_f64 of one node on two lanes, 2k (h = 0) and 2k + 1 (h = 1), for launches
// of few warps: half the conversions each, 500 instructions in a row (with those of
// k_tile64 around it) instead of 800.  Lane h holds populations h, h + 2, h + 4 and h + 6 in f[0 .. 3] and the
// force's component h, and receives the same populations of the result and the
// component w of the displacement.  The bits are step_f64's.  Every lane of the
// warp calls it.  (No signs on the FMA pipe and no results on the FP64 pipe: with
// one or two warps per scheduler both only lengthen the chain, 64 x 64 1.34
// against 1.41 us per step.  Nor are nodes of zeros told apart: 64 x 64 with one
// forced node, twelve steps, 37 -> 17 us, but every other launch lost 0.4 to 1.4 %, and a
// small lattice is filled within some tens of steps.)
template <bool GEN>
__device__ __forceinline__ void step_f64_half(const double f[4], double g, int h, const Coef<double>& c, double& w,
                                              double o[4]) {
    constexpr unsigned ALL = 0xffffffffu;
    uint32_t e = 0;
#pragma unroll
    for (int p = 0; p < 4; ++p) e = max(e, (uint32_t)__double2hiint(f[p]) & 0x7ff00000u);
    e = max(e, (uint32_t)__double2hiint(g) & 0x7ff00000u);
    e = max(e, __shfl_xor_sync(ALL, e, 1));
    const bool slow = !c.fixed || e - (100u << 20) > (1900u << 20);
    auto other = [&](int64_t v) { return __shfl_xor_sync(ALL, v, 1); };
    const int64_t t = -h;                                    // (v ^ t) - t: v on lane 0, -v on lane 1
    const int64_t A0 = to_fixed<false>(f[0], e, 0), A2 = to_fixed<false>(f[1], e, 0), B0 = to_fixed<false>(f[2], e, 0),
                  B1 = to_fixed<false>(f[3], e, 0), H = to_fixed<false>(g, e, 1);
    const int64_t sB = B0 + B1, dB = B0 - B1, sA = A0 + A2, dA = A0 - A2;
    const int64_t sBo = other(sB), dBo = other(dB), sAo = other(sA);
    const int64_t m = dB - ((dBo ^ t) - t);                  // m_12 = r - s, m_21 = s + r
    const int64_t U = dA + m + H;
    const int64_t X = mul_fixed(c.k11, ((sB - sBo) ^ t) - t);
    const int64_t S = mul_fixed(c.ks, sA + sAo + 2 * (sB + sBo)), D = mul_fixed(c.kd, ((sA - sAo) ^ t) - t);
    int64_t T = mul_fixed(c.kw12t, U), W = 0;                // (w_21 = w_12)
    if (GEN) {
        T += mul_fixed(c.k12, m);
        W = mul_fixed(c.k22, sB + sBo);
    }
    const int64_t To = other(T);
    const int64_t A = U + H - 4 * T, Ah = A >> 1, P = S + ((D ^ t) - t) - 2 * W;
    const int64_t Xs = W + ((X ^ t) - t), Z = T + ((To ^ t) - t);
    o[0] = from_fixed<false>(P + Ah, e);
    o[1] = from_fixed<false>(P - (A - Ah), e);
    o[2] = from_fixed<false>(Xs + Z, e);
    o[3] = from_fixed<false>(Xs - Z, e);
    w = from_fixed<false>(U, e);
    if (__any_sync(ALL, slow)) {
        double a[8], gx = __shfl_xor_sync(ALL, g, 1), gy = gx, u, v, r[8];
        if (h) gy = g;
        else gx = g;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const double q = __shfl_xor_sync(ALL, f[p], 1);
            a[2 * p] = h ? q : f[p];
            a[2 * p + 1] = h ? f[p] : q;
        }
        if (slow) {
            collide_populations<GEN>(moments(a), gx, gy, c, u, v, r);
#pragma unroll
            for (int p = 0; p < 4; ++p) o[p] = h ? r[2 * p + 1] : r[2 * p];
            w = h ? v : u;
        }
    }
}

// Shifted FP16 storage.  The equilibrium-type part of a post-collision state
// with first moments (c10, c01) is E = M^-1 (c10, c01, 0, 0, 0, theta c10,
// theta c01, 0):
//   E1 = k1 c10, E3 = -k1 c10, E2 = k1 c01, E4 = -k1 c01   (k1 = (1 - theta)/2)
//   E5 = k5 (c10 + c01), E6 = k5 (c01 - c10), E7 = -k5 (c10 + c01),
//   E8 = k5 (c10 - c01)                                     (k5 = theta/4)
// The stored deviation is N = f* - E = M^-1 (0, 0, m*_11, m*_s, m*_d,
// m*_12 - theta m*_10, m*_21 - theta m*_01, m*_22), which is O(eps) of f*.
// (Quarter form in and out: the m*_12 - theta m*_10 terms are divided by 4;
// qtheta = theta / 4.)
template <typename T>
__device__ __forceinline__ Mom<T> deviation_moments(const Mom<T>& s, T qtheta) {
    Mom<T> n = s;
    n.m10 = T(0);
    n.m01 = T(0);
    n.m12 = fmad(-qtheta, s.m10, s.m12);
    n.m21 = fmad(-qtheta, s.m01, s.m21);
    return n;
}

// Error-free FP32 transformations for the steady-state residual.  GB300's
// FP64 pipe issues about 1/64 of the FP32 rate, so the residual of FP32 and
// FP16-shifted storage evaluates the displacement in FP32 pairs (hi + lo)
// instead of FP64 per node: two_sum is Knuth's TwoSum (s + e == a + b
// exactly, six FP32 additions, no branch), fast_two_sum Dekker's form for
// |a| >= |b| (three additions).  Every operation is written with explicit
// rounding so that no compiler contraction or reassociation can touch it.
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

__device__ __forceinline__ float fast_two_sum(float a, float b, float& e) {
    const float s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
    return s;
}

// The displacement of eight FP32 pre-collision populations, u = mbar_10 =
// m_10 + g_x / 2 and v = mbar_01 (Eqs. coll10, coll01; Table 2), as FP32
// pairs (u_hi, u_lo, v_hi, v_lo).  The sums are the moment butterfly's
// (moments(), then collide's half force), so u_hi + u_lo carries exactly the
// value the butterfly rounds, with each addition's rounding error recovered
// by two_sum: m_12 = r - s with r = f5 - f7, s = f6 - f8, m_10 = (f1 - f3) +
// m_12, u = m_10 + g_x / 2 (and m_21 = r + s, m_01 = (f2 - f4) + m_21).  The
// error terms are summed in FP32, so the pair is exact to about 2^-44 of the
// largest partial sum; the hi parts are the FP32 values the collision uses.
__device__ __forceinline__ float4 exact_displacement(const float f[8], float gx, float gy) {
    float er, es, e12, e21, ea, eb, e10, e01, eu, ev;
    const float r = two_sum(f[4], -f[6], er);
    const float s = two_sum(f[5], -f[7], es);
    const float m12 = two_sum(r, -s, e12);
    const float m21 = two_sum(r, s, e21);
    const float a = two_sum(f[0], -f[2], ea);
    const float b = two_sum(f[1], -f[3], eb);
    const float m10 = two_sum(a, m12, e10);
    const float m01 = two_sum(b, m21, e01);
    const float u = two_sum(m10, 0.5f * gx, eu);
    const float v = two_sum(m01, 0.5f * gy, ev);
    const float ulo = __fadd_rn(__fadd_rn(__fadd_rn(eu, e10), __fadd_rn(ea, e12)), __fsub_rn(er, es));
    const float vlo = __fadd_rn(__fadd_rn(__fadd_rn(ev, e01), __fadd_rn(eb, e21)), __fadd_rn(er, es));
    float4 d;
    d.x = two_sum(u, ulo, d.y);
    d.z = two_sum(v, vlo, d.w);
    return d;
}

// Programmatic dependent launch.  A kernel launched with launch_after (below)
// starts as soon as its predecessor's blocks have exited, without waiting for
// the stream to see the predecessor completed: it calls after_predecessor()
// before it touches global memory, which waits until the predecessor's writes
// are visible.  Launches in a stream otherwise followed one another on a 2.05 us
// grid (a tile launch of 4.7 us took 6.25).  No kernel lets its successor
// start earlier than that: blocks of the next strip launch then took the slots
// the running one left and clumped (1024^2, 400 steps: 2.37 against 1.85 ms).
__device__ __forceinline__ void after_predecessor() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ int wrap_dec(int i, int n) { return i == 0 ? n - 1 : i - 1; }
__device__ __forceinline__ int wrap_inc(int i, int n) { return i + 1 == n ? 0 : i + 1; }

// ---------------------------------------------------------------------------
// The per-node arithmetic above for two nodes at a time, in the packed FP32 instructions of sm_103a (add / sub / fma .f32x2:
// two FP32 operations per issue slot).
//
// Every packed operation rounds each half as its scalar counterpart does, and
// the sums are those above up to powers of two and signs, which
// rounding commutes with; so a pair holds the values the scalar code computes
// (the sign of a zero aside).  Two things shape the form:
//   - the assembler may fuse a packed product into a following packed sum,
//     so the products of the relaxation (rmul above) are scalar
//     multiplications with explicit rounding, which it does not fuse; their
//     factors come from the constant bank;
//   - a packed constant needs a register pair, or two moves at each use, so
//     the factors 2, -1/2 and -4 of lbm_core.cuh are folded away: only 1/2 and
//     -2 remain.
using pair_t = unsigned long long;   // two FP32 values: low half first

__device__ __forceinline__ pair_t pk(float lo, float hi) {
    pair_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void unpk(pair_t p, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p));
}
__device__ __forceinline__ float pk_lo(pair_t p) {
    float lo, hi;
    unpk(p, lo, hi);
    return lo;
}
__device__ __forceinline__ float pk_hi(pair_t p) {
    float lo, hi;
    unpk(p, lo, hi);
    return hi;
}
__device__ __forceinline__ pair_t add2(pair_t a, pair_t b) {
    pair_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ pair_t sub2(pair_t a, pair_t b) {
    pair_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ pair_t fma2(pair_t a, pair_t b, pair_t c) {
    pair_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ pair_t splat(float v) { return pk(v, v); }

__device__ __forceinline__ pair_t mul1(float c, pair_t p) {   // rounded on its own
    float lo, hi;
    unpk(p, lo, hi);
    return pk(__fmul_rn(c, lo), __fmul_rn(c, hi));
}
__device__ __forceinline__ pair_t neg2(pair_t p) { return p ^ 0x8000000080000000ULL; }

// The factors of the pair form: Coef<float> with q_s doubled (moments2 halves
// m_s), and the two packed constants.  A kernel argument, so that the scalar
// factors are operands from the constant bank.
struct PairCoef {
    pair_t half, nhalf, nfour;
    float q11, qs2, qd, qw12t, q12, qw21t, q21, q22, qtheta, theta;
};

__host__ __device__ inline PairCoef pair_coef(const Coef<float>& c) {
    PairCoef d;
    d.half = 0x3f0000003f000000ULL;
    d.nhalf = 0xbf000000bf000000ULL;
    d.nfour = 0xc0800000c0800000ULL;
    d.q11 = c.q11;
    d.qs2 = 2.0f * c.qs;
    d.qd = c.qd;
    d.qw12t = c.qw12t;
    d.q12 = c.q12;
    d.qw21t = c.qw21t;
    d.q21 = c.q21;
    d.q22 = c.q22;
    d.qtheta = c.qtheta;
    d.theta = c.theta;
    return d;
}

// First stage of the moment butterfly (moments()): the sums and
// differences of opposite populations.  Populations 6 and 8 enter negated.
struct Opp2 {
    pair_t p, nq, r, s;         // f5 + f7, -(f6 + f8), f5 - f7, f6 - f8
    pair_t a, b, s13, s24;      // f1 - f3, f2 - f4, f1 + f3, f2 + f4
};

__device__ __forceinline__ Opp2 opposites2(pair_t f1, pair_t f2, pair_t f3, pair_t f4, pair_t f5, pair_t nf6,
                                           pair_t f7, pair_t nf8) {
    Opp2 o;
    o.p = add2(f5, f7);
    o.nq = add2(nf6, nf8);
    o.r = sub2(f5, f7);
    o.s = sub2(nf8, nf6);
    o.a = sub2(f1, f3);
    o.b = sub2(f2, f4);
    o.s13 = add2(f1, f3);
    o.s24 = add2(f2, f4);
    return o;
}

// The same from eight populations as they are.
__device__ __forceinline__ Opp2 opposites2(const pair_t f[8]) {
    Opp2 o = opposites2(f[0], f[1], f[2], f[3], f[4], 0, f[6], 0);
    o.nq = sub2(sub2(0, f[5]), f[7]);
    o.s = sub2(f[5], f[7]);
    return o;
}

struct Mom2 {
    pair_t m10, m01, m11, msh, md, m12, m21, m22;   // msh = m_s / 2
};

__device__ __forceinline__ Mom2 moments2(const Opp2& o, const PairCoef& c) {
    Mom2 m;
    m.m11 = add2(o.p, o.nq);
    m.m22 = sub2(o.p, o.nq);
    m.m12 = sub2(o.r, o.s);
    m.m21 = add2(o.r, o.s);
    m.m10 = add2(o.a, m.m12);
    m.m01 = add2(o.b, m.m21);
    m.msh = fma2(c.half, add2(o.s13, o.s24), m.m22);
    m.md = sub2(o.s13, o.s24);
    return m;
}

// Post-collision moments in the quarter form (collide()).
struct Post2 {
    pair_t m10, m01, m11, ms, md, m12, m21, m22;
};

template <bool GEN>
__device__ __forceinline__ Post2 collide2(const Mom2& m, pair_t gx, pair_t gy, const PairCoef& c) {
    Post2 s;
    const pair_t u = fma2(c.half, gx, m.m10), v = fma2(c.half, gy, m.m01);
    s.m10 = add2(m.m10, gx);
    s.m01 = add2(m.m01, gy);
    s.m11 = mul1(c.q11, m.m11);
    s.ms = mul1(c.qs2, m.msh);
    s.md = mul1(c.qd, m.md);
    if (GEN) {
        s.m12 = fma2(splat(c.qw12t), u, mul1(c.q12, m.m12));
        s.m21 = fma2(splat(c.qw21t), v, mul1(c.q21, m.m21));
        s.m22 = mul1(c.q22, m.m22);
    } else {
        s.m12 = mul1(c.qtheta, u);
        s.m21 = mul1(c.qtheta, v);
        s.m22 = 0;
    }
    return s;
}

// Back-transformation (populations()) up to the last sum of
// each population, which the caller takes one at a time in the order it needs
// them.
template <bool ZERO22>
struct Pop2 {
    pair_t A, B, P, Q, h1, h2, h3, h4;
    __device__ __forceinline__ Pop2(const Post2& s, const PairCoef& c) {
        A = fma2(c.nfour, s.m12, s.m10);
        B = fma2(c.nfour, s.m21, s.m01);
        h3 = add2(s.m12, s.m21);
        h4 = sub2(s.m21, s.m12);
        const pair_t t = ZERO22 ? s.ms : sub2(s.ms, add2(s.m22, s.m22));
        P = add2(t, s.md);
        Q = sub2(t, s.md);
        h1 = ZERO22 ? s.m11 : add2(s.m22, s.m11);
        h2 = ZERO22 ? s.m11 : sub2(s.m11, s.m22);
    }
    __device__ __forceinline__ pair_t f1(const PairCoef& c) const { return fma2(c.half, A, P); }
    __device__ __forceinline__ pair_t f2(const PairCoef& c) const { return fma2(c.half, B, Q); }
    __device__ __forceinline__ pair_t f3(const PairCoef& c) const { return fma2(c.nhalf, A, P); }
    __device__ __forceinline__ pair_t f4(const PairCoef& c) const { return fma2(c.nhalf, B, Q); }
    __device__ __forceinline__ pair_t f5() const { return add2(h1, h3); }
    __device__ __forceinline__ pair_t nf6() const { return sub2(h2, h4); }
    __device__ __forceinline__ pair_t f7() const { return sub2(h1, h3); }
    __device__ __forceinline__ pair_t nf8() const { return add2(h2, h4); }
    __device__ __forceinline__ void all(const PairCoef& c, pair_t f[8]) const {
        f[0] = f1(c);
        f[1] = f2(c);
        f[2] = f3(c);
        f[3] = f4(c);
        f[4] = f5();
        f[5] = neg2(nf6());
        f[6] = f7();
        f[7] = neg2(nf8());
    }
};

// The pair one column to the right (c_x = +1: the value pulled from x - 1) or
// to the left (from x + 1) of a warp whose lane l holds columns 2l, 2l + 1.
// The outermost column receives its own lane's value: a halo column.
__device__ __forceinline__ pair_t from_left(pair_t p) {
    float lo, hi;
    unpk(p, lo, hi);
    return pk(__shfl_up_sync(0xffffffffu, hi, 1), lo);
}
__device__ __forceinline__ pair_t from_right(pair_t p) {
    float lo, hi;
    unpk(p, lo, hi);
    return pk(hi, __shfl_down_sync(0xffffffffu, lo, 1));
}

// Launch a kernel that calls after_predecessor().
template <typename... P, typename... A>
inline cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace lbm
