// 64-bit fixed-point arithmetic of the propagation sweeps (host and device).
//
// Why integers: a GB300 SM retires one FP64 warp instruction in 64 cycles per sub-partition, but a
// 32 x 32 + 64 -> 64 bit multiply-add in 2.2 (measured: 67 and 2.2 cycles per warp instruction).  A
// product of two 64-bit fixed-point numbers to 64 bits is 4 such multiply-adds, a complex product 14,
// about 35 cycles instead of the 256 of its 4 FP64 FMAs, and it keeps 60 bits where a double keeps 53.
//
// Number format.  A value v is an int64 with a binary point fixed per quantity; for products it is
// split into balanced digits v = h 2^32 + l, l in [-2^31, 2^31) (so all partial products are signed and
// what is dropped has zero mean).  h h' goes into `acc`, h l' + l h' into `mid` (both 64-bit, several
// products may be added up); fold(acc, mid) = acc + (mid >> 32) is the product 2^-64, one multiply-add by 1,
// rounded to nearest by the 2^31 that `mid` starts from.  Only l l' is dropped.  Scales are chosen so
// that the products need no other shift.
//
// Scales (FULL_CN; fix_class per class, psi's per instance and slice):
//   psi    2^sigma with ||psi||_2 2^sigma in [2^(top-1), 2^top), top 60 or 61 (2-norm over the grid
//          points).  The step does not increase the 2-norm, and every intermediate is a solution of a
//          leading subsystem of A, whose inverse has 2-norm <= 1, so |D|, |Y| <= beta ||psi||,
//          |u| <= (1 + beta) ||psi||: no value leaves 62 bits
//   D, Y, u  as psi
//   gamma  2^64 in products (|gamma| <= beta <= 0.35), 2^58 in the pivot recurrence
//   Q, S   2^58, |Re Q|, |Im Q| < 16 for every |E| <= E_lim
// With a 2-norm near 2^60.5 one unit is 2^-60.5 of it; spread over N points, its rounding stays below
// that of the same sweep in double (tests/test_fixed_point_sweep.py and test_fixed_point_forms.py measure both against
// 113 bits).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

#ifndef __CUDACC__
#ifndef __host__
#define __host__
#define __device__
#endif
#ifndef __forceinline__
#define __forceinline__ inline
#endif
#endif

namespace tdse {

struct Digits {
    int32_t h, l;
};

struct FixClass {
    int32_t ok;             // FULL_CN has a fixed-point form (0: the FP64 sweep)
    int32_t num;            // NUMEROV_SPLIT has one
    int32_t top, xk, kv;
    int32_t ci;             // 2/beta = ci + cf 2^-64
    Digits cf;
    int64_t inv_b;          // 1/beta at 2^58
    double E_lim;
    double e_scale;         // field samples to fixed point
    double v_scale;         // dV sums back
};

// Per point: S0 at 2^58 (lo, hi), X = 2 dx^2 x as digits (l, h); and dV, mask (2^61) as digits.
struct FixPoint {
    int32_t s0_lo, s0_hi, x_l, x_h;
};
struct FixObs {
    int32_t v_l, v_h, m_l, m_h;
};

__host__ __device__ __forceinline__ Digits digits(int64_t v)
{
    const int32_t l = (int32_t)(uint32_t)(uint64_t)v;
    return Digits{(int32_t)((uint32_t)((uint64_t)v >> 32) + ((uint32_t)l >> 31)), l};
}
__host__ __device__ __forceinline__ int64_t undigits(Digits d)
{
    return (int64_t)(((uint64_t)(uint32_t)d.h << 32) + (uint64_t)(int64_t)d.l);
}
// -v - 1 (the negative of every digit but for one unit of the low one)
__host__ __device__ __forceinline__ Digits negative(Digits d) { return Digits{-d.h, ~d.l}; }

// a b + c, one instruction (spelled out: the 64-bit expression compiles to a wider multiply)
__host__ __device__ __forceinline__ int64_t mad(int32_t a, int32_t b, int64_t c)
{
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (int64_t)a * b + c;
#endif
}
__host__ __device__ __forceinline__ uint64_t madu(uint32_t a, uint32_t b, uint64_t c)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (uint64_t)a * b + c;
#endif
}
// acc + (mid >> 32)
__host__ __device__ __forceinline__ int64_t fold(int64_t acc, int64_t mid)
{
#ifdef __CUDA_ARCH__
    int64_t r;   // one multiply-add: a 64-bit add of a sign-extended word is three instructions
    asm("mad.wide.s32 %0, %1, 1, %2;" : "=l"(r) : "r"((int32_t)(uint32_t)((uint64_t)mid >> 32)), "l"(acc));
    return r;
#else
    return acc + (mid >> 32);
#endif
}

// (acc << L) + (mid >> R), 0 <= L < 32, 0 < R < 32
template <int L, int R>
__host__ __device__ __forceinline__ int64_t combine(int64_t acc, int64_t mid)
{
#ifdef __CUDA_ARCH__
    const uint32_t al = (uint32_t)(uint64_t)acc, ah = (uint32_t)((uint64_t)acc >> 32);
    const uint32_t ml = (uint32_t)(uint64_t)mid, mh = (uint32_t)((uint64_t)mid >> 32);
    const uint64_t x = L == 0 ? (uint64_t)acc : ((uint64_t)__funnelshift_l(al, ah, L) << 32) | (uint64_t)(al << L);
    const uint64_t y = ((uint64_t)(uint32_t)((int32_t)mh >> R) << 32) | (uint64_t)__funnelshift_r(ml, mh, R);
    return (int64_t)(x + y);
#else
    return (int64_t)(((uint64_t)acc << L) + (uint64_t)(mid >> R));
#endif
}
// x y 2^-(64 - L), rounded
template <int L>
__host__ __device__ __forceinline__ int64_t mul_fix(Digits x, Digits y)
{
    const int64_t mid = mad(x.h, y.l, mad(x.l, y.h, int64_t(1) << (31 - L)));
    if constexpr (L == 0) return fold(mad(x.h, y.h, 0), mid);
    else return combine<L, 32 - L>(mad(x.h, y.h, 0), mid);
}

// (a b + c d) 2^-64 + z, rounded
__host__ __device__ __forceinline__ int64_t mul2_fix(Digits a, Digits b, Digits c, Digits d, int64_t z = 0)
{
    return fold(mad(a.h, b.h, mad(c.h, d.h, z)), mad(a.h, b.l, mad(a.l, b.h, mad(c.h, d.l, mad(c.l, d.h, int64_t(1) << 31)))));
}

// D = -i gamma u: (Dr, Di) = (gr ui + gi ur, gi ui - gr ur)
__host__ __device__ __forceinline__ void mul_minus_i(Digits gr, Digits gi, Digits ur, Digits ui, int64_t& dr, int64_t& di)
{
    dr = mul2_fix(gr, ui, gi, ur);
    di = mul2_fix(gi, ui, negative(gr), ur);
}

// (2/beta) y - p
__host__ __device__ __forceinline__ int64_t update_fix(int32_t ci, Digits cf, Digits y, int64_t p)
{
    int64_t acc = mad(y.l, ci, -p);
    acc = (int64_t)((uint64_t)acc + ((uint64_t)((uint32_t)y.h * (uint32_t)ci) << 32));
    return fold(mad(cf.h, y.h, acc), mad(cf.h, y.l, mad(cf.l, y.h, int64_t(1) << 31)));
}

// ---- NUMEROV_SPLIT (tdse_numerov_fix.cuh)

// (a b + c d) 2^-62, rounded
__host__ __device__ __forceinline__ int64_t mul2_fix62(Digits a, Digits b, Digits c, Digits d)
{
    return combine<2, 30>(mad(a.h, b.h, mad(c.h, d.h, 0)),
                          mad(a.h, b.l, mad(a.l, b.h, mad(c.h, d.l, mad(c.l, d.h, int64_t(1) << 29)))));
}

// cos and sin of `turn` 2^-64 turns at 2^62, within a few units: the angle reduced to [-1/8, 1/8] turn and
// the Taylor polynomials to theta^18 and theta^19 (next term 3e-21), in fixed point: about 250
// instructions, where sincos takes about 50 FP64 instructions of 64 cycles.
__host__ __device__ __forceinline__ void fix_cos_sin(uint64_t turn, int64_t& c, int64_t& s)
{
    const int quad = (int)((turn + (uint64_t(1) << 61)) >> 62);
    const int64_t r = (int64_t)(turn - ((uint64_t)quad << 62));            // |r| <= 2^61
    const Digits th = digits(mul_fix<3>(digits(r), digits(3622009729038561421)));   // pi/2 2^61: theta at 2^62
    const Digits z = digits(mul_fix<2>(th, th));
    // (-1)^k / (2k)! and (-1)^k / (2k+1)! at 2^62
    const int64_t kc[10] = {4611686018427387904, -2305843009213693952, 192153584101141163, -6405119470038039, 114377133393536,
                            -1270857037706, 9627704831, -52899477, 220414, -720};
    const int64_t ks[10] = {4611686018427387904, -768614336404564651, 38430716820228233, -915017067148291, 12708570377060,
                            -115532457973, 740592679, -3526632, 12966, -38};
    int64_t a = kc[9], b = ks[9];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 8; k >= 0; --k) {
        a = kc[k] + mul_fix<2>(z, digits(a));
        b = ks[k] + mul_fix<2>(z, digits(b));
    }
    b = mul_fix<2>(th, digits(b));
    const int64_t c0 = (quad & 1) ? -b : a, s0 = (quad & 1) ? a : b;
    c = (quad & 2) ? -c0 : c0;
    s = (quad & 2) ? -s0 : s0;
}

__host__ __device__ __forceinline__ float rcp_f32(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / x;
#endif
}

// 2^116 / n for n in [2^55, 2^61): float seed r0 ~ 2^85 / n (|relative error e| < 2^-22) and one
// third-order Newton step.  e is carried in units of 2^-53 and below that, with e^2, in units of 2^-61
// (to 2^-53 alone its rounding acts alike on every step near the nucleus, and the error of the sweep
// grows with the number of steps): the result is within 2^-55 relative for n < 2^59 (|Q|^2 < 128), 2^-53 up to the
// end of the range, where the floors of the three terms, all one way, add up (tests/test_fixed_point_forms.py).
__host__ __device__ __forceinline__ int64_t recip_fix(int64_t n)
{
    const uint32_t nl = (uint32_t)(uint64_t)n, nh = (uint32_t)((uint64_t)n >> 32);
    const int32_t r0 = (int32_t)(rcp_f32((float)(int32_t)(uint32_t)((uint64_t)n >> 30)) * 36028797018963968.0f);
    const uint64_t p = madu((uint32_t)r0, nl, 0);
    const uint64_t q = madu((uint32_t)r0, nh, p >> 32);               // ~2^53
    const int32_t e = (int32_t)(0u - (uint32_t)q);                    // 1 - n r0 2^-85 = e 2^-53 - (p mod 2^32) 2^-85
    const int32_t f = ((int32_t)(mad(e, e, 0) >> 32) >> 13) - (int32_t)((uint32_t)p >> 24);
    return ((int64_t)r0 << 31) + (mad(r0, e, 0) >> 22) + (((r0 >> 16) * f) >> 14);
}

// One row of the pivot recurrence, from the previous row's gamma at 2^58 to this row's, S = S0 + X E.
__host__ __device__ __forceinline__ void gamma_row(int64_t inv_b, int64_t S, int64_t& gr, int64_t& gi)
{
    const Digits qr = digits(inv_b + gi), qi = digits(S - gr);
    // |Q|^2 at 2^52: acc + (mid >> 31)
    const int64_t n = combine<0, 31>(mad(qr.h, qr.h, mad(qi.h, qi.h, 0)), mad(qr.h, qr.l, mad(qi.h, qi.l, int64_t(1) << 30)));
    const Digits R = digits(recip_fix(n));   // 2^64 / |Q|^2
    gr = mul_fix<0>(qi, R);
    gi = mul_fix<0>(qr, R);
}

__host__ __device__ __forceinline__ int64_t diag_row(const FixPoint& t, Digits E)
{
    const int64_t s0 = (int64_t)(((uint64_t)(uint32_t)t.s0_hi << 32) | (uint32_t)t.s0_lo);
    return s0 + mul_fix<5>(Digits{t.x_h, t.x_l}, E);
}

// IEEE double to fixed point: v 2^sigma rounded to nearest, for |v| 2^sigma < 2^61.  Integer operations
// only (a conversion instruction occupies the FP64 pipe).
__host__ __device__ __forceinline__ int64_t double_to_fix(uint64_t bits, int sigma)
{
    const int e = (int)(bits >> 52) & 0x7ff;
    const uint64_t mant = ((bits & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0)) << 9;   // < 2^62
    int rs = 1084 - (e ? e : 1) - sigma;   // v = mant 2^-rs at this scale, rs >= 1
    rs = rs < 1 ? 1 : (rs > 63 ? 63 : rs);
    const int64_t u = (int64_t)((mant + (uint64_t(1) << (rs - 1))) >> rs);
    return (int64_t)bits < 0 ? -u : u;
}

// Fixed point to IEEE double bits: v 2^-sigma rounded to nearest, |v| < 2^63, result normal or zero.
__host__ __device__ __forceinline__ uint64_t fix_to_double(int64_t v, int sigma)
{
    const uint64_t u = v < 0 ? (uint64_t)0 - (uint64_t)v : (uint64_t)v;
    if (u == 0) return 0;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)u);
#else
    const int lz = __builtin_clzll(u);
#endif
    const uint64_t t = u << lz;                                      // leading one at bit 63
    const uint64_t m = (t >> 11) + ((t >> 10) & 1u);                  // 53 bits; a carry moves the exponent
    return ((uint64_t)(v < 0) << 63) | (((uint64_t)(1023 + 62 - lz - sigma) << 52) + m);
}

// v 2^k rounded, v = hi + lo a pair of doubles
inline int64_t pair_fix(double hi, double lo, int k) { return std::llrint(std::ldexp(hi, k)) + std::llrint(std::ldexp(lo, k)); }

// Fixed-point form of a class with spacing dx and time step dt (beta = dt / (4 dx^2)); s0_max, x_max,
// dv_max: bounds on |S0|, |X|, |dV| over the grid.
inline FixClass fix_class(int N, double dx, double dt, double s0_max, double x_max, double dv_max)
{
    FixClass f{};
    f.kv = dv_max > 0.0 && std::isfinite(dv_max) ? std::max(-40, (int)std::ceil(std::log2(dv_max))) : 0;
    f.v_scale = std::ldexp(1.0, f.kv - 61);
    const double beta = dt / (4.0 * dx * dx);
    // beta <= 0.35: gamma at 2^64 keeps its digit products in 63 bits; beta > 0.0715: Q < 16.  N: the sum
    // of (2j - N + 1) x low digit over a segment stays in 64 bits, and the rounding of one unit per
    // point, spread over N points, below double's (measured to 32768)
    if (!(beta >= 0.0715 && beta <= 0.35) || N > 32768) return f;
    if (!(s0_max < 15.0) || !std::isfinite(x_max) || !(x_max > 0.0) || !std::isfinite(dv_max)) return f;
    // 1/beta = 4 dx^2 / dt as a pair of doubles: its own rounding would act as a systematic error of
    // every step
    const double p = 4.0 * dx * dx, pl = 4.0 * std::fma(dx, dx, -dx * dx);
    const double ib = p / dt, ib_lo = (std::fma(-ib, dt, p) + pl) / dt;
    f.top = beta <= 0.25 ? 61 : 60;
    f.E_lim = 0.999 * (15.0 - s0_max) / x_max;   // |gamma| < 1 joins Q's components
    f.xk = (int)std::ceil(std::log2(x_max));
    if (std::abs(f.xk) > 60 || f.kv > 60) return f;
    f.inv_b = pair_fix(ib, ib_lo, 58);
    f.ci = (int)std::lrint(2.0 * ib);
    f.cf = digits(pair_fix(2.0 * ib - f.ci, 2.0 * ib_lo, 63) * 2);
    f.e_scale = std::ldexp(1.0, 56 + f.xk);       // X E: 2^(61 - xk) 2^(56 + xk) 2^-59 = 2^58
    f.ok = 1;
    return f;
}

// Table entries of point j: S0 = 2 + 2 dx^2 V (V its only rounded part), X = (2j - N + 1) dx^3 with
// dx^3 as a pair of doubles; dV and the mask m.
__host__ __device__ inline FixPoint fix_point(const FixClass& f, int j, int N, double dx, double V)
{
    const int64_t s0 = (int64_t(1) << 59) + llrint(ldexp(2.0 * dx * dx * V, 58));
    const double d2 = dx * dx, d2l = fma(dx, dx, -d2);
    const double d3 = d2 * dx, d3l = fma(d2, dx, -d3) + d2l * dx;
    const double w = 2.0 * j - (N - 1.0);
    const double x = w * d3, xl = fma(w, d3, -x) + w * d3l;
    const Digits X = digits(llrint(ldexp(x, 61 - f.xk)) + llrint(ldexp(xl, 61 - f.xk)));
    return FixPoint{(int32_t)(uint32_t)(uint64_t)s0, (int32_t)(uint32_t)((uint64_t)s0 >> 32), X.l, X.h};
}
__host__ __device__ inline FixObs fix_obs(const FixClass& f, double dV, double m)
{
    const Digits v = digits(llrint(ldexp(dV, 61 - f.kv))), q = digits(llrint(ldexp(m, 61)));
    return FixObs{v.l, v.h, q.l, q.h};
}

}  // namespace tdse
