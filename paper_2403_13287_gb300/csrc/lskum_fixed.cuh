// Fixed-point split fluxes of the FP64 form: one stencil member's flux
// difference G(q~_i) - G(q~_0) in 64-bit integers (IMAD.WIDE, shifts and adds).
//
// Why: an FP64 instruction holds its SM for 16 cycles (2 lanes per cycle and
// SM, measured; FP32 and logic 128, 32 x 32 -> 64 multiply-add 41-64), so the
// FP64 split fluxes left 90 % of the issue slots empty while the FP64 pipe was
// full. A 64 x 64 product keeping the high word costs three wide multiply-adds
// and two adds, 3-4 cycles instead of 16, and keeps 60 bits of its format's range
// where a double keeps 53 of its own size. The result is rounded to a double once
// per component. The flux launch went from 178 to 45 FP64 instructions per edge and
// from 6.82 to 2.20 ms at 2.5 million points (second order, RK4), its error against
// multiple precision is 2-8 times below that of the FP64 chain (slow transverse
// momenta, where it would not be, are left to FP64: fix_slow).
//
// With r = beta^(-1/2), S_t = u.t sqrt(beta), S_n likewise, every flux is a
// bounded function of (S_t, S_n) times a power of r times rho. For a direction
// d (transverse direction o), sgn the split sign and z = sgn S_d:
//   Phi = (1 + erf z)/2, E = exp(-z^2)/(2 sqrt(pi)), P = z Phi + E,
//   G0 = sgn rho r P,  G1 = rho r^2 (Phi/2 + z P),  G2 = sgn rho r^2 S_o P,
//   G3 = sgn rho r^3 ((hc + (S_t^2 + S_n^2)/2) P - E/4),
//   rho = exp(q1 + S_t^2 + S_n^2) r^5            (gamma = 1.4)
// which is split_flux (lskum_device.cuh) divided through by the powers of r.
// Formats: Qn is a 64-bit signed integer holding value 2^n. The comments give
// the range that each n leaves room for. A product's high word drops less than
// 1.25 units of its Qn.
//
// Taken when fix_state says so: beta in [2^-80, 2^80), S_t^2 + S_n^2 < 15.875
// with each component of sqrt(beta) (u, v) below 3.9375 (Mach 4.7), |q1| < 32,
// i.e. every state such flows meet; the FP64 form takes the others. The same
// code compiles on the host, where it is tested against multiple precision.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define LSKUM_FIX_FN __device__ __forceinline__
#define LSKUM_FIX_TABLE static __device__ __align__(64) const
#else
#include <cmath>
#include <cstring>
#define LSKUM_FIX_FN static inline
#define LSKUM_FIX_TABLE static const
#endif

namespace lskum {

#include "fix_tables.h"

// --- words of a double, float seeds, leading zeros -------------------------
LSKUM_FIX_FN int64_t fix_bits(double x)
{
#ifdef __CUDACC__
    return __double_as_longlong(x);
#else
    int64_t b;
    memcpy(&b, &x, 8);
    return b;
#endif
}
LSKUM_FIX_FN double fix_double(int64_t b)
{
#ifdef __CUDACC__
    return __longlong_as_double(b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}
// round(2^21 / sqrt(b)) within a unit or so, b the float with these bits in [1/2, 2)
LSKUM_FIX_FN int32_t fix_rsqrt_seed(uint32_t bits)
{
#ifdef __CUDACC__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(bits)));
    return __float_as_int(y + 4.0f) & 0x7fffff;   // [4, 8) has a unit of 2^-21
#else
    float b;
    memcpy(&b, &bits, 4);
    const float y = 1.0f / sqrtf(b) + 4.0f;
    int32_t v;
    memcpy(&v, &y, 4);
    return v & 0x7fffff;
#endif
}
LSKUM_FIX_FN int fix_clz(uint32_t x)   // x != 0
{
#ifdef __CUDACC__
    return __clz((int)x);
#else
    return __builtin_clz(x);
#endif
}
LSKUM_FIX_FN int32_t fix_mulhi32(int32_t a, int32_t b)
{
#ifdef __CUDACC__
    return __mulhi(a, b);
#else
    return (int32_t)(((int64_t)a * b) >> 32);
#endif
}
LSKUM_FIX_FN int fix_min(int a, int b) { return a < b ? a : b; }
LSKUM_FIX_FN int fix_max(int a, int b) { return a > b ? a : b; }
LSKUM_FIX_FN int64_t fix_min64(int64_t a, int64_t b) { return a < b ? a : b; }
LSKUM_FIX_FN int64_t fix_max64(int64_t a, int64_t b) { return a > b ? a : b; }
LSKUM_FIX_FN int64_t fix_shl(int64_t v, int s) { return (int64_t)((uint64_t)v << s); }

// --- products ---------------------------------------------------------------
// a = hi 2^32 + lo with lo signed, so that all partial products are signed
// 32 x 32 -> 64 multiply-adds. a must stay below 2^63 - 2^31 (hi is rounded
// up with lo), as every operand here does by its format.
struct FixOp {
    int32_t hi, lo;
};
LSKUM_FIX_FN FixOp fix_op(int64_t a)
{
    const int32_t lo = (int32_t)a;
    return FixOp{(int32_t)(a >> 32) + (int32_t)((uint32_t)lo >> 31), lo};
}
LSKUM_FIX_FN int64_t fix_value(FixOp a) { return fix_shl((int64_t)a.hi, 32) + a.lo; }
// a b 2^-64 within (-1.25, 0.25] (the low x low product is left out)
LSKUM_FIX_FN int64_t fix_mul(FixOp a, FixOp b)
{
    int64_t m = (int64_t)a.hi * b.lo;
    m += (int64_t)a.lo * b.hi;
    return (int64_t)a.hi * b.hi + (m >> 32);
}
// a b 2^(S-64), S small enough for the result's range
template <int S>
LSKUM_FIX_FN int64_t fix_mul_s(FixOp a, FixOp b)
{
    int64_t m = (int64_t)a.hi * b.lo;
    m += (int64_t)a.lo * b.hi;
    return fix_shl((int64_t)a.hi * b.hi, S) + (m >> (32 - S));
}
// a^2 2^(S-64)
template <int S>
LSKUM_FIX_FN int64_t fix_sqr_s(FixOp a)
{
    return fix_shl((int64_t)a.hi * a.hi, S) + (((int64_t)a.hi * a.lo) >> (31 - S));
}
// v with the sign flipped where m = -1 (unchanged where m = 0)
LSKUM_FIX_FN int64_t fix_flip(int64_t v, int64_t m) { return (v ^ m) - m; }

// v 2^e, rounded to nearest; e such that the result is a normal number
LSKUM_FIX_FN double fix_to_double(int64_t v, int e)
{
    const int64_t s = v >> 63;
    uint64_t a = (uint64_t)fix_flip(v, s);
    if (a == 0) return 0.0;
    if ((a >> 32) == 0) {
        a <<= 32;
        e -= 32;
    }
    const int lz = fix_clz((uint32_t)(a >> 32));
    a <<= lz;                                   // top bit 63: the value is 1.xx 2^(63 - lz + e)
    const uint64_t r = (a >> 11) + ((a >> 10) & 1u);   // 53 bits; a carry moves into the exponent
    return fix_double((int64_t)((r + ((uint64_t)(1023 + 62 - lz + e) << 52)) | ((uint64_t)s & 0x8000000000000000ull)));
}

// --- one state ----------------------------------------------------------------
struct FixState {
    int64_t St, Sn;        // Q61, |.| < 4
    int64_t H;             // Q59, hc + (St^2 + Sn^2)/2 < 9.7
    int64_t c0, c1, c3;    // rho r, rho r^2, rho r^3: c 2^e, e from n and k (fix_e0 ...)
    int64_t r;             // r 2^k in Q61, (0.7, 1.42)
    int n, k;              // exp(q1 + s2) = M 2^n, beta = b 4^k
};
LSKUM_FIX_FN int fix_e0(int n, int k) { return n - 6 * k - 58; }
LSKUM_FIX_FN int fix_e1(int n, int k) { return n - 7 * k - 57; }
LSKUM_FIX_FN int fix_e3(int n, int k) { return n - 8 * k - 57; }

// the double x times r/2 (R = r 2^61 in (0.7, 1.42), times 2^-k) as Q61; false
// from 3.9375 on
LSKUM_FIX_FN bool fix_scaled(double x, FixOp R, int k, int64_t &y)
{
    const int64_t b = fix_bits(x);
    const int e = (int)(b >> 52) & 0x7ff;
    const int64_t m = ((b & 0xfffffffffffffll) | 0x10000000000000ll) << 9;   // 1.xx in Q61
    const int64_t p = fix_mul(fix_op(m), R);                                 // Q58
    const int sh = e - 1021 - k, up = fix_max(fix_min(sh, 5), 0);
    const bool ok = sh <= 5 && (int32_t)(p >> 32) < (0x7e000000 >> up);
    const int64_t v = sh >= 0 ? fix_shl(p, up) : p >> fix_min(-sh, 63);
    y = e ? fix_flip(v, b >> 63) : 0;
    return ok;
}

// 2^62 for 1: a unit normal's component
LSKUM_FIX_FN int64_t fix_unit(double x)
{
#ifdef __CUDACC__
    return __double2ll_rn(x * 0x1p62);
#else
    return (int64_t)llrint(ldexp(x, 62));
#endif
}

// exp(x) = M 2^n, x in Q57 (|x| < 48), M in Q62, in (0.9999, 2 - 2^-13)
LSKUM_FIX_FN int64_t fix_exp(int64_t x, int &n)
{
    const int64_t y = fix_mul(fix_op(x), fix_op(LSKUM_FIX_LOG2E));   // log2, Q55
    const int64_t yr = y + (1ll << 42);
    n = (int)(yr >> 55);
    const int64_t T = kFixExp2[(int)(yr >> 43) & 4095];          // Q62
    const int64_t u = fix_shl(y, 21) >> 1;                       // Q62: 2 x the remainder in 1/4096, [-1, 1)
    const int32_t uh = (int32_t)(u >> 31);                       // Q31
    const int32_t t2 = LSKUM_FIX_A2 + fix_mulhi32(LSKUM_FIX_A3, uh);              // Q58
    const int64_t t1 = LSKUM_FIX_A1 + (((int64_t)t2 * uh) >> 14);                 // Q75
    const int64_t v = fix_mul(fix_op(t1), fix_op(u));                             // Q73
    return T + (fix_mul(fix_op(T), fix_op(v)) >> 9);
}

// The state q in the frame t = (ny, -nx), n = (nx, ny) (nx, ny in Q62); false
// if it lies outside the ranges of the formats
LSKUM_FIX_FN bool fix_state(const double q[4], FixOp nx, FixOp ny, FixState &s)
{
    // beta = -q4/2 = b 4^k, b in [1/2, 2): Q53 from q4's mantissa
    const int64_t b3 = fix_bits(q[3]);
    const int p = (int)((uint64_t)b3 >> 52) - 0x800 - 1024;
    bool ok = (unsigned)(p + 80) < 160u;        // negative, and |k| <= 40
    const int odd = p & 1, k = (p + 1) >> 1;
    const uint64_t b = (uint64_t)((b3 & 0xfffffffffffffll) | 0x10000000000000ll) << (1 - odd);
    // r = b^(-1/2): a seed Y 2^-21, then e = 1 - b Y^2 (exact to 2^-63) and
    // r = Y (1 + e/2 + 3 e^2/8), |e| < 2^-20
    const int32_t Y = fix_rsqrt_seed(((uint32_t)(b3 >> 29) & 0x7fffffu) | (uint32_t)(127 - odd) << 23);
    const uint64_t w = (uint64_t)(uint32_t)Y * (uint32_t)Y;
    uint64_t t = ((uint64_t)(uint32_t)b * (uint32_t)w) >> 32;
    t += (uint64_t)(uint32_t)(b >> 32) * (uint32_t)w;
    t += (uint64_t)(uint32_t)b * (uint32_t)(w >> 32);
    t += (uint64_t)((uint32_t)(b >> 32) * (uint32_t)(w >> 32)) << 32;
    const int64_t e = (int64_t)(0x8000000000000000ull - t);   // Q63
    const int32_t eh = (int32_t)(e >> 12);                      // Q51
    const int64_t c = (e >> 2) + ((3 * (int64_t)fix_mulhi32(eh, eh)) >> 11);   // Q62
    const int64_t r = ((int64_t)Y << 40) + (((int64_t)Y * c) >> 22);           // Q61
    const FixOp R = fix_op(r);
    // sqrt(beta) u = (q2, q3) r/2, turned into the frame
    int64_t y2, y3;
    ok &= fix_scaled(q[1], R, k, y2);
    ok &= fix_scaled(q[2], R, k, y3);
    const FixOp o2 = fix_op(y2), o3 = fix_op(y3);
    const int64_t St = fix_mul(o2, ny) - fix_mul(o3, nx);      // Q59, |.| < 8
    const int64_t Sn = fix_mul(o2, nx) + fix_mul(o3, ny);
    const int64_t s2 = fix_sqr_s<3>(fix_op(St)) + fix_sqr_s<3>(fix_op(Sn));   // Q57
    ok &= (uint32_t)(s2 >> 32) < 0x1fc00000u;                   // < 15.875
    s.St = fix_shl(St, 2);
    s.Sn = fix_shl(Sn, 2);
    s.H = (7ll << 57) + (s2 << 1);                              // hc = 1.75
    // rho r^-5 = exp(x), x = q1 + s2 in Q57, |q1| < 32
    const int64_t b1 = fix_bits(q[0]);
    const int e1 = (int)(b1 >> 52) & 0x7ff;
    ok &= e1 <= 1027;
    int64_t x = (((b1 & 0xfffffffffffffll) | 0x10000000000000ll) << 10) >> fix_max(fix_min(1028 - e1, 63), 0);
    x = fix_flip(x, b1 >> 63) + s2;
    int n;
    const FixOp M = fix_op(fix_exp(x, n));
    // r^2 <= 2 in Q61, r^4 <= 4 in Q60, r^6 <= 8 in Q59; the factors below 16, 22.7 and 32
    const FixOp r2 = fix_op(fix_sqr_s<3>(R));
    const FixOp r4 = fix_op(fix_sqr_s<2>(r2));
    s.c0 = fix_mul_s<1>(M, fix_op(fix_mul_s<2>(r4, r2)));        // Q58, below 2^62 like the others
    s.c1 = fix_mul_s<2>(fix_op(s.c0), R);                        // Q57
    s.c3 = fix_mul_s<3>(fix_op(s.c1), R);                        // Q57
    s.r = r;
    s.n = n;
    s.k = k;
    return ok;
}

// |S| below 2^-7, S in Q61. The formats leave S, and with it a transverse momentum
// flux, 2^-57.6 of the flux's scale rho r^2 (rms, measured); products in FP64
// carry about 2^-52.5 |S_o| instead, less from here on, which counts where one
// direction's weights are far above the other's (slow gas in a thin stencil).
LSKUM_FIX_FN bool fix_slow(int64_t S) { return (uint32_t)((int32_t)(S >> 32) + (1 << 22)) < (1u << 23); }

// c 2^e, c below 2^62, against another factor's exponent eo: c at the larger of
// the two (es)
LSKUM_FIX_FN int64_t fix_align_half(int64_t c, int e, int eo, int &es)
{
    es = fix_max(e, eo);
    return c >> fix_min(es - e, 63);
}
// the left shift that takes the larger of two such factors (c, and one with
// high word hi) into [2^61, 2^62)
LSKUM_FIX_FN int fix_top(int64_t c, uint32_t hi) { return fix_clz((uint32_t)((uint64_t)c >> 32) | hi) - 2; }

// Phi (Q62), E (Q62) and P (Q61) of z = sgn S_d, returned with z (Q61) as an operand
LSKUM_FIX_FN FixOp fix_phi_e(int64_t Sd, int64_t sgn, int64_t &Phi, int64_t &E, int64_t &P)
{
    const int64_t a = fix_flip(Sd, Sd >> 63);
    const int kr = (int)((a + (1ll << 49)) >> 50);
    const int64_t u = fix_shl(a, 14) >> 1;   // Q62: 2^12 (|z| - s_k), [-1, 1)
    const int32_t uh = (int32_t)(u >> 31);   // Q31
    const FixOp uo = fix_op(u);
#ifdef __CUDACC__
    int64_t t0, t1, e0, e1;
    int32_t t2, t3, t4, e2, e3, e4;
    {
        const longlong2 *row = reinterpret_cast<const longlong2 *>(kFixErf + kr);
        const longlong2 w0 = __ldg(row), w1 = __ldg(row + 1);
        const int4 w2 = __ldg(reinterpret_cast<const int4 *>(row + 2));
        const int2 w3 = __ldg(reinterpret_cast<const int2 *>(row + 3));
        t0 = w0.x; t1 = w0.y; e0 = w1.x; e1 = w1.y;
        t2 = w2.x; t3 = w2.y; t4 = w2.z; e2 = w2.w; e3 = w3.x; e4 = w3.y;
    }
#else
    const FixRow &row = kFixErf[kr];
    int64_t t0 = row.t0, t1 = row.t1, e0 = row.e0, e1 = row.e1;
    int32_t t2 = row.t2, t3 = row.t3, t4 = row.t4, e2 = row.e2, e3 = row.e3, e4 = row.e4;
#endif
    t3 += fix_mulhi32(t4, uh);
    e3 += fix_mulhi32(e4, uh);
    t2 += fix_mulhi32(t3, uh);
    e2 += fix_mulhi32(e3, uh);
    t1 += ((int64_t)t2 * uh) >> 12;
    e1 += ((int64_t)e2 * uh) >> 12;
    const int64_t T = t0 + (fix_mul(fix_op(t1), uo) >> 11);   // erf|z|/2, Q62
    E = e0 + (fix_mul(fix_op(e1), uo) >> 11);                 // exp(-z^2)/(2 sqrt(pi)), Q62
    const int64_t z = fix_flip(Sd, sgn);                      // Q61
    Phi = (1ll << 61) + fix_flip(T, z >> 63);                 // Q62
    const FixOp zo = fix_op(z);
    P = (E >> 1) + fix_shl(fix_mul(zo, fix_op(Phi)), 2);
    return zo;
}

// the bounded parts of one state's split flux with z = sgn S_d, So the
// transverse S: P in Q61, Phi/2 + z P in Q58, So P in Q58, H P - E/4 in Q57
LSKUM_FIX_FN void fix_parts(int64_t Sd, int64_t sgn, int64_t So, int64_t H, int64_t F[4])
{
    int64_t Phi, E, P;
    const FixOp zo = fix_phi_e(Sd, sgn, Phi, E, P);
    const FixOp Po = fix_op(P);
    F[0] = P;
    F[1] = (Phi >> 5) + fix_mul(zo, Po);
    F[2] = fix_mul(fix_op(So), Po);
    F[3] = fix_mul_s<1>(fix_op(H), Po) - (E >> 7);
}

// the parts times the state's (shifted) factors: c < 2^62 and F[0] < 2^63,
// |F[1..3]| < 2^62.4, so one, two more bits of the products fit
LSKUM_FIX_FN void fix_scale(FixOp c0, FixOp c1, FixOp c3, int64_t F[4])
{
    F[0] = fix_mul_s<1>(c0, fix_op(F[0]));
    F[1] = fix_mul_s<2>(c1, fix_op(F[1]));
    F[2] = fix_mul_s<2>(c1, fix_op(F[2]));
    F[3] = fix_mul_s<2>(c3, fix_op(F[3]));
}

// --- the q-derivative passes' parts ------------------------------------------
// Two doubles, each with an exponent of its own: x = X 2^(ex-1084), 2^61 <= |X| <
// 2^62 the op's value; a zero (or subnormal) component is X = 0 with an exponent
// below all others, so that the other one alone sets a product's scale. (One
// exponent for both, the larger one's, was 60 bits of the vector's size but not of
// a small component: a stencil stretched A : 1 lost log2(A) bits of h . g where the
// gradient runs across it, 8.8e-14 of |h.x g.x| + |h.y g.y| at 1000 : 1.)
constexpr int kFixZeroExponent = -8192;
struct FixPair {
    FixOp x, y;
    int ex, ey;   // biased exponents (0x7ff: not finite)
};
template <int Q>
LSKUM_FIX_FN int64_t fix_mantissa(int64_t b)   // 1.xx in Q<Q>, signed
{
    return fix_flip(((b & 0xfffffffffffffll) | 0x10000000000000ll) << (Q - 52), b >> 63);
}
LSKUM_FIX_FN FixPair fix_pair(double x, double y)
{
    const int64_t bx = fix_bits(x), by = fix_bits(y);
    const int ex = (int)(bx >> 52) & 0x7ff, ey = (int)(by >> 52) & 0x7ff;
    FixPair p;
    p.ex = ex ? ex : kFixZeroExponent;
    p.ey = ey ? ey : kFixZeroExponent;
    p.x = fix_op(ex ? fix_mantissa<61>(bx) : 0);
    p.y = fix_op(ey ? fix_mantissa<61>(by) : 0);
    return p;
}
// both components zero (or subnormal)
LSKUM_FIX_FN bool fix_pair_zero(const FixPair &p) { return fix_max(p.ex, p.ey) < 0; }
// A pair without loss in two words: a component's 53 bits leave the word's low 9
// to its exponent, e - 639 (1..511; 0 beside a zero). Both words 0 where the pair
// does not fit: the larger component outside 2^-127..2^128, the smaller one not
// zero and below 2^-383.
LSKUM_FIX_FN void fix_pack_pair(double x, double y, int64_t &wx, int64_t &wy)
{
    const FixPair p = fix_pair(x, y);
    const int e = fix_max(p.ex, p.ey) - 895;
    const int cx = p.ex < 0 ? 0 : p.ex - 639, cy = p.ey < 0 ? 0 : p.ey - 639;
    const bool fits = e >= 1 && e <= 255 && (cx > 0 || p.ex < 0) && (cy > 0 || p.ey < 0);
    wx = fits ? fix_value(p.x) | cx : 0;
    wy = fits ? fix_value(p.y) | cy : 0;
}
LSKUM_FIX_FN FixPair fix_unpack_pair(int64_t wx, int64_t wy)
{
    FixPair p;
    const int cx = (int)wx & 511, cy = (int)wy & 511;
    p.ex = cx ? cx + 639 : kFixZeroExponent;
    p.ey = cy ? cy + 639 : kFixZeroExponent;
    p.x = fix_op(wx & ~511ll);
    p.y = fix_op(wy & ~511ll);
    return p;
}
// the exponents of h and g for which fix_dot's result is a normal number: away
// from both ends by the 60 bits that a cancelling sum may lose
LSKUM_FIX_FN bool fix_dot_in_range(const FixPair &h, const FixPair &g)
{
    const int e = fix_max(h.ex + g.ex, h.ey + g.ey);
    return (unsigned)(e - 1100) < 1900u && fix_max(fix_max(h.ex, h.ey), fix_max(g.ex, g.ey)) < 0x7ff;
}
// h.x g.x + h.y g.y, rounded once: each product within 1.25 units of 2^-58 of
// itself, the smaller one shifted to the larger one's exponent (a unit more), so
// 2^-56 of the larger product before the rounding
LSKUM_FIX_FN double fix_dot(const FixPair &h, const FixPair &g)
{
    const int a = h.ex + g.ex, b = h.ey + g.ey, e = fix_max(a, b);
    const int64_t c = (fix_mul(h.x, g.x) >> fix_min(e - a, 63)) + (fix_mul(h.y, g.y) >> fix_min(e - b, 63));
    return fix_to_double(c, e - 2104);
}

// round(2^22 / f) within a unit or so, f the float with these bits in [1, 2)
LSKUM_FIX_FN int32_t fix_rcp_seed(uint32_t bits)
{
#ifdef __CUDACC__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(bits)));
    return __float_as_int(y + 2.0f) - 0x40000000;   // [2, 4) has a unit of 2^-22
#else
    float f;
    memcpy(&f, &bits, 4);
    const float y = 1.0f / f + 2.0f;
    int32_t v;
    memcpy(&v, &y, 4);
    return v - 0x40000000;
#endif
}

// 1/m in Q62 (in (0.5, 1]) of m in Q61, 2^61 <= m < 2^62
LSKUM_FIX_FN int64_t fix_rcp(int64_t m)
{
    const int32_t Y = fix_rcp_seed(0x3f800000u | ((uint32_t)(m >> 38) & 0x7fffffu));   // Q22
    // e = 1 - m Y exactly to 2^-63, r = Y (1 + e + e^2), |e| < 2^-21
    const uint64_t t = (((uint64_t)(uint32_t)m * (uint32_t)Y) >> 20) + (((uint64_t)(uint32_t)(m >> 32) * (uint32_t)Y) << 12);
    const int64_t e = (int64_t)(0x8000000000000000ull - t);       // Q63
    const int32_t eh = (int32_t)(e >> 11);                         // Q52
    const int64_t c = (e >> 1) + (fix_mulhi32(eh, eh) >> 10);      // Q62
    return ((int64_t)Y << 40) + (((int64_t)Y * c) >> 22);
}

// Venkatakrishnan's f(x, d) = N / M, N = x (x + 2d) + eps2,
// M = x (x + d) + 2 d^2 + eps2, for 0 <= x < 2d (so that f <= 1) and exponents
// within fix_phi_in_range. Everything is scaled by the power of two that takes
// the larger of d and sqrt(eps2) to order 1; N keeps an exponent of its own, so
// that a small f keeps its relative precision (2^-54 before the final rounding).
LSKUM_FIX_FN bool fix_phi_in_range(double d, double eps2)
{
    const int ed = (int)(fix_bits(d) >> 52), ee = (int)(fix_bits(eps2) >> 52);
    return (unsigned)(ed - 300) < 1400u && (unsigned)ee < 1700u;
}
LSKUM_FIX_FN double fix_phi(double x, double d, double eps2)
{
    const int64_t bx = fix_bits(x), bd = fix_bits(d), be = fix_bits(eps2);
    const int ex = (int)(bx >> 52), ed = (int)(bd >> 52), ee = (int)(be >> 52);
    const int p = fix_max(ed, 1023 + ((ee - 1022) >> 1));          // biased exponent of the scale
    const int64_t X = ex ? fix_mantissa<60>(bx) : 0;             // x = X 2^(ex - p), 1.xx in Q60
    const int ux = ex ? ex - p : -4096, ue = ee ? ee + 1023 - 2 * p : -4096;   // ux <= 1, ue <= 0
    const int64_t xs = X >> fix_min(1 - ux, 63);                    // x < 4 in Q59
    const int64_t ds = fix_mantissa<60>(bd) >> fix_min(p - ed + 1, 63);            // d < 2 in Q59
    const int64_t E = ee ? fix_mantissa<57>(be) : 0;             // eps2 = E 2^ue, 1.xx in Q57
    const int64_t T = fix_mul_s<2>(fix_op(X), fix_op(xs + 2 * ds)); // x (x + 2d) = T 2^ux, T < 16 in Q57
    const int un = fix_max(ux, ue);
    const int64_t N = (T >> fix_min(un - ux, 63)) + (E >> fix_min(un - ue, 63));   // Q57, times 2^un
    // M < 34 in Q56, at least 1/4
    const int64_t M = fix_mul_s<2>(fix_op(xs), fix_op(xs + ds)) + fix_sqr_s<3>(fix_op(ds)) + (E >> fix_min(1 - ue, 63));
    const int lz = fix_clz((uint32_t)((uint64_t)M >> 32)) - 2;
    const int64_t f = fix_mul_s<2>(fix_op(N), fix_op(fix_rcp(M << lz)));   // N / (M 2^(lz - 61)), Q57
    return un < -900 ? 0.0 : fix_to_double(f, un + lz - 62);      // below 2^-890: 0
}

// a - b where sign and exponent agree (the difference is then exact), in range
// for fix_to_double
LSKUM_FIX_FN bool fix_same_binade(double a, double b)
{
    const int64_t ba = fix_bits(a), x = ba ^ fix_bits(b);
    return ((uint64_t)x >> 52) == 0 && (unsigned)(((int)(ba >> 52) & 0x7ff) - 100) < 1900u;
}
LSKUM_FIX_FN double fix_difference(double a, double b)
{
    const int64_t ba = fix_bits(a), bb = fix_bits(b);
    return fix_to_double(fix_flip((ba & 0xfffffffffffffll) - (bb & 0xfffffffffffffll), ba >> 63),
                         ((int)(ba >> 52) & 0x7ff) - 1075);
}

// --- q-variables of a state ------------------------------------------------
// positive and of an exponent for which the forms below stay normal
LSKUM_FIX_FN bool fix_moderate(double x) { return (uint64_t)fix_bits(x) - (700ull << 52) < (700ull << 52); }

// 1/x of a moderate x, within 2^-59 before the final rounding
LSKUM_FIX_FN double fix_reciprocal(double x)
{
    const int64_t b = fix_bits(x);
    return fix_to_double(fix_rcp(fix_mantissa<61>(b)), 1023 - 62 - (int)(b >> 52));
}

// 1/y and x/y of moderate x and y from one reciprocal, each within 2^-57 before its
// one rounding (x (1/y) in FP64 rounds twice: of q4 = -rho/p that made 1.22e-16 rms
// where the FP64 division's was 1.05e-16)
LSKUM_FIX_FN void fix_quotient(double x, double y, double &ry, double &xy)
{
    const int64_t bx = fix_bits(x), by = fix_bits(y);
    const int ex = (int)(bx >> 52), ey = (int)(by >> 52);
    const int64_t r = fix_rcp(fix_mantissa<61>(by));                              // Q62
    ry = fix_to_double(r, 1023 - 62 - ey);
    xy = fix_to_double(fix_mul_s<2>(fix_op(fix_mantissa<61>(bx)), fix_op(r)), ex - ey - 61);   // Q61, (0.5, 2)
}

// log2 of a positive normal x's mantissa in Q60, [0, 1)
LSKUM_FIX_FN int64_t fix_log2_mantissa(double x)
{
    const int64_t b = fix_bits(x);
    const int j = (int)(b >> 42) & 1023;
#ifdef __CUDACC__
    const int4 w = __ldg(reinterpret_cast<const int4 *>(kFixLog2 + j));
    const int64_t lc = (int64_t)(((uint64_t)(uint32_t)w.y << 32) | (uint32_t)w.x);
    const uint32_t r = (uint32_t)w.z;
#else
    const int64_t lc = kFixLog2[j].log2c;
    const uint32_t r = kFixLog2[j].r;
#endif
    // u = 2^11 (m r - 1) in Q62, |u| < 1.001: the 1's 2^73 is 0 modulo 2^64
    const uint64_t m = (uint64_t)((b & 0xfffffffffffffll) | 0x10000000000000ll);
    const int64_t u = (int64_t)((((uint64_t)(uint32_t)m * r) >> 11) + (((m >> 32) * r) << 21));
    const int32_t uh = (int32_t)(u >> 32);                                        // Q30
    const FixOp uo = fix_op(u);
    const int32_t t4 = LSKUM_FIX_LOG_C4 + fix_mulhi32(LSKUM_FIX_LOG_C5, uh);      // Q66
    const int32_t t3 = LSKUM_FIX_LOG_C3 + fix_mulhi32(t4, uh);                    // Q64
    const int64_t t2 = LSKUM_FIX_LOG_C2 + (((int64_t)t3 * uh) >> 10);             // Q84
    const int64_t t1 = LSKUM_FIX_LOG_C1 + (fix_mul(fix_op(t2), uo) >> 10);        // Q72
    return lc + (fix_mul(fix_op(t1), uo) >> 10);                                  // Q60
}

// ln(rho) + 2.5 ln(beta), beta = rho/(2p), of moderate rho and p, which is
// (7 log2 rho - 5 log2 p - 5) ln2/2: within 2^-54 before the final rounding
// while the bracket is below 117, beyond that to about a unit in the last place
LSKUM_FIX_FN double fix_log_state(double rho, double p)
{
    const int n = 7 * ((int)(fix_bits(rho) >> 52) - 1023) - 5 * ((int)(fix_bits(p) >> 52) - 1023) - 5;
    const int64_t f = 7 * fix_log2_mantissa(rho) - 5 * fix_log2_mantissa(p);      // Q60, (-5, 7)
    const bool small = n >= -110 && n <= 110;
    const int64_t l = (small ? fix_shl(n, 56) : 0) + (f >> 4);                    // the bracket in Q56, half of it in Q57
    const double v = fix_to_double(fix_mul(fix_op(l), fix_op(LSKUM_FIX_LN2)), -56);
    return small ? v : v + (double)n * 0.34657359027997264;
}

}  // namespace lskum
