// Fixed-point split fluxes of the FP64 form: one stencil member's flux
// difference G(q~_i) - G(q~_0) in 64-bit integers (IMAD.WIDE, shifts and adds).
//
// Why: an FP64 instruction holds its SM for 16 cycles (2 lanes per cycle and
// SM, measured; FP32 and logic 128, 32 x 32 -> 64 multiply-add 41-64), so the
// FP64 split fluxes left 90 % of the issue slots empty while the FP64 pipe was
// full. A 64 x 64 product keeping the high word costs three wide multiply-adds
// and two adds, 3-4 cycles instead of 16, and keeps 60 bits where a double
// keeps 53. The result is rounded to a double once per component. The flux
// launch went from 178 to 50 FP64 warp instructions per edge and from 6.82 to
// 2.70 ms at 2.5 million points (second order, RK4), its error against multiple
// precision is 2-8 times below that of the FP64 chain.
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
// Taken when fix_state says so: beta in [2^-40, 2^40), S_t^2 + S_n^2 < 15.875
// with each component of sqrt(beta) (u, v) below 3.9375 (Mach 4.7), |q1| < 32,
// i.e. every state such flows meet; the FP64 form takes the others. The same code compiles on the host, where it is tested against
// multiple precision.
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
    int64_t c0, c1, c3;    // rho r, rho r^2, rho r^3: c 2^e
    int e0, e1, e3;
};

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
    // powers of r: r^2 <= 2 in Q61, r^4 <= 4 in Q60, r^6 <= 8 in Q59, r^7 < 11.4 and r^8 <= 16 in Q58
    const FixOp r2 = fix_op(fix_sqr_s<3>(R));
    const FixOp r4 = fix_op(fix_sqr_s<2>(r2));
    const FixOp r6 = fix_op(fix_mul_s<2>(r4, r2));
    const FixOp r7 = fix_op(fix_mul_s<2>(r6, R));
    const FixOp r8 = fix_op(fix_sqr_s<2>(r4));
    s.c0 = fix_mul_s<1>(M, r6);                                  // Q58, below 2^62 like the others
    s.c1 = fix_mul_s<1>(M, r7);                                  // Q57
    s.c3 = fix_mul_s<1>(M, r8);                                  // Q57
    s.e0 = n - 6 * k - 58;
    s.e1 = n - 7 * k - 57;
    s.e3 = n - 8 * k - 57;
    return ok;
}

// two factors c 2^e, both below 2^62, brought to one exponent (returned), the larger in [2^61, 2^62)
LSKUM_FIX_FN int fix_align(int64_t &ci, int ei, int64_t &c0, int e0)
{
    const int d = ei - e0;
    c0 >>= fix_max(fix_min(d, 63), 0);
    ci >>= fix_max(fix_min(-d, 63), 0);
    const int lz = fix_clz((uint32_t)((uint64_t)(ci | c0) >> 32)) - 2;
    ci <<= lz;
    c0 <<= lz;
    return fix_max(ei, e0) - lz;
}

// the bounded parts of one state's split flux with z = sgn S_d, So the
// transverse S: P in Q61, Phi/2 + z P in Q58, So P in Q58, H P - E/4 in Q57
LSKUM_FIX_FN void fix_parts(int64_t Sd, int64_t sgn, int64_t So, int64_t H, int64_t F[4])
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
    const int64_t E = e0 + (fix_mul(fix_op(e1), uo) >> 11);   // exp(-z^2)/(2 sqrt(pi)), Q62
    const int64_t z = fix_flip(Sd, sgn);                      // Q61
    const int64_t Phi = (1ll << 61) + fix_flip(T, z >> 63);   // Q62
    const FixOp zo = fix_op(z);
    const int64_t P = (E >> 1) + fix_shl(fix_mul(zo, fix_op(Phi)), 2);
    const FixOp Po = fix_op(P);
    F[0] = P;
    F[1] = (Phi >> 5) + fix_mul(zo, Po);
    F[2] = fix_mul(fix_op(So), Po);
    F[3] = fix_mul_s<1>(fix_op(H), Po) - (E >> 7);
}

// An edge's two states with their factors at common exponents
struct FixEdge {
    FixOp c0i, c1i, c3i, c00, c10, c30;
    int e0, e1, e3;
};
LSKUM_FIX_FN void fix_edge(const FixState &si, const FixState &s0, FixEdge &g)
{
    int64_t a = si.c0, b = s0.c0;
    g.e0 = fix_align(a, si.e0, b, s0.e0) + 2;
    g.c0i = fix_op(a);
    g.c00 = fix_op(b);
    a = si.c1, b = s0.c1;
    g.e1 = fix_align(a, si.e1, b, s0.e1) + 4;
    g.c1i = fix_op(a);
    g.c10 = fix_op(b);
    a = si.c3, b = s0.c3;
    g.e3 = fix_align(a, si.e3, b, s0.e3) + 5;
    g.c3i = fix_op(a);
    g.c30 = fix_op(b);
}

// G(q~_i) - G(q~_0) of one direction without the factors sgn of components
// 0, 2 and 3: [mass, d-momentum, o-momentum, energy]. sgn = 0 for G+, -1 for G-.
LSKUM_FIX_FN void fix_flux_difference(const FixEdge &g, const FixState &si, const FixState &s0, bool along_t,
                                      int64_t sgn, double dG[4])
{
    int64_t Fi[4], F0[4];
    fix_parts(along_t ? si.St : si.Sn, sgn, along_t ? si.Sn : si.St, si.H, Fi);
    fix_parts(along_t ? s0.St : s0.Sn, sgn, along_t ? s0.Sn : s0.St, s0.H, F0);
    // c < 2^62 and F[0] < 2^63, |F[1..3]| < 2^62.4: one, two more bits of the products fit
    dG[0] = fix_to_double(fix_mul_s<1>(g.c0i, fix_op(Fi[0])) - fix_mul_s<1>(g.c00, fix_op(F0[0])), g.e0);
    dG[1] = fix_to_double(fix_mul_s<2>(g.c1i, fix_op(Fi[1])) - fix_mul_s<2>(g.c10, fix_op(F0[1])), g.e1);
    dG[2] = fix_to_double(fix_mul_s<2>(g.c1i, fix_op(Fi[2])) - fix_mul_s<2>(g.c10, fix_op(F0[2])), g.e1);
    dG[3] = fix_to_double(fix_mul_s<2>(g.c3i, fix_op(Fi[3])) - fix_mul_s<2>(g.c30, fix_op(F0[3])), g.e3);
}

}  // namespace lskum
