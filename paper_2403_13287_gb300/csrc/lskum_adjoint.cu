// Vector-Jacobian product of the q-LSKUM residual (E10 with E11, E13-E15):
// U_bar = (dR/dU)^T R_bar and (x_bar, y_bar) = (dR/dx, dR/dy)^T R_bar, in
// FP64 or (mixed contexts, unlimited) FP32, for order 1 or 2.
//
// Reverse pass, every sum a gather (no atomics, bitwise reproducible):
//   flux      per point (owner of its edges): the transposed split-flux
//             Jacobians at both reconstructed states applied to the
//             cotangents (FP64: in the variables of the fixed-point fluxes,
//             k_adj_flux_pair, or through the regrouped split fluxes for
//             gamma != 1.4; FP32: forward-mode duals, 4 tangents), giving
//             cotangents of the owner's q~_0, of each neighbour's q~_i (kept
//             per edge) and of the sub-stencil weights;
//   gather    per point over its incoming edges (transpose CSR): the
//             neighbour-side cotangents;
//   limiter   (limiter_K > 0) back to the unlimited last iterate;
//   gradient  the K+1 least-squares passes of E15 in reverse (saved forward
//             iterates), each pass one kernel with an outgoing-edge loop
//             (owner terms, weight and offset cotangents) and an incoming-
//             edge loop (neighbour terms; FP64: in blocks of their own);
//   state     q_bar to U_bar through the E13 Jacobian;
//   geometry  once per product, and only if coordinate cotangents are asked
//             for: least-squares weight cotangents back to edge offsets
//             (a = M^-1 d with M = sum d d^T gives d_bar_k = b_k - B d_k,
//             b = M^-1 a_bar, B = sum (b a^T + a b^T)), then offsets to
//             points by one more gather.
#include <cub/cub.cuh>
#include <type_traits>

#include "lskum_adjoint.h"
#include "lskum_fixed.cuh"

namespace lskum {

namespace {

// ---------------------------------------------------------------------------
// forward-mode dual number with four tangents, over T (double, or float for
// the FP32 product)
// ---------------------------------------------------------------------------
template <class T>
struct D4T {
    T v, d[4];
};
using D4 = D4T<double>;

// elementary functions: in FP64 the forward kernels' own forms (the
// table-driven exp, and erf(S) with exp(-S^2) from one Taylor-table row),
// in FP32 the library's
[[maybe_unused]] __device__ __forceinline__ double m_exp(double x) { return exp_tab(x); }
__device__ __forceinline__ float m_exp(float x) { return expf(x); }
__device__ __forceinline__ double m_log(double x) { return log(x); }
__device__ __forceinline__ float m_log(float x) { return logf(x); }
__device__ __forceinline__ double m_sqrt(double x) { return sqrt(x); }
[[maybe_unused]] __device__ __forceinline__ float m_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double m_rsqrt(double x) { return rsqrt(x); }
__device__ __forceinline__ float m_rsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ void m_erf_gauss(double S, double &erfS, double &e) { erf_exp(S, erfS, e); }
__device__ __forceinline__ void m_erf_gauss(float S, float &erfS, float &e)
{
    erfS = erff(S);
    e = expf(-S * S);
}

template <class T>
__device__ __forceinline__ D4T<T> dconst(T v)
{
    D4T<T> r;
    r.v = v;
#pragma unroll
    for (int k = 0; k < 4; ++k) r.d[k] = T(0);
    return r;
}
template <class T>
__device__ __forceinline__ D4T<T> operator+(const D4T<T> &a, const D4T<T> &b)
{
    D4T<T> r;
    r.v = a.v + b.v;
#pragma unroll
    for (int k = 0; k < 4; ++k) r.d[k] = a.d[k] + b.d[k];
    return r;
}
template <class T>
__device__ __forceinline__ D4T<T> operator-(const D4T<T> &a, const D4T<T> &b)
{
    D4T<T> r;
    r.v = a.v - b.v;
#pragma unroll
    for (int k = 0; k < 4; ++k) r.d[k] = a.d[k] - b.d[k];
    return r;
}
template <class T>
__device__ __forceinline__ D4T<T> operator*(const D4T<T> &a, const D4T<T> &b)
{
    D4T<T> r;
    r.v = a.v * b.v;
#pragma unroll
    for (int k = 0; k < 4; ++k) r.d[k] = a.d[k] * b.v + a.v * b.d[k];
    return r;
}
template <class T>
__device__ __forceinline__ D4T<T> operator*(T s, const D4T<T> &a)
{
    D4T<T> r;
    r.v = s * a.v;
#pragma unroll
    for (int k = 0; k < 4; ++k) r.d[k] = s * a.d[k];
    return r;
}
template <class T>
__device__ __forceinline__ D4T<T> operator+(T s, const D4T<T> &a)
{
    D4T<T> r = a;
    r.v = s + a.v;
    return r;
}
// f(a) with f(a.v) = fv and f'(a.v) = df
template <class T>
__device__ __forceinline__ D4T<T> chain(const D4T<T> &a, T fv, T df)
{
    D4T<T> r;
    r.v = fv;
#pragma unroll
    for (int k = 0; k < 4; ++k) r.d[k] = df * a.d[k];
    return r;
}
template <class T>
__device__ __forceinline__ D4T<T> recip(const D4T<T> &a)
{
    const T r = T(1) / a.v;
    return chain(a, r, -r * r);
}
template <class T>
__device__ __forceinline__ D4T<T> dexp(const D4T<T> &a)
{
    const T e = m_exp(a.v);
    return chain(a, e, e);
}
template <class T>
__device__ __forceinline__ D4T<T> dlog(const D4T<T> &a)
{
    return chain(a, m_log(a.v), T(1) / a.v);
}
template <class T>
__device__ __forceinline__ D4T<T> dsqrt(const D4T<T> &a)
{
    const T s = m_sqrt(a.v);
    return chain(a, s, T(0.5) / s);
}

// The dual-number forms below serve the FP32 product; the FP64 product runs
// state_adjoint_rev (reverse mode through the forward kernels' regrouped
// split fluxes).
template <class T>
struct PrimDT {
    D4T<T> rho, u, v, p, sqb, rsb;
};

// inverse of E13 over duals: beta = -q4/2, u = -q2/q4, v = -q3/q4,
// rho = exp(q1 + beta |u|^2) beta^(-1/(gamma-1)), p = rho/(2 beta). From
// rsb = 1/sqrt(beta) and ib = 1/beta as the forward kernels form them:
// 1/q4 = -ib/2 (derivative -ib^2/4), sqrt(beta) = beta rsb (rsb/2),
// 1/sqrt(beta) (-rsb ib/2), and for gamma = 1.4 beta^-2.5 = rsb ib^2
// (-2.5 rsb ib^3) in place of exp(-2.5 ln beta)
template <class T>
__device__ __forceinline__ PrimDT<T> prim_d(const D4T<T> qt[4], T inv_gm1, bool g14)
{
    PrimDT<T> s;
    const D4T<T> beta = T(-0.5) * qt[3];
    const T rsb = m_rsqrt(beta.v), ib = rsb * rsb;
    const D4T<T> r = chain(qt[3], T(-0.5) * ib, T(-0.25) * ib * ib);
    s.u = T(-1) * (qt[1] * r);
    s.v = T(-1) * (qt[2] * r);
    s.sqb = chain(beta, beta.v * rsb, T(0.5) * rsb);
    s.rsb = chain(beta, rsb, T(-0.5) * rsb * ib);
    const D4T<T> ke = beta * (s.u * s.u + s.v * s.v);
    if (g14) {
        const T b25 = rsb * ib * ib;
        s.rho = dexp(qt[0] + ke) * chain(beta, b25, T(-2.5) * b25 * ib);
    } else {
        s.rho = dexp(qt[0] - inv_gm1 * dlog(beta) + ke);
    }
    s.p = T(-1) * (s.rho * r);
    return s;
}

// split flux along a direction over duals, in the paper's form
template <class T>
__device__ __forceinline__ void split_flux_d(T sgn, const PrimDT<T> &s, const D4T<T> &un, const D4T<T> &ut,
                                             T inv_gm1, D4T<T> G[4])
{
    const D4T<T> S = un * s.sqb;
    T erfv, e;
    m_erf_gauss(S.v, erfv, e);
    const D4T<T> erfS = chain(S, erfv, T(1.1283791670955126) * e);         // 2/sqrt(pi)
    const D4T<T> eS = chain(S, e, T(-2) * S.v * e);
    const D4T<T> A = T(0.5) * (T(1) + sgn * erfS);
    const D4T<T> B = T(0.28209479177387814) * (eS * s.rsb);                 // 1/(2 sqrt(pi))
    const D4T<T> rhoE = inv_gm1 * s.p + T(0.5) * (s.rho * (un * un + ut * ut));
    const D4T<T> m = un * A + sgn * B;
    G[0] = s.rho * m;
    G[1] = (s.p + s.rho * un * un) * A + sgn * (s.rho * un * B);
    G[2] = s.rho * ut * m;
    G[3] = (rhoE + s.p) * un * A + sgn * ((rhoE + T(0.5) * s.p) * B);
}

__device__ __forceinline__ void ld4(const double *a, int64_t p, double v[4])
{
    const double2 *a2 = reinterpret_cast<const double2 *>(a);
    const double2 lo = a2[2 * p], hi = a2[2 * p + 1];
    v[0] = lo.x; v[1] = lo.y; v[2] = hi.x; v[3] = hi.y;
}
__device__ __forceinline__ void st4(double *a, int64_t p, const double v[4])
{
    double2 *a2 = reinterpret_cast<double2 *>(a);
    a2[2 * p] = make_double2(v[0], v[1]);
    a2[2 * p + 1] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void ld8(const double *a, int64_t p, double v[8])
{
    ld4(a, 2 * p, v);
    ld4(a, 2 * p + 1, v + 4);
}
__device__ __forceinline__ void st8(double *a, int64_t p, const double v[8])
{
    st4(a, 2 * p, v);
    st4(a, 2 * p + 1, v + 4);
}
__device__ __forceinline__ void ld4(const float *a, int64_t p, float v[4])
{
    const float4 t = reinterpret_cast<const float4 *>(a)[p];
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void st4(float *a, int64_t p, const float v[4])
{
    reinterpret_cast<float4 *>(a)[p] = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void ld8(const float *a, int64_t p, float v[8])
{
    ld4(a, 2 * p, v);
    ld4(a, 2 * p + 1, v + 4);
}
__device__ __forceinline__ void st8(float *a, int64_t p, const float v[8])
{
    st4(a, 2 * p, v);
    st4(a, 2 * p + 1, v + 4);
}

// sub-stencil slots of an edge: x-sub (0 x+, 1 x-) and y-sub (2 y+, 3 y-), -1 if none
__device__ __forceinline__ int xsub(uint8_t m) { return (m & M_XPOS) ? 0 : ((m & M_XNEG) ? 1 : -1); }
__device__ __forceinline__ int ysub(uint8_t m) { return (m & M_YPOS) ? 2 : ((m & M_YNEG) ? 3 : -1); }
__device__ __forceinline__ bool sub_needed(uint8_t f, int k)
{
    return k >= 0 && (f == FLAG_INTERIOR || (f == FLAG_WALL && k != 2));
}

// cotangent of one reconstructed state: sum over the split fluxes it feeds,
// cs (frame order) against Gs and cn (frame order) against Gn, plus the
// flux values for the weight cotangents

template <class T>
__device__ __forceinline__ void state_adjoint(const T qt[4], T tx, T ty, T nx, T ny, bool use_s, T sg_s, bool use_n,
                                              T sg_n, const T cs[4], const T cn[4], T inv_gm1, bool g14, T qbar[4],
                                              T Gs[4], T Gn[4])
{
    D4T<T> q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        q[k] = dconst(qt[k]);
        q[k].d[k] = T(1);
    }
    const PrimDT<T> s = prim_d(q, inv_gm1, g14);
    const D4T<T> us = tx * s.u + ty * s.v;
    const D4T<T> un = nx * s.u + ny * s.v;
#pragma unroll
    for (int k = 0; k < 4; ++k) qbar[k] = T(0);
    if (use_s) {
        D4T<T> G[4];
        split_flux_d(sg_s, s, us, un, inv_gm1, G);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            Gs[c] = G[c].v;
#pragma unroll
            for (int k = 0; k < 4; ++k) qbar[k] += cs[c] * G[c].d[k];
        }
    }
    if (use_n) {
        D4T<T> G[4];
        split_flux_d(sg_n, s, un, us, inv_gm1, G);
        // Gn components are [mass, n-momentum, s-momentum, energy]
        const int fr[4] = {0, 2, 1, 3};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            Gn[fr[c]] = G[c].v;
#pragma unroll
            for (int k = 0; k < 4; ++k) qbar[k] += cn[fr[c]] * G[c].d[k];
        }
    }
}

// FP64 form of state_adjoint in reverse mode: the split fluxes in the forward
// kernels' regrouped form once, then their adjoint, so that
// q_bar = sum over the needed directions of (dG/dq~)^T c without forming the
// Jacobians. Primal, with (u_d, u_t) = (u.t, u.n) for the s direction and
// (u.n, u.t) for the n direction:
//   beta = -q4/2, r = beta^-1/2, hib = r^2/2 (= p/rho), u.t = (q2 tx + q3 ty) hib,
//   sqb = beta r, w2 = |u|^2, rho/2 = exp(q1 + beta w2)/2 beta^(-1/(gamma-1)),
//   h = (1/(gamma-1) + 1) hib + w2/2, qb = hib/2, rrc = (rho/2) r/sqrt(pi);
//   S = u_d sqb, fe = sgn erf S, Q = rho/2 (1 + fe), W = sgn rrc exp(-S^2),
//   G0 = u_d Q + W, G1 = u_d G0 + Q hib, G2 = u_t G0, G3 = h G0 - qb W.
__device__ __forceinline__ void state_adjoint_rev(const double qt[4], double tx, double ty, double nx, double ny,
                                                  bool use_s, double sg_s, bool use_n, double sg_n,
                                                  const double cs[4], const double cn[4], double inv_gm1, bool g14,
                                                  double qbar[4], double Gs[4], double Gn[4])
{
    const double beta = -0.5 * qt[3];
    const double rsb = m_rsqrt(beta), ib = rsb * rsb, hib = 0.5 * ib;
    const double qs = qt[1] * tx + qt[2] * ty, qn = qt[1] * nx + qt[2] * ny;
    const double us = qs * hib, un = qn * hib;
    const double sqb = beta * rsb;
    const double w2 = us * us + un * un;
    double hrho, fb = 1.0;   // fb = beta^-2.5 for gamma = 1.4
    if (g14) {
        fb = rsb * (ib * ib);
        hrho = exp_tab(qt[0] + beta * w2, -1) * fb;
    } else {
        hrho = exp_tab(qt[0] + beta * w2 - inv_gm1 * m_log(beta), -1);
    }
    const double h = (inv_gm1 + 1.0) * hib + 0.5 * w2;
    const double qb = 0.5 * hib;
    const double rrc = hrho * rsb * 0.5641895835477563;   // 1/sqrt(pi)
    double b_us = 0.0, b_un = 0.0, b_sqb = 0.0, b_hrho = 0.0, b_hib = 0.0, b_rrc = 0.0, b_h = 0.0, b_qb = 0.0;
    // one direction: primal G (in the direction's order) and its adjoint for cotangent c
    auto dir = [&](double ud, double ut, double sg, const double c[4], double G[4], double &b_ud, double &b_ut) {
        const double S = ud * sqb;
        double erfv, e;
        m_erf_gauss(S, erfv, e);
        const double fe = sg * erfv;
        const double Q = hrho + hrho * fe;
        const double W = sg * e * rrc;
        const double G0 = ud * Q + W;
        G[0] = G0;
        G[1] = ud * G0 + Q * hib;
        G[2] = ut * G0;
        G[3] = h * G0 - qb * W;
        const double bG0 = c[0] + c[1] * ud + c[2] * ut + c[3] * h;
        b_h += c[3] * G0;
        b_qb -= c[3] * W;
        b_ut += c[2] * G0;
        b_hib += c[1] * Q;
        const double bQ = c[1] * hib + bG0 * ud;
        const double bW = bG0 - c[3] * qb;
        b_ud += c[1] * G0 + bG0 * Q;
        b_rrc += bW * sg * e;
        b_hrho += bQ * (1.0 + fe);
        // fe = sgn erf S (erf' = 2/sqrt(pi) e), e = exp(-S^2) (e' = -2 S e)
        const double bS = (bQ * hrho * sg * 1.1283791670955126 - bW * sg * rrc * 2.0 * S) * e;
        b_ud += bS * sqb;
        b_sqb += bS * ud;
    };
    if (use_s) dir(us, un, sg_s, cs, Gs, b_us, b_un);
    if (use_n) {
        const double c[4] = {cn[0], cn[2], cn[1], cn[3]};   // Gn is [mass, n-momentum, s-momentum, energy]
        double G[4];
        dir(un, us, sg_n, c, G, b_un, b_us);
        Gn[0] = G[0];
        Gn[1] = G[2];
        Gn[2] = G[1];
        Gn[3] = G[3];
    }
    // per-state factors, in reverse
    b_hrho += b_rrc * rsb * 0.5641895835477563;
    double b_rsb = b_rrc * hrho * 0.5641895835477563;
    b_hib += 0.5 * b_qb + (inv_gm1 + 1.0) * b_h;
    double b_w2 = 0.5 * b_h;
    const double bx = b_hrho * hrho;   // d(rho/2)/dx = rho/2 for the exponent's argument x
    double b_beta = bx * w2;
    if (g14) b_beta += bx * (-2.5 * ib);   // beta^-2.5: relative derivative -2.5/beta
    else b_beta -= bx * inv_gm1 * ib;      // -ln(beta)/(gamma-1)
    b_w2 += bx * beta;
    b_us += 2.0 * us * b_w2;
    b_un += 2.0 * un * b_w2;
    b_beta += b_sqb * rsb;
    b_rsb += b_sqb * beta;
    const double b_qs = b_us * hib, b_qn = b_un * hib;
    b_hib += b_us * qs + b_un * qn;
    b_rsb += b_hib * rsb;                  // hib = rsb^2/2
    b_beta -= 0.5 * b_rsb * rsb * ib;      // rsb = beta^-1/2
    qbar[0] = bx;
    qbar[1] = b_qs * tx + b_qn * nx;
    qbar[2] = b_qs * ty + b_qn * ny;
    qbar[3] = -0.5 * b_beta;
}

// ---------------------------------------------------------------------------
// flux adjoint, owner side, one lane per point: the FP32 product, and FP64 with
// gamma != 1.4. GEOM: with the cotangents of weights and offsets.
// ---------------------------------------------------------------------------
// weights (w_s, w_n) and offset of an edge: the FP64 geometry, or its FP32 copy
// COPIES: the FP32 product's copies of the geometry are there (a kernel for each
// case: the choice inside the loops cost the product 13 %)
template <bool COPIES>
__device__ __forceinline__ void edge_geometry(const AdjParamsT<double> &P, int e, int i, double2 xy0, bool second,
                                              double &wx, double &wy, double &dx, double &dy)
{
    const double2 w = P.g.fxw[e];
    wx = w.x;
    wy = w.y;
    if (second) {
        const double2 xyi = P.g.xy[i];
        dx = xyi.x - xy0.x;
        dy = xyi.y - xy0.y;
    }
}
// (dx, dy, w_s, w_n) and (a_x, a_y) of an edge in FP32: the copies, or made here
__device__ __forceinline__ float4 float_edge(const DevGeom &g, int e, int i, double2 xy0)
{
    const double2 Pi = g.xy[i], w = g.fxw[e];
    return make_float4((float)(Pi.x - xy0.x), (float)(Pi.y - xy0.y), (float)w.x, (float)w.y);
}
template <bool COPIES>
__device__ __forceinline__ float2 float_weights(const AdjParamsT<float> &P, int e)
{
    if constexpr (COPIES) return __ldg(P.ea + e);
    const double2 a = P.g.lsw[e];
    return make_float2((float)a.x, (float)a.y);
}
template <bool COPIES>
__device__ __forceinline__ float4 float_offsets(const AdjParamsT<float> &P, int e, int i, double2 xy0)
{
    if constexpr (COPIES) return __ldg(P.ef + e);
    return float_edge(P.g, e, i, xy0);
}
template <bool COPIES>
__device__ __forceinline__ void edge_geometry(const AdjParamsT<float> &P, int e, int i, double2 xy0, bool, float &wx,
                                              float &wy, float &dx, float &dy)
{
    const float4 v = float_offsets<COPIES>(P, e, i, xy0);
    dx = v.x;
    dy = v.y;
    wx = v.z;
    wy = v.w;
}

// an exact double of a float; the FP32 one avoids the conversion instruction
// (FP64 pipe), subnormals become zero
__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(float v) { return f32_to_f64_ip(v); }

template <class T, bool GEOM, bool COPIES>
__global__ void __launch_bounds__(128) k_adj_flux(AdjParamsT<T> P)
{
    const DevGeom &g = P.g;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.n) return;
    const uint8_t f = g.flag[p] & 3;
    const bool second = P.order == 2;
    const T h = T(0.5);
    T qb0[4] = {0, 0, 0, 0}, gb0[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int e0 = g.off[p], e1 = g.off[p + 1];
    if (f == FLAG_FARFIELD) {
        // R = 0 there: no cotangent flows from this point
        for (int e = e0; e < e1; ++e) {
            st4(P.ebar, e, qb0);
            if (GEOM && !P.add) P.wbar[e] = make_double2(0.0, 0.0);
        }
        st4(P.qbar, p, qb0);
        if (second) st8(P.gbar, p, gb0);
        return;
    }
    const double2 xy0 = g.xy[p];
    const double2 n0d = g.nrm[p];
    const T nx = T(n0d.x), ny = T(n0d.y);
    const T tx = ny, ty = -nx;
    const T inv_gm1 = T(P.inv_gm1);
    T Rb[4], q0[4], g0[8];
    ld4(P.Rbar, p, Rb);
    // frame-order cotangent of R_local: R_global = (R0, R1 t + R2 n, R3)
    const T Rl[4] = {Rb[0], Rb[1] * tx + Rb[2] * ty, Rb[1] * nx + Rb[2] * ny, Rb[3]};
    ld4(P.q, p, q0);
    if (second) ld8(P.qg, p, g0);
    for (int e = e0; e < e1; ++e) {
        const int i = g.idx[e];
        const uint8_t m = g.mask[e];
        const int ks = xsub(m), kn = ysub(m);
        const bool us_ = sub_needed(f, ks), un_ = sub_needed(f, kn);
        T wx, wy, dx = T(0), dy = T(0);
        edge_geometry<COPIES>(P, e, i, xy0, second, wx, wy, dx, dy);
        T qti[4], qt0[4];
        ld4(P.q, i, qti);
        T gi[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) qt0[k] = q0[k];
        if (second) {
            ld8(P.qg, i, gi);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                qti[k] = qti[k] - h * (dx * gi[k] + dy * gi[4 + k]);
                qt0[k] = qt0[k] - h * (dx * g0[k] + dy * g0[4 + k]);
            }
        }
        T cs[4], cn[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            cs[k] = us_ ? wx * Rl[k] : T(0);
            cn[k] = un_ ? wy * Rl[k] : T(0);
        }
        T qbi[4], qbo[4], Gsi[4] = {0, 0, 0, 0}, Gni[4] = {0, 0, 0, 0}, Gs0[4] = {0, 0, 0, 0},
                              Gn0[4] = {0, 0, 0, 0};
        const T sgs = (m & M_XPOS) ? T(1) : T(-1), sgn = (m & M_YPOS) ? T(1) : T(-1);
        if (us_ || un_) {
            if constexpr (std::is_same<T, double>::value) {
                state_adjoint_rev(qti, tx, ty, nx, ny, us_, sgs, un_, sgn, cs, cn, inv_gm1, P.g14 != 0, qbi, Gsi, Gni);
                state_adjoint_rev(qt0, tx, ty, nx, ny, us_, sgs, un_, sgn, cs, cn, inv_gm1, P.g14 != 0, qbo, Gs0, Gn0);
            } else {
                state_adjoint(qti, tx, ty, nx, ny, us_, sgs, un_, sgn, cs, cn, inv_gm1, P.g14 != 0, qbi, Gsi, Gni);
                state_adjoint(qt0, tx, ty, nx, ny, us_, sgs, un_, sgn, cs, cn, inv_gm1, P.g14 != 0, qbo, Gs0, Gn0);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) qbi[k] = qbo[k] = T(0);
        }
        // R += w (G(q~_i) - G(q~_0)): + for the neighbour, - for the owner
        if constexpr (GEOM) {
            T wbx = T(0), wby = T(0);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                wbx += Rl[k] * (Gsi[k] - Gs0[k]);
                wby += Rl[k] * (Gni[k] - Gn0[k]);
            }
            double2 wb = P.add ? P.wbar[e] : make_double2(0.0, 0.0);
            if (us_) wb.x += to_f64(wbx);
            if (un_) wb.y += to_f64(wby);
            P.wbar[e] = wb;
        }
        st4(P.ebar, e, qbi);
        T dxb = T(0), dyb = T(0);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            qbo[k] = -qbo[k];
            qb0[k] += qbo[k];
            if (second) {
                // q~_0 = q_0 - (dx qx_0 + dy qy_0)/2
                gb0[k] -= h * dx * qbo[k];
                gb0[4 + k] -= h * dy * qbo[k];
                if constexpr (GEOM) {
                    dxb -= h * qbo[k] * g0[k];
                    dyb -= h * qbo[k] * g0[4 + k];
                }
            }
        }
        if constexpr (GEOM) {
            double2 db = P.dbar[e];
            db.x += to_f64(dxb);
            db.y += to_f64(dyb);
            P.dbar[e] = db;
        }
    }
    st4(P.qbar, p, qb0);
    if (second) st8(P.gbar, p, gb0);
}

// ---------------------------------------------------------------------------
// flux adjoint, owner side, FP64 with gamma = 1.4, two lanes per edge: lane 0
// differentiates at the neighbour's state, lane 1 at the point's own one.
//
// In the variables of the fixed-point fluxes (lskum_fixed.cuh) the adjoint is
// short: per direction with cotangent (r0, ra, ro, r3) of [mass, along,
// transverse, energy], J = sum of r G is
//   s0 P + a1 F1 + s2 So P + s3 F3,  s0 = sgn r0 C0, a1 = ra C1, s2 = sgn ro C1,
//   s3 = sgn r3 C3, F1 = Phi/2 + z P, F3 = H P - E/4, z = sgn S_d,
// and P' = Phi, F1' = 2 P, E' = -2 z E give
//   dJ/dz = (s0 + s2 So + s3 H) Phi + 2 a1 P + s3 z E/2,
//   dJ/dSo = s2 P, dJ/dH = s3 P, dJ/dx = J (all factors carry exp(x)),
//   dJ/dln r = 6 s0 P + 7 (a1 F1 + s2 So P) + 8 s3 F3.
// Then H = hc + (S_t^2 + S_n^2)/2, x = q1 + S_t^2 + S_n^2, S = (q2, q3).(t, n) r/2,
// r = (-q4/2)^(-1/2). J itself is what the weight's cotangent needs. Phi, E, P,
// F1, F3 and the factors come from the integer pipes: about 100 FP64
// instructions per lane and edge instead of 400 per edge in one lane, and J's
// rounding error is a fifth of the FP64 chain's. 40k points: 536 -> 186 us.
// ---------------------------------------------------------------------------
struct DirCotangent {
    double J;                        // sum of r G, without the weight
    double bd, bo, bH, bx, bl;       // w dJ/d(S_d, S_o, H, x, ln r)
};
__device__ __forceinline__ DirCotangent direction_cotangent(const FixState &s, bool along_t, unsigned long long sbit,
                                                            double Sd, double So, double H, double C0, double C1,
                                                            double C3, double r0, double ra, double ro, double r3,
                                                            double w)
{
    int64_t Phi_, E_, P_;
    const FixOp zo = fix_phi_e(along_t ? s.St : s.Sn, sbit ? -1 : 0, Phi_, E_, P_);
    const FixOp Po = fix_op(P_);
    const double Phi = fix_to_double(Phi_, -62), P = fix_to_double(P_, -61), P2 = fix_to_double(P_, -60);
    const double Eh = fix_to_double(E_, -63);                                       // E/2
    const double F1 = fix_to_double((Phi_ >> 5) + fix_mul(zo, Po), -58);
    const double F3 = fix_to_double(fix_mul_s<1>(fix_op(s.H), Po) - (E_ >> 7), -57);
    const double s0 = flip_sign(r0 * C0, sbit), a1 = ra * C1, s2 = flip_sign(ro * C1, sbit), y3 = r3 * C3, s3 = flip_sign(y3, sbit);
    const double K = fma(s3, H, fma(s2, So, s0));
    const double u1 = a1 * F1, u3 = s3 * F3, s2P = s2 * P, v = So * s2P, uv = u1 + v;
    DirCotangent o;
    o.J = fma(s0, P, uv + u3);
    const double Jl = fma(6.0, o.J, fma(2.0, u3, uv));
    const double Jz = fma(K, Phi, fma(a1, P2, y3 * (Sd * Eh)));    // sgn z = S_d
    o.bd = flip_sign(w, sbit) * Jz;
    o.bo = w * s2P;
    o.bH = w * (s3 * P);
    o.bx = w * o.J;
    o.bl = w * Jl;
    return o;
}

// a state outside the fixed-point ranges: the FP64 reverse mode
struct StateCotangent {
    double qb[4], Js, Jn;
};
__device__ __noinline__ StateCotangent state_cotangent_fp64(double q0, double q1, double q2, double q3, double2 n0,
                                                            int flags, double wx, double wy, double R0, double Rs,
                                                            double Rn, double R3, double inv_gm1)
{
    const double qt[4] = {q0, q1, q2, q3}, Rl[4] = {R0, Rs, Rn, R3};
    const bool us_ = flags & 1, un_ = flags & 2;
    double cs[4], cn[4], Gs[4] = {0.0, 0.0, 0.0, 0.0}, Gn[4] = {0.0, 0.0, 0.0, 0.0};
    for (int k = 0; k < 4; ++k) {
        cs[k] = us_ ? wx * Rl[k] : 0.0;
        cn[k] = un_ ? wy * Rl[k] : 0.0;
    }
    StateCotangent o;
    state_adjoint_rev(qt, n0.y, -n0.x, n0.x, n0.y, us_, flags & 4 ? 1.0 : -1.0, un_, flags & 8 ? 1.0 : -1.0, cs, cn,
                      inv_gm1, true, o.qb, Gs, Gn);
    o.Js = o.Jn = 0.0;
    for (int k = 0; k < 4; ++k) {
        o.Js += Rl[k] * Gs[k];
        o.Jn += Rl[k] * Gn[k];
    }
    return o;
}

template <bool GEOM>
__global__ void __launch_bounds__(128, 5) k_adj_flux_pair(AdjParams P)
{
    const DevGeom &g = P.g;
    const int64_t pp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 1;
    const int l = threadIdx.x & 1;
    const int64_t p = pp < g.n ? pp : g.n - 1;
    const uint8_t f = g.flag[p] & 3;
    const bool second = P.order == 2, live = pp < g.n;
    double qb0[4] = {0.0, 0.0, 0.0, 0.0}, gb0[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const int e0 = g.off[p], e1 = g.off[p + 1];
    if (live && l == 0 && f == FLAG_FARFIELD) {
        // R = 0 there: no cotangent flows from this point
        for (int e = e0; e < e1; ++e) {
            st4(P.ebar, e, qb0);
            if (GEOM && !P.add) P.wbar[e] = make_double2(0.0, 0.0);
        }
    }
    const int deg = live && f != FLAG_FARFIELD ? e1 - e0 : 0;
    const double2 xy0 = g.xy[p];
    const double2 n0 = g.nrm[p];
    const FixOp fnx = fix_op(fix_unit(n0.x)), fny = fix_op(fix_unit(n0.y));
    const double tx = n0.y, ty = -n0.x;
    double Rb[4], g0[8];
    ld4(P.Rbar, p, Rb);
    // frame-order cotangent of R_local: R_global = (R0, R1 t + R2 n, R3)
    const double Rs = Rb[1] * tx + Rb[2] * ty, Rn = Rb[1] * n0.x + Rb[2] * n0.y;
    if (second) ld8(P.qg, p, g0);
    // whole warps go through the longest row: the lanes exchange J by shuffles
    const int most = __reduce_max_sync(0xffffffffu, deg);
#pragma unroll 1
    for (int j = 0; j < most; ++j) {
        const bool act = j < deg;
        const int e = act ? e0 + j : e0;
        const int i = g.idx[e];
        const uint8_t m = g.mask[e];
        const bool us_ = sub_needed(f, xsub(m)), un_ = sub_needed(f, ysub(m));
        const double2 w = g.fxw[e];   // zero where the sub-stencil is not needed
        const int64_t row = l ? p : (int64_t)i;
        double qt[4], qb[4], Js, Jn;
        gather4(P.q, row, qt);
        double2 h = make_double2(0.0, 0.0);
        if (second) {
            if (g.hd) {
                h = g.hd[e];
            } else {
                const double2 xyi = g.xy[i];
                h = make_double2(0.5 * (xyi.x - xy0.x), 0.5 * (xyi.y - xy0.y));
            }
            double gr[8];
            gather8(P.qg, row, gr);
#pragma unroll
            for (int k = 0; k < 4; ++k) qt[k] = fma(-h.y, gr[4 + k], fma(-h.x, gr[k], qt[k]));
        }
        FixState s;
        if (fix_state(qt, fnx, fny, s)) {
            double St = fix_to_double(s.St, -61), Sn = fix_to_double(s.Sn, -61);
            const double H = fix_to_double(s.H, -59);
            const double C0 = fix_to_double(s.c0, fix_e0(s.n, s.k)), C1 = fix_to_double(s.c1, fix_e1(s.n, s.k)),
                         C3 = fix_to_double(s.c3, fix_e3(s.n, s.k)), hr = fix_to_double(s.r, -62 - s.k);
            // (as in the forward: a small one in FP64)
            if (fix_slow(s.St)) St = fma(qt[1], tx, qt[2] * ty) * hr;
            if (fix_slow(s.Sn)) Sn = fma(qt[1], n0.x, qt[2] * n0.y) * hr;
            const DirCotangent a = direction_cotangent(s, true, (m & M_XPOS) ? 0ull : kSignBit, St, Sn, H, C0, C1, C3,
                                                       Rb[0], Rs, Rn, Rb[3], w.x);
            const DirCotangent b = direction_cotangent(s, false, (m & M_YPOS) ? 0ull : kSignBit, Sn, St, H, C0, C1, C3,
                                                       Rb[0], Rn, Rs, Rb[3], w.y);
            Js = a.J;
            Jn = b.J;
            const double bx = a.bx + b.bx, d = fma(2.0, bx, a.bH + b.bH);
            const double bt = fma(St, d, a.bd + b.bo), bn = fma(Sn, d, a.bo + b.bd);
            const double bl = fma(St, bt, fma(Sn, bn, a.bl + b.bl));
            const double mt = bt * hr, mn = bn * hr;
            qb[0] = bx;
            qb[1] = fma(mt, tx, mn * n0.x);
            qb[2] = fma(mt, ty, mn * n0.y);
            qb[3] = bl * (hr * hr);
        } else {
            const StateCotangent o = state_cotangent_fp64(
                qt[0], qt[1], qt[2], qt[3], n0, (us_ ? 1 : 0) | (un_ ? 2 : 0) | ((m & M_XPOS) ? 4 : 0) | ((m & M_YPOS) ? 8 : 0),
                w.x, w.y, Rb[0], Rs, Rn, Rb[3], P.inv_gm1);
#pragma unroll
            for (int k = 0; k < 4; ++k) qb[k] = o.qb[k];
            Js = o.Js;
            Jn = o.Jn;
        }
        // R += w (G(q~_i) - G(q~_0)): + for the neighbour, - for the owner
        if constexpr (GEOM) {
            const double Jso = __shfl_xor_sync(0xffffffffu, Js, 1), Jno = __shfl_xor_sync(0xffffffffu, Jn, 1);
            if (act && l == 0) {
                double2 wb = P.add ? P.wbar[e] : make_double2(0.0, 0.0);
                if (us_) wb.x += Js - Jso;
                if (un_) wb.y += Jn - Jno;
                P.wbar[e] = wb;
            }
        }
        if (act && l == 0) st4(P.ebar, e, qb);
        if (act && l == 1) {
            double dxb = 0.0, dyb = 0.0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                qb0[k] -= qb[k];
                if (second) {
                    // q~_0 = q_0 - h.grad q_0, with the cotangent -qb; h = d/2
                    gb0[k] = fma(h.x, qb[k], gb0[k]);
                    gb0[4 + k] = fma(h.y, qb[k], gb0[4 + k]);
                    if constexpr (GEOM) {
                        dxb = fma(qb[k], g0[k], dxb);
                        dyb = fma(qb[k], g0[4 + k], dyb);
                    }
                }
            }
            if constexpr (GEOM) {
                if (second) {
                    double2 db = P.dbar[e];
                    db.x = fma(0.5, dxb, db.x);
                    db.y = fma(0.5, dyb, db.y);
                    P.dbar[e] = db;
                }
            }
        }
    }
    if (live && l == 1) {
        st4(P.qbar, p, qb0);
        if (second) st8(P.gbar, p, gb0);
    }
}

// half offset and full-stencil weights of incoming edge t: the copies in the order
// that they are read in, or the edge's own
__device__ __forceinline__ double2 edge_half_offset(const DevGeom &g, int e, int64_t src)
{
    if (g.hd) return g.hd[e];
    const double2 a = g.xy[src], b = g.xy[g.idx[e]];
    return make_double2(0.5 * (b.x - a.x), 0.5 * (b.y - a.y));
}
__device__ __forceinline__ double2 incoming_offset(const AdjParamsT<double> &P, int t)
{
    return P.thd ? __ldg(P.thd + t) : edge_half_offset(P.g, P.tedge[t], P.tsrc[t]);
}
__device__ __forceinline__ double2 incoming_weights(const AdjParamsT<double> &P, int t)
{
    return P.tlsw ? __ldg(P.tlsw + t) : P.g.lsw[P.tedge[t]];
}
__device__ __forceinline__ float4 float_incoming(const DevGeom &g, int e, int src)
{
    const double2 a = g.lsw[e], A = g.xy[src], B = g.xy[g.idx[e]];
    return make_float4((float)a.x, (float)a.y, (float)(B.x - A.x), (float)(B.y - A.y));
}
template <bool COPIES>
__device__ __forceinline__ void incoming(const AdjParamsT<double> &P, int t, double &hx, double &hy, double &ax, double &ay)
{
    const double2 hh = incoming_offset(P, t), a = incoming_weights(P, t);
    hx = hh.x;
    hy = hh.y;
    ax = a.x;
    ay = a.y;
}
template <bool COPIES>
__device__ __forceinline__ float4 float_incoming_edge(const AdjParamsT<float> &P, int t)
{
    if constexpr (COPIES) return __ldg(P.tf + t);
    return float_incoming(P.g, P.tedge[t], P.tsrc[t]);
}
template <bool COPIES>
__device__ __forceinline__ void incoming(const AdjParamsT<float> &P, int t, float &hx, float &hy, float &ax, float &ay)
{
    const float4 v = float_incoming_edge<COPIES>(P, t);
    ax = v.x;
    ay = v.y;
    hx = 0.5f * v.z;
    hy = 0.5f * v.w;
}

// start + a0 b0 + a1 b1
__device__ __forceinline__ double dot_rest(const double *a, const double *b, double start)
{
    return fma(a[1], b[1], fma(a[0], b[0], start));
}
// An offset's or weight's cotangent sums four components over the two lanes of a
// point: its x in the order 0 1 2 3 and its y in the order 2 3 0 1, so that the
// lanes go through both at once and hand the half-done sum over in the middle
// (half the FP64 additions of a lane for each sum).
// lane l of a pair holds components 2l and 2l + 1 of a, of x and of y: lane 1
// returns x0 + a.x, lane 0 y0 + a.y. start is this lane's part, x0 in lane 0 and y0
// in lane 1. Called by whole warps.
__device__ __forceinline__ double half_dot(int l, const double a[2], const double x[2], const double y[2], double start)
{
    const double mine[2] = {l ? y[0] : x[0], l ? y[1] : x[1]}, other[2] = {l ? x[0] : y[0], l ? x[1] : y[1]};
    return dot_rest(a, other, __shfl_xor_sync(0xffffffffu, dot_rest(a, mine, start), 1));
}

// ---------------------------------------------------------------------------
// flux adjoint, neighbour side: point p gathers the cotangents of q~_p over
// the edges that reach it
// ---------------------------------------------------------------------------
template <class T, bool GEOM, bool COPIES>
__global__ void __launch_bounds__(128) k_adj_flux_gather(AdjParamsT<T> P)
{
    const DevGeom &g = P.g;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.n) return;
    const bool second = P.order == 2;
    const T h = T(0.5);
    T qb[4], gb[8], gp[8];
    ld4(P.qbar, p, qb);
    if (second) {
        ld8(P.gbar, p, gb);
        if constexpr (GEOM) ld8(P.qg, p, gp);
    }
    const int t1 = P.toff[p + 1];
    for (int t = P.toff[p]; t < t1; ++t) {
        const int e = P.tedge[t];
        T eb[4];
        ld4(P.ebar, e, eb);
#pragma unroll
        for (int k = 0; k < 4; ++k) qb[k] += eb[k];
        if (second) {
            T hx, hy, ax, ay;
            incoming<COPIES>(P, t, hx, hy, ax, ay);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // q~_p = q_p - (dx qx_p + dy qy_p)/2 on this edge
                gb[k] -= hx * eb[k];
                gb[4 + k] -= hy * eb[k];
            }
            if constexpr (GEOM) {
                T dxb = T(0), dyb = T(0);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    dxb -= h * eb[k] * gp[k];
                    dyb -= h * eb[k] * gp[4 + k];
                }
                double2 d = P.dbar[e];
                d.x += to_f64(dxb);
                d.y += to_f64(dyb);
                P.dbar[e] = d;
            }
        }
    }
    st4(P.qbar, p, qb);
    if (second) st8(P.gbar, p, gb);
}

// the same in FP64 of order 2 with the offsets' cotangents: two lanes per point,
// two components each (half_dot). A point's incoming edges are a serial chain of
// dependent loads and FP64 sums: 37 -> 28 us at 40k points; at 640k (0.27 ms) the
// FP64 pipe bounds both forms.
__global__ void __launch_bounds__(128) k_adj_flux_gather_pair(AdjParams P)
{
    const int64_t n = P.g.n, pp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 1;
    const int l = threadIdx.x & 1, k0 = 2 * l;
    const bool live = pp < n;
    const int64_t p = live ? pp : n - 1;   // (lanes past the end take part in the shuffles)
    double qb[2], gx[2], gy[2], px[2], py[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        qb[k] = P.qbar[4 * p + k0 + k];
        gx[k] = P.gbar[8 * p + k0 + k];
        gy[k] = P.gbar[8 * p + 4 + k0 + k];
    }
    gather_c<2>(P.qg + 8 * p + k0, px);
    gather_c<2>(P.qg + 8 * p + 4 + k0, py);
    const int t0 = P.toff[p], deg = live ? P.toff[p + 1] - t0 : 0;
    const int most = __reduce_max_sync(0xffffffffu, deg);
#pragma unroll 1
    for (int j = 0; j < most; ++j) {
        double eb[2] = {0.0, 0.0};
        int e = 0;
        if (j < deg) {
            e = P.tedge[t0 + j];
            const double2 h = incoming_offset(P, t0 + j);
            const double2 v = *reinterpret_cast<const double2 *>(P.ebar + 4 * (int64_t)e + k0);
            eb[0] = v.x;
            eb[1] = v.y;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                qb[k] += eb[k];
                // q~_p = q_p - h.grad q_p on this edge
                gx[k] = fma(-h.x, eb[k], gx[k]);
                gy[k] = fma(-h.y, eb[k], gy[k]);
            }
        }
        const double d = half_dot(l, eb, px, py, 0.0);
        if (j < deg) {
            double *o = reinterpret_cast<double *>(P.dbar + e) + (1 - l);
            *o = fma(-0.5, d, *o);
        }
    }
    if (!live) return;
    store_c<2>(P.qbar + 4 * p + k0, qb);
    store_c<2>(P.gbar + 8 * p + k0, gx);
    store_c<2>(P.gbar + 8 * p + 4 + k0, gy);
}

// ---------------------------------------------------------------------------
// one least-squares pass of E15 in reverse. Forward (per component c):
//   g_p = sum_e a_e s_e,  s_e = (q_i - q_p) - [dx (gx'_i - gx'_p) + dy (gy'_i - gy'_p)]/2
// with g' the previous iterate (absent in the first-order pass). GEOM: with the
// cotangents of the weights and offsets; without them an outgoing edge only
// gives the owner's q its share, and no neighbour value is read for it (FP32 at
// 640k points: 228 -> 58 us a pass, half of it from the geometry's FP32 copies,
// which spare the FP64 pipe the conversions).
// ---------------------------------------------------------------------------
template <bool GEOM, bool COPIES>
__global__ void __launch_bounds__(128) k_adj_grad_fp32(AdjParamsT<float> P, const float *__restrict__ gprev,
                                                       const float *__restrict__ gbar_in,
                                                       float *__restrict__ gbar_out, int first)
{
    const DevGeom &g = P.g;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.n) return;
    const bool inner = gprev != nullptr;
    float qb[4], gb[8], qp[4], gbo[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    ld4(P.qbar, p, qb);
    ld8(gbar_in, p, gb);
    if constexpr (GEOM) ld4(P.q, p, qp);
    // an inner pass is sum_e a_e (q_i - q_0 - h_e.grad q_i) + grad q_0 / 2
    // (h_e the half offset; the terms in grad q_0 add up to grad q_0 / 2 since
    // sum_e a_e d_e^T = I, and the forward passes take them so), so grad q_0
    // gets gb / 2 and neither the weights nor the offsets see grad q_0
    if (inner) {
#pragma unroll
        for (int k = 0; k < 8; ++k) gbo[k] = 0.5f * gb[k];
    }
    // outgoing edges: owner terms, and the cotangents of a_e and of the offsets
    for (int e = g.off[p]; e < g.off[p + 1]; ++e) {
        const float2 a = float_weights<COPIES>(P, e);
        if constexpr (!GEOM) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float sb = a.x * gb[k] + a.y * gb[4 + k];
                qb[k] -= sb;
            }
        } else {
            const int i = g.idx[e];
            float qi[4], gi[8], hx = 0.0f, hy = 0.0f;
            ld4(P.q, i, qi);
            if (inner) {
                const float4 v = float_offsets<COPIES>(P, e, i, g.xy[p]);
                hx = 0.5f * v.x;
                hy = 0.5f * v.y;
                ld8(gprev, i, gi);
            }
            float abx = 0.0f, aby = 0.0f, dbx = 0.0f, dby = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float sb = a.x * gb[k] + a.y * gb[4 + k];
                float s = qi[k] - qp[k];
                if (inner) {
                    s = s - (hx * gi[k] + hy * gi[4 + k]);
                    // d_e = 2 h_e: d_bar = -(sb/2) grad q_i
                    dbx -= 0.5f * sb * gi[k];
                    dby -= 0.5f * sb * gi[4 + k];
                }
                qb[k] -= sb;
                abx += s * gb[k];
                aby += s * gb[4 + k];
            }
            double2 ab = first && !P.add ? make_double2(0.0, 0.0) : P.abar[e];
            ab.x += to_f64(abx);
            ab.y += to_f64(aby);
            P.abar[e] = ab;
            if (inner) {
                double2 db = P.dbar[e];
                db.x += to_f64(dbx);
                db.y += to_f64(dby);
                P.dbar[e] = db;
            }
        }
    }
    // incoming edges: the terms of this point as a neighbour
    const int t1 = P.toff[p + 1];
    for (int t = P.toff[p]; t < t1; ++t) {
        const int src = P.tsrc[t];
        float hx, hy, ax, ay;
        incoming<COPIES>(P, t, hx, hy, ax, ay);
        float gs[8];
        ld8(gbar_in, src, gs);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float sb = ax * gs[k] + ay * gs[4 + k];
            qb[k] += sb;
            if (inner) {
                gbo[k] -= hx * sb;
                gbo[4 + k] -= hy * sb;
            }
        }
    }
    st4(P.qbar, p, qb);
    if (inner) st8(gbar_out, p, gbo);
}

// The FP64 pass: the outgoing and the incoming edges of a point go to blocks of
// their own (blockIdx.y; twice the warps in flight, half the serial chain),
// which keep the q cotangent apart (qbar2: the owner's share, summed with qbar
// by k_adj_state), and the two-term products run on the integer pipes
// (fix_dot): 40 FP64 instructions per edge of 68. 87 -> 62 us a pass at 40k points.
// Two lanes per point, two components each, which add up a_bar and d_bar together
// (half_dot). One lane with all four: a residual product of 8k points 0.50 ms
// against 0.45, 64k 0.857 / 0.806, 160k 1.64 / 1.57, 640k 5.46 / 5.28. Blocks per SM
// (registers against warps) 5 / 6 / 7 / 8: 0.434 / 0.437 / 0.444 / 0.453 ms at 18k,
// 1.608 / 1.588 / 1.570 / 1.582 at 160k, 5.43 / 5.34 / 5.28 / 5.28 at 640k.
__device__ __forceinline__ double dot2(const FixPair &a, const FixPair &b, double ax, double ay, double bx, double by)
{
    if (fix_dot_in_range(a, b)) return fix_dot(a, b);
    return fix_pair_zero(b) ? 0.0 : fma(ay, by, ax * bx);   // both terms zero (or subnormal): nothing to add
}

template <bool GEOM>
__global__ void __launch_bounds__(128, GEOM ? 7 : 8) k_adj_grad_fp64(AdjParams P, const double *__restrict__ gprev,
                                                                    const double *__restrict__ gbar_in,
                                                                    double *__restrict__ gbar_out, int first)
{
    constexpr int C = 2;
    const DevGeom &g = P.g;
    const int64_t pp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 1;
    const int l = threadIdx.x & 1, k0 = C * l;
    const bool live = pp < g.n;
    const int64_t p = live ? pp : g.n - 1;   // (lanes past the end take part in the shuffles)
    const bool inner = gprev != nullptr;
    double qb[C], gx[C], gy[C];
    gather_c<C>(gbar_in + 8 * p + k0, gx);
    gather_c<C>(gbar_in + 8 * p + 4 + k0, gy);
    if (blockIdx.y == 0) {
        // outgoing edges: owner terms, and the cotangents of a_e and of the offsets
        FixPair gbp[C];
        double qp[C];
#pragma unroll
        for (int k = 0; k < C; ++k) {
            qb[k] = first ? 0.0 : P.qbar2[4 * p + k0 + k];
            gbp[k] = fix_pair(gx[k], gy[k]);
        }
        double2 xyp = make_double2(0.0, 0.0);
        if constexpr (GEOM) {
            gather_c<C>(P.q + 4 * p + k0, qp);
            if (!g.hd) xyp = g.xy[p];
        }
        const int e0 = g.off[p], deg = live ? g.off[p + 1] - e0 : 0;
        // whole warps go through the longest row where the lanes exchange sums by shuffles
        const int most = GEOM ? __reduce_max_sync(0xffffffffu, deg) : deg;
#pragma unroll 1
        for (int j = 0; j < most; ++j) {
            const bool act = j < deg;
            const int e = act ? e0 + j : e0;
            const double2 a = g.lsw[e];
            const FixPair ap = fix_pair(a.x, a.y);
            double sb[C];
#pragma unroll
            for (int k = 0; k < C; ++k) {
                sb[k] = dot2(ap, gbp[k], a.x, a.y, gx[k], gy[k]);
                if (act) qb[k] -= sb[k];
            }
            if constexpr (GEOM) {
                const int64_t i = g.idx[e];
                double qi[C], s[C], ix[C], iy[C];
                gather_c<C>(P.q + 4 * i + k0, qi);
#pragma unroll
                for (int k = 0; k < C; ++k) s[k] = qi[k] - qp[k];
                if (inner) {
                    double2 h;
                    if (g.hd) {
                        h = g.hd[e];
                    } else {
                        const double2 xyi = g.xy[i];
                        h = make_double2(0.5 * (xyi.x - xyp.x), 0.5 * (xyi.y - xyp.y));
                    }
                    const FixPair hp = fix_pair(h.x, h.y);
                    gather_c<C>(gprev + 8 * i + k0, ix);
                    gather_c<C>(gprev + 8 * i + 4 + k0, iy);
#pragma unroll
                    for (int k = 0; k < C; ++k) s[k] -= dot2(hp, fix_pair(ix[k], iy[k]), h.x, h.y, ix[k], iy[k]);
                }
                // a_bar += s gb, and with d_e = 2 h_e: d_bar -= (sb/2) grad q_i
                const bool start = first && !P.add;
                // (a lane starts one sum and ends, and stores, the other)
                double *const ab = reinterpret_cast<double *>(P.abar + e), *const db = reinterpret_cast<double *>(P.dbar + e);
                const double a1 = half_dot(l, s, gx, gy, start || !act ? 0.0 : ab[l]);
                if (act) ab[1 - l] = a1;
                if (inner) {   // (the same in every lane)
                    const double d1 = half_dot(l, sb, ix, iy, 0.0);
                    if (act) db[1 - l] = fma(-0.5, d1, db[1 - l]);
                }
            }
        }
        if (live) store_c<C>(P.qbar2 + 4 * p + k0, qb);
    } else {
        // incoming edges: the terms of this point as a neighbour; an inner pass
        // gives grad q_0 the cotangent gb / 2 (see k_adj_grad_fp32)
        if (!live) return;
        double ox[C], oy[C];
#pragma unroll
        for (int k = 0; k < C; ++k) {
            qb[k] = P.qbar[4 * p + k0 + k];
            ox[k] = 0.5 * gx[k];
            oy[k] = 0.5 * gy[k];
        }
        const int t1 = P.toff[p + 1];
#pragma unroll 1
        for (int t = P.toff[p]; t < t1; ++t) {
            const int64_t src = P.tsrc[t];
            const double2 a = incoming_weights(P, t);
            const FixPair ap = fix_pair(a.x, a.y);
            double sx[C], sy[C];
            gather_c<C>(gbar_in + 8 * src + k0, sx);
            gather_c<C>(gbar_in + 8 * src + 4 + k0, sy);
            double2 h = make_double2(0.0, 0.0);
            if (inner) h = incoming_offset(P, t);
#pragma unroll
            for (int k = 0; k < C; ++k) {
                const double sb = dot2(ap, fix_pair(sx[k], sy[k]), a.x, a.y, sx[k], sy[k]);
                qb[k] += sb;
                if (inner) {
                    ox[k] = fma(-h.x, sb, ox[k]);
                    oy[k] = fma(-h.y, sb, oy[k]);
                }
            }
        }
        store_c<C>(P.qbar + 4 * p + k0, qb);
        if (inner) {
            store_c<C>(gbar_out + 8 * p + k0, ox);
            store_c<C>(gbar_out + 8 * p + 4 + k0, oy);
        }
    }
}

// ---------------------------------------------------------------------------
// Venkatakrishnan's limiter in reverse. Forward (k_qgrad's limited pass, per
// component): g = phi g_raw with phi = f(x_m, d_m) when x_m < 2 d_m, else 1;
//   f(x, d) = N/M, N = x (x + 2d) + eps^2, M = x (x + d) + 2 d^2 + eps^2,
//   x_m = min(D+, -D-), D+- the largest / smallest q_i - q_0 over the stencil
//   and P_0 itself (0), d_m = max_e |h_e . g_raw| (h_e the half offset),
//   eps^2 = (K dmin)^3, dmin the nearest neighbour's distance.
// With G = gbar . g_raw (the cotangent of phi):
//   g_raw_bar = phi gbar + G f_d s h*          (h* the edge of d_m, s the sign
//                                               of h*.g_raw)
//   x_m = q_i - q_0 (D+) or q_0 - q_j (-D-): q_0 and the extreme neighbour get
//         -+ G f_x; the neighbour's share is handed over through lidx/lval
//         and added by k_adj_limit_gather
//   the offsets: d* = 2 h* gets G f_d s g_raw / 2, the nearest neighbour's
//         offset gets 3 K^3 dmin^2 G f_eps d/|d| (through eps^2)
// The choices: the first largest (smallest) q_i in row order, P_0's own winning
// ties (the forward takes the value of the largest rounded q_i - q_0 alone; where
// several differences round alike, q_i still tells which is the extreme one); the
// first largest |h . g_raw|; the first nearest neighbour by squared distance. Where phi = 1 the limiter is
// inactive and gbar passes through.
//
// With s = x + d and r = 1/M: f_x = (2 s - phi (x + s)) r, f_d = (2 x - phi (x + 4 d)) r,
// f_eps = (1 - phi) r = d (2 d - x) r^2.
//
// Four lanes per point, a component each; what they share is exchanged by
// shuffles: the offset of an edge that several components chose is written
// once, by the lowest of them. The FP64 pipe bounds it, so the searches compare
// bits (the extreme neighbours by q_i itself, the shifts by magnitude) and r
// comes from the integer pipes: 76 -> 33 us at 40k points, 700 -> 389 us at 640k.
// ---------------------------------------------------------------------------
// doubles in their order as integers (both zeros equal), and back
__device__ __forceinline__ long long ordered(double v)
{
    long long b = __double_as_longlong(v);
    if (b == (long long)kSignBit) b = 0;
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double unordered(long long b)
{
    return __longlong_as_double(b ^ ((b >> 63) & 0x7fffffffffffffffll));
}

__global__ void __launch_bounds__(128) k_adj_limit(AdjParams P, const double *__restrict__ graw,
                                                   const double *__restrict__ gbar_in, double *__restrict__ gbar_out,
                                                   int32_t *__restrict__ lidx, double *__restrict__ lval,
                                                   double limK)
{
    const DevGeom &g = P.g;
    const int64_t pp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
    const int k = threadIdx.x & 3;
    const bool live = pp < g.n;
    const int64_t p = live ? pp : g.n - 1;   // (lanes past the end take part in the shuffles)
    const double q0 = P.q[4 * p + k];
    const double grx = graw[8 * p + k], gry = graw[8 * p + 4 + k];
    const double gbx = gbar_in[8 * p + k], gby = gbar_in[8 * p + 4 + k];
    double2 P0 = make_double2(0.0, 0.0);
    if (!g.hd) P0 = g.xy[p];
    const int e1 = g.off[p + 1];
    long long mx = ordered(q0), mn = mx, hm = -1;   // largest and smallest q, bits of d_m (none yet)
    unsigned long long sh = 0;
    int emx = -1, emn = -1, eh = -1;
    double2 hh = make_double2(0.0, 0.0);
    for (int e = g.off[p]; e < e1; ++e) {
        const int i = g.idx[e];
        const long long qi = ordered(P.q[4 * (int64_t)i + k]);
        double2 h;
        if (g.hd) {
            h = g.hd[e];
        } else {
            const double2 Pi = g.xy[i];
            h = make_double2(0.5 * (Pi.x - P0.x), 0.5 * (Pi.y - P0.y));
        }
        if (qi > mx) {
            mx = qi;
            emx = e;
        }
        if (qi < mn) {
            mn = qi;
            emn = e;
        }
        const unsigned long long c = (unsigned long long)__double_as_longlong(fma(h.x, grx, h.y * gry));
        const long long ca = (long long)(c & ~kSignBit);
        if (ca > hm) {
            hm = ca;
            eh = e;
            sh = c & kSignBit;
            hh = h;
        }
    }
    const double dmx = unordered(mx) - q0, dmn = q0 - unordered(mn);
    const bool plus = dmx <= dmn;
    const double x = plus ? dmx : dmn, d = __longlong_as_double(hm), d2 = 2.0 * d;
    const bool on = live && eh >= 0 && x < d2;   // else phi = 1
    const double hK = g.dmin[p] * limK, hK2 = hK * hK;
    double gox = gbx, goy = gby, xb = 0.0, cx = 0.0, cy = 0.0, db = 0.0;
    int li = -1;
    if (on) {
        const double eps2 = hK2 * hK, s = x + d;
        const double N = fma(x, x + d2, eps2), M = fma(x, s, fma(d2, d, eps2));
        const double r = fix_moderate(M) ? fix_reciprocal(M) : 1.0 / M;
        double phi = N * r;
        phi = fma(fma(-M, phi, N), r, phi);
        const double G = r * fma(gbx, grx, gby * gry);
        const double gd = flip_sign(G * fma(-phi, fma(4.0, d, x), x + x), sh);
        gox = fma(phi, gbx, gd * hh.x);
        goy = fma(phi, gby, gd * hh.y);
        li = plus ? emx : emn;
        xb = G * fma(-phi, x + s, s + s);
        if (!plus) xb = -xb;
        // d* = 2 h*: its offset cotangent is half that of h*
        cx = 0.5 * gd * grx;
        cy = 0.5 * gd * gry;
        db = G * (r * (d * (d2 - x)));
    }
    const int mine = on ? eh : -1;
    bool lead = on;
    double sx = cx, sy = cy;
#pragma unroll
    for (int m = 1; m < 4; ++m) {
        const int eo = __shfl_xor_sync(0xffffffffu, mine, m);
        const double ox = __shfl_xor_sync(0xffffffffu, cx, m), oy = __shfl_xor_sync(0xffffffffu, cy, m);
        if (eo == mine) {
            sx += ox;
            sy += oy;
            if ((k ^ m) < k) lead = false;
        }
    }
    db += __shfl_xor_sync(0xffffffffu, db, 1);
    db += __shfl_xor_sync(0xffffffffu, db, 2);
    if (lead) {
        double2 o = P.dbar[eh];
        o.x += sx;
        o.y += sy;
        P.dbar[eh] = o;
    }
    __syncwarp();   // the nearest edge may be one of those
    if (live && k == 0 && db != 0.0) {
        const int e = P.near_e[p];
        const double2 u = P.near_u[p];
        const double dminb = 3.0 * limK * hK2 * db;
        double2 o = P.dbar[e];
        o.x = fma(dminb, u.x, o.x);
        o.y = fma(dminb, u.y, o.y);
        P.dbar[e] = o;
    }
    if (!live) return;
    if (li < 0) xb = 0.0;
    P.qbar[4 * p + k] -= xb;
    gbar_out[8 * p + k] = gox;
    gbar_out[8 * p + 4 + k] = goy;
    lidx[4 * p + k] = li;
    lval[4 * p + k] = xb;
}

// the extreme neighbours' share of the limiter's q cotangent (k_adj_limit),
// gathered over each point's incoming edges (no atomics)
__global__ void __launch_bounds__(128) k_adj_limit_gather(AdjParams P, const int32_t *__restrict__ lidx,
                                                          const double *__restrict__ lval)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P.g.n) return;
    const int t0 = P.toff[p], t1 = P.toff[p + 1];
    if (t0 == t1) return;
    double qb[4];
    ld4(P.qbar, p, qb);
    bool any = false;
    for (int t = t0; t < t1; ++t) {
        const int e = P.tedge[t];
        const int64_t src = P.tsrc[t];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (lidx[4 * src + k] == e) {
                qb[k] += lval[4 * src + k];
                any = true;
            }
        }
    }
    if (any) st4(P.qbar, p, qb);
}

// ---------------------------------------------------------------------------
// least-squares weights back to edge offsets (owner side). A system with
// M = sum d d^T and weights a = M^-1 d gives
//   d_bar_k = b_k - B d_k,  b = M^-1 a_bar,  B = sum (b a^T + a b^T).
// Full stencil: a_bar = abar, and with C = sum a_bar a^T over the forward's own
// weights B = M^-1 C + (M^-1 C)^T. (S = sum (a_bar d^T + d a_bar^T) and B = M^-1 S M^-1
// has the same count of operations but takes S through M^-1 twice: on a stencil
// stretched 1000 : 1 across both axes y_bar was 3e-9 off where the forward's
// conditioning gives 4e-11.) A sub-stencil takes one row of M^-1 d (frame (s, n)) as
// its weight, so a_bar is the weight's cotangent wb along that row, b = wb beta
// with beta the row of M^-1, A = M^-1 sum wb d and B = beta A^T + A beta^T.
//
// All M^-1 depend on the points alone: k_adj_plan forms them once per context,
// so a product needs one pass for C and the D = sum wb d, and one for the
// offsets' cotangents, with the B of an edge's two sub-stencils added up first:
// 39 FP64 instructions per edge (half offsets h where they are stored: D takes
// them, B is doubled instead). The sub-stencils stay in the frame that their
// weights were solved in: b and B d nearly cancel for a thin sub-stencil, and B
// turned to global axes lost seven digits there. 94 -> 63 us at 40k points, 823 -> 502 us at 640k.
// ---------------------------------------------------------------------------
struct Sym2 {
    double xx, xy, yy;
};
__device__ __forceinline__ Sym2 inverse2(const Sym2 &A)
{
    const double r = 1.0 / (A.xx * A.yy - A.xy * A.xy);
    return Sym2{A.yy * r, -A.xy * r, A.xx * r};
}
__device__ __forceinline__ double2 times(const Sym2 &A, double2 v)
{
    return make_double2(fma(A.xx, v.x, A.xy * v.y), fma(A.xy, v.x, A.yy * v.y));
}

// (s, n) of an offset; the same operations for d and for h = d/2
__device__ __forceinline__ double2 in_frame(double2 d, double2 n0)
{
    return make_double2(fma(d.x, n0.y, -(d.y * n0.x)), fma(d.x, n0.x, d.y * n0.y));
}

// plan [kAdjPlan][n]: M^-1 (xx, xy, yy) of the full stencil, then of each
// sub-stencil, zero where the point needs none
__global__ void __launch_bounds__(128) k_adj_plan(DevGeom g, double *__restrict__ plan, int32_t *__restrict__ near_e,
                                                  double2 *__restrict__ near_u)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, n = g.n;
    if (p >= n) return;
    const uint8_t f = g.flag[p] & 3;
    const double2 xy0 = g.xy[p], n0 = g.nrm[p];
    Sym2 M = {0, 0, 0};
    Sym2 Ms[4] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    // the nearest neighbour: the first of equals in row order
    int best = -1;
    double d2best = 0.0;
    double2 dbest = make_double2(0.0, 0.0);
    for (int e = g.off[p]; e < g.off[p + 1]; ++e) {
        const double2 xyi = g.xy[g.idx[e]];
        const double dx = xyi.x - xy0.x, dy = xyi.y - xy0.y;
        const double2 t = in_frame(make_double2(dx, dy), n0);
        const uint8_t m = g.mask[e];
        M.xx = fma(dx, dx, M.xx);
        M.xy = fma(dx, dy, M.xy);
        M.yy = fma(dy, dy, M.yy);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if ((k < 2 ? xsub(m) : ysub(m)) != k) continue;
            Ms[k].xx = fma(t.x, t.x, Ms[k].xx);
            Ms[k].xy = fma(t.x, t.y, Ms[k].xy);
            Ms[k].yy = fma(t.y, t.y, Ms[k].yy);
        }
        const double d2 = dx * dx + dy * dy;
        if (best < 0 || d2 < d2best) {
            best = e;
            d2best = d2;
            dbest = make_double2(dx, dy);
        }
    }
    const double dmin = g.dmin[p];
    near_e[p] = best;
    near_u[p] = dmin > 0.0 ? make_double2(dbest.x / dmin, dbest.y / dmin) : make_double2(0.0, 0.0);
    const Sym2 Mi = inverse2(M);
    plan[p] = Mi.xx;
    plan[n + p] = Mi.xy;
    plan[2 * n + p] = Mi.yy;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        Sym2 A = {0, 0, 0};
        if (sub_needed(f, k)) A = inverse2(Ms[k]);
        double *o = plan + (3 + 3 * k) * n + p;
        o[0] = A.xx;
        o[n] = A.xy;
        o[2 * n] = A.yy;
    }
}

__device__ __forceinline__ double2 half_offset(const DevGeom &g, int e, double2 xy0)
{
    if (g.hd) return g.hd[e];
    const double2 xyi = g.xy[g.idx[e]];
    return make_double2(0.5 * (xyi.x - xy0.x), 0.5 * (xyi.y - xy0.y));
}
// D += w h for the one of two sums the edge belongs to (selects instead of two predicated sums)
__device__ __forceinline__ void add_to(bool first, bool second, double w, double2 h, double2 &D0, double2 &D1)
{
    double2 t = first ? D0 : D1;
    t.x = fma(w, h.x, t.x);
    t.y = fma(w, h.y, t.y);
    if (first) D0 = t;
    if (second) D1 = t;
}
// 2 B of a sub-stencil from D / 2, and its beta (row 0 or 1 of M^-1)
__device__ __forceinline__ Sym2 sub_back(const double *__restrict__ plan, int64_t n, double2 D, int row, double2 &beta)
{
    const Sym2 Mi = {plan[0], plan[n], plan[2 * n]};
    beta = row ? make_double2(Mi.xy, Mi.yy) : make_double2(Mi.xx, Mi.xy);
    const double2 A = times(Mi, make_double2(4.0 * D.x, 4.0 * D.y));
    return Sym2{2.0 * beta.x * A.x, fma(beta.x, A.y, beta.y * A.x), 2.0 * beta.y * A.y};
}

__global__ void __launch_bounds__(128) k_adj_weights(AdjParams P)
{
    const DevGeom &g = P.g;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.n) return;
    const bool full = P.order == 2;
    double2 xy0 = make_double2(0.0, 0.0);
    if (!g.hd) xy0 = g.xy[p];
    const double2 n0 = g.nrm[p];
    const int e0 = g.off[p], e1 = g.off[p + 1];
    double2 C0 = make_double2(0.0, 0.0), C1 = C0;   // rows of C = sum a_bar a^T
    double2 D0 = C0, D1 = C0, D2 = C0, D3 = C0;
    for (int e = e0; e < e1; ++e) {
        const double2 h = half_offset(g, e, xy0), t = in_frame(h, n0);
        const int ks = xsub(g.mask[e]), kn = ysub(g.mask[e]);
        const double2 wb = P.wbar[e];
        if (full) {
            const double2 ab = P.abar[e], a = g.lsw[e];
            C0.x = fma(ab.x, a.x, C0.x);
            C0.y = fma(ab.x, a.y, C0.y);
            C1.x = fma(ab.y, a.x, C1.x);
            C1.y = fma(ab.y, a.y, C1.y);
        }
        add_to(ks == 0, ks == 1, wb.x, t, D0, D1);
        add_to(kn == 2, kn == 3, wb.y, t, D2, D3);
    }
    const double *pl = P.plan + p;
    const int64_t n = g.n;
    Sym2 Mi = {0, 0, 0}, B = {0, 0, 0};
    if (full) {
        Mi = Sym2{pl[0], pl[n], pl[2 * n]};
        // 2 B = 2 (Mi C + (Mi C)^T), for half offsets
        const double2 b0 = times(Mi, make_double2(C0.x, C1.x)), b1 = times(Mi, make_double2(C0.y, C1.y));   // columns of Mi C
        B = Sym2{4.0 * b0.x, 2.0 * (b0.y + b1.x), 4.0 * b1.y};
    }
    double2 beta0, beta1, beta2, beta3;
    const Sym2 B0 = sub_back(pl + 3 * n, n, D0, 0, beta0), B1 = sub_back(pl + 6 * n, n, D1, 0, beta1);
    const Sym2 B2 = sub_back(pl + 9 * n, n, D2, 1, beta2), B3 = sub_back(pl + 12 * n, n, D3, 1, beta3);
    const Sym2 zero = {0.0, 0.0, 0.0};
    for (int e = e0; e < e1; ++e) {
        const double2 h = half_offset(g, e, xy0), t = in_frame(h, n0);
        const int ks = xsub(g.mask[e]), kn = ysub(g.mask[e]);
        const double2 wb = P.wbar[e];
        double2 d = P.dbar[e];
        const Sym2 X = ks == 0 ? B0 : ks == 1 ? B1 : zero, Y = kn == 2 ? B2 : kn == 3 ? B3 : zero;
        const Sym2 C = {X.xx + Y.xx, X.xy + Y.xy, X.yy + Y.yy};
        const double wx = ks >= 0 ? wb.x : 0.0, wy = kn >= 0 ? wb.y : 0.0;
        const double2 bx = ks == 0 ? beta0 : beta1, by = kn == 2 ? beta2 : beta3;
        const double gs = fma(wx, bx.x, fma(wy, by.x, -fma(C.xx, t.x, C.xy * t.y)));
        const double gn = fma(wx, bx.y, fma(wy, by.y, -fma(C.xy, t.x, C.yy * t.y)));
        if (full) {
            const double2 ab = P.abar[e], b = times(Mi, ab), c = times(B, h);
            d.x += b.x - c.x;
            d.y += b.y - c.y;
        }
        // s = d.t, n = d.n with t = (n_y, -n_x)
        d.x = fma(gs, n0.y, fma(gn, n0.x, d.x));
        d.y = fma(-gs, n0.x, fma(gn, n0.y, d.y));
        P.dbar[e] = d;
    }
}

// offsets d_e = P_dst - P_src back to points: x_bar_p = sum_in d_bar - sum_out d_bar,
// plus the per-point cotangents already gathered in pxy (internal order, or nullptr)
__global__ void __launch_bounds__(256) k_adj_points(AdjParams P, const double2 *__restrict__ pxy,
                                                    double *__restrict__ xb_out, double *__restrict__ yb_out,
                                                    int accumulate)
{
    const DevGeom &g = P.g;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.n) return;
    double xb = 0.0, yb = 0.0;
    if (pxy) {
        xb = pxy[p].x;
        yb = pxy[p].y;
    }
    for (int t = P.toff[p]; t < P.toff[p + 1]; ++t) {
        const double2 d = P.dbar[P.tedge[t]];
        xb += d.x;
        yb += d.y;
    }
    for (int e = g.off[p]; e < g.off[p + 1]; ++e) {
        const double2 d = P.dbar[e];
        xb -= d.x;
        yb -= d.y;
    }
    const int32_t o = P.perm[p];
    if (xb_out) xb_out[o] = accumulate ? xb_out[o] + xb : xb;
    if (yb_out) yb_out[o] = accumulate ? yb_out[o] + yb : yb;
}

// q_bar to U_bar through E13, adds into Ub_acc ([n][4], internal order). With
// p = (gamma-1) (E - m^2/(2 rho)), m^2 = m1^2 + m2^2 and g = 1/(gamma-1):
//   q1 = ln rho + g ln(rho/(2p)) - m^2/(2 rho p), q2 = m1/p, q3 = m2/p, q4 = -rho/p,
// in reverse by hand (45 FP64 operations and two reciprocals per point)
// 1/x by the integer pipes, within 2^-59 before the rounding; extreme x divide.
// (k_adj_state, bound by the FP64 pipe, with two of them and 1/inv_gm1 from the
// host: 71 -> 52 us at 640k points)
__device__ __forceinline__ double reciprocal(double x) { return fix_moderate(x) ? fix_reciprocal(x) : 1.0 / x; }

template <class T>
__global__ void __launch_bounds__(256) k_adj_state(AdjParamsT<T> P, const double *__restrict__ U,
                                                   double *__restrict__ Ub_acc)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n = P.g.n;
    if (p >= n) return;
    double u[4], qb[4], ub[4];
    ld4(U, p, u);
    T qt[4];
    ld4(P.qbar, p, qt);
#pragma unroll
    for (int k = 0; k < 4; ++k) qb[k] = to_f64(qt[k]);
    if (P.qbar2) {
        ld4(P.qbar2, p, qt);
#pragma unroll
        for (int k = 0; k < 4; ++k) qb[k] += to_f64(qt[k]);
    }
    ld4(Ub_acc, p, ub);
    const double g = P.inv_gm1, gm1 = P.gm1;
    const double ir = reciprocal(u[0]), m1 = u[1] * ir, m2 = u[2] * ir;            // velocities
    const double ke = 0.5 * (u[1] * m1 + u[2] * m2);                          // m^2/(2 rho)
    const double pr = gm1 * (u[3] - ke), ip = reciprocal(pr);
    const double kp = ke * ip;                                                // m^2/(2 rho p)
    // cotangents at fixed p, and that of p
    const double rb = qb[0] * ir * (1.0 + g + kp) - qb[3] * ip;
    const double ab = ip * (qb[1] - qb[0] * m1), bb = ip * (qb[2] - qb[0] * m2);
    const double pb = ip * (qb[0] * (kp - g) - ip * (qb[1] * u[1] + qb[2] * u[2] - qb[3] * u[0]));
    // p through rho, m and E
    const double c = gm1 * pb;
    ub[0] += rb + c * (0.5 * (m1 * m1 + m2 * m2));
    ub[1] += ab - c * m1;
    ub[2] += bb - c * m2;
    ub[3] += c;
    st4(Ub_acc, p, ub);
}

// ---------------------------------------------------------------------------
// transpose CSR: incoming edges of every point, in edge order
// ---------------------------------------------------------------------------
__global__ void k_edge_src(int64_t n, const int32_t *__restrict__ off, int32_t *__restrict__ esrc)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    for (int e = off[p]; e < off[p + 1]; ++e) esrc[e] = (int32_t)p;
}

__global__ void k_iota(int64_t m, int32_t *__restrict__ v)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m) v[t] = (int32_t)t;
}

// toff[p] = first position of key p in the sorted keys (lower bound)
__global__ void k_toff(int64_t n, int64_t nnz, const int32_t *__restrict__ keys, int32_t *__restrict__ toff)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p > n) return;
    int64_t lo = 0, hi = nnz;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (keys[mid] < p) lo = mid + 1;
        else hi = mid;
    }
    toff[p] = (int32_t)lo;
}

__global__ void k_tsrc(int64_t nnz, const int32_t *__restrict__ tedge, const int32_t *__restrict__ esrc,
                       int32_t *__restrict__ tsrc)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nnz) tsrc[t] = esrc[tedge[t]];
}

// weights and half offset of incoming edge t (edge tedge[t] of point tsrc[t])
__global__ void k_incoming(int64_t nnz, DevGeom g, const int32_t *__restrict__ tedge, const int32_t *__restrict__ tsrc,
                           double2 *__restrict__ tlsw, double2 *__restrict__ thd)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nnz) return;
    const int e = tedge[t];
    tlsw[t] = g.lsw[e];
    thd[t] = edge_half_offset(g, e, tsrc[t]);
}

// the FP32 product's copies: the FP64 offsets and weights rounded once
__global__ void k_float_edges(DevGeom g, float4 *__restrict__ ef, float2 *__restrict__ ea)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.n) return;
    const double2 P0 = g.xy[p];
    for (int e = g.off[p]; e < g.off[p + 1]; ++e) {
        const double2 a = g.lsw[e];
        ef[e] = float_edge(g, e, g.idx[e], P0);
        ea[e] = make_float2((float)a.x, (float)a.y);
    }
}

__global__ void k_float_incoming(int64_t nnz, DevGeom g, const int32_t *__restrict__ tedge,
                                 const int32_t *__restrict__ tsrc, float4 *__restrict__ tf)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nnz) tf[t] = float_incoming(g, tedge[t], tsrc[t]);
}

unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t build_transpose_csr(int64_t n, int64_t nnz, const int32_t *off, const int32_t *idx, int32_t *toff,
                                int32_t *tedge, int32_t *tsrc, cudaStream_t s)
{
    int32_t *esrc = nullptr, *iota = nullptr, *keys = nullptr;
    void *tmp = nullptr;
    size_t tmp_bytes = 0;
    cudaError_t err = cudaSuccess;
    const int64_t m = nnz > 0 ? nnz : 1;
    do {
        if ((err = cudaMallocAsync(&esrc, m * sizeof(int32_t), s)) != cudaSuccess) break;
        if ((err = cudaMallocAsync(&iota, m * sizeof(int32_t), s)) != cudaSuccess) break;
        if ((err = cudaMallocAsync(&keys, m * sizeof(int32_t), s)) != cudaSuccess) break;
        k_edge_src<<<blocks(n, 256), 256, 0, s>>>(n, off, esrc);
        k_iota<<<blocks(m, 256), 256, 0, s>>>(nnz, iota);
        if ((err = cudaGetLastError()) != cudaSuccess) break;
        if (nnz > 0) {
            // stable: equal destinations keep edge order
            err = cub::DeviceRadixSort::SortPairs(nullptr, tmp_bytes, idx, keys, iota, tedge, (int)nnz, 0, 32, s);
            if (err != cudaSuccess) break;
            if ((err = cudaMallocAsync(&tmp, tmp_bytes, s)) != cudaSuccess) break;
            err = cub::DeviceRadixSort::SortPairs(tmp, tmp_bytes, idx, keys, iota, tedge, (int)nnz, 0, 32, s);
            if (err != cudaSuccess) break;
        }
        k_toff<<<blocks(n + 1, 256), 256, 0, s>>>(n, nnz, keys, toff);
        if (nnz > 0) k_tsrc<<<blocks(nnz, 256), 256, 0, s>>>(nnz, tedge, esrc, tsrc);
        err = cudaGetLastError();
    } while (0);
    if (tmp) cudaFreeAsync(tmp, s);
    if (keys) cudaFreeAsync(keys, s);
    if (iota) cudaFreeAsync(iota, s);
    if (esrc) cudaFreeAsync(esrc, s);
    return err;
}

cudaError_t build_incoming(const DevGeom &g, int64_t nnz, const int32_t *tedge, const int32_t *tsrc, double2 *tlsw,
                           double2 *thd, cudaStream_t s)
{
    if (nnz <= 0) return cudaSuccess;
    k_incoming<<<blocks(nnz, 256), 256, 0, s>>>(nnz, g, tedge, tsrc, tlsw, thd);
    return cudaGetLastError();
}

cudaError_t build_adj_plan(const DevGeom &g, double *plan, int32_t *near_e, double2 *near_u, cudaStream_t s)
{
    k_adj_plan<<<blocks(g.n, 128), 128, 0, s>>>(g, plan, near_e, near_u);
    return cudaGetLastError();
}

cudaError_t build_float_geometry(const DevGeom &g, int64_t nnz, const int32_t *tedge, const int32_t *tsrc, float4 *ef,
                                 float2 *ea, float4 *tf, cudaStream_t s)
{
    if (nnz <= 0) return cudaSuccess;
    k_float_edges<<<blocks(g.n, 128), 128, 0, s>>>(g, ef, ea);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    k_float_incoming<<<blocks(nnz, 256), 256, 0, s>>>(nnz, g, tedge, tsrc, tf);
    return cudaGetLastError();
}

// launches the kernel of T that fits: with the FP32 copies or without
template <class T, bool GEOM, bool COPIES>
static void adj_flux_owner(const AdjParamsT<T> &P, cudaStream_t s)
{
    if constexpr (std::is_same<T, double>::value) {
        if (P.g14) {
            k_adj_flux_pair<GEOM><<<blocks(P.g.n, 64), 128, 0, s>>>(P);
            return;
        }
    }
    k_adj_flux<T, GEOM, COPIES><<<blocks(P.g.n, 128), 128, 0, s>>>(P);
}
template <class T, bool GEOM, bool COPIES>
static void adj_flux_gather(const AdjParamsT<T> &P, cudaStream_t s)
{
    if constexpr (GEOM && std::is_same<T, double>::value) k_adj_flux_gather_pair<<<blocks(P.g.n, 64), 128, 0, s>>>(P);
    else k_adj_flux_gather<T, GEOM, COPIES><<<blocks(P.g.n, 128), 128, 0, s>>>(P);
}
template <class T, bool COPIES>
static cudaError_t adj_flux(const AdjParamsT<T> &P, bool geom, cudaStream_t s)
{
    if (geom) adj_flux_owner<T, true, COPIES>(P, s);
    else adj_flux_owner<T, false, COPIES>(P, s);
    const cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    if (geom && P.order == 2) adj_flux_gather<T, true, COPIES>(P, s);   // (order 1 has no offsets)
    else adj_flux_gather<T, false, COPIES>(P, s);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_adj_flux(const AdjParamsT<T> &P, bool geom, cudaStream_t s)
{
    if constexpr (std::is_same<T, float>::value) {
        if (!P.ef) return adj_flux<T, false>(P, geom, s);
    }
    return adj_flux<T, true>(P, geom, s);
}

template <class T>
cudaError_t launch_adj_grad(const AdjParamsT<T> &P, const T *gprev, const T *gbar_in, T *gbar_out, bool geom,
                            bool first, cudaStream_t s)
{
    const int f = first ? 1 : 0;
    const unsigned nb = blocks(P.g.n, 128);
    if constexpr (std::is_same<T, double>::value) {
        const dim3 pairs(blocks(P.g.n, 64), 2);
        if (geom) k_adj_grad_fp64<true><<<pairs, 128, 0, s>>>(P, gprev, gbar_in, gbar_out, f);
        else k_adj_grad_fp64<false><<<pairs, 128, 0, s>>>(P, gprev, gbar_in, gbar_out, f);
    } else if (P.ef) {
        if (geom) k_adj_grad_fp32<true, true><<<nb, 128, 0, s>>>(P, gprev, gbar_in, gbar_out, f);
        else k_adj_grad_fp32<false, true><<<nb, 128, 0, s>>>(P, gprev, gbar_in, gbar_out, f);
    } else {
        if (geom) k_adj_grad_fp32<true, false><<<nb, 128, 0, s>>>(P, gprev, gbar_in, gbar_out, f);
        else k_adj_grad_fp32<false, false><<<nb, 128, 0, s>>>(P, gprev, gbar_in, gbar_out, f);
    }
    return cudaGetLastError();
}

cudaError_t launch_adj_limit(const AdjParams &P, const double *graw, const double *gbar_in, double *gbar_out,
                             int32_t *lidx, double *lval, double limK, cudaStream_t s)
{
    k_adj_limit<<<blocks(P.g.n, 32), 128, 0, s>>>(P, graw, gbar_in, gbar_out, lidx, lval, limK);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    k_adj_limit_gather<<<blocks(P.g.n, 128), 128, 0, s>>>(P, lidx, lval);
    return cudaGetLastError();
}

cudaError_t launch_adj_weights(const AdjParams &P, cudaStream_t s)
{
    k_adj_weights<<<blocks(P.g.n, 128), 128, 0, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_adj_points(const AdjParams &P, const double2 *pxy, double *x_bar, double *y_bar, bool accumulate,
                              cudaStream_t s)
{
    k_adj_points<<<blocks(P.g.n, 256), 256, 0, s>>>(P, pxy, x_bar, y_bar, accumulate ? 1 : 0);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_adj_state(const AdjParamsT<T> &P, const double *U, double *Ub_acc, cudaStream_t s)
{
    k_adj_state<T><<<blocks(P.g.n, 256), 256, 0, s>>>(P, U, Ub_acc);
    return cudaGetLastError();
}

__global__ void k_to_float(int64_t m, const double *__restrict__ a, float *__restrict__ b)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m) b[t] = (float)a[t];
}

cudaError_t launch_to_float(int64_t m, const double *a, float *b, cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    k_to_float<<<blocks(m, 256), 256, 0, s>>>(m, a, b);
    return cudaGetLastError();
}

template cudaError_t launch_adj_flux<double>(const AdjParamsT<double> &, bool, cudaStream_t);
template cudaError_t launch_adj_flux<float>(const AdjParamsT<float> &, bool, cudaStream_t);
template cudaError_t launch_adj_grad<double>(const AdjParamsT<double> &, const double *, const double *, double *, bool,
                                             bool, cudaStream_t);
template cudaError_t launch_adj_grad<float>(const AdjParamsT<float> &, const float *, const float *, float *, bool,
                                            bool, cudaStream_t);
template cudaError_t launch_adj_state<double>(const AdjParamsT<double> &, const double *, double *, cudaStream_t);
template cudaError_t launch_adj_state<float>(const AdjParamsT<float> &, const double *, double *, cudaStream_t);

// ---------------------------------------------------------------------------
// pseudo-time update in forward (stage states for the reverse sweep) and in
// reverse. A stage maps U^n and a residual R to
//   U' = P(U^n - c dt R),
// P the boundary treatment: wall points lose the normal momentum (a symmetric
// projection), far-field points are reset to the free stream (no dependence).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_stage_fwd(StageParams S, const double *__restrict__ Un,
                                                   const double *__restrict__ R, double c,
                                                   double *__restrict__ Uout)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= S.n) return;
    const uint8_t f = S.flag[p] & 3;
    double u[4], r[4], o[4];
    ld4(Un, p, u);
    ld4(R, p, r);
    const double cdt = c * S.dt[p];
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = u[k] - cdt * r[k];
    if (f == FLAG_WALL) {
        const double2 n0 = S.nrm[p];
        const double mn = o[1] * n0.x + o[2] * n0.y;
        o[1] = o[1] - mn * n0.x;
        o[2] = o[2] - mn * n0.y;
    } else if (f == FLAG_FARFIELD) {
        const double *Ui = S.case_uinf ? S.case_uinf + 4 * (int)S.pcase[p] : S.Uinf;
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = Ui[k];
    }
    st4(Uout, p, o);
}

// reverse of one stage: v = P^T Ub_out; Uacc += v; dtbar (+)= -c sum_k R_k v_k;
// Rbar (+)= -c dt v (assigned when init, else added)
__global__ void __launch_bounds__(256) k_stage_adj(StageParams S, const double *__restrict__ Ub_out,
                                                   const double *__restrict__ R, double c, int init,
                                                   double *__restrict__ Uacc, double *__restrict__ dtbar,
                                                   double *__restrict__ Rbar)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= S.n) return;
    const uint8_t f = S.flag[p] & 3;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (f != FLAG_FARFIELD) {
        ld4(Ub_out, p, v);
        if (f == FLAG_WALL) {
            const double2 n0 = S.nrm[p];
            const double mn = v[1] * n0.x + v[2] * n0.y;
            v[1] = v[1] - mn * n0.x;
            v[2] = v[2] - mn * n0.y;
        }
    }
    double a[4], r[4], rb[4] = {0.0, 0.0, 0.0, 0.0};
    ld4(Uacc, p, a);
    ld4(R, p, r);
    if (!init) ld4(Rbar, p, rb);
    const double dt = S.dt[p];
    double tb = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        a[k] += v[k];
        tb -= c * r[k] * v[k];
        rb[k] -= c * dt * v[k];
    }
    st4(Uacc, p, a);
    st4(Rbar, p, rb);
    dtbar[p] = init ? tb : dtbar[p] + tb;
}

// reverse of the last RK4 stage U^{n+1} = P(U^n - dt/6 (R0 + 2 R1 + 2 R2 + R3))
__global__ void __launch_bounds__(256) k_stage_adj_rk4_final(StageParams S, const double *__restrict__ Ub_out,
                                                             const double *__restrict__ R0,
                                                             const double *__restrict__ R1,
                                                             const double *__restrict__ R2,
                                                             const double *__restrict__ R3,
                                                             double *__restrict__ Uacc, double *__restrict__ dtbar,
                                                             double *__restrict__ Rb0, double *__restrict__ Rb1,
                                                             double *__restrict__ Rb2, double *__restrict__ Rb3)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= S.n) return;
    const uint8_t f = S.flag[p] & 3;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (f != FLAG_FARFIELD) {
        ld4(Ub_out, p, v);
        if (f == FLAG_WALL) {
            const double2 n0 = S.nrm[p];
            const double mn = v[1] * n0.x + v[2] * n0.y;
            v[1] = v[1] - mn * n0.x;
            v[2] = v[2] - mn * n0.y;
        }
    }
    double a[4], r0[4], r1[4], r2[4], r3[4], b0[4], b1[4];
    ld4(Uacc, p, a);
    ld4(R0, p, r0);
    ld4(R1, p, r1);
    ld4(R2, p, r2);
    ld4(R3, p, r3);
    const double dt = S.dt[p];
    double tb = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        a[k] += v[k];
        tb -= (r0[k] + 2.0 * r1[k] + 2.0 * r2[k] + r3[k]) * v[k] / 6.0;
        b0[k] = -dt / 6.0 * v[k];
        b1[k] = -dt / 3.0 * v[k];
    }
    st4(Uacc, p, a);
    st4(Rb0, p, b0);
    st4(Rb1, p, b1);
    st4(Rb2, p, b1);
    st4(Rb3, p, b0);
    dtbar[p] = tb;
}

// reverse of timestep(): dt = CFL dmin / (|u| + 3 sqrt(p/rho)), dmin the
// distance to the nearest neighbour (the first of equals in row order)
__global__ void __launch_bounds__(256) k_dt_adj(StageParams S, const double *__restrict__ dmin,
                                                const int32_t *__restrict__ near_e, const double2 *__restrict__ near_u,
                                                double cfl, double inv_gm1, const double *__restrict__ U, const double *__restrict__ dtbar,
                                                double *__restrict__ Uacc, double2 *__restrict__ dbar)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= S.n) return;
    const double tb = dtbar[p];
    double u[4];
    ld4(U, p, u);
    D4 Ud[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        Ud[k] = dconst(u[k]);
        Ud[k].d[k] = 1.0;
    }
    const D4 rinv = recip(Ud[0]);
    const D4 uu = Ud[1] * rinv, vv = Ud[2] * rinv;
    const D4 pr = (1.0 / inv_gm1) * (Ud[3] - 0.5 * (Ud[0] * (uu * uu + vv * vv)));
    const D4 speed = dsqrt(uu * uu + vv * vv) + 3.0 * dsqrt(pr * rinv);
    const D4 inv_speed = recip(speed);
    double a[4];
    ld4(Uacc, p, a);
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] += tb * cfl * dmin[p] * inv_speed.d[k];
    st4(Uacc, p, a);
    // dmin = |P_i - P_0| of the nearest neighbour
    const double db = tb * cfl * inv_speed.v;
    const int e = near_e[p];
    const double2 dir = near_u[p];
    double2 d = dbar[e];
    d.x = fma(db, dir.x, d.x);
    d.y = fma(db, dir.y, d.y);
    dbar[e] = d;
}

// forces: Cp_w = (p_w - p_inf)/q_inf, (fx, fy) = -sum Cp n ds, Cl = fy cos a - fx sin a,
// Cd = fx cos a + fy sin a. Per wall entry: U cotangent at the wall point and
// the cotangent of its arc-length weight ds_w
__global__ void __launch_bounds__(256) k_forces_adj(int64_t nwall, double gamma, double qinf,
                                                    const int32_t *__restrict__ wall,
                                                    const double *__restrict__ ds,
                                                    const double2 *__restrict__ nrm,
                                                    const double *__restrict__ U, double fxb, double fyb,
                                                    double *__restrict__ Uacc, double *__restrict__ dsbar)
{
    const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nwall) return;
    const int p = wall[w];
    double u[4];
    ld4(U, p, u);
    const double rho = u[0], a = u[1] / rho, b = u[2] / rho;
    const double pr = (gamma - 1.0) * (u[3] - 0.5 * rho * (a * a + b * b));
    const double c = (pr - 1.0 / gamma) / qinf;
    const double2 n = nrm[p];
    const double fn = fxb * n.x + fyb * n.y;
    const double cb = -fn * ds[w];
    dsbar[w] = -c * fn;
    const double pb = cb / qinf, gm1 = gamma - 1.0;
    double ub[4];
    ld4(Uacc, p, ub);
    ub[0] += pb * gm1 * 0.5 * (a * a + b * b);
    ub[1] += -pb * gm1 * a;
    ub[2] += -pb * gm1 * b;
    ub[3] += pb * gm1;
    st4(Uacc, p, ub);
}

// ds_w = (|P_{w+1} - P_w| + |P_w - P_{w-1}|)/2 on the closed contour: point
// cotangents of the wall coordinates (added into pxy, internal order)
__global__ void __launch_bounds__(256) k_forces_xy_adj(int64_t nwall, const int32_t *__restrict__ wall,
                                                       const double2 *__restrict__ xy,
                                                       const double *__restrict__ dsbar,
                                                       double2 *__restrict__ pxy)
{
    const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nwall) return;
    const int64_t wp = (w + nwall - 1) % nwall, wn = (w + 1) % nwall;
    const double2 P = xy[wall[w]], Pp = xy[wall[wp]], Pn = xy[wall[wn]];
    const double lp = sqrt((P.x - Pp.x) * (P.x - Pp.x) + (P.y - Pp.y) * (P.y - Pp.y));
    const double ln = sqrt((Pn.x - P.x) * (Pn.x - P.x) + (Pn.y - P.y) * (Pn.y - P.y));
    // segment (w-1, w) feeds ds_{w-1} and ds_w; segment (w, w+1) feeds ds_w and ds_{w+1}
    const double gp = 0.5 * (dsbar[wp] + dsbar[w]) / lp, gn = 0.5 * (dsbar[w] + dsbar[wn]) / ln;
    double2 o = pxy[wall[w]];
    o.x += gp * (P.x - Pp.x) - gn * (Pn.x - P.x);
    o.y += gp * (P.y - Pp.y) - gn * (Pn.y - P.y);
    pxy[wall[w]] = o;
}

cudaError_t launch_stage_fwd(const StageParams &S, const double *Un, const double *R, double c, double *Uout,
                             cudaStream_t s)
{
    k_stage_fwd<<<blocks(S.n, 256), 256, 0, s>>>(S, Un, R, c, Uout);
    return cudaGetLastError();
}

cudaError_t launch_stage_adj(const StageParams &S, const double *Ub_out, const double *R, double c, bool init,
                             double *Uacc, double *dtbar, double *Rbar, cudaStream_t s)
{
    k_stage_adj<<<blocks(S.n, 256), 256, 0, s>>>(S, Ub_out, R, c, init ? 1 : 0, Uacc, dtbar, Rbar);
    return cudaGetLastError();
}

cudaError_t launch_stage_adj_rk4_final(const StageParams &S, const double *Ub_out, const double *const R[4],
                                       double *Uacc, double *dtbar, double *const Rb[4], cudaStream_t s)
{
    k_stage_adj_rk4_final<<<blocks(S.n, 256), 256, 0, s>>>(S, Ub_out, R[0], R[1], R[2], R[3], Uacc, dtbar, Rb[0],
                                                          Rb[1], Rb[2], Rb[3]);
    return cudaGetLastError();
}

cudaError_t launch_dt_adj(const StageParams &S, const AdjParams &P, double cfl, double inv_gm1, const double *U,
                          const double *dtbar, double *Uacc, cudaStream_t s)
{
    k_dt_adj<<<blocks(S.n, 256), 256, 0, s>>>(S, P.g.dmin, P.near_e, P.near_u, cfl, inv_gm1, U, dtbar,
                                                    Uacc, P.dbar);
    return cudaGetLastError();
}

cudaError_t launch_forces_adj(int64_t nwall, double gamma, double qinf, const int32_t *wall, const double *ds,
                              const double2 *nrm, const double2 *xy, const double *U, double fxb, double fyb,
                              double *Uacc, double *dsbar, double2 *pxy, cudaStream_t s)
{
    if (nwall <= 0) return cudaSuccess;
    k_forces_adj<<<blocks(nwall, 256), 256, 0, s>>>(nwall, gamma, qinf, wall, ds, nrm, U, fxb, fyb, Uacc, dsbar);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    k_forces_xy_adj<<<blocks(nwall, 256), 256, 0, s>>>(nwall, wall, xy, dsbar, pxy);
    return cudaGetLastError();
}

}  // namespace lskum
