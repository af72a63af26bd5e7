// Hot-path kernels of q-LSKUM (arXiv 2403.13287): q-derivatives (E14, E15),
// the fused flux residual + state update (E10-E12, E16 / RK4) and the
// reductions (residue, forces). One to four pairs of lanes per point in the flux
// kernel, two or four lanes in the q-derivative passes; the neighbour loop gathers
// q, q-derivatives and offsets of the stencil.
#include "lskum_device.cuh"
#include "lskum_fixed.cuh"
#include "lskum_kernels.h"

namespace lskum {

// --------------------------------------------------------------------------
// q_derivatives(): one least-squares solve of E15 per point.
//   first order (qg_old == nullptr):  grad q_0 = sum_e a_e (q_i - q_0)
//   inner iteration (Jacobi):         dq~ = dq - 1/2 [dx (qx_i - qx_0) + dy (qy_i - qy_0)]
// with the previous iterate qg_old read at every point and the new one
// written to qg_new (no point reads what this pass writes).
// --------------------------------------------------------------------------
// 1/M for a positive normal M: the approximate reciprocal of PTX
// (rcp.approx.ftz.f64) refined by two steps of Newton's iteration for 1/M,
// r <- r + r (1 - M r), each of which squares the relative error; the
// limiter's phi needs no correctly rounded quotient, and the limited
// q-derivative parity tests hold it to far below 1e-12.
__device__ __forceinline__ double rcp_newton(double M)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(M));
    double e = fma(-M, r, 1.0);
    r = fma(r, e, r);
    e = fma(-M, r, 1.0);
    return fma(r, e, r);
}

// Kinetic boundary mode: the q carried by the image (entry e of the image
// CSR) of a neighbour P_i of P_0, reconstructed (E14) with the image's half
// offset hs when recon: the reflection across the tangent line (normal n0)
// of P_i's own reconstruction q_i - h.grad q_i, h the reflection of hs
// (reflecting the gas reflects q1, q2 and every gradient, and the image of
// a field at the image of a point is the reflection of its value there);
// the free stream qf for a far-field image (zero gradient).
__device__ __forceinline__ void image_q(const DevGeom &g, int e, uint8_t m, double2 n0, const double *qf,
                                       const double *__restrict__ q, const double *__restrict__ qg, double2 hs,
                                       bool recon, double qi[4])
{
    if (m & M_IMG_FAR) {
#pragma unroll
        for (int k = 0; k < 4; ++k) qi[k] = qf[k];
        return;
    }
    const int i = g.iidx[e];
    load4(q, i, qi);
    if (recon) {
        double2 h = hs;
        reflect2(h.x, h.y, n0.x, n0.y);
        double gi[8];
        load8(qg, i, gi);
#pragma unroll
        for (int k = 0; k < 4; ++k) qi[k] = fma(-h.y, gi[4 + k], fma(-h.x, gi[k], qi[k]));
    }
    reflect2(qi[1], qi[2], n0.x, n0.y);
}

// Order-preserving integer image of a double (anything but NaN): its IEEE
// bits as a signed integer with the magnitude bits of negative values
// inverted, so that integer order is numeric order (-0 just below +0); the
// map is its own inverse. FP64 min/max issue at the FP64 rate on this part,
// 1/64 of the integer ALU rate, so the stencil extrema take this form.
__device__ __forceinline__ long long order_key(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffLL); }

// components k0 .. k0 + C - 1 (k0 a multiple of C) without an indexed array in memory
template <int C>
__device__ __forceinline__ void components(const double v[4], int k0, double o[C])
{
    if constexpr (C == 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = v[k];
    } else if constexpr (C == 2) {
        o[0] = k0 ? v[2] : v[0];
        o[1] = k0 ? v[3] : v[1];
    } else {
        const double a = (k0 & 1) ? v[1] : v[0], b = (k0 & 1) ? v[3] : v[2];
        o[0] = (k0 & 2) ? b : a;
    }
}

// Kinds of q-derivative pass (the template argument PASS): QG_INNER an inner
// iteration, QG_LIMIT the limiter applied at its end, QG_EXTREMA a first
// pass that also stores the limiter's extremum measure for a limited inner
// pass that follows.
enum { QG_LIMIT = 1, QG_INNER = 2, QG_EXTREMA = 4 };

// d_m = max_e |h_e . (sx, sy)| of each component, bit for bit the value of
// the plain FP64 loop over the edges, with FP64 products only on the edges
// that can hold the maximum. An FP32 pass bounds every edge's value: with
// a = hf_x sf and b = hf_y tf (h, sx, sy rounded to FP32), the FP32
// v = |a + b| lies within 4.01 u (|h_x sx| + |h_y sy|) of the FP64 |r_e|
// (u = 2^-24: the three roundings to FP32, the two products and the sum,
// each within u relative; r_e within 2^-52 of the exact value), and the
// margin c = 2^-20 (|a| + |b|) + 2^-120 exceeds that with room for the
// roundings of c, v - c and v + c (the absolute term covers FP32 underflow).
// So L = max_e fl(v - c) <= max_e |r_e|, and the edge holding the maximum
// has fl(v + c) >= L. A second FP32 pass marks the edges with
// !(fl(v + c) < L) (a NaN or an overflow marks the edge too); the marked
// edges (one bit each: at most LSKUM_MAX_DEGREE = 25) are then evaluated in
// FP64 exactly as the plain loop evaluates them.
template <int C>
__device__ __forceinline__ void largest_shift_screened(const DevGeom &g, int e0, int e1, const double sx[C],
                                                       const double sy[C], unsigned long long dm[C])
{
    constexpr float kMargin = 9.5367431640625e-07f;  // 2^-20 = 16 u
    constexpr float kTiny = 7.52316384526264e-37f;   // 2^-120
    float sf[C], tf[C], L[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
        sf[k] = f64_to_f32(sx[k]);
        tf[k] = f64_to_f32(sy[k]);
        L[k] = 0.0f;
    }
    for (int e = e0; e < e1; ++e) {
        const float2 h = g.hd_f[e];
#pragma unroll
        for (int k = 0; k < C; ++k) {
            const float a = h.x * sf[k], b = h.y * tf[k];
            const float c = fmaf(kMargin, fabsf(a) + fabsf(b), kTiny);
            L[k] = fmaxf(L[k], fabsf(a + b) - c);
        }
    }
    uint32_t cand[C];
#pragma unroll
    for (int k = 0; k < C; ++k) cand[k] = 0u;
    for (int e = e0; e < e1; ++e) {
        const float2 h = g.hd_f[e];
        const uint32_t bit = 1u << (e - e0);
#pragma unroll
        for (int k = 0; k < C; ++k) {
            const float a = h.x * sf[k], b = h.y * tf[k];
            const float c = fmaf(kMargin, fabsf(a) + fabsf(b), kTiny);
            if (!(fabsf(a + b) + c < L[k])) cand[k] |= bit;
        }
    }
#pragma unroll
    for (int k = 0; k < C; ++k) {
        uint32_t m = cand[k];
        while (m) {
            const int j = __ffs(m) - 1;
            m &= m - 1;
            const double2 h = g.hd[e0 + j];
            dm[k] = max(dm[k], abs_bits(fma(h.x, sx[k], h.y * sy[k])));
        }
    }
}

// One pass, by kind:
//   first:  G1 = sum_e a_e (q_i - q_0), the first-order solve;
//   inner:  G1 - sum_e a_e (h_e . grad q_i) + grad q_0 / 2, which is the sum
//           of a_e (q_i - q_0 - h_e . (grad q_i - grad q_0)) over the stencil
//           (h_e the half offset (P_i - P_0)/2): the weights a_e = M^-1 d_e,
//           M = sum_e d_e d_e^T, satisfy sum_e a_e d_e^T = I, so the terms in
//           grad q_0 add up to grad q_0 / 2, and the first-order part is the
//           stored G1 (g1) of the same state.
// The limiter scales each component of the result by Venkatakrishnan's
// phi = min over every reconstruction shift +-h_e.grad q of
// f(D, d) = (D^2 + eps^2 + 2Dd) / (D^2 + 2d^2 + Dd + eps^2), D the stencil
// maximum minus q_0 for a positive shift, the minimum minus q_0 for a
// negative one, eps^2 = (K min_e |P_i - P_0|)^3. With x = |D| and
// d = |shift|, f = N/M has N - M = d (x - 2d): f < 1 exactly when x < 2d;
// f increases in x up to x = 2d + sqrt(8d^2 + eps^2) > 2d and stays above 1
// beyond; and for fixed x < 2d it decreases in d. So phi is 1 unless
// x_m = min(D+, -D-) < 2 d_m, d_m the largest |h_e.grad q|, and then it is
// f(x_m, d_m): one quotient per component (a reciprocal and two Newton steps).
// KIN: the kinetic boundary mode (mirror images in g.ioff...; a separate
// instantiation keeps the plain kernel's registers as they are)
// The FP64 pipe bounds the pass (16 SM cycles per warp instruction). Per edge
// and component the inner pass keeps two FP64 fused multiply-adds (s -= a c);
// c = h . grad q_i comes from the integer pipes (fix_dot), q_i - q_0 of the
// first pass too where it is exact, and the limiter's quotient (fix_phi): pass
// average 0.700 -> 0.456 ms at 2.5 million points.
// LANES lanes per point, 4 / LANES components each: every lane runs the point's
// whole edge loop in row order, so the arithmetic of a component is the same
// bit for bit whatever LANES is, and a small cloud spreads over more warps with
// a shorter serial chain in each.
template <bool KIN, int PASS, int LANES>
__global__ void __launch_bounds__(128) k_qgrad(DevGeom g, const double *__restrict__ q,
                                               const double *__restrict__ qg_old, const double *__restrict__ g1,
                                               double *__restrict__ qg_new, double *__restrict__ ext, double limK,
                                               double *__restrict__ raw)
{
    constexpr bool INNER = (PASS & QG_INNER) != 0, LIMIT = (PASS & QG_LIMIT) != 0;
    constexpr bool EXTR = !INNER && (PASS & (QG_LIMIT | QG_EXTREMA)) != 0;   // extrema found here
    constexpr int C = 4 / LANES;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t p = t / LANES;
    const int k0 = (int)(t % LANES) * C;   // this lane's components: k0 .. k0 + C - 1
    if (p >= g.n) return;
    double sx[C], sy[C];
    // order keys of the largest and smallest q_i - q_0 (P_0's own difference: +0)
    long long kmax[C], kmin[C];
    const int e0 = g.off[p], e1 = g.off[p + 1];
    double2 xy0 = make_double2(0.0, 0.0);
    if ((INNER || LIMIT) && !g.hd) xy0 = g.xy[p];
    auto half_offset = [&](int e, int64_t i) {
        if (g.hd) return g.hd[e];
        const double2 xyi = g.xy[i];
        return make_double2(0.5 * (xyi.x - xy0.x), 0.5 * (xyi.y - xy0.y));
    };
    if constexpr (!INNER) {
        double q0[C];
        gather_c<C>(q + 4 * p + k0, q0);
#pragma unroll
        for (int k = 0; k < C; ++k) {
            sx[k] = sy[k] = 0.0;
            kmax[k] = kmin[k] = 0;
        }
        auto add = [&](const double *qi, double2 a) {
#pragma unroll
            for (int k = 0; k < C; ++k) {
                // on the integer pipe where that is exact (the same bits)
                const double dq = fix_same_binade(qi[k], q0[k]) ? fix_difference(qi[k], q0[k]) : qi[k] - q0[k];
                if constexpr (EXTR) {
                    const long long key = order_key(__double_as_longlong(dq));
                    kmax[k] = max(kmax[k], key);
                    kmin[k] = min(kmin[k], key);
                }
                sx[k] = fma(a.x, dq, sx[k]);
                sy[k] = fma(a.y, dq, sy[k]);
            }
        };
        for (int e = e0; e < e1; ++e) {
            double qi[C];
            gather_c<C>(q + 4 * (int64_t)g.idx[e] + k0, qi);
            add(qi, g.lsw[e]);
        }
        if constexpr (KIN) {
            // kinetic boundary mode: the mirror images of the neighbours
            const int f0 = g.ioff[p], f1 = g.ioff[p + 1];
            if (f0 < f1) {
                const double2 n0 = g.nrm[p];
                const double *qf = g.qinf + 4 * (g.pcase ? (int)g.pcase[p] : 0);
                for (int e = f0; e < f1; ++e) {
                    double qi[4], qk[C];
                    image_q(g, e, g.imask[e], n0, qf, q, nullptr, make_double2(0.0, 0.0), false, qi);
                    components<C>(qi, k0, qk);
                    add(qk, g.ilsw[e]);
                }
            }
        }
    } else {
        gather_c<C>(g1 + 8 * p + k0, sx);
        gather_c<C>(g1 + 8 * p + 4 + k0, sy);
        for (int e = e0; e < e1; ++e) {
            const int64_t i = g.idx[e];
            const double2 a = g.lsw[e];
            double gx[C], gy[C];
            gather_c<C>(qg_old + 8 * i + k0, gx);
            gather_c<C>(qg_old + 8 * i + 4 + k0, gy);
            // h . grad q_i in fixed point: half of the FP64 pipe's work moves to
            // the integer pipes, which are idle otherwise
            int64_t hx, hy;   // the half offset in its stored form, made here in mixed contexts
            if (g.hfx) {
                const longlong2 w = __ldg(g.hfx + e);
                hx = w.x;
                hy = w.y;
            } else {
                const double2 h = half_offset(e, i);
                fix_pack_pair(h.x, h.y, hx, hy);
            }
            const FixPair hp = fix_unpack_pair(hx, hy);
#pragma unroll
            for (int k = 0; k < C; ++k) {
                const FixPair gp = fix_pair(gx[k], gy[k]);
                double c = 0.0;
                if (fix_dot_in_range(hp, gp)) {
                    c = fix_dot(hp, gp);
                } else if (!fix_pair_zero(gp)) {
                    const double2 h = half_offset(e, i);
                    c = fma(h.y, gy[k], h.x * gx[k]);
                }
                sx[k] = fma(-a.x, c, sx[k]);
                sy[k] = fma(-a.y, c, sy[k]);
            }
        }
        if constexpr (KIN) {
            // a wall image's q~ is the reflection of q_i - h.grad q_i, h the
            // reflection of the image's half offset, so its correction is the
            // reflection of h.grad q_i; far-field images carry no gradient
            const int f0 = g.ioff[p], f1 = g.ioff[p + 1];
            if (f0 < f1) {
                const double2 n0 = g.nrm[p];
                for (int e = f0; e < f1; ++e) {
                    if (g.imask[e] & M_IMG_FAR) continue;
                    const double2 a = g.ilsw[e];
                    double2 h = g.ihd[e];
                    reflect2(h.x, h.y, n0.x, n0.y);
                    double gi[8], c[4], ck[C];
                    load8(qg_old, g.iidx[e], gi);
#pragma unroll
                    for (int k = 0; k < 4; ++k) c[k] = fma(-h.y, gi[4 + k], -h.x * gi[k]);
                    reflect2(c[1], c[2], n0.x, n0.y);
                    components<C>(c, k0, ck);
#pragma unroll
                    for (int k = 0; k < C; ++k) {
                        sx[k] = fma(a.x, ck[k], sx[k]);
                        sy[k] = fma(a.y, ck[k], sy[k]);
                    }
                }
            }
        }
        double tx[C], ty[C];
        gather_c<C>(qg_old + 8 * p + k0, tx);
        gather_c<C>(qg_old + 8 * p + 4 + k0, ty);
#pragma unroll
        for (int k = 0; k < C; ++k) {
            sx[k] = fma(0.5, tx[k], sx[k]);
            sy[k] = fma(0.5, ty[k], sy[k]);
        }
    }
    // x_m = min(D+, -D-) per component
    double xm[C];
    if constexpr (EXTR) {
#pragma unroll
        for (int k = 0; k < C; ++k)
            xm[k] = __longlong_as_double((long long)min((unsigned long long)kmax[k],
                                                        abs_bits(__longlong_as_double(order_key(kmin[k])))));
    }
    if constexpr (LIMIT) {
        if constexpr (INNER) gather_c<C>(ext + 4 * p + k0, xm);
        if (raw) {   // the iterate before the limiter (a reverse pass needs both)
            store_c<C>(raw + 8 * p + k0, sx);
            store_c<C>(raw + 8 * p + 4 + k0, sy);
        }
        unsigned long long dm[C];   // bits of d_m (non-negative doubles order as integers)
#pragma unroll
        for (int k = 0; k < C; ++k) dm[k] = 0;
        if (g.hd_f && e1 - e0 <= 32) {
            largest_shift_screened<C>(g, e0, e1, sx, sy, dm);
        } else {
            for (int e = e0; e < e1; ++e) {
                const double2 h = half_offset(e, g.idx[e]);
#pragma unroll
                for (int k = 0; k < C; ++k) dm[k] = max(dm[k], abs_bits(fma(h.x, sx[k], h.y * sy[k])));
            }
        }
        if constexpr (KIN) {
            for (int e = g.ioff[p]; e < g.ioff[p + 1]; ++e) {
                const double2 h = g.ihd[e];
#pragma unroll
                for (int k = 0; k < C; ++k) dm[k] = max(dm[k], abs_bits(fma(h.x, sx[k], h.y * sy[k])));
            }
        }
        const double hK = g.dmin[p] * limK;
        const double eps2 = hK * hK * hK;
#pragma unroll
        for (int k = 0; k < C; ++k) {
            // f(x, d) = N / M, N = x (x + 2d) + eps^2, M = x (x + d) + (2d^2 + eps^2):
            // in fixed point (13 FP64 instructions fewer per component), in FP64
            // for extreme exponents. Non-negative doubles order as their bits.
            const double x = xm[k], d = __longlong_as_double((long long)dm[k]);
            double phi = 1.0;
            if (fix_phi_in_range(d, eps2)) {
                if (__double_as_longlong(x) < (long long)dm[k] + (1ll << 52)) phi = fix_phi(x, d, eps2);
            } else if (x < 2.0 * d) {
                const double N = fma(x, x + 2.0 * d, eps2);
                phi = N * rcp_newton(fma(x, x + d, fma(2.0 * d, d, eps2)));
            }
            sx[k] *= phi;
            sy[k] *= phi;
        }
    } else if constexpr (EXTR) {
        store_c<C>(ext + 4 * p + k0, xm);
    }
    store_c<C>(qg_new + 8 * p + k0, sx);
    store_c<C>(qg_new + 8 * p + 4 + k0, sy);
}

// --------------------------------------------------------------------------
// flux_residual() + timestep() + state_update() (+ residue partials), fused.
// For each neighbour P_i of P_0 (frame t = (ny, -nx), n = (nx, ny)):
//   q~_i = q_i - 1/2 (dx qx_i + dy qy_i),  q~_0 = q_0 - 1/2 (dx qx_0 + dy qy_0)   (E14)
//   R += w_s [Gs(q~_i) - Gs(q~_0)] + w_n [Gn(q~_i) - Gn(q~_0)]                    (E11)
// where Gs is Gx+ or Gx- and Gn is Gy+ or Gy- by the edge's sub-stencil.
// --------------------------------------------------------------------------
struct FluxParams {
    DevGeom g;
    Gas gas;
    const double *q;    // [n][4] q of the state being evaluated
    const double *qg;   // [n][8] q-derivatives, or nullptr (first order)
    const double *Un;   // [n][4] U^n (update modes)
    double *Uout;       // [n][4] next stage state / U^{n+1}
    double *acc;        // [n][4] RK4 accumulator
    double *qout;       // [n][4] q of Uout
    double *dt;         // [n] local time step (computed at stage 0)
    double *R;          // [n][4] residual output (residual mode)
    double *norm_part;  // per warp: pair of R_rho^2 sums (stage 0), see warp_residue_pair
    int *status;        // [0] status bits, [1] smallest offending internal point
    const uint16_t *pcase;    // per point: its case in a batch, or nullptr (one case)
    const double *case_uinf;  // [cases][4] free stream per case, or nullptr (gas.Uinf)
    double cfl;
    int order;
    int mode;   // 0 residual only, 1 forward Euler, 2 RK4
    int stage;  // RK4 stage 0..3
};

__device__ __forceinline__ void flag_nonphysical(int *status, int64_t p)
{
    atomicOr(status, STATUS_NONPHYSICAL);
    atomicMin(status + 1, (int)p);
}

// The residual R of point p (one lane per point, whole warps of consecutive
// points): written out, or the time step, the state update and the residue partials
template <bool KIN>
__device__ __forceinline__ void state_update(const FluxParams &P, int64_t p, bool live, uint8_t flag, const double Rg[4])
{
    const DevGeom &g = P.g;
    if (P.mode == 0) {
        if (live) store4(P.R, p, Rg);
        return;
    }

    // ---- time step and state update ----
    if (live) {
        double Un[4], Unew[4];
        load4(P.Un, p, Un);
        double dt;
        if (P.mode == 1 || P.stage == 0) {
            // timestep(): dt = CFL min|P_i - P_0| / (|u| + 3 sqrt(p/rho))
            const double rho = Un[0], u = Un[1] / rho, v = Un[2] / rho;
            const double pr = (P.gas.gamma - 1.0) * (Un[3] - 0.5 * rho * (u * u + v * v));
            dt = P.cfl * g.dmin[p] / (sqrt(u * u + v * v) + 3.0 * sqrt(pr / rho));
            P.dt[p] = dt;
        } else {
            dt = P.dt[p];
        }
        if (P.mode == 1) {
#pragma unroll
            for (int k = 0; k < 4; ++k) Unew[k] = Un[k] - dt * Rg[k];
        } else {
            double a[4];
            if (P.stage == 0) {
#pragma unroll
                for (int k = 0; k < 4; ++k) a[k] = Rg[k];
            } else {
                load4(P.acc, p, a);
                if (P.stage < 3) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) a[k] = a[k] + 2.0 * Rg[k];
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) a[k] = a[k] + Rg[k];
                }
            }
            if (P.stage < 3) {
                store4(P.acc, p, a);
                const double c = (P.stage == 2) ? dt : 0.5 * dt;
#pragma unroll
                for (int k = 0; k < 4; ++k) Unew[k] = Un[k] - c * Rg[k];
            } else {
                const double c = dt / 6.0;
#pragma unroll
                for (int k = 0; k < 4; ++k) Unew[k] = Un[k] - c * a[k];
            }
        }
        if (flag == FLAG_WALL) {
            const double2 n0 = g.nrm[p];
            const double mn = Unew[1] * n0.x + Unew[2] * n0.y;
            Unew[1] = Unew[1] - mn * n0.x;
            Unew[2] = Unew[2] - mn * n0.y;
        } else if (flag == FLAG_FARFIELD && !KIN) {
            const double *Ui = P.case_uinf ? P.case_uinf + 4 * (int)P.pcase[p] : P.gas.Uinf;
#pragma unroll
            for (int k = 0; k < 4; ++k) Unew[k] = Ui[k];
        }
        store4(P.Uout, p, Unew);
        double qn[4];
        if (!q_from_U(Unew, P.gas, qn)) flag_nonphysical(P.status, p);
        store4(P.qout, p, qn);
    }

    // ---- residue partials: a pair of R_rho^2 sums per warp, at stage 0 ----
    if (P.mode == 1 || P.stage == 0) warp_residue_pair(P.pcase, p, live, Rg[0] * Rg[0], P.norm_part);
}

// One member's term of E11 is w_s [Gs(q~_i) - Gs(q~_0)] + w_n [Gn(q~_i) - Gn(q~_0)],
// Gs = Gx+ or Gx- and Gn = Gy+ or Gy- by the member's sub-stencil bits m, in
// the frame (t, n) of P_0.
struct Vec4 {
    double v[4];
};
struct StateFluxes {
    double t[4], n[4];   // [mass, along, transverse, energy]
    bool ok;
};

// both directions' split fluxes of one state in FP64, for members outside the
// fixed-point form's ranges: each lane of a pair takes its own state, as there
// (a residual of 160k points all at Mach 7: 0.88 ms with both states in each
// lane, 0.71 ms so). Not inlined: it keeps its registers out of the loop that
// hardly ever calls it.
__device__ __noinline__ StateFluxes state_fluxes_fp64(Vec4 q, unsigned long long st, unsigned long long sn, double2 n0,
                                                      Gas gas)
{
    StateFluxes o;
    Prim s;
    o.ok = prim_from_q(q.v, gas, n0.y, -n0.x, n0, s);
    split_flux(st, s, s.us, s.un, s.Ss, o.t);
    split_flux(sn, s, s.un, s.us, s.Sn, o.n);
    return o;
}

// the member's whole term in FP64 by one lane (gamma != 1.4), R in the order
// [mass, s-momentum, n-momentum, energy]
__device__ __forceinline__ void edge_residual(const double qti[4], const double qt0[4], uint8_t m, double2 w,
                                              double2 n0, double tx, double ty, const Gas &gas, double R[4],
                                              bool &ok)
{
    // equal reconstructed states have dG = 0 exactly (compared as bit patterns,
    // on the integer pipe; +0 against -0 only costs a flux evaluation giving dG = 0)
    if (((__double_as_longlong(qti[0]) ^ __double_as_longlong(qt0[0])) |
         (__double_as_longlong(qti[1]) ^ __double_as_longlong(qt0[1])) |
         (__double_as_longlong(qti[2]) ^ __double_as_longlong(qt0[2])) |
         (__double_as_longlong(qti[3]) ^ __double_as_longlong(qt0[3]))) == 0)
        return;
    Prim si, s0;
    ok &= prim_from_q(qti, gas, tx, ty, n0, si);
    ok &= prim_from_q(qt0, gas, tx, ty, n0, s0);
    // w != 0 tested on the bits (integer pipe; +-0 are the zeros)
    if ((__double_as_longlong(w.x) & ~(long long)kSignBit) != 0) {
        const unsigned long long sg = (m & M_XPOS) ? 0ull : kSignBit;
        double Gi[4], G0[4];
        split_flux(sg, si, si.us, si.un, si.Ss, Gi);
        split_flux(sg, s0, s0.us, s0.un, s0.Ss, G0);
#pragma unroll
        for (int k = 0; k < 4; ++k) R[k] += w.x * __dsub_rn(Gi[k], G0[k]);
    }
    if ((__double_as_longlong(w.y) & ~(long long)kSignBit) != 0) {
        const unsigned long long sg = (m & M_YPOS) ? 0ull : kSignBit;
        double Gi[4], G0[4];
        split_flux(sg, si, si.un, si.us, si.Sn, Gi);
        split_flux(sg, s0, s0.un, s0.us, s0.Sn, G0);
        // Gn components are [mass, n-momentum, s-momentum, energy]
        R[0] += w.y * __dsub_rn(Gi[0], G0[0]);
        R[1] += w.y * __dsub_rn(Gi[2], G0[2]);
        R[2] += w.y * __dsub_rn(Gi[1], G0[1]);
        R[3] += w.y * __dsub_rn(Gi[3], G0[3]);
    }
}

__device__ __forceinline__ uint32_t other_lane(uint32_t v) { return __shfl_xor_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ int64_t other_lane(int64_t v)
{
    const uint32_t lo = other_lane((uint32_t)v), hi = other_lane((uint32_t)((uint64_t)v >> 32));
    return (int64_t)(((uint64_t)hi << 32) | lo);
}
__device__ __forceinline__ double other_lane(double v)
{
    return __longlong_as_double(other_lane((int64_t)__double_as_longlong(v)));
}

// (u.t, u.n) of a q-vector, u = -(q2, q3)/q4. Not inlined: hardly ever needed, and
// the loop that calls it has no registers to spare
__device__ __noinline__ double2 frame_velocity(double q2, double q3, double q4, double2 n0)
{
    const double r = -1.0 / q4;
    return make_double2(fma(q2, n0.y, -(q3 * n0.x)) * r, fma(q2, n0.x, q3 * n0.y) * r);
}

// One member of a point's stencil, evaluated by two neighbouring lanes: lane 0
// holds the neighbour's reconstructed state, lane 1 the point's own one (qt).
// Each turns its state into fixed point and forms the products c F of both
// directions; then lane 0 takes the difference of the fluxes along t, lane 1
// that along n: d = [mass, along, transverse, energy]. Called by whole warps;
// act is the same in both lanes of a pair, and pairs without a member
// (act = false) take part in the shuffles only and get d = 0.
__device__ __forceinline__ void member_difference(bool act, int l, const double qt[4], uint32_t m, double2 w, double2 n0,
                                                  FixOp nx, FixOp ny, const Gas &gas, double d[4], bool &ok)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = 0.0;
    // equal reconstructed states have dG = 0 exactly (compared as bit patterns);
    // the last component decides almost always
    // (every lane takes part in every shuffle and vote: no && or ?: before them)
    const int64_t other3 = other_lane((int64_t)__double_as_longlong(qt[3]));
    bool differ = act && other3 != __double_as_longlong(qt[3]);
    if (__any_sync(0xffffffffu, act && !differ)) {
        bool any = false;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int64_t o = other_lane((int64_t)__double_as_longlong(qt[k]));
            any |= o != __double_as_longlong(qt[k]);
        }
        differ = act && (differ || any);
    }
    if (!__any_sync(0xffffffffu, differ)) return;
    const bool xp = (m & M_XPOS) != 0, yp = (m & M_YPOS) != 0;
    const unsigned long long sbit = (l ? yp : xp) ? 0ull : kSignBit;   // of this lane's direction
    FixState s;
    bool fixed = fix_state(qt, nx, ny, s);
    // (bit 0: in range; bits 1 and 2: slow along t and along n)
    const uint32_t mine = (fixed ? 1u : 0u) | (fix_slow(s.St) ? 2u : 0u) | (fix_slow(s.Sn) ? 4u : 0u);
    const uint32_t both = mine & other_lane(mine);
    fixed = (both & 1u) != 0;
    if (__any_sync(0xffffffffu, differ && fixed)) {
        if (!fixed) s.St = s.Sn = 0;   // an index of the tables; the result is not used
        // the two states' factors at common exponents
        const int en = (int)other_lane((uint32_t)s.n), ek = (int)other_lane((uint32_t)s.k);
        int e0, e1, e3;
        const int64_t c0 = fix_align_half(s.c0, fix_e0(s.n, s.k), fix_e0(en, ek), e0);
        const int64_t c1 = fix_align_half(s.c1, fix_e1(s.n, s.k), fix_e1(en, ek), e1);
        const int64_t c3 = fix_align_half(s.c3, fix_e3(s.n, s.k), fix_e3(en, ek), e3);
        const int z0 = fix_top(c0, other_lane((uint32_t)((uint64_t)c0 >> 32)));
        const int z1 = fix_top(c1, other_lane((uint32_t)((uint64_t)c1 >> 32)));
        const int z3 = fix_top(c3, other_lane((uint32_t)((uint64_t)c3 >> 32)));
        const FixOp o0 = fix_op(c0 << z0), o1 = fix_op(c1 << z1), o3 = fix_op(c3 << z3);
        int64_t Ft[4], Fn[4];
        fix_parts(s.St, xp ? 0 : -1, s.Sn, s.H, Ft);
        fix_scale(o0, o1, o3, Ft);
        fix_parts(s.Sn, yp ? 0 : -1, s.St, s.H, Fn);
        fix_scale(o0, o1, o3, Fn);
        // lane 0: G_t(neighbour) - G_t(own), lane 1: G_n(neighbour) - G_n(own);
        // the products lack the factor sgn of components 0, 2 and 3
        const bool use = differ && fixed;
        // both transverse velocities small: that momentum's flux as velocity times
        // mass flux in FP64 (fix_slow says why; a step of 2.5 million points 16.10 ->
        // 16.27 ms, and 16.41 with this after the loop, which spills more)
        const bool slow_o = use && (both & (l ? 2u : 4u)) != 0;
        double d2 = 0.0;
        if (__any_sync(0xffffffffu, slow_o)) {
            const double2 u = frame_velocity(qt[1], qt[2], qt[3], n0);
            const double gt = fix_to_double(Ft[0], e0 - z0 + 2) * u.y, gn = fix_to_double(Fn[0], e0 - z0 + 2) * u.x;
            const double r = other_lane(l ? gt : gn);
            d2 = l ? __dsub_rn(r, gn) : __dsub_rn(gt, r);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t r = other_lane(l ? Ft[k] : Fn[k]);
            const double v =
                fix_to_double(l ? r - Fn[k] : Ft[k] - r, k == 0 ? e0 - z0 + 2 : k == 3 ? e3 - z3 + 5 : e1 - z1 + 4);
            if (use) d[k] = k == 1 ? v : flip_sign(k == 2 && slow_o ? d2 : v, sbit);
        }
    }
    const bool slow = differ && !fixed;
    if (__any_sync(0xffffffffu, slow)) {
        StateFluxes f;
#pragma unroll
        for (int k = 0; k < 4; ++k) f.t[k] = f.n[k] = 0.0;
        if (slow) {
            Vec4 q;
#pragma unroll
            for (int k = 0; k < 4; ++k) q.v[k] = qt[k];
            f = state_fluxes_fp64(q, xp ? 0ull : kSignBit, yp ? 0ull : kSignBit, n0, gas);
            ok &= f.ok;
        }
        // an unfused subtraction of the two rounded fluxes, so equal states give
        // exactly zero (a contracted fma(rho_i, m_i, -rho_0 m_0) would leave a
        // product's rounding); a direction of weight zero adds nothing, whatever
        // its difference
        const bool use = slow && (__double_as_longlong(l ? w.y : w.x) & ~(long long)kSignBit) != 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double r = other_lane(l ? f.t[k] : f.n[k]);
            const double v = l ? __dsub_rn(r, f.n[k]) : __dsub_rn(f.t[k], r);
            if (use) d[k] = v;
        }
    }
}

// The sums over a point's members, in row order whatever PAIRS: A[k] += w d[k].
// One pair of lanes takes its own members (all four components). Several pairs
// hand their differences over through shared memory, and pair p sums component
// p of all of them (2 pairs: 2p and 2p + 1), so that no addition is done
// twice: by shuffles each lane summed everything, PAIRS times the FP64 work (4
// pairs 29.1 -> 25.6 us at 3k points, 38.1 -> 34.1 at 10k; 2 pairs 71.8 -> 69.4 at 40k).
template <int PAIRS>
struct Members {
    static constexpr int C = PAIRS == 1 ? 4 : PAIRS == 2 ? 2 : 1;   // components a lane sums
    static constexpr int kStride = 34;                              // doubles: the reads of a component meet no bank twice
    double A[C];
    __device__ __forceinline__ Members()
    {
#pragma unroll
        for (int k = 0; k < C; ++k) A[k] = 0.0;
    }
    static __device__ __forceinline__ int first() { return C * ((threadIdx.x >> 1) % PAIRS); }
    // called by whole warps; x: 5 kStride doubles of the warp's own
    __device__ __forceinline__ void add(double w, const double d[4], double *x)
    {
        if constexpr (PAIRS == 1) {
#pragma unroll
            for (int k = 0; k < 4; ++k) A[k] = fma(w, d[k], A[k]);
        } else {
            const int t = threadIdx.x & 31, base = (t & ~(2 * PAIRS - 1)) | (t & 1);
            __syncwarp();   // the last round's reads are done
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k * kStride + t] = d[k];
            x[4 * kStride + t] = w;
            __syncwarp();
            const double *row = x + first() * kStride + base;
#pragma unroll
            for (int j = 0; j < PAIRS; ++j) {
                const double wj = x[4 * kStride + base + 2 * j];
#pragma unroll
                for (int k = 0; k < C; ++k) A[k] = fma(wj, row[k * kStride + 2 * j], A[k]);
            }
        }
    }
    // all four sums of a lane's direction, in every lane
    __device__ __forceinline__ void all(double *x, double S[4]) const
    {
        if constexpr (PAIRS == 1) {
#pragma unroll
            for (int k = 0; k < 4; ++k) S[k] = A[k];
        } else {
            const int t = threadIdx.x & 31, base = (t & ~(2 * PAIRS - 1)) | (t & 1);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < C; ++k) x[(first() + k) * kStride + base] = A[k];
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 4; ++k) S[k] = x[k * kStride + base];
        }
    }
};

// What bounds it at large sizes: the FP64 pipe (68 % busy: the reconstruction,
// the sums, the state update), the integer multipliers (62 %) and ALUs (58 %),
// 66 % of the issue slots; at a few thousand points one warp's chain of rounds.
// 64 registers and a few spills, for 32 warps per SM, beat 80 (24 warps) and 128
// (16): 2.30 / 2.48 / 2.67 ms at 2.5 million points when they were compared, 2.20 now.
// One lane per member with both states took 2.58 ms and a chain twice as long.
// Two lanes per member (member_difference), PAIRS pairs of lanes per point. With
// one pair the members of a row follow one another; with 2 or 4 each pair takes
// every second or fourth, and the differences are added in row order all the
// same (Members), so that a small cloud spreads over more warps with a
// fraction of the serial chain and every launch gives the same bits. The state
// update runs afterwards with one lane per point (R through shared memory).
template <int PAIRS>
struct FluxShape {
    static constexpr int kThreads = PAIRS == 4 ? 256 : 128, kPoints = kThreads / (2 * PAIRS);
    static_assert(kPoints % 32 == 0, "whole warps of points");
};
template <bool KIN, int PAIRS>
__global__ void __launch_bounds__(FluxShape<PAIRS>::kThreads, PAIRS == 1 ? 8 : PAIRS == 2 ? 6 : 2) k_flux_update(FluxParams P)
{
    constexpr int POINTS = FluxShape<PAIRS>::kPoints;
    __shared__ double2 s_R[POINTS][2];
    constexpr int kWarps = PAIRS == 1 ? 0 : FluxShape<PAIRS>::kThreads / 32, kRow = 5 * Members<PAIRS>::kStride;
    __shared__ double s_members[kWarps * kRow + 1];
    double *const xw = s_members + (PAIRS == 1 ? 0 : (threadIdx.x >> 5) * kRow);
    const DevGeom &g = P.g;
    {
        const int l = threadIdx.x & 1, pair = (threadIdx.x >> 1) % PAIRS, pt = threadIdx.x / (2 * PAIRS);
        const int64_t pp = (int64_t)blockIdx.x * POINTS + pt, p = pp < g.n ? pp : g.n - 1;
        const uint8_t flag = g.flag[p] & 3;  // bit 7 marks FP64 closures in mixed contexts
        // far-field points are held at the free stream, except in the kinetic boundary mode
        const bool work = pp < g.n && (flag != FLAG_FARFIELD || KIN);
        const double2 n0 = g.nrm[p];
        const FixOp fnx = fix_op(fix_unit(n0.x)), fny = fix_op(fix_unit(n0.y));
        const bool second = P.order == 2;
        const int e0 = g.off[p], deg = work ? g.off[p + 1] - e0 : 0;
        double2 xy0 = make_double2(0.0, 0.0);
        if (second && !g.hd) xy0 = g.xy[p];
        Members<PAIRS> sums;
        bool ok = true;
        // whole warps go through the longest row's rounds: the members exchange by shuffles
        const int most = __reduce_max_sync(0xffffffffu, (deg + PAIRS - 1) / PAIRS);
#pragma unroll 1
        for (int r = 0; r < most; ++r) {
            const int j = r * PAIRS + pair;
            const int e = j < deg ? e0 + j : e0;
            const double2 w = g.fxw[e];
            // weights outside every needed sub-stencil are +0 exactly: tested on the bits
            const bool act = j < deg && (__double_as_longlong(w.x) | __double_as_longlong(w.y)) != 0;
            const int i = g.idx[e];
            const int64_t row = l ? p : (int64_t)i;
            double qt[4], d[4];
            gather4(P.q, row, qt);
            if (second) {
                double2 h;
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
            member_difference(act, l, qt, g.mask[e], w, n0, fnx, fny, P.gas, d, ok);
            sums.add(l ? w.y : w.x, d, xw);
        }
        if constexpr (KIN) {
            // kinetic boundary mode: the mirror images of the neighbours
            const int f0 = g.ioff[p], nim = work ? g.ioff[p + 1] - f0 : 0;
            const int imost = __reduce_max_sync(0xffffffffu, (nim + PAIRS - 1) / PAIRS);
            const double *qf = g.qinf + 4 * (g.pcase ? (int)g.pcase[p] : 0);
#pragma unroll 1
            for (int r = 0; r < imost; ++r) {
                const int j = r * PAIRS + pair;
                const bool act = j < nim;
                double2 w = make_double2(0.0, 0.0);
                uint8_t m = 0;
                double qt[4], d[4];
                gather4(P.q, p, qt);
                if (act) {
                    const int e = f0 + j;
                    w = g.ifxw[e];
                    m = g.imask[e];
                    const double2 hs = g.ihd[e];
                    if (l == 0) {
                        image_q(g, e, m, n0, qf, P.q, P.qg, hs, second, qt);
                    } else if (second) {
                        double gr[8];
                        gather8(P.qg, p, gr);
#pragma unroll
                        for (int k = 0; k < 4; ++k) qt[k] = fma(-hs.y, gr[4 + k], fma(-hs.x, gr[k], qt[k]));
                    }
                }
                member_difference(act, l, qt, m, w, n0, fnx, fny, P.gas, d, ok);
                sums.add(l ? w.y : w.x, d, xw);
            }
        }
        if (!ok) flag_nonphysical(P.status, p);
        // lane 0 holds the sums along t, lane 1 those along n: R in the order
        // [mass, s-momentum, n-momentum, energy]
        double A[4], N[4];
        sums.all(xw, A);
#pragma unroll
        for (int k = 0; k < 4; ++k) N[k] = other_lane(A[k]);
        if (threadIdx.x % (2 * PAIRS) == 0) {
            const double Rs = A[1] + N[2], Rn = A[2] + N[1];
            const double tx = n0.y, ty = -n0.x;
            s_R[pt][0] = make_double2(A[0] + N[0], Rs * tx + Rn * n0.x);
            s_R[pt][1] = make_double2(Rs * ty + Rn * n0.y, A[3] + N[3]);
        }
    }
    __syncthreads();
    if (threadIdx.x >= POINTS) return;
    const int64_t p = (int64_t)blockIdx.x * POINTS + threadIdx.x;
    const bool live = p < g.n;
    const uint8_t flag = live ? g.flag[p] & 3 : FLAG_FARFIELD;
    const double2 R01 = s_R[threadIdx.x][0], R23 = s_R[threadIdx.x][1];
    const double Rg[4] = {R01.x, R01.y, R23.x, R23.y};

    state_update<KIN>(P, p, live, flag, Rg);
}

// One lane per point, all in FP64: gamma != 1.4, which the fixed-point form does
// not cover
template <bool KIN>
__global__ void __launch_bounds__(128) k_flux_update_fp64(FluxParams P)
{
    const DevGeom &g = P.g;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double Rg[4] = {0.0, 0.0, 0.0, 0.0};
    const bool live = p < g.n;
    uint8_t flag = FLAG_FARFIELD;
    if (live) flag = g.flag[p] & 3;  // bit 7 marks FP64 closures in mixed contexts
    // far-field points are held at the free stream, except in the kinetic boundary mode
    if (live && (flag != FLAG_FARFIELD || KIN)) {
        const double2 xy0 = g.xy[p];
        const double2 n0 = g.nrm[p];
        const double tx = n0.y, ty = -n0.x;
        double q0[4], g0[8];
        load4(P.q, p, q0);
        const bool second = P.order == 2;
        if (second) load8(P.qg, p, g0);
        double R[4] = {0.0, 0.0, 0.0, 0.0};
        bool ok = true;
        const int e0 = g.off[p], e1 = g.off[p + 1];
        for (int e = e0; e < e1; ++e) {
            const double2 w = g.fxw[e];
            // weights outside every needed sub-stencil are +0 exactly: tested on the bits
            if ((__double_as_longlong(w.x) | __double_as_longlong(w.y)) == 0) continue;
            const int i = g.idx[e];
            const uint8_t m = g.mask[e];
            double qti[4], qt0[4];
            load4(P.q, i, qti);
#pragma unroll
            for (int k = 0; k < 4; ++k) qt0[k] = q0[k];
            if (second) {
                double2 h;
                if (g.hd) {
                    h = g.hd[e];
                } else {
                    const double2 xyi = g.xy[i];
                    h = make_double2(0.5 * (xyi.x - xy0.x), 0.5 * (xyi.y - xy0.y));
                }
                double gi[8];
                load8(P.qg, i, gi);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    qti[k] = fma(-h.y, gi[4 + k], fma(-h.x, gi[k], qti[k]));
                    qt0[k] = fma(-h.y, g0[4 + k], fma(-h.x, g0[k], qt0[k]));
                }
            }
            edge_residual(qti, qt0, m, w, n0, tx, ty, P.gas, R, ok);
        }
        if constexpr (KIN) {
            // kinetic boundary mode: the mirror images of the neighbours
            const int f0 = g.ioff[p], f1 = g.ioff[p + 1];
            const double *qf = g.qinf + 4 * (g.pcase ? (int)g.pcase[p] : 0);
            for (int e = f0; e < f1; ++e) {
                const double2 w = g.ifxw[e];
                const uint8_t m = g.imask[e];
                const double2 hs = g.ihd[e];
                double qti[4], qt0[4];
                image_q(g, e, m, n0, qf, P.q, P.qg, hs, second, qti);
#pragma unroll
                for (int k = 0; k < 4; ++k) qt0[k] = second ? fma(-hs.y, g0[4 + k], fma(-hs.x, g0[k], q0[k])) : q0[k];
                edge_residual(qti, qt0, m, w, n0, tx, ty, P.gas, R, ok);
            }
        }
        if (!ok) flag_nonphysical(P.status, p);
        Rg[0] = R[0];
        Rg[1] = R[1] * tx + R[2] * n0.x;
        Rg[2] = R[1] * ty + R[2] * n0.y;
        Rg[3] = R[3];
    }
    state_update<KIN>(P, p, live, flag, Rg);
}

// residue() of every case = sqrt(sum R_rho^2)/n_case from the per-warp
// pairs, in a fixed order. Case c owns points [start[c], start[c+1]); a warp
// whose first point lies in c contributes its first sum, a warp that starts
// in the case before contributes its second. Stage 1: block (j, c) sums
// chunk j (kResidueChunk warps) of case c; stage 2: one block sums each
// case's chunks and writes out[(*counter) * ncases + c], then advances the
// counter (so one captured iteration can be replayed), bounded by cap.
static constexpr int kResidueChunk = 2048;

__global__ void __launch_bounds__(256) k_residue_chunks(const double *__restrict__ part,
                                                        const int64_t *__restrict__ start, int maxchunks,
                                                        double *__restrict__ chunk)
{
    const int c = blockIdx.y, j = blockIdx.x;
    const int64_t p0 = start[c], p1 = start[c + 1];
    const int64_t w0 = p0 >> 5, w1 = (p1 - 1) >> 5;
    const int64_t a = w0 + (int64_t)j * kResidueChunk;
    const int64_t b = min(w1 + 1, a + kResidueChunk);
    double s = 0.0;
    for (int64_t w = a + threadIdx.x; w < b; w += blockDim.x) s += part[2 * w + ((w << 5) >= p0 ? 0 : 1)];
    __shared__ double sm[256];
    sm[threadIdx.x] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) sm[threadIdx.x] += sm[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) chunk[(int64_t)c * maxchunks + j] = sm[0];
}

__global__ void __launch_bounds__(256) k_residue_finish(const double *__restrict__ chunk,
                                                        const int64_t *__restrict__ start, int ncases, int maxchunks,
                                                        double *__restrict__ out_base, int *counter, int cap)
{
    __shared__ double sm[256];
    const int it = *counter;
    for (int c = 0; c < ncases; ++c) {
        const int64_t p0 = start[c], p1 = start[c + 1];
        const int64_t nw = ((p1 - 1) >> 5) - (p0 >> 5) + 1;
        const int nch = (int)((nw + kResidueChunk - 1) / kResidueChunk);
        double s = 0.0;
        for (int j = threadIdx.x; j < nch; j += blockDim.x) s += chunk[(int64_t)c * maxchunks + j];
        sm[threadIdx.x] = s;
        __syncthreads();
        for (int h = 128; h > 0; h >>= 1) {
            if (threadIdx.x < h) sm[threadIdx.x] += sm[threadIdx.x + h];
            __syncthreads();
        }
        if (threadIdx.x == 0 && it >= 0 && it < cap) out_base[(int64_t)it * ncases + c] = sqrt(sm[0]) / (double)(p1 - p0);
        __syncthreads();
    }
    if (threadIdx.x == 0) *counter = it + 1;
}

int residue_chunks(int64_t case_points) { return (int)((((case_points + 31) >> 5) + 1 + kResidueChunk - 1) / kResidueChunk); }

// q-variables of every point from U (used when a state is loaded)
__global__ void __launch_bounds__(256) k_q_from_U(int64_t n, Gas gas, const double *__restrict__ U,
                                                  double *__restrict__ q, int *status)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    double u[4], qq[4];
    load4(U, p, u);
    if (!q_from_U(u, gas, qq)) flag_nonphysical(status, p);
    store4(q, p, qq);
}

// timestep() alone: dt = CFL min|P_i - P_0| / (|u| + 3 sqrt(p/rho)) from U
__global__ void __launch_bounds__(256) k_timestep(int64_t n, Gas gas, double cfl,
                                                  const double *__restrict__ dmin,
                                                  const double *__restrict__ U, double *__restrict__ dt)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    double Un[4];
    load4(U, p, Un);
    const double rho = Un[0], u = Un[1] / rho, v = Un[2] / rho;
    const double pr = (gas.gamma - 1.0) * (Un[3] - 0.5 * rho * (u * u + v * v));
    dt[p] = cfl * dmin[p] / (sqrt(u * u + v * v) + 3.0 * sqrt(pr / rho));
}

// forces: per wall point (contour order) Cp and -Cp n ds; one block sums them
__global__ void __launch_bounds__(256) k_forces(int64_t nwall, Gas gas, double qinf,
                                                const int32_t *__restrict__ wall,
                                                const double *__restrict__ ds,
                                                const double2 *__restrict__ nrm,
                                                const double *__restrict__ U, double cosa, double sina,
                                                double *__restrict__ cp, double *__restrict__ clcd)
{
    __shared__ double sx[256], sy[256];
    double fx = 0.0, fy = 0.0;
    const double p_inf = 1.0 / gas.gamma;
    for (int64_t w = threadIdx.x; w < nwall; w += blockDim.x) {
        const int p = wall[w];
        double u[4];
        load4(U, p, u);
        const double rho = u[0], a = u[1] / rho, b = u[2] / rho;
        const double pr = (gas.gamma - 1.0) * (u[3] - 0.5 * rho * (a * a + b * b));
        const double c = (pr - p_inf) / qinf;
        cp[w] = c;
        const double2 n = nrm[p];
        fx -= c * n.x * ds[w];
        fy -= c * n.y * ds[w];
    }
    sx[threadIdx.x] = fx;
    sy[threadIdx.x] = fy;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sx[threadIdx.x] += sx[threadIdx.x + w];
            sy[threadIdx.x] += sy[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        clcd[0] = sy[0] * cosa - sx[0] * sina;
        clcd[1] = sx[0] * cosa + sy[0] * sina;
    }
}

// ----------------------------------------------------------------------------
// launchers
// ----------------------------------------------------------------------------
static inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <bool KIN, int LANES>
static void qgrad_pass(int pass, const DevGeom &g, const double *q, const double *qg_old, const double *g1,
                       double *qg_new, double *ext, double limK, double *raw, cudaStream_t s)
{
    const unsigned nb = blocks_for(LANES * g.n, 128);
    switch (pass) {
    case 0: k_qgrad<KIN, 0, LANES><<<nb, 128, 0, s>>>(g, q, qg_old, g1, qg_new, ext, limK, raw); break;
    case QG_EXTREMA: k_qgrad<KIN, QG_EXTREMA, LANES><<<nb, 128, 0, s>>>(g, q, qg_old, g1, qg_new, ext, limK, raw); break;
    case QG_LIMIT: k_qgrad<KIN, QG_LIMIT, LANES><<<nb, 128, 0, s>>>(g, q, qg_old, g1, qg_new, ext, limK, raw); break;
    case QG_INNER: k_qgrad<KIN, QG_INNER, LANES><<<nb, 128, 0, s>>>(g, q, qg_old, g1, qg_new, ext, limK, raw); break;
    default: k_qgrad<KIN, QG_INNER | QG_LIMIT, LANES><<<nb, 128, 0, s>>>(g, q, qg_old, g1, qg_new, ext, limK, raw); break;
    }
}

cudaError_t launch_qgrad(const DevGeom &g, const double *q, const double *qg_old, const double *g1,
                         double *qg_new, double *ext, double limiter_K, cudaStream_t s, double *raw)
{
    const bool inner = qg_old != nullptr, limit = limiter_K > 0.0;
    if (inner && (!g1 || (limit && !ext))) return cudaErrorInvalidValue;
    const int pass = inner ? (QG_INNER | (limit ? QG_LIMIT : 0)) : limit ? QG_LIMIT : ext ? QG_EXTREMA : 0;
    // Lanes per point (the same bits either way). A small cloud is bound by the
    // serial chain of a warp and by idle SMs, and 4 lanes shorten the one and
    // fill the other: pass average 14.4 against 18.8 us at 3k points, 18.0
    // against 19.7 at 40k, 28.8 against 30.3 at 93k. From there on (both 42.0 us at
    // 160k, 74.8 against 72.8 at 320k) the index, weight and offset work that every
    // lane repeats counts more. One lane with all four components: 27 us at 3k.
    const bool four = g.n < 120000;
    if (g.ioff) {
        if (four) qgrad_pass<true, 4>(pass, g, q, qg_old, g1, qg_new, ext, limiter_K, raw, s);
        else qgrad_pass<true, 2>(pass, g, q, qg_old, g1, qg_new, ext, limiter_K, raw, s);
    } else if (four) {
        qgrad_pass<false, 4>(pass, g, q, qg_old, g1, qg_new, ext, limiter_K, raw, s);
    } else {
        qgrad_pass<false, 2>(pass, g, q, qg_old, g1, qg_new, ext, limiter_K, raw, s);
    }
    return cudaGetLastError();
}

int64_t residue_parts(int64_t n) { return 2 * ((n + 31) / 32); }

template <int PAIRS>
static void flux_pairs(const FluxParams &P, cudaStream_t s)
{
    constexpr int T = FluxShape<PAIRS>::kThreads;
    const unsigned nb = blocks_for(P.g.n, FluxShape<PAIRS>::kPoints);
    if (P.g.ioff) k_flux_update<true, PAIRS><<<nb, T, 0, s>>>(P);
    else k_flux_update<false, PAIRS><<<nb, T, 0, s>>>(P);
}

cudaError_t launch_flux(const DevGeom &g, const Gas &gas, const FluxLaunch &L, cudaStream_t s)
{
    FluxParams P;
    P.g = g;
    P.gas = gas;
    P.q = L.q; P.qg = L.qg; P.Un = L.Un; P.Uout = L.Uout; P.acc = L.acc; P.qout = L.qout;
    P.dt = L.dt; P.R = L.R; P.norm_part = L.norm_part; P.status = L.status;
    P.pcase = L.pcase; P.case_uinf = L.case_uinf;
    P.cfl = L.cfl; P.order = L.order; P.mode = L.mode; P.stage = L.stage;
    // Pairs of lanes per point (the same bits whichever): more while the cloud
    // leaves SMs idle and the launch is one warp's serial chain. 4 / 2 pairs take
    // 25 / 38 us at 3k points, 33 / 42 at 10k, 53 / 46 at 20k and 81 / 70 at 40k,
    // 2 / 1 pairs 96 / 95 at 64k, 127 / 130 at 93k, 194 / 187 at 160k and 357 /
    // 323 at 320k (lanes without a member in a point's last round). 8 pairs gain
    // 1.4 us at 3k and lose above.
    if (!gas.g14) {
        if (g.ioff) k_flux_update_fp64<true><<<blocks_for(g.n, 128), 128, 0, s>>>(P);
        else k_flux_update_fp64<false><<<blocks_for(g.n, 128), 128, 0, s>>>(P);
    } else if (g.n < 14000) {
        flux_pairs<4>(P, s);
    } else if (g.n < 120000) {
        flux_pairs<2>(P, s);
    } else {
        flux_pairs<1>(P, s);
    }
    return cudaGetLastError();
}

cudaError_t launch_residue_finish(const double *part, const int64_t *case_start, int ncases, int maxchunks,
                                  double *chunk, double *out_base, int *counter, int cap, cudaStream_t s)
{
    k_residue_chunks<<<dim3(maxchunks, ncases), 256, 0, s>>>(part, case_start, maxchunks, chunk);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    k_residue_finish<<<1, 256, 0, s>>>(chunk, case_start, ncases, maxchunks, out_base, counter, cap);
    return cudaGetLastError();
}

cudaError_t launch_q_from_U(int64_t n, const Gas &gas, const double *U, double *q, int *status,
                            cudaStream_t s)
{
    k_q_from_U<<<blocks_for(n, 256), 256, 0, s>>>(n, gas, U, q, status);
    return cudaGetLastError();
}

cudaError_t launch_timestep(int64_t n, const Gas &gas, double cfl, const double *dmin, const double *U,
                            double *dt, cudaStream_t s)
{
    k_timestep<<<blocks_for(n, 256), 256, 0, s>>>(n, gas, cfl, dmin, U, dt);
    return cudaGetLastError();
}

cudaError_t launch_forces(int64_t nwall, const Gas &gas, double qinf, const int32_t *wall,
                          const double *ds, const double2 *nrm, const double *U, double cosa,
                          double sina, double *cp, double *clcd, cudaStream_t s)
{
    k_forces<<<1, 256, 0, s>>>(nwall, gas, qinf, wall, ds, nrm, U, cosa, sina, cp, clcd);
    return cudaGetLastError();
}

}  // namespace lskum
