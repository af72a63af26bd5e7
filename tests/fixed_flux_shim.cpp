// Host build of the fixed-point split fluxes (csrc/lskum_fixed.cuh) for the CPU tests.
#include "lskum_fixed.cuh"

using namespace lskum;

// n members: states qi, q0 ([n][4]), normals, direction (along t or n), split
// sign; dG[n][4] = G(qi) - G(q0) in [mass, along, transverse, energy], ok[n]
extern "C" void fixed_flux(long n, const double *qi, const double *q0, const double *nx, const double *ny,
                           const int *along, const int *sgn, double *dG, int *ok)
{
    for (long e = 0; e < n; ++e) {
        FixState si, s0;
        const FixOp a = fix_op(fix_unit(nx[e])), b = fix_op(fix_unit(ny[e]));
        const bool oi = fix_state(qi + 4 * e, a, b, si), o0 = fix_state(q0 + 4 * e, a, b, s0);
        ok[e] = oi && o0;
        if (!ok[e]) continue;
        // the two states' factors at common exponents, as the two lanes of the kernel share them
        int e0, e1, e3;
        int64_t ci[3] = {si.c0, si.c1, si.c3}, c0[3] = {s0.c0, s0.c1, s0.c3};
        const int ei[3] = {fix_e0(si.n, si.k), fix_e1(si.n, si.k), fix_e3(si.n, si.k)};
        const int eo[3] = {fix_e0(s0.n, s0.k), fix_e1(s0.n, s0.k), fix_e3(s0.n, s0.k)};
        int *ex[3] = {&e0, &e1, &e3};
        const int up[3] = {2, 4, 5};
        for (int j = 0; j < 3; ++j) {
            ci[j] = fix_align_half(ci[j], ei[j], eo[j], *ex[j]);
            c0[j] = fix_align_half(c0[j], eo[j], ei[j], *ex[j]);
            const int z = fix_top(ci[j], (uint32_t)((uint64_t)c0[j] >> 32));
            ci[j] <<= z;
            c0[j] <<= z;
            *ex[j] += up[j] - z;
        }
        const bool t = along[e] != 0;
        const int64_t m = sgn[e] < 0 ? -1 : 0;
        int64_t Fi[4], F0[4];
        fix_parts(t ? si.St : si.Sn, m, t ? si.Sn : si.St, si.H, Fi);
        fix_parts(t ? s0.St : s0.Sn, m, t ? s0.Sn : s0.St, s0.H, F0);
        fix_scale(fix_op(ci[0]), fix_op(ci[1]), fix_op(ci[2]), Fi);
        fix_scale(fix_op(c0[0]), fix_op(c0[1]), fix_op(c0[2]), F0);
        const int es[4] = {e0, e1, e1, e3};
        double d[4];
        for (int k = 0; k < 4; ++k) d[k] = fix_to_double(Fi[k] - F0[k], es[k]);
        const double s = sgn[e];
        dG[4 * e] = s * d[0];
        dG[4 * e + 1] = d[1];
        dG[4 * e + 2] = s * d[2];
        dG[4 * e + 3] = s * d[3];
    }
}

// the parts of one state's flux (fix_parts) for S and the transverse S in Q61, H in Q59
extern "C" void fixed_parts(long n, const long long *Sd, const long long *So, const long long *H, long long *F)
{
    for (long e = 0; e < n; ++e) {
        int64_t f[4];
        fix_parts(Sd[e], 0, So[e], H[e], f);
        for (int k = 0; k < 4; ++k) F[4 * e + k] = f[k];
    }
}

extern "C" void fixed_exp(long n, const long long *x, long long *M, int *m)
{
    for (long e = 0; e < n; ++e) M[e] = fix_exp(x[e], m[e]);
}

// c F through fix_top and the last product: (ci, c0) at exponent 0 -> the aligned pair's high-word products with F
extern "C" void fixed_scaled(long n, const long long *ci, const long long *c0, const long long *F, long long *gi,
                             long long *g0, int *ex)
{
    for (long e = 0; e < n; ++e) {
        int64_t a = ci[e], b = c0[e];
        const int z = fix_top(a, (uint32_t)((uint64_t)b >> 32));
        a <<= z;
        b <<= z;
        ex[e] = -z;
        gi[e] = fix_mul(fix_op(a), fix_op(F[e]));
        g0[e] = fix_mul(fix_op(b), fix_op(F[e]));
    }
}

// h . g of rows [hx, hy, gx, gy], h through its stored form; ok: in range
extern "C" void fixed_dot(long n, const double *a, double *c, int *ok)
{
    for (long e = 0; e < n; ++e) {
        int64_t wx, wy;
        fix_pack_pair(a[4 * e], a[4 * e + 1], wx, wy);
        const FixPair h = fix_unpack_pair(wx, wy), g = fix_pair(a[4 * e + 2], a[4 * e + 3]);
        ok[e] = fix_dot_in_range(h, g);
        c[e] = ok[e] ? fix_dot(h, g) : 0.0;
    }
}

// f(x, d) of rows [x, d, eps2] where x < 2 d
extern "C" void fixed_phi(long n, const double *a, double *f, int *ok)
{
    for (long e = 0; e < n; ++e) {
        ok[e] = fix_phi_in_range(a[3 * e + 1], a[3 * e + 2]);
        f[e] = ok[e] && a[3 * e] < 2.0 * a[3 * e + 1] ? fix_phi(a[3 * e], a[3 * e + 1], a[3 * e + 2]) : 1.0;
    }
}

extern "C" void fixed_difference(long n, const double *a, double *d, int *ok)
{
    for (long e = 0; e < n; ++e) {
        ok[e] = fix_same_binade(a[2 * e], a[2 * e + 1]);
        d[e] = ok[e] ? fix_difference(a[2 * e], a[2 * e + 1]) : 0.0;
    }
}

// rows [rho, p]: ln(rho) + 2.5 ln(rho/(2p)) and 1/rho; ok: both moderate
extern "C" void fixed_log(long n, const double *a, double *l, double *r, int *ok)
{
    for (long e = 0; e < n; ++e) {
        ok[e] = fix_moderate(a[2 * e]) && fix_moderate(a[2 * e + 1]);
        l[e] = ok[e] ? fix_log_state(a[2 * e], a[2 * e + 1]) : 0.0;
        r[e] = ok[e] ? fix_reciprocal(a[2 * e]) : 0.0;
    }
}
