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
        FixEdge g;
        fix_edge(si, s0, g);
        double d[4];
        fix_flux_difference(g, si, s0, along[e] != 0, sgn[e] < 0 ? -1 : 0, d);
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

// c F through fix_align and the last product: (ci, c0) at exponent 0 -> the aligned pair's high-word products with F
extern "C" void fixed_scaled(long n, const long long *ci, const long long *c0, const long long *F, long long *gi,
                             long long *g0, int *ex)
{
    for (long e = 0; e < n; ++e) {
        int64_t a = ci[e], b = c0[e];
        ex[e] = fix_align(a, 0, b, 0);
        gi[e] = fix_mul(fix_op(a), fix_op(F[e]));
        g0[e] = fix_mul(fix_op(b), fix_op(F[e]));
    }
}
