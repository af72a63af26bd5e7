// Host build of what a state passes through (csrc/lskum_fixed.cuh), for the CPU tests.
#include "lskum_fixed.cuh"

using namespace lskum;

// rows [x, y]: 1/y and x/y; ok: both moderate
extern "C" void fixed_quotient(long n, const double *a, double *r, double *q, int *ok)
{
    for (long e = 0; e < n; ++e) {
        r[e] = q[e] = 0.0;
        ok[e] = fix_moderate(a[2 * e]) && fix_moderate(a[2 * e + 1]);
        if (ok[e]) fix_quotient(a[2 * e], a[2 * e + 1], r[e], q[e]);
    }
}
