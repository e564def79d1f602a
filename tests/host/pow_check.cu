// Host check of the fixed-point power (lbm_fixed.cuh; compiled with nvcc for
// the host only, no GPU): its error against long double arithmetic, over the
// shear rates and exponents of the power law, over the whole range it admits,
// and at the ends of the table intervals.  Prints the largest errors in units
// in the last place of the result.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include "lbm_fixed.cuh"

using namespace lbm;

static uint64_t bits(double x)
{
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
}
static double at(uint64_t b)
{
    double x;
    memcpy(&x, &b, 8);
    return x;
}
static double worst = 0.0;
static int bad = 0;
static void check(double x, double e)
{
    if (!pow_in_range(bits(x), bits(e))) return;
    const double got = pow_fixed(bits(x), bits(e));
    const long double want = powl((long double)x, (long double)e);
    int ex;
    frexpl(want, &ex);
    const double err = (double)(fabsl((long double)got - want) / ldexpl(1.0L, ex - 53));
    if (!(err <= worst)) worst = err;
    if (err != err) bad++;
}
static double uniform() { return drand48(); }

int main()
{
    srand48(1);
    for (int i = 0; i < 2000000; i++) check(exp((uniform() * 20.0 - 5.0)), 2.0 * uniform() - 1.0);
    const double law = worst;
    worst = 0.0;
    for (int i = 0; i < 2000000; i++) check(at(bits(1.0) + (uint64_t)(uniform() * 9007199254740992.0 * 59) ), 4.0 * uniform() - 2.0);
    for (int i = 0; i < 2000000; i++) check(at(bits(0x1p-60) + (uint64_t)(uniform() * 9007199254740992.0 * 59)), 4.0 * uniform() - 2.0);
    for (int E = -60; E < 60; E++)
        for (int j = 0; j <= 64; j++)
            for (int d = -2; d <= 2; d++)
                for (double e : {-0.4, -0.2, 0.0, 0.4, 1.0, -1.999, 1e-9, 0x1p-70, 5e-324})
                    check(at(bits(ldexp(1.0 + j / 64.0, E)) + d), e);
    const double all = worst;
    if (pow_fixed(bits(1.0), bits(0.3)) != 1.0 || pow_fixed(bits(7.5), bits(0.0)) != 1.0 ||
        pow_fixed(bits(4.0), bits(0.5)) != 2.0)
        bad++;
    for (double x : {0.0, -1.0, 0x1p60, 0x1p-61, 5e-324, (double)INFINITY, (double)NAN})
        if (pow_in_range(bits(x), bits(0.5))) bad++;
    for (double e : {2.0, -2.0, (double)INFINITY, (double)NAN})
        if (pow_in_range(bits(1.5), bits(e))) bad++;
    printf("%s law %.4f all %.4f\n", bad ? "FAILED" : "OK", law, all);
    return bad ? 1 : 0;
}
