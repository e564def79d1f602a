// Host check of what the fixed-point collision (lbm_collide_fixed.cuh) admits:
// every state it takes has to come back as the same collision in long double
// gives it, however far from ordinary flows, and every other state has to be
// refused with nothing changed.  A value that leaves its 64-bit format wraps
// by 16 of its units, which moves a population by 1e-3 at least; rounding
// moves one by less than 1e-9 (sums and products by some 2^-60; the power law,
// whose rate is clamped at gamma_1, by 2^-58 over the strain there, 5e-8 at
// the scales drawn here), so 1e-9 tells them apart.
//   rest:   fluids at rest, densities through both limits;
//   box:    populations over their whole range, heat over (-1, 1);
//   walks:  from an ordinary node along random directions, out to the limits,
//           with the last state taken and the first refused found by bisection;
//   flows:  ordinary ones, nearly all of which have to be taken.
#define main ordinary_flows
#include "fixed_check.cu"   // Par and the collision in type R
#undef main

static long g_failed = 0, g_taken = 0, g_all = 0;

static Par draw_par()
{
    const double L = 32.0 * pow(2.0, 6.0 * drand48()), Ma = 0.02 + 0.3 * drand48(), Uc = Ma / sqrt(3.0), Ra = pow(10.0, 3.0 + 3.0 * drand48());
    const double eps = drand48() < 0.3 ? 1.0 : 0.2501 + 0.74 * drand48(), n = drand48() < 0.2 ? 1.0 : 0.5 + drand48();
    const double Feps = eps < 1.0 && drand48() < 0.8 ? 1.75 / sqrt(150.0 * eps * eps * eps) : 0.0;
    return Par{eps, 6.2 * Uc * Uc / L, 1.0 / (3.0 * Uc * L / sqrt(Ra) + 0.5), 0.1 + 1.8 * drand48(), 0.1 + 1.8 * drand48(), n, L / Uc,
               6.2 / pow(sqrt(Ra), 2.0 - n) * Uc * L, pow(10.0, -3.0 + 3.0 * drand48()) * L * L, Feps, 1};
}

// Whether the state is taken; counts a failure where it comes back wrong.
static bool check(const Par &p, const FixedParams &fp, const double f[9], const double g[5], double tau, const char *what)
{
    double c[9], d[5], t = tau;
    for (int i = 0; i < 9; i++) c[i] = f[i];
    for (int i = 0; i < 5; i++) d[i] = g[i];
    const double sK = sqrt(p.K);
    const bool ok = collide_fixed(fp, 3.0 * p.nu_ref, p.Feps > 0.0, p.eps / (4.0 * p.K), p.eps / p.K, p.eps * p.Feps / (2.0 * sK),
                                  p.eps * p.Feps / sK, c, d, t);
    g_all++;
    g_taken += ok;
    bool wrong = false;
    double worst = 0.0;
    if (ok) {
        long double F[9], G[5], T = tau;
        for (int i = 0; i < 9; i++) F[i] = f[i];
        for (int i = 0; i < 5; i++) G[i] = g[i];
        plain<long double>(p, F, G, T);
        for (int i = 0; i < 9; i++) worst = fmax(worst, (double)fabsl(c[i] - F[i]));
        for (int i = 0; i < 5; i++) worst = fmax(worst, (double)fabsl(d[i] - G[i]));
        worst = fmax(worst, (double)fabsl((t - T) / T));
        wrong = !(worst < 1e-9);
    } else {
        for (int i = 0; i < 9; i++) wrong |= !(c[i] == f[i]);
        for (int i = 0; i < 5; i++) wrong |= !(d[i] == g[i]);
        wrong |= !(t == tau);
    }
    if (wrong && g_failed++ < 20) {
        double r = 0.0;
        for (int i = 0; i < 9; i++) r += f[i];
        printf("%s: %s, off by %.2e: rho %.6f f %.5f %.5f %.5f %.5f %.5f %.5f %.5f %.5f %.5f g %.4f %.4f %.4f %.4f %.4f tau %.4f eps %.3f\n", what,
               ok ? "taken" : "refused but changed", worst, r, f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], f[8], g[0], g[1], g[2], g[3],
               g[4], tau, p.eps);
    }
    return ok;
}
static FixedParams fixed_of(const Par &p)
{
    return fixed_params(p.eps, p.gbeta, p.omegaT, p.s_e, p.s_p, p.n, p.scale, 0.01, 1e6, p.clamp);
}
static const double W[9] = {4. / 9, 1. / 9, 1. / 9, 1. / 9, 1. / 9, 1. / 36, 1. / 36, 1. / 36, 1. / 36};
static const double EX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, EY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};

static void ordinary(const Par &p, double size, double f[9], double g[5], double &tau)
{
    const double vx = u(size), vy = u(size), T = 0.5 + 0.5 * u(1.0), r = 1.0 + u(0.05);
    for (int i = 0; i < 9; i++) {
        const double eu = EX[i] * vx + EY[i] * vy;
        f[i] = W[i] * r * (1.0 + 3.0 * eu + (4.5 * eu * eu - 1.5 * (vx * vx + vy * vy)) / p.eps) * (1.0 + u(0.1 * size));
    }
    for (int i = 0; i < 5; i++) g[i] = (i == 0 ? T / 3 : T / 6 * (1.0 + 3.0 * (EX[i] * vx + EY[i] * vy))) * (1.0 + u(0.1 * size));
    tau = 0.5 + 3.0 * p.nu_ref * pow(10.0, u(1.0) * (p.n - 1.0));
}

int main()
{
    srand48(11);
    // rest
    for (int k = 0; k < 400; k++) {
        const Par p = draw_par();
        const FixedParams fp = fixed_of(p);
        if (!fp.ok) g_failed++, printf("parameters refused\n");
        for (double r = 0.40; r < 2.2; r += 0.005) {
            double f[9], g[5];
            for (int i = 0; i < 9; i++) f[i] = W[i] * r;
            for (int i = 0; i < 5; i++) g[i] = i == 0 ? 1. / 6 : 1. / 12;
            check(p, fp, f, g, 0.8, "rest");
        }
    }
    // box: one to nine populations drawn large, the rest small or at rest; the
    // momentum often balanced, as it is limited
    long box0 = g_taken;
    for (long k = 0; k < 1500000; k++) {
        const Par p = draw_par();
        const FixedParams fp = fixed_of(p);
        double f[9], g[5];
        const double rho = 0.45 + 1.7 * drand48(), mix = drand48();
        double s = 0.0;
        for (int i = 0; i < 9; i++) s += f[i] = drand48() < 0.4 ? pow(2.0, -14.0 * drand48()) : drand48();
        for (int i = 0; i < 9; i++) f[i] *= rho / s;
        if (drand48() < 0.7)   // nearly balanced against the opposite direction
            for (int a : {1, 2, 5, 6}) {
                const int b = a + 2;
                const double m = 0.5 * (f[a] + f[b]), d = 0.5 * (f[a] - f[b]) * drand48() * drand48();
                f[a] = m + d;
                f[b] = m - d;
            }
        for (int i = 0; i < 9; i++) f[i] = mix * f[i] + (1.0 - mix) * W[i] * rho;
        const double T = 0.5 + 1.3 * u(1.0), wide = drand48() < 0.5 ? 1.0 : 0.1;
        for (int i = 0; i < 5; i++) g[i] = drand48() < 0.3 ? u(1.0) : (i == 0 ? T / 3 : T / 6) + wide * u(0.6);
        if (drand48() < 0.3) g[4] = T - (g[0] + g[1] + g[2] + g[3]);
        check(p, fp, f, g, drand48() < 0.5 ? 0.5 + drand48() : 0.25 * pow(2.0, 12.0 * drand48()), "box");
    }
    box0 = g_taken - box0;
    // walks
    for (int k = 0; k < 20000; k++) {
        Par p = draw_par();
        const FixedParams fp = fixed_of(p);
        double f[9], g[5], tau, df[9], dg[5];
        ordinary(p, 0.05, f, g, tau);
        const int kind = k % 4;   // all, flow alone, heat alone, one moment's direction
        for (int i = 0; i < 9; i++) df[i] = kind == 2 ? 0.0 : u(1.0) * (kind == 0 ? W[i] : 1.0);
        for (int i = 0; i < 5; i++) dg[i] = kind == 1 ? 0.0 : u(1.0);
        if (kind == 3) {
            const int m = (k / 4) % 6;
            for (int i = 0; i < 5; i++) dg[i] = 0.0;
            for (int i = 0; i < 9; i++) {
                const double e2 = EX[i] * EX[i] + EY[i] * EY[i];
                df[i] = m == 0 ? W[i] : m == 1 ? 3.0 * e2 - 4.0 : m == 2 ? 4.0 - 10.5 * e2 + 4.5 * e2 * e2 : m == 3 ? EX[i] * EX[i] - EY[i] * EY[i]
                                  : m == 4 ? EX[i] * EY[i] : W[i] * EX[i] * (k & 64 ? 1.0 : -1.0);
                if (k & 32) df[i] = -df[i];
            }
        }
        auto at = [&](double a) {
            double x[9], y[5];
            for (int i = 0; i < 9; i++) x[i] = f[i] + a * df[i];
            for (int i = 0; i < 5; i++) y[i] = g[i] + a * dg[i];
            return check(p, fp, x, y, tau, "walk");
        };
        double in = 0.0, out = -1.0;
        for (double a = 1e-3; a < 4.0; a *= 1.2)
            if (at(a))
                in = a;
            else if (out < 0.0)
                out = a;
        if (out > in)
            for (int b = 0; b < 50; b++) {
                const double a = 0.5 * (in + out);
                (at(a) ? in : out) = a;
            }
    }
    // flows
    long taken = g_taken, all = g_all;
    for (int k = 0; k < 200000; k++) {
        const Par p = draw_par();
        double f[9], g[5], tau;
        ordinary(p, pow(10.0, -8.0 + 7.0 * drand48()), f, g, tau);
        check(p, fixed_of(p), f, g, tau < 1000.0 ? tau : 1000.0, "flow");
    }
    const double part = (double)(g_taken - taken) / (g_all - all);
    if (!(part > 0.97)) g_failed++;
    printf("%s %ld failed; taken: %ld in the box, %ld in all, flows %.4f\n", g_failed ? "FAILED" : "OK", g_failed, box0, g_taken, part);
    return g_failed ? 1 : 0;
}
