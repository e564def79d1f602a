// Host check of the fixed-point collision (lbm_collide_fixed.cuh; compiled
// with nvcc for the host only, no GPU) against the same collision in long
// double, written here in moment space, and beside the plain FP64 form of
// that collision: largest and root-mean-square error of the post-collision
// populations and of the relaxation time for both, over flows near rest,
// ordinary and strong ones, both laws, both drags and several parameters.
// Values outside the admitted ranges have to be refused with nothing changed.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include "lbm_collide_fixed.cuh"

using namespace lbm;

struct Par {
    double eps, gbeta, omegaT, s_e, s_p, n, scale, nu_ref, K, Feps;
    int clamp;
};

// The collision in type R, from the moments' definitions.
template <class R>
static void plain(const Par &p, R f[9], R g[5], R &tau)
{
    const R sax = (f[1] + f[2]) + (f[3] + f[4]), sdg = (f[5] + f[6]) + (f[7] + f[8]);
    const R rho = f[0] + sax + sdg;
    const R jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]), jy = (f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8]);
    const R T = g[0] + (g[1] + g[2]) + (g[3] + g[4]);
    const R eps = R(p.eps), Gy = R(p.gbeta) * (T - R(0.5));
    const R vx = jx / rho, vy = jy / rho + eps * Gy / 2, vm = sqrt(vx * vx + vy * vy);
    const R nup = (tau - R(0.5)) / 3;
    const R c0 = R(0.5) + eps / (4 * R(p.K)) * nup, c1 = R(p.eps * p.Feps / (2.0 * sqrt(p.K)));
    const R den = c0 + sqrt(c0 * c0 + c1 * vm), ux = vx / den, uy = vy / den;
    const R drag = -(eps / R(p.K) * nup + 2 * c1 * vm / den), Fx = drag * ux, Fy = drag * uy + eps * Gy;
    const R e = 2 * sdg - 4 * f[0] - sax, ep = 4 * f[0] - 2 * sax + sdg;
    const R qx = -2 * (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]), qy = -2 * (f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8]);
    const R pxx = (f[1] + f[3]) - (f[2] + f[4]), pxy = (f[5] + f[7]) - (f[6] + f[8]);
    const R ri = rho / eps, u2 = 3 * ri * (ux * ux + uy * uy), eeq = u2 - 2 * rho, peq = rho - u2;
    const R xeq = ri * (ux * ux - uy * uy), yeq = ri * ux * uy;
    const R A = R(1.4) / 6 * (e - eeq), B = (pxx - xeq) / (2 * tau), C = (pxy - yeq) / tau;
    const R gs = 3 / rho * sqrt(A * A + B * B + C * C) * R(p.scale);
    R D;
    if (p.clamp) {
        const R gc = gs < R(0.01) ? R(0.01) : (gs > R(1e6) ? R(1e6) : gs);
        D = pow(gc, R(p.n) - 1);
    } else {
        D = gs < R(0.01) ? R(1) : (gs <= R(1e6) ? pow(gs, R(p.n) - 1) : pow(R(1e6), R(p.n) - 1));
    }
    tau = 3 * R(p.nu_ref) * D + R(0.5);
    const R w = 1 / tau, uF = ux * Fx + uy * Fy;
    const R es = e - R(1.4) * (e - eeq) + R(0.3) * 6 * ri * uF, ps = ep - R(1.4) * (ep - peq) - R(0.3) * 6 * ri * uF;
    const R jxs = rho * (ux + Fx / 2), jys = rho * (uy + Fy / 2);
    const R qxs = qx - R(1.2) * (qx + rho * ux) - R(0.4) * rho * Fx, qys = qy - R(1.2) * (qy + rho * uy) - R(0.4) * rho * Fy;
    const R xs = pxx - w * (pxx - xeq) + (1 - w / 2) * 2 * ri * (ux * Fx - uy * Fy);
    const R ys = pxy - w * (pxy - yeq) + (1 - w / 2) * ri * (ux * Fy + uy * Fx);
    const R a0 = rho / 9, a1 = es / 36, a2 = ps / 36, a3 = jxs / 6, a4 = qxs / 12, a5 = jys / 6, a6 = qys / 12, a7 = xs / 4, a8 = ys / 4;
    const R ax = a0 - a1 - 2 * a2, dg = a0 + 2 * a1 + a2;
    f[0] = a0 - 4 * a1 + 4 * a2;
    f[1] = ax + (a3 - 2 * a4) + a7;
    f[2] = ax + (a5 - 2 * a6) - a7;
    f[3] = ax - (a3 - 2 * a4) + a7;
    f[4] = ax - (a5 - 2 * a6) - a7;
    f[5] = dg + (a3 + a4) + (a5 + a6) + a8;
    f[6] = dg - (a3 + a4) + (a5 + a6) - a8;
    f[7] = dg - (a3 + a4) - (a5 + a6) + a8;
    f[8] = dg + (a3 + a4) - (a5 + a6) - a8;
    const R n1 = g[1] - g[3], n2 = g[2] - g[4], n3 = (g[1] + g[2]) + (g[3] + g[4]) - 4 * g[0], n4 = (g[1] + g[3]) - (g[2] + g[4]);
    const R wT = R(p.omegaT), n1s = n1 - wT * (n1 - T * ux), n2s = n2 - wT * (n2 - T * uy);
    const R n3s = n3 - R(p.s_e) * (n3 + 2 * T / 3), n4s = n4 - R(p.s_p) * n4;
    g[0] = T / 5 - n3s / 5;
    g[1] = T / 5 + n3s / 20 + n1s / 2 + n4s / 4;
    g[2] = T / 5 + n3s / 20 + n2s / 2 - n4s / 4;
    g[3] = T / 5 + n3s / 20 - n1s / 2 + n4s / 4;
    g[4] = T / 5 + n3s / 20 - n2s / 2 - n4s / 4;
}

static double u(double a) { return a * (2.0 * drand48() - 1.0); }

int main()
{
    srand48(7);
    const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    int failed = 0;
    long taken = 0, all = 0;
    for (int law = 0; law < 2; law++)
        for (double eps : {1.0, 0.6, 0.3})
            for (double n : {0.6, 1.0, 1.4})
                for (double size : {1e-12, 1e-6, 1e-3, 0.03, 0.1}) {
                    double top[2][3] = {}, sum[2][3] = {};
                    const double L = 64 << (int)(drand48() * 6), Uc = 0.1 / sqrt(3.0), Ra = 1e5;
                    Par p{eps, 6.2 * Uc * Uc / L, 1.0 / (3.0 * Uc * L / sqrt(Ra) + 0.5), 1.5, 1.5, n, L / Uc,
                          6.2 / pow(sqrt(Ra), 2.0 - n) * Uc * L, pow(10.0, -2.0 + u(1.0)) * L * L,
                          eps < 1.0 ? 1.75 / sqrt(150.0 * eps * eps * eps) : 0.0, law};
                    const double g1 = 0.01, g2 = 1e6;
                    const FixedParams fp = fixed_params(p.eps, p.gbeta, p.omegaT, p.s_e, p.s_p, p.n, p.scale, g1, g2, law);
                    if (fp.ok != (law == 1 || n == 1.0)) failed++;
                    if (!fp.ok) continue;   // a law with jumps: left to FP64
                    const int M = 4000;
                    for (int q = 0; q < M; q++) {
                        double f[9], g[5], tau, vx = u(size), vy = u(size), T = 0.5 + 0.5 * u(1.0), r = 1.0 + u(size);
                        for (int i = 0; i < 9; i++) {
                            const double w = i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0), eu = ex[i] * vx + ey[i] * vy;
                            f[i] = w * r * (1.0 + 3.0 * eu + (4.5 * eu * eu - 1.5 * (vx * vx + vy * vy)) / eps) * (1.0 + u(0.1 * size));
                        }
                        for (int i = 0; i < 5; i++)
                            g[i] = (i == 0 ? T / 3 : T / 6 * (1.0 + 3.0 * (ex[i] * vx + ey[i] * vy))) * (1.0 + u(0.1 * size));
                        tau = 0.5 + 3.0 * p.nu_ref * pow(10.0, u(1.0) * (n - 1.0));
                        long double F[9], G[5], t = tau;
                        double a[9], b[5], ta = tau, c[9], d[5], tc = tau;
                        for (int i = 0; i < 9; i++) F[i] = a[i] = c[i] = f[i];
                        for (int i = 0; i < 5; i++) G[i] = b[i] = d[i] = g[i];
                        plain<long double>(p, F, G, t);
                        plain<double>(p, a, b, ta);
                        const double sK = sqrt(p.K);
                        const bool ok = collide_fixed(fp, 3.0 * p.nu_ref, p.Feps > 0.0, p.eps / (4.0 * p.K),
                                                      p.eps / p.K, p.eps * p.Feps / (2.0 * sK), p.eps * p.Feps / sK, c, d, tc);
                        all++;
                        if (!ok) {
                            for (int i = 0; i < 9; i++) failed += c[i] != f[i];
                            for (int i = 0; i < 5; i++) failed += d[i] != g[i];
                            failed += tc != tau;
                            continue;
                        }
                        taken++;
                        for (int s = 0; s < 2; s++) {
                            const double *x = s ? c : a, *y = s ? d : b, tt = s ? tc : ta;
                            for (int i = 0; i < 9; i++) {
                                const double er = (double)fabsl(x[i] - F[i]);
                                top[s][0] = fmax(top[s][0], er);
                                sum[s][0] += er * er;
                            }
                            for (int i = 0; i < 5; i++) {
                                const double er = (double)fabsl(y[i] - G[i]);
                                top[s][1] = fmax(top[s][1], er);
                                sum[s][1] += er * er;
                            }
                            const double er = (double)fabsl(tt - t) / tau;
                            top[s][2] = fmax(top[s][2], er);
                            sum[s][2] += er * er;
                        }
                    }
                    // the fixed-point form may not be further off than the FP64 one, largest or on average
                    for (int k = 0; k < 3; k++) {
                        const bool worse = top[1][k] > top[0][k] * 1.05 + 1e-20 || sum[1][k] > sum[0][k] * 1.05 + 1e-38;
                        if (worse || getenv("SHOW"))
                            printf("law %d eps %.1f n %.1f size %.0e L %.0f %s: max %.2e (FP64 %.2e), rms %.2e (%.2e)%s\n", law, eps, n, size, L,
                                   k == 0 ? "f" : (k == 1 ? "g" : "tau"), top[1][k], top[0][k], sqrt(sum[1][k] / M), sqrt(sum[0][k] / M),
                                   worse ? " WORSE" : "");
                        failed += worse;
                    }
                }
    // refused: values out of range, one at a time
    {
        const FixedParams fp = fixed_params(0.6, 1e-4, 1.0, 1.5, 1.5, 0.6, 1e3, 0.01, 1e6, 1);
        const double bads[] = {0.0, -0.1, 1.0, 1e-6, 1e300, (double)INFINITY, (double)NAN};
        for (int i = 0; i < 9; i++)
            for (double v : bads) {
                double f[9] = {4. / 9, 1. / 9, 1. / 9, 1. / 9, 1. / 9, 1. / 36, 1. / 36, 1. / 36, 1. / 36}, g[5] = {1. / 6, 1. / 12, 1. / 12, 1. / 12, 1. / 12}, t = 0.8;
                if (!collide_fixed(fp, 0.9, true, 1e-4, 4e-4, 1e-3, 2e-3, f, g, t)) failed++;
                f[i] = v;
                if (collide_fixed(fp, 0.9, true, 1e-4, 4e-4, 1e-3, 2e-3, f, g, t)) failed++;
            }
        for (int i = 0; i < 6; i++)
            for (double v : {1.0, -1.0, 1e300, (double)INFINITY, (double)NAN}) {
                double f[9] = {4. / 9, 1. / 9, 1. / 9, 1. / 9, 1. / 9, 1. / 36, 1. / 36, 1. / 36, 1. / 36}, g[5] = {1. / 6, 1. / 12, 1. / 12, 1. / 12, 1. / 12}, t = 0.8;
                if (i < 5) g[i] = v; else t = v == 1.0 ? 0.1 : v;
                if (collide_fixed(fp, 0.9, true, 1e-4, 4e-4, 1e-3, 2e-3, f, g, t)) failed++;
            }
    }
    printf("%s taken %.4f\n", failed ? "FAILED" : "OK", (double)taken / all);
    return failed ? 1 : 0;
}
