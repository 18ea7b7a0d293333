// Errors of the block fixed-point collision (lbm_fixed.cuh, compiled for the host)
// and of the same collision in FP64 against long double, by kind of flow and tau.
// First a line "wild" with the largest error, in units of the cell's largest value, over
// cells far from equilibrium at every size the range takes in, and how many it took in.
// Then one line each: kind model tau, rms error of the values (FP64 form, fixed
// point), rms and mean error of the x momentum (FP64 form, fixed point) and the
// number of cells; everything relative to the largest |s_i| or |F| of the cell.
#include <cmath>
#include <cstdio>
#include <random>

#include "lbm_fixed.cuh"
using namespace lbm;
typedef long double X;

static void fp64_form(double s[Q], double om, const double F[3], bool inc) {
    double r = s[0];
    for (int p = 0; p < NPAIR; ++p) r += s[pair_first(p)] + s[opp(pair_first(p))];
    const double j[3] = {
        fma(0.5, F[0], (((s[1] - s[2]) + (s[7] - s[10])) + ((s[8] - s[9]) + (s[11] - s[14]))) + (s[12] - s[13])),
        fma(0.5, F[1], (((s[3] - s[4]) + (s[7] - s[10])) + ((s[9] - s[8]) + (s[15] - s[18]))) + (s[16] - s[17])),
        fma(0.5, F[2], (((s[5] - s[6]) + (s[11] - s[14])) + ((s[13] - s[12]) + (s[15] - s[18]))) + (s[17] - s[16]))};
    const double rho = inc ? 1.0 : 1.0 + r, inv = 1.0 / rho, u[3] = {j[0] * inv, j[1] * inv, j[2] * inv};
    const double omc = 1.0 - om, c = 1.0 - 0.5 * om, nusq = -1.5 * fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0]));
    const double uF = fma(u[2], F[2], fma(u[1], F[1], u[0] * F[0]));
    s[0] = fma(omc, s[0], fma(om * (1.0 / 3.0) * rho, nusq, fma(-c, uF, om * (1.0 / 3.0) * r)));
    for (int p = 0; p < NPAIR; ++p) {
        const int i = pair_first(p), o = opp(i);
        const double h = i <= 6 ? 1.0 : 0.5, w = h / 18.0, k = om * (1.0 / 18.0);
        const double a = h * fma(-1.0 / 6.0 * c, uF, k * r), b = h * (k * rho);
        const double e = ex(i) * u[0] + ey(i) * u[1] + ez(i) * u[2], eF = ex(i) * F[0] + ey(i) * F[1] + ez(i) * F[2];
        const double E = fma(e, 9.0 * c * w * eF, fma(b, fma(4.5, e * e, nusq), a));
        const double P = fma(3.0 * b, e, 3.0 * c * w * eF);
        s[i] = fma(omc, s[i], E + P);
        s[o] = fma(omc, s[o], E - P);
    }
}

static void extended(const double s[Q], X om, const double F[3], bool inc, X out[Q]) {
    X r = 0, j[3] = {X(F[0]) / 2, X(F[1]) / 2, X(F[2]) / 2};
    for (int i = 0; i < Q; ++i) {
        r += s[i];
        j[0] += X(ex(i)) * s[i];
        j[1] += X(ey(i)) * s[i];
        j[2] += X(ez(i)) * s[i];
    }
    const X rho = inc ? X(1) : 1 + r, u[3] = {j[0] / rho, j[1] / rho, j[2] / rho};
    const X usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2], uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2];
    for (int i = 0; i < Q; ++i) {
        const X w = X(1) / (i == 0 ? 3 : (i <= 6 ? 18 : 36));
        const X eu = ex(i) * u[0] + ey(i) * u[1] + ez(i) * u[2], eF = X(ex(i)) * F[0] + X(ey(i)) * F[1] + X(ez(i)) * F[2];
        out[i] = (1 - om) * s[i] + om * w * (r + rho * (3 * eu + X(4.5) * eu * eu - X(1.5) * usq)) +
                 (1 - om / 2) * w * (3 * (eF - uF) + 9 * eu * eF);
    }
}

struct Sum {
    X sq = 0, j2 = 0, j1 = 0;
    void add(const double s[Q], const X x[Q], double top) {
        X dj = 0;
        for (int i = 0; i < Q; ++i) {
            const X d = (s[i] - x[i]) / top;
            sq += d * d;
            dj += ex(i) * d;
        }
        j2 += dj * dj;
        j1 += dj;
    }
};

// Populations that add up in rho and j as far as the range allows: signs that follow a
// random direction, or one for all, sizes near the cell's largest.
static void wild() {
    std::mt19937_64 gen(5);
    std::uniform_real_distribution<double> U(-1, 1);
    X worst = 0;
    int n = 0;
    for (int t = 0; t < 400000; ++t) {
        const double size = ldexp(1.0, -2 - t % 9) * (0.75 + 0.25 * U(gen)), bias = U(gen), d[3] = {U(gen), U(gen), U(gen)};
        const bool inc = t & 1, force = t & 2;
        const double om = 1.0 + 0.999 * U(gen), flat = U(gen) * U(gen);
        double s[Q], f[Q], F[3] = {0, 0, 0}, top = 0;
        for (int i = 0; i < Q; ++i) {
            const double p = ex(i) * d[0] + ey(i) * d[1] + ez(i) * d[2];
            s[i] = f[i] = size * (1 + 0.1 * U(gen)) * (i == 0 || p == 0 ? bias : (p > 0 ? 1 : -1) * (1 - fabs(flat)) + flat);
            top = fmax(top, fabs(s[i]));
        }
        for (int c = 0; c < 3 && force; ++c) F[c] = size * U(gen);
        FixedMom m;
        if (!(force ? fixed_moments<true>(f, F[0], F[1], F[2], m) : fixed_moments<false>(f, 0, 0, 0, m))) continue;
        if (force)
            fixed_collide<true>(f, m, fixed_k(om), inc);
        else
            fixed_collide<false>(f, m, fixed_k(om), inc);
        X x[Q];
        extended(s, om, F, inc, x);
        for (int i = 0; i < Q; ++i) {
            top = fmax(top, (double)fabsl(x[i]));
            top = fmax(top, fabs(F[i % 3]));
        }
        for (int i = 0; i < Q; ++i) worst = fmaxl(worst, fabsl(f[i] - x[i]) / top);
        ++n;
    }
    printf("wild %Lg %d\n", worst, n);
}

int main() {
    wild();
    const struct { const char *name; double rho, u, noise, F; } kinds[] = {
        {"flow", 0.01, 0.03, 1e-3, 0},      {"rough", 0.02, 0.05, 0.05, 0}, {"still", 0.2, 1e-9, 1e-3, 0},
        {"slow", 0.01, 1e-4, 1e-2, 0},      {"fast", 0.2, 0.2, 1e-2, 0},    {"noise", 0, 0, 1.0, 0},
        {"tiny", 3e-31, 1e-30, 0.05, 1e-33}, {"driven", 0.01, 0.03, 1e-3, 1e-3},
        {"pushed", 1e-8, 1e-8, 0.1, 0.01}};
    const double taus[] = {0.5005, 0.55, 0.6, 0.9, 1.0, 2.0, 5.0, 50.0};
    std::mt19937_64 gen(1);
    std::normal_distribution<double> N(0, 1);
    std::uniform_real_distribution<double> U(-1, 1);
    for (const auto &k : kinds)
        for (int inc = 0; inc < 2; ++inc)
            for (double tau : taus) {
                const double om = 1.0 / tau, size = k.u + k.rho > 0 ? k.u + 0.3 * k.rho : 0.01;
                const FixedK fk = fixed_k(om);
                Sum a, b;
                int n = 0;
                for (int t = 0; t < 4000; ++t) {
                    const double u[3] = {k.u * U(gen), k.u * U(gen), k.u * U(gen)}, r = k.rho * U(gen);
                    const double F[3] = {k.F * U(gen), k.F * U(gen), k.F * U(gen)};
                    double s[Q], f[Q], top = 0;
                    for (int i = 0; i < Q; ++i) {
                        const double eu = ex(i) * u[0] + ey(i) * u[1] + ez(i) * u[2];
                        const double usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
                        s[i] = weight(i) * (r + (1 + r) * (3 * eu + 4.5 * eu * eu - 1.5 * usq) + size * k.noise * N(gen));
                        top = fmax(top, fabs(s[i]));
                        f[i] = s[i];
                    }
                    for (int c = 0; c < 3; ++c) top = fmax(top, fabs(F[c]));
                    X x[Q];
                    extended(s, om, F, inc, x);
                    FixedMom m;
                    if (!(k.F ? fixed_moments<true>(f, F[0], F[1], F[2], m) : fixed_moments<false>(f, 0, 0, 0, m))) continue;
                    if (k.F)
                        fixed_collide<true>(f, m, fk, inc);
                    else
                        fixed_collide<false>(f, m, fk, inc);
                    fp64_form(s, om, F, inc);
                    a.add(s, x, top);
                    b.add(f, x, top);
                    ++n;
                }
                printf("%s %d %g %Lg %Lg %Lg %Lg %Lg %Lg %d\n", k.name, inc, tau, sqrtl(a.sq / n / Q), sqrtl(b.sq / n / Q),
                       sqrtl(a.j2 / n), sqrtl(b.j2 / n), a.j1 / n, b.j1 / n, n);
            }
}
