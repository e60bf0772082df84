// The local adjoints of the direct adjoint step (lbfd_adjoint_cell.cuh) against
// central differences of their forward forms, and the WENO3 partials at the
// smallest epsilon.  Prints the largest deviation of the collision's adjoint and
// of the WENO3 partials, and the number of partials that change when line and
// epsilon are scaled by powers of two down to that epsilon.  Built and run on
// the CPU by tests/test_adjoint_cell_host.py; no GPU call is made.
#include <cmath>
#include <cstdio>

#include "lbfd_adjoint_cell.cuh"

using namespace lbfd;

static unsigned long long state = 1;
static double uniform()  // in [-1, 1)
{
    state = state * 6364136223846793005ull + 1442695040888963407ull;
    return (double)(state >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

// fourth-order central difference of f at x[k]
template <typename F>
static double difference(double* x, double h, F f)
{
    const double x0 = *x;
    double v[4];
    const double at[4] = {-2.0, -1.0, 1.0, 2.0};
    for (int j = 0; j < 4; ++j) {
        *x = x0 + at[j] * h;
        v[j] = f();
    }
    *x = x0;
    return ((v[0] - v[3]) + 8.0 * (v[2] - v[1])) / (12.0 * h);
}

static double collision()
{
    double worst = 0.0;
    for (int t = 0; t < 200; ++t) {
        double x[13];  // m0, m1, m2, rho, irho, u, gam, Lam
        for (double& v : x) v = 0.03 * uniform();
        x[6] = 0.7 + 0.3 * uniform();
        x[7] = (1.0 + 0.1 * uniform()) / x[6];
        double lg[9];
        for (double& v : lg) v = uniform();
        const double rs = -0.54, rb = 0.3;
        auto in = [&] { return Collision2{x[0], {x[1], x[2]}, {x[3], x[4], x[5]}, x[6], x[7], {x[8], x[9]},
                                          {x[10], x[11]}, x[12]}; };
        Collision2 b{};
        collide2_adjoint(in(), rs, rb, lg, b, nullptr);
        const double adj[13] = {b.m0, b.m1[0], b.m1[1], b.m2[0], b.m2[1], b.m2[2], b.rho, b.irho, b.u[0], b.u[1],
                                b.gam[0], b.gam[1], b.Lam};
        double scale = 0.0;
        for (const double v : adj) scale = std::fmax(scale, std::fabs(v));
        for (int k = 0; k < 13; ++k) {
            const double d = difference(&x[k], 1e-4, [&] {
                Collision2 unused{};
                double g[9], s = 0.0;
                collide2_adjoint(in(), rs, rb, lg, unused, g);
                for (int i = 0; i < 9; ++i) s += lg[i] * g[i];
                return s;
            });
            worst = std::fmax(worst, std::fabs(d - adj[k]) / scale);
        }
    }
    return worst;
}

static double weno(int* scaled)
{
    double worst = 0.0;
    *scaled = 0;
    for (int t = 0; t < 800; ++t) {
        double v[5], w[5], z[5];
        for (double& y : v) y = uniform();
        const bool neg = t & 1, near = t & 2;
        const double eps = 1.0;
        conv_partials(v, neg, eps, near, w);
        for (int j = 0; j < 5; ++j) {
            const double d = difference(&v[j], 1e-3, [&] { return conv_partials(v, neg, eps, near, z); });
            worst = std::fmax(worst, std::fabs(d - w[j]));
        }
        const double s = std::ldexp(1.0, -124);  // epsilon 2^-248 = 2.2e-75
        double u[5];
        for (int j = 0; j < 5; ++j) u[j] = s * v[j];
        const double r = conv_partials(v, neg, eps, near, z), rs = conv_partials(u, neg, s * s * eps, near, z);
        *scaled += rs != s * r;
        for (int j = 0; j < 5; ++j) *scaled += z[j] != w[j];
    }
    return worst;
}

int main()
{
    int scaled;
    const double c = collision(), w = weno(&scaled);
    printf("%.3e %.3e %d\n", c, w, scaled);
    return 0;
}
