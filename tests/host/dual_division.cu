// Forward-mode division: the largest error of a quotient's derivative, in units
// of the FP32 unit roundoff times |a b' / b^2| (the size of the two terms that
// nearly cancel), over n pairs whose derivatives nearly cancel.  Built and run
// on the CPU by tests/test_dual_division_host.py; no GPU call is made.
#include <cmath>
#include <cstdio>

#include "lbfd_dual.cuh"

static unsigned long long state = 1;
static float uniform(float lo, float hi)
{
    state = state * 6364136223846793005ull + 1442695040888963407ull;
    return lo + (hi - lo) * (float)((state >> 40) * (1.0 / 16777216.0));
}

int main()
{
    using D = lbfd::Dual<float, 4>;
    double worst = 0.0;
    for (int i = 0; i < 1000000; ++i) {
        D a, b;
        a.v = uniform(0.5f, 50.f);
        b.v = uniform(0.5f, 50.f);
        for (int k = 0; k < 4; ++k) {
            b.d[k] = uniform(0.5f, 2.f);
            a.d[k] = (float)((double)a.v / b.v * b.d[k] * (1.0 + uniform(-1e-4f, 1e-4f)));
        }
        const D q = a / b;
        for (int k = 0; k < 4; ++k) {
            const double term = (double)a.v / b.v * b.d[k] / b.v, exact = a.d[k] / (double)b.v - term;
            worst = std::fmax(worst, std::fabs(q.d[k] - exact) / term * 16777216.0);
        }
    }
    printf("%.6f\n", worst);
    return 0;
}
