// repeat_step (qp_df.h) against taking its steps one by one, bit for bit:
// increments from far below to far above the last place of x, ties, starts at
// and next to powers of two, paths through zero, zero, infinities and NaN.
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>

#include "qp_df.h"

using namespace qp;

static long bad = 0, checked = 0;

template <class S>
static void check(double x, int n, const S &s)
{
    double a = x;
    for (int k = 0; k < n; ++k) a = s.one(a);
    const double b = repeat_step(x, n, s);
    ++checked;
    if (d2u(a) != d2u(b) && !(a != a && b != b)) {
        if (++bad < 10) printf("# x %a n %d: %a, got %a\n", x, n, a, b);
    }
}

int main()
{
    std::mt19937_64 g(7);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    const int counts[] = {0, 1, 2, 3, 4, 5, 17, 250, 1000};
    for (int t = 0; t < 400000; ++t) {
        const int n = counts[g() % 9];
        double x = std::ldexp(U(g), (int)(g() % 24) - 12);
        double d = std::ldexp(U(g), (int)(g() % 70) - 64);
        const int how = (int)(g() % 8);
        if (how == 0) x = std::ldexp(x < 0 ? -1.0 : 1.0, (int)(g() % 12) - 6);           // a power of two
        if (how == 1) x = std::nextafter(std::ldexp(1.0, (int)(g() % 12) - 6), g() % 2 ? 9e9 : 0);
        if (how == 2) d = (g() % 2 ? 0.5 : 1.5) * std::ldexp(U(g) < 0 ? -1.0 : 1.0, std::ilogb(x) - 52);  // tie
        if (how == 3) d = -x / (double)(1 + g() % 300);                                   // through zero
        if (how == 4) d = std::ldexp((double)(2 * (g() % 4096) + 1), std::ilogb(x) - 53);  // tie, wider
        check(x, n, StepFloat((float)d));
        const double b = U(g);
        check(x, n, StepProduct{b, d / b});
        check(x, n, StepProduct{0.5, 2.0 * d});
    }
    const double odd[] = {0.0, -0.0, INFINITY, -INFINITY, NAN, 1e300, -1e300, 5e-324, 1e-300, 1.0};
    const float inc[] = {0.0f, -0.0f, 1e-40f, 1e30f, -1e30f, INFINITY, NAN, 1e-20f, 0.03f};
    for (double x : odd)
        for (float f : inc)
            for (int n : counts) {
                check(x, n, StepFloat(f));
                check(x, n, StepProduct{0.25, 4.0 * (double)f});
            }
    printf("checked %ld\nwrong %ld\n", checked, bad);
    return 0;
}
