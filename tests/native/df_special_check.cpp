// Host check of the mixed path's conversions (qp_df.h) on infinities, NaN and
// the largest floats: each gives what the FP64 expression gives.
// Prints one line per check: "<name> <failures>" and exits 0.
#include <float.h>
#include <math.h>
#include <stdio.h>

#include "qp_df.h"

static bool same(double a, double b) { return isnan(a) ? isnan(b) != 0 : a == b; }

int main()
{
    const float special[] = {INFINITY, -INFINITY, NAN, -NAN, FLT_MAX, -FLT_MAX, FLT_MIN, 1.0f, 0.0f};
    const double base[] = {0.0, 1.0, -3.5, 1e-30, 1e-5, 1e30, 1e37, -1e38, 1e39, 1e40, -1e41,
                           1e60, INFINITY, -INFINITY, NAN};
    int f_to_d = 0, merge = 0, add = 0, split = 0;
    for (float f : special) {
        if (!same(qp::f_to_d(f), (double)f)) ++f_to_d;
        // a double-float's low part is 0 here, or not a number beside an infinity
        if (!same(qp::merge_df({f, 0.0f}), (double)f)) ++merge;
        if (!same(qp::merge_df({1.0f, f}), 1.0 + (double)f)) ++merge;
        for (double d : base) {
            if (isfinite(f) && isfinite(d)) continue;
            if (!same(qp::add_fd(d, f), d + (double)f)) ++add;
        }
    }
    // a depth that became not a number in double-float arithmetic stays so
    const qp::df2 t = qp::df_add_f({1.0f, 0.0f}, NAN);
    if (!isnan(qp::merge_df(t))) ++split;
    printf("f_to_d %d\nmerge %d\nadd_fd %d\ndepth %d\n", f_to_d, merge, add, split);
    return 0;
}
