// Sturm count of a real symmetric tridiagonal matrix, shared by the
// eigensolvers of small and large cells.
#pragma once

namespace kald {

// The number of negative pivots q_j of the LDL^T factorisation of T - x I (the
// eigenvalues below x).  The pivots are
// carried as ratios q_j = a_j / a_{j-1} of the leading principal minors,
// a_j = (d_j - x) a_{j-1} - e_{j-1}^2 a_{j-2} (a_{-1} = 1, a_{-2} = 0), which is
// the pivot recurrence q_j = d_j - x - e_{j-1}^2 / q_{j-1} without a division
// in the dependency chain.  A zero minor (a pivot exactly 0) is replaced by
// -pivmin a_{j-1}; the pair (a_j, a_{j-1}) is rescaled by 2^-400 or 2^400
// (exact) whenever a_j leaves [2^-400, 2^400].  Sign, zero and exponent tests
// work on the bit patterns.
__device__ inline int sturm_count(int n, const double *__restrict__ d, const double *__restrict__ e2, double x,
                           double pivmin) {
    int cnt = 0;
    double am = 1.0, amm = 0.0;                        // a_{j-1}, a_{j-2}
    for (int j = 0; j < n; ++j) {
        const double t = (j > 0) ? e2[j - 1] * amm : 0.0;
        double a = fma(d[j] - x, am, -t);
        if ((__double_as_longlong(a) << 1) == 0) a = -pivmin * am;
        cnt += (__double_as_longlong(a) ^ __double_as_longlong(am)) < 0;   // q_j < 0
        const int ex = (__double2hiint(a) >> 20) & 0x7ff;
        if (ex > 1023 + 400) {
            a *= 0x1p-400;
            am *= 0x1p-400;
        } else if (ex < 1023 - 400) {
            a *= 0x1p+400;
            am *= 0x1p+400;
        }
        amm = am;
        am = a;
    }
    return cnt;
}

}  // namespace kald
