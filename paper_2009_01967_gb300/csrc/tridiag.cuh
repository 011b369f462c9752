// Sturm count of a real symmetric tridiagonal matrix, shared by the
// eigensolvers of small and large cells.
#pragma once

namespace kald {

// The rare steps of sturm_count: a zero minor (a pivot exactly 0) is replaced by
// -pivmin a_{j-1}, and the pair is rescaled by 2^-400 or 2^400 (exact) when a has left
// [2^-400, 2^400].  Not inlined: predicated off in the loop, its five multiplications
// took their slots of the FP64 unit (64 cycles each for a warp) in every step.
static __device__ __noinline__ double2 sturm_rescale(double a, double am, double pivmin) {
    if ((__double_as_longlong(a) << 1) == 0) a = -pivmin * am;
    const int ex = (__double2hiint(a) >> 20) & 0x7ff;
    if (ex > 1023 + 400) {
        a *= 0x1p-400;
        am *= 0x1p-400;
    } else if (ex < 1023 - 400) {
        a *= 0x1p+400;
        am *= 0x1p+400;
    }
    return make_double2(a, am);
}

// The number of negative pivots q_j of the LDL^T factorisation of T - x I (the
// eigenvalues below x).  The pivots are
// carried as ratios q_j = a_j / a_{j-1} of the leading principal minors,
// a_j = (d_j - x) a_{j-1} - e_{j-1}^2 a_{j-2} (a_{-1} = 1, a_{-2} = 0), which is
// the pivot recurrence q_j = d_j - x - e_{j-1}^2 / q_{j-1} without a division
// in the dependency chain.  Sign, zero and exponent tests work on the bit patterns;
// three FP64 operations per step.
__device__ inline int sturm_count(int n, const double *__restrict__ d, const double *__restrict__ e2, double x,
                           double pivmin) {
    int cnt = 0;
    double am = 1.0, amm = 0.0;                        // a_{j-1}, a_{j-2}
    for (int j = 0; j < n; ++j) {
        const double t = (j > 0) ? e2[j - 1] * amm : 0.0;
        double a = fma(d[j] - x, am, -t);
        const int ex = (__double2hiint(a) >> 20) & 0x7ff;
        const int neg = __double2hiint(am);
        if ((unsigned)(ex - (1023 - 400)) > 800u) {
            const bool zero = (__double_as_longlong(a) << 1) == 0;
            const double2 r = sturm_rescale(a, am, pivmin);
            if (zero) cnt += 1;                        // -pivmin a_{j-1}: a negative pivot
            else cnt += (__double2hiint(a) ^ neg) < 0; // q_j < 0
            a = r.x;
            am = r.y;
        } else {
            cnt += (__double2hiint(a) ^ neg) < 0;
        }
        amm = am;
        am = a;
    }
    return cnt;
}

}  // namespace kald
