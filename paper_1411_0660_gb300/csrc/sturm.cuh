// sturm.cuh -- eigenvalue counts of a symmetric tridiagonal matrix from its leading minors.
#pragma once

namespace mbl {

// Number of eigenvalues of T(d, e2) below x from the leading minors p_i = (d_i - x) p_{i-1} - e2_{i-1} p_{i-2} themselves (Givens,
// 1954): their sign changes.  Three FP64 operations a row where the quotient form's division takes some
// thirty, on a part with two FP64 FMAs a clock and SM.  T scaled to a norm of about 1 (so that two rows
// change a minor by no more than 2^+-400: a zero minor is replaced by -2^-200 times the last, as the
// quotient form replaces a zero pivot); both minors are rescaled when they leave [2^-300, 2^300].
__device__ __forceinline__ int sturm_count_minors(int m, const double *d, const double *e2, double x) {
    double p0 = 1.0, p1 = d[0] - x;
    if (p1 == 0.0) p1 = -0x1p-200;
    int c = __double2hiint(p1) < 0;
    for (int i = 1; i < m; ++i) {
        double p2 = fma(d[i] - x, p1, -(e2[i - 1] * p0));
        if (p2 == 0.0) p2 = p1 * -0x1p-200;
        c += (__double2hiint(p2) ^ __double2hiint(p1)) < 0;
        p0 = p1;
        p1 = p2;
        if (i & 1) {
            const int x0 = (__double2hiint(p0) >> 20) & 0x7ff, x1 = (__double2hiint(p1) >> 20) & 0x7ff, xm = max(x0, x1);
            if ((unsigned)(xm - 723) > 600u) {
                const double f = __hiloint2double((2046 - xm) << 20, 0);
                p0 *= f;
                p1 *= f;
            }
        }
    }
    return c;
}

}  // namespace mbl
