// What the readbacks form in integers (csrc/lbm_fixed.cuh), on the host, for
// tests/test_fixed_point_readback_cpu.py.
#include "lbm_fixed.cuh"

using namespace lbmk;

// Deviations d[n][27]: their sum and the first moment along x; taken[n]: 1 where the
// integer sums apply.
extern "C" void deviation_sums(long n, const float *d, double *m0, double *jx, int *taken)
{
    for (long i = 0; i < n; i++) {
        float v[27];
        i64 X[27];
        int em;
        for (int a = 0; a < 27; a++) v[a] = d[27 * i + a];
        taken[i] = fx_load_dev(v, em, X) == FXD_TAKEN;
        if (!taken[i]) continue;
        FxSums27<i64> s;
        fx_sums27(X, s);
        m0[i] = fx_value(s.rho, 182 - em);
        jx[i] = fx_value(s.jx, 182 - em);
    }
}

// 1/x as the readbacks form it.
extern "C" void reciprocals(long n, const double *x, double *r)
{
    for (long i = 0; i < n; i++) r[i] = fx_recip(x[i]);
}
