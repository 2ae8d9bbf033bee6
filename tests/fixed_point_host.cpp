// The fixed-point collisions of csrc/lbm_fixed.cuh on the host, for
// tests/test_fixed_point_cpu.py.  f: [n][q] populations, replaced by the results;
// P: [n][dim] force or source shapes; ok[n]: 1 where the fixed-point form applies.
#include "lbm_fixed.cuh"

using namespace lbmk;

template <int Q, class Collide>
static void run(long n, double *f, int *ok, Collide collide)
{
    for (long i = 0; i < n; i++) {
        double v[Q];
        for (int a = 0; a < Q; a++) v[a] = f[i * Q + a];
        const int em = fx_emax(v), k = FxGrid<Q>::S + 1023 - em;
        int bad = fx_in_range(em) ? 0 : -1;
        if (bad == 0) {
            i64 X[Q];
            if constexpr (Q == 9) {  // the kernels' own way in: see fixed_step9 and fixed_step5
                fx_load_int<9, false>(v, em, X);
                for (int a = 0; a < 9; a++) bad |= (int)fx_hi(fx_bits(v[a]));
            } else if constexpr (Q == 5) {
                fx_load_int<5, true>(v, em, X);
            } else {
                fx_load(v, k, X);
            }
            collide(i, v, X, k, em, bad);
            for (int a = 0; a < Q; a++)
                v[a] = Q == 5 ? fx_value_signed(X[a], k, bad) : fx_value_pos(X[a], k + 1, bad);
        }
        ok[i] = bad >= 0;
        for (int a = 0; a < Q; a++) f[i * Q + a] = v[a];
    }
}

extern "C" void fixed27(long n, double *f, const double *P, double apre, double apost, double wb, double ws, int xo, int *ok)
{
    run<27>(n, f, ok, [&](long i, const double (&v)[27], i64 (&X)[27], int k, int em, int &bad) {
        FxForce F[3] = {{0, 0}, {0, 0}, {0, 0}};
        for (int d = 0; d < (xo ? 1 : 3); d++)
            if (!fx_force(P[3 * i + d], 0.25 * apre, 0.25 * (apre + apost), k, em, (unsigned)fx_bits(v[13]) >> (8 * d), F[d]))
                bad = -1;
        FxSums27<i64> s;
        fx_sums27(X, s);
        if (xo) fx_collide27<true>(s, F, fx_rates27(wb, ws), X, bad);
        else fx_collide27<false>(s, F, fx_rates27(wb, ws), X, bad);
    });
}

extern "C" void fixed15(long n, double *f, const double *P, double apre, double apost, double wb, double ws, int xo, int *ok)
{
    run<15>(n, f, ok, [&](long i, const double (&v)[15], i64 (&X)[15], int k, int em, int &bad) {
        FxForce F[3] = {{0, 0}, {0, 0}, {0, 0}};
        for (int d = 0; d < (xo ? 1 : 3); d++)
            if (!fx_force(P[3 * i + d], 0.25 * apre, 0.25 * (apre + apost), k, em, (unsigned)fx_bits(v[0]) >> (8 * d), F[d]))
                bad = -1;
        FxSums15<i64> s;
        fx_sums15(X, s);
        if (xo) fx_collide15<true>(s, F, fx_rates27(wb, ws), X, bad);
        else fx_collide15<false>(s, F, fx_rates27(wb, ws), X, bad);
    });
}

extern "C" void fixed9(long n, double *f, const double *P, double apre, double apost, double w3, double w4, double w5, int xo,
                       int *ok)
{
    run<9>(n, f, ok, [&](long i, const double (&v)[9], i64 (&X)[9], int k, int em, int &bad) {
        FxForce F[2] = {{0, 0}, {0, 0}};
        for (int d = 0; d < (xo ? 1 : 2); d++)
            if (!fx_force(P[2 * i + d], 0.25 * apre, 0.25 * (apre + apost), k, em, (unsigned)fx_bits(v[0]) >> (8 * d), F[d]))
                bad = -1;
        FxSums9<i64> s;
        fx_sums9(X, s);
        if (xo) fx_collide9<true>(s, F, fx_rates9(w3, w4, w5), X, bad);
        else fx_collide9<false>(s, F, fx_rates9(w3, w4, w5), X, bad);
    });
}

extern "C" void fixed5(long n, double *f, const double *P, double apre, double apost, const double *om, double ux, double uy,
                       int *ok)
{
    const FxCoef5 c = fx_coef5(om[1] / 2, om[2] / 2, om[3] / 4, om[4] / 4, ux, uy);
    run<5>(n, f, ok, [&](long i, const double (&v)[5], i64 (&X)[5], int k, int em, int &bad) {
        FxForce S;
        if (!c.ok || !fx_force(P[i], 0.5 * apre, 0.5 * (apre + apost), k - 1, em, (unsigned)fx_bits(v[0]), S)) bad = -1;
        fx_collide5(X, S.h1, S.h2, c);
    });
}
