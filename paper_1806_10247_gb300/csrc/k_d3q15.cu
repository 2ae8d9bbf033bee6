// D3Q15 fused stream + collide step, FP64: the 3D cascaded method of
// Appendix A with the symmetrized operator-split force.
//
// Per node: pull the 15 populations (Eq. 22b with halfway bounce-back or
// periodic wrap), raw moments of Eq. g8 (the corner populations through an
// 8-point sign transform), the pre-collision half force of Eq. 8A, the
// cascaded changes g_4..g_14 of Eq. 6A, the force change g_1..g_3 of
// Eq. 13A and the populations f + K g (Eq. 2A), again through the sign
// transform on the corners.  Three readings of the appendix are built in:
// the trace bracket of g_9 relaxes towards its equilibrium rho (as printed
// the rest state would not be a fixed point); the populations are K g
// exactly (the printed f^p_12 has the sign of g_13 flipped); the product in
// the fourth-order bracket of g_14 is that of the post-collision second
// central moments kappa_xx, kappa_yy divided by rho.  With a time-dependent
// force the first moments change by (F_pre + F_post)/2, i.e.
// g_1..3 = (F_pre + F_post)/20.
#include "lbm_d3q15.cuh"
#include "lbm_internal.h"
#include "lbm_lattices.cuh"
#include "lbm_tiles.cuh"

namespace lbmk {
namespace {

constexpr int kBlock = 256;

// omega_4..omega_8 (shear), omega_9 (trace), omega_10..omega_13, omega_14
struct Rates15 {
    double s, b, t, q;
};

// F = a_pre P (Eq. 8A), Fq = a_post P (second half step).
__device__ __forceinline__ void collide(double (&f)[15], const double (&F)[3], const double (&Fq)[3],
                                        const Rates15 &w)
{
    // Axis pairs and the corner sign transform: S_{ijk} = sum_c s_x^i s_y^j s_z^k f_c.
    const double axs = f[1] + f[2], axd = f[1] - f[2];
    const double ays = f[3] + f[4], ayd = f[3] - f[4];
    const double azs = f[5] + f[6], azd = f[5] - f[6];
    const double A1 = f[7] + f[8], B1 = f[7] - f[8];      // y+, z+
    const double A2 = f[9] + f[10], B2 = f[9] - f[10];    // y-, z+
    const double A3 = f[11] + f[12], B3 = f[11] - f[12];  // y+, z-
    const double A4 = f[13] + f[14], B4 = f[13] - f[14];  // y-, z-
    const double P1 = A1 + A2, Q1 = A1 - A2, P2 = A3 + A4, Q2 = A3 - A4;
    const double R1 = B1 + B2, T1 = B1 - B2, R2 = B3 + B4, T2 = B3 - B4;
    const double S = P1 + P2, Sz = P1 - P2, Sy = Q1 + Q2, Syz = Q1 - Q2;
    const double Sx = R1 + R2, Sxz = R1 - R2, Sxy = T1 + T2, Sxyz = T1 - T2;

    // Raw moments (Eq. g8): on D3Q15 every cubic and quartic monomial of the
    // basis lives on the corners only.
    const double rho = f[0] + axs + ays + azs + S;
    const double kxx = axs + S, kyy = ays + S, kzz = azs + S;
    const double kxy = Sxy, kxz = Sxz, kyz = Syz;
    const double kxyy = Sx, kxxy = Sy, kxxz = Sz, kxyz = Sxyz, kxxyy = S;

    // Eq. 8A: half-forced momentum J = rho u.
    const double jx0 = axd + Sx, jy0 = ayd + Sy, jz0 = azd + Sz;
    const double Jx = fma(0.5, F[0], jx0), Jy = fma(0.5, F[1], jy0), Jz = fma(0.5, F[2], jz0);
    const double ir = __drcp_rn(rho);
    const double ux = Jx * ir, uy = Jy * ir, uz = Jz * ir;

    // Eq. 6A.  Second order: central moments about u.
    const double cxx = kxx - Jx * ux, cyy = kyy - Jy * uy, czz = kzz - Jz * uz;
    const double g4 = -0.125 * w.s * (kxy - Jx * uy);
    const double g5 = -0.125 * w.s * (kxz - Jx * uz);
    const double g6 = -0.125 * w.s * (kyz - Jy * uz);
    const double g7 = -0.25 * w.s * (cxx - cyy);
    const double g8 = -(w.s / 12.0) * (cxx + cyy - 2.0 * czz);
    const double g9 = (w.b / 18.0) * (rho - (cxx + cyy + czz));
    const double h3 = g7 + g8 + 3.0 * g9;  // the combination the cubic cascades share
    const double g10 = 0.0625 * w.t * (-kxyy + 2.0 * uy * kxy + ux * kyy - 2.0 * Jx * uy * uy) + uy * g4 +
                       0.125 * ux * (h3 - 2.0 * g7);
    const double g11 = 0.0625 * w.t * (-kxxy + 2.0 * ux * kxy + uy * kxx - 2.0 * Jx * ux * uy) + ux * g4 +
                       0.125 * uy * h3;
    const double g12 = 0.0625 * w.t * (-kxxz + 2.0 * ux * kxz + uz * kxx - 2.0 * Jx * ux * uz) + ux * g5 +
                       0.125 * uz * h3;
    const double g13 = 0.125 * w.t * (-kxyz + ux * kyz + uy * kxz + uz * kxy - 2.0 * Jx * uy * uz) + uz * g4 +
                       uy * g5 + ux * g6;
    // post-collision kappa_xx, kappa_yy (the changes of K_7, K_8, K_9 to them)
    const double cxx_p = cxx + 2.0 * (g7 + g8) + 6.0 * g9;
    const double cyy_p = cyy + 2.0 * (g8 - g7) + 6.0 * g9;
    const double ux2 = ux * ux, uy2 = uy * uy;
    const double g14 = 0.0625 * w.q *
                           (-kxxyy + 2.0 * ux * kxyy + 2.0 * uy * kxxy - ux2 * kyy - uy2 * kxx -
                            4.0 * ux * uy * kxy + cxx_p * cyy_p * ir + 3.0 * Jx * ux * uy2) -
                       2.0 * ux * uy * g4 + 0.125 * (ux2 - uy2) * g7 - 0.125 * (ux2 + uy2) * g8 -
                       (0.375 * (ux2 + uy2) + 0.5) * g9 + 2.0 * ux * g10 + 2.0 * uy * g11;

    // Eq. 13A with the two half steps.
    const double g1 = 0.05 * (F[0] + Fq[0]), g2 = 0.05 * (F[1] + Fq[1]), g3 = 0.05 * (F[2] + Fq[2]);

    // f + K g.  Rest and axes:
    f[0] += 32.0 * g14 - 2.0 * g9;
    const double bx = g7 + g8 - g9 - 8.0 * g14, ox = g1 - 8.0 * g10;
    const double by = g8 - g7 - g9 - 8.0 * g14, oy = g2 - 8.0 * g11;
    const double bz = -2.0 * g8 - g9 - 8.0 * g14, oz = g3 - 8.0 * g12;
    f[1] += bx + ox;
    f[2] += bx - ox;
    f[3] += by + oy;
    f[4] += by - oy;
    f[5] += bz + oz;
    f[6] += bz - oz;
    // corners: c0 + s_x cx + s_y cy + s_z cz + s_x s_y g4 + s_x s_z g5 + s_y s_z g6 + s_x s_y s_z g13
    const double c0 = g9 + 2.0 * g14, cx = g1 + 2.0 * g10, cy = g2 + 2.0 * g11, cz = g3 + 2.0 * g12;
    const double U0 = c0 + cz, Ux = cx + g5, Uy = cy + g6, Uxy = g4 + g13;  // z = +1
    const double V0 = c0 - cz, Vx = cx - g5, Vy = cy - g6, Vxy = g4 - g13;  // z = -1
    const double a0 = U0 + Uy, ax = Ux + Uxy, b0 = U0 - Uy, bxx = Ux - Uxy;
    const double c0m = V0 + Vy, cxm = Vx + Vxy, d0 = V0 - Vy, dx = Vx - Vxy;
    f[7] += a0 + ax;
    f[8] += a0 - ax;
    f[9] += b0 + bxx;
    f[10] += b0 - bxx;
    f[11] += c0m + cxm;
    f[12] += c0m - cxm;
    f[13] += d0 + dx;
    f[14] += d0 - dx;
}

// One node's step in fixed point (omega_10 .. omega_14 = 1): shape(d) gives the
// force shape's component d, q1 = a_pre / 4 and q2 = (a_pre + a_post) / 4, put(a,
// f) takes a result.
template <bool FORCED, bool XO, class Shape, class Put>
__device__ __forceinline__ FxStep fixed_step15(const double (&f)[15], const FxRates &w, double q1, double q2, Shape shape,
                                             Put put)
{
    const int em = fx_emax(f);
    const int k = FxGrid<15>::S + 1023 - em;
    if (!fx_in_range(em)) return FX_NOT;
    int bad = 0;
    FxForce F[3] = {{0, 0}, {0, 0}, {0, 0}};
    if (FORCED) {
        const unsigned dither = (unsigned)fx_bits(f[0]);
#pragma unroll
        for (int d = 0; d < (XO ? 1 : 3); d++)
            if (!fx_force(shape(d), q1, q2, k, em, dither >> (8 * d), F[d])) bad = -1;
        if (bad < 0) return FX_NOT;
    }
    i64 X[15];
    fx_load(f, k, X);
    FxSums15<i64> s;
    fx_sums15(X, s);
    fx_collide15<XO>(s, F, w, X, bad);
#pragma unroll
    for (int a = 0; a < 15; a++) put(a, fx_value_pos(X[a], k + 1, bad));
    return bad >= 0 ? FX_DONE : FX_GIVEN_UP;
}

template <class Shape>
__device__ __forceinline__ void double_step15(double (&f)[15], const Rates15 &w, bool forced, double apre, double apost,
                                              Shape shape)
{
    double F[3] = {0.0, 0.0, 0.0}, Fq[3] = {0.0, 0.0, 0.0};
    if (forced) {
#pragma unroll
        for (int d = 0; d < 3; d++) {
            const double P = shape(d);
            F[d] = apre * P;
            Fq[d] = apost * P;
        }
    }
    collide(f, F, Fq, w);
}

// FIX: the fixed-point form (omega_10 .. omega_14 = 1).  XO: the force acts
// along x only.  Both checked on the host.
template <int FK, bool FIX, bool XO>
__global__ void __launch_bounds__(kBlock)
k_step(const __grid_constant__ Planes<double, 15> P, Geom g, FieldDev Fd, double apre, double apost, Rates15 w,
       FxRates fx, double q1, double q2)
{
    step_begin();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    int x, y, z;
    node_xyz(g, i, x, y, z);
    double f[15];
    load_pulled<LD3Q15>(P, g, x, y, z, i, f);
    auto shape = [&](int d) { return field_value(Fd, FK, d, x, y, z, i); };
    if (FIX) {
        const FxStep r = fixed_step15<FK != FK_NONE, XO>(f, fx, q1, q2, shape, [&](int a, double v) { P.out[a][i] = v; });
        if (r == FX_DONE) return;
        if (r == FX_GIVEN_UP) load_pulled<LD3Q15>(P, g, x, y, z, i, f);
    }
    double_step15(f, w, FK != FK_NONE, apre, apost, shape);
#pragma unroll
    for (int a = 0; a < 15; a++) P.out[a][i] = f[a];
}

// Batched form; a step's amplitudes per item in Amp64.
// One node of a batched launch (member `it`, node i; B staged in shared memory).
__device__ __forceinline__ void batch_node(const BatchItem &B, const BatchLaunch &L, int it, int i)
{
    const Geom &g = B.g;
    const int p = B.parity + L.parity;
    const double *fin = B.buf[p & 1];
    double *fout = B.buf[(p + 1) & 1];
    const Amp64 ap = L.pairs ? L.pairs[(size_t)L.k * L.count + it] : L.inl[it];
    int x, y, z;
    node_xyz(g, i, x, y, z);
    double f[15];
    load_pulled<LD3Q15>(fin, g, x, y, z, i, f);
    if (L.mrho) fused_fields<LD3Q15>(B, L, it, i, x, y, z, f, 2.0 * ap.q1);  // fused readback of f(t)'s fields
    const bool forced = B.fkind != FK_NONE;
    auto shape = [&](int d) { return forced ? field_value(B.F, B.fkind, d, x, y, z, i) : 0.0; };
    const Rates15 w{B.coef[0], B.coef[1], B.coef[2], B.coef[3]};
    if (w.t == 1.0 && w.q == 1.0) {  // uniform over the member
        const FxStep r =
            fixed_step15<true, false>(f, B.fx, ap.q1, ap.q2, shape, [&](int a, double v) { fout[a * g.Np + i] = v; });
        if (r == FX_DONE) return;
        if (r == FX_GIVEN_UP) load_pulled<LD3Q15>(fin, g, x, y, z, i, f);
    }
    double_step15(f, w, forced, ap.pre, ap.g, shape);
#pragma unroll
    for (int a = 0; a < 15; a++) fout[a * g.Np + i] = f[a];
}

template <int TB, int MODE>
__global__ void __launch_bounds__(TB)
k_batch(const __grid_constant__ BatchLaunch L)
{
    batch_tiles<TB, MODE>(L, [](const BatchItem &B, const BatchLaunch &L2, int it, int i) { batch_node(B, L2, it, i); });
}

}  // namespace

void d3q15_batch_coef(const double omega[9], BatchItem &item)
{
    item.coef[0] = omega[2];
    item.coef[1] = omega[1];
    item.coef[2] = omega[3];
    item.coef[3] = omega[4];
    item.fx = fx_rates27(omega[1], omega[2]);
}

cudaError_t d3q15_batch_step(const BatchLaunch &L, int nblocks, int tile, cudaStream_t s)
{
    LBM_TILED_LAUNCH(k_batch, L, nblocks, tile, s);
}

int d3q15_batch_resident(int tile)
{
    LBM_TILED_RESIDENT(k_batch, tile);
}

cudaError_t d3q15_step(const LaunchArgs &a)
{
    const Rates15 w{a.omega[2], a.omega[1], a.omega[3], a.omega[4]};
    const FxRates fx = fx_rates27(a.omega[1], a.omega[2]);
    const double q1 = 0.25 * a.apre, q2 = 0.25 * (a.apre + a.apost);
    const Planes<double, 15> P = make_planes<double, 15>(a.fin, a.fout, a.g.Np);
    const bool fix = w.t == 1.0 && w.q == 1.0, xo = force_x_only(a.fkind, a.F, 3);
    const int block = spread_block(a.g.N, kBlock), grid = (a.g.N + block - 1) / block;
#define STEP15(FK, FIX, XO) launch_step(a.overlap, k_step<FK, FIX, XO>, grid, block, a.stream, P, a.g, a.F, a.apre, a.apost, w, fx, q1, q2)
    switch (a.fkind) {
    case FK_NONE:
        if (fix) STEP15(FK_NONE, true, false);
        else STEP15(FK_NONE, false, false);
        break;
    case FK_CONST:
        if (fix && xo) STEP15(FK_CONST, true, true);
        else if (fix) STEP15(FK_CONST, true, false);
        else STEP15(FK_CONST, false, false);
        break;
    default:
        if (fix && xo) STEP15(FK_GENERAL, true, true);
        else if (fix) STEP15(FK_GENERAL, true, false);
        else STEP15(FK_GENERAL, false, false);
        break;
    }
#undef STEP15
    return cudaGetLastError();
}

}  // namespace lbmk
