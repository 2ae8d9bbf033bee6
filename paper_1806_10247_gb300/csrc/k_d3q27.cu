// D3Q27 cascaded (central-moment) LB step with Strang-split body force, FP64,
// one thread per node, pull form.  arXiv:1806.10247 states the 3D method for
// D3Q15 (Appendix A) and notes that it extends to D3Q27; this is that
// extension by the generic central-moment procedure:
//
//   raw moments m_abc (a,b,c in {0,1,2})  ->  pre-collision half force on the
//   first moments (Eq. 8A analogue: m_100 += F_pre/2, ...)  ->  central moments
//   about u = m_1/rho  ->  relaxation (trace with omega_bulk towards rho,
//   deviatoric and off-diagonal second order with omega_shear towards 0, every
//   moment of order n = 3..6 with omega_n towards its Maxwellian value)  ->
//   raw moments  ->  post-collision force along K_1 = e (Eqs. 12A-13A
//   analogue, g_1 = (F_pre + F_post)/2 / 18 since sum_alpha e_x^2 = 18)  ->
//   populations.
//
// The transforms are factorised along the axes (three passes of nine 1D
// transforms on the moment orders 0, 1, 2 of the velocities -1, 0, +1), so a
// node costs ~400 FP64 operations instead of the ~1500 of dense 27 x 27
// transforms.  Moment index k = a + 3 b + 9 c matches the velocity index
// alpha = (ex+1) + 3 (ey+1) + 9 (ez+1) position by position.
#include <utility>

#include "lbm_internal.h"
#include "lbm_lattices.cuh"
#include "lbm_tiles.cuh"

namespace lbmk {
namespace {

struct Rates27 {
    double wb, ws, w3, w4, w5, w6;
};

// Populations at velocities -1, 0, +1 -> raw moments of order 0, 1, 2.
__device__ __forceinline__ void raw_fwd(double &a, double &b, double &c)
{
    const double s = c + a, d = c - a;
    a = s + b;
    b = d;
    c = s;
}
// Raw moments -> central moments about u (binomial shift, one axis).
__device__ __forceinline__ void shift_fwd(double m0, double &m1, double &m2, double u)
{
    const double k1 = fma(-u, m0, m1);
    m2 = fma(-u, m1 + k1, m2);
    m1 = k1;
}

// The way back runs on HALVED moments: every axis on which a moment has order
// 1 or 2 contributes a factor 1/2 (m~_abc = m_abc / 2^(#nonzero orders)).  The
// inverse 1D transform of a halved triple (m0, m1/2, m2/2) is then
// f_-1 = m2/2 - m1/2, f_0 = m0 - m2, f_+1 = m2/2 + m1/2: three operations per
// line instead of four, and the factors cost nothing where they land on
// constants (relaxation rates, equilibrium values, force coefficients).
//
// Halved raw moments of order 0, 1, 2 -> populations at -1, 0, +1.
__device__ __forceinline__ void raw_bwd_h(double &m0, double &m1, double &m2)
{
    const double fm = m2 - m1, fp = m2 + m1, f0 = fma(-2.0, m2, m0);
    m0 = fm;
    m1 = f0;
    m2 = fp;
}

// Apply a 1D operation to the nine triples along axis `ax` (0 x, 1 y, 2 z).
template <int AX, class Op>
__device__ __forceinline__ void along(double (&m)[27], Op op)
{
    constexpr int st = AX == 0 ? 1 : (AX == 1 ? 3 : 9);
#pragma unroll
    for (int t = 0; t < 9; t++) {
        // base index of the t-th line along AX
        const int p = AX == 0 ? 3 * t : (AX == 1 ? (t % 3) + 9 * (t / 3) : t);
        op(m[p], m[p + st], m[p + 2 * st]);
    }
}

// The back-shift, halved central moments about u -> halved raw moments (per line, uh =
// u / 2: m1 = k1 + u k0 and m2 = k2 + 2 u k1 + u^2 k0 with the halves carried along),
// with a compile-time zero pattern: bit k of Z set means m[k]
// is exactly 0 on entry (the unit-rates collision leaves 16 of the 27 halved
// central moments at 0).  An operation with a known-zero operand is left out
// and its value taken as is: fma(a, 0, x) = x, fma(a, x, 0) = a x, x + 0 = x
// (equal to the full operation up to the sign of a zero result).
template <int AX>
__host__ __device__ constexpr int line_base(int t)
{
    return AX == 0 ? 3 * t : (AX == 1 ? (t % 3) + 9 * (t / 3) : t);
}
template <int AX>
__host__ __device__ constexpr int line_stride()
{
    return AX == 0 ? 1 : (AX == 1 ? 3 : 9);
}

// Zero pattern after the back-shift along AX: on a line (k0, k1, k2), the new k1
// is 0 when k0 and k1 are, the new k2 when all three are.
template <int AX>
__host__ __device__ constexpr unsigned shift_zeros(unsigned z)
{
    unsigned r = z;
    for (int t = 0; t < 9; t++) {
        const int p0 = line_base<AX>(t), p1 = p0 + line_stride<AX>(), p2 = p0 + 2 * line_stride<AX>();
        const bool z01 = ((z >> p0) & 1u) && ((z >> p1) & 1u), z012 = z01 && ((z >> p2) & 1u);
        r = (r & ~(1u << p1) & ~(1u << p2)) | (z01 ? 1u << p1 : 0u) | (z012 ? 1u << p2 : 0u);
    }
    return r;
}

template <unsigned Z, int AX, int T>
__device__ __forceinline__ void shift_line(double (&m)[27], double u, double uh)
{
    constexpr int p0 = line_base<AX>(T), p1 = p0 + line_stride<AX>(), p2 = p0 + 2 * line_stride<AX>();
    constexpr bool z0 = (Z >> p0) & 1u, z1 = (Z >> p1) & 1u, z2 = (Z >> p2) & 1u;
    if constexpr (z0 && z1) {
        return;  // m1 = 0, and k2 keeps its value
    } else {
        double m1;
        if constexpr (z0) m1 = m[p1];
        else if constexpr (z1) m1 = uh * m[p0];
        else m1 = fma(uh, m[p0], m[p1]);
        double s;
        if constexpr (z1) s = m1;
        else s = m[p1] + m1;
        if constexpr (z2) m[p2] = u * s;
        else m[p2] = fma(u, s, m[p2]);
        m[p1] = m1;
    }
}

template <unsigned Z, int AX, int... T>
__device__ __forceinline__ void shift_lines(double (&m)[27], double u, double uh, std::integer_sequence<int, T...>)
{
    (shift_line<Z, AX, T>(m, u, uh), ...);
}

// Halved post-collision central moments about u -> populations: back-shift,
// the post-collision force in moment space, inverse raw transform.  Z: the
// moments known to be exactly 0 on entry (see shift_line).  XO: the force has
// no y and z components (their terms, additions of 0, are left out).
template <unsigned Z, bool XO>
__device__ __forceinline__ void finish(double (&m)[27], double ux, double uy, double uz, const double (&F)[3],
                                       const double (&Fq)[3])
{
    const double hx = 0.5 * ux, hy = 0.5 * uy, hz = 0.5 * uz;
    constexpr unsigned Zy = shift_zeros<0>(Z), Zz = shift_zeros<1>(Zy);
    shift_lines<Z, 0>(m, ux, hx, std::make_integer_sequence<int, 9>{});
    shift_lines<Zy, 1>(m, uy, hy, std::make_integer_sequence<int, 9>{});
    shift_lines<Zz, 2>(m, uz, hz, std::make_integer_sequence<int, 9>{});

    // K_1 g_1 in moment space, g = (F_pre + F_post) / 36: e_x changes m_100 by
    // 18 g, m_120 and m_102 by 12 g, m_122 by 8 g (halved: 9 g, 3 g, 3 g, g).
    // m_100 = rho u already carries F_pre / 2 (the pre-collision shift), so
    // only F_post / 2 is added to it.
    {
        const double sx = F[0] + Fq[0];
        m[1] = fma(0.25, Fq[0], m[1]);
        m[7] = fma(sx, 1.0 / 12.0, m[7]); m[19] = fma(sx, 1.0 / 12.0, m[19]); m[25] = fma(sx, 1.0 / 36.0, m[25]);
        if constexpr (!XO) {
            const double sy = F[1] + Fq[1], sz = F[2] + Fq[2];
            m[3] = fma(0.25, Fq[1], m[3]);
            m[9] = fma(0.25, Fq[2], m[9]);
            m[5] = fma(sy, 1.0 / 12.0, m[5]); m[21] = fma(sy, 1.0 / 12.0, m[21]); m[23] = fma(sy, 1.0 / 36.0, m[23]);
            m[11] = fma(sz, 1.0 / 12.0, m[11]); m[15] = fma(sz, 1.0 / 12.0, m[15]); m[17] = fma(sz, 1.0 / 36.0, m[17]);
        }
    }

    along<2>(m, [](double &a, double &b, double &c) { raw_bwd_h(a, b, c); });
    along<1>(m, [](double &a, double &b, double &c) { raw_bwd_h(a, b, c); });
    along<0>(m, [](double &a, double &b, double &c) { raw_bwd_h(a, b, c); });
}

// F: pre-collision force a_pre P; Fq: post-collision force a_post P; XO: the
// force has no y and z components.
template <bool XO = false>
__device__ __forceinline__ void collide(double (&m)[27], const double (&F)[3], const double (&Fq)[3],
                                        const Rates27 &w)
{
    along<0>(m, [](double &a, double &b, double &c) { raw_fwd(a, b, c); });
    along<1>(m, [](double &a, double &b, double &c) { raw_fwd(a, b, c); });
    along<2>(m, [](double &a, double &b, double &c) { raw_fwd(a, b, c); });

    // Pre-collision half force on the first moments; velocity u = m_1 / rho.
    m[1] = fma(0.5, F[0], m[1]);
    if constexpr (!XO) {
        m[3] = fma(0.5, F[1], m[3]);
        m[9] = fma(0.5, F[2], m[9]);
    }
    const double rho = m[0];
    const double rinv = recip_density(rho);
    const double ux = m[1] * rinv, uy = m[3] * rinv, uz = m[9] * rinv;

    along<0>(m, [ux](double &a, double &b, double &c) { shift_fwd(a, b, c, ux); });
    along<1>(m, [uy](double &a, double &b, double &c) { shift_fwd(a, b, c, uy); });
    along<2>(m, [uz](double &a, double &b, double &c) { shift_fwd(a, b, c, uz); });

    // Relaxation of the central moments; the results are written halved.
    {
        const double T = m[2] + m[6] + m[18];
        const double D1 = m[2] - m[6], D2 = m[2] - m[18];
        const double Ts = fma(w.wb, rho - T, T);
        const double rs = 1.0 - w.ws;
        const double rh = 0.5 * rs, rq = 0.25 * rs;
        const double D1h = rh * D1, D2h = rh * D2;  // halved relaxed deviatoric parts
        const double kxx = fma(Ts, 1.0 / 6.0, (D1h + D2h) * (1.0 / 3.0));
        m[2] = kxx;
        m[6] = kxx - D1h;
        m[18] = kxx - D2h;
        m[4] *= rq;   // 110
        m[10] *= rq;  // 101
        m[12] *= rq;  // 011
        m[1] = 0.0;   // first central moments vanish after the half force
        m[3] = 0.0;
        m[9] = 0.0;
        const double r3 = 1.0 - w.w3, r4 = 1.0 - w.w4, r5 = 1.0 - w.w5;
        const double r3q = 0.25 * r3, r3e = 0.125 * r3;
        m[5] *= r3q; m[7] *= r3q; m[11] *= r3q; m[15] *= r3q; m[19] *= r3q; m[21] *= r3q; m[13] *= r3e;
        // m~_220 = (1 - w4) m_220 / 4 + w4 (rho / 9) / 4
        const double r4q = 0.25 * r4, e4 = (w.w4 * (1.0 / 36.0)) * rho;
        m[8] = fma(r4q, m[8], e4);
        m[20] = fma(r4q, m[20], e4);
        m[24] = fma(r4q, m[24], e4);
        const double r4e = 0.125 * r4, r5e = 0.125 * r5;
        m[14] *= r4e; m[16] *= r4e; m[22] *= r4e;
        m[17] *= r5e; m[23] *= r5e; m[25] *= r5e;
        m[26] = fma(0.125 * (1.0 - w.w6), m[26], (w.w6 * (1.0 / 216.0)) * rho);
    }

    finish<0u, XO>(m, ux, uy, uz, F, Fq);
}

// Halved central moments the unit-rates collision leaves exactly 0: all but
// 000, 200, 020, 002, 110, 101, 011, 220, 202, 022, 222 (index a + 3b + 9c).
constexpr unsigned kNonZeroW1 = (1u << 0) | (1u << 2) | (1u << 6) | (1u << 18) | (1u << 4) | (1u << 10) | (1u << 12) |
                                (1u << 8) | (1u << 20) | (1u << 24) | (1u << 26);
constexpr unsigned kZeroW1 = ((1u << 27) - 1u) & ~kNonZeroW1;

// The same collision when omega_3 = omega_4 = omega_5 = omega_6 = 1 (the
// paper's choice for the higher moments, Sec. 6): every central moment of
// order 3..6 lands exactly on its Maxwellian value, so only the raw moments of
// order <= 2 are formed (partial transforms) and the forward shift reduces to
// the six second-order central moments.
template <bool XO = false>
__device__ __forceinline__ void collide_w1(double (&m)[27], const double (&F)[3], const double (&Fq)[3],
                                           const Rates27 &w)
{
    along<0>(m, [](double &a, double &b, double &c) { raw_fwd(a, b, c); });
    // Line (b, c) along x holds M0, M1, M2 at m[3b + 9c + 0..2]; e_y = b - 1, e_z = c - 1.
    double Y0[3], Y1[3], Y2[3], X0[3], X1[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const double s = m[9 * c + 6] + m[9 * c], d = m[9 * c + 6] - m[9 * c];
        Y0[c] = s + m[9 * c + 3];
        Y1[c] = d;
        Y2[c] = s;
        X0[c] = (m[9 * c + 7] + m[9 * c + 1]) + m[9 * c + 4];
        X1[c] = m[9 * c + 7] - m[9 * c + 1];
    }
    const double rho = (Y0[2] + Y0[0]) + Y0[1];
    double jz = Y0[2] - Y0[0];
    const double kzz = Y0[2] + Y0[0];
    double jy = (Y1[2] + Y1[0]) + Y1[1];
    const double kyz = Y1[2] - Y1[0];
    const double kyy = (Y2[2] + Y2[0]) + Y2[1];
    double jx = (X0[2] + X0[0]) + X0[1];
    const double kxz = X0[2] - X0[0];
    const double kxy = (X1[2] + X1[0]) + X1[1];
    const double kxx = ((m[2] + m[5]) + (m[8] + m[11])) + ((m[14] + m[17]) + (m[20] + m[23])) + m[26];

    jx = fma(0.5, F[0], jx);
    if constexpr (!XO) {
        jy = fma(0.5, F[1], jy);
        jz = fma(0.5, F[2], jz);
    }
    const double rinv = recip_density(rho);
    const double ux = jx * rinv, uy = jy * rinv, uz = jz * rinv;

    // Second-order central moments (the first ones vanish) and their relaxation.
    const double cxx = fma(-jx, ux, kxx), cyy = fma(-jy, uy, kyy), czz = fma(-jz, uz, kzz);
    const double T = cxx + cyy + czz;
    const double D1 = cxx - cyy, D2 = cxx - czz;
    const double Ts = fma(w.wb, rho - T, T);
    const double rs = 1.0 - w.ws;
    const double rh = 0.5 * rs, rq = 0.25 * rs;
    const double D1h = rh * D1, D2h = rh * D2;
    const double sxx = fma(Ts, 1.0 / 6.0, (D1h + D2h) * (1.0 / 3.0));
    // halved post-collision central moments (orders 3..6 at their Maxwellian values)
#pragma unroll
    for (int k = 0; k < 27; k++) m[k] = 0.0;
    m[0] = rho;
    m[2] = sxx;
    m[6] = sxx - D1h;
    m[18] = sxx - D2h;
    m[4] = rq * fma(-jx, uy, kxy);
    m[10] = rq * fma(-jx, uz, kxz);
    m[12] = rq * fma(-jy, uz, kyz);
    const double e4 = rho * (1.0 / 36.0);
    m[8] = e4;
    m[20] = e4;
    m[24] = e4;
    m[26] = rho * (1.0 / 216.0);
    finish<kZeroW1, XO>(m, ux, uy, uz, F, Fq);
}

// One node's step in fixed point (unit higher rates): get() pulls the
// populations, shape(d) gives the force shape's component d, q1 = a_pre / 4 and
// q2 = (a_pre + a_post) / 4, put(a, f) stores a result.
template <bool FORCED, bool XO, class Shape, class Put>
__device__ __forceinline__ FxStep fixed_step27(const double (&f)[27], const FxRates &w, double q1, double q2, Shape shape,
                                             Put put)
{
    const int em = fx_emax(f);
    const int k = FxGrid<27>::S + 1023 - em;
    if (!fx_in_range(em)) return FX_NOT;
    int bad = 0;
    FxForce F[3] = {{0, 0}, {0, 0}, {0, 0}};
    if (FORCED) {
        const unsigned dither = (unsigned)fx_bits(f[13]);
#pragma unroll
        for (int d = 0; d < (XO ? 1 : 3); d++)
            if (!fx_force(shape(d), q1, q2, k, em, dither >> (8 * d), F[d])) bad = -1;
        if (bad < 0) return FX_NOT;
    }
    i64 X[27];
    fx_load(f, k, X);
    FxSums27<i64> s;
    fx_sums27(X, s);
    fx_collide27<XO>(s, F, w, X, bad);
#pragma unroll
    for (int a = 0; a < 27; a++) put(a, fx_value_pos(X[a], k + 1, bad));
    return bad >= 0 ? FX_DONE : FX_GIVEN_UP;
}

// The FP64 form of a node's step.
template <bool W1, bool XO, class Shape>
__device__ __forceinline__ void double_step27(double (&m)[27], const Rates27 &w, bool forced, double apre, double apost,
                                              Shape shape)
{
    double F[3] = {0.0, 0.0, 0.0}, Fq[3] = {0.0, 0.0, 0.0};
    if (forced) {
#pragma unroll
        for (int d = 0; d < (XO ? 1 : 3); d++) {
            const double P = shape(d);
            F[d] = apre * P;
            Fq[d] = apost * P;
        }
    }
    if (W1) collide_w1<XO>(m, F, Fq, w);
    else collide<XO>(m, F, Fq, w);
}

// 6 resident blocks of 128 threads (80 registers, 40 bytes spilled): the step
// waits for the conversions' results and for integer chains more than for
// memory, so warps in flight matter.  Kolmogorov 256^3 FP64, 4 steps and the
// fields: 2 blocks of 256 threads 9.63 ms, 4 of 128 8.41, 5 of 128 8.37, 6 of 128
// 8.16; 8 or 10 of 64 8.38 / 8.36.
constexpr int kStepBlock = 128, kStepMinBlocks = 6;

// The step loads its populations over the read-only path; overlapped steps (see
// step_wait) may not, and the plain loads cost this kernel 2.5 % (160^3, 8 steps
// and the fields: 3.59 / 3.65 ms).  The launches that overlap hides are 8 % of 64^3
// (0.637 -> 0.584 ms for 16 steps and the fields), 1.5 % of 96^3 and nothing from 102^3 on:
// the line lies between the two.  No step_next: a grid of 152 to 912 blocks
// leaves room on every SM, and blocks placed while those of the step before still
// run come to lie unevenly (40^3: 0.270 ms apart, 0.293 so, 0.233 with the
// blocks placed as the earlier ones end).
constexpr int kOverlapNodes = 1 << 20;

// XO: the force has no y and z components (checked on the host).  OV: an
// overlapped step.
template <int FK, bool W1, bool XO, bool OV>
__global__ void __launch_bounds__(kStepBlock, W1 ? kStepMinBlocks : 1)
k_step(const __grid_constant__ Planes<double, 27> P, Geom g, FieldDev Fd, double apre, double apost, Rates27 w,
       FxRates fx, double q1, double q2)
{
    if (OV) step_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    int x, y, z;
    node_xyz(g, i, x, y, z);
    double m[27];
    load_pulled<LD3Q27, !OV>(P, g, x, y, z, i, m);
    auto shape = [&](int d) { return field_value(Fd, FK, d, x, y, z, i); };
    if (W1) {
        const FxStep r = fixed_step27<FK != FK_NONE, XO>(m, fx, q1, q2, shape, [&](int a, double v) { P.out[a][i] = v; });
        if (r == FX_DONE) return;
        if (r == FX_GIVEN_UP) load_pulled<LD3Q27, !OV>(P, g, x, y, z, i, m);
    }
    double_step27<W1, XO>(m, w, FK != FK_NONE, apre, apost, shape);
#pragma unroll
    for (int a = 0; a < 27; a++) P.out[a][i] = m[a];
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
    double m[27];
    load_pulled<LD3Q27>(fin, g, x, y, z, i, m);
    // fused readback of f(t)'s fields
    if (L.mrho) fused_fields<LD3Q27>(B, L, it, i, x, y, z, m, 2.0 * ap.q1);
    const bool forced = B.fkind != FK_NONE;
    auto shape = [&](int d) { return forced ? field_value(B.F, B.fkind, d, x, y, z, i) : 0.0; };
    auto put = [&](int a, double v) { fout[a * g.Np + i] = v; };
    const Rates27 w{B.coef[0], B.coef[1], B.coef[2], B.coef[3], B.coef[4], B.coef[5]};
    if (B.variant == 3) {  // uniform over the member
        const FxStep r = fixed_step27<true, true>(m, B.fx, ap.q1, ap.q2, shape, put);
        if (r == FX_DONE) return;
        if (r == FX_GIVEN_UP) load_pulled<LD3Q27>(fin, g, x, y, z, i, m);
        double_step27<true, true>(m, w, forced, ap.pre, ap.g, shape);
    } else if (B.variant == 1) {
        const FxStep r = fixed_step27<true, false>(m, B.fx, ap.q1, ap.q2, shape, put);
        if (r == FX_DONE) return;
        if (r == FX_GIVEN_UP) load_pulled<LD3Q27>(fin, g, x, y, z, i, m);
        double_step27<true, false>(m, w, forced, ap.pre, ap.g, shape);
    } else {
        double_step27<false, false>(m, w, forced, ap.pre, ap.g, shape);
    }
#pragma unroll
    for (int a = 0; a < 27; a++) put(a, m[a]);
}

// At most 128 registers: 16 warps per SM at every tile size.
template <int TB, int MODE>
__global__ void __launch_bounds__(TB, 512 / TB) k_batch(const __grid_constant__ BatchLaunch L)
{
    batch_tiles<TB, MODE>(L, [](const BatchItem &B, const BatchLaunch &L2, int it, int i) { batch_node(B, L2, it, i); });
}

bool high_rates_one(const double *om) { return om[3] == 1.0 && om[4] == 1.0 && om[5] == 1.0 && om[6] == 1.0; }

}  // namespace

// coef[0..5] = omega[1..6]
void d3q27_batch_coef(const double omega[9], BatchItem &item)
{
    for (int k = 0; k < 6; k++) item.coef[k] = omega[k + 1];
    item.fx = fx_rates27(omega[1], omega[2]);
}

cudaError_t d3q27_batch_step(const BatchLaunch &L, int nblocks, int tile, cudaStream_t s)
{
    LBM_TILED_LAUNCH(k_batch, L, nblocks, tile, s);
}

int d3q27_batch_resident(int tile)
{
    LBM_TILED_RESIDENT(k_batch, tile);
}

bool d3q27_high_rates_one(const double omega[9]) { return high_rates_one(omega); }

cudaError_t d3q27_step(const LaunchArgs &a)
{
    Rates27 w{a.omega[1], a.omega[2], a.omega[3], a.omega[4], a.omega[5], a.omega[6]};
    const int block = spread_block(a.g.N, kStepBlock), grid = (a.g.N + block - 1) / block;
    const double q1 = 0.25 * a.apre, q2 = 0.25 * (a.apre + a.apost);
    const bool w1 = high_rates_one(a.omega);
    const Planes<double, 27> P = make_planes<double, 27>(a.fin, a.fout, a.g.Np);
    const bool xo = force_x_only(a.fkind, a.F, 3);
    const FxRates fx = fx_rates27(a.omega[1], a.omega[2]);
    const bool ov = w1 && a.g.N <= kOverlapNodes;
#define STEP27(FK, W1, XO, OV) \
    launch_step(OV && a.overlap, k_step<FK, W1, XO, OV>, grid, block, a.stream, P, a.g, a.F, a.apre, a.apost, w, fx, q1, q2)
#define STEP27_W1(FK, XO) (ov ? STEP27(FK, true, XO, true) : STEP27(FK, true, XO, false))
    switch (a.fkind) {
    case FK_NONE: return w1 ? STEP27_W1(FK_NONE, false) : STEP27(FK_NONE, false, false, false);
    case FK_CONST:
        return !w1 ? STEP27(FK_CONST, false, false, false) : xo ? STEP27_W1(FK_CONST, true) : STEP27_W1(FK_CONST, false);
    default:
        return !w1 ? STEP27(FK_GENERAL, false, false, false)
                   : xo ? STEP27_W1(FK_GENERAL, true) : STEP27_W1(FK_GENERAL, false);
    }
#undef STEP27_W1
#undef STEP27
}

}  // namespace lbmk
