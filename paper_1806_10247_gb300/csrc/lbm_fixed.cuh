// FP64 steps in fixed point.
//
// This GPU issues 1.69 FP64 adds, multiplies or multiply-adds per clock and SM
// (2.0 conversions between FP64 and integers), but 62 64-bit integer adds and
// about 5 signed 64 x 64 -> high-64 products, and the two kinds of unit work
// side by side.  So the step kernels of the FP64 storage convert a node's
// populations to 64-bit integers at one scale per node, run the moment
// transforms and the collision on those, and convert the results back.
//
// Scale: with E the exponent of the node's largest |f|, X = f 2^(S - E),
// rounded to nearest even, |X| < 2^(S + 1).  S (FxGrid) leaves the headroom
// that the sums of the lattice need and keeps S - 52 bits below the last bit
// of the largest population (3 on D3Q27, 5 on D2Q9): the sums and differences
// of the transforms are then exact, and a product rounds at 2^-S of the
// largest population, where an FP64 operation on quantities of the size of rho
// rounds at 2^-53 of rho.  Mass and momentum are carried without any rounding
// between the two conversions.  The result is rounded to FP64 once, to nearest
// even.
//
// What the fixed-point form does not take is left to the FP64 form of that node: known
// before any of its work, a population that is not finite, an exponent outside
// [kEmaxLo, kEmaxHi] (a scalar on a background of 0) or a force as large as the
// populations; found on the way, |u| >= 1/2, a density far below the largest population, a
// result that is negative or below 2^-25 of the largest population (FxStep).
//
// Everything here compiles for the host too (tests run it against 64-bit and
// wider arithmetic on the CPU).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#include <math.h>
#include <string.h>
#define FX_HD inline
#endif

namespace lbmk {

// What a node's step in fixed point did: FX_DONE, FX_NOT (nothing: the populations are as
// they were) or FX_GIVEN_UP (its results are void, the populations to be pulled again:
// keeping them beside the fixed-point values would cost registers at every node).
enum FxStep { FX_DONE, FX_NOT, FX_GIVEN_UP };

typedef long long i64;
typedef unsigned long long u64;

// ---- words ------------------------------------------------------------------
FX_HD u64 fx_bits(double x)
{
#ifdef __CUDA_ARCH__
    return (u64)__double_as_longlong(x);
#else
    u64 b;
    memcpy(&b, &x, 8);
    return b;
#endif
}
FX_HD double fx_double(u64 b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((i64)b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}
FX_HD unsigned fx_hi(u64 b) { return (unsigned)(b >> 32); }

// High 64 bits of the signed product.
FX_HD i64 fx_mul(i64 a, i64 b)
{
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (i64)(((__int128)a * b) >> 64);
#endif
}
// x 2^n for a normal x or 0 (which becomes a value below 2^(n - 1000)): an
// integer add on the exponent, no FP64 operation.
FX_HD double fx_ldexp(double x, int n) { return fx_double(fx_bits(x) + ((u64)(unsigned)n << 52)); }
// Round to nearest even.
FX_HD i64 fx_round(double x)
{
#ifdef __CUDA_ARCH__
    return __double2ll_rn(x);
#else
    return llrint(x);
#endif
}
FX_HD double fx_to_double(i64 x)
{
#ifdef __CUDA_ARCH__
    return __ll2double_rn(x);
#else
    return (double)x;
#endif
}
// About 1/x to 2^-22, x > 0.
FX_HD float fx_rcp_approx(float x)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / x;
#endif
}
FX_HD unsigned fx_float_bits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    unsigned b;
    memcpy(&b, &x, 4);
    return b;
#endif
}
FX_HD float fx_float(unsigned b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    memcpy(&x, &b, 4);
    return x;
#endif
}
// A positive normal float as a double: the exponent field re-biased, the mantissa
// moved up (no FP64 conversion).
FX_HD double fx_widen(float x)
{
    return fx_double(((u64)fx_float_bits(x) << 29) + ((u64)(1023 - 127) << 52));
}
// 1/x for a positive normal x (biased exponent 3 .. 2043), correctly rounded: a 22-bit
// reciprocal of the mantissa r with one third-order correction, r (1 + e + e^2), e = 1 -
// x r, is within 0.51 units of the last place; with X and Y the mantissas of x and of that
// result as integers, 2^105 - X Y (known from its low 64 bits, as it is below X in
// magnitude) tells whether a neighbour is nearer.  Three FP64 operations and about
// fifteen of the integer unit, where the maths library's reciprocal takes about seven of
// the FP64 unit, which bounds the readbacks.
FX_HD double fx_recip(double x)
{
    constexpr u64 kMant = 0x000fffffffffffffull, kLead = 0x0010000000000000ull;
    const u64 b = fx_bits(x);
    const u64 m = (b & kMant) | 0x3ff0000000000000ull;      // mantissa in [1, 2)
    const double r = fx_widen(fx_rcp_approx(fx_float(0x3f800000u | ((unsigned)(m >> 29) & 0x7fffffu))));
    const double e = fma(-fx_double(m), r, 1.0);
    const double p = fma(e, e, e);
    u64 y = fx_bits(fma(r, p, r));
    const i64 X = (i64)((b & kMant) | kLead);
    const i64 R2 = (i64)(0ull - 2ull * (u64)X * ((y & kMant) | kLead));
    if (R2 > X) y++;
    if (R2 < -X) y--;
    return fx_ldexp(fx_double(y), 1023 - (int)(b >> 52));
}

// ---- scale --------------------------------------------------------------------
constexpr int kEmaxLo = 500, kEmaxHi = 1073;  // biased exponents the fixed-point forms take (2^-523 .. 2^50)

// S by lattice: after the forward transform the grid is refined by one bit (so
// that half of a first moment is an integer), and the largest sum formed is the
// trace of the second moments, at most sum |e|^2 = 54 (D3Q27), 30 (D3Q15), 12
// (D2Q9) times the largest population: 54 2^(S + 2) < 2^63 and so on.
template <int Q>
struct FxGrid;
template <>
struct FxGrid<27> {
    static constexpr int S = 55;
};
template <>
struct FxGrid<15> {
    static constexpr int S = 56;
};
template <>
struct FxGrid<9> {
    static constexpr int S = 57;
};
template <>
struct FxGrid<5> {
    static constexpr int S = 57;
};

// Biased exponent of the largest |f|.
template <int Q>
FX_HD int fx_emax(const double (&f)[Q])
{
    unsigned m = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < Q; a++) {
        const unsigned h = fx_hi(fx_bits(f[a])) & 0x7fffffffu;
        m = h > m ? h : m;
    }
    return (int)(m >> 20);
}
FX_HD bool fx_in_range(int emax) { return (unsigned)(emax - kEmaxLo) <= (unsigned)(kEmaxHi - kEmaxLo); }

// Populations at the node's scale; k = S + 1023 - emax.
template <int Q>
FX_HD void fx_load(const double (&f)[Q], int k, i64 (&X)[Q])
{
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < Q; a++) X[a] = fx_round(fx_ldexp(f[a], k));
}

// The same in integers alone (a conversion costs half a clock of the FP64 unit,
// this about a tenth of the integer units'), to nearest with halves away from
// zero: exact for values within S - 52 binary orders of the largest.  SIGNED =
// false takes |f|.
template <int Q, bool SIGNED>
FX_HD void fx_load_int(const double (&f)[Q], int emax, i64 (&X)[Q])
{
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < Q; a++) {
        const u64 b = fx_bits(f[a]);
        const int e = (int)(fx_hi(b) >> 20) & 0x7ff;
        const int sh = emax - e < 63 ? emax - e : 63;
        const u64 m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
        const i64 v = (i64)(((m << (FxGrid<Q>::S - 51)) >> sh) + 1) >> 1;
        const i64 s = (i64)b >> 63;
        X[a] = SIGNED ? (v ^ s) - s : v;
    }
}

// FP32 deviations as integers X = d 2^(182 - em), em the biased exponent of the largest:
// 24-bit values, 32 bits below the largest one's last, rounded towards zero.  Not taken:
// em below 56, where the leading bit that a zero or a subnormal value does not have
// (added to every value) would not yet be shifted out, and a value that is not finite.
enum FxDev { FXD_ZERO, FXD_TAKEN, FXD_NOT };
template <int Q>
FX_HD FxDev fx_load_dev(const float (&d)[Q], int &em, i64 (&X)[Q])
{
    unsigned m = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < Q; a++) {
        const unsigned b = fx_float_bits(d[a]) & 0x7fffffffu;
        m = b > m ? b : m;
    }
    em = (int)(m >> 23);
    if (m == 0) return FXD_ZERO;
    if (em < 56 || em >= 255) return FXD_NOT;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < Q; a++) {
        const unsigned b = fx_float_bits(d[a]);
        const int sh = em - (int)((b >> 23) & 0xffu);
        const u64 v = (u64)((b & 0x7fffffu) | 0x800000u) << 32 >> (sh < 63 ? sh : 63);
        const i64 s = (i64)((int)b >> 31);
        X[a] = ((i64)v ^ s) - s;
    }
    return FXD_TAKEN;
}

// X 2^-k, rounded to nearest even; 0 gives 0.
FX_HD double fx_value(i64 X, int k)
{
    const double d = fx_to_double(X);
    return X == 0 ? 0.0 : fx_ldexp(d, -k);
}

// The same for 2^32 <= X < 2^62, without an FP64 conversion: shift the leading
// bit to bit 62, round away the 10 bits below FP64's last one (to nearest
// even), add the exponent.  `bad` goes negative for any other X.
FX_HD double fx_value_pos(i64 X, int k, int &bad)
{
    const unsigned hi = (unsigned)((u64)X >> 32);
    bad |= (int)hi - 1;
#ifdef __CUDA_ARCH__
    unsigned n;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(n) : "r"(hi));
    n -= 1u;
#else
    if ((int)hi <= 0) return 0.0;
    const unsigned n = (unsigned)__builtin_clz(hi) - 1u;
#endif
    u64 v = (u64)X << n;
    v += 0x1ffull + ((v >> 10) & 1ull);
    v >>= 10;
    // v = 2^52 .. 2^53: its leading bit adds one to the exponent field
    return fx_double(v + ((u64)(unsigned)(1023 + 51 + 10 - k - (int)n) << 52));
}

// The same for values of either sign, 2^32 <= |X| < 2^62.
FX_HD double fx_value_signed(i64 X, int k, int &bad)
{
    const i64 s = X >> 63;
    return fx_double(fx_bits(fx_value_pos((X ^ s) - s, k, bad)) | ((u64)X & 0x8000000000000000ull));
}

// fx_value with its FP64 conversion left to |X| < 2^32, for kernels that the FP64 unit bounds.
FX_HD double fx_value_int(i64 X, int k)
{
    int bad = 0;
    const double v = fx_value_signed(X, k, bad);
    return bad >= 0 ? v : fx_value(X, k);
}

// ---- force --------------------------------------------------------------------
// Fixed-point form of a force along one axis at a node, on the refined grid
// (scale 2^(k + 1)): h1 = F_pre / 4 (half of the pre-collision half force),
// h2 = (F_pre + F_post) / 4.  h2 enters the momentum of every step, so it is
// rounded with 8 more bits and a dither from the node's own low bits: a fixed
// rounding would add up over a steady run.
struct FxForce {
    i64 h1, h2;
};
// q1 = a_pre / 4, q2 = (a_pre + a_post) / 4, P the shape's value.  With q2 = 2
// q1 (an envelope that does not change over the step; compared by its bits, an
// FP64 comparison costs as much as the product) one product and one conversion do.
FX_HD bool fx_force(double P, double q1, double q2, int k, int emax, unsigned dither, FxForce &F)
{
    const double f2 = q2 * P;
    unsigned m = fx_hi(fx_bits(f2)) & 0x7fffffffu;
    F.h2 = (fx_round(fx_ldexp(f2, k + 9)) + (i64)(dither & 0xffu)) >> 8;
    if (fx_bits(q2) == fx_bits(q1) + (1ull << 52)) {
        F.h1 = F.h2 >> 1;
    } else {
        const double f1 = q1 * P;
        const unsigned m1 = fx_hi(fx_bits(f1)) & 0x7fffffffu;
        m = m1 > m ? m1 : m;
        F.h1 = fx_round(fx_ldexp(f1, k + 1));
    }
    return (int)(m >> 20) <= emax - 6;
}

// ---- velocity -----------------------------------------------------------------
// 2^64 / rho to a relative 2^-52; bad < 0 when rho is not above 2^52.
FX_HD double fx_reciprocal(i64 rho, int &bad)
{
    const int rh = (int)(rho >> 32);
    bad |= rh - (1 << 20);
    const double r = fx_ldexp(fx_to_double(rho), -32);
    const double x = fx_widen(fx_rcp_approx((float)rh));
    // x (1 + e + e^2) with e = 1 - r x, |e| < 2^-19
    const double e = fma(-r, x, 1.0);
    const double p = fma(e, e, e);
    return fx_ldexp(fma(x, p, x), 32);
}
// j / rho 2^64 for |j| < rho / 2, ri = 2^64 / rho; bad < 0 for a larger |j|.
FX_HD i64 fx_ratio(i64 j, i64 rho, double ri, int &bad)
{
    // rho / 2 - 1 - |j| >= 0 (the shift is exact up to one unit)
    bad |= (int)((((rho >> 1) - 1) - (j < 0 ? -j : j)) >> 32);
    return fx_round(fx_to_double(j) * ri);
}

// Constants as fractions of 2^64.
constexpr i64 kFx3 = 0x5555555555555555ll;   // 1/3
constexpr i64 kFx6 = 0x2aaaaaaaaaaaaaabll;   // 1/6
constexpr i64 kFx9 = 0x1c71c71c71c71c72ll;   // 1/9
constexpr i64 kFx36 = 0x071c71c71c71c71cll;  // 1/36
constexpr i64 kFx216 = 0x012f684bda12f685ll; // 1/216

// Relaxation factors of a launch: shear (1 - omega_s) 2^63 and bulk
// (omega_b - 1) 2^63 (D3Q27); D2Q9: (1 - omega_4) 2^62, (1 - omega_5) 2^62 and
// (omega_3 - 1) 2^62.
struct FxRates {
    i64 a, b, c;
};
inline i64 fx_fraction(double x, int bits)
{
    const double v = x * (double)(1ll << (bits - 1)) * 2.0, top = 9223372036854774784.0;  // 2^63 - 1024
    return (i64)(v > top ? top : (v < -top ? -top : v));
}
inline FxRates fx_rates27(double wb, double ws) { return FxRates{fx_fraction(1.0 - ws, 63), fx_fraction(wb - 1.0, 63), 0}; }
inline FxRates fx_rates9(double w3, double w4, double w5)
{
    return FxRates{fx_fraction(1.0 - w4, 62), fx_fraction(1.0 - w5, 62), fx_fraction(w3 - 1.0, 62)};
}

// ---- D3Q27 --------------------------------------------------------------------
// The forward sums of a node's populations (fixed point or any other type), as
// far as a unit-rates collision and a readback need them.
template <class V>
struct FxSums27 {
    V rho, jx, jy, jz, xx, yy, zz, xy, xz, yz;
};
template <class V>
FX_HD void fx_sums27(const V (&f)[27], FxSums27<V> &s)
{
    V a0[9], a1[9], a2[9];  // lines along x: order 0, 1, 2
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int t = 0; t < 9; t++) {
        const V e = f[3 * t + 2] + f[3 * t];
        a0[t] = e + f[3 * t + 1];
        a1[t] = f[3 * t + 2] - f[3 * t];
        a2[t] = e;
    }
    V Y0[3], Y1[3], Y2[3], X0[3], X1[3];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int c = 0; c < 3; c++) {
        const V e = a0[3 * c + 2] + a0[3 * c];
        Y0[c] = e + a0[3 * c + 1];
        Y1[c] = a0[3 * c + 2] - a0[3 * c];
        Y2[c] = e;
        X0[c] = a1[3 * c + 2] + a1[3 * c] + a1[3 * c + 1];
        X1[c] = a1[3 * c + 2] - a1[3 * c];
    }
    s.zz = Y0[2] + Y0[0];
    s.rho = s.zz + Y0[1];
    s.jz = Y0[2] - Y0[0];
    s.jy = Y1[2] + Y1[0] + Y1[1];
    s.yz = Y1[2] - Y1[0];
    s.yy = Y2[2] + Y2[0] + Y2[1];
    s.jx = X0[2] + X0[0] + X0[1];
    s.xz = X0[2] - X0[0];
    s.xy = X1[2] + X1[0] + X1[1];
    s.xx = ((a2[0] + a2[1]) + (a2[2] + a2[3])) + ((a2[4] + a2[5]) + (a2[6] + a2[7])) + a2[8];
}

// One line of the halved back-shift (k0, k1/2, k2/2 central -> raw); UH = U / 2.
FX_HD void fx_shift(i64 k0, i64 &k1, i64 &k2, i64 U, i64 UH)
{
    const i64 m1 = k1 + fx_mul(k0, UH);
    k2 += fx_mul(k1 + m1, U);
    k1 = m1;
}
// Lines with known zeros: k1 = k2 = 0 on entry; k0 = k2 = 0.
FX_HD void fx_shift_k0(i64 k0, i64 &k1, i64 &k2, i64 U, i64 UH)
{
    k1 = fx_mul(k0, UH);
    k2 = fx_mul(k1, U);
}
// k2 = 0 on entry.
FX_HD void fx_shift_k01(i64 k0, i64 &k1, i64 &k2, i64 U, i64 UH)
{
    const i64 m1 = k1 + fx_mul(k0, UH);
    k2 = fx_mul(k1 + m1, U);
    k1 = m1;
}
FX_HD void fx_shift_k1(i64 k1, i64 &k2, i64 U) { k2 = fx_mul(k1 + k1, U); }
// k1 = 0 on entry.
FX_HD void fx_shift_k02(i64 k0, i64 &k1, i64 &k2, i64 U, i64 UH)
{
    k1 = fx_mul(k0, UH);
    k2 += fx_mul(k1, U);
}
// k1 known (half of a first moment), its central value 0.
FX_HD void fx_shift_first(i64 k1, i64 &k2, i64 U) { k2 += fx_mul(k1, U); }

FX_HD void fx_back(i64 &m0, i64 &m1, i64 &m2)
{
    const i64 a = m2 - m1, b = m2 + m1;
    m1 = m0 - m2 - m2;
    m0 = a;
    m2 = b;
}

// The D3Q27 collision with omega_3 .. omega_6 = 1 (see k_d3q27.cu collide_w1
// for the steps): s are the sums on the grid k, force F per axis (axes 1 and 2
// unused with XO).  m: post-collision populations on the grid k + 1.
template <bool XO>
FX_HD void fx_collide27(const FxSums27<i64> &s, const FxForce (&F)[3], const FxRates &w, i64 (&m)[27], int &bad)
{
    // halves of the half-forced first moments on the refined grid: j / 2 there is j here
    const i64 hx = s.jx + F[0].h1, hy = XO ? s.jy : s.jy + F[1].h1, hz = XO ? s.jz : s.jz + F[2].h1;
    const i64 rho = s.rho + s.rho;
    const i64 j[3] = {hx + hx, hy + hy, hz + hz};
    const double ri = fx_reciprocal(rho, bad);
    const i64 U[3] = {fx_ratio(j[0], rho, ri, bad), fx_ratio(j[1], rho, ri, bad), fx_ratio(j[2], rho, ri, bad)};
    const i64 cxx = s.xx + s.xx - fx_mul(j[0], U[0]), cyy = s.yy + s.yy - fx_mul(j[1], U[1]);
    const i64 czz = s.zz + s.zz - fx_mul(j[2], U[2]);
    const i64 cxy = s.xy + s.xy - fx_mul(j[0], U[1]), cxz = s.xz + s.xz - fx_mul(j[0], U[2]);
    const i64 cyz = s.yz + s.yz - fx_mul(j[1], U[2]);
    // relaxation: Ts = T + omega_b (rho - T); halved deviatoric parts
    i64 Ts = rho;
    if (w.b != 0) {
        const i64 d = fx_mul(rho - (cxx + cyy + czz), w.b);
        Ts += d + d;
    }
    const i64 D1h = fx_mul(cxx - cyy, w.a), D2h = fx_mul(cxx - czz, w.a);
    const i64 sxx = fx_mul(Ts, kFx6) + fx_mul(D1h + D2h, kFx3);
    const i64 wq = w.a >> 1;
    const i64 e4 = fx_mul(rho, kFx36);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int q = 0; q < 27; q++) m[q] = 0;
    m[0] = rho;
    m[1] = hx;
    m[3] = hy;
    m[9] = hz;
    m[2] = sxx;
    m[6] = sxx - D1h;
    m[18] = sxx - D2h;
    m[4] = fx_mul(cxy, wq);
    m[10] = fx_mul(cxz, wq);
    m[12] = fx_mul(cyz, wq);
    m[8] = m[20] = m[24] = e4;
    m[26] = fx_mul(rho, kFx216);
    const i64 ux = U[0], uy = U[1], uz = U[2], uhx = ux >> 1, uhy = uy >> 1, uhz = uz >> 1;
    // along x: (b, c) = (0,0) (1,0) (2,0) (0,1) (1,1) (0,2) (2,2); the other lines are 0
    fx_shift_first(m[1], m[2], ux);
    fx_shift_k1(m[4], m[5], ux);
    fx_shift_k02(m[6], m[7], m[8], ux, uhx);
    fx_shift_k1(m[10], m[11], ux);
    fx_shift_k0(m[12], m[13], m[14], ux, uhx);
    fx_shift_k02(m[18], m[19], m[20], ux, uhx);
    fx_shift_k02(m[24], m[25], m[26], ux, uhx);
    // along y, lines (a, c)
    fx_shift_first(m[3], m[6], uy);
    fx_shift(m[1], m[4], m[7], uy, uhy);
    fx_shift(m[2], m[5], m[8], uy, uhy);
    fx_shift_k1(m[12], m[15], uy);
    fx_shift_k01(m[10], m[13], m[16], uy, uhy);
    fx_shift_k01(m[11], m[14], m[17], uy, uhy);
    fx_shift_k02(m[18], m[21], m[24], uy, uhy);
    fx_shift_k02(m[19], m[22], m[25], uy, uhy);
    fx_shift_k02(m[20], m[23], m[26], uy, uhy);
    // along z, lines (a, b)
    fx_shift_first(m[9], m[18], uz);
    fx_shift(m[1], m[10], m[19], uz, uhz);
    fx_shift(m[2], m[11], m[20], uz, uhz);
    fx_shift(m[3], m[12], m[21], uz, uhz);
    fx_shift(m[4], m[13], m[22], uz, uhz);
    fx_shift(m[5], m[14], m[23], uz, uhz);
    fx_shift(m[6], m[15], m[24], uz, uhz);
    fx_shift(m[7], m[16], m[25], uz, uhz);
    fx_shift(m[8], m[17], m[26], uz, uhz);
    // post-collision force: m_100 gains F_post / 2, m_120 and m_102 (F_pre +
    // F_post) / 3, m_122 (F_pre + F_post) 2 / 9; halved per nonzero order
    m[1] = s.jx + F[0].h2;
    {
        const i64 g3 = fx_mul(F[0].h2, kFx3), g9 = fx_mul(F[0].h2, kFx9);
        m[7] += g3;
        m[19] += g3;
        m[25] += g9;
    }
    if (!XO) {
        m[3] = s.jy + F[1].h2;
        m[9] = s.jz + F[2].h2;
        const i64 g3 = fx_mul(F[1].h2, kFx3), g9 = fx_mul(F[1].h2, kFx9);
        m[5] += g3;
        m[21] += g3;
        m[23] += g9;
        const i64 h3 = fx_mul(F[2].h2, kFx3), h9 = fx_mul(F[2].h2, kFx9);
        m[11] += h3;
        m[15] += h3;
        m[17] += h9;
    }
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int t = 0; t < 9; t++) fx_back(m[t], m[t + 9], m[t + 18]);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int t = 0; t < 9; t++) fx_back(m[t % 3 + 9 * (t / 3)], m[t % 3 + 9 * (t / 3) + 3], m[t % 3 + 9 * (t / 3) + 6]);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int t = 0; t < 9; t++) fx_back(m[3 * t], m[3 * t + 1], m[3 * t + 2]);
}

// ---- D2Q9 ---------------------------------------------------------------------
template <class V>
struct FxSums9 {
    V rho, jx, jy, xx, yy, xy;
};
template <class V>
FX_HD void fx_sums9(const V (&f)[9], FxSums9<V> &s)
{
    const V s0 = f[1] + f[3], d0 = f[1] - f[3];  // row ey = 0
    const V s1 = f[5] + f[6], d1 = f[5] - f[6];  // row ey = +1
    const V s2 = f[8] + f[7], d2 = f[8] - f[7];  // row ey = -1
    const V B0 = f[2] + s1, C0 = f[4] + s2;
    s.yy = B0 + C0;
    s.rho = f[0] + s0 + s.yy;
    s.jx = d0 + d1 + d2;
    s.jy = B0 - C0;
    s.xx = s0 + s1 + s2;
    s.xy = d1 - d2;
}

// The D2Q9 collision with omega_6 .. omega_8 = 1 (see k_d2q9.cu collide_w1).
template <bool XO>
FX_HD void fx_collide9(const FxSums9<i64> &s, const FxForce (&F)[2], const FxRates &w, i64 (&f)[9], int &bad)
{
    const i64 hx = s.jx + F[0].h1, hy = XO ? s.jy : s.jy + F[1].h1;
    const i64 rho = s.rho + s.rho;
    const i64 j[2] = {hx + hx, hy + hy};
    const double ri = fx_reciprocal(rho, bad);
    const i64 ux = fx_ratio(j[0], rho, ri, bad), uy = fx_ratio(j[1], rho, ri, bad), uhx = ux >> 1, uhy = uy >> 1;
    const i64 cxx = s.xx + s.xx - fx_mul(j[0], ux), cyy = s.yy + s.yy - fx_mul(j[1], uy);
    const i64 cxy = s.xy + s.xy - fx_mul(j[0], uy);
    // (T + omega_3 (2 rho / 3 - T)) / 4, (1 - omega_4) D / 4, (1 - omega_5) c_xy / 4
    const i64 r6 = fx_mul(rho, kFx6);
    i64 Tq = r6;
    if (w.c != 0) Tq += fx_mul(4 * r6 - (cxx + cyy), w.c);
    const i64 Dq = fx_mul(cxx - cyy, w.a);
    i64 m20 = Tq + Dq, m02 = Tq - Dq, m11 = fx_mul(cxy, w.b);
    i64 m22 = fx_mul(rho, kFx36), m21, m12;
    // back-shift along x, then along y (halved moments)
    fx_shift_first(hx, m20, ux);
    fx_shift_k1(m11, m21, ux);
    fx_shift_k02(m02, m12, m22, ux, uhx);
    fx_shift_first(hy, m02, uy);
    fx_shift(hx, m11, m12, uy, uhy);
    fx_shift(m20, m21, m22, uy, uhy);
    // post-collision force: m_10 gains F_post / 2, m_12 (F_pre + F_post) / 3 (halved: / 12)
    i64 m10 = s.jx + F[0].h2, m01 = hy;
    m12 += fx_mul(F[0].h2, kFx3);
    if (!XO) {
        m01 = s.jy + F[1].h2;
        m21 += fx_mul(F[1].h2, kFx3);
    }
    i64 a0 = rho, b0 = m01, c0 = m02, a1 = m10, b1 = m11, c1 = m12, a2 = m20, b2 = m21, c2 = m22;
    fx_back(a0, b0, c0);  // x-order 0; e_y = -1, 0, +1
    fx_back(a1, b1, c1);
    fx_back(a2, b2, c2);
    fx_back(a0, a1, a2);  // e_y = -1: e_x = -1, 0, +1
    fx_back(b0, b1, b2);
    fx_back(c0, c1, c2);
    f[0] = b1;
    f[1] = b2;
    f[3] = b0;
    f[2] = c1;
    f[5] = c2;
    f[6] = c0;
    f[4] = a1;
    f[8] = a2;
    f[7] = a0;
}

// ---- D2Q5 ---------------------------------------------------------------------
// Step coefficients of a uniform advecting velocity (k_d2q5.cu Coef5) as
// fractions of 2^63: h1 = A1 phi - c1 kx, h2 = A2 phi - c2 ky, h3 = P3 phi + X3
// kx + Y3 ky + S3 (kxx + kyy), h4 = P4 phi + X4 kx + Y4 ky + D4 (kxx - kyy).  ok
// = 0 where that form does not apply: an advecting velocity near 1 and above, or a
// P3 that is not below 1 (both components large, omega_1 and omega_2 near 2).
struct FxCoef5 {
    i64 A1, c1, A2, c2, P3, X3, Y3, S3, P4, X4, Y4, D4;
    int ok;
};
inline FxCoef5 fx_coef5(double c1, double c2, double c3, double c4, double ux, double uy)
{
    FxCoef5 k{};
    // With rates in (0, 2) (c1, c2 < 1, c3, c4 < 1/2) and |u| < 0.9 the others are below
    // 1: X3 = ux (2 c3 - c1), P4 = (c1 - c4) ux^2 - (c2 - c4) uy^2 and so on.  P3 = c3 (2/3
    // - ux^2 - uy^2) + c1 ux^2 + c2 uy^2 goes up to 1.6.
    const double P3 = c3 * (2.0 / 3.0 - ux * ux - uy * uy) + c1 * ux * ux + c2 * uy * uy;
    k.ok = ux > -0.9 && ux < 0.9 && uy > -0.9 && uy < 0.9 && P3 > -0.99 && P3 < 0.99;
    if (!k.ok) return k;
    // products of fractions, in integers: 2^-62 instead of FP64's 2^-53
    auto mul = [](i64 a, i64 b) { return 2 * fx_mul(a, b); };
    const i64 C1 = fx_fraction(c1, 63), C2 = fx_fraction(c2, 63), C3 = fx_fraction(c3, 63), C4 = fx_fraction(c4, 63);
    const i64 X = fx_fraction(ux, 63), Y = fx_fraction(uy, 63), X2 = mul(X, X), Y2 = mul(Y, Y);
    k.A1 = mul(C1, X);
    k.c1 = C1;
    k.A2 = mul(C2, Y);
    k.c2 = C2;
    const i64 q1 = mul(C1, X2), q2 = mul(C2, Y2), r3 = mul(C3, X2) + mul(C3, Y2), r4 = mul(C4, X2) - mul(C4, Y2);
    k.P3 = mul(C3, kFx3) - r3 + q1 + q2;  // c3 (2/3 - ux^2 - uy^2) + c1 ux^2 + c2 uy^2
    k.X3 = 2 * mul(C3, X) - mul(C1, X);
    k.Y3 = 2 * mul(C3, Y) - mul(C2, Y);
    k.S3 = -C3;
    k.P4 = q1 - q2 - r4;
    k.X4 = 2 * mul(C4, X) - mul(C1, X);
    k.Y4 = mul(C2, Y) - 2 * mul(C4, Y);
    k.D4 = -C4;
    return k;
}

constexpr i64 kFx5 = 0x3333333333333333ll;  // 1/5

// The scalar step at a uniform velocity: h = S_pre / 2, t = (S_pre + S_post) / 2
// (what the zeroth moment gains).  The rest population is what the others leave
// of the exact total.
FX_HD void fx_collide5(i64 (&g)[5], i64 h, i64 t, const FxCoef5 &c)
{
    const i64 kx = g[1] - g[3], ky = g[2] - g[4], sx = g[1] + g[3], sy = g[2] + g[4];
    const i64 phi0 = g[0] + (sx + sy), phi = phi0 + h;
    const i64 p2 = phi + phi, x2 = kx + kx, y2 = ky + ky, s2 = 2 * (sx + sy), d2 = 2 * (sx - sy);
    const i64 h1 = fx_mul(p2, c.A1) - fx_mul(x2, c.c1), h2 = fx_mul(p2, c.A2) - fx_mul(y2, c.c2);
    const i64 h3 = fx_mul(t, kFx5) + fx_mul(p2, c.P3) + fx_mul(x2, c.X3) + fx_mul(y2, c.Y3) + fx_mul(s2, c.S3);
    const i64 h4 = fx_mul(p2, c.P4) + fx_mul(x2, c.X4) + fx_mul(y2, c.Y4) + fx_mul(d2, c.D4);
    const i64 e1 = h3 + h4, e2 = h3 - h4;
    g[1] += e1 + h1;
    g[2] += e2 + h2;
    g[3] += e1 - h1;
    g[4] += e2 - h2;
    g[0] = phi0 + t - ((g[1] + g[2]) + (g[3] + g[4]));
}

// ---- D3Q15 --------------------------------------------------------------------
// Axis pairs and the corner sign transform of a node's populations (k_d3q15.cu).
template <class V>
struct FxSums15 {
    V rho, jx, jy, jz, xx, yy, zz, xy, xz, yz;
};
template <class V>
FX_HD void fx_sums15(const V (&f)[15], FxSums15<V> &s)
{
    const V A1 = f[7] + f[8], B1 = f[7] - f[8];      // y+, z+
    const V A2 = f[9] + f[10], B2 = f[9] - f[10];    // y-, z+
    const V A3 = f[11] + f[12], B3 = f[11] - f[12];  // y+, z-
    const V A4 = f[13] + f[14], B4 = f[13] - f[14];  // y-, z-
    const V P1 = A1 + A2, Q1 = A1 - A2, P2 = A3 + A4, Q2 = A3 - A4;
    const V R1 = B1 + B2, T1 = B1 - B2, R2 = B3 + B4, T2 = B3 - B4;
    const V S = P1 + P2, axs = f[1] + f[2], ays = f[3] + f[4], azs = f[5] + f[6];
    s.xx = axs + S;
    s.yy = ays + S;
    s.zz = azs + S;
    s.rho = f[0] + axs + ays + s.zz;
    s.jx = f[1] - f[2] + (R1 + R2);
    s.jy = f[3] - f[4] + (Q1 + Q2);
    s.jz = f[5] - f[6] + (P1 - P2);
    s.xy = T1 + T2;
    s.xz = R1 - R2;
    s.yz = Q1 - Q2;
}

// The D3Q15 collision with omega_10 .. omega_14 = 1 (w.a, w.b as on D3Q27): the
// relaxed second-order central moments, third-order ones 0 and the fourth-order
// one kappa_xx kappa_yy / rho give the raw moments of the fifteen monomials,
//   m_xyy = ux m_yy + 2 uy k_xy, m_xxy = uy m_xx + 2 ux k_xy, m_xxz = uz m_xx + 2 ux k_xz,
//   m_xyz = ux m_yz + uy k_xz + uz k_xy, m_xxyy = k_xxyy + ux m_xyy + uy (uy k_xx + 2 ux k_xy),
// and those the populations: the corners by the sign transform (/ 8), the axis
// pairs from what the corners leave of the second and first moments, the rest
// population from what all of them leave of rho, so that mass and momentum are
// carried exactly.  f: populations on the grid k + 1.
template <bool XO>
FX_HD void fx_collide15(const FxSums15<i64> &s, const FxForce (&F)[3], const FxRates &w, i64 (&f)[15], int &bad)
{
    const i64 hx = s.jx + F[0].h1, hy = XO ? s.jy : s.jy + F[1].h1, hz = XO ? s.jz : s.jz + F[2].h1;
    const i64 rho = s.rho + s.rho;
    const i64 j[3] = {hx + hx, hy + hy, hz + hz};
    const double ri = fx_reciprocal(rho, bad);
    const i64 ux = fx_ratio(j[0], rho, ri, bad), uy = fx_ratio(j[1], rho, ri, bad), uz = fx_ratio(j[2], rho, ri, bad);
    const i64 pxx = fx_mul(j[0], ux), pyy = fx_mul(j[1], uy), pzz = fx_mul(j[2], uz);
    const i64 pxy = fx_mul(j[0], uy), pxz = fx_mul(j[0], uz), pyz = fx_mul(j[1], uz);
    const i64 cxx = s.xx + s.xx - pxx, cyy = s.yy + s.yy - pyy, czz = s.zz + s.zz - pzz;
    i64 Ts = rho;
    if (w.b != 0) {
        const i64 d = fx_mul(rho - (cxx + cyy + czz), w.b);
        Ts += d + d;
    }
    // relaxed central moments: trace Ts, deviatoric and off-diagonal parts by 1 - omega
    const i64 D1 = 2 * fx_mul(cxx - cyy, w.a), D2 = 2 * fx_mul(cxx - czz, w.a);
    const i64 kxx = fx_mul(Ts + D1 + D2, kFx3), kyy = kxx - D1, kzz = kxx - D2;
    const i64 kxy = 2 * fx_mul(s.xy + s.xy - pxy, w.a), kxz = 2 * fx_mul(s.xz + s.xz - pxz, w.a);
    const i64 kyz = 2 * fx_mul(s.yz + s.yz - pyz, w.a);
    // kappa_xx / rho as a fraction of 2^64 (below 1/2: the trace is about rho)
    const i64 V = fx_ratio(kxx, rho, ri, bad);
    const i64 mxx = kxx + pxx, myy = kyy + pyy, mzz = kzz + pzz;
    const i64 mxy = kxy + pxy, mxz = kxz + pxz, myz = kyz + pyz;
    i64 mxyy = fx_mul(myy, ux) + 2 * fx_mul(kxy, uy);
    const i64 xk = 2 * fx_mul(kxy, ux);
    i64 mxxy = fx_mul(mxx, uy) + xk;
    i64 mxxz = fx_mul(mxx, uz) + 2 * fx_mul(kxz, ux);
    const i64 mxyz = fx_mul(myz, ux) + fx_mul(kxz, uy) + fx_mul(kxy, uz);
    const i64 mxxyy = fx_mul(kyy, V) + fx_mul(mxyy, ux) + fx_mul(fx_mul(kxx, uy) + xk, uy);
    // force: the first moments gain (F_pre + F_post) / 2 in all, the cubic ones 2 / 5 (F_pre + F_post)
    const i64 f2x = F[0].h2 + F[0].h2;
    mxyy += f2x - fx_mul(f2x, kFx5);  // 8 / 5 h2
    i64 tx = s.jx + F[0].h2, ty = s.jy, tz = s.jz;         // halves of the new first moments
    if (!XO) {
        const i64 f2y = F[1].h2 + F[1].h2, f2z = F[2].h2 + F[2].h2;
        mxxy += f2y - fx_mul(f2y, kFx5);
        mxxz += f2z - fx_mul(f2z, kFx5);
        ty += F[1].h2;
        tz += F[2].h2;
    }
    // corners: (S + sx Sx + sy Sy + sz Sz + sx sy Sxy + sx sz Sxz + sy sz Syz + sx sy sz Sxyz) / 8
    {
        const i64 U0 = mxxyy + mxxz, Ux = mxyy + mxz, Uy = mxxy + myz, Uxy = mxy + mxyz;  // z = +1
        const i64 V0 = mxxyy - mxxz, Vx = mxyy - mxz, Vy = mxxy - myz, Vxy = mxy - mxyz;  // z = -1
        const i64 a0 = U0 + Uy, ax = Ux + Uxy, b0 = U0 - Uy, bx = Ux - Uxy;
        const i64 c0 = V0 + Vy, cx = Vx + Vxy, d0 = V0 - Vy, dx = Vx - Vxy;
        f[7] = (a0 + ax) >> 3;
        f[8] = (a0 - ax) >> 3;
        f[9] = (b0 + bx) >> 3;
        f[10] = (b0 - bx) >> 3;
        f[11] = (c0 + cx) >> 3;
        f[12] = (c0 - cx) >> 3;
        f[13] = (d0 + dx) >> 3;
        f[14] = (d0 - dx) >> 3;
    }
    // what the corners hold of the zeroth and first moments
    const i64 A1 = f[7] + f[8], A2 = f[9] + f[10], A3 = f[11] + f[12], A4 = f[13] + f[14];
    const i64 S = (A1 + A2) + (A3 + A4);
    const i64 Cx = (f[7] - f[8]) + (f[9] - f[10]) + (f[11] - f[12]) + (f[13] - f[14]);
    const i64 Cy = (A1 - A2) + (A3 - A4), Cz = (A1 + A2) - (A3 + A4);
    const i64 ex = mxx - S, ey = myy - S, ez = mzz - S;
    const i64 ox = tx + tx - Cx, oy = ty + ty - Cy, oz = tz + tz - Cz;
    f[1] = (ex + ox) >> 1;
    f[2] = f[1] - ox;
    f[3] = (ey + oy) >> 1;
    f[4] = f[3] - oy;
    f[5] = (ez + oz) >> 1;
    f[6] = f[5] - oz;
    f[0] = rho - S - (f[1] + f[2]) - (f[3] + f[4]) - (f[5] + f[6]);
}

}  // namespace lbmk
