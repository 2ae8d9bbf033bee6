// Velocity sets as compile-time traits, and the per-node helpers that every
// kernel of a lattice shares: pulling the streamed populations of a node and
// the zeroth/first moments.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lbm_device.cuh"
#include "lbm_fixed.cuh"

namespace lbmk {

// D2Q9, Sec. 4 Eq. 15: 0 rest, 1 +x, 2 +y, 3 -x, 4 -y, 5 (+,+), 6 (-,+), 7 (-,-), 8 (+,-).
struct LD2Q9 {
    static constexpr int Q = 9, DIM = 2, ID = 1;
    __host__ __device__ static constexpr int ex(int a) { return (a == 1 || a == 5 || a == 8) ? 1 : ((a == 3 || a == 6 || a == 7) ? -1 : 0); }
    __host__ __device__ static constexpr int ey(int a) { return (a == 2 || a == 5 || a == 6) ? 1 : ((a == 4 || a == 7 || a == 8) ? -1 : 0); }
    __host__ __device__ static constexpr int ez(int) { return 0; }
    __host__ __device__ static constexpr int opp(int a) { return a == 0 ? 0 : (a <= 4 ? ((a + 1) % 4) + 1 : ((a - 3) % 4) + 5); }
    // rest-state populations per unit density (4/9, 1/9, 1/36)
    __host__ __device__ static constexpr double w(int a) { return a == 0 ? 4.0 / 9.0 : (a <= 4 ? 1.0 / 9.0 : 1.0 / 36.0); }
};

// D2Q5, Sec. 5 Eq. 34: 0 rest, 1 +x, 2 +y, 3 -x, 4 -y.
struct LD2Q5 {
    static constexpr int Q = 5, DIM = 2, ID = 3;
    __host__ __device__ static constexpr int ex(int a) { return a == 1 ? 1 : (a == 3 ? -1 : 0); }
    __host__ __device__ static constexpr int ey(int a) { return a == 2 ? 1 : (a == 4 ? -1 : 0); }
    __host__ __device__ static constexpr int ez(int) { return 0; }
    __host__ __device__ static constexpr int opp(int a) { return a == 0 ? 0 : ((a + 1) % 4) + 1; }
    // rest-state populations per unit scalar (1/3, 1/6): moments 1, 0, 1/3
    __host__ __device__ static constexpr double w(int a) { return a == 0 ? 1.0 / 3.0 : 1.0 / 6.0; }
};

// D3Q27 in tensor order: a = (ex+1) + 3 (ey+1) + 9 (ez+1); the opposite of a is 26 - a.
struct LD3Q27 {
    static constexpr int Q = 27, DIM = 3, ID = 2;
    __host__ __device__ static constexpr int ex(int a) { return a % 3 - 1; }
    __host__ __device__ static constexpr int ey(int a) { return (a / 3) % 3 - 1; }
    __host__ __device__ static constexpr int ez(int a) { return a / 9 - 1; }
    __host__ __device__ static constexpr int opp(int a) { return 26 - a; }
    // rest-state populations per unit density: product of (1/6, 2/3, 1/6) per axis
    __host__ __device__ static constexpr double w1(int e) { return e == 0 ? 2.0 / 3.0 : 1.0 / 6.0; }
    __host__ __device__ static constexpr double w(int a) { return w1(ex(a)) * w1(ey(a)) * w1(ez(a)); }
};

// Source offset of the pull f_a(x) = f^p_a(x - e_a) (Eq. 22b / Eq. 40b) with
// periodic wrap, or the node itself with opp = true when x - e_a lies beyond a
// halfway bounce-back wall (the population comes back reversed).
__device__ __forceinline__ int pull_off(const Geom &g, int x, int y, int z, int ex, int ey, int ez,
                                        bool &opp)
{
    int sx = x - ex, sy = y - ey, sz = z - ez;
    opp = false;
    if (ex != 0 && (sx < 0 || sx >= g.nx)) {
        if (g.wall[0]) opp = true;
        else sx = (sx < 0) ? sx + g.nx : sx - g.nx;
    }
    if (ey != 0 && (sy < 0 || sy >= g.ny)) {
        if (g.wall[1]) opp = true;
        else sy = (sy < 0) ? sy + g.ny : sy - g.ny;
    }
    if (ez != 0 && (sz < 0 || sz >= g.nz)) {
        if (g.wall[2]) opp = true;
        else sz = (sz < 0) ? sz + g.nz : sz - g.nz;
    }
    if (opp) return x + g.nx * (y + g.ny * z);
    return sx + g.nx * (sy + g.ny * sz);
}

// Populations are loaded with plain loads, not over the read-only path: a step may
// be launched before the one it follows has ended, and that path is for data that
// nothing writes during a kernel's life.
//
// step_wait: wait until the step before has ended and its results are visible.
// step_next: let the next step's blocks be placed from here on (without it, as
// this step's blocks end).  In a loop of steps each launch but the first asks for
// that overlap (launch_step): its blocks are in place, their code fetched, when the
// step before ends.  Of a launch without the attribute both instructions do
// nothing.  16 steps of a 512 x 256 channel and its fields: FP64 172 -> 131 us, FP32
// 86 -> 65; 256 x 192 FP64 scalar 102 -> 60.
__device__ __forceinline__ void step_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void step_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// First statement of a step kernel that takes both at once.
__device__ __forceinline__ void step_begin()
{
    step_wait();
    step_next();
}

// Pulled populations of node i = (x, y, z): get(p, k) returns the stored
// value of plane p at node k.  A node that has no wall beside it takes every
// population along its wrapped periodic offset (no per-population test, so a
// warp whose nodes straddle a periodic edge does not diverge); a node next to
// a wall tests each population with pull_off.
template <class L, class V, class Get>
__device__ __forceinline__ void pull_node(const Geom &g, int x, int y, int z, int i, V (&f)[L::Q], Get get)
{
    const bool wall_x = g.wall[0] && (x == 0 || x == g.nx - 1);
    const bool wall_y = g.wall[1] && (y == 0 || y == g.ny - 1);
    const bool wall_z = L::DIM == 3 && g.wall[2] && (z == 0 || z == g.nz - 1);
    if (!(wall_x || wall_y || wall_z)) {
        // offset of the source node for e = +1 (coordinate - 1) and e = -1
        // (coordinate + 1) along each axis, wrapped
        const int sy = g.nx;
        const int xm = x == 0 ? g.nx - 1 : -1, xp = x == g.nx - 1 ? 1 - g.nx : 1;
        const int ym = y == 0 ? (g.ny - 1) * sy : -sy, yp = y == g.ny - 1 ? (1 - g.ny) * sy : sy;
        int zm = 0, zp = 0;
        if (L::DIM == 3) {
            const int sz = g.nx * g.ny;
            zm = z == 0 ? (g.nz - 1) * sz : -sz;
            zp = z == g.nz - 1 ? (1 - g.nz) * sz : sz;
        }
#pragma unroll
        for (int a = 0; a < L::Q; a++) {
            const int ex = L::ex(a), ey = L::ey(a), ez = L::ez(a);
            const int row = i + (ey == 1 ? ym : (ey == -1 ? yp : 0)) + (ez == 1 ? zm : (ez == -1 ? zp : 0));
            f[a] = get(a, row + (ex == 1 ? xm : (ex == -1 ? xp : 0)));
        }
        return;
    }
#pragma unroll
    for (int a = 0; a < L::Q; a++) {
        const int ex = L::ex(a), ey = L::ey(a), ez = L::ez(a);
        if (ex == 0 && ey == 0 && ez == 0) {
            f[a] = get(a, i);
        } else {
            bool opp;
            const int off = pull_off(g, x, y, z, ex, ey, ez, opp);
            f[a] = get(opp ? L::opp(a) : a, off);
        }
    }
}

template <class L>
__device__ __forceinline__ void load_pulled(const double *__restrict__ fin, const Geom &g, int x, int y,
                                            int z, int i, double (&f)[L::Q])
{
    pull_node<L>(g, x, y, z, i, f, [&](int p, int k) { return fin[p * g.Np + k]; });
}

// Base pointers of the Q population planes of a step's source and
// destination buffers, passed in the launch arguments: a kernel then
// addresses plane a of node k with one multiply-add on a parameter instead of
// forming the 64-bit product a * Np per access.
template <class T, int Q>
struct Planes {
    const T *in[Q];
    T *out[Q];
};

template <class T, int Q>
inline Planes<T, Q> make_planes(const void *fin, void *fout, long long Np)
{
    Planes<T, Q> P;
    for (int a = 0; a < Q; a++) {
        P.in[a] = static_cast<const T *>(fin) + a * Np;
        P.out[a] = static_cast<T *>(fout) + a * Np;
    }
    return P;
}

// Reduced-precision storage: conversions of a stored deviation to/from float.
template <class T> struct Dev;
template <> struct Dev<float> {
    __device__ static float get(const float *p) { return *p; }
    __device__ static float to_store(float v) { return v; }
};
// 16-bit values are loaded as plain unsigned shorts (a native load the compiler
// can schedule freely) and reinterpreted.
template <> struct Dev<__half> {
    __device__ static float get(const __half *p)
    {
        return __half2float(__ushort_as_half(*reinterpret_cast<const unsigned short *>(p)));
    }
    __device__ static __half to_store(float v) { return __float2half_rn(v); }
};
template <> struct Dev<__nv_bfloat16> {
    __device__ static float get(const __nv_bfloat16 *p)
    {
        return __bfloat162float(__ushort_as_bfloat16(*reinterpret_cast<const unsigned short *>(p)));
    }
    __device__ static __nv_bfloat16 to_store(float v) { return __float2bfloat16_rn(v); }
};

// Pulled deviations of a node (as float) from stored planes of type T.
template <class L, class T>
__device__ __forceinline__ void load_pulled_dev(const T *__restrict__ fin, const Geom &g, int x, int y, int z,
                                                int i, float (&d)[L::Q])
{
    pull_node<L>(g, x, y, z, i, d, [&](int p, int k) { return Dev<T>::get(fin + p * g.Np + k); });
}

// The same pulls through a plane table in the launch arguments.  RO: over the
// read-only path (a kernel that nothing overlaps).
template <class L, bool RO = false>
__device__ __forceinline__ void load_pulled(const Planes<double, L::Q> &P, const Geom &g, int x, int y, int z,
                                            int i, double (&f)[L::Q])
{
    pull_node<L>(g, x, y, z, i, f, [&](int p, int k) { return RO ? __ldg(P.in[p] + k) : P.in[p][k]; });
}
template <class L, class T>
__device__ __forceinline__ void load_pulled_dev(const Planes<T, L::Q> &P, const Geom &g, int x, int y, int z,
                                                int i, float (&d)[L::Q])
{
    pull_node<L>(g, x, y, z, i, d, [&](int p, int k) { return Dev<T>::get(P.in[p] + k); });
}

// Zeroth and first moments of a node's populations in any arithmetic.
template <class L, class V>
__device__ __forceinline__ void sum_moments(const V (&f)[L::Q], V &m0, V (&j)[3])
{
    if constexpr (L::Q == 27) {
        FxSums27<V> s;
        fx_sums27(f, s);
        m0 = s.rho;
        j[0] = s.jx;
        j[1] = s.jy;
        j[2] = s.jz;
    } else if constexpr (L::Q == 9) {
        FxSums9<V> s;
        fx_sums9(f, s);
        m0 = s.rho;
        j[0] = s.jx;
        j[1] = s.jy;
        j[2] = V(0);
    } else {
        m0 = f[0];
        j[0] = j[1] = j[2] = V(0);
#pragma unroll
        for (int a = 1; a < L::Q; a++) {
            m0 += f[a];
            if (L::ex(a) == 1) j[0] += f[a];
            if (L::ex(a) == -1) j[0] -= f[a];
            if (L::ey(a) == 1) j[1] += f[a];
            if (L::ey(a) == -1) j[1] -= f[a];
            if (L::ez(a) == 1) j[2] += f[a];
            if (L::ez(a) == -1) j[2] -= f[a];
        }
    }
}

// Zeroth and first moments of a node as every FP64 readback and reduction
// forms them: summed in fixed point (lbm_fixed.cuh), where the sums are exact,
// and rounded once; a node outside the fixed-point range is summed in FP64.  The
// FP64 sums of D3Q27 took 40 clocks of an SM's FP64 unit per node, the four
// conversions back take 2 (INT: none, for a readback inside a step, which the FP64 unit
// bounds more tightly).  D2Q5's four FP64 adds stay.
template <class L, bool INT = false>
__device__ __forceinline__ void zeroth_first(const double (&f)[L::Q], double &m0, double (&j)[3])
{
    const int em = fx_emax(f);
    if (L::Q != 5 && fx_in_range(em)) {
        const int k = FxGrid<L::Q>::S + 1023 - em;
        i64 X[L::Q], M, J[3];
        fx_load_int<L::Q, true>(f, em, X);
        sum_moments<L>(X, M, J);
        m0 = INT ? fx_value_int(M, k) : fx_value(M, k);
#pragma unroll
        for (int d = 0; d < 3; d++) j[d] = d < L::DIM ? (INT ? fx_value_int(J[d], k) : fx_value(J[d], k)) : 0.0;
        return;
    }
    sum_moments<L>(f, m0, j);
}

// The same sums of FP32 deviations: every value becomes a 24-bit integer
// shifted to the node's scale (32 bits below the largest deviation's last),
// without an FP64 conversion per value: converting to FP64 and adding there
// took 53 clocks of the FP64 unit per D3Q27 node, this takes about 8 of the
// integer units (moments of a 384^3 FP32 lattice: 9.5 -> 2.0 ms, the memory's
// time 1.2).
template <class L>
__device__ __forceinline__ void zeroth_first(const float (&d)[L::Q], double &m0, double (&j)[3])
{
    int em;
    i64 X[L::Q];
    const FxDev r = fx_load_dev(d, em, X);
    if (r == FXD_ZERO) {  // a node at the reference state
        m0 = j[0] = j[1] = j[2] = 0.0;
        return;
    }
    if (r == FXD_TAKEN) {
        i64 M, J[3];
        sum_moments<L>(X, M, J);
        const int k = 23 + 32 + 127 - em;  // X = d 2^k
        m0 = fx_value(M, k);
#pragma unroll
        for (int q = 0; q < 3; q++) j[q] = q < L::DIM ? fx_value(J[q], k) : 0.0;
        return;
    }
    double dd[L::Q];
#pragma unroll
    for (int a = 0; a < L::Q; a++) dd[a] = (double)d[a];
    sum_moments<L>(dd, m0, j);
}

// Whether fx_recip takes a density (a negative one's exponent is above 2047).
__device__ __forceinline__ bool recip_takes(double rho)
{
    const unsigned e = fx_hi(fx_bits(rho)) >> 20;
    return e > 2u && e < 2044u;
}
// The correctly rounded 1/rho of the readbacks.
__device__ __forceinline__ double recip_density(double rho) { return recip_takes(rho) ? fx_recip(rho) : __drcp_rn(rho); }
// j / rho of the reductions is over_density(j, sh) * density_recip(rho, sh): where rho lies
// near an end of the FP64 range (its reciprocal need not be an FP64 number) both are
// scaled by 2^700 or 2^-700 first (sh > 0, < 0).  NaN for a density that is not positive and finite.
__device__ __forceinline__ double over_density(double j, int sh)
{
    return sh == 0 ? j : j * (sh > 0 ? 0x1p700 : 0x1p-700);
}
__device__ __forceinline__ double density_recip(double rho, int &sh)
{
    sh = 0;
    if (!recip_takes(rho)) {
        const u64 b = fx_bits(rho);
        if (b - 1u >= 0x7fefffffffffffffull) return fx_double(0x7ff8000000000000ull);
        sh = b >> 52 < 3u ? 1 : -1;
        rho = over_density(rho, sh);
    }
    return fx_recip(rho);
}

// Whether component c of a shape is known to vanish everywhere.
__device__ __forceinline__ bool field_zero(const FieldDev &F, int kind, int c)
{
    return kind == FK_NONE || (kind == FK_CONST ? F.cval[c] == 0.0 : ((F.zmask >> c) & 1) != 0);
}

// The packed fields of a node from its zeroth and first moments, as every
// readback writes them: rho (phi for the scalar lattice) at rho[off + i],
// velocity component d at u[dim * off + d * N + i] = j_d (1/rho); with `forced`
// the pre-collision half force / source (a_pre / 2) P is included (Eq. 25 / 43;
// ahalf = a_pre / 2, components that vanish everywhere are left out), in
// one fused multiply-add: every rounding is spelt out, so that every kernel that
// forms the fields gives the same bits.
template <class L>
__device__ __forceinline__ void store_fields(double m0, const double (&j)[3], bool forced, double ahalf, const FieldDev &F,
                                             int fkind, int x, int y, int z, int i, int N, long long off, double *rho,
                                             double *u)
{
    if (L::Q == 5) {
        rho[off + i] = forced ? __fma_rn(ahalf, field_value(F, fkind, 0, x, y, z, i), m0) : m0;
        return;
    }
    rho[off + i] = m0;
    const double rinv = recip_density(m0);
#pragma unroll
    for (int d = 0; d < L::DIM; d++) {
        double jd = j[d];
        if (forced && !field_zero(F, fkind, d)) jd = __fma_rn(ahalf, field_value(F, fkind, d, x, y, z, i), jd);
        u[L::DIM * off + (long long)d * N + i] = __dmul_rn(jd, rinv);
    }
}

// Copy an object into shared memory cooperatively (word by word); the caller
// synchronises.  Used to give every thread of a block one copy of its batch
// descriptor without repeated global loads.
template <class Obj>
__device__ __forceinline__ void stage_to_shared(Obj &dst, const Obj &src)
{
    static_assert(sizeof(Obj) % 4 == 0, "word copy");
    const unsigned *s = reinterpret_cast<const unsigned *>(&src);
    unsigned *d = reinterpret_cast<unsigned *>(&dst);
    for (int k = threadIdx.x; k < (int)(sizeof(Obj) / 4); k += blockDim.x) d[k] = __ldg(s + k);
}

// Coordinates of node i = x + nx (y + ny z).
__device__ __forceinline__ void node_xyz(const Geom &g, int i, int &x, int &y, int &z)
{
    const int r = div_invariant(i, g.mx, g.lx);
    x = i - r * g.nx;
    z = div_invariant(r, g.my, g.ly);
    y = r - z * g.ny;
}

// Coordinates of node i = x + nx y of a 2D lattice.
__device__ __forceinline__ void node_xy(const Geom &g, int i, int &x, int &y)
{
    y = div_invariant(i, g.mx, g.lx);
    x = i - y * g.nx;
}

}  // namespace lbmk
