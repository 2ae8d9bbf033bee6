// Where the warm-start network's kernels find their values: pixels of a batch, the
// sources of taps, positions on a line.  Included by k_nn.cu; compiles for the host too
// (tests run it on the CPU).
#pragma once

#ifdef __CUDACC__
#define NN_HD __host__ __device__ __forceinline__
#else
#define NN_HD inline
#endif

namespace nnix {

struct Shape {
    int n, ci, co, d, h, w;  // batch, channels in/out, spatial extents
    int kd, kh, kw;          // kernel extents (odd)
    int dd, dh, dw;          // dilations
    NN_HD long long in_count() const { return (long long)n * ci * d * h * w; }
    NN_HD long long out_count() const { return (long long)n * co * d * h * w; }
};

// The kernels' index type I: int, or long long for batches of 2^31 positions and more
// (narrow() decides), whose divisions take several times as long.
template <class I>
struct Index;
template <>
struct Index<int> {
    typedef unsigned U;
};
template <>
struct Index<long long> {
    typedef unsigned long long U;
};

// Offset of value `at` of channel c inside a sample, sp values a channel.
template <class I>
NN_HD long long plane_offset(int c, I sp, I at)
{
    return (long long)c * sp + at;
}

// Pixel coordinates of pixel q of a batch.
template <class I>
struct Pixel {
    int n, d, h, w;  // sample, place inside it
    I p;             // position inside it
};
template <class I>
NN_HD Pixel<I> pixel_at(const Shape &s, I q)
{
    typedef typename Index<I>::U U;
    const U sp = (U)((I)s.d * s.h * s.w);
    Pixel<I> x;
    x.n = (int)((U)q / sp);
    x.p = (I)((U)q - (U)x.n * sp);
    const U r = (U)x.p / (U)s.w;
    x.w = (int)((U)x.p - r * (U)s.w);
    x.d = (int)(r / (U)s.h);
    x.h = (int)(r - (U)x.d * (U)s.h);
    return x;
}
// Position of the source pixel of tap (a, f, e), shifted by sgn * dilation; -1 outside.
template <class I>
NN_HD I tap_source(const Shape &s, const Pixel<I> &x, int a, int f, int e, int sgn)
{
    const int zd = x.d + sgn * s.dd * (a - (s.kd - 1) / 2);
    const int zh = x.h + sgn * s.dh * (f - (s.kh - 1) / 2);
    const int zw = x.w + sgn * s.dw * (e - (s.kw - 1) / 2);
    const bool in = (unsigned)zd < (unsigned)s.d && (unsigned)zh < (unsigned)s.h && (unsigned)zw < (unsigned)s.w;
    return in ? ((I)zd * s.h + zh) * s.w + zw : (I)-1;
}
// The images as one line of positions: every row of w pixels is followed by hw
// empty ones, hw the largest shift along w of a tap that can meet a pixel at all (one below
// w), so that position + shift is the shifted pixel of the same row, or an empty one, for
// every |shift| <= hw.  Taps further out have no source anywhere.
template <class I>
struct Line {
    I hw, wp;       // reach, positions per row
    I total;        // positions of the batch
    I sp;
};
// Taps on either side of the middle one that can meet a pixel along w.
NN_HD int taps_in_reach(const Shape &s)
{
    const int all = (s.kw - 1) / 2, some = (s.w - 1) / s.dw;
    return all < some ? all : some;
}
template <class I>
NN_HD Line<I> line_of(const Shape &s)
{
    Line<I> l;
    l.hw = s.dw * taps_in_reach(s);
    l.wp = s.w + l.hw;
    l.sp = (I)s.d * s.h * s.w;
    l.total = (I)s.n * s.d * s.h * l.wp;
    return l;
}
// Sample, plane, row and column of a position; w < 0 outside the batch and on empty positions.
template <class I>
NN_HD Pixel<I> position_at(const Shape &s, const Line<I> &l, I q)
{
    typedef typename Index<I>::U U;
    Pixel<I> x;
    x.n = x.d = x.h = 0;
    x.p = 0;
    x.w = -1;
    if (q < 0 || q >= l.total) return x;
    const U r = (U)q / (U)l.wp;
    const I w = q - (I)(r * (U)l.wp);
    const U z = r / (U)s.h;
    x.h = (int)(r - z * (U)s.h);
    x.n = (int)(z / (U)s.d);
    x.d = (int)(z - (U)x.n * (U)s.d);
    x.w = w < s.w ? (int)w : -1;
    return x;
}
// Whether positions, a tile and its taps past the last one among them, and offsets
// inside a channel are 32-bit numbers.
inline bool narrow(const Shape &s)
{
    const Line<long long> l = line_of<long long>(s);
    return l.sp < (1LL << 30) && l.total + l.hw < (1LL << 31) - (1LL << 21);
}

}  // namespace nnix
