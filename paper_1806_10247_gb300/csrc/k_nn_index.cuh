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

// Offset of value `at` of channel c inside a sample, sp values a channel.
NN_HD long long plane_offset(int c, int sp, int at) { return (long long)c * sp + at; }

// Pixel coordinates of pixel q of a batch (32-bit: the launchers check the sizes).
struct Pixel {
    int n, p;        // sample, position inside it
    int d, h, w;
};
NN_HD Pixel pixel_at(const Shape &s, unsigned q)
{
    const unsigned sp = (unsigned)(s.d * s.h * s.w);
    Pixel x;
    x.n = (int)(q / sp);
    x.p = (int)(q - (unsigned)x.n * sp);
    const unsigned r = (unsigned)x.p / (unsigned)s.w;
    x.w = x.p - (int)(r * (unsigned)s.w);
    x.d = (int)(r / (unsigned)s.h);
    x.h = (int)(r - (unsigned)x.d * (unsigned)s.h);
    return x;
}
// Position of the source pixel of tap (a, f, e), shifted by sgn * dilation; -1 outside.
NN_HD int tap_source(const Shape &s, const Pixel &x, int a, int f, int e, int sgn)
{
    const int zd = x.d + sgn * s.dd * (a - (s.kd - 1) / 2);
    const int zh = x.h + sgn * s.dh * (f - (s.kh - 1) / 2);
    const int zw = x.w + sgn * s.dw * (e - (s.kw - 1) / 2);
    const bool in = (unsigned)zd < (unsigned)s.d && (unsigned)zh < (unsigned)s.h && (unsigned)zw < (unsigned)s.w;
    return in ? (zd * s.h + zh) * s.w + zw : -1;
}
// The images as one line of positions: every row of w pixels is followed by hw
// empty ones, hw the largest shift along w of a tap that can meet a pixel at all (one below
// w), so that position + shift is the shifted pixel of the same row, or an empty one, for
// every |shift| <= hw.  Taps further out have no source anywhere.
struct Line {
    int hw, wp;       // reach, positions per row
    unsigned total;   // positions of the batch
    int sp;
};
// Taps on either side of the middle one that can meet a pixel along w.
NN_HD int taps_in_reach(const Shape &s)
{
    const int all = (s.kw - 1) / 2, some = (s.w - 1) / s.dw;
    return all < some ? all : some;
}
NN_HD Line line_of(const Shape &s)
{
    Line l;
    l.hw = s.dw * taps_in_reach(s);
    l.wp = s.w + l.hw;
    l.sp = s.d * s.h * s.w;
    l.total = (unsigned)s.n * (unsigned)(s.d * s.h) * (unsigned)l.wp;
    return l;
}
// Sample, plane, row and column of a position; w < 0 outside the batch and on empty positions.
NN_HD Pixel position_at(const Shape &s, const Line &l, int q)
{
    Pixel x;
    x.n = x.d = x.h = x.p = 0;
    x.w = -1;
    if (q < 0 || (unsigned)q >= l.total) return x;
    const unsigned r = (unsigned)q / (unsigned)l.wp;
    const int w = q - (int)(r * (unsigned)l.wp);
    const unsigned z = r / (unsigned)s.h;
    x.h = (int)(r - z * (unsigned)s.h);
    x.n = (int)(z / (unsigned)s.d);
    x.d = (int)(z - (unsigned)x.n * (unsigned)s.d);
    x.w = w < s.w ? w : -1;
    return x;
}

}  // namespace nnix
