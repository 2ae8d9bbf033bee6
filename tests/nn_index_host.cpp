// The index arithmetic of csrc/k_nn_index.cuh on the host, for tests/test_nn_index_cpu.py.
#include "k_nn_index.cuh"

using namespace nnix;

static Shape shape_of(const int *v)
{
    return Shape{v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], v[9], v[10], v[11]};
}

// Offsets, inside a sample, of channel c[i]'s source of tap[i] (a, f, e) of pixel q[i];
// -1 outside.  n: the pixels' samples.
template <class I>
static void gather(const Shape &s, long count, const long long *q, const int *c, const int *tap, int sgn, long long *n,
                   long long *off)
{
    const I sp = (I)s.d * s.h * s.w;
    for (long i = 0; i < count; i++) {
        const Pixel<I> x = pixel_at<I>(s, (I)q[i]);
        const I at = tap_source(s, x, tap[3 * i], tap[3 * i + 1], tap[3 * i + 2], sgn);
        n[i] = x.n;
        off[i] = at >= 0 ? plane_offset(c[i], sp, at) : -1;
    }
}
extern "C" void gather_offsets(const int *v, long count, const long long *q, const int *c, const int *tap, int sgn,
                               long long *n, long long *off)
{
    const Shape s = shape_of(v);
    if (narrow(s)) gather<int>(s, count, q, c, tap, sgn, n, off);
    else gather<long long>(s, count, q, c, tap, sgn, n, off);
}

// The line of positions: total[0], reach[0]; of positions q[i]: sample n, plane d, row h, column w.
template <class I>
static void line(const Shape &s, long count, const long long *q, int *pos, long long *total, long long *reach)
{
    const Line<I> l = line_of<I>(s);
    *total = l.total;
    *reach = l.hw;
    for (long i = 0; i < count; i++) {
        const Pixel<I> x = position_at<I>(s, l, (I)q[i]);
        const int at[4] = {x.n, x.d, x.h, x.w};
        for (int k = 0; k < 4; k++) pos[4 * i + k] = at[k];
    }
}
extern "C" int positions(const int *v, long count, const long long *q, int *pos, long long *total, long long *reach)
{
    const Shape s = shape_of(v);
    if (narrow(s)) line<int>(s, count, q, pos, total, reach);
    else line<long long>(s, count, q, pos, total, reach);
    return narrow(s);
}
