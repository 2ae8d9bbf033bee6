// The index arithmetic of csrc/k_nn_index.cuh on the host, for tests/test_nn_index_cpu.py.
#include "k_nn_index.cuh"

using namespace nnix;

static Shape shape_of(const int *v)
{
    return Shape{v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], v[9], v[10], v[11]};
}

// Offsets, inside a sample, of channel c[i]'s source of tap[i] (a, f, e) of pixel q[i];
// -1 outside.  n: the pixels' samples.
extern "C" void gather_offsets(const int *v, long count, const long long *q, const int *c, const int *tap, int sgn,
                               long long *n, long long *off)
{
    const Shape s = shape_of(v);
    const int sp = s.d * s.h * s.w;
    for (long i = 0; i < count; i++) {
        const Pixel x = pixel_at(s, (unsigned)q[i]);
        const int at = tap_source(s, x, tap[3 * i], tap[3 * i + 1], tap[3 * i + 2], sgn);
        n[i] = x.n;
        off[i] = at >= 0 ? plane_offset(c[i], sp, at) : -1;
    }
}
