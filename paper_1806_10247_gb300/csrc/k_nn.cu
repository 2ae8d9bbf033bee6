// Kernels of the learned warm start: a small 3D convolutional network trained
// and evaluated on the GPU (forward, backward, loss, Adam).  Activations are
// FP32 in [batch][channel][D][H][W] layout; weights are read either as FP32 or
// as BF16 (the trained network's storage form), always accumulated in FP32.
// The paper has no counterpart: this supports the warm start of the LB
// iteration, which alone decides the converged field.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>

#include "../../include/lbm.h"
#include "k_nn_index.cuh"
#include "k_nn_tc.cuh"

namespace {

using namespace nnix;

constexpr int kT = 256;
thread_local std::string g_nn_error;

int nn_fail(int code, const char *fmt, ...)
{
    char buf[256];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_nn_error = buf;
    return code;
}

__device__ __forceinline__ float wload(const void *w, int bf16, long long i)
{
    if (bf16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(w)[i]);
    return reinterpret_cast<const float *>(w)[i];
}

// y[n,o,p] = b[o] + sum_{i,tap} w[o,i,tap] x[n,i,p + shift(tap)], zero padding.
__global__ void __launch_bounds__(kT)
k_conv_fwd(const float *__restrict__ x, const void *__restrict__ w, int bf16, const float *__restrict__ b,
           float *__restrict__ y, Shape s, int act)
{
    const long long idx = (long long)blockIdx.x * kT + threadIdx.x;
    if (idx >= s.out_count()) return;
    const int v = idx % s.w;
    long long r = idx / s.w;
    const int hh = r % s.h;
    r /= s.h;
    const int dd = r % s.d;
    r /= s.d;
    const int o = r % s.co;
    const int n = (int)(r / s.co);
    float acc = b[o];
    const int taps = s.kd * s.kh * s.kw;
    for (int i = 0; i < s.ci; i++) {
        const float *xi = x + ((long long)n * s.ci + i) * s.d * s.h * s.w;
        const long long wbase = ((long long)o * s.ci + i) * taps;
        for (int a = 0; a < s.kd; a++) {
            const int zd = dd + s.dd * (a - (s.kd - 1) / 2);
            if (zd < 0 || zd >= s.d) continue;
            for (int c = 0; c < s.kh; c++) {
                const int zh = hh + s.dh * (c - (s.kh - 1) / 2);
                if (zh < 0 || zh >= s.h) continue;
                for (int e = 0; e < s.kw; e++) {
                    const int zw = v + s.dw * (e - (s.kw - 1) / 2);
                    if (zw < 0 || zw >= s.w) continue;
                    acc = fmaf(wload(w, bf16, wbase + (a * s.kh + c) * s.kw + e), xi[((long long)zd * s.h + zh) * s.w + zw],
                               acc);
                }
            }
        }
    }
    y[idx] = act == 1 ? tanhf(acc) : acc;
}

// gx[n,i,p] = sum_{o,tap} w[o,i,tap] gy[n,o,p - shift(tap)]  (transposed convolution).
__global__ void __launch_bounds__(kT)
k_conv_bwd_in(const float *__restrict__ gy, const void *__restrict__ w, int bf16, float *__restrict__ gx, Shape s)
{
    const long long idx = (long long)blockIdx.x * kT + threadIdx.x;
    if (idx >= s.in_count()) return;
    const int v = idx % s.w;
    long long r = idx / s.w;
    const int hh = r % s.h;
    r /= s.h;
    const int dd = r % s.d;
    r /= s.d;
    const int i = r % s.ci;
    const int n = (int)(r / s.ci);
    const int taps = s.kd * s.kh * s.kw;
    float acc = 0.0f;
    for (int o = 0; o < s.co; o++) {
        const float *go = gy + ((long long)n * s.co + o) * s.d * s.h * s.w;
        const long long wbase = ((long long)o * s.ci + i) * taps;
        for (int a = 0; a < s.kd; a++) {
            const int zd = dd - s.dd * (a - (s.kd - 1) / 2);
            if (zd < 0 || zd >= s.d) continue;
            for (int c = 0; c < s.kh; c++) {
                const int zh = hh - s.dh * (c - (s.kh - 1) / 2);
                if (zh < 0 || zh >= s.h) continue;
                for (int e = 0; e < s.kw; e++) {
                    const int zw = v - s.dw * (e - (s.kw - 1) / 2);
                    if (zw < 0 || zw >= s.w) continue;
                    acc = fmaf(wload(w, bf16, wbase + (a * s.kh + c) * s.kw + e), go[((long long)zd * s.h + zh) * s.w + zw],
                               acc);
                }
            }
        }
    }
    gx[idx] = acc;
}

__device__ __forceinline__ float block_sum(float v)
{
    __shared__ float sh[kT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    v = threadIdx.x < kT / 32 ? sh[threadIdx.x] : 0.0f;
    if (warp == 0)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;  // valid in thread 0
}

// One block per weight (o, i, tap) and, after those, one per bias o:
// gw = sum_{n,p} gy[n,o,p] x[n,i,p + shift(tap)],  gb = sum_{n,p} gy[n,o,p].
// Fixed summation order: deterministic.
__global__ void __launch_bounds__(kT)
k_conv_bwd_w(const float *__restrict__ x, const float *__restrict__ gy, float *__restrict__ gw, float *__restrict__ gb,
             Shape s)
{
    const int taps = s.kd * s.kh * s.kw;
    const long long nweights = (long long)s.co * s.ci * taps;
    const long long bid = blockIdx.x;
    const long long sp = (long long)s.d * s.h * s.w;
    float acc = 0.0f;
    if (bid < nweights) {
        const int tap = bid % taps;
        const int i = (bid / taps) % s.ci;
        const int o = (int)(bid / ((long long)taps * s.ci));
        const int e = tap % s.kw, c = (tap / s.kw) % s.kh, a = tap / (s.kw * s.kh);
        const int sd = s.dd * (a - (s.kd - 1) / 2), sh = s.dh * (c - (s.kh - 1) / 2), sw = s.dw * (e - (s.kw - 1) / 2);
        for (long long q = threadIdx.x; q < (long long)s.n * sp; q += kT) {
            const int n = (int)(q / sp);
            const long long p = q % sp;
            const int v = p % s.w, hh = (p / s.w) % s.h, dd = (int)(p / ((long long)s.w * s.h));
            const int zd = dd + sd, zh = hh + sh, zw = v + sw;
            if (zd < 0 || zd >= s.d || zh < 0 || zh >= s.h || zw < 0 || zw >= s.w) continue;
            acc = fmaf(gy[((long long)n * s.co + o) * sp + p],
                       x[((long long)n * s.ci + i) * sp + ((long long)zd * s.h + zh) * s.w + zw], acc);
        }
        acc = block_sum(acc);
        if (threadIdx.x == 0) gw[bid] = acc;
    } else {
        const int o = (int)(bid - nweights);
        for (long long q = threadIdx.x; q < (long long)s.n * sp; q += kT) {
            const int n = (int)(q / sp);
            acc += gy[((long long)n * s.co + o) * sp + q % sp];
        }
        acc = block_sum(acc);
        if (threadIdx.x == 0) gb[o] = acc;
    }
}

// g *= 1 - y^2, four values per thread where both arrays are 16-byte aligned.
__global__ void __launch_bounds__(kT)
k_tanh_bwd(float *__restrict__ g, const float *__restrict__ y, long long count, int vec)
{
    const long long i = (long long)blockIdx.x * kT + threadIdx.x;
    if (vec && 4 * i + 4 <= count) {
        float4 a = reinterpret_cast<float4 *>(g)[i];
        const float4 b = __ldg(reinterpret_cast<const float4 *>(y) + i);
        a.x *= 1.0f - b.x * b.x;
        a.y *= 1.0f - b.y * b.y;
        a.z *= 1.0f - b.z * b.z;
        a.w *= 1.0f - b.w * b.w;
        reinterpret_cast<float4 *>(g)[i] = a;
        return;
    }
    for (long long k = 4 * i; k < 4 * i + 4 && k < count; k++) g[k] *= 1.0f - y[k] * y[k];
}

// g = 2 (y - t) / count and the partial sums of (y - t)^2 of kMseBlocks blocks
// at most (one block took 0.3 ms for 524,288 values, the memory's time is 1 us);
// k_mse_final adds them in order: loss = mean((y - t)^2).
constexpr int kMseBlocks = 304;
__device__ __forceinline__ double block_sum_f64(double acc)
{
    __shared__ double sh[kT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    acc = threadIdx.x < kT / 32 ? sh[threadIdx.x] : 0.0;
    if (threadIdx.x < 32)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    return acc;  // valid in thread 0
}
__global__ void __launch_bounds__(kT)
k_mse(const float *__restrict__ y, const float *__restrict__ t, float *__restrict__ g, long long count,
      double *__restrict__ part)
{
    double acc = 0.0;
    const float scale = 2.0f / (float)count;
    for (long long i = (long long)blockIdx.x * kT + threadIdx.x; i < count; i += (long long)gridDim.x * kT) {
        const float d = y[i] - t[i];
        g[i] = scale * d;
        acc += (double)d * (double)d;
    }
    acc = block_sum_f64(acc);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}
__global__ void __launch_bounds__(kT) k_mse_final(const double *__restrict__ part, int n, long long count,
                                                  double *__restrict__ loss)
{
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += kT) acc += part[i];
    acc = block_sum_f64(acc);
    if (threadIdx.x == 0) *loss = acc / (double)count;
}

// Adam (bias-corrected) on FP32 master weights; also refreshes the BF16 copy.
__global__ void __launch_bounds__(kT)
k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
       __nv_bfloat16 *__restrict__ pb, long long count, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const long long i = (long long)blockIdx.x * kT + threadIdx.x;
    if (i >= count) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (pb) pb[i] = __float2bfloat16_rn(pi);
}

__global__ void __launch_bounds__(kT) k_to_bf16(const float *__restrict__ p, __nv_bfloat16 *__restrict__ pb, long long count)
{
    const long long i = (long long)blockIdx.x * kT + threadIdx.x;
    if (i < count) pb[i] = __float2bfloat16_rn(p[i]);
}

int launched(const char *what)
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return nn_fail(LBM_ECUDA, "%s: %s", what, cudaGetErrorString(e));
    return LBM_OK;
}

unsigned grid_of(long long count, int block) { return (unsigned)((count + block - 1) / block); }

// ------------------------------------------------ tensor-core convolutions ---
// With BF16 weights (the trained network's storage form) the convolutions run
// as implicit GEMMs on the tensor cores (tcgen05, BF16 operands, FP32
// accumulation in tensor memory): activations and incoming gradients are
// rounded to BF16 as they are staged, every product is exact and the sums are
// FP32.  Tiles: kM = 128 pixels (or weight rows) by up to kMaxKp padded K
// values and kMaxNp padded output channels; one thread stages one row.

// Bit 0 set when a tensor-core wait ran out (read and cleared by lbm_nn_tc_status).
__device__ int g_tc_status;

int round16(int v) { return (v + 15) / 16 * 16; }

enum TcMode { TC_FWD = 0, TC_BWD_IN = 1 };

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    unsigned u;
    memcpy(&u, &v, sizeof u);
    return u;
}

// Forward pass and input gradient.
// TC_FWD:    y[n,o,p] = act(b[o] + sum_{i,tap} w[o,i,tap] x[n,i,p + shift(tap)])
//            rows: pixels of y; K = (i, tap); N = o.
// TC_BWD_IN: gx[n,i,p] = sum_{o,tap} w[o,i,tap] gy[n,o,p - shift(tap)]
//            rows: pixels of x; K = (o, tap); N = i.
// K runs over the gathered channels, then over the taps: the order of the FP32 sums
// is part of the result, since the next layer rounds it to BF16.  A thread gathers
// its pixel's row of K, eight values to a 16-byte row of a core matrix.  A block
// keeps the weights in shared memory and walks over the 128-pixel tiles blockIdx.x,
// blockIdx.x + gridDim.x, ...  TAPS = 9 (1 x 3 x 3): the nine source positions are
// found once per pixel and (channel, tap) of every value is known at compile time;
// 0: any taps, counted along.  For the shapes that the staged form below does not take.
template <int MODE, int TAPS, class I>
__global__ void __launch_bounds__(nntc::kM, TAPS ? 5 : 1)
k_tc_conv(const float *__restrict__ in, const __nv_bfloat16 *__restrict__ w, const float *__restrict__ b,
          float *__restrict__ out, Shape s, int act, int Kp, int Np)
{
    using namespace nntc;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long mbar;
    __shared__ uint32_t tmem_base;
    unsigned char *As = smem;
    unsigned char *Bs = smem + kM * Kp * 2;
    const int tid = threadIdx.x;
    const int taps = s.kd * s.kh * s.kw;
    const int cin = MODE == TC_FWD ? s.ci : s.co;    // channels of the gathered operand
    const int cout = MODE == TC_FWD ? s.co : s.ci;   // channels of the result
    const int K = cin * taps;
    const int sgn = MODE == TC_FWD ? 1 : -1;
    const I sp = (I)s.d * s.h * s.w;
    const I npix = s.n * sp, ntiles = (npix + kM - 1) / kM;
    const uint32_t ncols = tmem_cols(Np);
    const uint32_t lboA = (kM / 8) * 128, lboB = (uint32_t)(Np / 8) * 128;
    if (tid < 32) tmem_alloc(smem_u32(&tmem_base), ncols);
    if (tid == 0) mbar_init(smem_u32(&mbar));
    for (int idx = tid; idx < Np * (Kp >> 3); idx += kM) {
        const int k8 = idx / Np, r = idx - k8 * Np;  // r: output channel
        __nv_bfloat16 v[8];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const int k = 8 * k8 + j, c = k / taps, tap = k - c * taps;
            v[j] = __float2bfloat16_rn(0.f);
            if (r < cout && k < K)
                v[j] = MODE == TC_FWD ? w[((long long)r * s.ci + c) * taps + tap]
                                      : w[((long long)c * s.ci + r) * taps + tap];
        }
        uint4 u;
        memcpy(&u, v, sizeof u);
        *reinterpret_cast<uint4 *>(Bs + core_off(r, 8 * k8, Np)) = u;
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = tmem_base;
    bool ok = true;
    uint32_t phase = 0;
    for (I tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const I q = tile * kM + tid;
        const bool valid = q < npix;
        const Pixel<I> x = pixel_at<I>(s, valid ? q : 0);
        const float *base = in + (long long)x.n * cin * sp;
        auto put8 = [&](int k8, const float (&v)[8]) {
            *reinterpret_cast<uint4 *>(As + core_off(tid, 8 * k8, kM)) = make_uint4(
                pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
        };
        if constexpr (TAPS == 9) {
            I at[9];
#pragma unroll
            for (int tap = 0; tap < 9; tap++) at[tap] = valid ? tap_source(s, x, 0, tap / 3, tap % 3, sgn) : (I)-1;
            // over every group of the padded K: eight channels' taps are nine groups, and a
            // channel count that is an odd multiple of eight leaves one of zeros beyond them
            for (int k0 = 0; k0 < (Kp >> 3); k0 += 9) {
                const int c0 = 8 * (k0 / 9);
                const float *src = base + (long long)c0 * sp;
#pragma unroll
                for (int g = 0; g < 9; g++) {
                    const int k8 = k0 + g;
                    if (k8 >= (Kp >> 3)) break;
                    float v[8];
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const int c = (8 * g + j) / 9, tap = (8 * g + j) % 9;
                        v[j] = at[tap] >= 0 && c0 + c < cin ? __ldg(src + plane_offset(c, sp, at[tap])) : 0.f;
                    }
                    put8(k8, v);
                }
            }
        } else {
            int c = 0, a = 0, f = 0, e = 0;
            for (int k8 = 0; k8 < (Kp >> 3); k8++) {
                float v[8];
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const I at = valid && c < cin ? tap_source(s, x, a, f, e, sgn) : (I)-1;
                    v[j] = at >= 0 ? __ldg(base + plane_offset(c, sp, at)) : 0.f;
                    if (++e == s.kw) {
                        e = 0;
                        if (++f == s.kh) {
                            f = 0;
                            if (++a == s.kd) {
                                a = 0;
                                c++;
                            }
                        }
                    }
                }
                put8(k8, v);
            }
        }
        fence_smem_to_async();
        fence_before_sync();
        __syncthreads();
        fence_after_sync();
        if (tid == 0) {
            issue_tile(tmem, smem_u32(As), lboA, smem_u32(Bs), lboB, Kp, Np);
            mma_commit(smem_u32(&mbar));
        }
        ok = __syncthreads_and(mbar_wait_bounded(smem_u32(&mbar), phase));
        fence_after_sync();
        phase ^= 1u;
        if (!ok) break;
        for (int c0 = 0; c0 < Np; c0 += 16) {
            float v[16];
            tmem_load16(tmem + ((uint32_t)(32 * (tid >> 5)) << 16) + (uint32_t)c0, v);
            if (valid) {
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const int o = c0 + j;
                    if (o < cout) {
                        float r = v[j];
                        if (MODE == TC_FWD) {
                            r += b[o];
                            if (act == 1) r = tanhf(r);
                        }
                        out[((long long)x.n * cout + o) * sp + x.p] = r;
                    }
                }
            }
        }
        // the next tile's MMAs overwrite the accumulators every warp has just read
        fence_before_sync();
    }
    if (!ok) {
        if (tid == 0) atomicOr(&g_tc_status, 1);
        mbar_wait_bounded(smem_u32(&mbar), phase ^ 1u);  // the MMAs end before their accumulators are freed
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (tid < 32) tmem_dealloc(tmem, ncols);
}

// The same for 1 x 3 x 3 taps and up to 16 channels (every layer of the network), with
// each value loaded three times instead of nine: a block stages, for each of the
// three rows of taps, the 128 positions of its tile and the hw positions on either
// side as BF16, eight channels (16 bytes) a position; a thread then reads the sixteen
// channels of its nine taps from there and writes its row of K.  16 -> 16 channels,
// dilation 8, 32 x 128^2 pixels, forward: 61 us (the memory's time is 10); the gather
// above, nine loads a value from L1 and L2, 88; a division per gathered value and a block
// per tile about 900.  Now bound by instruction issue: tanh, the staging and the rows of K.
// The staged positions on either side of a tile grow with the dilation: 32 x 128^2, 16 -> 16
// channels, dilation 8, 16, 24, 63, 127: 57, 70, 73, 88, 166 us, gathered 74, 72, 72, 71, 67; 2
// x 256 x 2048, 8, 16, 24, 127, 868: 112, 143, 143, 246, 1615, gathered 157, 157, 157, 152, 153.
constexpr int kStagedChannels = 16, kStagedReach = 16;
template <int MODE>
__global__ void __launch_bounds__(nntc::kM)
k_tc_conv_staged(const float *__restrict__ in, const __nv_bfloat16 *__restrict__ w, const float *__restrict__ b,
          float *__restrict__ out, Shape s, int act, int Kp, int Np)
{
    using namespace nntc;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long mbar;
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x;
    const int cin = MODE == TC_FWD ? s.ci : s.co;    // channels of the gathered operand
    const int cout = MODE == TC_FWD ? s.co : s.ci;   // channels of the result
    const int sgn = MODE == TC_FWD ? 1 : -1;
    const Line<int> l = line_of<int>(s);
    constexpr int G8 = kStagedChannels / 8;           // channel groups of eight
    const int R = (kM + 2 * l.hw + 7) / 8 * 8;        // staged positions
    constexpr int segs = 3, taps = 9;
    const int K = cin * taps;
    unsigned char *St = smem;
    unsigned char *As = St + segs * G8 * R * 16;
    unsigned char *Bs = As + kM * Kp * 2;
    const int ntiles = (l.total + kM - 1) / kM;
    const uint32_t ncols = tmem_cols(Np);
    const uint32_t lboA = (kM / 8) * 128, lboB = (uint32_t)(Np / 8) * 128;
    if (tid < 32) tmem_alloc(smem_u32(&tmem_base), ncols);
    if (tid == 0) mbar_init(smem_u32(&mbar));
    for (int idx = tid; idx < Np * (Kp >> 3); idx += kM) {
        const int k8 = idx / Np, r = idx - k8 * Np;  // r: output channel
        __nv_bfloat16 v[8];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const int k = 8 * k8 + j, c = k / taps, tap = k - c * taps;
            v[j] = __float2bfloat16_rn(0.f);
            if (r < cout && k < K)
                v[j] = MODE == TC_FWD ? w[((long long)r * s.ci + c) * taps + tap]
                                      : w[((long long)c * s.ci + r) * taps + tap];
        }
        uint4 u;
        memcpy(&u, v, sizeof u);
        *reinterpret_cast<uint4 *>(Bs + core_off(r, 8 * k8, Np)) = u;
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = tmem_base;
    bool ok = true;
    uint32_t phase = 0;
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const int q0 = tile * kM;
        for (int j = tid; j < kM + 2 * l.hw; j += kM) {
            const Pixel<int> x = position_at(s, l, q0 + j - l.hw);
            const float *base = in + (long long)x.n * cin * l.sp + x.w;
            for (int seg = 0; seg < segs; seg++) {
                const int zh = x.h + sgn * s.dh * (seg - 1);
                const bool have = x.w >= 0 && (unsigned)zh < (unsigned)s.h;
                const float *src = base + (have ? (x.d * s.h + zh) * s.w : 0);
                unsigned char *dst = St + ((seg * G8) * R + j) * 16;
#pragma unroll
                for (int g = 0; g < G8; g++) {
                    float v[8];
#pragma unroll
                    for (int i = 0; i < 8; i++) {
                        const int c = 8 * g + i;
                        v[i] = have && c < cin ? __ldg(src + (long long)c * l.sp) : 0.f;
                    }
                    *reinterpret_cast<uint4 *>(dst + g * R * 16) = make_uint4(
                        pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
                }
            }
        }
        __syncthreads();
        {
            // half words of word c / 2 of tap's vector: channels c, c + 1
            unsigned v[taps][8];
#pragma unroll
            for (int tap = 0; tap < taps; tap++) {
                const int at = tid + l.hw + sgn * s.dw * (tap % 3 - 1);
#pragma unroll
                for (int g = 0; g < G8; g++) {
                    const uint4 u = *reinterpret_cast<const uint4 *>(St + ((tap / 3 * G8 + g) * R + at) * 16);
                    v[tap][4 * g] = u.x;
                    v[tap][4 * g + 1] = u.y;
                    v[tap][4 * g + 2] = u.z;
                    v[tap][4 * g + 3] = u.w;
                }
            }
#pragma unroll
            for (int k8 = 0; k8 < kStagedChannels * taps / 8; k8++) {
                if (k8 >= (Kp >> 3)) break;
                unsigned o[4];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int k0 = 8 * k8 + 2 * j, k1 = k0 + 1, c0 = k0 / taps, c1 = k1 / taps;
                    o[j] = __byte_perm(v[k0 % taps][c0 / 2], v[k1 % taps][c1 / 2],
                                       (c0 & 1 ? 0x32 : 0x10) | (c1 & 1 ? 0x7600 : 0x5400));
                }
                *reinterpret_cast<uint4 *>(As + core_off(tid, 8 * k8, kM)) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
        fence_smem_to_async();
        fence_before_sync();
        __syncthreads();
        fence_after_sync();
        if (tid == 0) {
            issue_tile(tmem, smem_u32(As), lboA, smem_u32(Bs), lboB, Kp, Np);
            mma_commit(smem_u32(&mbar));
        }
        ok = __syncthreads_and(mbar_wait_bounded(smem_u32(&mbar), phase));
        fence_after_sync();
        phase ^= 1u;
        if (!ok) break;
        const Pixel<int> x = position_at(s, l, q0 + tid);
        float *dst = out + (long long)x.n * cout * l.sp + (x.d * s.h + x.h) * s.w + x.w;
        for (int c0 = 0; c0 < Np; c0 += 16) {
            float v[16];
            tmem_load16(tmem + ((uint32_t)(32 * (tid >> 5)) << 16) + (uint32_t)c0, v);
            if (x.w >= 0) {
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const int o = c0 + j;
                    if (o < cout) {
                        float r = v[j];
                        if (MODE == TC_FWD) {
                            r += b[o];
                            if (act == 1) r = tanhf(r);
                        }
                        dst[(long long)o * l.sp] = r;
                    }
                }
            }
        }
        // the next tile's MMAs overwrite the accumulators every warp has just read
        fence_before_sync();
    }
    if (!ok) {
        if (tid == 0) atomicOr(&g_tc_status, 1);
        mbar_wait_bounded(smem_u32(&mbar), phase ^ 1u);  // the MMAs end before their accumulators are freed
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (tid < 32) tmem_dealloc(tmem, ncols);
}

// Weight gradient, partial sums: block g accumulates, over the 128-position
// chunks c = g, g + G, ... of the line of positions, the rows r = tap * ci + i of
// part[g][r][o] = sum_p x[n,i,p + shift(tap)] gy[n,o,p]
// (rows: weight entries, `tiles` tiles of 128; K: positions; N: o), and in FP32
// the sums of gy, bpart[g][o].  k_tc_reduce_w adds the G partial sums in a fixed
// order.  A thread loads the value of one position (and the first 2 hw threads
// one of the halo) once per row of taps and channel, rounds it once and stores
// it in the kw columns that its taps along w put it in.  FAR: tap by tap, for dilations of
// a chunk and more, where the taps' positions lie apart, for taps out of reach and for 64-bit positions (2 x 256 x 2048 positions, 16
// channels, dilation 868: 243 us, with the whole halo 1214; dilation 127: 260 with it).
// Columns are stored two bytes at a time; the core matrices lie kPad bytes further apart along K than
// they are long, so that the 32 columns of a warp fall on 16 different banks (two
// columns share a word).
constexpr int kPad = 16;
template <int N16, bool FAR>
__global__ void __launch_bounds__(nntc::kM)
k_tc_conv_bwd_w(const float *__restrict__ x, const float *__restrict__ gy, float *__restrict__ part,
                float *__restrict__ bpart, Shape s, int G, int tiles)
{
    using namespace nntc;
    using I = typename std::conditional<FAR, long long, int>::type;
    constexpr int Np = 16 * N16;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long mbar;
    __shared__ uint32_t tmem_base;
    __shared__ float bsum[kM / 32][Np];
    const int tid = threadIdx.x;
    const Line<I> l = line_of<I>(s);
    const int segs = s.kd * s.kh, Kw = s.ci * segs * s.kw, rows = (Kw + 7) / 8 * 8;
    const uint32_t lboA = (uint32_t)rows * 16 + kPad, lboB = (uint32_t)Np * 16 + kPad;
    unsigned char *Bs = smem;
    unsigned char *As = smem + (kM / 8) * lboB;  // last: the rows past `rows` of the last tile read what follows
    const int mid = (s.kw - 1) / 2, reach = FAR ? taps_in_reach(s) : mid;
    if (FAR && reach < mid) {  // the columns of the taps without a source stay 0
        for (uint32_t k = tid; k < kM / 8 * lboA / 16; k += kM) reinterpret_cast<uint4 *>(As)[k] = make_uint4(0, 0, 0, 0);
    }
    const I nchunks = (l.total + kM - 1) / kM;
    const int g = blockIdx.x;
    const uint32_t ncols = tmem_cols(tiles * Np);
    if (tid < 32) tmem_alloc(smem_u32(&tmem_base), ncols);
    if (tid == 0) mbar_init(smem_u32(&mbar));
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = tmem_base;
    float bacc[Np];
#pragma unroll
    for (int o = 0; o < Np; o++) bacc[o] = 0.f;
    bool ok = true;
    int round = 0;
    for (I c = g; c < nchunks && ok; c += G, round++) {
        const I q0 = c * kM;
        {
            const Pixel<I> px = position_at<I>(s, l, q0 + tid);
            const bool valid = px.w >= 0;
            const float *src = gy + (long long)px.n * s.co * l.sp + (valid ? ((I)px.d * s.h + px.h) * s.w + px.w : 0);
            unsigned char *col = Bs + (tid >> 3) * lboB + (tid & 7) * 2;
#pragma unroll
            for (int o = 0; o < Np; o++) {
                const float v = valid && o < s.co ? __ldg(src + (long long)o * l.sp) : 0.f;
                bacc[o] += v;
                *reinterpret_cast<__nv_bfloat16 *>(col + o * 16) = __float2bfloat16_rn(v);
            }
        }
        // j: a position less q0, its value into the columns of the taps first .. last
        int first = mid - reach, last = FAR ? first : s.kw - 1;
        for (I j = tid - l.hw; FAR ? first <= mid + reach : j < kM + l.hw; j += FAR ? s.dw : kM) {
            const Pixel<I> px = position_at<I>(s, l, q0 + j);
            const float *base = x + (long long)px.n * s.ci * l.sp + px.w;
            for (int seg = 0; seg < segs; seg++) {
                const int a = seg / s.kh, f = seg - a * s.kh;
                const int zd = px.d + s.dd * (a - (s.kd - 1) / 2), zh = px.h + s.dh * (f - (s.kh - 1) / 2);
                const bool have = px.w >= 0 && (unsigned)zd < (unsigned)s.d && (unsigned)zh < (unsigned)s.h;
                const float *src = base + (have ? ((I)zd * s.h + zh) * s.w : 0);
                for (int i0 = 0; i0 < s.ci; i0 += 8) {
                    __nv_bfloat16 v[8];
#pragma unroll
                    for (int i = 0; i < 8; i++)
                        v[i] = __float2bfloat16_rn(have && i0 + i < s.ci ? __ldg(src + (long long)(i0 + i) * l.sp) : 0.f);
                    for (int e = FAR ? first : 0; e <= last; e++) {
                        const int k = (int)(j - (I)s.dw * (e - mid));
                        if ((unsigned)k >= (unsigned)kM) continue;
                        unsigned char *dst = As + (k >> 3) * lboA + (k & 7) * 2 + ((seg * s.kw + e) * s.ci + i0) * 16;
#pragma unroll
                        for (int i = 0; i < 8; i++)
                            if (i0 + i < s.ci) *reinterpret_cast<__nv_bfloat16 *>(dst + i * 16) = v[i];
                    }
                }
            }
            if (FAR) last = ++first;
        }
        fence_smem_to_async();
        fence_before_sync();
        __syncthreads();
        fence_after_sync();
        if (tid == 0) {
            const uint32_t id = idesc_bf16(kM, Np), a0 = smem_u32(As), b0 = smem_u32(Bs);
            for (int t = 0; t < tiles; t++)
                for (int k = 0; k < kM / 16; k++)
                    mma_bf16(tmem + (uint32_t)(t * Np), smem_desc(a0 + (uint32_t)t * kM * 16 + 2u * k * lboA, lboA, 128),
                             smem_desc(b0 + 2u * k * lboB, lboB, 128), id, (round > 0 || k > 0) ? 1u : 0u);
            mma_commit(smem_u32(&mbar));
        }
        // the next chunk overwrites the operands: wait for this chunk's MMAs
        ok = __syncthreads_and(mbar_wait_bounded(smem_u32(&mbar), (uint32_t)(round & 1)));
        fence_after_sync();
    }
    if (ok) {
        for (int t = 0; t < tiles; t++)
#pragma unroll
            for (int c0 = 0; c0 < Np; c0 += 16) {
                float v[16];
                tmem_load16(tmem + ((uint32_t)(32 * (tid >> 5)) << 16) + (uint32_t)(t * Np + c0), v);
                const long long r = (long long)g * tiles * kM + t * kM + tid;
#pragma unroll
                for (int j = 0; j < 16; j++) part[r * Np + c0 + j] = round > 0 ? v[j] : 0.f;
            }
    } else {
        if (tid == 0) atomicOr(&g_tc_status, 1);
        mbar_wait_bounded(smem_u32(&mbar), (uint32_t)((round - 1) & 1));
    }
#pragma unroll
    for (int o = 0; o < Np; o++) {
        float v = bacc[o];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
        if ((tid & 31) == 0) bsum[tid >> 5][o] = v;
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (tid < Np) bpart[g * Np + tid] = (bsum[0][tid] + bsum[1][tid]) + (bsum[2][tid] + bsum[3][tid]);
    if (tid < 32) tmem_dealloc(tmem, ncols);
}

// gw[o][i][tap] = sum_g part[g][tap * ci + i][o], and after the Kw rows gb[o] =
// sum_g bpart[g][o].  One block per row: thread t adds the partial sums g = t / 16,
// t / 16 + 16, ... of channel o0 + t % 16, then the sixteen are added in order (a
// fixed order: deterministic).
__global__ void __launch_bounds__(kT)
k_tc_reduce_w(const float *__restrict__ part, const float *__restrict__ bpart, float *__restrict__ gw,
              float *__restrict__ gb, int ci, int co, int taps, int G, int Mp, int Np)
{
    __shared__ float sh[16][17];
    const int r = blockIdx.x, Kw = ci * taps, lane = threadIdx.x & 15, row = threadIdx.x >> 4;
    const int tap = r / ci, i = r - tap * ci;
    const float *src = r < Kw ? part + (long long)r * Np : bpart;
    const long long stride = r < Kw ? (long long)Mp * Np : Np;
    for (int o0 = 0; o0 < co; o0 += 16) {
        float acc = 0.f;
#pragma unroll 4
        for (int g = row; g < G; g += 16) acc += src[g * stride + o0 + lane];
        sh[row][lane] = acc;
        __syncthreads();
        if (row == 0 && o0 + lane < co) {
            float t = 0.f;
#pragma unroll
            for (int k = 0; k < 16; k++) t += sh[k][lane];
            if (r < Kw) gw[((long long)(o0 + lane) * ci + i) * taps + tap] = t;
            else gb[o0 + lane] = t;
        }
        __syncthreads();
    }
}

// Scratch of one call, allocated and freed in stream order from a pool of the
// library's own (one per device; it keeps at most kPoolKeep bytes between uses),
// so that calls on different streams and threads never share it.
constexpr size_t kPoolKeep = 64u << 20;
std::mutex g_pool_mu;
cudaMemPool_t g_pool[64] = {};

cudaMemPool_t scratch_pool()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lock(g_pool_mu);
    if (!g_pool[dev]) {
        cudaMemPoolProps p{};
        p.allocType = cudaMemAllocationTypePinned;
        p.handleTypes = cudaMemHandleTypeNone;
        p.location.type = cudaMemLocationTypeDevice;
        p.location.id = dev;
        cudaMemPool_t pool = nullptr;
        if (cudaMemPoolCreate(&pool, &p) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        unsigned long long keep = kPoolKeep;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        g_pool[dev] = pool;
    }
    return g_pool[dev];
}

void *scratch_alloc(size_t bytes, cudaStream_t st)
{
    cudaMemPool_t pool = scratch_pool();
    void *p = nullptr;
    if (!pool || cudaMallocFromPoolAsync(&p, bytes, pool, st) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}

// The shapes the tensor-core kernels take: what a tile holds (include/lbm.h).
bool tc_fits(const Shape &s, int cin, int cout)
{
    return round16(cin * s.kd * s.kh * s.kw) <= nntc::kMaxKp && round16(cout) <= nntc::kMaxNp;
}

// Blocks of a kernel that an SM holds at once, times the SMs, by registers, shared
// memory, tensor memory columns and threads, at most `most`.  (The occupancy query answers 1 for
// kernels that allocate tensor memory.)
template <class K>
unsigned resident_grid(K kernel, size_t smem, int ncols, int most = 2048 / nntc::kM)
{
    int dev = 0, sms = 152, per_sm = 512 / ncols;
    cudaFuncAttributes a{};
    if (cudaFuncGetAttributes(&a, kernel) == cudaSuccess) {
        const int regs = (a.numRegs + 7) / 8 * 8 * nntc::kM;
        per_sm = std::min(per_sm, 65536 / regs);
        per_sm = std::min(per_sm, (int)(227 * 1024 / (smem + a.sharedSizeBytes + 1024)));
    } else {
        cudaGetLastError();
    }
    per_sm = std::max(1, std::min(per_sm, most));
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (unsigned)(per_sm * sms);
}

template <class K, class... A>
int tc_launch(K kernel, long long tiles, size_t smem, int Np, cudaStream_t st, const char *what, A... args)
{
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return nn_fail(LBM_ECUDA, "%s: %s", what, cudaGetErrorString(e));
    const unsigned most = resident_grid(kernel, smem, nntc::tmem_cols(Np));
    kernel<<<tiles < most ? (unsigned)tiles : most, nntc::kM, smem, st>>>(args...);
    return launched(what);
}

template <int MODE>
int tc_conv_launch(const float *in, const void *w, const float *b, float *out, const Shape &s, int act,
                   cudaStream_t st, const char *what)
{
    const int cin = MODE == TC_FWD ? s.ci : s.co, cout = MODE == TC_FWD ? s.co : s.ci, Np = round16(cout);
    const __nv_bfloat16 *wb = reinterpret_cast<const __nv_bfloat16 *>(w);
    const int taps = s.kd * s.kh * s.kw, Kp = round16(cin * taps);
    const size_t smem = (size_t)(nntc::kM + Np) * Kp * 2;
    const bool small = narrow(s);
    const long long npix = (long long)s.n * s.d * s.h * s.w, tiles = (npix + nntc::kM - 1) / nntc::kM;
    if (small && s.kd == 1 && s.kh == 3 && s.kw == 3) {
        const Line<int> l = line_of<int>(s);
        const size_t stage = (size_t)3 * (kStagedChannels / 8) * ((nntc::kM + 2 * (size_t)l.hw + 7) / 8 * 8) * 16;
        if (cin <= kStagedChannels && l.hw <= kStagedReach && l.hw == s.dw)
            return tc_launch(k_tc_conv_staged<MODE>, (l.total + nntc::kM - 1) / nntc::kM, smem + stage, Np, st, what, in,
                             wb, b, out, s, act, Kp, Np);
        return tc_launch(k_tc_conv<MODE, 9, int>, tiles, smem, Np, st, what, in, wb, b, out, s, act, Kp, Np);
    }
    if (small) return tc_launch(k_tc_conv<MODE, 0, int>, tiles, smem, Np, st, what, in, wb, b, out, s, act, Kp, Np);
    return tc_launch(k_tc_conv<MODE, 0, long long>, tiles, smem, Np, st, what, in, wb, b, out, s, act, Kp, Np);
}

template <int N16, bool FAR>
int tc_conv_bwd_w_launch(const float *x, const float *gy, float *gw, float *gb, const Shape &s, cudaStream_t st)
{
    constexpr int Np = 16 * N16;
    const int taps = s.kd * s.kh * s.kw, Kw = s.ci * taps, rows = (Kw + 7) / 8 * 8;
    const int tiles = (Kw + nntc::kM - 1) / nntc::kM, Mp = tiles * nntc::kM;
    const long long nchunks = (line_of<long long>(s).total + nntc::kM - 1) / nntc::kM;
    const size_t smem = (size_t)(nntc::kM / 8) * (rows * 16 + kPad + Np * 16 + kPad) + (size_t)(Mp - rows) * 16;
    cudaError_t e = cudaFuncSetAttribute(k_tc_conv_bwd_w<N16, FAR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return nn_fail(LBM_ECUDA, "conv3d_backward(weights): %s", cudaGetErrorString(e));
    // The number of partial sums is part of the result (its last bits), so it does not follow
    // the registers that the compiler takes: 7, 6, 5 and 4 blocks per SM fit for 16 to 64 channels.
    unsigned G = resident_grid(k_tc_conv_bwd_w<N16, FAR>, smem, nntc::tmem_cols(tiles * Np), 8 - N16);
    if (G > nchunks) G = (unsigned)nchunks;
    float *part = static_cast<float *>(scratch_alloc((size_t)G * (Mp + 1) * Np * sizeof(float), st));
    if (!part) return nn_fail(LBM_ENOMEM, "conv3d_backward: tensor-core workspace");
    float *bpart = part + (size_t)G * Mp * Np;
    k_tc_conv_bwd_w<N16, FAR><<<G, nntc::kM, smem, st>>>(x, gy, part, bpart, s, (int)G, tiles);
    k_tc_reduce_w<<<Kw + 1, kT, 0, st>>>(part, bpart, gw, gb, s.ci, s.co, taps, (int)G, Mp, Np);
    const int rc = launched("conv3d_backward(weights)");
    cudaFreeAsync(part, st);
    return rc;
}

template <int N16>
int tc_conv_bwd_w(const float *x, const float *gy, float *gw, float *gb, const Shape &s, cudaStream_t st)
{
    return s.dw >= nntc::kM || taps_in_reach(s) < (s.kw - 1) / 2 || !narrow(s) ? tc_conv_bwd_w_launch<N16, true>(x, gy, gw, gb, s, st)
                            : tc_conv_bwd_w_launch<N16, false>(x, gy, gw, gb, s, st);
}

int check_shape(const int *sp, const int *k, const int *dil, int n, int ci, int co, Shape &s)
{
    if (!sp || !k || !dil) return nn_fail(LBM_EINVAL, "shape, kernel and dilation are required");
    if (n < 1 || ci < 1 || co < 1) return nn_fail(LBM_EINVAL, "batch and channel counts must be >= 1");
    for (int d = 0; d < 3; d++) {
        if (sp[d] < 1) return nn_fail(LBM_EINVAL, "spatial extents must be >= 1");
        if (k[d] < 1 || (k[d] & 1) == 0) return nn_fail(LBM_EINVAL, "kernel extents must be odd");
        if (dil[d] < 1) return nn_fail(LBM_EINVAL, "dilations must be >= 1");
    }
    s = Shape{n, ci, co, sp[0], sp[1], sp[2], k[0], k[1], k[2], dil[0], dil[1], dil[2]};
    if (s.in_count() > (1LL << 40) || s.out_count() > (1LL << 40)) return nn_fail(LBM_EINVAL, "tensor too large");
    return LBM_OK;
}

}  // namespace

extern "C" {

const char *lbm_nn_last_error(void) { return g_nn_error.c_str(); }

int lbm_nn_tc_status(int *status)
{
    if (!status) return nn_fail(LBM_EINVAL, "tc_status: status is NULL");
    int v = 0, zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_tc_status, sizeof v);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_tc_status, &zero, sizeof zero);
    if (e != cudaSuccess) return nn_fail(LBM_ECUDA, "tc_status: %s", cudaGetErrorString(e));
    *status = v;
    return LBM_OK;
}

int lbm_nn_conv3d_forward(const float *x, const void *w, int w_bf16, const float *b, float *y, int n, int ci, int co,
                          const int dhw[3], const int k[3], const int dil[3], int act, void *stream)
{
    Shape s;
    int rc = check_shape(dhw, k, dil, n, ci, co, s);
    if (rc != LBM_OK) return rc;
    if (!x || !w || !b || !y) return nn_fail(LBM_EINVAL, "conv3d_forward: NULL pointer");
    if (act != 0 && act != 1) return nn_fail(LBM_EINVAL, "conv3d_forward: act must be 0 or 1");
    if (w_bf16 && tc_fits(s, ci, co))
        return tc_conv_launch<TC_FWD>(x, w, b, y, s, act, (cudaStream_t)stream, "conv3d_forward");
    k_conv_fwd<<<grid_of(s.out_count(), kT), kT, 0, (cudaStream_t)stream>>>(x, w, w_bf16, b, y, s, act);
    return launched("conv3d_forward");
}

int lbm_nn_conv3d_backward(const float *x, const void *w, int w_bf16, const float *gy, float *gx, float *gw, float *gb,
                           int n, int ci, int co, const int dhw[3], const int k[3], const int dil[3], void *stream)
{
    Shape s;
    int rc = check_shape(dhw, k, dil, n, ci, co, s);
    if (rc != LBM_OK) return rc;
    if (!x || !w || !gy || !gw || !gb) return nn_fail(LBM_EINVAL, "conv3d_backward: NULL pointer");
    cudaStream_t st = (cudaStream_t)stream;
    const int taps = s.kd * s.kh * s.kw;
    if (gx) {
        if (w_bf16 && tc_fits(s, co, ci)) {
            rc = tc_conv_launch<TC_BWD_IN>(gy, w, nullptr, gx, s, 0, st, "conv3d_backward(input)");
        } else {
            k_conv_bwd_in<<<grid_of(s.in_count(), kT), kT, 0, st>>>(gy, w, w_bf16, gx, s);
            rc = launched("conv3d_backward(input)");
        }
        if (rc != LBM_OK) return rc;
    }
    if (w_bf16 && ci * taps <= nntc::kMaxKp && round16(co) <= nntc::kMaxNp)
        switch (round16(co) / 16) {
        case 1: return tc_conv_bwd_w<1>(x, gy, gw, gb, s, st);
        case 2: return tc_conv_bwd_w<2>(x, gy, gw, gb, s, st);
        case 3: return tc_conv_bwd_w<3>(x, gy, gw, gb, s, st);
        default: return tc_conv_bwd_w<4>(x, gy, gw, gb, s, st);
        }
    const long long blocks = (long long)co * ci * taps + co;
    k_conv_bwd_w<<<(unsigned)blocks, kT, 0, st>>>(x, gy, gw, gb, s);
    return launched("conv3d_backward(weights)");
}

int lbm_nn_tanh_backward(float *g, const float *y, long long count, void *stream)
{
    if (!g || !y || count < 0) return nn_fail(LBM_EINVAL, "tanh_backward: bad arguments");
    if (count == 0) return LBM_OK;
    const int vec = (reinterpret_cast<uintptr_t>(g) | reinterpret_cast<uintptr_t>(y)) % 16 == 0;
    k_tanh_bwd<<<grid_of((count + 3) / 4, kT), kT, 0, (cudaStream_t)stream>>>(g, y, count, vec);
    return launched("tanh_backward");
}

int lbm_nn_mse(const float *y, const float *t, float *g, long long count, double *loss, void *stream)
{
    if (!y || !t || !g || !loss || count < 1) return nn_fail(LBM_EINVAL, "mse: bad arguments");
    cudaStream_t st = (cudaStream_t)stream;
    const long long want = (count + 4 * kT - 1) / (4 * kT);
    const int blocks = (int)(want < kMseBlocks ? want : kMseBlocks);
    double *part = static_cast<double *>(scratch_alloc(blocks * sizeof(double), st));
    if (!part) return nn_fail(LBM_ENOMEM, "mse: workspace");
    k_mse<<<blocks, kT, 0, st>>>(y, t, g, count, part);
    k_mse_final<<<1, kT, 0, st>>>(part, blocks, count, loss);
    const int rc = launched("mse");
    cudaFreeAsync(part, st);
    return rc;
}

int lbm_nn_adam(float *p, const float *g, float *m, float *v, void *p_bf16, long long count, double lr, double b1,
                double b2, double eps, long long step, void *stream)
{
    if (!p || !g || !m || !v || count < 0 || step < 1) return nn_fail(LBM_EINVAL, "adam: bad arguments");
    if (count == 0) return LBM_OK;
    const float c1 = (float)(1.0 - pow(b1, (double)step)), c2 = (float)(1.0 - pow(b2, (double)step));
    k_adam<<<grid_of(count, kT), kT, 0, (cudaStream_t)stream>>>(p, g, m, v, (__nv_bfloat16 *)p_bf16, count, (float)lr,
                                                                 (float)b1, (float)b2, (float)eps, c1, c2);
    return launched("adam");
}

int lbm_nn_to_bf16(const float *p, void *p_bf16, long long count, void *stream)
{
    if (!p || !p_bf16 || count < 0) return nn_fail(LBM_EINVAL, "to_bf16: bad arguments");
    if (count == 0) return LBM_OK;
    k_to_bf16<<<grid_of(count, kT), kT, 0, (cudaStream_t)stream>>>(p, (__nv_bfloat16 *)p_bf16, count);
    return launched("to_bf16");
}

}  // extern "C"
