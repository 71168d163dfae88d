// nn_backward.cu -- the element-wise part of the bf16 network's backward
// pass, fused: what lies between two convolutions runs as one kernel that
// reads the incoming gradient once and writes the bfloat16 gradient that the
// next convolutions read (the FP32 gradient of the pre-activation itself is
// not stored).  Bias and weight gradients leave per-block partial sums, which
// one kernel adds for all layers at the end of the pass.
//
// All of it is bound by memory.  Measured on GB300 at 64^3 x 4, 16 channels
// in the finest level: the output head's backward 212 us in nine kernels ->
// 35 us in one; pooling gradient, skip sum, activation and bias 87 us in
// three -> 33 us; the 25 final sums 250 us -> 36 us; the 13 weight
// transposes 47 us -> 10 us.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "nn.h"

namespace lbm {
namespace nn {

namespace {

constexpr float kSlope = 0.1f;  // leaky ReLU
constexpr int kThreads = 256;

__device__ __forceinline__ float4 load4(const __nv_bfloat16 *p)
{
    const uint2 q = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&q.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&q.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 load4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void add4(float4 &s, const float4 &a)
{
    s.x += a.x;
    s.y += a.y;
    s.z += a.z;
    s.w += a.w;
}
__device__ __forceinline__ uint2 narrow4(const float4 &g)
{
    const __nv_bfloat162 lo = __floats2bfloat162_rn(g.x, g.y), hi = __floats2bfloat162_rn(g.z, g.w);
    uint2 pk;
    pk.x = *reinterpret_cast<const unsigned *>(&lo);
    pk.y = *reinterpret_cast<const unsigned *>(&hi);
    return pk;
}

// The gradient g of a layer's output, its activation's derivative applied
// and narrowed to dyn; the layer's bias gradient as partials[block][c].
//  kPlain: g as it is.
//  kUp2:   g is the gradient of the upsampled tensor (edge 2n): the sum of
//          the eight children.
//  kPool:  g plus an eighth of the gradient h of the pooled tensor (edge n / 2).
// Four channels per thread.  The grid stride is a multiple of the c / 4
// groups, so a thread always meets the same four channels and sums them.
template <GradSource SRC>
__global__ void __launch_bounds__(kThreads)
    grad_narrow_kernel(const float *__restrict__ g, const float *__restrict__ h,
                       const __nv_bfloat16 *__restrict__ yout, __nv_bfloat16 *__restrict__ dyn, unsigned len4, int n,
                       int c4, float *__restrict__ partials)
{
    chain_wait();
    chain_release();
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    const int c = 4 * c4;
    for (unsigned i = blockIdx.x * kThreads + threadIdx.x; i < len4; i += gridDim.x * kThreads) {
        float4 v;
        if constexpr (SRC == GradSource::kPlain) {
            v = load4(g + 4 * static_cast<size_t>(i));
        } else {
            const unsigned q = i % c4;
            unsigned r = i / c4;
            const unsigned x = r % n;
            r /= n;
            const unsigned y = r % n;
            r /= n;
            const unsigned z = r % n, b = r / n;
            if constexpr (SRC == GradSource::kUp2) {
                const unsigned m = 2 * n;
                const float *p = g + ((((static_cast<size_t>(b) * m + 2 * z) * m + 2 * y) * m + 2 * x) * c + 4 * q);
                v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    add4(v, load4(p + ((static_cast<size_t>(k >> 2) * m + ((k >> 1) & 1)) * m + (k & 1)) * c));
            } else {
                const unsigned m = n / 2;
                v = load4(g + 4 * static_cast<size_t>(i));
                const float4 a = load4(h + ((((static_cast<size_t>(b) * m + z / 2) * m + y / 2) * m + x / 2) * c + 4 * q));
                add4(v, make_float4(0.125f * a.x, 0.125f * a.y, 0.125f * a.z, 0.125f * a.w));
            }
        }
        const float4 o = load4(yout + 4 * static_cast<size_t>(i));
        if (!(o.x > 0.f)) v.x *= kSlope;
        if (!(o.y > 0.f)) v.y *= kSlope;
        if (!(o.z > 0.f)) v.z *= kSlope;
        if (!(o.w > 0.f)) v.w *= kSlope;
        reinterpret_cast<uint2 *>(dyn)[i] = narrow4(v);
        add4(acc, v);
    }
    __shared__ float4 red[kThreads];
    red[threadIdx.x] = acc;
    __syncthreads();
    if (static_cast<int>(threadIdx.x) < c4) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = threadIdx.x; k < kThreads; k += c4) add4(t, red[k]);
        *reinterpret_cast<float4 *>(partials + static_cast<size_t>(blockIdx.x) * c + 4 * threadIdx.x) = t;
    }
}

// The output head (1^3, 16 -> 5, no activation) and the layer before it: per
// voxel the loss term and d = 2 (out - target) / len; the head's weight
// gradient d x h and bias gradient d (FP32); the gradient of h from d rounded
// to bfloat16 and the weights, then h's activation derivative, narrowed to
// dyn, and that layer's bias gradient.  Per block: partials[block] =
// (head weights [5][16], head biases [5], bias gradient [16]) and the loss.
constexpr int kHeadIn = 16, kHeadOut = 5;
constexpr int kHeadSums = kHeadOut * kHeadIn + kHeadOut + kHeadIn;

__global__ void __launch_bounds__(kThreads)
    head_backward_kernel(const __nv_bfloat16 *__restrict__ out, const float *__restrict__ target,
                         const __nv_bfloat16 *__restrict__ h, const __nv_bfloat16 *__restrict__ w,
                         __nv_bfloat16 *__restrict__ dyn, long long voxels, float *__restrict__ partials,
                         double *__restrict__ loss)
{
    __shared__ float ws[kHeadOut][kHeadIn];
    for (int e = threadIdx.x; e < kHeadOut * kHeadIn; e += kThreads) ws[e / kHeadIn][e % kHeadIn] = __bfloat162float(w[e]);
    __syncthreads();
    chain_wait();
    chain_release();
    constexpr int C = kHeadIn / 2;  // two threads per voxel, eight channels each
    const int c0 = C * (threadIdx.x & 1);
    const float scale = 2.0f / static_cast<float>(voxels * kHeadOut);
    float dw[kHeadOut][C], db[kHeadOut], dh[C];
    double sq = 0.0;
#pragma unroll
    for (int i = 0; i < C; ++i) {
        dh[i] = 0.f;
#pragma unroll
        for (int o = 0; o < kHeadOut; ++o) dw[o][i] = 0.f;
    }
#pragma unroll
    for (int o = 0; o < kHeadOut; ++o) db[o] = 0.f;
    for (long long v = (blockIdx.x * static_cast<long long>(kThreads) + threadIdx.x) / 2; v < voxels;
         v += static_cast<long long>(gridDim.x) * (kThreads / 2)) {
        float x[C];
        const uint4 u = *reinterpret_cast<const uint4 *>(h + v * kHeadIn + c0);
        const unsigned word[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&word[j]));
            x[2 * j] = f.x;
            x[2 * j + 1] = f.y;
        }
        float e[kHeadOut], dn[kHeadOut];  // dn: d rounded as the tensor cores' operands are
#pragma unroll
        for (int o = 0; o < kHeadOut; ++o) {
            e[o] = __bfloat162float(out[v * kHeadOut + o]) - target[v * kHeadOut + o];
            const float d = scale * e[o];
            db[o] += d;
#pragma unroll
            for (int i = 0; i < C; ++i) dw[o][i] = fmaf(d, x[i], dw[o][i]);
            dn[o] = __bfloat162float(__float2bfloat16_rn(d));
        }
        // the two threads share the squares (FP64 runs at 1/64 of the FP32
        // rate and would otherwise bound the kernel)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float m = c0 == 0 ? e[k] : (k < 2 ? e[3 + k] : 0.f);
            sq += static_cast<double>(m) * m;
        }
        float g[C];
#pragma unroll
        for (int i = 0; i < C; ++i) {
            float r = 0.f;
#pragma unroll
            for (int o = 0; o < kHeadOut; ++o) r = fmaf(dn[o], ws[o][c0 + i], r);
            if (!(x[i] > 0.f)) r *= kSlope;
            dh[i] += r;
            g[i] = r;
        }
        const uint2 lo = narrow4(make_float4(g[0], g[1], g[2], g[3])), hi = narrow4(make_float4(g[4], g[5], g[6], g[7]));
        *reinterpret_cast<uint4 *>(dyn + v * kHeadIn + c0) = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
    // fixed-order sums: a shuffle tree over a warp's threads of the same half,
    // then the warps in order
    __shared__ float red[kThreads / 32][kHeadSums];
    __shared__ double redl[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto total = [&](float s, int at, bool mine) {
#pragma unroll
        for (int d = 16; d > 1; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if (mine) red[warp][at] = s;
    };
#pragma unroll
    for (int o = 0; o < kHeadOut; ++o) {
#pragma unroll
        for (int i = 0; i < C; ++i) total(dw[o][i], o * kHeadIn + c0 + i, lane < 2);
        total(db[o], kHeadOut * kHeadIn + o, lane == 0);
    }
#pragma unroll
    for (int i = 0; i < C; ++i) total(dh[i], kHeadOut * kHeadIn + kHeadOut + c0 + i, lane < 2);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, d);
    if (lane == 0) redl[warp] = sq;
    __syncthreads();
    for (int k = threadIdx.x; k < kHeadSums; k += kThreads) {
        float s = 0.f;
        for (int i = 0; i < kThreads / 32; ++i) s += red[i][k];
        partials[static_cast<size_t>(blockIdx.x) * kHeadSums + k] = s;
    }
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < kThreads / 32; ++i) s += redl[i];
        loss[blockIdx.x] = s;
    }
}

// Adds the partial sums of many arrays at once: out[i] = sum over chunks of
// partials[chunk * stride + i], i < len, in a fixed order.  A block covers E
// consecutive elements of one array with 256 / E lanes over the chunks; lane
// l adds chunks l, l + L, ... into four interleaved sums, and the lanes are
// then added in order.  The block after the last array's adds the loss.
__global__ void __launch_bounds__(kThreads) sum_all_kernel(const __grid_constant__ SumList list)
{
    __shared__ float red[kThreads];
    chain_wait();
    chain_release();
    const int b = static_cast<int>(blockIdx.x);
    if (b == list.first[list.count]) {
        __shared__ double redd[kThreads];
        double s = 0.0;
        for (int i = threadIdx.x; i < list.loss_parts; i += kThreads) s += list.loss_partials[i];
        redd[threadIdx.x] = s;
        __syncthreads();
        for (int o = kThreads / 2; o > 0; o >>= 1) {
            if (static_cast<int>(threadIdx.x) < o) redd[threadIdx.x] += redd[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) *list.loss = redd[0] * list.loss_scale;
        return;
    }
    int k = 0;
    while (b >= list.first[k + 1]) ++k;
    const SumArray &A = list.a[k];
    const int E = A.width, L = kThreads / E;
    const int e = threadIdx.x % E, lane = threadIdx.x / E;
    const int i = (b - list.first[k]) * E + e;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    if (i < A.len) {
        const float *p = A.partials + i;
        const size_t st = A.stride;
        int c = lane;
        for (; c + 3 * L < A.chunks; c += 4 * L) {
            s0 += p[c * st];
            s1 += p[(c + L) * st];
            s2 += p[(c + 2 * L) * st];
            s3 += p[(c + 3 * L) * st];
        }
        for (; c < A.chunks; c += L) s0 += p[c * st];
    }
    red[threadIdx.x] = (s0 + s1) + (s2 + s3);
    __syncthreads();
    if (lane == 0 && i < A.len) {
        float tot = 0.f;
        for (int l = 0; l < L; ++l) tot += red[l * E + e];
        A.out[i] = tot;
    }
}

// The output head's forward pass, y[v][co] = b[co] + sum_ci h[v][ci] w[co][ci]
// rounded to bfloat16, for 16 input channels: one voxel per thread, its
// channels in two 16-byte loads.  TO = float stores the rounded value widened.
template <typename TO>
__global__ void __launch_bounds__(kThreads)
    head_forward_kernel(const __nv_bfloat16 *__restrict__ h, const __nv_bfloat16 *__restrict__ w,
                        const float *__restrict__ bias, TO *__restrict__ y, long long voxels)
{
    __shared__ float ws[kHeadOut][kHeadIn], bs[kHeadOut];
    for (int e = threadIdx.x; e < kHeadOut * kHeadIn; e += kThreads) ws[e / kHeadIn][e % kHeadIn] = __bfloat162float(w[e]);
    if (threadIdx.x < kHeadOut) bs[threadIdx.x] = bias[threadIdx.x];
    __syncthreads();
    chain_wait();
    chain_release();
    const long long v = blockIdx.x * static_cast<long long>(kThreads) + threadIdx.x;
    if (v >= voxels) return;
    float x[kHeadIn];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint4 u = reinterpret_cast<const uint4 *>(h + v * kHeadIn)[k];
        const unsigned word[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&word[j]));
            x[8 * k + 2 * j] = f.x;
            x[8 * k + 2 * j + 1] = f.y;
        }
    }
#pragma unroll
    for (int o = 0; o < kHeadOut; ++o) {
        float r = bs[o];
#pragma unroll
        for (int i = 0; i < kHeadIn; ++i) r = fmaf(x[i], ws[o][i], r);
        const __nv_bfloat16 q = __float2bfloat16_rn(r);
        if constexpr (sizeof(TO) == 4) y[v * kHeadOut + o] = __bfloat162float(q);
        else y[v * kHeadOut + o] = q;
    }
}

// Every listed layer's weights transposed for the input gradient:
// wt[tap][ci][co] = w[26 - tap][co][ci], at the same offset.
__global__ void __launch_bounds__(kThreads)
    flip_all_kernel(const __nv_bfloat16 *__restrict__ w, __nv_bfloat16 *__restrict__ wt, const __grid_constant__ FlipList list)
{
    chain_wait();
    chain_release();
    const int i = static_cast<int>(blockIdx.x * kThreads + threadIdx.x);
    if (i >= list.first[list.count]) return;
    int k = 0;
    while (i >= list.first[k + 1]) ++k;
    const int j = i - list.first[k], cin = list.cin[k], cout = list.cout[k];
    const int co = j % cout, ci = j / cout % cin, tap = j / (cout * cin);
    wt[list.offset[k] + j] = w[list.offset[k] + (static_cast<size_t>(26 - tap) * cout + co) * cin + ci];
}

}  // namespace

cudaError_t grad_narrow(GradSource src, const float *g, const float *h, const __nv_bfloat16 *yout, __nv_bfloat16 *dyn,
                        long long voxels, int n, int c, float *partials, cudaStream_t s)
{
    const long long len4 = voxels * c / 4;
    // the grid stride stays below 2^32 and is a multiple of c / 4
    if (c % 4 != 0 || kThreads % (c / 4) != 0 || len4 >= (1LL << 31)) return cudaErrorInvalidValue;
    const unsigned l = static_cast<unsigned>(len4);
    switch (src) {
    case GradSource::kPlain:
        return launch_chained(grad_narrow_kernel<GradSource::kPlain>, kGradBlocks, kThreads, 0, s, true, g, h, yout, dyn, l, n,
                              c / 4, partials);
    case GradSource::kUp2:
        return launch_chained(grad_narrow_kernel<GradSource::kUp2>, kGradBlocks, kThreads, 0, s, true, g, h, yout, dyn, l, n,
                              c / 4, partials);
    default:
        return launch_chained(grad_narrow_kernel<GradSource::kPool>, kGradBlocks, kThreads, 0, s, true, g, h, yout, dyn, l, n,
                              c / 4, partials);
    }
}

template <typename TO>
cudaError_t head_forward(const __nv_bfloat16 *h, const __nv_bfloat16 *w, const float *bias, TO *y, long long voxels,
                         cudaStream_t s)
{
    const long long blocks = (voxels + kThreads - 1) / kThreads;
    if (blocks >= (1LL << 31)) return cudaErrorInvalidValue;
    return launch_chained(head_forward_kernel<TO>, static_cast<unsigned>(blocks), kThreads, 0, s, true, h, w, bias, y, voxels);
}
template cudaError_t head_forward<float>(const __nv_bfloat16 *, const __nv_bfloat16 *, const float *, float *, long long,
                                         cudaStream_t);
template cudaError_t head_forward<__nv_bfloat16>(const __nv_bfloat16 *, const __nv_bfloat16 *, const float *,
                                                 __nv_bfloat16 *, long long, cudaStream_t);

size_t head_partial_floats() { return static_cast<size_t>(kHeadBlocks) * kHeadSums; }

cudaError_t head_backward(const __nv_bfloat16 *out, const float *target, const __nv_bfloat16 *h, const __nv_bfloat16 *w,
                          __nv_bfloat16 *dyn, long long voxels, float *partials, double *loss_partials, float *dw,
                          float *db, float *db_before, SumList &sums, cudaStream_t s)
{
    const cudaError_t e = launch_chained(head_backward_kernel, kHeadBlocks, kThreads, 0, s, true, out, target, h, w, dyn,
                                         voxels, partials, loss_partials);
    constexpr int kw = kHeadOut * kHeadIn;
    sums.add(partials, kHeadSums, dw, kw, kHeadBlocks);
    sums.add(partials + kw, kHeadSums, db, kHeadOut, kHeadBlocks);
    sums.add(partials + kw + kHeadOut, kHeadSums, db_before, kHeadIn, kHeadBlocks);
    sums.loss_partials = loss_partials;
    sums.loss_parts = kHeadBlocks;
    sums.loss_scale = 1.0 / static_cast<double>(voxels * kHeadOut);
    return e;
}

void SumList::add(const float *partials, size_t stride, float *out, int len, int chunks)
{
    SumArray &A = a[count];
    A.partials = partials;
    A.out = out;
    A.stride = stride;
    A.len = len;
    A.chunks = chunks;
    // few chunks: a thread per element; many: a line, or a sector, of
    // elements per block and the other threads as lanes over the chunks
    A.width = chunks <= 32 ? kThreads : (chunks <= 128 ? 32 : 8);
    first[count + 1] = first[count] + (len + A.width - 1) / A.width;
    ++count;
}

cudaError_t sum_all(const SumList &list, cudaStream_t s)
{
    return launch_chained(sum_all_kernel, list.first[list.count] + 1, kThreads, 0, s, true, list);
}

cudaError_t flip_all(const __nv_bfloat16 *w, __nv_bfloat16 *wt, const FlipList &list, cudaStream_t s)
{
    const int len = list.first[list.count];
    return launch_chained(flip_all_kernel, (len + kThreads - 1) / kThreads, kThreads, 0, s, true, w, wt, list);
}

}  // namespace nn
}  // namespace lbm
