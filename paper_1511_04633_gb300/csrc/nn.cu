// nn.cu -- kernels of the warm-start surrogate: a 3-D convolutional U-Net
// that maps a cavity's parameters (Ra, wall type) to an approximate steady
// state (u, v, w, theta).  Forward and backward passes, the loss and the
// Adam update are all here; surrogate.cu strings them together.
//
// Layout: activations channels-last [n][z][y][x][c] (c fastest), weights of a
// k^3 convolution [tap][cout][cin] (cin fastest), taps ordered
// (dz, dy, dx) with dx fastest, each in -(k/2)..(k/2); zero padding.  The
// storage type of activations and weights is float or bfloat16 (T); every
// sum accumulates in FP32; gradients are FP32.  Every reduction runs in a
// fixed order (per-block partials, then an ordered finishing pass), so the
// training is bitwise repeatable.
#include <atomic>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "internal.h"
#include "nn.h"

namespace lbm {
namespace nn {

namespace {

template <typename T>
__device__ __forceinline__ float ldf(const T *p);
template <>
__device__ __forceinline__ float ldf<float>(const float *p) { return *p; }
template <>
__device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16 *p) { return __bfloat162float(*p); }

template <typename T>
__device__ __forceinline__ void stf(T *p, float v);
template <>
__device__ __forceinline__ void stf<float>(float *p, float v) { *p = v; }
template <>
__device__ __forceinline__ void stf<__nv_bfloat16>(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

constexpr float kSlope = 0.1f;  // leaky ReLU

// ---------------------------------------------------------------- convolution

// Direct convolution, one block per (sample, z, 8 x 8 tile of (y, x), group
// of 32 output channels).  The input tile with its halo and the weights of
// the group are staged in shared memory 8 input channels at a time; each of
// the 256 threads owns 2 voxels x 4 output channels (64 x 32 / 256).
constexpr int kTile = 8;
constexpr int kCoTile = 32;
constexpr int kCiChunk = 8;

template <typename TI, typename TW, typename TO, int K>
__global__ void __launch_bounds__(256) conv3d_kernel(const TI *__restrict__ x, const TW *__restrict__ w,
                                                     const float *__restrict__ bias,
                                                     TO *__restrict__ y, int n, int cin, int cout,
                                                     int act)
{
    constexpr int R = K / 2;
    constexpr int H = kTile + 2 * R;  // halo tile edge
    __shared__ float xs[K][H][H][kCiChunk];
    // weights padded to 9 per output channel: the 8 channel groups of a warp
    // then hit 8 different banks
    __shared__ float ws[K * K * K][kCoTile][kCiChunk + 1];
    const int tiles = n / kTile;
    int bid = blockIdx.x;
    const int tx0 = (bid % tiles) * kTile;
    bid /= tiles;
    const int ty0 = (bid % tiles) * kTile;
    bid /= tiles;
    const int z = bid % n;
    const int b = bid / n;
    const int co0 = blockIdx.y * kCoTile;
    const int t = threadIdx.x;
    // thread -> 2 voxels (vx, vx + 32 in the flattened 8 x 8 tile) x 4 channels
    const int cg = t & 7;          // channel group: channels co0 + cg*4 .. +3
    const int v0 = t >> 3;         // 0..31
    float acc[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    const long long plane = static_cast<long long>(n) * n;
    const TI *xb = x + static_cast<long long>(b) * n * plane * cin;
    for (int ci0 = 0; ci0 < cin; ci0 += kCiChunk) {
        // stage the input halo tile for channels ci0 .. ci0 + 7
        for (int e = t; e < K * H * H * kCiChunk; e += 256) {
            const int c = e % kCiChunk;
            int r = e / kCiChunk;
            const int hx = r % H;
            r /= H;
            const int hy = r % H;
            const int hz = r / H;
            const int gz = z + hz - R, gy = ty0 + hy - R, gx = tx0 + hx - R;
            float v = 0.f;
            if (gz >= 0 && gz < n && gy >= 0 && gy < n && gx >= 0 && gx < n && ci0 + c < cin)
                v = ldf(xb + ((static_cast<long long>(gz) * n + gy) * n + gx) * cin + ci0 + c);
            xs[hz][hy][hx][c] = v;
        }
        for (int e = t; e < K * K * K * kCoTile * kCiChunk; e += 256) {
            const int c = e % kCiChunk;
            int r = e / kCiChunk;
            const int co = r % kCoTile;
            const int tap = r / kCoTile;
            float v = 0.f;
            if (co0 + co < cout && ci0 + c < cin)
                v = ldf(w + (static_cast<long long>(tap) * cout + co0 + co) * cin + ci0 + c);
            ws[tap][co][c] = v;
        }
        __syncthreads();
#pragma unroll 1
        for (int tap = 0; tap < K * K * K; ++tap) {
            const int dz = tap / (K * K), dy = (tap / K) % K, dx = tap % K;
#pragma unroll
            for (int c = 0; c < kCiChunk; ++c) {
                float xv[2], wv[4];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int v = v0 + 32 * i;
                    xv[i] = xs[dz][(v >> 3) + dy][(v & 7) + dx][c];
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) wv[j] = ws[tap][cg * 4 + j][c];
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xv[i], wv[j], acc[i][j]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int v = v0 + 32 * i;
        const int gy = ty0 + (v >> 3), gx = tx0 + (v & 7);
        TO *yo = y + (((static_cast<long long>(b) * n + z) * n + gy) * n + gx) * cout;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int co = co0 + cg * 4 + j;
            if (co >= cout) continue;
            float r = acc[i][j] + (bias ? bias[co] : 0.f);
            if (act) r = r > 0.f ? r : kSlope * r;
            stf(yo + co, r);
        }
    }
}

// Tensor-core convolution for bfloat16 inputs and weights (implicit GEMM
// with mma.sync m16n8k16, FP32 accumulation).  One block of 4 warps per
// (sample, z, 8 x 8 tile of (y, x), 32 output channels): GEMM rows are the
// 64 voxels of the tile, columns the 32 channels, and the reduction runs
// over taps x input channels in chunks of 16.  The input halo tile and the
// weights of one z-plane of taps are staged in shared memory with 24-element
// strides per voxel / channel, which keeps the fragment loads free of bank
// conflicts (8 rows x 12 words cover the 32 banks).  Warp w owns tile rows
// 16w..16w+15 (two y-rows of 8 voxels) and all 4 column tiles.
constexpr int kMmaStride = 24;

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                               unsigned b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int K, typename TO>
__global__ void __launch_bounds__(128) conv3d_mma_kernel(const __nv_bfloat16 *__restrict__ x,
                                                         const __nv_bfloat16 *__restrict__ w,
                                                         const float *__restrict__ bias,
                                                         TO *__restrict__ y, int n, int cin, int cout,
                                                         int act)
{
    constexpr int R = K / 2;
    constexpr int H = kTile + 2 * R;
    __shared__ __align__(16) __nv_bfloat16 xs[K][H][H][kMmaStride];
    __shared__ __align__(16) __nv_bfloat16 ws[K * K][kCoTile][kMmaStride];
    const int tiles = n / kTile;
    int bid = blockIdx.x;
    const int tx0 = (bid % tiles) * kTile;
    bid /= tiles;
    const int ty0 = (bid % tiles) * kTile;
    bid /= tiles;
    const int z = bid % n;
    const int b = bid / n;
    const int co0 = blockIdx.y * kCoTile;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int g = lane >> 2, tig = lane & 3;
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = 0.f;
    const long long plane = static_cast<long long>(n) * n;
    const __nv_bfloat16 *xb = x + static_cast<long long>(b) * n * plane * cin;
    const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
    for (int ci0 = 0; ci0 < cin; ci0 += 16) {
        // input halo tile: 16-byte granules of 8 channels
        for (int e = t; e < K * H * H * 2; e += 128) {
            const int half = e & 1;
            int r = e >> 1;
            const int hx = r % H;
            r /= H;
            const int hy = r % H;
            const int hz = r / H;
            const int gz = z + hz - R, gy = ty0 + hy - R, gx = tx0 + hx - R;
            const int c = ci0 + 8 * half;
            uint4 v = zero4;
            if (gz >= 0 && gz < n && gy >= 0 && gy < n && gx >= 0 && gx < n && c < cin)
                v = *reinterpret_cast<const uint4 *>(xb + ((static_cast<long long>(gz) * n + gy) * n + gx) * cin + c);
            *reinterpret_cast<uint4 *>(&xs[hz][hy][hx][8 * half]) = v;
        }
        for (int tz = 0; tz < K; ++tz) {
            __syncthreads();  // previous plane's weights fully consumed
            for (int e = t; e < K * K * kCoTile * 2; e += 128) {
                const int half = e & 1;
                int r = e >> 1;
                const int co = r % kCoTile;
                const int tp = r / kCoTile;
                const int c = ci0 + 8 * half;
                uint4 v = zero4;
                if (co0 + co < cout && c < cin)
                    v = *reinterpret_cast<const uint4 *>(
                        w + (static_cast<long long>(tz * K * K + tp) * cout + co0 + co) * cin + c);
                *reinterpret_cast<uint4 *>(&ws[tp][co][8 * half]) = v;
            }
            __syncthreads();
#pragma unroll
            for (int tp = 0; tp < K * K; ++tp) {
                const int ty = tp / K, tx = tp % K;
                // A: rows g (voxel (2 warp, g)) and g + 8 (voxel (2 warp + 1, g))
                const __nv_bfloat16 *r0 = &xs[tz][2 * warp + ty][g + tx][0];
                const __nv_bfloat16 *r1 = &xs[tz][2 * warp + 1 + ty][g + tx][0];
                unsigned a[4];
                a[0] = *reinterpret_cast<const unsigned *>(r0 + 2 * tig);
                a[1] = *reinterpret_cast<const unsigned *>(r1 + 2 * tig);
                a[2] = *reinterpret_cast<const unsigned *>(r0 + 2 * tig + 8);
                a[3] = *reinterpret_cast<const unsigned *>(r1 + 2 * tig + 8);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const __nv_bfloat16 *wc = &ws[tp][8 * j + g][0];
                    const unsigned b0 = *reinterpret_cast<const unsigned *>(wc + 2 * tig);
                    const unsigned b1 = *reinterpret_cast<const unsigned *>(wc + 2 * tig + 8);
                    mma_bf16_16816(acc[j], a, b0, b1);
                }
            }
        }
        __syncthreads();  // xs consumed before the next chunk overwrites it
    }
    // epilogue: c0, c1 -> row g; c2, c3 -> row g + 8; columns 2 tig, 2 tig + 1
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int gy = ty0 + 2 * warp + half, gx = tx0 + g;
        TO *yo = y + (((static_cast<long long>(b) * n + z) * n + gy) * n + gx) * cout;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int co = co0 + 8 * j + 2 * tig + q;
                if (co >= cout) continue;
                float r = acc[j][2 * half + q] + (bias ? bias[co] : 0.f);
                if (act) r = r > 0.f ? r : kSlope * r;
                stf(yo + co, r);
            }
        }
    }
}

// Tensor-core weight gradient for bfloat16 inputs and output gradients:
// dw[tap][co][ci] = sum over voxels v of dy[v][co] x[v + tap][ci] is a GEMM
// with M = output channels, N = input channels and K = voxels.  One block of
// 4 warps per (tap, group of 64 output channels, group of 32 input channels,
// chunk of voxels); each stage stages 64 voxels of dy and of the shifted x
// transposed ([channel][voxel], 72-element rows: conflict-free fragment
// loads), then every warp runs 4 k-steps x 4 mma for its 16 output channels.
// Partial sums per chunk go to partials[chunk][tap][co][ci].
constexpr int kWgVox = 64;
constexpr int kWgRow = kWgVox + 8;

template <int K>
__global__ void __launch_bounds__(128) wgrad_mma_kernel(const __nv_bfloat16 *__restrict__ x,
                                                        const __nv_bfloat16 *__restrict__ dy,
                                                        float *__restrict__ partials, int batch, int n,
                                                        int cin, int cout, int chunk, int co_groups)
{
    constexpr int R = K / 2;
    constexpr int TAPS = K * K * K;
    __shared__ __align__(16) __nv_bfloat16 sa[64][kWgRow];  // dy^T: [co][voxel]
    __shared__ __align__(16) __nv_bfloat16 sb[32][kWgRow];  // x_tap^T: [ci][voxel]
    int bid = blockIdx.x;
    const int tap = bid % TAPS;
    bid /= TAPS;
    const int cog = bid % co_groups;
    const int cig = bid / co_groups;
    const int co0 = cog * 64, ci0 = cig * 32;
    const int dz = tap / (K * K) - R, dyo = (tap / K) % K - R, dx = tap % K - R;
    const long long total = static_cast<long long>(batch) * n * n * n;
    const long long v_begin = static_cast<long long>(blockIdx.y) * chunk;
    const long long v_end = v_begin + chunk < total ? v_begin + chunk : total;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int g = lane >> 2, tig = lane & 3;
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = 0.f;
    const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
    for (long long vb = v_begin; vb < v_end; vb += kWgVox) {
        // dy granules: 64 voxels x 8 granules of 8 output channels
        for (int e = t; e < kWgVox * 8; e += 128) {
            const int vi = e >> 3, gr = e & 7;
            const int co = co0 + 8 * gr;
            uint4 v = zero4;
            if (vb + vi < v_end && co < cout)
                v = *reinterpret_cast<const uint4 *>(dy + (vb + vi) * cout + co);
            const __nv_bfloat16 *h = reinterpret_cast<const __nv_bfloat16 *>(&v);
#pragma unroll
            for (int q = 0; q < 8; ++q) sa[8 * gr + q][vi] = h[q];
        }
        // x granules at the voxel shifted by the tap: 64 voxels x 4 granules
        for (int e = t; e < kWgVox * 4; e += 128) {
            const int vi = e >> 2, gr = e & 3;
            const int ci = ci0 + 8 * gr;
            uint4 v = zero4;
            if (vb + vi < v_end && ci < cin) {
                long long r = vb + vi;
                const int gx = static_cast<int>(r % n);
                r /= n;
                const int gy = static_cast<int>(r % n);
                r /= n;
                const int gz = static_cast<int>(r % n);
                const long long bb = r / n;
                const int sz = gz + dz, sy = gy + dyo, sx = gx + dx;
                if (sz >= 0 && sz < n && sy >= 0 && sy < n && sx >= 0 && sx < n)
                    v = *reinterpret_cast<const uint4 *>(x + (((bb * n + sz) * n + sy) * n + sx) * cin + ci);
            }
            const __nv_bfloat16 *h = reinterpret_cast<const __nv_bfloat16 *>(&v);
#pragma unroll
            for (int q = 0; q < 8; ++q) sb[8 * gr + q][vi] = h[q];
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < kWgVox / 16; ++ks) {
            const __nv_bfloat16 *r0 = &sa[16 * warp + g][16 * ks];
            const __nv_bfloat16 *r1 = &sa[16 * warp + g + 8][16 * ks];
            unsigned a[4];
            a[0] = *reinterpret_cast<const unsigned *>(r0 + 2 * tig);
            a[1] = *reinterpret_cast<const unsigned *>(r1 + 2 * tig);
            a[2] = *reinterpret_cast<const unsigned *>(r0 + 2 * tig + 8);
            a[3] = *reinterpret_cast<const unsigned *>(r1 + 2 * tig + 8);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const __nv_bfloat16 *bc = &sb[8 * j + g][16 * ks];
                const unsigned b0 = *reinterpret_cast<const unsigned *>(bc + 2 * tig);
                const unsigned b1 = *reinterpret_cast<const unsigned *>(bc + 2 * tig + 8);
                mma_bf16_16816(acc[j], a, b0, b1);
            }
        }
        __syncthreads();
    }
    float *out = partials + (static_cast<long long>(blockIdx.y) * TAPS + tap) * cout * cin;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int co = co0 + 16 * warp + g + (q >> 1) * 8;
            const int ci = ci0 + 8 * j + 2 * tig + (q & 1);
            if (co < cout && ci < cin) out[static_cast<long long>(co) * cin + ci] = acc[j][q];
        }
}

// Tensor-core weight gradient of a 3^3 convolution, all 27 taps per block:
// dw[tap][co][ci] = sum over voxels v of dy[v][co] x[v + tap][ci].  A block
// owns 16 output x 16 input channels and a run of 8 x 8 x 4 voxel tiles of
// the batch.  Per tile it stages dy (256 voxels) and the x halo (10 x 10 x 6
// voxels) once, unmodified (channels-last rows padded to 24 elements, which
// keeps the 8 rows of every ldmatrix conflict-free), and every tap reads the
// shifted x rows straight from the halo: ldmatrix takes one row address per
// thread, so the shift costs nothing.  The transposed 8 x 8 loads
// (ldmatrix .trans) turn the channels-last rows into the A = dy^T (co x
// voxels) and B = x_tap (voxels x ci) fragments of mma.m16n8k16.  Warp w
// accumulates taps w, w + 8, w + 16 (and w + 24 < 27) for both 8-channel
// halves of ci: 6 or 8 accumulator tiles.  The block's sums over its tiles go
// to partials[chunk][tap][co][ci], summed in chunk order afterwards.
// What bounds it: the fragment loads, 35 of 512 B per 16 voxels for 54 MMAs.
// The next tile's copies (cp.async) run under the current tile's MMAs, two
// blocks per SM; staging and multiplying in turn with three blocks took 78
// us instead of 68 us for 16 x 16 channels at 64^3 x 4, 28 instead of 23
// us for 64 x 64 at 16^3 x 4.
constexpr int kWtX = 8, kWtY = 8, kWtZ = 4;                  // voxel tile
constexpr int kWtHX = kWtX + 2, kWtHY = kWtY + 2, kWtHZ = kWtZ + 2;
constexpr int kWtVox = kWtX * kWtY * kWtZ;                   // 256
constexpr int kWtHalo = kWtHX * kWtHY * kWtHZ;               // 600
constexpr int kWtRow = 24;                                   // bf16 per staged row

__device__ __forceinline__ void ldsm_x4_trans(unsigned (&r)[4], const void *p)
{
    const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}

// Shared memory of one stage: the x halo, then the dy tile (rows of kWtRow).
constexpr unsigned kWtStage = (kWtHalo + kWtVox) * kWtRow * 2u;

__device__ __forceinline__ void wt_copy16(void *dst, const void *src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     static_cast<unsigned>(__cvta_generic_to_shared(dst))),
                 "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

__global__ void __launch_bounds__(256, 2) wgrad_taps_kernel(const __nv_bfloat16 *__restrict__ x,
                                                            const __nv_bfloat16 *__restrict__ dy,
                                                            float *__restrict__ partials, int n,
                                                            int cin, int cout, int tiles_per_sample,
                                                            int total_tiles, int tiles_per_block)
{
    extern __shared__ __align__(16) unsigned char wt_smem[];
    chain_wait();
    chain_release();
    typedef __nv_bfloat16 Row[kWtRow];
    const int ci_tiles = cin > 8 ? cin / 16 : 1;
    const int co0 = (blockIdx.x / ci_tiles) * 16, ci0 = (blockIdx.x % ci_tiles) * 16;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int ntap = warp + 24 < 27 ? 4 : 3;
    float acc[4][2][4], sum[4][2][4];  // of the tile (tensor cores), of the run
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = sum[i][j][q] = 0.f;
    const int tx_n = n / kWtX, ty_n = n / kWtY;
    // ldmatrix row of this thread: matrix j = lane / 8, row r = lane % 8
    const int mj = lane >> 3, mr = lane & 7;
    const int t_begin = blockIdx.y * tiles_per_block;
    const int t_end = min(t_begin + tiles_per_block, total_tiles);
    // copies of one tile into stage s (one group per thread)
    auto load = [&](int tile, int s) {
        Row *xs = reinterpret_cast<Row *>(wt_smem + s * kWtStage), *gs = xs + kWtHalo;
        const int b = tile / tiles_per_sample;
        int r = tile % tiles_per_sample;
        const int x0 = (r % tx_n) * kWtX;
        r /= tx_n;
        const int y0 = (r % ty_n) * kWtY;
        const int z0 = (r / ty_n) * kWtZ;
        const long long sample = static_cast<long long>(b) * n * n * n;
        // x halo: 600 voxels x 2 granules of 8 channels (zero outside the
        // grid and beyond cin)
        for (int e = t; e < kWtHalo * 2; e += 256) {
            const int half = e & 1, h = e >> 1;
            const int hx = h % kWtHX, hy = (h / kWtHX) % kWtHY, hz = h / (kWtHX * kWtHY);
            const int gx = x0 + hx - 1, gy = y0 + hy - 1, gz = z0 + hz - 1;
            const int c = ci0 + 8 * half;
            const bool in = gx >= 0 && gx < n && gy >= 0 && gy < n && gz >= 0 && gz < n && c < cin;
            const __nv_bfloat16 *p = x + (sample + (static_cast<long long>(gz) * n + gy) * n + gx) * cin + c;
            wt_copy16(&xs[h][8 * half], in ? p : x, in);
        }
        // dy tile: 256 voxels x 2 granules
        for (int e = t; e < kWtVox * 2; e += 256) {
            const int half = e & 1, vi = e >> 1;
            const int vx = vi % kWtX, vy = (vi / kWtX) % kWtY, vz = vi / (kWtX * kWtY);
            wt_copy16(&gs[vi][8 * half],
                      dy + (sample + (static_cast<long long>(z0 + vz) * n + y0 + vy) * n + x0 + vx) * cout + co0 + 8 * half,
                      true);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (t_begin < t_end) load(t_begin, 0);
    for (int tile = t_begin; tile < t_end; ++tile) {
        const int s = (tile - t_begin) & 1;
        if (tile + 1 < t_end) {
            load(tile + 1, s ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const Row *xs = reinterpret_cast<const Row *>(wt_smem + s * kWtStage), *gs = xs + kWtHalo;
#pragma unroll 2
        for (int ks = 0; ks < kWtVox / 16; ++ks) {
            // k-step ks: voxels 16 ks .. 16 ks + 15 = two x-rows (z, y), (z, y + 1)
            const int vz = ks / (kWtY / 2), vy = 2 * (ks % (kWtY / 2));
            unsigned a[4];
            // A = dy^T: matrices (v 0-7, co 0-7), (v 0-7, co 8-15), (v 8-15, co 0-7), (v 8-15, co 8-15)
            ldsm_x4_trans(a, &gs[16 * ks + 8 * (mj >> 1) + mr][8 * (mj & 1)]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i < ntap) {
                    const int tap = warp + 8 * i;
                    const int dz = tap / 9, dyy = (tap / 3) % 3, dx = tap % 3;
                    // B rows: voxel row (mj & 1) of the k-step, x = mr, shifted by the tap;
                    // matrices (v 0-7, ci 0-7), (v 8-15, ci 0-7), (v 0-7, ci 8-15), (v 8-15, ci 8-15)
                    const int h = ((vz + dz) * kWtHY + vy + (mj & 1) + dyy) * kWtHX + mr + dx;
                    unsigned bb[4];
                    ldsm_x4_trans(bb, &xs[h][8 * (mj >> 1)]);
                    mma_bf16_16816(acc[i][0], a, bb[0], bb[1]);
                    mma_bf16_16816(acc[i][1], a, bb[2], bb[3]);
                }
            }
        }
        // the tensor cores' additions truncate: their chains end with the tile
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    sum[i][j][q] += acc[i][j][q];
                    acc[i][j][q] = 0.f;
                }
        __syncthreads();  // the stage is free for the tile after the next
    }
    // acc[i][j]: rows co0 + g (+8), columns ci0 + 8 j + 2 tig (+1)
    const int g = lane >> 2, tig = lane & 3;
    float *out = partials + static_cast<long long>(blockIdx.y) * 27 * cout * cin;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (i >= ntap) continue;
        const int tap = warp + 8 * i;
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int co = co0 + g + 8 * (q >> 1);
                const int ci = ci0 + 8 * j + 2 * tig + (q & 1);
                if (ci < cin)
                    out[(static_cast<long long>(tap) * cout + co) * cin + ci] = sum[i][j][q];
            }
    }
}

// Weight gradient of a 1^3 convolution with few channels (the output head):
// dw[co][ci] = sum over voxels of dy[v][co] x[v][ci] on CUDA cores.  Each
// thread sums a strided set of voxels into CO x CI registers; the block
// reduces its threads in a fixed tree and writes partials[block][co][ci].
template <typename TI, int CO, int CI>
__global__ void __launch_bounds__(256) wgrad_small_kernel(const TI *__restrict__ x,
                                                          const float *__restrict__ dy,
                                                          float *__restrict__ partials, long long voxels,
                                                          int cin, int cout, long long chunk)
{
    float acc[CO][CI];
#pragma unroll
    for (int o = 0; o < CO; ++o)
#pragma unroll
        for (int i = 0; i < CI; ++i) acc[o][i] = 0.f;
    const long long v0 = blockIdx.x * chunk;
    const long long v1 = v0 + chunk < voxels ? v0 + chunk : voxels;
    for (long long v = v0 + threadIdx.x; v < v1; v += 256) {
        float xv[CI], gv[CO];
#pragma unroll
        for (int i = 0; i < CI; ++i) xv[i] = i < cin ? ldf(x + v * cin + i) : 0.f;
#pragma unroll
        for (int o = 0; o < CO; ++o) gv[o] = o < cout ? dy[v * cout + o] : 0.f;
#pragma unroll
        for (int o = 0; o < CO; ++o)
#pragma unroll
            for (int i = 0; i < CI; ++i) acc[o][i] = fmaf(gv[o], xv[i], acc[o][i]);
    }
    // fixed-order reduction: warp shuffle tree, then the 8 warps in order
    __shared__ float red[8][CO * CI];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 0; o < CO; ++o)
#pragma unroll
        for (int i = 0; i < CI; ++i) {
            float v = acc[o][i];
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
            if (lane == 0) red[warp][o * CI + i] = v;
        }
    __syncthreads();
    for (int k = threadIdx.x; k < CO * CI; k += 256) {
        const int o = k / CI, i = k % CI;
        if (o >= cout || i >= cin) continue;
        float v = 0.f;
        for (int w = 0; w < 8; ++w) v += red[w][k];
        partials[(static_cast<long long>(blockIdx.x) * cout + o) * cin + i] = v;
    }
}

__device__ __forceinline__ void ldsm_x4(unsigned (&r)[4], const void *p)
{
    const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}

template <typename T>
__device__ __forceinline__ void st2(T *p, float a, float b);
template <>
__device__ __forceinline__ void st2<float>(float *p, float a, float b)
{
    *reinterpret_cast<float2 *>(p) = make_float2(a, b);
}
template <>
__device__ __forceinline__ void st2<__nv_bfloat16>(__nv_bfloat16 *p, float a, float b)
{
    *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a, b);
}

// Tensor-core 3^3 convolution (implicit GEMM, mma.m16n8k16, FP32
// accumulation) over 8 x 8 x 4 voxel tiles: a block owns one tile of one
// sample and 8 NT output channels.  For every 16 input channels it stages
// the x halo (10 x 10 x 6 voxels) and the weights of all 27 taps for its
// channels (rows padded to 24 elements: conflict-free ldmatrix), then runs
// the 27 taps as shifted GEMMs: ldmatrix takes one row address per thread,
// so tap (dz, dy, dx) just reads the halo rows shifted by it.  Warp w owns
// voxel rows 32 w .. 32 w + 31 (two m16 tiles) and all NT n8 tiles.
// Dynamic shared memory: (600 + 27 * 8 NT) rows of 24 bfloat16.
template <int NT, typename TO>
__global__ void __launch_bounds__(256) conv3d_tc_kernel(const __nv_bfloat16 *__restrict__ x,
                                                        const __nv_bfloat16 *__restrict__ w,
                                                        const float *__restrict__ bias,
                                                        TO *__restrict__ y, int n, int cin, int cout,
                                                        int act)
{
    constexpr int CO = 8 * NT;
    extern __shared__ __align__(16) unsigned char conv_smem[];
    __nv_bfloat16(*xs)[kWtRow] = reinterpret_cast<__nv_bfloat16(*)[kWtRow]>(conv_smem);
    __nv_bfloat16(*ws)[kWtRow] = xs + kWtHalo;  // [tap * CO + co]
    const int tx_n = n / kWtX, ty_n = n / kWtY, tz_n = n / kWtZ;
    int r = blockIdx.x;
    const int x0 = (r % tx_n) * kWtX;
    r /= tx_n;
    const int y0 = (r % ty_n) * kWtY;
    r /= ty_n;
    const int z0 = (r % tz_n) * kWtZ;
    const int b = r / tz_n;
    const int co0 = blockIdx.y * CO;
    const long long sample = static_cast<long long>(b) * n * n * n;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int mj = lane >> 3, mr = lane & 7;
    float acc[2][NT][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
    const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
    for (int ci0 = 0; ci0 < cin; ci0 += 16) {
        for (int e = t; e < kWtHalo * 2; e += 256) {
            const int half = e & 1, h = e >> 1;
            const int hx = h % kWtHX, hy = (h / kWtHX) % kWtHY, hz = h / (kWtHX * kWtHY);
            const int gx = x0 + hx - 1, gy = y0 + hy - 1, gz = z0 + hz - 1;
            const int c = ci0 + 8 * half;
            uint4 v = zero4;
            if (gx >= 0 && gx < n && gy >= 0 && gy < n && gz >= 0 && gz < n && c < cin)
                v = *reinterpret_cast<const uint4 *>(
                    x + (sample + (static_cast<long long>(gz) * n + gy) * n + gx) * cin + c);
            *reinterpret_cast<uint4 *>(&xs[h][8 * half]) = v;
        }
        for (int e = t; e < 27 * CO * 2; e += 256) {
            const int half = e & 1, row = e >> 1;
            const int co = row % CO, tap = row / CO;
            const int c = ci0 + 8 * half;
            uint4 v = zero4;
            if (co0 + co < cout && c < cin)
                v = *reinterpret_cast<const uint4 *>(w + (static_cast<long long>(tap) * cout + co0 + co) * cin + c);
            *reinterpret_cast<uint4 *>(&ws[row][8 * half]) = v;
        }
        __syncthreads();
#pragma unroll 1
        for (int tap = 0; tap < 27; ++tap) {
            const int dz = tap / 9, dyy = (tap / 3) % 3, dx = tap % 3;
            unsigned a[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                // m16 tile 2 warp + i: voxel x-rows (vz, vy) and (vz, vy + 1)
                const int mt = 2 * warp + i;
                const int vz = mt / (kWtY / 2), vy = 2 * (mt % (kWtY / 2));
                const int h = ((vz + dz) * kWtHY + vy + (mj & 1) + dyy) * kWtHX + mr + dx;
                ldsm_x4(a[i], &xs[h][8 * (mj >> 1)]);
            }
#pragma unroll
            for (int j = 0; j < NT; j += 2) {
                // n8 tiles j, j + 1: matrices (co j, ci 0-7), (co j, ci 8-15), (co j+1, ...)
                unsigned bb[4];
                ldsm_x4(bb, &ws[tap * CO + 8 * (j + (mj >> 1)) + mr][8 * (mj & 1)]);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    mma_bf16_16816(acc[i][j], a[i], bb[0], bb[1]);
                    mma_bf16_16816(acc[i][j + 1], a[i], bb[2], bb[3]);
                }
            }
        }
        __syncthreads();
    }
    const int g = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int mt = 2 * warp + i;
        const int vz = mt / (kWtY / 2), vy = 2 * (mt % (kWtY / 2));
#pragma unroll
        for (int hrow = 0; hrow < 2; ++hrow) {
            const long long vox = sample + (static_cast<long long>(z0 + vz) * n + y0 + vy + hrow) * n + x0 + g;
            TO *yo = y + vox * cout;
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const int co = co0 + 8 * j + 2 * tig;
                if (co >= cout) continue;
                float v0 = acc[i][j][2 * hrow] + (bias ? bias[co] : 0.f);
                float v1 = acc[i][j][2 * hrow + 1] + (bias ? bias[co + 1] : 0.f);
                if (act) {
                    v0 = v0 > 0.f ? v0 : kSlope * v0;
                    v1 = v1 > 0.f ? v1 : kSlope * v1;
                }
                st2(yo + co, v0, v1);
            }
        }
    }
}

// A 1^3 convolution with few channels (the output head and its input
// gradient) on CUDA cores: one voxel per thread, the weights and bias in
// shared memory, y[v][co] = act(sum_ci x[v][ci] w[co][ci] + b[co]).
template <typename TI, typename TW, typename TO, int CI, int CO>
__global__ void __launch_bounds__(256) conv1x1_small_kernel(const TI *__restrict__ x, const TW *__restrict__ w,
                                                            const float *__restrict__ bias, TO *__restrict__ y,
                                                            long long voxels, int cin, int cout, int act)
{
    __shared__ float ws[CO][CI];
    __shared__ float bs[CO];
    for (int e = threadIdx.x; e < CO * CI; e += blockDim.x) {
        const int o = e / CI, i = e % CI;
        ws[o][i] = (o < cout && i < cin) ? ldf(w + o * cin + i) : 0.f;
    }
    for (int o = threadIdx.x; o < CO; o += blockDim.x) bs[o] = (bias && o < cout) ? bias[o] : 0.f;
    __syncthreads();
    for (long long v = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; v < voxels;
         v += static_cast<long long>(gridDim.x) * blockDim.x) {
        float xv[CI];
#pragma unroll
        for (int i = 0; i < CI; ++i) xv[i] = i < cin ? ldf(x + v * cin + i) : 0.f;
#pragma unroll
        for (int o = 0; o < CO; ++o) {
            if (o >= cout) break;
            float r = bs[o];
#pragma unroll
            for (int i = 0; i < CI; ++i) r = fmaf(xv[i], ws[o][i], r);
            if (act) r = r > 0.f ? r : kSlope * r;
            stf(y + v * cout + o, r);
        }
    }
}

// out = bfloat16(in)
__global__ void narrow_kernel(const float *__restrict__ in, __nv_bfloat16 *__restrict__ out, long long len)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        out[i] = __float2bfloat16_rn(in[i]);
}

// Weight gradient of a k^3 convolution: dw[tap][co][ci] = sum over samples
// and voxels of dy[v][co] * x[v + tap][ci].  One block per (tap, chunk of
// voxels); thread t owns input channel ci = t % cin and the output channels
// t / cin + j * (256 / cin), and sums its chunk in order (cin must divide
// 256; cin, cout <= 128).  partials[chunk][tap][co][ci] are summed in order
// afterwards.
template <typename TI, int K>
__global__ void __launch_bounds__(256) conv3d_wgrad_kernel(const TI *__restrict__ x,
                                                           const float *__restrict__ dy,
                                                           float *__restrict__ partials, int batch,
                                                           int n, int cin, int cout, int chunk)
{
    constexpr int R = K / 2;
    constexpr int VB = 32;  // voxels staged per round
    __shared__ float xs[VB][128];
    __shared__ float gs[VB][128];
    const int tap = blockIdx.x;
    const int dz = tap / (K * K) - R, dyo = (tap / K) % K - R, dx = tap % K - R;
    const long long total = static_cast<long long>(batch) * n * n * n;
    const long long v_begin = static_cast<long long>(blockIdx.y) * chunk;
    const long long v_end = v_begin + chunk < total ? v_begin + chunk : total;
    const int ci = threadIdx.x % cin;
    const int co0 = threadIdx.x / cin;
    const int step = 256 / cin;
    const int nco = (cout - co0 + step - 1) / step;  // output channels of this thread (<= 64)
    float acc[64];
#pragma unroll
    for (int k = 0; k < 64; ++k) acc[k] = 0.f;
    for (long long vb = v_begin; vb < v_end; vb += VB) {
        const int nv = static_cast<int>(v_end - vb < VB ? v_end - vb : VB);
        for (int e = threadIdx.x; e < VB * cin; e += 256) {
            const int c = e % cin, vi = e / cin;
            float val = 0.f;
            if (vi < nv) {
                long long v = vb + vi;
                const int gx = static_cast<int>(v % n);
                v /= n;
                const int gy = static_cast<int>(v % n);
                v /= n;
                const int gz = static_cast<int>(v % n);
                const long long bb = v / n;
                const int sz = gz + dz, sy = gy + dyo, sx = gx + dx;
                if (sz >= 0 && sz < n && sy >= 0 && sy < n && sx >= 0 && sx < n)
                    val = ldf(x + (((bb * n + sz) * n + sy) * n + sx) * cin + c);
            }
            xs[vi][c] = val;
        }
        for (int e = threadIdx.x; e < VB * cout; e += 256) {
            const int c = e % cout, vi = e / cout;
            gs[vi][c] = vi < nv ? dy[(vb + vi) * cout + c] : 0.f;
        }
        __syncthreads();
#pragma unroll 1
        for (int vi = 0; vi < nv; ++vi) {
            const float xv = xs[vi][ci];
#pragma unroll
            for (int k = 0; k < 64; ++k)
                if (k < nco) acc[k] = fmaf(gs[vi][co0 + k * step], xv, acc[k]);
        }
        __syncthreads();
    }
    float *out = partials + (static_cast<long long>(blockIdx.y) * gridDim.x + tap) * cout * cin;
#pragma unroll
    for (int k = 0; k < 64; ++k)
        if (k < nco) out[(co0 + k * step) * cin + ci] = acc[k];
}

// out[i] = sum over chunks of partials[chunk][i], in a fixed order: a block
// covers E consecutive elements (E = 32, or the power of two >= len when len
// is smaller) with 256 / E lanes of chunks; lane l adds chunks l, l + L, ...
// into four interleaved sums (chunk c goes to sum (c / L) % 4), and the lanes
// are then added in order.  Threads with consecutive elements read
// consecutive floats of one chunk.
__global__ void __launch_bounds__(256) sum_chunks_kernel(const float *__restrict__ partials,
                                                         float *__restrict__ out, long long len,
                                                         int chunks, int E)
{
    __shared__ float red[256];
    const int L = 256 / E;
    const int e = threadIdx.x % E, lane = threadIdx.x / E;
    const long long i = static_cast<long long>(blockIdx.x) * E + e;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    if (i < len) {
        int c = lane;
        for (; c + 3 * L < chunks; c += 4 * L) {
            s0 += partials[static_cast<long long>(c) * len + i];
            s1 += partials[static_cast<long long>(c + L) * len + i];
            s2 += partials[static_cast<long long>(c + 2 * L) * len + i];
            s3 += partials[static_cast<long long>(c + 3 * L) * len + i];
        }
        for (; c < chunks; c += L) s0 += partials[static_cast<long long>(c) * len + i];
    }
    red[threadIdx.x] = (s0 + s1) + (s2 + s3);
    __syncthreads();
    if (lane == 0 && i < len) {
        float tot = 0.f;
        for (int l = 0; l < L; ++l) tot += red[l * E + e];
        out[i] = tot;
    }
}

// Bias gradient partials: per block of voxels, the sum of dy over them.
// Thread t adds channel t % cout of voxels lane, lane + lanes, ... (lane =
// t / cout, lanes = 256 / cout; four interleaved sums), so a warp reads
// consecutive floats; the lanes are then summed in order.
__global__ void __launch_bounds__(256) bias_grad_kernel(const float *__restrict__ dy,
                                                        float *__restrict__ partials, long long voxels,
                                                        int cout, long long chunk)
{
    __shared__ float red[256];
    const int lanes = 256 / cout;
    const int c = threadIdx.x % cout, lane = threadIdx.x / cout;
    const long long v0 = static_cast<long long>(blockIdx.x) * chunk;
    const long long v1 = v0 + chunk < voxels ? v0 + chunk : voxels;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    if (lane < lanes) {
        long long v = v0 + lane;
        for (; v + 3 * lanes < v1; v += 4 * lanes) {
            s0 += dy[v * cout + c];
            s1 += dy[(v + lanes) * cout + c];
            s2 += dy[(v + 2 * lanes) * cout + c];
            s3 += dy[(v + 3 * lanes) * cout + c];
        }
        for (; v < v1; v += lanes) s0 += dy[v * cout + c];
    }
    red[threadIdx.x] = (s0 + s1) + (s2 + s3);
    __syncthreads();
    if (threadIdx.x < cout) {
        float tot = 0.f;
        for (int l = 0; l < lanes; ++l) tot += red[l * cout + threadIdx.x];
        partials[static_cast<long long>(blockIdx.x) * cout + threadIdx.x] = tot;
    }
}

// dy_pre = dy * slope where the (leaky ReLU) output was negative.
template <typename T>
__global__ void act_backward_kernel(const T *__restrict__ yout, float *__restrict__ dy, long long len)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        if (!(ldf(yout + i) > 0.f)) dy[i] *= kSlope;
}

// The leaky-ReLU backward (when act) fused with the bfloat16 copy of the
// resulting gradient: dy[i] *= slope where the output was not positive, then
// dyn[i] = bfloat16(dy[i]).  Four elements per thread (len % 4 == 0).
template <typename T>
__global__ void act_backward_narrow_kernel(const T *__restrict__ yout, float *__restrict__ dy,
                                           __nv_bfloat16 *__restrict__ dyn, long long len4, int act)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len4;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        float4 g = reinterpret_cast<float4 *>(dy)[i];
        if (act) {
            const long long e = 4 * i;
            if (!(ldf(yout + e) > 0.f)) g.x *= kSlope;
            if (!(ldf(yout + e + 1) > 0.f)) g.y *= kSlope;
            if (!(ldf(yout + e + 2) > 0.f)) g.z *= kSlope;
            if (!(ldf(yout + e + 3) > 0.f)) g.w *= kSlope;
            reinterpret_cast<float4 *>(dy)[i] = g;
        }
        __nv_bfloat162 lo = __floats2bfloat162_rn(g.x, g.y), hi = __floats2bfloat162_rn(g.z, g.w);
        uint2 pk;
        pk.x = *reinterpret_cast<unsigned *>(&lo);
        pk.y = *reinterpret_cast<unsigned *>(&hi);
        reinterpret_cast<uint2 *>(dyn)[i] = pk;
    }
}

// act_backward_narrow_kernel that also sums the bias gradient: with a grid
// of a fixed number of blocks the grid stride is a multiple of the cout / 4
// channel groups, so every thread sees the same four channels and sums them;
// each block adds its threads per channel group in thread order and writes
// partials[block][cout].
template <typename T>
__global__ void __launch_bounds__(256) act_backward_narrow_bias_kernel(const T *__restrict__ yout,
                                                                       float *__restrict__ dy,
                                                                       __nv_bfloat16 *__restrict__ dyn,
                                                                       long long len4, int act, int c4,
                                                                       float *__restrict__ partials)
{
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len4;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        float4 g = reinterpret_cast<float4 *>(dy)[i];
        if (act) {
            const long long e = 4 * i;
            if (!(ldf(yout + e) > 0.f)) g.x *= kSlope;
            if (!(ldf(yout + e + 1) > 0.f)) g.y *= kSlope;
            if (!(ldf(yout + e + 2) > 0.f)) g.z *= kSlope;
            if (!(ldf(yout + e + 3) > 0.f)) g.w *= kSlope;
            reinterpret_cast<float4 *>(dy)[i] = g;
        }
        __nv_bfloat162 lo = __floats2bfloat162_rn(g.x, g.y), hi = __floats2bfloat162_rn(g.z, g.w);
        uint2 pk;
        pk.x = *reinterpret_cast<unsigned *>(&lo);
        pk.y = *reinterpret_cast<unsigned *>(&hi);
        reinterpret_cast<uint2 *>(dyn)[i] = pk;
        acc.x += g.x;
        acc.y += g.y;
        acc.z += g.z;
        acc.w += g.w;
    }
    __shared__ float4 red[256];
    red[threadIdx.x] = acc;
    __syncthreads();
    if (static_cast<int>(threadIdx.x) < c4) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = threadIdx.x; k < 256; k += c4) {
            t.x += red[k].x;
            t.y += red[k].y;
            t.z += red[k].z;
            t.w += red[k].w;
        }
        float *o = partials + static_cast<long long>(blockIdx.x) * 4 * c4 + 4 * threadIdx.x;
        o[0] = t.x;
        o[1] = t.y;
        o[2] = t.z;
        o[3] = t.w;
    }
}

// wt[tap][ci][co] = w[K^3 - 1 - tap][co][ci] (weights of the transposed
// convolution, in the storage type).
template <typename TW>
__global__ void flip_transpose_kernel(const TW *__restrict__ w, TW *__restrict__ wt, int taps,
                                      int cout, int cin)
{
    const long long len = static_cast<long long>(taps) * cout * cin;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int co = static_cast<int>(i % cout);
        long long r = i / cout;
        const int ci = static_cast<int>(r % cin);
        const int tap = static_cast<int>(r / cin);
        wt[i] = w[(static_cast<long long>(taps - 1 - tap) * cout + co) * cin + ci];
    }
}

// ---------------------------------------------------------------- pooling, upsampling, skips

// Four consecutive channels as one access (c % 4 == 0).
struct F4 {
    float v[4];
};
template <typename T>
__device__ __forceinline__ F4 ld4(const T *p);
template <>
__device__ __forceinline__ F4 ld4<float>(const float *p)
{
    const float4 q = *reinterpret_cast<const float4 *>(p);
    return F4{{q.x, q.y, q.z, q.w}};
}
template <>
__device__ __forceinline__ F4 ld4<__nv_bfloat16>(const __nv_bfloat16 *p)
{
    const uint2 q = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&q.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&q.y));
    return F4{{a.x, a.y, b.x, b.y}};
}
template <typename T>
__device__ __forceinline__ void st4(T *p, const F4 &f);
template <>
__device__ __forceinline__ void st4<float>(float *p, const F4 &f)
{
    *reinterpret_cast<float4 *>(p) = make_float4(f.v[0], f.v[1], f.v[2], f.v[3]);
}
template <>
__device__ __forceinline__ void st4<__nv_bfloat16>(__nv_bfloat16 *p, const F4 &f)
{
    __nv_bfloat162 a = __floats2bfloat162_rn(f.v[0], f.v[1]), b = __floats2bfloat162_rn(f.v[2], f.v[3]);
    uint2 q;
    q.x = *reinterpret_cast<unsigned *>(&a);
    q.y = *reinterpret_cast<unsigned *>(&b);
    *reinterpret_cast<uint2 *>(p) = q;
}

// Element i of a [batch][n][n][n][c] tensor handled as (voxel, group of 4
// channels): i = voxel * c4 + q.  Voxel coordinates from the flat index.
// 32-bit divisions where they suffice: with 64-bit
// ones the kernels below were bound by them (up2_add at 64^3 x 4, 16
// channels: 29 us against 25, and 16 us with 16-byte accesses).
__device__ __forceinline__ void voxel_xyz(long long v, int n, int &x, int &y, int &z, long long &b)
{
    if (v < (1LL << 32)) {
        unsigned u = static_cast<unsigned>(v), d = static_cast<unsigned>(n);
        x = static_cast<int>(u % d);
        u /= d;
        y = static_cast<int>(u % d);
        u /= d;
        z = static_cast<int>(u % d);
        b = u / d;
        return;
    }
    x = static_cast<int>(v % n);
    v /= n;
    y = static_cast<int>(v % n);
    v /= n;
    z = static_cast<int>(v % n);
    b = v / n;
}

// i / d and i % d, in 32 bits where i fits.
__device__ __forceinline__ long long div_mod(long long i, int d, int &rem)
{
    if (i < (1LL << 32)) {
        const unsigned u = static_cast<unsigned>(i), q = u / static_cast<unsigned>(d);
        rem = static_cast<int>(u - q * static_cast<unsigned>(d));
        return q;
    }
    const long long q = i / d;
    rem = static_cast<int>(i - q * d);
    return q;
}

// G = 4 N consecutive channels in N 4-channel accesses (bf16: N = 2 makes one
// 16-byte access of each).
template <int N>
struct FN {
    F4 f[N];
};
template <typename T, int N>
__device__ __forceinline__ FN<N> ldn(const T *p)
{
    FN<N> r;
    if constexpr (std::is_same_v<T, __nv_bfloat16> && N == 2) {
        const uint4 u = *reinterpret_cast<const uint4 *>(p);
        const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w[k]));
            r.f[k / 2].v[2 * (k % 2)] = v.x;
            r.f[k / 2].v[2 * (k % 2) + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) r.f[k] = ld4(p + 4 * k);
    }
    return r;
}
template <typename T, int N>
__device__ __forceinline__ void stn(T *p, const FN<N> &r)
{
    if constexpr (std::is_same_v<T, __nv_bfloat16> && N == 2) {
        unsigned w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(r.f[k / 2].v[2 * (k % 2)], r.f[k / 2].v[2 * (k % 2) + 1]);
            w[k] = *reinterpret_cast<const unsigned *>(&h);
        }
        *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) st4(p + 4 * k, r.f[k]);
    }
}

// 2 x 2 x 2 average pooling, n -> n / 2 (channels in groups of 4 N)
template <typename T, int N>
__global__ void avgpool2_kernel(const T *__restrict__ x, T *__restrict__ y, int batch, int n, int c)
{
    chain_wait();
    chain_release();
    const int m = n / 2, c4 = c / (4 * N);
    const long long len = static_cast<long long>(batch) * m * m * m * c4;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        int q, ox, oy, oz;
        long long b;
        const long long vox = div_mod(i, c4, q);
        voxel_xyz(vox, m, ox, oy, oz, b);
        FN<N> s;
#pragma unroll
        for (int j = 0; j < 4 * N; ++j) s.f[j / 4].v[j % 4] = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int zz = 2 * oz + (k >> 2), yy = 2 * oy + ((k >> 1) & 1), xx = 2 * ox + (k & 1);
            const FN<N> a = ldn<T, N>(x + (((b * n + zz) * n + yy) * n + xx) * c + 4 * N * q);
#pragma unroll
            for (int j = 0; j < 4 * N; ++j) s.f[j / 4].v[j % 4] += a.f[j / 4].v[j % 4];
        }
#pragma unroll
        for (int j = 0; j < 4 * N; ++j) s.f[j / 4].v[j % 4] *= 0.125f;
        stn<T, N>(y + 4 * N * i, s);
    }
}

// gradient of avgpool2: dx = dy / 8 broadcast (FP32)
__global__ void avgpool2_backward_kernel(const float *__restrict__ dy, float *__restrict__ dx,
                                         int batch, int n, int c)
{
    const int m = n / 2, c4 = c / 4;
    const long long len = static_cast<long long>(batch) * n * n * n * c4;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        int q, xx, yy, zz;
        long long b;
        const long long vox = div_mod(i, c4, q);
        voxel_xyz(vox, n, xx, yy, zz, b);
        F4 a = ld4(dy + (((b * m + zz / 2) * m + yy / 2) * m + xx / 2) * c + 4 * q);
#pragma unroll
        for (int j = 0; j < 4; ++j) a.v[j] *= 0.125f;
        st4(dx + 4 * i, a);
    }
}

// nearest upsampling x2 (n -> 2n), plus an optional skip added: y = up(x) + s
template <typename T, int N>
__global__ void up2_add_kernel(const T *__restrict__ x, const T *__restrict__ skip, T *__restrict__ y,
                               int batch, int n, int c)
{
    chain_wait();
    chain_release();
    const int m = 2 * n, c4 = c / (4 * N);
    const long long len = static_cast<long long>(batch) * m * m * m * c4;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        int q, xx, yy, zz;
        long long b;
        const long long vox = div_mod(i, c4, q);
        voxel_xyz(vox, m, xx, yy, zz, b);
        FN<N> v = ldn<T, N>(x + (((b * n + zz / 2) * n + yy / 2) * n + xx / 2) * c + 4 * N * q);
        if (skip) {
            const FN<N> sk = ldn<T, N>(skip + 4 * N * i);
#pragma unroll
            for (int j = 0; j < 4 * N; ++j) v.f[j / 4].v[j % 4] += sk.f[j / 4].v[j % 4];
        }
        stn<T, N>(y + 4 * N * i, v);
    }
}

// gradient of nearest upsampling: dx = sum of the 8 children of dy (FP32)
__global__ void up2_backward_kernel(const float *__restrict__ dy, float *__restrict__ dx, int batch,
                                    int n, int c)
{
    const int m = 2 * n, c4 = c / 4;
    const long long len = static_cast<long long>(batch) * n * n * n * c4;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        int q, ox, oy, oz;
        long long b;
        const long long vox = div_mod(i, c4, q);
        voxel_xyz(vox, n, ox, oy, oz, b);
        F4 s{{0.f, 0.f, 0.f, 0.f}};
        for (int k = 0; k < 8; ++k) {
            const int zz = 2 * oz + (k >> 2), yy = 2 * oy + ((k >> 1) & 1), xx = 2 * ox + (k & 1);
            const F4 a = ld4(dy + (((b * m + zz) * m + yy) * m + xx) * c + 4 * q);
#pragma unroll
            for (int j = 0; j < 4; ++j) s.v[j] += a.v[j];
        }
        st4(dx + 4 * i, s);
    }
}

// a += b, four floats per thread (len % 4 == 0)
__global__ void add_inplace_kernel(float *__restrict__ a, const float *__restrict__ b, long long len4)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len4;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        float4 x = reinterpret_cast<float4 *>(a)[i];
        const float4 y = reinterpret_cast<const float4 *>(b)[i];
        x.x += y.x;
        x.y += y.y;
        x.z += y.z;
        x.w += y.w;
        reinterpret_cast<float4 *>(a)[i] = x;
    }
}

// ---------------------------------------------------------------- loss, optimiser, features

// Mean squared error: per-block partial sums of (y - t)^2 and dy = 2 (y - t) / len.
template <typename T>
__global__ void __launch_bounds__(256) mse_kernel(const T *__restrict__ yp, const float *__restrict__ tgt,
                                                  float *__restrict__ dy, double *__restrict__ partials,
                                                  long long len)
{
    __shared__ double sh[256];
    double s = 0.0;
    const float scale = 2.0f / static_cast<float>(len);
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < len; i += static_cast<long long>(gridDim.x) * 256) {
        const float d = ldf(yp + i) - tgt[i];
        s += static_cast<double>(d) * d;
        if (dy) dy[i] = scale * d;
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
}

__global__ void sum_doubles_kernel(const double *__restrict__ partials, int n, double scale,
                                   double *__restrict__ out)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double s = 0.0;
    for (int i = 0; i < n; ++i) s += partials[i];
    *out = s * scale;
}

// Adam (Kingma & Ba 2015) on FP32 master weights; the storage copy is
// refreshed from the master.  bc1 = 1 - beta1^t, bc2 = 1 - beta2^t.
template <typename TW>
__global__ void adam_kernel(float *__restrict__ master, TW *__restrict__ wstore,
                            const float *__restrict__ grad, float *__restrict__ m1,
                            float *__restrict__ m2, long long len, float lr, float beta1,
                            float beta2, float eps, float bc1, float bc2)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const float g = grad[i];
        const float a = beta1 * m1[i] + (1.f - beta1) * g;
        const float b = beta2 * m2[i] + (1.f - beta2) * g * g;
        m1[i] = a;
        m2[i] = b;
        const float mh = a / bc1, vh = b / bc2;
        const float wv = master[i] - lr * mh / (sqrtf(vh) + eps);
        master[i] = wv;
        stf(wstore + i, wv);
    }
}

template <typename TW>
__global__ void copy_to_store_kernel(const float *__restrict__ master, TW *__restrict__ wstore,
                                     long long len)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        stf(wstore + i, master[i]);
}

// Input features of one sample, channels-last [z][y][x][kFeatures]:
//  0: (log10 Ra - 4.5) / 1.5   1..3: one-hot wall type   4..6: x, y, z in [-1, 1]
//  7: the conduction profile 1/2 - Y (Y = (y + 1/2)/n)
template <typename T>
__global__ void features_kernel(const double *__restrict__ ra, const int *__restrict__ wall,
                                T *__restrict__ out, int batch, int n)
{
    // the per-sample feature (log10 Ra - 4.5) / 1.5, once per block (FP64 is slow)
    extern __shared__ float feat_ra[];
    chain_wait();
    chain_release();
    for (int b = threadIdx.x; b < batch; b += blockDim.x)
        feat_ra[b] = static_cast<float>((log10(ra[b]) - 4.5) / 1.5);
    __syncthreads();
    const long long vox = static_cast<long long>(n) * n * n;
    const long long len = batch * vox;
    const float h = 1.0f / n;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        int xx, yy, zz;
        long long b;
        voxel_xyz(i, n, xx, yy, zz, b);
        const int wl = wall[b];
        const F4 lo{{feat_ra[b], wl == 1 ? 1.f : 0.f, wl == 2 ? 1.f : 0.f, wl == 3 ? 1.f : 0.f}};
        const F4 hi{{2.f * (xx + 0.5f) * h - 1.f, 2.f * (yy + 0.5f) * h - 1.f, 2.f * (zz + 0.5f) * h - 1.f,
                     0.5f - (yy + 0.5f) * h}};
        st4(out + i * kFeatures, lo);
        st4(out + i * kFeatures + 4, hi);
    }
}

// Trilinear resampling of one channels-last sample [m^3][c] (cell-centred
// grids on the same unit cube) to planar fields: channel k (< 5) becomes
// plane[k] of out ([*][N^3], float), as scale[k] * value + offset[k].
struct ResampleMap {
    int plane[5];
    float scale[5], offset[5];
};

template <typename T>
__global__ void resample_kernel(const T *__restrict__ in, int m, int c, float *__restrict__ out, int N,
                                const ResampleMap map)
{
    const long long vox = static_cast<long long>(N) * N * N;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < vox;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int xx = static_cast<int>(i % N);
        const int yy = static_cast<int>((i / N) % N);
        const int zz = static_cast<int>(i / (static_cast<long long>(N) * N));
        // position in input cell units, clamped to the range of cell centres
        auto coord = [&](int k, int &i0, float &f) {
            float p = (k + 0.5f) * m / N - 0.5f;
            p = fminf(fmaxf(p, 0.f), static_cast<float>(m - 1));
            i0 = static_cast<int>(floorf(p));
            if (i0 > m - 2) i0 = m - 2 > 0 ? m - 2 : 0;
            f = p - i0;
            if (m == 1) f = 0.f;
        };
        int x0, y0, z0;
        float fx, fy, fz;
        coord(xx, x0, fx);
        coord(yy, y0, fy);
        coord(zz, z0, fz);
        const int x1 = m > 1 ? x0 + 1 : x0, y1 = m > 1 ? y0 + 1 : y0, z1 = m > 1 ? z0 + 1 : z0;
        for (int k = 0; k < c && k < 5; ++k) {
            auto at = [&](int z, int y, int x) {
                return ldf(in + ((static_cast<long long>(z) * m + y) * m + x) * c + k);
            };
            const float c00 = at(z0, y0, x0) * (1 - fx) + at(z0, y0, x1) * fx;
            const float c01 = at(z0, y1, x0) * (1 - fx) + at(z0, y1, x1) * fx;
            const float c10 = at(z1, y0, x0) * (1 - fx) + at(z1, y0, x1) * fx;
            const float c11 = at(z1, y1, x0) * (1 - fx) + at(z1, y1, x1) * fx;
            const float c0 = c00 * (1 - fy) + c01 * fy, c1 = c10 * (1 - fy) + c11 * fy;
            out[map.plane[k] * vox + i] = fmaf(map.scale[k], c0 * (1 - fz) + c1 * fz, map.offset[k]);
        }
    }
}

template <typename T>
__global__ void widen_kernel(const T *__restrict__ in, float *__restrict__ out, long long len)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        out[i] = ldf(in + i);
}

__global__ void fill_kernel(float *__restrict__ p, float v, long long len)
{
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < len;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        p[i] = v;
}

// Training target of one sample from planar fields, channels-last:
// out[v] = ((u_x, u_y, u_z) / u_c, theta, (rho - 1) / (3 u_c^2)).
__global__ void target_kernel(const float *__restrict__ u, const float *__restrict__ theta,
                              const float *__restrict__ rho, long long vox, float inv_uc,
                              float *__restrict__ out)
{
    const float inv_r = inv_uc * inv_uc / 3.0f;
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < vox;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        out[5 * i + 0] = u[i] * inv_uc;
        out[5 * i + 1] = u[vox + i] * inv_uc;
        out[5 * i + 2] = u[2 * vox + i] * inv_uc;
        out[5 * i + 3] = theta[i];
        out[5 * i + 4] = rho ? (rho[i] - 1.0f) * inv_r : 0.0f;
    }
}

// Elements per block of sum_chunks_kernel and its grid: one thread per
// element when there are few chunks, else 32 elements (fewer when len is
// smaller) with the remaining threads as lanes over the chunks.
int sum_width(long long len, int chunks)
{
    if (chunks <= 16) return 256;
    int e = 1;
    while (e < 32 && e < len) e *= 2;
    return e;
}
unsigned sum_blocks(long long len, int chunks)
{
    const int e = sum_width(len, chunks);
    return static_cast<unsigned>((len + e - 1) / e);
}

unsigned flat_blocks(long long len)
{
    long long b = (len + 255) / 256;
    if (b > 152 * 64) b = 152 * 64;
    if (b < 1) b = 1;
    return static_cast<unsigned>(b);
}

}  // namespace

// ---------------------------------------------------------------- launchers

// Streaming multiprocessors of the current device (152 on GB300), asked once
// per device.
int sm_count()
{
    static std::atomic<int> cached[64];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return 152;
    }
    if (dev >= 0 && dev < 64 && (sms = cached[dev].load(std::memory_order_relaxed)) > 0) return sms;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        return 152;
    }
    if (dev >= 0 && dev < 64) cached[dev].store(sms, std::memory_order_relaxed);
    return sms;
}

// 32 output channels per block, unless that leaves most SMs idle (the 8^3
// level: 32 blocks of 32 channels at batch 4): 16 per block doubles the
// blocks.  Every output accumulates the same MMAs in the same order either way.
bool mma_sync_takes_32(long long voxel_tiles, int cout)
{
    return cout % 32 == 0 && voxel_tiles * (cout / 32) >= 2LL * sm_count();
}

template <typename TI, typename TW, typename TO>
cudaError_t conv3d(const TI *x, const TW *w, const float *bias, TO *y, int batch, int n, int cin,
                   int cout, int k, int act, cudaStream_t s, bool chained)
{
    if (n % kTile != 0 || (k != 1 && k != 3)) return cudaErrorInvalidValue;
    if (k == 1 && cin <= 16 && cout <= 16 && (cin < 8 || cout < 8)) {
        const long long voxels = static_cast<long long>(batch) * n * n * n;
        conv1x1_small_kernel<TI, TW, TO, 16, 16><<<flat_blocks(voxels), 256, 0, s>>>(x, w, bias, y, voxels, cin,
                                                                                  cout, act);
        return cudaGetLastError();
    }
    const int tiles = n / kTile;
    dim3 grid(static_cast<unsigned>(tiles) * tiles * n * batch, (cout + kCoTile - 1) / kCoTile);
    if constexpr (std::is_same_v<TI, __nv_bfloat16> && std::is_same_v<TW, __nv_bfloat16>) {
        // tensor cores: channels are read in 16-byte granules of 8, so the
        // channel count and both base pointers must keep 16-byte alignment
        const bool aligned =
            ((reinterpret_cast<unsigned long long>(x) | reinterpret_cast<unsigned long long>(w)) & 15ull) == 0;
        UmmaPlan plan;
        if (k == 3 && conv3d_umma_takes(x, w, y, batch, n, cin, cout, static_cast<int>(sizeof(TO)), &plan))
            return conv3d_umma(plan, x, w, bias, y, batch, n, cin, cout, act, s, chained);
        if (k == 3 && aligned && (cin == 8 || cin % 16 == 0) && cout % 16 == 0 && n % kWtX == 0 &&
            n % kWtZ == 0) {
            const unsigned vtiles = static_cast<unsigned>(batch) * (n / kWtX) * (n / kWtY) * (n / kWtZ);
            // the dynamic shared memory exceeds the 48 KB default: opt in (per
            // call, so every device the kernel runs on gets the attribute)
            cudaError_t e;
            if (mma_sync_takes_32(vtiles, cout)) {
                const int smem = (kWtHalo + 27 * 32) * kWtRow * 2;
                e = cudaFuncSetAttribute(conv3d_tc_kernel<4, TO>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
                if (e != cudaSuccess) return e;
                conv3d_tc_kernel<4, TO><<<dim3(vtiles, cout / 32), 256, smem, s>>>(x, w, bias, y, n, cin, cout, act);
            } else {
                const int smem = (kWtHalo + 27 * 16) * kWtRow * 2;
                e = cudaFuncSetAttribute(conv3d_tc_kernel<2, TO>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
                if (e != cudaSuccess) return e;
                conv3d_tc_kernel<2, TO><<<dim3(vtiles, cout / 16), 256, smem, s>>>(x, w, bias, y, n, cin, cout, act);
            }
            return cudaGetLastError();
        }
        if (cin % 8 == 0 && aligned) {
            if (k == 3)
                conv3d_mma_kernel<3, TO><<<grid, 128, 0, s>>>(x, w, bias, y, n, cin, cout, act);
            else
                conv3d_mma_kernel<1, TO><<<grid, 128, 0, s>>>(x, w, bias, y, n, cin, cout, act);
            return cudaGetLastError();
        }
    }
    if (k == 3)
        conv3d_kernel<TI, TW, TO, 3><<<grid, 256, 0, s>>>(x, w, bias, y, n, cin, cout, act);
    else
        conv3d_kernel<TI, TW, TO, 1><<<grid, 256, 0, s>>>(x, w, bias, y, n, cin, cout, act);
    return cudaGetLastError();
}

int conv3d_wgrad_chunks(const void *x, const void *dy, int batch, int n, int cin, int cout)
{
    const unsigned long long bases = reinterpret_cast<unsigned long long>(x) | reinterpret_cast<unsigned long long>(dy);
    if ((bases & 15ull) != 0 || cout % 16 != 0 || (cin != 8 && cin % 16 != 0) || n % kWtX != 0) return 0;
    const long long blocks_per_chunk = static_cast<long long>(cout / 16) * (cin > 8 ? cin / 16 : 1);
    const long long tiles = static_cast<long long>(batch) * (n / kWtX) * (n / kWtY) * (n / kWtZ);
    // one wave of 2 resident blocks per SM: fewer chunks keep the final sum
    // over chunks short
    const long long most = std::min((152 * 2 + blocks_per_chunk - 1) / blocks_per_chunk, tiles);
    const long long per = (tiles + most - 1) / most;
    return static_cast<int>((tiles + per - 1) / per);
}

cudaError_t conv3d_wgrad_partials(const __nv_bfloat16 *x, const __nv_bfloat16 *dy, float *partials, int chunks, int batch,
                                  int n, int cin, int cout, cudaStream_t s)
{
    const int tiles_per_sample = (n / kWtX) * (n / kWtY) * (n / kWtZ);
    const long long tiles = static_cast<long long>(batch) * tiles_per_sample;
    const long long per = (tiles + chunks - 1) / chunks;
    const dim3 grid(static_cast<unsigned>(cout / 16 * (cin > 8 ? cin / 16 : 1)), static_cast<unsigned>(chunks));
    const cudaError_t e =
        cudaFuncSetAttribute(wgrad_taps_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kWtStage);
    if (e != cudaSuccess) return e;
    return launch_chained(wgrad_taps_kernel, grid, 256, 2 * kWtStage, s, true, x, dy, partials, n, cin, cout,
                          tiles_per_sample, static_cast<int>(tiles), static_cast<int>(per));
}

cudaError_t conv3d_wgrad_bf16(const __nv_bfloat16 *x, const __nv_bfloat16 *dy, float *dw, float *scratch,
                              size_t scratch_floats, int batch, int n, int cin, int cout, int k,
                              cudaStream_t s)
{
    const bool aligned =
        ((reinterpret_cast<unsigned long long>(x) | reinterpret_cast<unsigned long long>(dy)) & 15ull) == 0;
    if (cin % 8 != 0 || cout % 8 != 0 || !aligned || (k != 1 && k != 3)) return cudaErrorInvalidValue;
    int chunks3 = k == 3 ? conv3d_wgrad_chunks(x, dy, batch, n, cin, cout) : 0;
    if (chunks3 > 0) {
        const long long len = 27LL * cin * cout;
        while (chunks3 > 1 && static_cast<size_t>(chunks3 * len) > scratch_floats) chunks3 /= 2;
        if (static_cast<size_t>(chunks3 * len) > scratch_floats) return cudaErrorInvalidValue;
        cudaError_t e = conv3d_wgrad_partials(x, dy, scratch, chunks3, batch, n, cin, cout, s);
        if (e != cudaSuccess) return e;
        sum_chunks_kernel<<<sum_blocks(len, chunks3), 256, 0, s>>>(scratch, dw, len, chunks3, sum_width(len, chunks3));
        return cudaGetLastError();
    }
    const long long total = static_cast<long long>(batch) * n * n * n;
    const int taps = k * k * k;
    const int cogs = (cout + 63) / 64, cigs = (cin + 31) / 32;
    const long long pairs = static_cast<long long>(cin) * cout;
    const long long blocks_per_chunk = static_cast<long long>(taps) * cogs * cigs;
    long long chunks = (152 * 16 + blocks_per_chunk - 1) / blocks_per_chunk;
    const long long max_chunks = (total + kWgVox - 1) / kWgVox;
    if (chunks > max_chunks) chunks = max_chunks;
    while (chunks > 1 && static_cast<size_t>(chunks * taps * pairs) > scratch_floats) chunks /= 2;
    if (static_cast<size_t>(chunks * taps * pairs) > scratch_floats) return cudaErrorInvalidValue;
    // chunks of whole stages
    long long chunk = (total + chunks - 1) / chunks;
    chunk = (chunk + kWgVox - 1) / kWgVox * kWgVox;
    chunks = (total + chunk - 1) / chunk;
    dim3 grid(static_cast<unsigned>(blocks_per_chunk), static_cast<unsigned>(chunks));
    if (k == 3)
        wgrad_mma_kernel<3><<<grid, 128, 0, s>>>(x, dy, scratch, batch, n, cin, cout, static_cast<int>(chunk), cogs);
    else
        wgrad_mma_kernel<1><<<grid, 128, 0, s>>>(x, dy, scratch, batch, n, cin, cout, static_cast<int>(chunk), cogs);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long len = taps * pairs;
    sum_chunks_kernel<<<sum_blocks(len, static_cast<int>(chunks)), 256, 0, s>>>(
        scratch, dw, len, static_cast<int>(chunks), sum_width(len, static_cast<int>(chunks)));
    return cudaGetLastError();
}

template <typename TI>
cudaError_t conv3d_wgrad(const TI *x, const float *dy, float *dw, float *scratch,
                         size_t scratch_floats, int batch, int n, int cin, int cout, int k,
                         cudaStream_t s)
{
    const long long total = static_cast<long long>(batch) * n * n * n;
    if (k == 1 && cout <= 8 && cin <= 16) {
        long long blocks = 152 * 4;
        if (blocks > total) blocks = total;
        const long long pairs = static_cast<long long>(cin) * cout;
        while (blocks > 1 && static_cast<size_t>(blocks * pairs) > scratch_floats) blocks /= 2;
        const long long chunk = (total + blocks - 1) / blocks;
        blocks = (total + chunk - 1) / chunk;
        if (cout <= 5)
            wgrad_small_kernel<TI, 5, 16><<<static_cast<unsigned>(blocks), 256, 0, s>>>(x, dy, scratch, total, cin,
                                                                                        cout, chunk);
        else
            wgrad_small_kernel<TI, 8, 16><<<static_cast<unsigned>(blocks), 256, 0, s>>>(x, dy, scratch, total, cin,
                                                                                        cout, chunk);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        sum_chunks_kernel<<<sum_blocks(pairs, static_cast<int>(blocks)), 256, 0, s>>>(
        scratch, dw, pairs, static_cast<int>(blocks), sum_width(pairs, static_cast<int>(blocks)));
        return cudaGetLastError();
    }
    if (cin > 128 || cout > 128 || 256 % cin != 0) return cudaErrorInvalidValue;
    const int taps = k * k * k;
    const long long pairs = static_cast<long long>(cin) * cout;
    // chunks of voxels: enough blocks to fill the GPU, bounded by the scratch
    long long chunks = (152 * 8 + taps - 1) / taps;
    if (chunks > total) chunks = total;
    while (chunks > 1 && static_cast<size_t>(chunks * taps * pairs) > scratch_floats) chunks /= 2;
    if (static_cast<size_t>(chunks * taps * pairs) > scratch_floats) return cudaErrorInvalidValue;
    const int chunk = static_cast<int>((total + chunks - 1) / chunks);
    chunks = (total + chunk - 1) / chunk;
    dim3 grid(taps, static_cast<unsigned>(chunks));
    if (k == 3)
        conv3d_wgrad_kernel<TI, 3><<<grid, 256, 0, s>>>(x, dy, scratch, batch, n, cin, cout, chunk);
    else
        conv3d_wgrad_kernel<TI, 1><<<grid, 256, 0, s>>>(x, dy, scratch, batch, n, cin, cout, chunk);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long len = taps * pairs;
    sum_chunks_kernel<<<sum_blocks(len, static_cast<int>(chunks)), 256, 0, s>>>(
        scratch, dw, len, static_cast<int>(chunks), sum_width(len, static_cast<int>(chunks)));
    return cudaGetLastError();
}

cudaError_t bias_grad(const float *dy, float *db, float *scratch, size_t scratch_floats,
                      long long voxels, int cout, cudaStream_t s)
{
    if (cout < 1 || cout > 256) return cudaErrorInvalidValue;
    long long blocks = 152 * 2;
    if (blocks > voxels) blocks = voxels;
    while (blocks > 1 && static_cast<size_t>(blocks * cout) > scratch_floats) blocks /= 2;
    const long long chunk = (voxels + blocks - 1) / blocks;
    blocks = (voxels + chunk - 1) / chunk;
    bias_grad_kernel<<<static_cast<unsigned>(blocks), 256, 0, s>>>(dy, scratch, voxels, cout, chunk);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    sum_chunks_kernel<<<sum_blocks(cout, static_cast<int>(blocks)), 256, 0, s>>>(
        scratch, db, cout, static_cast<int>(blocks), sum_width(cout, static_cast<int>(blocks)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t act_backward_narrow(const T *yout, float *dy, __nv_bfloat16 *dyn, long long len, int act,
                                cudaStream_t s)
{
    const bool aligned =
        ((reinterpret_cast<unsigned long long>(dy) & 15ull) | (reinterpret_cast<unsigned long long>(dyn) & 7ull)) == 0;
    if (len % 4 != 0 || !aligned) return cudaErrorInvalidValue;
    act_backward_narrow_kernel<T><<<flat_blocks(len / 4), 256, 0, s>>>(yout, dy, dyn, len / 4, act);
    return cudaGetLastError();
}

template <typename T>
cudaError_t act_backward_narrow_bias(const T *yout, float *dy, __nv_bfloat16 *dyn, long long voxels, int cout,
                                     int act, float *db, float *scratch, size_t scratch_floats, cudaStream_t s)
{
    constexpr int kBlocks = 152 * 4;
    const bool aligned =
        ((reinterpret_cast<unsigned long long>(dy) & 15ull) | (reinterpret_cast<unsigned long long>(dyn) & 7ull)) == 0;
    if (cout % 4 != 0 || 256 % (cout / 4) != 0 || !aligned || static_cast<size_t>(kBlocks) * cout > scratch_floats)
        return cudaErrorInvalidValue;
    const long long len4 = voxels * cout / 4;
    act_backward_narrow_bias_kernel<T><<<kBlocks, 256, 0, s>>>(yout, dy, dyn, len4, act, cout / 4, scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    sum_chunks_kernel<<<sum_blocks(cout, kBlocks), 256, 0, s>>>(scratch, db, cout, kBlocks, sum_width(cout, kBlocks));
    return cudaGetLastError();
}

template <typename T>
cudaError_t act_backward(const T *yout, float *dy, long long len, cudaStream_t s)
{
    act_backward_kernel<T><<<flat_blocks(len), 256, 0, s>>>(yout, dy, len);
    return cudaGetLastError();
}

template <typename TW>
cudaError_t flip_transpose(const TW *w, TW *wt, int k, int cout, int cin, cudaStream_t s)
{
    const int taps = k * k * k;
    flip_transpose_kernel<TW><<<flat_blocks(static_cast<long long>(taps) * cout * cin), 256, 0, s>>>(
        w, wt, taps, cout, cin);
    return cudaGetLastError();
}

template <typename T>
cudaError_t avgpool2(const T *x, T *y, int batch, int n, int c, cudaStream_t s)
{
    if (c % 4 != 0) return cudaErrorInvalidValue;
    const long long len = static_cast<long long>(batch) * (n / 2) * (n / 2) * (n / 2) * (c / 4);
    if (std::is_same_v<T, __nv_bfloat16> && c % 8 == 0)
        return launch_chained(avgpool2_kernel<T, 2>, flat_blocks(len / 2), 256, 0, s, true, x, y, batch, n, c);
    return launch_chained(avgpool2_kernel<T, 1>, flat_blocks(len), 256, 0, s, true, x, y, batch, n, c);
}

cudaError_t avgpool2_backward(const float *dy, float *dx, int batch, int n, int c, cudaStream_t s)
{
    if (c % 4 != 0) return cudaErrorInvalidValue;
    const long long len = static_cast<long long>(batch) * n * n * n * (c / 4);
    avgpool2_backward_kernel<<<flat_blocks(len), 256, 0, s>>>(dy, dx, batch, n, c);
    return cudaGetLastError();
}

template <typename T>
cudaError_t up2_add(const T *x, const T *skip, T *y, int batch, int n, int c, cudaStream_t s)
{
    if (c % 4 != 0) return cudaErrorInvalidValue;
    const long long len = static_cast<long long>(batch) * 8LL * n * n * n * (c / 4);
    if (std::is_same_v<T, __nv_bfloat16> && c % 8 == 0)
        return launch_chained(up2_add_kernel<T, 2>, flat_blocks(len / 2), 256, 0, s, true, x, skip, y, batch, n, c);
    return launch_chained(up2_add_kernel<T, 1>, flat_blocks(len), 256, 0, s, true, x, skip, y, batch, n, c);
}

cudaError_t up2_backward(const float *dy, float *dx, int batch, int n, int c, cudaStream_t s)
{
    if (c % 4 != 0) return cudaErrorInvalidValue;
    const long long len = static_cast<long long>(batch) * n * n * n * (c / 4);
    up2_backward_kernel<<<flat_blocks(len), 256, 0, s>>>(dy, dx, batch, n, c);
    return cudaGetLastError();
}

cudaError_t add_inplace(float *a, const float *b, long long len, cudaStream_t s)
{
    if (len % 4 != 0) return cudaErrorInvalidValue;
    add_inplace_kernel<<<flat_blocks(len / 4), 256, 0, s>>>(a, b, len / 4);
    return cudaGetLastError();
}

template <typename T>
cudaError_t mse(const T *yp, const float *tgt, float *dy, double *partials, double *loss,
                long long len, cudaStream_t s)
{
    const unsigned blocks = 256;
    mse_kernel<T><<<blocks, 256, 0, s>>>(yp, tgt, dy, partials, len);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    sum_doubles_kernel<<<1, 32, 0, s>>>(partials, blocks, 1.0 / static_cast<double>(len), loss);
    return cudaGetLastError();
}

template <typename TW>
cudaError_t adam(float *master, TW *wstore, const float *grad, float *m1, float *m2, long long len,
                 float lr, float beta1, float beta2, float eps, int t, cudaStream_t s)
{
    const float bc1 = 1.f - powf(beta1, static_cast<float>(t));
    const float bc2 = 1.f - powf(beta2, static_cast<float>(t));
    adam_kernel<TW><<<flat_blocks(len), 256, 0, s>>>(master, wstore, grad, m1, m2, len, lr, beta1,
                                                     beta2, eps, bc1, bc2);
    return cudaGetLastError();
}

template <typename TW>
cudaError_t copy_to_store(const float *master, TW *wstore, long long len, cudaStream_t s)
{
    copy_to_store_kernel<TW><<<flat_blocks(len), 256, 0, s>>>(master, wstore, len);
    return cudaGetLastError();
}

template <typename T>
cudaError_t features(const double *ra, const int *wall, T *out, int batch, int n, cudaStream_t s)
{
    const size_t smem = static_cast<size_t>(batch) * sizeof(float);
    if (smem > 48 * 1024) return cudaErrorInvalidValue;
    // one wave of blocks: each pays the FP64 logarithm once
    const unsigned blocks = std::min(flat_blocks(static_cast<long long>(batch) * n * n * n), 152u * 8u);
    return launch_chained(features_kernel<T>, blocks, 256, smem, s, true, ra, wall, out, batch, n);
}

template <typename T>
cudaError_t resample(const T *in, int m, int c, float *out, int N, const int plane[5],
                     const float scale[5], const float offset[5], cudaStream_t s)
{
    ResampleMap map;
    for (int k = 0; k < 5; ++k) {
        map.plane[k] = plane[k];
        map.scale[k] = scale[k];
        map.offset[k] = offset[k];
    }
    resample_kernel<T><<<flat_blocks(static_cast<long long>(N) * N * N), 256, 0, s>>>(in, m, c, out, N, map);
    return cudaGetLastError();
}

template <typename T>
cudaError_t widen(const T *in, float *out, long long len, cudaStream_t s)
{
    widen_kernel<T><<<flat_blocks(len), 256, 0, s>>>(in, out, len);
    return cudaGetLastError();
}

cudaError_t narrow(const float *in, __nv_bfloat16 *out, long long len, cudaStream_t s)
{
    narrow_kernel<<<flat_blocks(len), 256, 0, s>>>(in, out, len);
    return cudaGetLastError();
}

cudaError_t fill(float *p, float v, long long len, cudaStream_t s)
{
    fill_kernel<<<flat_blocks(len), 256, 0, s>>>(p, v, len);
    return cudaGetLastError();
}

cudaError_t target_from_fields(const float *u, const float *theta, const float *rho, long long vox,
                               float inv_uc, float *out, cudaStream_t s)
{
    target_kernel<<<flat_blocks(vox), 256, 0, s>>>(u, theta, rho, vox, inv_uc, out);
    return cudaGetLastError();
}

// explicit instantiations for float and bfloat16 storage
#define DMRT_NN_INST(T)                                                                        \
    template cudaError_t conv3d<T, T, T>(const T *, const T *, const float *, T *, int, int, int, \
                                         int, int, int, cudaStream_t, bool);                    \
    template cudaError_t conv3d_wgrad<T>(const T *, const float *, float *, float *, size_t, int, \
                                         int, int, int, int, cudaStream_t);                     \
    template cudaError_t act_backward<T>(const T *, float *, long long, cudaStream_t);          \
    template cudaError_t act_backward_narrow<T>(const T *, float *, __nv_bfloat16 *, long long, int, \
                                                cudaStream_t);                                  \
    template cudaError_t act_backward_narrow_bias<T>(const T *, float *, __nv_bfloat16 *, long long, int, int, \
                                                     float *, float *, size_t, cudaStream_t);   \
    template cudaError_t flip_transpose<T>(const T *, T *, int, int, int, cudaStream_t);        \
    template cudaError_t avgpool2<T>(const T *, T *, int, int, int, cudaStream_t);              \
    template cudaError_t up2_add<T>(const T *, const T *, T *, int, int, int, cudaStream_t);    \
    template cudaError_t mse<T>(const T *, const float *, float *, double *, double *,          \
                                long long, cudaStream_t);                                       \
    template cudaError_t adam<T>(float *, T *, const float *, float *, float *, long long,      \
                                 float, float, float, float, int, cudaStream_t);                \
    template cudaError_t copy_to_store<T>(const float *, T *, long long, cudaStream_t);         \
    template cudaError_t features<T>(const double *, const int *, T *, int, int, cudaStream_t); \
    template cudaError_t resample<T>(const T *, int, int, float *, int, const int *, const float *, \
                                     const float *, cudaStream_t);                                 \
    template cudaError_t widen<T>(const T *, float *, long long, cudaStream_t);

DMRT_NN_INST(float)
DMRT_NN_INST(__nv_bfloat16)
#undef DMRT_NN_INST
// input gradients of bf16 layers on tensor cores: bf16 gradients, FP32 out
template cudaError_t conv3d<__nv_bfloat16, __nv_bfloat16, float>(const __nv_bfloat16 *,
                                                                const __nv_bfloat16 *, const float *,
                                                                float *, int, int, int, int, int, int,
                                                                cudaStream_t, bool);
// input gradients of bf16 layers: FP32 gradients through bf16 weights
template cudaError_t conv3d<float, __nv_bfloat16, float>(const float *, const __nv_bfloat16 *,
                                                        const float *, float *, int, int, int, int,
                                                        int, int, cudaStream_t, bool);

}  // namespace nn
}  // namespace lbm
