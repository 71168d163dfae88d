// conv_umma.cu -- 3^3 convolutions of the surrogate on the 5th-generation
// tensor cores (tcgen05.mma, accumulators in tensor memory).
//
// Both kernels are implicit GEMMs of M = 128 voxels x N = CO output channels
// x K = 16 input channels per instruction.  Operands sit in shared memory in
// the canonical K-major core-matrix layout (8 rows x 16 bytes): the 8 rows
// of an A core matrix are 8 consecutive x voxels of the staged halo, so tap
// (dz, dy, dx) is the same descriptor shifted by whole voxels; the weights
// are staged as [tap][kg][co] x 16 B (kg: group of 8 input channels).
//
// Roles of a CTA's nine warps: 0-3 epilogue (TMEM lane = voxel), 4 issues the
// MMAs, 5-8 load.  The loaders copy 16-byte pieces (8 channels of a voxel)
// with cp.async, zero-filled outside the grid, a few groups deep; the pieces
// of a voxel are neighbours in memory, so a warp's copies cover whole lines.
// (Tiled TMA copies of the same pieces were as fast, 42 against 43 us for
// the 64^3 x 4 layer of 16 channels, but need a tensor map per call.)
//
// What bounds them.  An MMA reads its 128 x 16 A tile (4 KB) and its B tile
// (CO x 32 B) from shared memory at 128 B per cycle, 32 + CO / 4 cycles, more
// than its arithmetic for CO <= 64.  Issuing one costs more than that if its
// descriptors are computed in a branch of one lane (see umma::mma_bf16): the
// deep layers took 1.4 to 2 times as long.
//
// Measured on GB300, kernel time per layer, before (a kernel that staged,
// multiplied and waited in turn; mma.sync at 8^3) and now:
//   16^3 x 4, 64 -> 64     29.1 -> 14.8 us     16^3 x 1, 64 -> 64    27.6 -> 8.9 us
//   8^3 x 4, 128 -> 128    44.4 -> 16.6 us     16^3 x 4, 32 -> 64    15.4 -> 11.2 us
//   64^3 x 2, 64 -> 64      561 -> 163 us      64^3 x 1, 128 -> 128  1057 -> 263 us
//   64^3 x 4, 16 -> 16     42.1 -> 37.6 us     32^3 x 4, 32 -> 32    20.9 -> 17.5 us
//   56^3 x 8, 16 -> 64      317 -> 232 us      (mma.sync before)
// (880 TFLOP/s at 64^3, 128 -> 128: 47 % of the measured bf16 rate.)  The wide
// kernel's outputs are bitwise those of the mma.sync kernel: the K = 16 slices
// are added in the same order, and tcgen05 and mma.sync add a slice alike.  The
// narrow one adds the slices of a tap one after another, which is the same
// for up to 16 input channels.
//
// Each wait is bounded; one that runs out sets *err, and the CTA drains its
// copies and MMAs before it releases its TMEM and exits.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "nn.h"
#include "umma.cuh"

namespace lbm {
namespace nn {

namespace {

constexpr float kSlope = 0.1f;  // leaky ReLU

constexpr int kThreads = 288;          // 4 epilogue warps, the MMA warp, 4 loader warps
constexpr int kLoaders = 128;
constexpr int kMmaWarp = 4;
constexpr unsigned kWaitPolls = 1u << 22;  // ~0.3 s of polling before giving up

// Tile of 8 x 16 voxels of a plane and its halo.
constexpr int kX = 8, kY = 16, kHX = kX + 2, kHY = kY + 2;
constexpr int kHaloRow = kHX * kHY;  // voxels of a halo plane

// Eight consecutive channels in one or two 16-byte stores (p 16-byte aligned).
__device__ __forceinline__ void store8(float *p, const float *v)
{
    reinterpret_cast<float4 *>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4 *>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void store8(__nv_bfloat16 *p, const float *v)
{
    uint4 u;
    __nv_bfloat162 h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    memcpy(&u, h, sizeof u);
    *reinterpret_cast<uint4 *>(p) = u;
}

// Sixteen consecutive channels (p 16-byte aligned; wide: 32-byte aligned).  A
// warp's lanes store to 32 different lines, and each store instruction visits
// every line: 32-byte stores make half the visits of 16-byte ones (48^3 x 6,
// 16 -> 32 channels, FP32 output: 47.4 -> 41.6 us).
__device__ __forceinline__ void store32(void *p, const uint4 &a, const uint4 &b)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z),
                 "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}
template <typename TO>
__device__ __forceinline__ void store16(TO *p, const float *v, bool wide)
{
    if (!wide) {
        store8(p, v);
        store8(p + 8, v + 8);
    } else if constexpr (sizeof(TO) == 4) {
        uint4 u[4];
        memcpy(u, v, sizeof u);
        store32(p, u[0], u[1]);
        store32(p + 8, u[2], u[3]);
    } else {
        __nv_bfloat162 h[8];
        uint4 u[2];
#pragma unroll
        for (int i = 0; i < 8; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        memcpy(u, h, sizeof u);
        store32(p, u[0], u[1]);
    }
}
template <typename TO>
__device__ __forceinline__ bool wide_stores(const TO *y)
{
    return (reinterpret_cast<unsigned long long>(y) & 31ull) == 0;
}

// Copy 16 bytes to shared memory, or zeros if !valid (src stays readable).
__device__ __forceinline__ void copy16(uint32_t dst, const void *src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(umma::smem_u32(bar)) : "memory");
}

// Bias and activation of 16 channels, in place.
__device__ __forceinline__ void finish16(float (&v)[16], const float *bias, int act)
{
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float a = v[i] + bias[i];
        v[i] = act && a <= 0.f ? kSlope * a : a;
    }
}

// ---------------------------------------------------------------- few channels

// cin <= 8 KG <= 32 and cout = CO <= 32: the planes of all 8 x 16 columns,
// column by column, are divided evenly among the resident CTAs (whole
// columns or runs of 16 planes left SMs with 3 or 4 CTAs: 43 against 38 us
// at 64^3 x 4); a CTA walks
// its range with the weights of all taps resident, one run of planes per
// column it meets.  Halo planes go through a ring of kRing slots (two more
// than a run's planes); the accumulator alternates over kAcc TMEM buffers,
// so copies, MMAs and epilogue of different planes overlap.  Per plane the
// MMAs run tap by tap, the K = 16 slices inside.
constexpr int kRing = 6;
constexpr int kAcc = 4;
constexpr int kMinRun = 2;
template <int KG>
constexpr unsigned plane_bytes() { return KG * kHaloRow * 16u; }
constexpr unsigned kHead = 512;  // mbarriers, TMEM slot, biases
template <int CO, int KG>
constexpr unsigned narrow_smem() { return kHead + kRing * plane_bytes<KG>() + 27u * KG * CO * 16u; }

// The run of planes from place g (column by column, n planes each) to the end
// of its column or of the range.
struct Run {
    int x0, y0, z_begin, z_end;
    long long b;
    __device__ __forceinline__ Run(long long g, long long g_end, int n)
    {
        long long r = g / n;
        z_begin = static_cast<int>(g - r * n);
        z_end = static_cast<int>(min(static_cast<long long>(n), z_begin + (g_end - g)));
        x0 = static_cast<int>(r % (n / kX)) * kX;
        r /= n / kX;
        y0 = static_cast<int>(r % (n / kY)) * kY;
        b = r / (n / kY);
    }
};

template <int CO, int KG, typename TO>
__global__ void __launch_bounds__(kThreads, KG == 2 ? 4 : 2)
    conv3d_umma_narrow_kernel(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ w,
                              const float *__restrict__ bias, TO *__restrict__ y, int n, int cin, int act,
                              long long planes, int *err)
{
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem);  // [kRing]: a slot holds its plane
    uint64_t *empty = full + kRing;                        // [kRing]: the MMAs that read it are done
    uint64_t *acc_full = empty + kRing;                    // [kAcc]: a plane's MMAs are done
    uint64_t *acc_empty = acc_full + kAcc;                 // [kAcc]: its accumulator was read
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acc_empty + kAcc);
    float *bs = reinterpret_cast<float *>(smem + 256);
    static_assert(8 * (2 * kRing + 2 * kAcc) + 4 <= 256 && 256 + 4 * CO <= kHead, "head layout");
    unsigned char *ring = smem + kHead;
    constexpr unsigned kPlane = plane_bytes<KG>();
    unsigned char *wsm = ring + kRing * kPlane;
    constexpr uint32_t kCols = kAcc * CO;
    const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
    const long long g_begin = planes * blockIdx.x / gridDim.x, g_end = planes * (blockIdx.x + 1) / gridDim.x;
    if (t == 0) {
        for (int k = 0; k < kRing; ++k) {
            umma::mbar_init(&full[k], kLoaders);
            umma::mbar_init(&empty[k], 1);
        }
        for (int k = 0; k < kAcc; ++k) {
            umma::mbar_init(&acc_full[k], 1);
            umma::mbar_init(&acc_empty[k], 4);  // one arrival per epilogue warp
        }
    }
    if (warp == 0) umma::tmem_alloc(tslot, kCols);
    if (t < CO) bs[t] = bias ? bias[t] : 0.f;
    // weights as [tap][kg][co] x 16 B, read in memory order, four loads in flight
    constexpr int kWeights = 27 * KG * CO;
#pragma unroll
    for (int e0 = 0; e0 < kWeights; e0 += 4 * kThreads) {
        uint4 v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = e0 + i * kThreads + t, kg = e % KG;
            v[i] = make_uint4(0u, 0u, 0u, 0u);
            if (e < kWeights && 8 * kg < cin)
                v[i] = *reinterpret_cast<const uint4 *>(w + static_cast<long long>(e / KG) * cin + 8 * kg);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = e0 + i * kThreads + t, kg = e % KG, co = e / KG % CO, tap = e / (KG * CO);
            if (e < kWeights) *reinterpret_cast<uint4 *>(wsm + ((tap * KG + kg) * CO + co) * 16) = v[i];
        }
    }
    umma::fence_proxy_async_smem();
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    chain_wait();
    chain_release();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);  // known to be uniform
    bool ok = true;
    if (warp > kMmaWarp) {
        // ---- loaders: thread's pieces (kg, hx, hy) of every plane, kg fastest
        const int lt = t - 32 * (kMmaWarp + 1);
        constexpr int kPieces = KG * kHaloRow, kPer = (kPieces + kLoaders - 1) / kLoaders;
        const uint32_t ring_s = umma::smem_u32(ring);
        const long long stride = static_cast<long long>(n) * n * cin;
        constexpr int kDepth = 3;  // planes of copies in flight
        static_assert(kRing >= kDepth + 2, "the planes that free a slot have been handed over");
        int k = 0, handed = 0;  // planes loaded and handed over
        auto hand_over = [&] {
            umma::fence_proxy_async_smem();
            arrive(&full[handed++ % kRing]);
        };
        for (long long g = g_begin; g < g_end && ok;) {
            const Run run(g, g_end, n);
            int src[kPer];  // element offset in the plane, -1: outside the grid
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int e = lt + i * kLoaders, kg = e % KG, h = e / KG;
                const int gx = run.x0 + h % kHX - 1, gy = run.y0 + h / kHX - 1;
                src[i] = gx >= 0 && gx < n && gy >= 0 && gy < n && 8 * kg < cin ? (gy * n + gx) * cin + 8 * kg : -1;
            }
            const __nv_bfloat16 *sample = x + run.b * n * stride;
            for (int p = run.z_begin - 1; p <= run.z_end; ++p, ++k) {
                const int slot = k % kRing;
                if (k >= kRing)
                    ok = umma::mbar_wait(&empty[slot], static_cast<uint32_t>(k / kRing - 1) & 1u, kWaitPolls);
                if (!ok) break;
                const bool in = p >= 0 && p < n;
                const __nv_bfloat16 *plane = sample + (in ? p : 0) * stride;
#pragma unroll
                for (int i = 0; i < kPer; ++i) {
                    const int e = lt + i * kLoaders, kg = e % KG, h = e / KG;
                    if (e < kPieces)
                        copy16(ring_s + slot * kPlane + (kg * kHaloRow + h) * 16, plane + max(src[i], 0),
                               in && src[i] >= 0);
                }
                copy_commit();
                if (k >= kDepth - 1) {
                    copy_wait<kDepth - 1>();
                    hand_over();
                }
            }
            g += run.z_end - run.z_begin;
        }
        copy_wait<0>();
        if (ok)
            while (handed < k) hand_over();
        else if (lt == 0) atomicExch(err, 1);
    } else if (warp == kMmaWarp) {
        {
            const uint32_t leader = umma::elect_one();
            constexpr uint32_t idesc = umma::idesc_bf16_f32(128, CO);
            const uint64_t a_base = umma::smem_desc(umma::smem_u32(ring), kHaloRow * 16, kHX * 16);
            const uint64_t b_base = umma::smem_desc(umma::smem_u32(wsm), CO * 16, 128);
            int j = 0, k = 0;  // planes computed; ring index of plane z - 1
            auto wait_slot = [&](int i) {
                return umma::mbar_wait(&full[i % kRing], static_cast<uint32_t>(i / kRing) & 1u, kWaitPolls);
            };
            for (long long g = g_begin; g < g_end && ok;) {
                const Run run(g, g_end, n);
                for (int z = run.z_begin; z < run.z_end; ++z, ++j, ++k) {
                    const int buf = j % kAcc;
                    // the accumulator's previous plane has been read out
                    if (j >= kAcc)
                        ok = umma::mbar_wait(&acc_empty[buf], static_cast<uint32_t>(j / kAcc - 1) & 1u, kWaitPolls);
                    ok = ok && wait_slot(k) && wait_slot(k + 1) && wait_slot(k + 2);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    umma::fence_after_sync();
                    uint64_t a_plane[3];
#pragma unroll
                    for (int dz = 0; dz < 3; ++dz)
                        a_plane[dz] = a_base + static_cast<uint64_t>((((k + dz) % kRing) * kPlane) >> 4);
                    const uint32_t dacc = tmem + buf * CO;
#pragma unroll
                    for (int tap = 0; tap < 27; ++tap) {
                        const int dz = tap / 9, dy = (tap / 3) % 3, dx = tap % 3;
#pragma unroll
                        for (int kc = 0; kc < KG / 2; ++kc) {
                            const uint64_t ad = a_plane[dz] + static_cast<uint64_t>(dy * kHX + dx + 2 * kc * kHaloRow);
                            const uint64_t bd = b_base + static_cast<uint64_t>((tap * KG + 2 * kc) * CO);
                            umma::mma_bf16(dacc, ad, bd, idesc, (tap > 0 || kc > 0) ? 1u : 0u, leader);
                        }
                    }
                    umma::commit(&acc_full[buf], leader);
                    umma::commit(&empty[k % kRing], leader);  // plane z - 1 is not read again
                }
                if (ok) {  // nor are the last two planes of the run
                    umma::commit(&empty[k % kRing], leader);
                    umma::commit(&empty[(k + 1) % kRing], leader);
                    k += 2;
                }
                g += run.z_end - run.z_begin;
            }
            if (!ok) {
                if (leader) atomicExch(err, 1);
                // MMAs still in flight end before TMEM is released
                if (j > 0) (void)umma::mbar_wait(&acc_full[(j - 1) % kAcc], static_cast<uint32_t>((j - 1) / kAcc) & 1u, kWaitPolls);
            }
        }
    } else {
        // ---- epilogue: warp w holds TMEM lanes 32 w .. 32 w + 31 (voxel m, x fastest)
        const int m = 32 * warp + lane;
        int j = 0;
        for (long long g = g_begin; g < g_end && ok;) {
            const Run run(g, g_end, n);
            TO *yo = y + (((run.b * n + run.z_begin) * n + run.y0 + m / kX) * n + run.x0 + m % kX) * CO;
            for (int z = run.z_begin; z < run.z_end; ++z, ++j, yo += static_cast<long long>(n) * n * CO) {
                const int buf = j % kAcc;
                ok = umma::mbar_wait(&acc_full[buf], static_cast<uint32_t>(j / kAcc) & 1u, kWaitPolls);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                umma::fence_after_sync();
#pragma unroll
                for (int c16 = 0; c16 < CO; c16 += 16) {
                    float v[16];
                    umma::ld_32x32b_x16(tmem + (static_cast<uint32_t>(32 * warp) << 16) + buf * CO + c16, v);
                    if (c16 + 16 == CO) {
                        // the accumulator may take another plane's MMAs
                        umma::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) arrive(&acc_empty[buf]);
                    }
                    finish16(v, bs + c16, act);
                    store16(yo + c16, v, wide_stores(y));
                }
            }
            g += run.z_end - run.z_begin;
        }
        if (!ok && lane == 0) atomicExch(err, 1);
    }
    umma::fence_before_sync();
    __syncthreads();
    if (warp == 0) umma::tmem_dealloc(tmem, kCols);
}

// ---------------------------------------------------------------- many channels

// Any cin (8, or a multiple of 16) and cout (a multiple of CO): a CTA owns R
// tiles of 128 voxels, stacked along z, times CO output channels, and runs
// over the input channels 16 at a time.  A stage holds 16 channels of the
// tiles' halo and the CO x 27 weights; kStages of them are in flight.  Every
// accumulator sums channel group by channel group and within a group tap by
// tap, whatever R, CO and the tile shape.
//  PAIR = false: a tile is 8 x 16 voxels of one plane (n a multiple of 16);
//    halo [kg][z R + 2][y 18][x 10] x 16 B.
//  PAIR = true: a tile is 8 x 8 voxels of two planes (n a multiple of 8).
//    The M rows are 16 rows of 8 voxels at one pitch, so each dy has a copy
//    of its own with exactly 8 y rows per plane:
//    halo [kg][dy 3][z 2 R + 2][y 8][x 10] x 16 B.
template <bool PAIR>
__host__ __device__ constexpr int halo_voxels(int R)
{
    return PAIR ? 3 * (2 * R + 2) * 8 * kHX : (R + 2) * kHaloRow;
}
template <int CO, bool PAIR>
__host__ __device__ constexpr unsigned stage_bytes(int R)
{
    return 32u * halo_voxels<PAIR>(R) + 27u * 2u * CO * 16u;
}
template <bool PAIR>
__host__ __device__ constexpr unsigned table_bytes(int R)
{
    return (4u * halo_voxels<PAIR>(R) + 15u) / 16u * 16u;
}
constexpr int kMaxStages = 4;

template <int CO, int R, bool PAIR, typename TO>
__global__ void __launch_bounds__(kThreads)
    conv3d_umma_wide_kernel(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ w,
                            const float *__restrict__ bias, TO *__restrict__ y, int n, int cin, int cout, int act,
                            int stages, int *err)
{
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem);  // [kMaxStages]
    uint64_t *empty = full + kMaxStages;                   // [kMaxStages]
    uint64_t *done = empty + kMaxStages;                   // all chunks are multiplied
    uint64_t *drained = done + 1;                          // after a failed wait: the MMAs in flight have ended
    uint32_t *tslot = reinterpret_cast<uint32_t *>(drained + 1);
    float *bs = reinterpret_cast<float *>(smem + 128);
    static_assert(8 * (2 * kMaxStages + 2) + 4 <= 128 && 128 + 4 * CO <= kHead, "head layout");
    constexpr int kVoxels = halo_voxels<PAIR>(R);
    int *offsets = reinterpret_cast<int *>(smem + kHead);  // [voxels]: element offset in the sample, -1 outside
    unsigned char *buf = smem + kHead + table_bytes<PAIR>(R);
    constexpr unsigned kStage = stage_bytes<CO, PAIR>(R);
    const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
    constexpr int TY = PAIR ? 8 : 16, TZ = PAIR ? 2 : 1;
    const int tx_n = n / kX, ty_n = n / TY, tz_n = n / (TZ * R);
    int r = blockIdx.x;
    const int x0 = (r % tx_n) * kX;
    r /= tx_n;
    const int y0 = (r % ty_n) * TY;
    r /= ty_n;
    const int z0 = (r % tz_n) * TZ * R;
    const int b = r / tz_n;
    const int co0 = blockIdx.y * CO;
    const long long sample = static_cast<long long>(b) * n * n * n;
    const int chunks = (cin + 15) / 16;
    constexpr uint32_t kCols = R * CO < 32 ? 32 : R * CO;
    if (t == 0) {
        for (int k = 0; k < kMaxStages; ++k) {
            umma::mbar_init(&full[k], kLoaders);
            umma::mbar_init(&empty[k], 1);
        }
        umma::mbar_init(done, 1);
        umma::mbar_init(drained, 1);
    }
    if (warp == 0) umma::tmem_alloc(tslot, kCols);
    if (t < CO) bs[t] = bias ? bias[co0 + t] : 0.f;
    for (int h = t; h < kVoxels; h += kThreads) {
        int gx = x0 + h % kHX - 1, gy, gz;
        if constexpr (PAIR) {
            const int rows = h / kHX, planes = 2 * R + 2;
            gy = y0 + rows % 8 + rows / (8 * planes) - 1;
            gz = z0 + rows / 8 % planes - 1;
        } else {
            gy = y0 + h / kHX % kHY - 1;
            gz = z0 + h / kHaloRow - 1;
        }
        const bool in = gx >= 0 && gx < n && gy >= 0 && gy < n && gz >= 0 && gz < n;
        offsets[h] = in ? ((gz * n + gy) * n + gx) * cin : -1;
    }
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    chain_wait();
    chain_release();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);  // known to be uniform
    bool ok = true;
    if (warp > kMmaWarp) {
        // ---- loaders: a stage is one group of copies per thread
        const int lt = t - 32 * (kMmaWarp + 1);
        const __nv_bfloat16 *xs = x + sample * cin;
        auto landed = [&](int c) {
            umma::fence_proxy_async_smem();
            arrive(&full[c % stages]);
        };
        int c = 0;
        for (; c < chunks; ++c) {
            const int s = c % stages;
            // with two stages the MMAs that free this one wait for the other
            if (c >= 2 && stages == 2) {
                copy_wait<0>();
                landed(c - 1);
            }
            if (c >= stages) ok = umma::mbar_wait(&empty[s], static_cast<uint32_t>(c / stages - 1) & 1u, kWaitPolls);
            if (!ok) break;
            const uint32_t hs = umma::smem_u32(buf + s * kStage);
            const int ci0 = 16 * c;
            const bool two = ci0 + 8 < cin;  // cin = 8 fills only the first group
#pragma unroll 4
            for (int e = lt; e < 2 * kVoxels; e += kLoaders) {
                const int kg = e & 1, h = e >> 1, off = offsets[h];
                copy16(hs + (kg * kVoxels + h) * 16, xs + max(off, 0) + (kg && two ? ci0 + 8 : ci0), off >= 0 && (!kg || two));
            }
            const uint32_t ws = hs + 32u * kVoxels;
#pragma unroll 4
            for (int e = lt; e < 27 * 2 * CO; e += kLoaders) {
                const int kg = e & 1, co = (e >> 1) % CO, tap = e / (2 * CO);
                copy16(ws + ((tap * 2 + kg) * CO + co) * 16,
                       w + (static_cast<long long>(tap) * cout + co0 + co) * cin + (kg && two ? ci0 + 8 : ci0), !kg || two);
            }
            copy_commit();
            if (c == 1 || (c >= 2 && stages > 2)) {
                copy_wait<1>();
                landed(c - 1);
            }
        }
        copy_wait<0>();
        if (ok) landed(c - 1);
        else if (lt == 0) atomicExch(err, 1);
    } else if (warp == kMmaWarp) {
        const uint32_t leader = umma::elect_one();
        constexpr uint32_t idesc = umma::idesc_bf16_f32(128, CO);
        bool issued = false;
        for (int c = 0; c < chunks; ++c) {
            const int s = c % stages;
            ok = umma::mbar_wait(&full[s], static_cast<uint32_t>(c / stages) & 1u, kWaitPolls);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            umma::fence_after_sync();
            const uint32_t hs = umma::smem_u32(buf + s * kStage);
            const uint64_t a_base = umma::smem_desc(hs, kVoxels * 16, kHX * 16);
            const uint64_t b_base = umma::smem_desc(hs + 32u * kVoxels, CO * 16, 128);
#pragma unroll
            for (int tap = 0; tap < 27; ++tap) {
                const int dz = tap / 9, dy = (tap / 3) % 3, dx = tap % 3;
                // different accumulators follow one another
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int row = PAIR ? (dy * (2 * R + 2) + 2 * i + dz) * 8 : (i + dz) * kHY + dy;
                    umma::mma_bf16(tmem + i * CO, a_base + static_cast<uint64_t>(row * kHX + dx),
                                   b_base + static_cast<uint64_t>(tap * 2 * CO), idesc, (c > 0 || tap > 0) ? 1u : 0u,
                                   leader);
                }
            }
            umma::commit(c + 1 < chunks ? &empty[s] : done, leader);
            issued = true;
        }
        if (!ok) {
            if (leader) atomicExch(err, 1);
            // MMAs still in flight end before TMEM is released (`done` stays
            // open: the epilogue's wait runs out too and nothing is stored)
            if (issued) {
                umma::commit(drained, leader);
                (void)umma::mbar_wait(drained, 0, kWaitPolls);
            }
        }
    } else {
        // ---- epilogue
        ok = umma::mbar_wait(done, 0, kWaitPolls);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
            umma::fence_after_sync();
            const int m = 32 * warp + lane;
            for (int i = 0; i < R; ++i) {
                const int yy = y0 + (PAIR ? m / kX % 8 : m / kX), zz = z0 + TZ * i + (PAIR ? m / 64 : 0);
                TO *yo = y + (sample + (static_cast<long long>(zz) * n + yy) * n + x0 + m % kX) * cout + co0;
#pragma unroll
                for (int c16 = 0; c16 < CO; c16 += 16) {
                    float v[16];
                    umma::ld_32x32b_x16(tmem + (static_cast<uint32_t>(32 * warp) << 16) + i * CO + c16, v);
                    finish16(v, bs + c16, act);
                    store16(yo + c16, v, wide_stores(y));
                }
            }
        } else if (lane == 0) {
            atomicExch(err, 1);
        }
    }
    umma::fence_before_sync();
    __syncthreads();
    if (warp == 0) umma::tmem_dealloc(tmem, kCols);
}

// ---------------------------------------------------------------- launch

// Device word: not zero once a tcgen05 convolution's wait has run out.
__device__ int g_umma_err;

int *umma_error_word()
{
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_umma_err) != cudaSuccess) return nullptr;
    return static_cast<int *>(p);
}

constexpr unsigned kSmemPerCta = 227u * 1024u, kSmemPerSm = 228u * 1024u;

template <int CO, int KG, typename TO>
cudaError_t launch_narrow(const __nv_bfloat16 *x, const __nv_bfloat16 *w, const float *bias, TO *y, int batch, int n,
                          int cin, int act, int *err, cudaStream_t s, bool chained)
{
    constexpr unsigned smem = narrow_smem<CO, KG>();
    auto kernel = conv3d_umma_narrow_kernel<CO, KG, TO>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    // resident CTAs per SM: shared memory (and 1 KB the runtime reserves per
    // CTA), TMEM columns, the launch bounds
    const int per_sm = std::min({KG == 2 ? 4 : 2, static_cast<int>(kSmemPerSm / (smem + 1024u)), 512 / (kAcc * CO)});
    // every resident CTA takes an equal share, of at least kMinRun planes (a
    // run loads two planes more than it computes; runs of at least 4 left SMs
    // idle: 32^3, 32 -> 32 channels 14.5 -> 12.4 us back to back)
    const long long planes = static_cast<long long>(batch) * (n / kX) * (n / kY) * n;
    const long long ctas = std::min<long long>(std::max(1, per_sm) * sm_count(), (planes + kMinRun - 1) / kMinRun);
    return launch_chained(kernel, static_cast<unsigned>(ctas), kThreads, smem, s, chained, x, w, bias, y, n, cin, act,
                          planes, err);
}

// The time of a layer: CTAs run in rounds of as many as an SM holds.  A round
// takes the set-up, R epilogue tiles in sequence and the chunks' MMAs (an M =
// 128, K = 16 MMA about 32 + CO / 4 cycles: its operands come from shared
// memory at 128 B per cycle); every CTA of the busiest SM takes the copies of
// its chunks (29 KB per us and SM; with 8 input channels half of a stage is
// only zeroed) and the stores of its output.  Fitted to 2400 timings (n 8 to
// 64, 1 to 8 samples, 8 to 128 channels on either side): half of them are
// within 6 %, nine in ten within 14 %.
template <int CO, int R, bool PAIR>
void consider(UmmaPlan &best, long long tiles, int nz, int cin, int cout, int out_bytes, int sms)
{
    if (cout % CO != 0 || nz % R != 0) return;
    const int chunks = (cin + 15) / 16;
    constexpr unsigned kFixed = kHead + table_bytes<PAIR>(R), kStage = stage_bytes<CO, PAIR>(R);
    int stages = std::min(chunks, kMaxStages);
    while (stages > 1 && kFixed + stages * kStage > kSmemPerCta) --stages;
    if (kFixed + stages * kStage > kSmemPerCta || (stages < 2 && chunks > 1)) return;
    const int per_sm = std::min({static_cast<int>(kSmemPerSm / (kFixed + stages * kStage + 1024u)),
                                 512 / std::max(32, R * CO), 65536 / (kThreads * 64)});
    const long long per = (tiles / R * (cout / CO) + sms - 1) / sms;  // CTAs of the busiest SM
    const long long rounds = (per + per_sm - 1) / per_sm;
    const double mma = 27.0 * R * (32.0 + CO / 4) / 1900.0, kb = kStage / 1024.0 * (cin == 8 ? 0.4 : 1.0);
    const double us = 3.5 + rounds * (1.2 + 0.69 * R + 0.315 * chunks * mma) +
                      per * (0.0345 * chunks * kb + 0.59 * R * CO / 64.0 * (out_bytes / 2));
    if (best.co == 0 || us < best.us) best = {CO, R, stages, us};
}

template <bool PAIR>
UmmaPlan wide_shape(int batch, int n, int cin, int cout, int out_bytes)
{
    const int nz = PAIR ? n / 2 : n;
    const long long tiles = static_cast<long long>(batch) * (n / kX) * (n / (PAIR ? 8 : 16)) * nz;
    const int sms = sm_count();
    UmmaPlan sh;
    consider<64, 4, PAIR>(sh, tiles, nz, cin, cout, out_bytes, sms);
    consider<64, 1, PAIR>(sh, tiles, nz, cin, cout, out_bytes, sms);
    consider<32, 4, PAIR>(sh, tiles, nz, cin, cout, out_bytes, sms);
    consider<32, 1, PAIR>(sh, tiles, nz, cin, cout, out_bytes, sms);
    consider<16, 4, PAIR>(sh, tiles, nz, cin, cout, out_bytes, sms);
    consider<16, 1, PAIR>(sh, tiles, nz, cin, cout, out_bytes, sms);
    return sh;
}

template <int CO, int R, bool PAIR, typename TO>
cudaError_t launch_wide(const UmmaPlan &sh, long long tiles, const __nv_bfloat16 *x, const __nv_bfloat16 *w,
                        const float *bias, TO *y, int n, int cin, int cout, int act, int *err, cudaStream_t s,
                        bool chained)
{
    const unsigned smem = kHead + table_bytes<PAIR>(R) + sh.stages * stage_bytes<CO, PAIR>(R);
    auto kernel = conv3d_umma_wide_kernel<CO, R, PAIR, TO>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kernel, dim3(static_cast<unsigned>(tiles / R), cout / CO), kThreads, smem, s, chained, x, w, bias,
                          y, n, cin, cout, act, sh.stages, err);
}

template <bool PAIR, typename TO>
cudaError_t run_wide(const UmmaPlan &sh, const __nv_bfloat16 *x, const __nv_bfloat16 *w, const float *bias, TO *y, int batch, int n,
                     int cin, int cout, int act, int *err, cudaStream_t s, bool chained)
{
    const long long tiles = static_cast<long long>(batch) * (n / kX) * (n / (PAIR ? 8 : 16)) * (PAIR ? n / 2 : n);
    auto go = [&](auto co, auto r) {
        return launch_wide<decltype(co)::value, decltype(r)::value, PAIR, TO>(sh, tiles, x, w, bias, y, n, cin, cout, act,
                                                                              err, s, chained);
    };
    auto by_r = [&](auto co) {
        return sh.R == 4 ? go(co, std::integral_constant<int, 4>{}) : go(co, std::integral_constant<int, 1>{});
    };
    switch (sh.co) {
    case 64: return by_r(std::integral_constant<int, 64>{});
    case 32: return by_r(std::integral_constant<int, 32>{});
    case 16: return by_r(std::integral_constant<int, 16>{});
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

int tensor_core_errors(bool reset)
{
    int *p = umma_error_word();
    if (!p) return -1;
    int v = 0;
    if (cudaMemcpy(&v, p, sizeof v, cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    if (reset && cudaMemset(p, 0, sizeof v) != cudaSuccess) return -1;
    return v;
}

// On unless DMRT_NN_NO_TCGEN05 is set in the environment (read once).  A
// sample's element offsets are 32-bit; the tiles are a grid dimension.
// Where n is an odd multiple of 8, a tile of two planes stages its halo three
// times, and layers of few input channels, or of output channels that are
// not a multiple of 32, are faster on mma.sync, which gives the same bits:
// with FP32 output 24^3 x 8, 16 -> 16 18.6 us here and 12.8 there, 40^3 x 3, 16
// -> 16 25.0 and 20.6, but 24^3 x 8, 128 -> 128 224 and 375.  The mma.sync
// kernel's time is within 5 % of the fit below; the tcgen05 one is taken where
// it is estimated 4 % and (beyond the shortest) 1.5 us faster.  Of 353 layers
// none is then slower than on mma.sync by more than 2 %, and 13 would be
// faster here by 3 % or more.
bool conv3d_umma_takes(const void *x, const void *w, const void *y, int batch, int n, int cin, int cout, int out_bytes,
                       UmmaPlan *plan)
{
    static const bool on = std::getenv("DMRT_NN_NO_TCGEN05") == nullptr;
    const unsigned long long bases = reinterpret_cast<unsigned long long>(x) | reinterpret_cast<unsigned long long>(w) |
                                     reinterpret_cast<unsigned long long>(y);
    const long long vox = static_cast<long long>(n) * n * n;
    if (!(on && (bases & 15ull) == 0 && (cin == 8 || cin % 16 == 0) && cout % 16 == 0 && n % 8 == 0 &&
          vox * cin < (1LL << 31) && vox * batch / 128 < (1LL << 31) && cout / 16 < 65536))
        return false;
    if (n % kY == 0) {
        const bool narrow = cin <= 32 && (cout == 16 || cout == 32);
        if (!narrow) *plan = wide_shape<false>(batch, n, cin, cout, out_bytes);
        return true;
    }
    *plan = wide_shape<true>(batch, n, cin, cout, out_bytes);
    const double chunks = (cin + 15) / 16;
    const long long sms = sm_count(), blocks = vox * batch / 256 * (cout / 16);  // mma.sync blocks of 16 channels
    const double mma_sync = mma_sync_takes_32(vox * batch / 256, cout)
                                ? 4.4 + chunks * (2.1 + 3.9 * static_cast<double>((blocks / 2 + sms - 1) / sms))
                                : 3.6 + chunks * (2.3 + 2.64 * static_cast<double>((blocks + sms - 1) / sms));
    return 1.04 * plan->us + (mma_sync > 11.0 ? 1.5 : 0.0) <= mma_sync;
}

template <typename TO>
cudaError_t conv3d_umma(const UmmaPlan &plan, const __nv_bfloat16 *x, const __nv_bfloat16 *w, const float *bias, TO *y,
                        int batch, int n, int cin, int cout, int act, cudaStream_t s, bool chained)
{
    int *err = umma_error_word();
    if (!err) return cudaErrorInvalidValue;
    if (plan.co == 0) {
        if (cout == 16 && cin <= 16) return launch_narrow<16, 2, TO>(x, w, bias, y, batch, n, cin, act, err, s, chained);
        if (cout == 16) return launch_narrow<16, 4, TO>(x, w, bias, y, batch, n, cin, act, err, s, chained);
        if (cin <= 16) return launch_narrow<32, 2, TO>(x, w, bias, y, batch, n, cin, act, err, s, chained);
        return launch_narrow<32, 4, TO>(x, w, bias, y, batch, n, cin, act, err, s, chained);
    }
    if (n % kY == 0) return run_wide<false, TO>(plan, x, w, bias, y, batch, n, cin, cout, act, err, s, chained);
    return run_wide<true, TO>(plan, x, w, bias, y, batch, n, cin, cout, act, err, s, chained);
}

template cudaError_t conv3d_umma<float>(const UmmaPlan &, const __nv_bfloat16 *, const __nv_bfloat16 *, const float *,
                                        float *, int, int, int, int, int, cudaStream_t, bool);
template cudaError_t conv3d_umma<__nv_bfloat16>(const UmmaPlan &, const __nv_bfloat16 *, const __nv_bfloat16 *,
                                                const float *, __nv_bfloat16 *, int, int, int, int, int, cudaStream_t,
                                                bool);

}  // namespace nn
}  // namespace lbm
