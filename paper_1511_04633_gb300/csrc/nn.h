// nn.h -- launchers of the surrogate's kernels (nn.cu); see nn.cu for the
// layouts.  Every launcher returns the CUDA error of its launches.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace lbm {
namespace nn {

// The network's kernels follow one another with programmatic dependent
// launch: the next kernel's blocks start, and set up what does not depend on
// the one before (barriers, TMEM, weights), while that one drains.  A kernel
// launched so calls chain_wait() before it touches activations or gradients
// and chain_release() after it, never before: whatever the next kernel
// does ahead of its own wait then comes after the kernel before this one, and
// weights are always older than that.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool chained,
                                  A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Input features per voxel (see features_kernel).
constexpr int kFeatures = 8;

// y = act(conv_k(x, w) + bias), k in {1, 3}, n a multiple of 8; act: 0 none,
// 1 leaky ReLU (slope 0.1).  bias may be null.  bfloat16 x and w (cin a
// multiple of 8) run on tensor cores; other types on CUDA cores.  chained:
// w and bias are older than the kernel launched last on s (launch_chained).
template <typename TI, typename TW, typename TO>
cudaError_t conv3d(const TI *x, const TW *w, const float *bias, TO *y, int batch, int n, int cin,
                   int cout, int k, int act, cudaStream_t s, bool chained = false);

// Streaming multiprocessors of the current device (152 on GB300).
int sm_count();

// The mma.sync convolution: 32 output channels per block (else 16)?  Voxel
// tiles are of 8 x 8 x 4.
bool mma_sync_takes_32(long long voxel_tiles, int cout);

// The 3^3 convolutions of bfloat16 x and w on the tcgen05 tensor cores
// (conv_umma.cu): taken where the channel counts are multiples of 16 (cin
// also 8), n a multiple of 8 and the three arrays 16-byte aligned, if they
// are the faster ones; *plan then says how.
struct UmmaPlan {
    int co = 0, R = 1, stages = 1;  // the wide kernel's tile; co = 0: the narrow kernel
    double us = 0.0;                // estimated time
};
bool conv3d_umma_takes(const void *x, const void *w, const void *y, int batch, int n, int cin, int cout, int out_bytes,
                       UmmaPlan *plan);
template <typename TO>
cudaError_t conv3d_umma(const UmmaPlan &plan, const __nv_bfloat16 *x, const __nv_bfloat16 *w, const float *bias, TO *y,
                        int batch, int n, int cin, int cout, int act, cudaStream_t s, bool chained);

// dw (FP32, [tap][cout][cin]) of conv3d; scratch holds the per-chunk partials.
template <typename TI>
cudaError_t conv3d_wgrad(const TI *x, const float *dy, float *dw, float *scratch,
                         size_t scratch_floats, int batch, int n, int cin, int cout, int k,
                         cudaStream_t s);

// the same on tensor cores, with the output gradient in bfloat16; requires
// cin and cout multiples of 8 and 16-byte aligned x and dy
// (cudaErrorInvalidValue otherwise).
cudaError_t conv3d_wgrad_bf16(const __nv_bfloat16 *x, const __nv_bfloat16 *dy, float *dw, float *scratch,
                              size_t scratch_floats, int batch, int n, int cin, int cout, int k,
                              cudaStream_t s);

// Not zero if a bounded wait of a tcgen05 convolution has run out (that
// launch's output is incomplete); reset = true clears it.  -1 on a CUDA error.
int tensor_core_errors(bool reset);

cudaError_t bias_grad(const float *dy, float *db, float *scratch, size_t scratch_floats,
                      long long voxels, int cout, cudaStream_t s);

// dy *= slope where the leaky-ReLU output yout is not positive.
template <typename T>
cudaError_t act_backward(const T *yout, float *dy, long long len, cudaStream_t s);

// act_backward (if act) and then dyn = bfloat16(dy), in one pass; len % 4 == 0,
// dy 16-byte and dyn 8-byte aligned.
template <typename T>
cudaError_t act_backward_narrow(const T *yout, float *dy, __nv_bfloat16 *dyn, long long len, int act,
                                cudaStream_t s);

// act_backward_narrow over voxels x cout values plus the bias gradient db[co]
// = sum over voxels of dy[v][co], in a fixed order; cout % 4 == 0 and cout / 4
// dividing 256; `scratch` holds 608 * cout partial sums.
template <typename T>
cudaError_t act_backward_narrow_bias(const T *yout, float *dy, __nv_bfloat16 *dyn, long long voxels, int cout,
                                     int act, float *db, float *scratch, size_t scratch_floats, cudaStream_t s);

// ---- the fused backward pass of the bf16 network (nn_backward.cu)

constexpr int kGradBlocks = 152 * 4;  // blocks of grad_narrow: chunks of its bias sums
constexpr int kHeadBlocks = 152 * 2;  // blocks of head_backward
constexpr int kMaxSums = 40;

// Arrays whose per-chunk partial sums sum_all adds (and the loss).
struct SumArray {
    const float *partials;
    float *out;
    size_t stride;
    int len, chunks, width;
};
struct SumList {
    int count = 0;
    int first[kMaxSums + 1] = {0};  // first block of each array, then the number of blocks
    SumArray a[kMaxSums];
    const double *loss_partials = nullptr;
    double *loss = nullptr;
    int loss_parts = 0;
    double loss_scale = 1.0;
    void add(const float *partials, size_t stride, float *out, int len, int chunks);
};
cudaError_t sum_all(const SumList &list, cudaStream_t s);

// Where grad_narrow's gradient comes from.
enum class GradSource { kPlain, kUp2, kPool };
cudaError_t grad_narrow(GradSource src, const float *g, const float *h, const __nv_bfloat16 *yout, __nv_bfloat16 *dyn,
                        long long voxels, int n, int c, float *partials, cudaStream_t s);

// The 16 -> 5 output head (bf16 h and w; y bf16, or its value widened).
template <typename TO>
cudaError_t head_forward(const __nv_bfloat16 *h, const __nv_bfloat16 *w, const float *bias, TO *y, long long voxels,
                         cudaStream_t s);

// The 16 -> 5 output head's backward with the loss; adds its sums to `sums`.
size_t head_partial_floats();
cudaError_t head_backward(const __nv_bfloat16 *out, const float *target, const __nv_bfloat16 *h, const __nv_bfloat16 *w,
                          __nv_bfloat16 *dyn, long long voxels, float *partials, double *loss_partials, float *dw,
                          float *db, float *db_before, SumList &sums, cudaStream_t s);

// Layers whose weights flip_all transposes, w and wt at the same offsets.
constexpr int kMaxFlips = 16;
struct FlipList {
    int count = 0;
    int first[kMaxFlips + 1] = {0};  // first element of each layer, then their number
    long long offset[kMaxFlips];
    int cin[kMaxFlips], cout[kMaxFlips];
};
cudaError_t flip_all(const __nv_bfloat16 *w, __nv_bfloat16 *wt, const FlipList &list, cudaStream_t s);

// The weight gradient of a 3^3 convolution as `chunks` partial sums of
// [27][cout][cin], to be added by sum_all: conv3d_wgrad_chunks of them, 0
// where the shape does not take this path (then use conv3d_wgrad_bf16).
int conv3d_wgrad_chunks(const void *x, const void *dy, int batch, int n, int cin, int cout);
cudaError_t conv3d_wgrad_partials(const __nv_bfloat16 *x, const __nv_bfloat16 *dy, float *partials, int chunks, int batch,
                                  int n, int cin, int cout, cudaStream_t s);

// weights of the transposed convolution (input gradient = conv3d with them)
template <typename TW>
cudaError_t flip_transpose(const TW *w, TW *wt, int k, int cout, int cin, cudaStream_t s);

template <typename T>
cudaError_t avgpool2(const T *x, T *y, int batch, int n, int c, cudaStream_t s);
cudaError_t avgpool2_backward(const float *dy, float *dx, int batch, int n, int c, cudaStream_t s);
template <typename T>
cudaError_t up2_add(const T *x, const T *skip, T *y, int batch, int n, int c, cudaStream_t s);
cudaError_t up2_backward(const float *dy, float *dx, int batch, int n, int c, cudaStream_t s);
cudaError_t add_inplace(float *a, const float *b, long long len, cudaStream_t s);

// loss = mean((yp - tgt)^2) into *loss (device double); dy = d loss / d yp.
template <typename T>
cudaError_t mse(const T *yp, const float *tgt, float *dy, double *partials, double *loss,
                long long len, cudaStream_t s);

template <typename TW>
cudaError_t adam(float *master, TW *wstore, const float *grad, float *m1, float *m2, long long len,
                 float lr, float beta1, float beta2, float eps, int t, cudaStream_t s);
template <typename TW>
cudaError_t copy_to_store(const float *master, TW *wstore, long long len, cudaStream_t s);

template <typename T>
cudaError_t features(const double *ra, const int *wall, T *out, int batch, int n, cudaStream_t s);

// trilinear resampling of one channels-last sample [m^3][c] (c <= 5) to
// planar fields: channel k into plane[k] of out, as scale[k] * v + offset[k]
template <typename T>
cudaError_t resample(const T *in, int m, int c, float *out, int N, const int plane[5],
                     const float scale[5], const float offset[5], cudaStream_t s);

// out = bfloat16(in), rounded to nearest
cudaError_t narrow(const float *in, __nv_bfloat16 *out, long long len, cudaStream_t s);
// out = (float) in; p[0..len) = v; training target from planar fields
template <typename T>
cudaError_t widen(const T *in, float *out, long long len, cudaStream_t s);
cudaError_t fill(float *p, float v, long long len, cudaStream_t s);
cudaError_t target_from_fields(const float *u, const float *theta, const float *rho, long long vox,
                               float inv_uc, float *out, cudaStream_t s);

}  // namespace nn
}  // namespace lbm
