// step_split.cu -- the fused double-MRT time step (arXiv:1511.04633, Eqs.
// (14), (19), (29)) of one walled cavity with ODD rows, two cells per thread:
// the cells (x, y, z0) and (x, y, z0 + 1), z0 even.  The pairs of step_pair.cu
// need an even row length, for the aligned two-element accesses; here every
// value is loaded and stored on its own (a warp's accesses are runs of 32
// cells of a slab, whatever the row length), and only the collision is
// packed (collide_from<F2>), which is what bounds the one-cell kernels: they
// execute 685 instructions per 16-bit cell.  The two cells share their x and
// y faces, so most of the wall logic is shared too.  The values stored are
// bitwise those of step_kernel and step_inplace_kernel.
//
// Measured on GB300, per step, one cell per thread -> this kernel: 101 x 75 x
// 61 in place FP16 14.8 -> 11.4 us, two buffers BF16 13.6 -> 11.3, FP32 15.4
// -> 13.3; 255^3 BF16 419 -> 377 us (in place 404 -> 357), FP32 559 -> 557.
// It executes half the instructions but holds half the warps for the same
// cells, so it pays where those fill the SMs (step_split_pays): 69^3 BF16 11.8
// -> 8.6 us, 45^3 4.7 -> 3.9, but 47^3 4.7 -> 5.2.
//
// A slab's cells are numbered flat (c = y nx + x), 128 per block, so no lane
// idles at the end of a row; y = c / nx is a multiplication (RowDivisor).
#include "pair_body.cuh"
#include "residual.cuh"

namespace lbm {

namespace {

constexpr int kSplitThreads = 128;
constexpr int kSplitBlocks = 5;     // 96 registers, as the paired kernels
constexpr int kSplitBlocksRes = 4;

struct SplitCoords {
    unsigned c0, c1;  // cell indices; c1 = c0 where the slab has no partner
    bool two;         // the second cell exists
    bool valid;
    PairFaces faces;  // x and y faces of both cells; zlo of cell 0, zhi of the last cell
    float th_lin;
};

__device__ __forceinline__ SplitCoords split_coords(const StepGeometry &S, const RowDivisor &D)
{
    SplitCoords p;
    const unsigned nxy = static_cast<unsigned>(S.nx) * S.ny;
    const unsigned c = blockIdx.x * kSplitThreads + threadIdx.x;
    const int z0 = 2 * static_cast<int>(blockIdx.y);
    const unsigned y = D.divide(c), x = c - y * S.nx;
    p.valid = c < nxy;
    p.two = z0 + 1 < S.nz;
    p.c0 = static_cast<unsigned>(z0) * nxy + c;
    p.c1 = p.two ? p.c0 + nxy : p.c0;
    p.faces = {x == 0, x + 1 == static_cast<unsigned>(S.nx), y == 0, y + 1 == static_cast<unsigned>(S.ny), z0 == 0,
               z0 + 2 >= S.nz};
    p.th_lin = theta_linear(static_cast<int>(y), S.inv_ny);
    return p;
}

// Does link q of cell 0 / cell 1 enter (IN: pull) or leave (!IN: push)
// through a face?  Cell 1 never touches z = 0, and cell 0 touches z = nz - 1
// only where it has no partner.
template <int Q, bool IN>
__device__ __forceinline__ void split_outside(const SplitCoords &p, bool &o0, bool &o1)
{
    constexpr int s = IN ? 1 : -1;
    constexpr int ex = s * plane_ex<Q>(), ey = s * plane_ey<Q>(), ez = s * plane_ez<Q>();
    bool xy = false;
    if constexpr (ex == 1) xy = xy || p.faces.xlo;
    if constexpr (ex == -1) xy = xy || p.faces.xhi;
    if constexpr (ey == 1) xy = xy || p.faces.ylo;
    if constexpr (ey == -1) xy = xy || p.faces.yhi;
    o0 = o1 = xy;
    if constexpr (ez == 1) o0 = o0 || p.faces.zlo;
    if constexpr (ez == -1) {
        o0 = o0 || (p.faces.zhi && !p.two);
        o1 = o1 || p.faces.zhi;
    }
}

// Pull of both cells (pull_pair's rules, each value loaded on its own).
template <int WALL, typename T, typename Off>
__device__ __forceinline__ void pull_split(const T *B0, const T *B1, const Off &O, const SplitCoords &p, F2 d[19], F2 g[7])
{
    static_for<0, kPlanes>([&](auto I) {
        constexpr int q = decltype(I)::value;
        bool o0, o1;
        split_outside<q, true>(p, o0, o1);
        const unsigned nb = O.template nb<q>(), bb = O.template bb<q>();
        float v0, v1;
        if constexpr (Off::kLocal) {
            v0 = Pair<T>::gld1(B0 + nb);
            v1 = Pair<T>::gld1(B1 + nb);
        } else {
            v0 = Pair<T>::gld1(B0 + (o0 ? bb : nb));
            v1 = Pair<T>::gld1(B1 + (o1 ? bb : nb));
        }
        if constexpr (q > 19) {
            constexpr int axis = plane_ex<q>() != 0 ? 0 : (plane_ey<q>() != 0 ? 1 : 2);
            if constexpr (dirichlet_axis<WALL>(axis)) {
                float tw;
                if constexpr (axis == 1) tw = (plane_ey<q>() == 1) ? 0.5f : -0.5f;
                else tw = p.th_lin;
                v0 = o0 ? fmaf(wall_coef<T>(), tw, -v0) : v0;  // anti-bounce-back
                v1 = o1 ? fmaf(wall_coef<T>(), tw, -v1) : v1;
            }
        }
        if constexpr (q < 19) d[q] = F2(v0, v1);
        else g[q - 19] = F2(v0, v1);
    });
}

// Store a pair's value, the second cell's only if it exists.
template <typename T, bool SR>
__device__ __forceinline__ void store_both(T *p0, T *p1, bool two, F2 v, unsigned r)
{
    if constexpr (std::is_same_v<T, float>) {
        *p0 = v.v.x;
        if (two) *p1 = v.v.y;
    } else {
        const unsigned w = Pair<T>::template pack<SR>(v, r);
        *reinterpret_cast<unsigned short *>(p0) = static_cast<unsigned short>(w);
        if (two) *reinterpret_cast<unsigned short *>(p1) = static_cast<unsigned short>(w >> 16);
    }
}

// The random bits of both cells at step number `step` (see pair_bits).
__device__ __forceinline__ unsigned split_bits(const SplitCoords &p, unsigned step)
{
    const unsigned salt = pcg_hash(step);
    return __byte_perm(pcg_hash(p.c0 ^ salt), pcg_hash(p.c1 ^ salt), 0x5410);
}

// The residual terms of both cells (residual_pair with separate addresses).
__device__ __forceinline__ void residual_split(const ResidualArgs &R, const SplitCoords &p, const float p0[4],
                                               const float p1[4], float2 th, float2 ux, float2 uy, float2 uz, DF acc[4])
{
    float t0[4], t1[4] = {0.f, 0.f, 0.f, 0.f};
    const int have_prev = *R.points > 0.0;
    residual_cell_terms(have_prev, th.x, ux.x, uy.x, uz.x, p0, t0);
    if (p.two) residual_cell_terms(have_prev, th.y, ux.y, uy.y, uz.y, p1, t1);
    const float2 now[4] = {th, ux, uy, uz};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        R.snap[k * R.cells + p.c0] = now[k].x;
        if (p.two) R.snap[k * R.cells + p.c1] = now[k].y;
        acc[k] = df_two_sum(t0[k], t1[k]);
    }
}

template <int WALL, typename T, bool SR, bool RES>
__global__ void __launch_bounds__(kSplitThreads, RES ? kSplitBlocksRes : kSplitBlocks)
    step_split_kernel(const T *__restrict__ src, T *__restrict__ dst, const StepGeometry S,
                      const CollideParams C, const ResidualArgs R, const RowDivisor D)
{
    // programmatic dependent launch, as in the one-cell kernel
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const SplitCoords p = split_coords(S, D);
    DF acc[4] = {};
    if (p.valid) {
        F2 d[19], g[7];
        float p0[4], p1[4];
        if constexpr (RES) {
            residual_cell_load(R, p.c0, p0);
            residual_cell_load(R, p.c1, p1);
        }
        pull_split<WALL, T>(src + p.c0, src + p.c1, TableOffsets{S}, p, d, g);
        const Conserved<F2> m0 = conserved<F2, Pair<T>::kShift>(d, g);
        const float2 th = m0.Tu.v, ux = m0.vx.v, uy = m0.vy.v, uz = m0.vz.v;
        unsigned r01 = 0;
        if constexpr (SR) {
            const size_t counter_at = static_cast<size_t>(kPlanes) * S.plane;
            const unsigned step = *reinterpret_cast<const unsigned *>(src + counter_at);
            if (p.c0 == 0) *reinterpret_cast<unsigned *>(dst + counter_at) = step + 1u;
            r01 = split_bits(p, step);
        }
        T *D0 = dst + p.c0, *D1 = dst + p.c1;
        const unsigned plane = opaque(S.plane);
        collide_from<F2, Pair<T>::kShift>(C, d, g, m0, plane_sink([&](auto I, F2 v) {
            constexpr int q = decltype(I)::value;
            store_both<T, SR>(D0 + q * plane, D1 + q * plane, p.two, v, SR ? plane_bits<q>(r01) : 0u);
        }));
        if constexpr (RES) residual_split(R, p, p0, p1, th, ux, uy, uz, acc);
    }
    if constexpr (RES) residual_block_store(acc, R.partials);
}

// The two in-place phases (step_inplace.cu); PHASE 2 as in step_pair.cu.
template <int WALL, typename T, bool SR, int PHASE, bool RES>
__global__ void __launch_bounds__(kSplitThreads, RES ? kSplitBlocksRes : kSplitBlocks)
    step_inplace_split_kernel(T *__restrict__ A, const InplaceGeometry SI, const CollideParams C,
                              const ResidualArgs R, const RowDivisor D)
{
    const StepGeometry &S = SI.load;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const SplitCoords p = split_coords(S, D);
    DF acc[4] = {};
    if (p.valid) {
        F2 d[19], g[7];
        float p0[4], p1[4];
        if constexpr (RES) {
            residual_cell_load(R, p.c0, p0);
            residual_cell_load(R, p.c1, p1);
        }
        if constexpr (PHASE == 0) pull_split<WALL, T>(A + p.c0, A + p.c1, TableOffsets{S}, p, d, g);
        else if constexpr (PHASE == 1) pull_split<WALL, T>(A + p.c0, A + p.c1, LocalOffsets{S.plane}, p, d, g);
        else pull_split<WALL, T>(A + p.c0, A + p.c1, LocalOppOffsets{S.plane}, p, d, g);
        const Conserved<F2> m0 = conserved<F2, Pair<T>::kShift>(d, g);
        const float2 th = m0.Tu.v, ux = m0.vx.v, uy = m0.vy.v, uz = m0.vz.v;
        unsigned r01 = 0;
        if constexpr (SR) {
            unsigned *ctr = reinterpret_cast<unsigned *>(A + static_cast<size_t>(kPlanes) * S.plane);
            const unsigned step = ctr[PHASE != 0];
            if (p.c0 == 0) ctr[PHASE == 0] = step + 1u;
            r01 = split_bits(p, step);
        }
        T *D0 = A + p.c0, *D1 = A + p.c1;
        const unsigned plane = opaque(S.plane);
        collide_from<F2, Pair<T>::kShift>(C, d, g, m0, plane_sink([&](auto I, F2 v) {
            constexpr int q = decltype(I)::value;
            const unsigned r = SR ? plane_bits<q>(r01) : 0u;
            if constexpr (PHASE == 1) {
                store_both<T, SR>(D0 + plane_opp<q>() * plane, D1 + plane_opp<q>() * plane, p.two, v, r);
            } else if constexpr (PHASE == 2) {
                store_both<T, SR>(D0 + q * plane, D1 + q * plane, p.two, v, r);
            } else {
                bool l0, l1;  // the link leaves the box
                split_outside<q, false>(p, l0, l1);
                const unsigned sn = static_cast<unsigned>(SI.sn[q]), sb = static_cast<unsigned>(SI.sb[q]);
                store_both<T, SR>(D0 + (l0 ? sb : sn), D1 + (l1 ? sb : sn), p.two, v, r);
            }
        }));
        if constexpr (RES) residual_split(R, p, p0, p1, th, ux, uy, uz, acc);
    }
    if constexpr (RES) residual_block_store(acc, R.partials);
}

cudaLaunchConfig_t split_config(const Geometry &G, cudaStream_t s, cudaLaunchAttribute *attr, bool pdl)
{
    cudaLaunchConfig_t cfg = {};
    const unsigned nxy = static_cast<unsigned>(G.nx) * G.ny;
    cfg.gridDim = dim3((nxy + kSplitThreads - 1) / kSplitThreads, (G.nz + 1) / 2);
    cfg.blockDim = dim3(kSplitThreads);
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cfg;
}

// f(std::true_type / std::false_type for stochastic stores) for the storage
// type and wall of the launch.
template <typename F>
cudaError_t split_dispatch(int wall, int storage, bool stochastic, F &&f)
{
    const cudaError_t e = dispatch(wall, storage, [&](auto W, auto *tp) {
        using T = std::remove_pointer_t<decltype(tp)>;
        if constexpr (decltype(W)::value == 0) {
            return cudaErrorInvalidValue;
        } else {
            if constexpr (!std::is_same_v<T, float>) {
                if (stochastic) return f(W, tp, std::true_type{});
            }
            return f(W, tp, std::false_type{});
        }
    });
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

bool step_split_supported(int wall, const Geometry &G)
{
    return wall >= 1 && wall <= 3 && static_cast<long long>(G.nx) * G.ny < (1LL << 28) - kSplitThreads;
}

// For small boxes both kernels' times are steps of their blocks per SM (152).
// Two buffers, FP32 and 16-bit, us per step: one cell per thread 2.5 to 3.4 for
// up to 3 blocks, 4.1 to 5.1 for 4 to 7, 4.6 to 6.4 for 8 to 10, 5.6 to 7.4 for
// 11 and 12; this kernel 2.5 to 2.8 for 1, 2.8 to 4.2 for 2, 3.7 to 4.6 up to
// 2.5, 4.8 to 6.1 up to 5 (the hardware spreads more than 380 blocks
// unevenly), 5.7 to 7.3 for 6.  Each row of the table: up to so many blocks of
// this kernel, it is taken from so many one-cell blocks on, FP32 and 16-bit;
// beyond it, from 1.8 times its own (thin boxes pair a slab with none).  Of
// 2346 timed cases, most of them chosen near these lines, 67 are slower than on
// the one-cell kernels by 2 % or more (15 by 10 to 19 %) and 111 would gain 3 % or
// more here; all together they gain 14 %.  Boxes below 60,000 cells, or of more
// than one round of blocks below 300,000, stay on the one-cell kernels.
bool step_split_pays(const Geometry &G, int storage)
{
    const long long cells = static_cast<long long>(G.nx) * G.ny * G.nz;
    const long long blocks = static_cast<long long>(split_blocks(G));
    if (cells < 300000 && (cells < 60000 || blocks > 152 * kSplitBlocks)) return false;
    const long long one_cell = static_cast<long long>((G.nx + 31) / 32) * ((G.ny + 3) / 4) * G.nz;
    constexpr int kLine[][3] = {{152, 456, 456}, {290, 530, 530}, {380, 520, 520}, {608, 1474, 1307}, {760, 1094, 1094}};
    for (const auto &l : kLine)
        if (blocks <= l[0]) return one_cell >= l[storage == 0 ? 1 : 2];
    return 5 * one_cell >= 9 * blocks;
}

size_t split_blocks(const Geometry &G)
{
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = split_config(G, nullptr, attr, false);
    return static_cast<size_t>(cfg.gridDim.x) * cfg.gridDim.y;
}

cudaError_t launch_step_split(int wall, int storage, bool stochastic, const void *src, void *dst, const StepGeometry &S,
                              const Geometry &G, const CollideParams &C, cudaStream_t s, bool pdl, const ResidualArgs *res)
{
    if (!step_split_supported(wall, G)) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = split_config(G, s, attr, pdl);
    const ResidualArgs R = res ? *res : ResidualArgs{};
    const RowDivisor D(static_cast<unsigned>(G.nx));
    return split_dispatch(wall, storage, stochastic, [&](auto W, auto *tp, auto sr) {
        using T = std::remove_pointer_t<decltype(tp)>;
        constexpr int WL = decltype(W)::value;
        constexpr bool SRv = decltype(sr)::value;
        const T *a = static_cast<const T *>(src);
        T *b = static_cast<T *>(dst);
        return res ? cudaLaunchKernelEx(&cfg, step_split_kernel<WL, T, SRv, true>, a, b, S, C, R, D)
                   : cudaLaunchKernelEx(&cfg, step_split_kernel<WL, T, SRv, false>, a, b, S, C, R, D);
    });
}

cudaError_t launch_step_inplace_split(int wall, int storage, bool stochastic, void *buf, int phase,
                                      const InplaceGeometry &SI, const Geometry &G, const CollideParams &C,
                                      cudaStream_t s, bool pdl, const ResidualArgs *res)
{
    if (!step_split_supported(wall, G) || phase < 0 || phase > 2 || (phase == 2 && res)) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = split_config(G, s, attr, pdl);
    const ResidualArgs R = res ? *res : ResidualArgs{};
    const RowDivisor D(static_cast<unsigned>(G.nx));
    return split_dispatch(wall, storage, stochastic, [&](auto W, auto *tp, auto sr) {
        using T = std::remove_pointer_t<decltype(tp)>;
        constexpr int WL = decltype(W)::value;
        constexpr bool SRv = decltype(sr)::value;
        T *A = static_cast<T *>(buf);
        auto run = [&](auto ph, auto rs) {
            return cudaLaunchKernelEx(
                &cfg, step_inplace_split_kernel<WL, T, SRv, decltype(ph)::value, decltype(rs)::value>, A, SI, C, R, D);
        };
        using std::integral_constant;
        if (phase == 2) return run(integral_constant<int, 2>{}, std::false_type{});
        if (res)
            return phase == 0 ? run(integral_constant<int, 0>{}, std::true_type{})
                              : run(integral_constant<int, 1>{}, std::true_type{});
        return phase == 0 ? run(integral_constant<int, 0>{}, std::false_type{})
                          : run(integral_constant<int, 1>{}, std::false_type{});
    });
}

}  // namespace lbm
