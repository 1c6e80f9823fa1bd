// pot_backward.cu -- analytic derivatives of the render (App. B.3.2), the
// optimiser step on the leaves (Sec. 3.3), the MSE loss of a ray batch (Sec. 3,
// NeRF loss) and pixel-ray generation for training batches.
//
// Backward, per ray (replaying the forward walk, so segments and the early-
// stop point are the forward's):
//   c_i = S(x_i),  x_i = sum_k k_{i,k} Y_k,  w_i = T_i (1 - e^{-sigma_i delta_i})
//   dC/dx_i      = w_i c_i (1 - c_i)                         (colour derivative, chain rule)
//   dC/dk_{i,k}  = dC/dx_i Y_k                               (basis constant along the ray)
//   dC/dsigma_i  = delta_i [ c_i T_{i+1} - S_i ],  S_i = sum_{k>i} w_k c_k + T_N bg
//                = delta_i [ c_i T_{i+1} - (C - sum_{k<=i} w_k c_k) ]
// i.e. the paper's two passes: the composited colour C (the forward output,
// or a first in-kernel pass) minus a running prefix.  Zero for sigma <= 0.
// Gradients of L = sum_rays <dL/dC, C> are scattered with float reductions
// (16-byte vector reductions where the row allows).  With POT_BWD_AGG, lanes
// of a warp that composite the same leaf in the same step first sum their
// contributions with warp shuffles (warp-aggregated atomics) and one lane per
// leaf issues the reductions.
#include <cmath>

#include "pot_render.cuh"
#include "pot_segments_internal.h"

#ifndef POT_BWD_AGG
// warp-aggregated gradient scatter (lanes sharing a leaf reduce by shuffles
// first).  Off: measured slower on 2^18-ray batches of the main tree, both for
// random pixels (1.28 vs 0.86 ms) and for random 4 x 8 pixel tiles, whose
// lanes do share leaves (0.75 vs 0.53 ms): the match and the 49-value shuffle
// tree cost more than the float reductions they save.
#define POT_BWD_AGG 0
#endif

namespace pot {

namespace {

__device__ __forceinline__ void red_add(float *a, float v)
{
    asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(a), "f"(v) : "memory");
}

__device__ __forceinline__ void red_add4(float *a, float x, float y, float z, float w)
{
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(a), "f"(x), "f"(y), "f"(z),
                 "f"(w)
                 : "memory");
}

// The terms of one leaf segment (App. B.3.2), given T_i (Tr) and the colour
// composited in front of it (prefix): the colour derivative gx_c =
// dL/dC_c w c_c (1 - c_c) (times Y_k for coefficient k) and the density
// derivative gsd (0 for sigma <= 0); Tr and prefix move past the segment.
// Returns whether sigma > 0.  The same operations as the forward's shading.
template <int K, typename T, typename YT>
__device__ __forceinline__ bool segment_terms(const T *sig_arr, const T *sh_arr, int leaf, float delta, const YT &Y,
                                              const float g[3], const float ctot[3], float prefix[3], float &Tr,
                                              float gx[3], float &gsd)
{
    const float sraw = Store<T>::load_sigma(sig_arr, leaf);
    const float sig = fmaxf(sraw, 0.f);
    float x[3];
    leaf_sh_dot<K, T>(sh_arr, leaf, Y, x, nullptr);
    const float e = exp_ftz(-sig * delta);  // same operations as the forward
    const float w = Tr * (1.f - e);
    const float Tn = Tr * e;
    float gs = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float col = sigmoidf_(x[c]);
        prefix[c] = fmaf(w, col, prefix[c]);
        gx[c] = g[c] * w * col * (1.f - col);
        gs = fmaf(g[c], fmaf(col, Tn, -(ctot[c] - prefix[c])), gs);
    }
    gsd = sraw > 0.f ? gs * delta : 0.f;  // zero for sigma <= 0 (same leaf: same sign)
    Tr = Tn;
    return sraw > 0.f;
}

template <int K, typename T>
struct GradVisitor {
    static constexpr bool kBasis = true, kVote = false;
    const T *sig_arr;
    const T *sh_arr;
    float gamma;
    float g[3];       // dL/dC of the ray
    float ctot[3];    // C of the ray (background included)
    float prefix[3];  // sum over composited segments of w c
    float Tr;
    float rest;       // the frame's
    float *grad_sigma;
    float *grad_sh;
    template <typename YT>
    __device__ __forceinline__ bool operator()(int leaf, float delta, const YT &Y)
    {
        float gx[3], gsd;
        const bool pos = segment_terms<K, T>(sig_arr, sh_arr, leaf, delta * rest, Y, g, ctot, prefix, Tr, gx, gsd);
        float *row = grad_sh + (int64_t)leaf * (3 * K);
#if POT_BWD_AGG
        // lanes compositing the same leaf: sum over the group with a shuffle
        // tree over its members (ranked by lane); the lowest lane scatters
        const unsigned act = __activemask();
        const unsigned grp = __match_any_sync(act, leaf);
        const unsigned shared_lanes = __ballot_sync(act, __popc(grp) > 1);
        if (shared_lanes) {
            const int lane = threadIdx.x & 31;
            if (grp != (1u << lane)) {
                const int n = __popc(grp);
                const int rank = __popc(grp & ((1u << lane) - 1u));
                const int nmax = (int)__reduce_max_sync(shared_lanes, (unsigned)n);
                float v[3 * K];
#pragma unroll
                for (int j = 0; j < 3 * K; ++j) v[j] = gx[j % 3] * Y[j / 3];
                for (int o = 1; o < nmax; o <<= 1) {
                    const bool has = rank + o < n;
                    const int src = has ? (int)__fns(grp, (unsigned)lane, o + 1) : lane;
#pragma unroll
                    for (int j = 0; j < 3 * K; ++j) {
                        const float t = __shfl_sync(shared_lanes, v[j], src);
                        if (has) v[j] += t;
                    }
                    const float t = __shfl_sync(shared_lanes, gsd, src);
                    if (has) gsd += t;
                }
                if (rank == 0) {
                    if ((3 * K) % 4 == 0) {
#pragma unroll
                        for (int j = 0; j < 3 * K; j += 4) red_add4(row + j, v[j], v[j + 1], v[j + 2], v[j + 3]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 3 * K; ++j) red_add(row + j, v[j]);
                    }
                    if (pos) red_add(grad_sigma + leaf, gsd);
                }
                return Tr < gamma;
            }
        }
#endif
        if ((3 * K) % 4 == 0) {
#pragma unroll
            for (int j = 0; j < 3 * K; j += 4)
                red_add4(row + j, gx[j % 3] * Y[j / 3], gx[(j + 1) % 3] * Y[(j + 1) / 3],
                         gx[(j + 2) % 3] * Y[(j + 2) / 3], gx[(j + 3) % 3] * Y[(j + 3) / 3]);
        } else {
#pragma unroll
            for (int j = 0; j < 3 * K; ++j) red_add(row + j, gx[j % 3] * Y[j / 3]);
        }
        if (pos) red_add(grad_sigma + leaf, gsd);
        return Tr < gamma;
    }
};

// The mean of a launch's squared errors: each warp's sum (in its first lane) joins its block's and the grid's in
// double, and the block that adds the last one writes the rounded mean.  Every thread of every block calls it.
template <int BLOCK>
__device__ __forceinline__ void finish_loss(double warp_sum, LossSum *s, double count, float *loss)
{
    __shared__ double part[BLOCK / 32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = warp_sum;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double sum = 0.0;
    for (int w = 0; w < BLOCK / 32; ++w) sum += part[w];
    atomicAdd(&s->sum, sum);
    __threadfence();
    if (atomicAdd(&s->blocks, 1ull) == gridDim.x - 1) {  // every block's sum is in
        __threadfence();
        *loss = (float)(*(volatile double *)&s->sum / count);
    }
}

struct BackwardParams {
    RenderParams r;
    const float *grad_rgb;
    const float *rgb_fwd;  // NULL: computed by a first pass
    float *grad_sigma;
    float *grad_sh;
    // fused MSE mode: dL/dC = mse_scale (C - target), L = sum (C - target)^2 / (3 n_rays)
    const float *target;
    float *loss;
    LossSum *loss_sum;     // zero before the launch
    float *rgb_out;        // optional copy of C
    float mse_scale;
    // non-null: the kernel runs only if *run_if != 0 (the walking backward as
    // the fallback of the per-record backward, whose records overflowed)
    const unsigned long long *run_if;
};

// What the backward kernel is given per ray.
enum BackwardMode { kGradAndColour = 0, kGrad = 1, kMseTarget = 2 };

#ifndef POT_BACKWARD_MIN_BLOCKS
// resident blocks per SM: 3 (12 warps, 168 registers).  4 blocks: 692 against
// 702 us on 2^18 random pixels of the depth-9 tree, but 2928 against 2649 us where
// every ray meets a leaf (see rays_min_blocks); 5: 814 us; 6: 908 us
#define POT_BACKWARD_MIN_BLOCKS 3
#endif
// With bricks or without an index a step waits for loads in turn, and where a
// segment's own registers are few (K <= 4: 80 hold it without spills) 24 warps are
// better, 10^6 random rays: depth 10, degree 1, no index 2564 -> 2280 us, bricks
// 1631 -> 1501 us, degree 0 2409 -> 1940 and 1461 -> 1236 us, 2^18 rays about half
// of that gain, up to 40,000 within 3 % (4 and 5 blocks: 2552, 2557 us).  At degree
// 3, whose registers spill, 200,000 rays (depth 9, bricks) take 591 instead of 445 us.
constexpr int backward_min_blocks(Lookup l, int K)
{
    return l == kLookAny && K <= 4 ? 6 : POT_BACKWARD_MIN_BLOCKS;
}

// MODE kGradAndColour: dL/dC and C given; kGrad: dL/dC given, C from a first
// walk; kMseTarget: C from a first walk, then dL/dC of the MSE against the
// target, C optionally written out.  The loss: each ray's squared error in float,
// summed over a warp by shuffles, over the warp's tiles, the block and the grid in
// double (one double reduction per block), and rounded once by the block that
// finishes last.  A float sum of one rounded addition per warp was off by 1.1e-6 of
// the loss at 20,011 rays (2,504 warps), by 2.6e-5 at 100,003 rays whose errors were
// all alike.  The call of 20,011 rays 85 -> 88 us.
template <int K, typename T, Lookup LOOKUP, int MODE>
__global__ void __launch_bounds__(kBlock, backward_min_blocks(LOOKUP, K))
    backward_kernel(const __grid_constant__ BackwardParams bp)
{
    POT_WALK_SHARED(K)
    const RenderParams &p = bp.r;
    if (bp.run_if && *bp.run_if == 0ull) return;
    const int lane = threadIdx.x & 31;
    const T *sig_arr = static_cast<const T *>(p.sigma);
    const T *sh_arr = static_cast<const T *>(p.sh);
    int taken = 0, slot;
    double wsum = 0.0;  // squared error of the warp's rays (MSE mode)
    for (unsigned long long tile; next_tile(p, lane, taken, tile, slot);) {
        const int64_t ray = (int64_t)tile * 32 + slot;
        float lsum = 0.f;  // this ray's squared error (MSE mode)
        const bool has = slot < 32 && ray < p.n_rays;
        float o[3], d[3];
        GradVisitor<K, T> gv;
        gv.sig_arr = sig_arr;
        gv.sh_arr = sh_arr;
        gv.gamma = p.gamma;
        gv.Tr = 1.f;
        gv.rest = p.frame.rest;
        gv.grad_sigma = bp.grad_sigma;
        gv.grad_sh = bp.grad_sh;
        if (has) {
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                o[r] = __ldg(p.ray_o + 3 * ray + r);
                d[r] = __ldg(p.ray_d + 3 * ray + r);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) gv.prefix[c] = gv.ctot[c] = gv.g[c] = 0.f;
        if (MODE == kGradAndColour) {
            if (has) {
#pragma unroll
                for (int c = 0; c < 3; ++c) gv.ctot[c] = __ldg(bp.rgb_fwd + 3 * ray + c);
            }
        } else {
            ShadeVisitor<K, T, false> sv{sig_arr, sh_arr, nullptr, p.gamma, {0.f, 0.f, 0.f}, 1.f, 0, nullptr,
                                         p.frame.rate};
            walk_rays<K, T, LOOKUP, false>(p, stk, ysm, wst, has, o, d, p.near, p.far, sv);
#pragma unroll
            for (int c = 0; c < 3; ++c) gv.ctot[c] = fmaf(sv.Tr, p.bg[c], sv.col[c]);
        }
        if (has) {
            if (MODE == kMseTarget) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float r = gv.ctot[c] - __ldg(bp.target + 3 * ray + c);
                    lsum = fmaf(r, r, lsum);
                    gv.g[c] = bp.mse_scale * r;
                    if (bp.rgb_out) bp.rgb_out[3 * ray + c] = gv.ctot[c];
                }
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) gv.g[c] = __ldg(bp.grad_rgb + 3 * ray + c);
            }
        }
        walk_rays<K, T, LOOKUP, false>(p, stk, ysm, wst, has && (gv.g[0] != 0.f || gv.g[1] != 0.f || gv.g[2] != 0.f), o, d, p.near,
                        p.far, gv);
        if (MODE == kMseTarget) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
            wsum += (double)lsum;
        }
    }
    if (MODE == kMseTarget) finish_loss<kBlock>(wsum, bp.loss_sum, 3.0 * (double)p.n_rays, bp.loss);
}

template <typename T>
cudaError_t launch_backward_t(const BackwardParams &bp, int K, int mode, cudaStream_t s)
{
    using Fn = void (*)(const BackwardParams);
    const bool dense = dense_index(bp.r);
    Fn fn = mode == kGradAndColour ? POT_PICK_WALK(backward_kernel, K, T, dense, kGradAndColour)
          : mode == kGrad          ? POT_PICK_WALK(backward_kernel, K, T, dense, kGrad)
                                   : POT_PICK_WALK(backward_kernel, K, T, dense, kMseTarget);
    if (!fn) return cudaErrorInvalidValue;
    const size_t smem = walk_smem_bytes(bp.r.cells == nullptr);
    unsigned grid = 0;
    cudaError_t e = persistent_grid(fn, smem, bp.r, &grid);
    if (e != cudaSuccess) return e;
    fn<<<grid, kBlock, smem, s>>>(bp);
    count_launch();
    return cudaGetLastError();
}

// ---- gradients from recorded segments ---------------------------------------
// One thread per record of pot_render_rays_record: the record gives the leaf,
// delta_i, T_i and P_i, the ray gives dL/dC, C and the SH basis at its
// direction; GradVisitor then does exactly the per-segment work of the walking
// backward (same operations, so the same per-segment terms bit for bit).

constexpr int kFlatBlock = 256;  // threads per block of the kernels without a walk

// The per-ray SH basis in registers (the interface of SmemY).
template <int K>
struct RegY {
    float v[K];
    __device__ __forceinline__ float operator[](int k) const { return v[k]; }
    __device__ __forceinline__ void fetch(float *yv, int k0, int k1) const
    {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k >= k0 && k <= k1) yv[k] = v[k];
    }
};

struct SegBackwardParams {
    SegmentBuffer sb;
    int64_t n_rays;    // records naming a ray or leaf outside these ranges are skipped
    int64_t n_leaves;
    // non-null: visit the records in the order perm[0 .. *n_perm) (by bin of
    // leaves, so that the reductions of neighbouring threads meet the same
    // gradient rows in L2); null: in slot order
    const unsigned *perm;
    const unsigned *n_perm;
    const void *sigma;
    const void *sh;
    const float *ray_d;
    const float *grad_rgb;
    const float *rgb_fwd;
    float *grad_sigma;
    float *grad_sh;
};

#ifndef POT_SEGBWD_MIN_BLOCKS
// resident blocks per SM: 3 (at most 80 registers, no spills; 4 blocks spill 12 bytes at 64)
#define POT_SEGBWD_MIN_BLOCKS 3
#endif

// How a warp sums 32 records into gradient rows: groups of kLanes lanes, each
// lane holding kVec adjacent values of a row (kPer times, kLanes * kVec apart),
// each group taking kRecs consecutive records.
template <int K>
struct RowShape {
    static constexpr int kVec = (3 * K) % 4 == 0 ? 4 : 1;
    static constexpr int kLanes = 3 * K / kVec < 32 ? 3 * K / kVec : 32;
    static constexpr int kPer = (3 * K / kVec + kLanes - 1) / kLanes;
    static constexpr int kGroups = 32 / kLanes;
    static constexpr int kRecs = (32 + kGroups - 1) / kGroups;
    // a warp's shared memory, in floats: per record dL/dx as three float4 {x0 x1 x2 x0}, {x1 x2 x0 x1},
    // {x2 x0 x1 x2} (a lane's four values start with channel 4 l mod 3), the basis (an odd row length keeps
    // the rows of 32 lanes, and of two groups, on distinct banks), and the leaves
    static constexpr int kBasisRow = K | 1;
    static constexpr int kBasis = 32 * 12, kLeaf = kBasis + 32 * kBasisRow, kFloats = (kLeaf + 32 + 3) / 4 * 4;
};

// Whole warps step over the records together, one record per lane.  Lanes next
// to each other that hold records of the same leaf (records in leaf order, or
// neighbouring rays of one forward step in slot order) form a run.  A record's
// row is the product of its three colour derivatives and its basis, so the
// warp leaves both in shared memory and sums rows from there: a group of lanes
// holds a whole row (12 lanes x 4 values at K = 16), walks its share of the
// records and, at the end of a run, adds the row with one reduction instruction
// of adjacent lanes.
//
// What bounds it: the float reductions and the gather of each record's ray and
// leaf.  One reduction of adjacent 16-byte vectors per row moves whole sectors;
// it replaced 12 reductions per run of one lane each (a scan of the 49 values
// over the run by shuffles, 735 instructions a warp), whose 16 bytes each were a
// request of their own.  With the sort's passes, 2^18 rays on the depth-9 tree
// (4.2 M records, degree 3): 537 -> 391 us.
template <int K, typename T>
__global__ void __launch_bounds__(kFlatBlock, POT_SEGBWD_MIN_BLOCKS) segment_backward_kernel(const SegBackwardParams q)
{
    if (q.sb.state[1] != 0ull) return;  // the records overflowed: the walking backward runs instead
    const unsigned long long handed = q.sb.state[0];
    const int64_t used = q.perm ? (int64_t)*q.n_perm
                       : handed < (unsigned long long)q.sb.capacity ? (int64_t)handed : q.sb.capacity;
    const int lane = threadIdx.x & 31;
    const T *sig_arr = static_cast<const T *>(q.sigma);
    const T *sh_arr = static_cast<const T *>(q.sh);
    using S = RowShape<K>;
    __shared__ float4 rows_sh[kFlatBlock / 32 * S::kFloats / 4];
    float *ws = reinterpret_cast<float *>(rows_sh) + (threadIdx.x >> 5) * S::kFloats;  // this warp's part
    const int group = lane / S::kLanes, in_row = lane % S::kLanes;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); k0 < used; k0 += stride) {
        const int64_t k = k0 + lane;
        int leaf = -1;  // -1: no terms on this lane
        float gx[3] = {0.f, 0.f, 0.f}, gsd = 0.f;
        RegY<K> Y;
#pragma unroll
        for (int j = 0; j < K; ++j) Y.v[j] = 0.f;
        if (k < used) {
            const int64_t i = q.perm ? (int64_t)q.perm[k] : k;
            const float4 a = __ldg(q.sb.rec + 2 * i);
            const int ray = __float_as_int(a.x), lf = __float_as_int(a.y);
            // unused slots (ray -1) and records naming a ray or leaf out of range are skipped
            if (ray >= 0 && ray < q.n_rays && lf >= 0 && lf < q.n_leaves) {
                float g[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) g[c] = __ldg(q.grad_rgb + 3 * (int64_t)ray + c);
                if (g[0] != 0.f || g[1] != 0.f || g[2] != 0.f) {
                    const float4 b4 = __ldg(q.sb.rec + 2 * i + 1);
                    float ctot[3], prefix[3] = {b4.x, b4.y, b4.z}, d[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) ctot[c] = __ldg(q.rgb_fwd + 3 * (int64_t)ray + c);
#pragma unroll
                    for (int c = 0; c < 3; ++c) d[c] = __ldg(q.ray_d + 3 * (int64_t)ray + c);
                    // the basis exactly as the walk computes it (Walker::begin)
                    const float len = sqrtf(fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2])));
                    const float invlen = __frcp_rn(len);
                    sh_basis<K>(d[0] * invlen, d[1] * invlen, d[2] * invlen, Y.v);
                    float Tr = a.w;
                    segment_terms<K, T>(sig_arr, sh_arr, lf, a.z, Y, g, ctot, prefix, Tr, gx, gsd);
                    leaf = lf;
                }
            }
        }
        const int next = __shfl_down_sync(0xffffffffu, leaf, 1);
        const unsigned ends = __ballot_sync(0xffffffffu, lane == 31 || leaf != next);  // last records of runs
        if (__all_sync(0xffffffffu, leaf < 0)) continue;
        if (S::kVec == 4) {
            float4 *x = reinterpret_cast<float4 *>(ws) + 3 * lane;
            x[0] = make_float4(gx[0], gx[1], gx[2], gx[0]);
            x[1] = make_float4(gx[1], gx[2], gx[0], gx[1]);
            x[2] = make_float4(gx[2], gx[0], gx[1], gx[2]);
        } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) ws[3 * lane + c] = gx[c];
        }
#pragma unroll
        for (int j = 0; j < K; ++j) ws[S::kBasis + lane * S::kBasisRow + j] = Y.v[j];
        reinterpret_cast<int *>(ws)[S::kLeaf + lane] = leaf;
        __syncwarp();
        if (group < S::kGroups) {
            float acc[S::kPer][S::kVec];
#pragma unroll
            for (int u = 0; u < S::kPer; ++u)
#pragma unroll
                for (int v = 0; v < S::kVec; ++v) acc[u][v] = 0.f;
            const int r_end = min(32, (group + 1) * S::kRecs);
            for (int r = group * S::kRecs; r < r_end; ++r) {
                const float *y = ws + S::kBasis + r * S::kBasisRow;
                if (S::kVec == 4) {
                    const float4 x = reinterpret_cast<const float4 *>(ws)[3 * r + in_row % 3];
                    const float y0 = y[4 * in_row / 3], y1 = y[4 * in_row / 3 + 1];
                    acc[0][0] = fmaf(x.x, y0, acc[0][0]);
                    acc[0][1 % S::kVec] = fmaf(x.y, in_row % 3 == 2 ? y1 : y0, acc[0][1 % S::kVec]);
                    acc[0][2 % S::kVec] = fmaf(x.z, in_row % 3 == 0 ? y0 : y1, acc[0][2 % S::kVec]);
                    acc[0][3 % S::kVec] = fmaf(x.w, y1, acc[0][3 % S::kVec]);
                } else {
#pragma unroll
                    for (int u = 0; u < S::kPer; ++u) {
                        const int j = u * S::kLanes + in_row;
                        if (j < 3 * K) acc[u][0] = fmaf(ws[3 * r + j % 3], y[j / 3], acc[u][0]);
                    }
                }
                if (((ends >> r) & 1u) || r + 1 == r_end) {
                    const int lf = reinterpret_cast<const int *>(ws)[S::kLeaf + r];
                    if (lf >= 0) {
                        float *row = q.grad_sh + (int64_t)lf * (3 * K);
                        if (S::kVec == 4) {
                            red_add4(row + 4 * in_row, acc[0][0], acc[0][1 % S::kVec], acc[0][2 % S::kVec],
                                     acc[0][3 % S::kVec]);
                        } else {
#pragma unroll
                            for (int u = 0; u < S::kPer; ++u) {
                                const int j = u * S::kLanes + in_row;
                                if (j < 3 * K) red_add(row + j, acc[u][0]);
                            }
                        }
                    }
#pragma unroll
                    for (int u = 0; u < S::kPer; ++u)
#pragma unroll
                        for (int v = 0; v < S::kVec; ++v) acc[u][v] = 0.f;
                }
            }
        }
        // the density derivative: summed over the run by shuffles, complete in its last lane
        const unsigned before = ends & ((1u << lane) - 1u);
        const int run0 = before ? 32 - __clz(before) : 0;
        float gs = gsd;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float v = __shfl_up_sync(0xffffffffu, gs, d);
            if (lane - d >= run0) gs += v;
        }
        if (leaf >= 0 && ((ends >> lane) & 1u) && gs != 0.f) red_add(q.grad_sigma + leaf, gs);
        __syncwarp();  // the next records overwrite the rows
    }
}

template <typename T>
cudaError_t launch_segment_backward_t(const SegBackwardParams &q, int K, cudaStream_t s)
{
    using Fn = void (*)(const SegBackwardParams);
    Fn fn = K == 1 ? segment_backward_kernel<1, T> : K == 4 ? segment_backward_kernel<4, T>
          : K == 9 ? segment_backward_kernel<9, T> : K == 16 ? segment_backward_kernel<16, T>
          : K == 25 ? segment_backward_kernel<25, T> : nullptr;
    if (!fn) return cudaErrorInvalidValue;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kFlatBlock, 0);
    if (e != cudaSuccess) return e;
    // one wave of resident blocks, no more than the slots could need
    int64_t blocks = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    const int64_t need = (q.sb.capacity + kFlatBlock - 1) / kFlatBlock;
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    fn<<<(unsigned)blocks, kFlatBlock, 0, s>>>(q);
    count_launch();
    return cudaGetLastError();
}

// ---- recorded segments in leaf order ----------------------------------------
// The records are visited leaf by leaf: one pass counts the records per leaf
// and notes each record's leaf and place among its leaf's, a scan gives every
// leaf a range of positions, and a second pass puts the record numbers there
// (without atomics).  A leaf's records are then adjacent, so the per-record
// kernel merges them within a warp, and neighbouring threads reduce into
// neighbouring gradient rows.  The leaves' ranges need no particular order: the
// scan runs over tiles of leaves, each of which draws its range from a counter.

struct SegBinParams {
    SegBackwardParams s;
    SegmentBins b;
};

constexpr int kScanBlock = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanBlock * kScanItems;  // counts per scan block

// A record's leaf, or -1 for an unused slot or one naming an out-of-range ray
// or leaf.
__device__ __forceinline__ int record_leaf(const SegBackwardParams &q, int64_t i, int64_t used)
{
    if (i >= used) return -1;
    const float4 a = __ldg(q.sb.rec + 2 * i);
    const int ray = __float_as_int(a.x), leaf = __float_as_int(a.y);
    if (ray < 0 || ray >= q.n_rays || leaf < 0 || leaf >= q.n_leaves) return -1;
    return leaf;
}

__device__ __forceinline__ int64_t records_used(const SegmentBuffer &sb)
{
    const unsigned long long handed = sb.state[0];
    return handed < (unsigned long long)sb.capacity ? (int64_t)handed : sb.capacity;
}

// Pass 1: records per leaf, and each record's leaf and place.  Whole warps step
// together so that lanes with the same leaf (neighbouring rays of one step)
// share one atomic, found with a match.
__global__ void __launch_bounds__(kFlatBlock) leaf_count_kernel(const SegBinParams q)
{
    if (q.s.sb.state[1] != 0ull) return;
    const int64_t used = records_used(q.s.sb);
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); i0 < used; i0 += stride) {
        const int64_t i = i0 + lane;
        const int leaf = record_leaf(q.s, i, used);
        const unsigned m = __match_any_sync(0xffffffffu, leaf);
        const int leader = __ffs(m) - 1;
        unsigned base = 0;
        if (leaf >= 0 && lane == leader) base = atomicAdd(q.b.start + leaf, (unsigned)__popc(m));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (i < used) q.b.place[i] = make_uint2((unsigned)leaf, base + __popc(m & ((1u << lane) - 1u)));
    }
}

// Pass 2: each record's number to its position.
__global__ void __launch_bounds__(kFlatBlock) leaf_scatter_kernel(const SegBinParams q)
{
    if (q.s.sb.state[1] != 0ull) return;
    const int64_t used = records_used(q.s.sb);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < used; i += (int64_t)gridDim.x * blockDim.x) {
        const uint2 v = q.b.place[i];
        if ((int)v.x >= 0) q.b.perm[q.b.start[v.x] + v.y] = (unsigned)i;
    }
}

// Exclusive scan of one value per thread over a block of kScanBlock threads;
// *total = the block's sum.
__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned *total)
{
    __shared__ unsigned warp_sum[kScanBlock / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
    }
    if (lane == 31) warp_sum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        unsigned w = warp_sum[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned t = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += t;
        }
        warp_sum[lane] = w;
    }
    __syncthreads();
    *total = warp_sum[kScanBlock / 32 - 1];
    return (wid ? warp_sum[wid - 1] : 0u) + incl - v;
}

// Counts become first positions, a tile of kScanTile leaves per block.
__global__ void __launch_bounds__(kScanBlock) leaf_ranges_kernel(const SegBinParams q)
{
    __shared__ unsigned tile_base;
    if (q.s.sb.state[1] != 0ull) return;
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    unsigned c[kScanItems], v = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        c[u] = base + u < q.b.n_bins ? q.b.start[base + u] : 0u;
        v += c[u];
    }
    unsigned total;
    unsigned run = block_exclusive_scan(v, &total);
    if (threadIdx.x == 0) tile_base = total ? atomicAdd(q.b.n_perm, total) : 0u;
    __syncthreads();
    if (total == 0) return;
    run += tile_base;
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        if (base + u < q.b.n_bins) q.b.start[base + u] = run;
        run += c[u];
    }
}

template <typename T>
cudaError_t launch_leaf_order_t(const SegBinParams &q, int K, cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // count and scatter passes: a few waves of blocks over the slots (grid-stride)
    int64_t blocks = (q.s.sb.capacity + kFlatBlock - 1) / kFlatBlock;
    if (blocks > 8 * (int64_t)sms) blocks = 8 * (int64_t)sms;
    if (blocks < 1) blocks = 1;
    const int64_t n_tiles = (q.b.n_bins + kScanTile - 1) / kScanTile;
    leaf_count_kernel<<<(unsigned)blocks, kFlatBlock, 0, s>>>(q);
    leaf_ranges_kernel<<<(unsigned)n_tiles, kScanBlock, 0, s>>>(q);
    leaf_scatter_kernel<<<(unsigned)blocks, kFlatBlock, 0, s>>>(q);
    count_launch(3);
    // the per-record kernel over the records in leaf order
    SegBackwardParams sq = q.s;
    sq.perm = q.b.perm;
    sq.n_perm = q.b.n_perm;
    return launch_segment_backward_t<T>(sq, K, s);
}

// ---- optimiser step on the leaves ------------------------------------------
struct StepParams {
    int64_t L;
    float lr_sigma, lr_sh, alpha, beta1, beta2, eps;
    float bc1, bc2;   // Adam bias corrections 1 - beta^t
    bool zero_stays;  // the divisor is above 0 for every v >= 0, so that 0 over it is 0
};

// Whether the update of a value whose quotient's numerator is num changes it.  A
// leaf that no ray met has num = 0 and often v = 0, which the IEEE root and
// quotients take to their slow paths; its value stays as it is, without them.
// Adam after 1,000 rays on 10.7 M leaves of degree 2: 2203 -> 1272 us (6.6 TB/s),
// after 2^18 rays on 4.0 M 764 -> 559 us; with no gradient 0, 2 to 4 % longer (4.3 M
// leaves of degree 2, RMSprop 471 -> 493 us, Adam 578 -> 597 us).
__device__ __forceinline__ bool moves(const StepParams &sp, float num, float v)
{
    return num != 0.f || !(v >= 0.f) || !sp.zero_stays;
}

// One parameter's update; m and v are its optimiser state (v unused by SGD,
// m only by Adam).
template <int KIND>
__device__ __forceinline__ float step_one(const StepParams &sp, float x, float g, float lr, float &m, float &v)
{
    if (KIND == POT_SGD) {
        x -= lr * g;
    } else if (KIND == POT_RMSPROP) {
        v = sp.alpha * v + (1.f - sp.alpha) * g * g;
        if (moves(sp, lr * g, v)) x -= lr * g / (sqrtf(v) + sp.eps);
    } else {
        m = sp.beta1 * m + (1.f - sp.beta1) * g;
        v = sp.beta2 * v + (1.f - sp.beta2) * g * g;
        if (moves(sp, (lr / sp.bc1) * m, v)) x -= (lr / sp.bc1) * m / (sqrtf(v) / sqrtf(sp.bc2) + sp.eps);
    }
    return x;
}

// State of value j (public order: sigma part, then SH part): RMSprop v at
// state[j]; Adam m at state[j], v at state[N + j].
template <int KIND>
__device__ __forceinline__ void load_state(const float *state, int64_t N, int64_t j, float &m, float &v)
{
    if (KIND == POT_RMSPROP) v = state[j];
    if (KIND == POT_ADAM) {
        m = state[j];
        v = state[N + j];
    }
}
template <int KIND>
__device__ __forceinline__ void store_state(float *state, int64_t N, int64_t j, float m, float v)
{
    if (KIND == POT_RMSPROP) state[j] = v;
    if (KIND == POT_ADAM) {
        state[j] = m;
        state[N + j] = v;
    }
}

// The step streams L (1 + 3K) values through 3 (SGD) to 7 (Adam) arrays and is
// bound by HBM.  Work goes in units of kStepUnit values, first the densities,
// then the SH values in the gradients' order; a thread takes every kStepBlock-th
// value of a unit and has the loads of all of them in flight before the first
// update.  Accesses are 4 bytes and adjacent across a warp, as the state's SH part
// starts at an offset of L floats, which no vector access can count on.  (One
// value per thread and iteration moved 4.6 TB/s, or 6.7 TB/s with 16-byte vectors
// where the leaves were a multiple of 4: the RMSprop step of 4,026,531 leaves at
// degree 3 860 -> 556 us = 7.1 TB/s, of 4,026,528 leaves 587 -> 551 us, of 4.0 M
// leaves at degree 2, whose records are padded, 541 -> 442 us; 120 M values with
// gradients anywhere: Adam 514 -> 498 us at degree 1, 661 -> 597 us at degree 2, SGD
// 217 -> 203 and 444 -> 301 us.)
constexpr int kStepBlock = 256, kStepPer = 8, kStepUnit = kStepBlock * kStepPer;

template <int KIND, int K>
__global__ void __launch_bounds__(kStepBlock) k_step(StepParams sp, float *__restrict__ sigma, float *__restrict__ sh,
                                                     const float *__restrict__ gs, const float *__restrict__ gsh,
                                                     float *__restrict__ state)
{
    constexpr int K3 = 3 * K, STRIDE = sh_stride<float>(K);
    const int64_t N = sp.L * (1 + K3);
    const int64_t sig_units = (sp.L + kStepUnit - 1) / kStepUnit;
    const int64_t units = sig_units + (sp.L * K3 + kStepUnit - 1) / kStepUnit;
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        const bool dens = u < sig_units;
        const int64_t base = (dens ? u : u - sig_units) * kStepUnit, end = dens ? sp.L : sp.L * K3;
        const int64_t row0 = base / K3;
        const int rem = (int)(base - row0 * K3);
        const float *grad = dens ? gs : gsh;
        float *param = dens ? sigma : sh, *st = dens ? state : state + sp.L;
        const float lr = dens ? sp.lr_sigma : sp.lr_sh;
        float x[kStepPer], g[kStepPer], m[kStepPer], v[kStepPer];
        // a value's place in the padded records: its row and column, by 32-bit division by a constant
        auto at = [&](int i) -> int64_t {
            const int e = i * kStepBlock + (int)threadIdx.x;
            if (dens || STRIDE == K3) return base + e;
            const unsigned r = (unsigned)(rem + e) / (unsigned)K3;
            return (row0 + r) * STRIDE + ((unsigned)(rem + e) - r * (unsigned)K3);
        };
#pragma unroll
        for (int i = 0; i < kStepPer; ++i) {
            const int64_t j = base + i * kStepBlock + threadIdx.x;
            m[i] = v[i] = x[i] = g[i] = 0.f;
            if (j < end) {
                x[i] = param[at(i)];
                g[i] = grad[j];
                load_state<KIND>(st, N, j, m[i], v[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < kStepPer; ++i) {
            const int64_t j = base + i * kStepBlock + threadIdx.x;
            if (j < end) {
                param[at(i)] = step_one<KIND>(sp, x[i], g[i], lr, m[i], v[i]);
                store_state<KIND>(st, N, j, m[i], v[i]);
            }
        }
    }
}

template <int KIND>
void launch_step_kind(const StepParams &sp, int K, unsigned grid, float *sig, float *sh, const float *gs,
                      const float *gsh, float *state, cudaStream_t s)
{
    switch (K) {
    case 1: k_step<KIND, 1><<<grid, kStepBlock, 0, s>>>(sp, sig, sh, gs, gsh, state); break;
    case 4: k_step<KIND, 4><<<grid, kStepBlock, 0, s>>>(sp, sig, sh, gs, gsh, state); break;
    case 9: k_step<KIND, 9><<<grid, kStepBlock, 0, s>>>(sp, sig, sh, gs, gsh, state); break;
    case 16: k_step<KIND, 16><<<grid, kStepBlock, 0, s>>>(sp, sig, sh, gs, gsh, state); break;
    default: k_step<KIND, 25><<<grid, kStepBlock, 0, s>>>(sp, sig, sh, gs, gsh, state); break;
    }
}

// ---- MSE loss of a ray batch: L = mean over n*3 of (rgb - target)^2 --------
// (the blocks' sums joined in double: float reductions of up to 4,096 blocks were off
// by 8e-7 of the loss at 200,003 random rays and by 4.6e-5 at 2^20 whose errors were
// all alike; a training step of 2^18 rays 1529 -> 1533 us)
__global__ void k_mse(int64_t n3, const float *rgb, const float *target, float *grad, LossSum *sum, float *loss)
{
    const float scale = 2.f / (float)n3;
    float acc = 0.f;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n3; j += (int64_t)gridDim.x * blockDim.x) {
        const float r = rgb[j] - target[j];
        acc = fmaf(r, r, acc);
        if (grad) grad[j] = scale * r;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    finish_loss<kFlatBlock>((double)acc, sum, (double)n3, loss);
}

// ---- pixel rays (the camera expression of the public header) ----------------
__global__ void k_camera_rays(const pot_camera *cams, int n_cams, int64_t per_cam, int W, int64_t n,
                              const int64_t *pixels, float *o, float *d)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t pix = pixels ? pixels[k] : k;
        int64_t cam = pix / per_cam;
        if (cam < 0 || cam >= n_cams) cam = cam < 0 ? 0 : n_cams - 1;  // guarded by the host check
        const int64_t rem = pix - cam * per_cam;
        const int j = (int)(rem / W), i = (int)(rem - (int64_t)j * W);
        const pot_camera *c = cams + cam;
        const float xc = __fdiv_rn(__fsub_rn(__fadd_rn((float)i, 0.5f), c->cx), c->fx);
        const float yc = -__fdiv_rn(__fsub_rn(__fadd_rn((float)j, 0.5f), c->cy), c->fy);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            d[3 * k + r] = __fsub_rn(__fadd_rn(__fmul_rn(c->c2w[r][0], xc), __fmul_rn(c->c2w[r][1], yc)),
                                     c->c2w[r][2]);
            o[3 * k + r] = c->c2w[r][3];
        }
    }
}

__global__ void k_pixel_range(int64_t n, const int64_t *pixels, int64_t total, unsigned *flag)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        if (pixels[k] < 0 || pixels[k] >= total) atomicOr(flag, 1u);
}

unsigned grid_n(int64_t n)
{
    int64_t b = (n + 255) / 256;
    return (unsigned)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

}  // namespace

cudaError_t launch_backward(const RenderParams &r, const float *grad_rgb, const float *rgb_fwd, float *grad_sigma,
                            float *grad_sh, int dtype, int K, cudaStream_t s)
{
    BackwardParams bp{r, grad_rgb, rgb_fwd, grad_sigma, grad_sh, nullptr, nullptr, nullptr, nullptr, 0.f};
    const int mode = rgb_fwd ? kGradAndColour : kGrad;
    switch (dtype) {
    case POT_F32: return launch_backward_t<float>(bp, K, mode, s);
    case POT_F16: return launch_backward_t<__half>(bp, K, mode, s);
    default: return launch_backward_t<__nv_bfloat16>(bp, K, mode, s);
    }
}

cudaError_t launch_mse_backward(const RenderParams &r, const float *target, float *rgb_out, float *loss, LossSum *sum,
                                float *grad_sigma, float *grad_sh, int dtype, int K, cudaStream_t s)
{
    BackwardParams bp{r, nullptr, nullptr, grad_sigma, grad_sh, target, loss, sum, rgb_out,
                      2.f / (3.f * (float)r.n_rays)};
    switch (dtype) {
    case POT_F32: return launch_backward_t<float>(bp, K, kMseTarget, s);
    case POT_F16: return launch_backward_t<__half>(bp, K, kMseTarget, s);
    default: return launch_backward_t<__nv_bfloat16>(bp, K, kMseTarget, s);
    }
}

cudaError_t launch_backward_recorded(const RenderParams &r, int64_t n_leaves, const SegmentBuffer &sb,
                                     const SegmentBins *bins, const float *grad_rgb, const float *rgb_fwd,
                                     float *grad_sigma, float *grad_sh, int dtype, int K, cudaStream_t s)
{
    SegBackwardParams q{sb,      r.n_rays,   n_leaves, nullptr,    nullptr,   r.sigma,
                        r.sh,    r.ray_d,    grad_rgb, rgb_fwd,    grad_sigma, grad_sh};
    cudaError_t e;
    if (bins) {
        const SegBinParams bq{q, *bins};
        switch (dtype) {
        case POT_F32: e = launch_leaf_order_t<float>(bq, K, s); break;
        case POT_F16: e = launch_leaf_order_t<__half>(bq, K, s); break;
        case POT_BF16: e = launch_leaf_order_t<__nv_bfloat16>(bq, K, s); break;
        default: return cudaErrorInvalidValue;
        }
    } else {
        switch (dtype) {
        case POT_F32: e = launch_segment_backward_t<float>(q, K, s); break;
        case POT_F16: e = launch_segment_backward_t<__half>(q, K, s); break;
        case POT_BF16: e = launch_segment_backward_t<__nv_bfloat16>(q, K, s); break;
        default: return cudaErrorInvalidValue;
        }
    }
    if (e != cudaSuccess) return e;
    // the fallback: every ray walked again, only if the records overflowed
    BackwardParams bp{r, grad_rgb, rgb_fwd, grad_sigma, grad_sh, nullptr, nullptr, nullptr, nullptr, 0.f,
                      sb.state + 1};
    switch (dtype) {
    case POT_F32: return launch_backward_t<float>(bp, K, kGradAndColour, s);
    case POT_F16: return launch_backward_t<__half>(bp, K, kGradAndColour, s);
    default: return launch_backward_t<__nv_bfloat16>(bp, K, kGradAndColour, s);
    }
}

cudaError_t launch_step(pot_tree *t, int kind, float lr_sigma, float lr_sh, float alpha, float beta1, float beta2,
                        float eps, int step, const float *gs, const float *gsh, float *state, cudaStream_t s)
{
    StepParams sp;
    sp.L = t->n_leaves;
    sp.lr_sigma = lr_sigma;
    sp.lr_sh = lr_sh;
    sp.alpha = alpha;
    sp.beta1 = beta1;
    sp.beta2 = beta2;
    sp.eps = eps;
    sp.bc1 = (float)(1.0 - std::pow((double)beta1, (double)step));
    sp.bc2 = (float)(1.0 - std::pow((double)beta2, (double)step));
    sp.zero_stays = eps > 0.f && (kind != POT_ADAM || sp.bc2 > 0.f);
    if (sp.L == 0) return cudaSuccess;
    int64_t units = (sp.L + kStepUnit - 1) / kStepUnit + (sp.L * 3 * t->K + kStepUnit - 1) / kStepUnit;
    if (units > (1 << 30)) units = 1 << 30;
    const unsigned g = (unsigned)units;
    float *sig = static_cast<float *>(t->sigma);
    float *sh = static_cast<float *>(t->sh);
    if (kind == POT_SGD) launch_step_kind<POT_SGD>(sp, t->K, g, sig, sh, gs, gsh, state, s);
    else if (kind == POT_RMSPROP) launch_step_kind<POT_RMSPROP>(sp, t->K, g, sig, sh, gs, gsh, state, s);
    else launch_step_kind<POT_ADAM>(sp, t->K, g, sig, sh, gs, gsh, state, s);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_mse(int64_t n, const float *rgb, const float *target, float *grad, float *loss, LossSum *sum,
                       cudaStream_t s)
{
    k_mse<<<grid_n(3 * n), kFlatBlock, 0, s>>>(3 * n, rgb, target, grad, sum, loss);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_camera_rays(const pot_camera *d_cams, int n_cams, int W, int H, int64_t n, const int64_t *pixels,
                               float *o, float *d, unsigned *d_flag, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    if (pixels) {
        k_pixel_range<<<grid_n(n), 256, 0, s>>>(n, pixels, (int64_t)n_cams * W * H, d_flag);
        count_launch();
    }
    k_camera_rays<<<grid_n(n), 256, 0, s>>>(d_cams, n_cams, (int64_t)W * H, W, n, pixels, o, d);
    count_launch();
    return cudaGetLastError();
}

}  // namespace pot
