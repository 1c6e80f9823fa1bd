// pot_render.cuh -- forward render kernel of the PlenOctree path (sm_103a).
//
// One warp renders one tile of 32 rays at a time (4 x 8 pixels of a camera,
// or 32 consecutive explicit rays); warps take tiles from a global counter
// until none is left (persistent grid, one wave of resident blocks).  Per ray:
//   a1 pinhole ray (fp32 expression of the public header)
//   a2 clip to the tree box and to [near, far]
//   a3 locate the cell: one load from the tree's cell index (leaf, or the
//      empty box around the voxel; two loads in the brick layout), or, for
//      trees without one, a descent of the child array from the deepest
//      ancestor the new voxel shares with the previous one (ancestor stack in
//      shared memory)
//   a4 exit time of the cell (double-float plane crossings, the earliest of
//      three chosen with selects); an empty node of any size is crossed in one
//      step (Sec. 3.2 "Rendering")
//   a5 leaf fetch: sigma and the SH record in 32-byte (or 16-byte) vector loads
//   a6 colour: sigmoid of the SH dot product, basis evaluated once per ray
//      because it is constant along the ray (App. B.3.2)
//   a7 composite: w = T (1 - exp(-max(sigma,0) delta)), C += w c (Eq. 1)
//   a8 stop once T < gamma (Sec. 3.2), add T * bg (App. B.3.2), store.
#pragma once

#include "pot_device.cuh"
#include "pot_internal.h"

namespace pot {

constexpr int kBlock = 256;
#ifndef POT_RENDER_MIN_BLOCKS
#define POT_RENDER_MIN_BLOCKS 4  // resident blocks per SM the register budget is cut for (64 registers)
#endif

// Fixed-point ray times.  A walk measures time from the clip range's entry
// tin in units of 2^-s, s such that the whole clip range [tin, tout] is at
// least 2^49 and below 2^50 units, and keeps it in 64-bit integers.  The
// crossing times of one axis's planes are then an arithmetic progression
// nx, nx + hs, nx + 2 hs, ... whose terms are exact sums: advancing by one
// plane, or by the j planes of a box, gives the same time whichever way the
// plane is reached, so leaf segments do not depend on how empty space is
// stepped over, and comparisons need no error bounds.  nx and hs are rounded
// from double-float values once per ray (a voxel is about 2^41 units at
// depth 9 and 2^38 at depth 12: rounding hs moves a crossing by at most 2^-33
// and 2^-27 of a voxel, the double-float inputs by about as much).
// Axes along which the ray does not move, and planes it would reach only after
// its range, have nx or hs = kTimeNever; nx + j hs stays below 2^63 for every
// j < 2^kMaxDepth.
constexpr int64_t kTimeNever = 1ll << 50;
constexpr int kTimeRangeExp = 49;

// (a - tin) 2^s, not below 0, s split into the factors s1 s2 so that neither
// overflows.  (The parts of a crossing time need not be ordered: where a
// plane's offset from the origin cancels, all of it is in a.lo.)
__device__ __forceinline__ int64_t fixed_time(df a, df tin, float s1, float s2)
{
    float ah, al, hi, e;
    two_sum(a.hi, a.lo, ah, al);
    two_sum(ah, -tin.hi, hi, e);
    const float lo = __fadd_rn(e, __fsub_rn(al, tin.lo));
    const float f = __fmul_rn(__fmul_rn(hi, s1), s2);
    if (!(f < (float)kTimeNever)) return kTimeNever;  // also NaN
    const int64_t t = __float2ll_rn(fmaxf(f, -(float)kTimeNever)) + __float2ll_rn(__fmul_rn(__fmul_rn(lo, s1), s2));
    return t < 0 ? 0 : t;
}

__device__ __forceinline__ float exp2_int(int x) { return __int_as_float((127 + x) << 23); }

// One ray's walk through the octree (a2-a4) as resumable state: begin() sets
// the ray up (clip, locate, first cell); cross_empty() and cross_leaf() advance
// past the cell the ray is in, the latter calling vis(leaf, delta, Y) for a
// segment of positive length (Y: the SH basis at the ray direction); all three
// return false once the walk is over (vis returned true, far clip, or the ray
// left the box).  The next cell is located before vis runs on the current one,
// so that its load overlaps the shading.
//
// The walk runs in the mirrored grid in which every component of the direction
// is >= 0 (voxel q of an axis with d < 0 stands for voxel R - 1 - q): every
// step adds to coordinates, boxes are left through their upper faces, and the
// mirror is one XOR of the cell's index offset, whose fields are bit fields of
// the coordinates.
//
// What bounds it: issue slots, and the integer pipe among them (a 64-bit
// compare or add takes two of its half-rate instructions).  The walk it
// replaced recomputed three double-float crossing times at every step (about 45
// instructions) and located positions by an fp32 estimate with a branch to an
// exact test near faces, its per-axis constants in shared memory (three 16-byte
// loads per step).  Both, 40 views of 800 x 800 on the depth-9 tree: f16 leaves
// 8.30 -> 6.55 ms (warp instructions 7.23 -> 5.45 G), f32 9.01 -> 8.02 ms (L1
// data-pipe wavefronts 2.08 -> 1.81 G); one 256 x 256 view of a depth-8 tree
// 137 -> 95 us; weights of 6 views 1048 -> 831 us.  Tried: separate inner loops
// for empty boxes and leaves (lanes at a leaf wait for the others: 8.32 ms for
// f16), one shared exit-time computation for both kinds of cell (6.28 against
// 6.05 ms).
template <int K, typename T>
struct Walker {
    int64_t nx[3], hs[3];  // time of the next plane and between planes, per axis
    int64_t t, tout;
    int q[3];              // mirrored voxel
    uint32_t flip;         // the mirror, in the form of the tree's cell lookup
    float unit;            // world length of one time unit
    int cell;              // entry of voxel q: leaf >= 0, or an empty box (cell_code_*)
    int lvl_valid, step_i;
    // rows of shared memory: the per-ray SH basis, and 1 / hs per axis (read
    // only where a box of more than one voxel is left), which saves registers
    float *ysm;
    float4 *st;
    __device__ __forceinline__ SmemY<K, kBlock> Y() const { return {ysm}; }

    // a3: the entry of mirrored voxel q: one load from the cell index when the
    // tree has one (two in the brick layout), else a descent from the deepest
    // ancestor q shares with voxel pq (whose path the stack holds up to
    // lvl_valid)
    __device__ __forceinline__ int locate(const RenderParams &p, int32_t *stk, const int pq[3])
    {
        const int D = p.depth;
        if (p.cells) {
            if (!p.btab)
                return __ldg(p.cells + (cell_index_offset((uint32_t)q[0], (uint32_t)q[1], (uint32_t)q[2], D) ^ flip));
            const uint32_t bk = brick_of((uint32_t)q[0], (uint32_t)q[1], (uint32_t)q[2], D);
            const uint32_t in = in_brick((uint32_t)q[0], (uint32_t)q[1], (uint32_t)q[2]);
            // brick layout: the brick's code, or its stored entries
            const uint32_t f = flip >> 27, fin = ((f & 1u) | (f & 2u) << 1 | (f & 4u) << 2) * 3u;
            const int b = __ldg(p.btab + (bk ^ (flip & 0x7FFFFFFu)));
            return b >= 0 ? __ldg(p.cells + (((int64_t)b << 6) | (in ^ fin))) : b;
        }
        const unsigned diff = (unsigned)((q[0] ^ pq[0]) | (q[1] ^ pq[1]) | (q[2] ^ pq[2]));
        const int lc = diff ? D - 32 + __clz(diff) : D - 1;  // level of the common ancestor
        int l = min(lc, lvl_valid);
        int node = stk[l * kBlock];
        int out = 0;
        for (; l < D; ++l) {
            const int b = D - 1 - l;
            const int s = ((((q[0] >> b) & 1) << 2) | (((q[1] >> b) & 1) << 1) | ((q[2] >> b) & 1)) ^ (int)flip;
            const int c = __ldg(p.child + (int64_t)node * 8 + s);
            if (c > 0 && l < D - 1) {
                node = c;
                stk[(l + 1) * kBlock] = c;
                continue;
            }
            out = c < 0 ? -c - 1 : cell_code_node(l + 1, D);  // an empty slot: an empty node of level l + 1
            break;
        }
        lvl_valid = min(l, D - 1);
        return out;
    }

    __device__ __forceinline__ bool begin(const RenderParams &p, int32_t *stk, const float o[3], const float d[3],
                                          float near, float far)
    {
        const int R = p.R;
        const float h = p.h, invh = p.invh;
        const float len = sqrtf(fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2])));
        if (!(len > 0.f) || !(len < 3.0e38f)) return false;
        const float invlen = __frcp_rn(len);
        {
            float Yt[K];
            sh_basis<K>(d[0] * invlen, d[1] * invlen, d[2] * invlen, Yt);
            SmemY<K, kBlock>::store(ysm, Yt);
        }
        float Ahi[3], Alo[3], rd[3];  // A = lo - o exactly, 1 / d
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            two_sum(p.lo[a], -o[a], Ahi[a], Alo[a]);
            rd[a] = d[a] != 0.f ? __frcp_rn(d[a]) : 0.f;
        }
        // a2: clip range in units of the ray parameter t (position o + t d)
        df tin = {near * invlen, 0.f}, tend = {far * invlen, 0.f};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (d[a] == 0.f) {
                float s, e;
                two_sum(o[a], -p.lo[a], s, e);
                const bool inside = (s > 0.f || (s == 0.f && e >= 0.f)) && (s < p.size || (s == p.size && e < 0.f));
                if (!inside) return false;
            } else {
                df t0 = cross_time(0, h, Ahi[a], Alo[a], d[a], rd[a]);
                df t1 = cross_time(R, h, Ahi[a], Alo[a], d[a], rd[a]);
                if (d[a] < 0.f) {
                    df tmp = t0;
                    t0 = t1;
                    t1 = tmp;
                }
                if (df_lt(tin, t0)) tin = t0;
                if (df_lt(t1, tend)) tend = t1;
            }
        }
        if (!df_lt(tin, tend)) return false;
        // the unit of time: 2^-s, s from the exponent of the range
        const int s = kTimeRangeExp + 127 - (int)(__float_as_uint(df_sub(tend, tin)) >> 23);
        const float s1 = exp2_int(s / 2), s2 = exp2_int(s - s / 2);
        unit = __fmul_rn(__fmul_rn(len, exp2_int(-(s / 2))), exp2_int(s / 2 - s));
        tout = fixed_time(tend, tin, s1, s2);
        flip = 0;
        float rh[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            // error bound of the fp32 voxel-coordinate estimate, in voxels
            const float margin = (fabsf(tend.hi * d[a]) + fabsf(Ahi[a])) * invh * 3.8146973e-6f + 1e-6f;
            const int v = min(max(locate_axis(tin, d[a], Ahi[a], Alo[a], h, invh, margin), 0), R - 1);
            const bool neg = d[a] < 0.f;
            q[a] = neg ? R - 1 - v : v;
            if (neg) flip |= 4u >> a;
            nx[a] = hs[a] = kTimeNever;
            if (d[a] != 0.f) {
                nx[a] = fixed_time(cross_time(neg ? v : v + 1, h, Ahi[a], Alo[a], d[a], rd[a]), tin, s1, s2);
                const float ard = fabsf(rd[a]), th = __fmul_rn(h, ard);
                hs[a] = fixed_time({th, __fmul_rn(__fmaf_rn(-th, fabsf(d[a]), h), ard)}, {0.f, 0.f}, s1, s2);
            }
            // planes per 2^20 units, a little below the true value (see cross_empty)
            rh[a] = __fmul_rn(__fdividef(1048576.f, __ll2float_rn(hs[a])), 1.f - 9.5367432e-7f);
        }
        *st = make_float4(rh[0], rh[1], rh[2], 0.f);
        // the mirror as an XOR mask: child slots (no index), entry offsets (dense), or brick offsets
        // with a flag per axis of the in-brick offset in bits 27-29 (brick layout)
        if (p.cells) {
            const uint32_t fx = flip & 4u ? R - 1 : 0, fy = flip & 2u ? R - 1 : 0, fz = flip & 1u ? R - 1 : 0;
            const uint32_t bk = brick_of(fx, fy, fz, p.depth);
            flip = p.btab ? bk | flip << 27 : (bk << 6) | in_brick(fx, fy, fz);
        }
        lvl_valid = 0;
        if (!p.cells) stk[0] = 0;  // the stack exists only for trees without a cell index
        cell = locate(p, stk, q);
        t = 0;
        step_i = 0;
        return true;
    }

    template <typename Visitor>
    __device__ __forceinline__ bool step(const RenderParams &p, int32_t *stk, Visitor &vis)
    {
        const int leaf = cell;  // < 0: an empty box
        const int pq[3] = {q[0], q[1], q[2]};
        int64_t texit;
        // a4: exit time of the current cell, the earliest of its upper faces, and
        // the voxel entered there: every plane with a time <= texit has been
        // crossed (past a leaf, one; a tie's other plane is then crossed in a
        // step of no length).  The next cell is located ahead of shading the
        // current leaf.
        if (leaf >= 0) {
            const bool x01 = nx[0] <= nx[1];
            const int64_t t01 = x01 ? nx[0] : nx[1];
            const bool x2 = nx[2] < t01;
            texit = x2 ? nx[2] : t01;
            const bool x[3] = {!x2 && x01, !x2 && !x01, x2};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (x[a]) {
                    nx[a] += hs[a];
                    ++q[a];
                }
            }
        } else {
            int64_t ex[3] = {nx[0], nx[1], nx[2]};
            const uint32_t m = cell & 0xFFFF, e = (cell >> 16) & 0xFF;
#pragma unroll
            for (int a = 0; a < 3; ++a)
                ex[a] += (int64_t)((uint64_t)((m & ~(uint32_t)q[a]) + e) * (uint64_t)hs[a]);
            texit = min(ex[0], min(ex[1], ex[2]));
            // planes crossed = floor((texit - nx) / hs) + 1, by an fp32 estimate that is exact or one too low
            // (its factor and its addend are low by 2^-20, over the rounding errors, and at most 2^12 planes
            // are crossed), then the exact test of the next plane
            const float4 rh = *st;
            const float r[3] = {rh.x, rh.y, rh.z};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const uint32_t c = __float2uint_rd(fmaf((float)(int)((texit - nx[a]) >> 20), r[a], 1.f - 9.5367432e-7f));
                nx[a] += (int64_t)((uint64_t)c * (uint64_t)hs[a]);
                q[a] += c;
                if (nx[a] <= texit) {
                    nx[a] += hs[a];
                    ++q[a];
                }
            }
        }
        const bool last = texit >= tout, capped = !last && step_i >= p.step_cap;
        if (capped) *p.err = 1u;  // device error word: a plain store, no branch around an atomic
        bool stop = last || capped;
        ++step_i;
        // outside the grid: its far planes' times may differ from tout by the rounding of hs
        if (!stop && (unsigned)(q[0] | q[1] | q[2]) >= (unsigned)p.R) stop = true;
        if (!stop) cell = locate(p, stk, pq);
        const int64_t dt = min(texit, tout) - t;
        t = texit;
        if (leaf >= 0 && dt > 0) {
            if (vis(leaf, __fmul_rn(__ll2float_rn(dt), unit), Y())) return false;
        }
        return !stop;
    }
};

// Per-thread scratch of a walk in shared memory: the SH basis (SmemY) and the
// walker's row of per-axis constants, and the ancestor stack [kMaxDepth][kBlock] in
// dynamic shared memory, which a launch provides (walk_smem_bytes) only when
// some tree of it has no cell index; without it the space goes to L1.
// Declared once per kernel.
#define POT_WALK_SHARED(K)                                          \
    extern __shared__ int32_t walk_stack_sh[];                      \
    __shared__ float4 walk_y_sh[kBlock * SmemY<K, kBlock>::kRow4];   \
    __shared__ float4 walk_st_sh[kBlock];                           \
    int32_t *stk = walk_stack_sh + threadIdx.x;                     \
    float *ysm = reinterpret_cast<float *>(walk_y_sh + threadIdx.x * SmemY<K, kBlock>::kRow4); \
    float4 *wst = walk_st_sh + threadIdx.x;                         \
    (void)ysm;                                                      \
    (void)wst;

inline size_t walk_smem_bytes(bool need_stack)
{
    return need_stack ? sizeof(int32_t) * kMaxDepth * kBlock : 0;
}

// Grid of a persistent walk kernel: one wave of resident blocks (SMs x blocks
// per SM for this kernel and shared memory), no more blocks than tiles need.
template <typename Fn>
cudaError_t persistent_grid(Fn fn, size_t smem, int64_t n_tiles, int max_blocks, unsigned *grid)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBlock, smem);
    if (e != cudaSuccess) return e;
    int64_t blocks = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    const int64_t need = (n_tiles + (kBlock / 32) - 1) / (kBlock / 32);
    if (blocks > need) blocks = need;
    if (max_blocks > 0 && blocks > max_blocks) blocks = max_blocks;
    if (blocks < 1) blocks = 1;
    *grid = (unsigned)blocks;
    return cudaSuccess;
}

// The whole walk of one ray.
template <int K, typename T, typename Visitor>
__device__ __forceinline__ void walk_ray(const RenderParams &p, int32_t *stk, float *ysm, float4 *wst,
                                         const float o[3], const float d[3], float near, float far, Visitor &vis)
{
    Walker<K, T> w;
    w.ysm = ysm;
    w.st = wst;
    if (!w.begin(p, stk, o, d, near, far)) return;
    while (w.step(p, stk, vis)) {
    }
}

// a5-a8 for one leaf segment: fetch, colour, composite, early stop.
template <int K, typename T, bool COUNT>
struct ShadeVisitor {
    const T *sig_arr;
    const T *sh_arr;
    uint8_t *touched;
    float gamma;
    float col[3];
    float Tr;
    int nseg;
    const void *cb;  // codebook (cb16 leaves only)
    template <typename YT>
    __device__ __forceinline__ bool operator()(int leaf, float delta, const YT &Y)
    {
        const float sig = fmaxf(Store<T>::load_sigma(sig_arr, leaf), 0.f);
        float x[3];
        leaf_colour_dot<K, T>(sh_arr, leaf, Y, x, cb);
        const float e = exp_ftz(-sig * delta);  // transmittance of the segment
        const float w = Tr * (1.f - e);
#pragma unroll
        for (int c = 0; c < 3; ++c) col[c] = fmaf(w, sigmoidf_(x[c]), col[c]);
        Tr *= e;
        if (COUNT) {
            ++nseg;
            touched[leaf] = 1;
        }
        return Tr < gamma;  // a8 early stop (gamma = 0 never stops)
    }
};

// Ray (origin, direction, clip range, output index) of slot `slot` (0..31) of
// tile `tile`: kTileW x kTileH pixels of a camera (tiles interleaved over groups of
// adjacent cameras) or 32 consecutive explicit rays.  False for slots outside
// the image or past the last ray.
template <bool CAMS>
__device__ __forceinline__ bool tile_ray(const RenderParams &p, unsigned long long tile, int slot, float o[3],
                                         float d[3], float &near, float &far, int64_t &ray)
{
    if (CAMS) {
        // tiles of a group of G consecutive cameras are interleaved: the same
        // tile of each camera of the group in turn, so neighbouring views
        // (which touch nearly the same leaves) share L1/L2
        // 32-bit arithmetic: the host keeps tile counts below 2^32
        const uint32_t tl = (uint32_t)tile;
        const uint32_t G = (uint32_t)p.view_group;
        const uint32_t per_group = (uint32_t)p.tiles_per_cam * G;
        const uint32_t group = tl / per_group;
        const uint32_t in_group = tl - group * per_group;
        const uint32_t gsize = min(G, (uint32_t)p.n_cams - group * G);
        const int64_t cam = (int64_t)(group * G + in_group % gsize);
        const uint32_t rem = in_group / gsize;
        const int ty = (int)(rem / (uint32_t)p.tiles_x);
        const int tx = (int)(rem - (uint32_t)ty * (uint32_t)p.tiles_x);
        const int i = tx * kTileW + (slot % kTileW);
        const int j = ty * kTileH + (slot / kTileW);
        if (i >= p.W || j >= p.H) return false;
        ray = (cam * p.H + j) * p.W + i;
        const pot_camera *c = p.cams + cam;
        // a1: pixel ray, each operation rounded once in the stated order
        const float xc = __fdiv_rn(__fsub_rn(__fadd_rn((float)i, 0.5f), c->cx), c->fx);
        const float yc = -__fdiv_rn(__fsub_rn(__fadd_rn((float)j, 0.5f), c->cy), c->fy);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            d[r] = __fsub_rn(__fadd_rn(__fmul_rn(c->c2w[r][0], xc), __fmul_rn(c->c2w[r][1], yc)), c->c2w[r][2]);
            o[r] = c->c2w[r][3];
        }
        near = c->near;
        far = c->far;
        return true;
    }
    ray = (int64_t)tile * 32 + slot;
    if (ray >= p.n_rays) return false;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        o[r] = __ldg(p.ray_o + 3 * ray + r);
        d[r] = __ldg(p.ray_d + 3 * ray + r);
    }
    near = p.near;
    far = p.far;
    return true;
}

template <int K, typename T, bool COUNT>
__device__ __forceinline__ void store_ray(const RenderParams &p, int64_t ray, const ShadeVisitor<K, T, COUNT> &v)
{
#pragma unroll
    for (int c = 0; c < 3; ++c) p.rgb[3 * ray + c] = fmaf(v.Tr, p.bg[c], v.col[c]);
    if (p.t_final) p.t_final[ray] = v.Tr;
    if (COUNT) p.seg_count[ray] = v.nseg;
}

// Forward render, one tile per warp at a time: the warp takes the next tile
// once all 32 of its rays are done.
template <int K, typename T, bool CAMS, bool COUNT>
__global__ void __launch_bounds__(kBlock, POT_RENDER_MIN_BLOCKS) render_kernel(const RenderParams p)
{
    POT_WALK_SHARED(K)
    const int lane = threadIdx.x & 31;
    const T *sig_arr = static_cast<const T *>(p.sigma);
    const T *sh_arr = static_cast<const T *>(p.sh);
    for (;;) {
        unsigned long long tile = 0;
        if (lane == 0) tile = atomicAdd(p.tile_counter, 1ull);
        tile = __shfl_sync(0xffffffffu, tile, 0);
        if (tile >= (unsigned long long)p.n_tiles) break;
        float o[3], d[3], near, far;
        int64_t ray;
        if (tile_ray<CAMS>(p, tile, lane, o, d, near, far, ray)) {
            ShadeVisitor<K, T, COUNT> v{sig_arr, sh_arr, p.leaf_touched, p.gamma, {0.f, 0.f, 0.f}, 1.f, 0,
                                        p.codebook};
            walk_ray<K, T>(p, stk, ysm, wst, o, d, near, far, v);
            store_ray<K, T, COUNT>(p, ray, v);
        }
    }
}

template <typename T>
cudaError_t launch_render_t(const RenderParams &p, int K, bool cams, bool count, cudaStream_t s,
                            int max_blocks)
{
    using Fn = void (*)(const RenderParams);
    Fn fn = nullptr;
#define POT_PICK(KK)                                                                            \
    if (K == KK)                                                                                \
        fn = cams ? (count ? render_kernel<KK, T, true, true> : render_kernel<KK, T, true, false>) \
                  : (count ? render_kernel<KK, T, false, true> : render_kernel<KK, T, false, false>);
    POT_PICK(1)
    POT_PICK(4)
    POT_PICK(9)
    POT_PICK(16)
    POT_PICK(25)
#undef POT_PICK
    if (!fn) return cudaErrorInvalidValue;
    const size_t smem = walk_smem_bytes(p.cells == nullptr);
    unsigned grid = 0;
    cudaError_t e = persistent_grid(fn, smem, p.n_tiles, max_blocks, &grid);
    if (e != cudaSuccess) return e;
    fn<<<grid, kBlock, smem, s>>>(p);
    count_launch();
    return cudaGetLastError();
}

}  // namespace pot
