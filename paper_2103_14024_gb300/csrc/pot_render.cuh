// pot_render.cuh -- forward render kernel of the PlenOctree path (sm_103a).
//
// One warp renders one tile of 32 rays at a time (4 x 8 pixels of a camera,
// or 32 consecutive explicit rays).  Large calls: one wave of resident blocks,
// whose warps take tiles from a global counter until none is left; calls whose
// tiles are all resident at once: a tile per warp by its place in the grid, or
// a part of one (one_wave, next_tile).  Per ray:
//   a1 pinhole ray (fp32 expression of the public header)
//   a2 clip to the tree box and to [near, far]
//   a3 locate the cell: one load from the tree's cell index (leaf, or the
//      empty box around the voxel; two loads in the brick layout), or, for
//      trees without one, a descent of the child array from the deepest
//      ancestor the new voxel shares with the previous one (ancestor stack in
//      shared memory)
//   a4 exit time of the cell (64-bit fixed point, the earliest of three upper
//      faces); an empty node of any size is crossed in one step (Sec. 3.2
//      "Rendering")
//   a5 leaf fetch: sigma and the SH record in 32-byte (or 16-byte) vector loads
//   a6 colour: sigmoid of the SH dot product, basis evaluated once per ray
//      because it is constant along the ray (App. B.3.2)
//   a7 composite: w = T (1 - exp(-max(sigma,0) delta)), C += w c (Eq. 1)
//   a8 stop once T < gamma (Sec. 3.2), add T * bg (App. B.3.2), store.
#pragma once

#include "pot_device.cuh"
#include "pot_internal.h"

namespace pot {

// How a walk finds the cell of a voxel: the dense cell index, its brick
// layout, or whichever the tree has (the descent of the child array included).
enum Lookup { kLookDense, kLookBrick, kLookAny };

// Threads per block of the walk kernels, and the blocks per SM that their
// register budget is cut for: 6 blocks, 24 warps, 80 registers with the dense
// index.  The walk and the shading need about 75; at 64 registers (32 warps) the
// loop spills, which lone views, bound by the latency of their longest rays,
// pay for (256 x 256 f16 109 against 89 us, 800 x 800 f32 350 against 320 us)
// and full launches do not notice (40 views: f16 5.68 against 5.65 ms, f32 7.31
// against 7.32 ms).  72 registers (28 warps): 89 us, 340 us, 5.65 ms, 7.33 ms.
// With bricks a step waits for two loads in turn, and more warps are better (one
// full-HD view at depth 10: 28 warps 744, 32 warps 768, 24 warps 801 us), but float
// records of degree 3 and 4 keep 24: at 72 registers their loads wait for one
// another, or spill (nine 100 x 100 views of the depth-8 degree-4 tree 263 -> 221 us,
// of the depth-9 degree-3 tree 360 -> 279 us, 20 of 800 x 800 2750 -> 2745 and
// 3497 -> 3455 us; 16-bit records of degree 4 2230 -> 2249 us, so they stay at 28).
// Explicit rays need not have neighbours in their warp, and then every lane
// brings its own lines: with the dense index fewer resident warps keep more of them in L1.  4 blocks
// against 6, 2^18 random pixels of 100 views on the depth-9 tree (one in four
// meets a leaf): render_rays 368 against 400 us, where every ray meets a leaf
// 725 against 934 us; the recording forward 440 against 494 and 860 against
// 1118 us (3 and 2 blocks the same within 1 %, as their registers allow 4).
// The descent of the child array, a chain of loads, wants 24 warps there (no
// index, 2^18 random pixels: 736 against 805 us), and trees with bricks run the same
// instance (depth 9, degree 3, 200,000 random rays with bricks / without an index:
// 24 warps 350 / 497, 20 warps 374 / 545, 28 warps 334 / 487, 32 warps 425 / 559 us;
// 50,000 rays 229 / 354, 222 / 340, 282 / 411, 362 / 501 us).
constexpr int kBlock = 128;
#ifndef POT_RENDER_MIN_BLOCKS
#define POT_RENDER_MIN_BLOCKS 6
#endif
template <int K, typename T>
constexpr int render_min_blocks(Lookup l)
{
    return l == kLookBrick && (K < 16 || sizeof(T) < 4) ? 7 : POT_RENDER_MIN_BLOCKS;
}
constexpr int rays_min_blocks(Lookup l) { return l == kLookAny ? 6 : 4; }  // explicit rays

// Fixed-point ray times.  A walk measures time from the clip range's entry
// tin in units of 2^-kTimeFrac, with the ray's direction scaled by a power of
// two to a length in [1, 2) and the box to an edge in [1, 2) (WalkFrame), and
// keeps it in 64-bit integers: the clip range is below 2^51 units.  The
// crossing times of one axis's planes are then an arithmetic progression
// nx, nx + hs, nx + 2 hs, ... whose terms are exact sums: advancing by one
// plane, or by the j planes of a box, gives the same time whichever way the
// plane is reached, so leaf segments do not depend on how empty space is
// stepped over, and comparisons need no error bounds.  nx and hs are rounded
// from double-float values once per ray (a voxel is at least 2^39 units at
// depth 9 and 2^36 at depth 12: rounding hs moves a crossing by at most 2^-31
// and 2^-25 of a voxel).
// Axes along which the ray does not move, and planes it would reach only after
// its range, have nx or hs = kTimeNever; nx + j hs stays below 2^63 for the
// j < 2^11 planes of any box.
constexpr int64_t kTimeNever = 1ll << 51;
constexpr float kTimeScale = (float)(1ll << kTimeFrac);

// hi + lo (lo below hi's last bits, or both small) in time units.
__device__ __forceinline__ int64_t fixed_time(float hi, float lo)
{
    const float f = __fmul_rn(hi, kTimeScale);
    if (!(f < (float)kTimeNever)) return kTimeNever;  // also NaN
    if (f < -(float)kTimeNever) return -kTimeNever;
    return __float2ll_rn(f) + __float2ll_rn(__fmul_rn(lo, kTimeScale));
}
__device__ __forceinline__ int64_t fixed_time_since(df a, df tin)
{
    float hi, e;
    two_sum(a.hi, -tin.hi, hi, e);
    return fixed_time(hi, __fadd_rn(e, __fsub_rn(a.lo, tin.lo)));
}

__device__ __forceinline__ float exp2_int(int x) { return __int_as_float((127 + x) << 23); }

// One ray's walk through the octree (a2-a4) as resumable state: begin() sets
// the ray up (clip, locate, first cell); approach() and step() advance past the
// cell the ray is in, an empty box or any, the latter calling vis(leaf, delta, Y) for a
// segment of positive length (delta: times frame.rest the world's length; Y: the SH
// basis at the ray direction); all three
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
//
// LOOKUP: how cells are found, fixed for the kernels where it pays (kLookAny
// asks the tree).  It saves branches, but matters more for the load of the next
// entry: where several lookups meet, the loaded register is copied, and the
// copy waits for the load before the shading's loads are issued (40 views, f16:
// 6.05 -> 5.68 ms; one full-HD view of a depth-10 tree with bricks: 807 -> 768 us).
template <int K, typename T, Lookup LOOKUP>
struct Walker {
    static constexpr bool DENSE = LOOKUP == kLookDense, BRICK = LOOKUP == kLookBrick;
    int64_t nx[3], hs[3];  // time of the next plane and between planes, per axis
    int64_t t, tout;
    int q[3];              // mirrored voxel
    uint32_t flip;         // the mirror, in the form of the tree's cell lookup
    float unit;            // length of one time unit
    int cell;              // entry of voxel q: leaf >= 0, or an empty box (cell_code_*)
    int step_i;
    // rows of shared memory: the per-ray SH basis, and 1 / hs per axis (read
    // only where an empty box is left), which saves registers
    float *ysm;
    float4 *st;
    __device__ __forceinline__ SmemY<K, kBlock> Y() const { return {ysm}; }

    // a3: the entry of mirrored voxel q: one load from the cell index when the
    // tree has one (two in the brick layout), else a descent from the deepest
    // ancestor q shares with voxel pq (whose path the stack holds up to
    // the level in its last row)
    __device__ __forceinline__ int locate(const RenderParams &p, int32_t *stk, const int pq[3])
    {
        const int D = p.depth;
        if (DENSE || BRICK || p.cells) {
            if (DENSE || (!BRICK && !p.btab))
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
        int l = min(lc, stk[kMaxDepth * kBlock]);
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
        stk[kMaxDepth * kBlock] = min(l, D - 1);
        return out;
    }

    // Leaves the unit direction in the first three floats of the basis row.
    __device__ __forceinline__ bool begin(const RenderParams &p, int32_t *stk, const float o[3], const float dw[3],
                                          float near, float far, float u[3])
    {
        const int R = p.R;
        const float h = p.frame.h, invh = p.frame.invh;
        const float len = sqrtf(fmaf(dw[0], dw[0], fmaf(dw[1], dw[1], dw[2] * dw[2])));
        if (!(len > 0.f) || !(len < 3.0e38f)) return false;
        const float invlen = __frcp_rn(len);
#pragma unroll
        for (int a = 0; a < 3; ++a) u[a] = dw[a] * invlen;
        // the direction scaled to a length in [1, 2)
        const int el = (int)(__float_as_uint(len) >> 23) - 127;
        const float ds = exp2_int(-el), il = invlen * exp2_int(el);
        unit = __fmul_rn(__fmul_rn(len, ds), p.frame.unit);
        float d[3], rd[3], Ahi[3], Alo[3], th[3], tl[3];  // A = lo - o exactly, 1 / d, time across the box
        bool move[3];
        // a2: clip range in scaled time (position o + t d)
        df tin = {near * p.frame.ws * il, 0.f}, tend = {far * p.frame.ws * il, 0.f};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            two_sum(p.lo[a], -o[a], Ahi[a], Alo[a]);
            move[a] = dw[a] != 0.f;
            if (!move[a]) {
                // -(lo - o) in [0, size), decided exactly
                const float s = -Ahi[a], e = -Alo[a];
                const bool inside = (s > 0.f || (s == 0.f && e >= 0.f)) && (s < p.size || (s == p.size && e < 0.f));
                if (!inside) return false;
            }
            Ahi[a] *= p.frame.ws;
            Alo[a] *= p.frame.ws;
            // no component is so small that its times leave the float range: those below 2^-125 and 2^-126 |A| count
            // as that much (their sign still decides the side of a plane that a ray starts on)
            d[a] = copysignf(fmaxf(fabsf(dw[a] * ds), fmaf(fabsf(Ahi[a]), 1.1754944e-38f, 2.3509887e-38f)), dw[a]);
            rd[a] = rcp_ftz(d[a]);
            // the box's two planes, A / d and (A + size) / d, the sum taken before the division: along a slow
            // axis A / d and size / d are large, and their roundings would stay where they cancel
            const df t0 = quotient(Ahi[a], Alo[a], d[a], rd[a]);
            float s1, e1;
            two_sum(Ahi[a], p.frame.size, s1, e1);
            const df t1 = quotient(s1, __fadd_rn(Alo[a], e1), d[a], rd[a]);
            th[a] = __fmul_rn(p.frame.size, rd[a]);
            tl[a] = __fmul_rn(__fmaf_rn(-th[a], d[a], p.frame.size), rd[a]);
            const bool neg = dw[a] < 0.f;
            const df t_in = neg ? t1 : t0, t_out = neg ? t0 : t1;
            if (move[a] && df_lt(tin, t_in)) tin = t_in;
            if (move[a] && df_lt(t_out, tend)) tend = t_out;
        }
        // (an offset beyond the floats: so far from a tiny box that no ray to it resolves it)
        if (!df_lt(tin, tend) || !(fabsf(Ahi[0]) + fabsf(Ahi[1]) + fabsf(Ahi[2]) < 3.4e38f)) return false;
        tout = fixed_time_since(tend, tin);
        flip = 0;
        float rh[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const bool neg = dw[a] < 0.f;
            if (neg) flip |= 4u >> a;
            // the voxel entered: an fp32 estimate low by its error bound, so exact or too low (by one unless
            // the origin is far away), then exact tests of its upper plane's time (a point on a plane belongs
            // to the voxel above).  The bound: 8 roundings of 2^-24 (|t d| + |A|) / h (3 of tin.hi, for tin.lo;
            // of A, the sum, 1 / h, the product and a subtraction one each), taken as 10, and on a mirrored
            // axis 2 of R 2^-25 (R - g, less the margin), taken as 8
            const float g = __fmul_rn(__fmaf_rn(tin.hi, d[a], -Ahi[a]), invh);
            const float margin = (fabsf(tin.hi * d[a]) + fabsf(Ahi[a])) * invh * 5.9604645e-7f +
                                 (1e-6f + (neg ? (float)R * 2.3841858e-7f : 0.f));
            int v = min(max(__float2int_rd((neg ? (float)R - g : g) - margin), 0), R - 1);
            hs[a] = fixed_time(fabsf(th[a]) * exp2_int(-p.depth), (neg ? -tl[a] : tl[a]) * exp2_int(-p.depth));
            if (!move[a]) {
                v = min(max(voxel_exact(o[a], p.lo[a], h / p.frame.ws, invh * p.frame.ws, R), 0), R - 1);
                nx[a] = hs[a] = kTimeNever;
            } else {
                for (;; ++v) {
                    nx[a] = fixed_time_since(cross_time(neg ? R - 1 - v : v + 1, h, Ahi[a], Alo[a], d[a], rd[a]), tin);
                    if (nx[a] > 0 || v == R - 1) break;
                }
            }
            nx[a] = nx[a] < 0 ? 0 : nx[a];
            q[a] = v;
            // planes per 2^20 units, a little below the true value (see step)
            rh[a] = fabsf(d[a]) * (invh * (exp2_int(20 - kTimeFrac) * (1.f - 9.5367432e-7f)));
        }
        *st = make_float4(rh[0], rh[1], rh[2], 0.f);
        // the mirror as an XOR mask: child slots (no index), entry offsets (dense), or brick offsets
        // with a flag per axis of the in-brick offset in bits 27-29 (brick layout)
        if (DENSE || BRICK || p.cells) {
            const uint32_t fx = flip & 4u ? R - 1 : 0, fy = flip & 2u ? R - 1 : 0, fz = flip & 1u ? R - 1 : 0;
            if (BRICK || (!DENSE && p.btab)) flip = brick_of(fx, fy, fz, p.depth) | flip << 27;
            else flip = cell_index_offset(fx, fy, fz, p.depth);
        }
        if (!DENSE && !BRICK && !p.cells) stk[0] = stk[kMaxDepth * kBlock] = 0;  // the stack exists only for trees without a cell index
        cell = locate(p, stk, q);
        t = 0;
        step_i = 0;
        return true;
    }

    // The SH basis at the unit direction that begin() left in its row.
    __device__ __forceinline__ void basis(const float u[3])
    {
        float Yt[K];
        sh_basis<K>(u[0], u[1], u[2], Yt);
        SmemY<K, kBlock>::store(ysm, Yt);
    }

    // One step of a lane in an empty box, its whole warp being in empty space:
    // the box is crossed; false when the ray ends in it.
    __device__ __forceinline__ bool approach(const RenderParams &p, int32_t *stk)
    {
        const int pq[3] = {q[0], q[1], q[2]};
        t = leave_box();
        if (t >= tout) return false;
        if (step_i >= p.step_cap) {
            *p.err = 1u;
            return false;
        }
        ++step_i;
        if ((unsigned)(q[0] | q[1] | q[2]) >= (unsigned)p.R) return false;
        cell = locate(p, stk, pq);
        return true;
    }

    // a4 for an empty box: the exit time, the earliest of its upper faces; every
    // plane with a time <= it has then been crossed: floor((texit - nx) / hs) + 1
    // of them per axis, by an fp32 estimate that is exact or one too low (its
    // factor and its addend are low by 2^-20, over the rounding errors, and at
    // most 2^12 planes are crossed), then the exact test of the next plane.
    __device__ __forceinline__ int64_t leave_box()
    {
        const uint32_t m = cell & 0xFFFF, e = (cell >> 16) & 0xFF;
        int64_t ex[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            ex[a] = nx[a] + (int64_t)((uint64_t)((m & ~(uint32_t)q[a]) + e) * (uint64_t)hs[a]);
        const int64_t texit = min(ex[0], min(ex[1], ex[2]));
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
        return texit;
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
            texit = leave_box();
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
// walker's row of constants, and the ancestor stack [kMaxDepth + 1][kBlock] in
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
    return need_stack ? sizeof(int32_t) * (kMaxDepth + 1) * kBlock : 0;
}

// Whether a launch may use the kLookDense instance of a kernel that has no other than kLookAny.
inline bool dense_index(const RenderParams &p) { return p.cells && !p.btab; }

// FN<K, T, LOOKUP, ...> for the K of a tree; null for another K.
#define POT_PICK_K(FN, K, T, LOOKUP, ...)                                                                       \
    ((K) == 1 ? FN<1, T, LOOKUP, ##__VA_ARGS__> : (K) == 4 ? FN<4, T, LOOKUP, ##__VA_ARGS__>                    \
     : (K) == 9 ? FN<9, T, LOOKUP, ##__VA_ARGS__> : (K) == 16 ? FN<16, T, LOOKUP, ##__VA_ARGS__>                \
     : (K) == 25 ? FN<25, T, LOOKUP, ##__VA_ARGS__> : nullptr)
#define POT_PICK_WALK(FN, K, T, DENSE, ...)                                                                     \
    ((DENSE) ? POT_PICK_K(FN, K, T, kLookDense, ##__VA_ARGS__) : POT_PICK_K(FN, K, T, kLookAny, ##__VA_ARGS__))

// The next tile of a warp, and the lane's slot in it (0..31; 32 for a lane that
// takes none): from the launch's counter until none is left, or, without one,
// once, by the warp's place in the grid.  Launches with fewer tiles than warps
// that could be resident split them: the time of such a launch is that of its
// slowest warp, and with fewer rays a warp takes fewer sides of the branches, waits
// for fewer lines per load and ends with its own rays.  False when there is none.
__device__ __forceinline__ bool next_tile(const RenderParams &p, int lane, int &taken, unsigned long long &tile,
                                          int &slot)
{
    slot = lane;
    if (p.tile_counter) {
        tile = 0;
        if (lane == 0) tile = atomicAdd(p.tile_counter, 1ull);
        tile = __shfl_sync(0xffffffffu, tile, 0);
    } else {
        if (taken++) return false;
        const unsigned warp = blockIdx.x * (kBlock / 32) + (threadIdx.x >> 5);
        const int rays = 32 >> p.part_log2;
        tile = warp >> p.part_log2;
        slot = lane < rays ? (int)(warp & ((1u << p.part_log2) - 1u)) * rays + lane : 32;
    }
    return tile < (unsigned long long)p.n_tiles;
}

// Grid of a walk kernel: all warps of all tiles without a counter, else one wave of resident blocks (SMs x blocks
// per SM for this kernel and shared memory), no more blocks than tiles need.
template <typename Fn>
cudaError_t persistent_grid(Fn fn, size_t smem, const RenderParams &p, unsigned *grid)
{
    const int64_t warps = p.tile_counter ? p.n_tiles : p.n_tiles << p.part_log2;
    const int64_t need = (warps + (kBlock / 32) - 1) / (kBlock / 32);
    if (!p.tile_counter) {
        *grid = (unsigned)(need < 1 ? 1 : need);
        return cudaSuccess;
    }
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBlock, smem);
    if (e != cudaSuccess) return e;
    int64_t blocks = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    *grid = (unsigned)blocks;
    return cudaSuccess;
}

// The walks of a warp's 32 rays (every lane calls it; has: whether it has a
// ray).  APPROACH (tiles of pixels, whose rays meet the scene together): while
// no lane has met a leaf the warp crosses empty space in a loop of its own,
// without the leaf side of step(), and the SH basis is evaluated once some lane
// has, so tiles that see no leaf never do.
template <int K, typename T, Lookup LOOKUP, bool APPROACH, typename Visitor>
__device__ __forceinline__ void walk_rays(const RenderParams &p, int32_t *stk, float *ysm, float4 *wst, bool has,
                                          const float o[3], const float d[3], float near, float far, Visitor &vis)
{
    Walker<K, T, LOOKUP> w;
    w.ysm = ysm;
    w.st = wst;
    float u[3] = {0.f, 0.f, 1.f};
    has = has && w.begin(p, stk, o, d, near, far, u);
    if (APPROACH) {
        while (!__any_sync(0xffffffffu, has && w.cell >= 0)) {
            if (has) has = w.approach(p, stk);
            if (!__any_sync(0xffffffffu, has)) return;
        }
    }
    if (Visitor::kBasis && has) w.basis(u);
    if (Visitor::kVote) {
        while (__any_sync(0xffffffffu, has)) {
            if (has) has = w.step(p, stk, vis);
        }
    } else {
        while (has) has = w.step(p, stk, vis);
    }
}

// a5-a8 for one leaf segment: fetch, colour, composite, early stop.
template <int K, typename T, bool COUNT>
struct ShadeVisitor {
    static constexpr bool kBasis = true, kVote = false;
    const T *sig_arr;
    const T *sh_arr;
    uint8_t *touched;
    float gamma;
    float col[3];
    float Tr;
    int nseg;
    const void *cb;  // codebook (cb16 leaves only)
    float rate;      // the frame's, from the launch's parameters: an operand, not a register
    template <typename YT>
    __device__ __forceinline__ bool operator()(int leaf, float delta, const YT &Y)
    {
        const float sig = fmaxf(Store<T>::load_sigma(sig_arr, leaf), 0.f);
        float x[3];
        leaf_colour_dot<K, T>(sh_arr, leaf, Y, x, cb);
        const float e = exp2_ftz((-sig * delta) * rate);  // transmittance of the segment
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
        const uint32_t group = p.by_group(tl);
        const uint32_t in_group = tl - group * per_group;
        const uint32_t gsize = min(G, (uint32_t)p.n_cams - group * G);
        const uint32_t rem = gsize == G ? p.by_view(in_group) : p.by_last(in_group);
        const int64_t cam = (int64_t)(group * G + in_group - rem * gsize);
        const int ty = (int)p.by_row(rem);
        const int tx = (int)(rem - (uint32_t)ty * (uint32_t)p.tiles_x);
        const int i = tx * kTileW + (slot % kTileW);
        const int j = ty * kTileH + (slot / kTileW);
        if (slot >= 32 || i >= p.W || j >= p.H) return false;
        ray = (cam * p.H + j) * p.W + i;
        const pot_camera *c = p.cams ? p.cams + cam : p.few_cams + cam;
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
    if (slot >= 32 || ray >= p.n_rays) return false;
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
template <int K, typename T, Lookup LOOKUP, bool CAMS, bool COUNT>
__global__ void __launch_bounds__(kBlock, CAMS ? render_min_blocks<K, T>(LOOKUP) : rays_min_blocks(LOOKUP))
    render_kernel(const __grid_constant__ RenderParams p)
{
    POT_WALK_SHARED(K)
    const int lane = threadIdx.x & 31;
    const T *sig_arr = static_cast<const T *>(p.sigma);
    const T *sh_arr = static_cast<const T *>(p.sh);
    int taken = 0, slot;
    for (unsigned long long tile; next_tile(p, lane, taken, tile, slot);) {
        float o[3], d[3], near, far;
        int64_t ray;
        const bool has = tile_ray<CAMS>(p, tile, slot, o, d, near, far, ray);
        ShadeVisitor<K, T, COUNT> v{sig_arr, sh_arr, p.leaf_touched, p.gamma, {0.f, 0.f, 0.f}, 1.f, 0, p.codebook,
                                    p.frame.rate};
        walk_rays<K, T, LOOKUP, CAMS>(p, stk, ysm, wst, has, o, d, near, far, v);
        if (has) store_ray<K, T, COUNT>(p, ray, v);
    }
}

template <typename T>
cudaError_t launch_render_t(const RenderParams &p, int K, bool cams, bool count, cudaStream_t s)
{
    using Fn = void (*)(const RenderParams);
    Fn fn = nullptr;
    // counting launches (measurement) and explicit rays have fewer instances of their own
    const Lookup look = p.btab ? kLookBrick : p.cells ? kLookDense : kLookAny;
#define POT_PICK(KK)                                                                  \
    if (K == KK)                                                                      \
        fn = cams ? (count                ? render_kernel<KK, T, kLookAny, true, true>   \
                     : look == kLookDense ? render_kernel<KK, T, kLookDense, true, false> \
                     : look == kLookBrick ? render_kernel<KK, T, kLookBrick, true, false> \
                                          : render_kernel<KK, T, kLookAny, true, false>)  \
                  : (count                ? render_kernel<KK, T, kLookAny, false, true>   \
                     : look == kLookDense ? render_kernel<KK, T, kLookDense, false, false> \
                                          : render_kernel<KK, T, kLookAny, false, false>);
    POT_PICK(1)
    POT_PICK(4)
    POT_PICK(9)
    POT_PICK(16)
    POT_PICK(25)
#undef POT_PICK
    if (!fn) return cudaErrorInvalidValue;
    const size_t smem = walk_smem_bytes(p.cells == nullptr);
    unsigned grid = 0;
    cudaError_t e = persistent_grid(fn, smem, p, &grid);
    if (e != cudaSuccess) return e;
    RenderParams q = p;
    if (cams) set_tile_divs(q);
    fn<<<grid, kBlock, smem, s>>>(q);
    count_launch();
    return cudaGetLastError();
}

}  // namespace pot
