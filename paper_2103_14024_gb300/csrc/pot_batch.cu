// pot_batch.cu -- one launch renders many requests: different trees, cameras,
// resolutions and outputs (the work list of a continuous-batching server).
//
// The host groups the items by (SH coefficients, leaf dtype, layout of the cell
// index, rate of the walk's frame); each group is one launch.  Every item contributes tiles of kTileW x kTileH pixels (as pot_render);
// each warp renders the tile of its place in the grid and finds its item among
// the items' first-tile offsets.  The per-ray code (walk + shading) is the
// same as pot_render's, so a request renders bit-identically alone or in a mix.
#include <algorithm>
#include <cmath>
#include <memory>
#include <utility>
#include <vector>

#include "pot_render.cuh"

namespace pot {

namespace {

struct BatchItem {
    const int32_t *child;
    const int32_t *cells;
    const int32_t *btab;
    const void *sigma;
    const void *sh;
    const void *codebook;
    int depth, R;
    float lo[3];
    float size;
    WalkFrame frame;
    float bg[3];
    float gamma;
    int W, H, tiles_x;
    FastDiv by_row;
    int64_t tile_begin;
    float *rgb;
    float *t_final;
    pot_camera cam;
};

struct BatchParams {
    const BatchItem *items;
    int n_items;
    int64_t n_tiles;
    unsigned int *err;
    int overlaps;  // launched while the previous group's last blocks run
    float rate;    // the frames'
};

template <int K, typename T, Lookup LOOKUP>
__global__ void __launch_bounds__(kBlock, render_min_blocks<K, T>(LOOKUP)) batch_kernel(const BatchParams bp)
{
    POT_WALK_SHARED(K)
    const int lane = threadIdx.x & 31;
    // the next group may start once this group's blocks have all started (see launch_batch_t)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // short blocks: every warp renders one tile and the block ends, so a
    // launch frees its SM slots tile by tile and launches of higher-priority
    // streams (small requests) start between them
    {
        const unsigned long long tile = (unsigned long long)blockIdx.x * (kBlock / 32) + (threadIdx.x >> 5);
        if (tile >= (unsigned long long)bp.n_tiles) return;
        // item owning the tile: the last item with tile_begin <= tile, by a
        // warp-wide search -- each round the 32 lanes test 32 evenly spaced
        // items of [lo, hi] at once and the range shrinks to one stride (one
        // round up to 32 items, two up to 1024), instead of a chain of
        // dependent loads of a binary search.  items[lo].tile_begin <= tile
        // holds throughout (item 0 begins at tile 0).
        int lo = 0, hi = bp.n_items - 1;
        while (hi > lo) {
            const int stride = (hi - lo + 32) / 32;
            const int cand = lo + lane * stride;
            const bool ok = cand <= hi && bp.items[cand].tile_begin <= (int64_t)tile;
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            lo += (31 - __clz(m)) * stride;
            hi = min(hi, lo + stride - 1);
        }
        const BatchItem &it = bp.items[lo];
        // 32-bit arithmetic: an item has at most 2^31 pixels
        const uint32_t rem = (uint32_t)((int64_t)tile - it.tile_begin);
        const int ty = (int)it.by_row(rem);
        const int tx = (int)(rem - (uint32_t)ty * (uint32_t)it.tiles_x);
        const int i = tx * kTileW + (lane % kTileW);
        const int j = ty * kTileH + (lane / kTileW);
        const bool has = i < it.W && j < it.H;
        RenderParams p;
        p.child = it.child;
        p.cells = it.cells;
        p.btab = it.btab;
        p.depth = it.depth;
        p.R = it.R;
        p.lo[0] = it.lo[0];
        p.lo[1] = it.lo[1];
        p.lo[2] = it.lo[2];
        p.size = it.size;
        p.frame = it.frame;
        p.step_cap = 3 * it.R + 16;
        p.err = bp.err;
        const pot_camera *c = &it.cam;
        float o[3], d[3];
        const float xc = __fdiv_rn(__fsub_rn(__fadd_rn((float)i, 0.5f), c->cx), c->fx);
        const float yc = -__fdiv_rn(__fsub_rn(__fadd_rn((float)j, 0.5f), c->cy), c->fy);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            d[r] = __fsub_rn(__fadd_rn(__fmul_rn(c->c2w[r][0], xc), __fmul_rn(c->c2w[r][1], yc)), c->c2w[r][2]);
            o[r] = c->c2w[r][3];
        }
        const T *sig_arr = static_cast<const T *>(it.sigma);
        const T *sh_arr = static_cast<const T *>(it.sh);
        ShadeVisitor<K, T, false> v{sig_arr, sh_arr, nullptr, it.gamma, {0.f, 0.f, 0.f}, 1.f, 0, it.codebook,
                                    bp.rate};
        walk_rays<K, T, LOOKUP, true>(p, stk, ysm, wst, has, o, d, c->near, c->far, v);
        if (has) {
            const int64_t px = (int64_t)j * it.W + i;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) it.rgb[3 * px + ch] = fmaf(v.Tr, it.bg[ch], v.col[ch]);
            if (it.t_final) it.t_final[px] = v.Tr;
        }
    }
    // a group is not done before the groups ahead of it are
    if (bp.overlaps && blockIdx.x == 0 && threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Groups follow each other on the stream, and each ends with its longest rays
// on a few SMs.  A group after the first is launched programmatically: its
// blocks start as soon as all blocks of the previous group have (groups read
// only descriptors and trees that were there before the first, and write
// outputs of their own, see outputs_overlap), and its block 0 waits for the previous group before it
// ends, so that whatever follows the call on the stream waits for all groups.
// Mixed requests on trees of degree 1, 2 and 3 (f16), one group each: 2 of
// 256 x 256 88 -> 59 us, 3 of them 275 -> 168 us, 6 of up to 800 x 800 598 -> 517 us,
// 24 of up to 1920 x 1080 3490 -> 3425 us.
template <typename T>
cudaError_t launch_batch_t(const BatchParams &bp, int K, Lookup look, bool need_stack, cudaStream_t s)
{
    using Fn = void (*)(const BatchParams);
    Fn fn = look == kLookDense ? POT_PICK_K(batch_kernel, K, T, kLookDense)
          : look == kLookBrick ? POT_PICK_K(batch_kernel, K, T, kLookBrick)
                               : POT_PICK_K(batch_kernel, K, T, kLookAny);
    if (!fn) return cudaErrorInvalidValue;
    const size_t smem = walk_smem_bytes(need_stack);
    const int64_t blocks = (bp.n_tiles + kBlock / 32 - 1) / (kBlock / 32);
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)(blocks > 0 ? blocks : 1);
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kBlock);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = bp.overlaps ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, bp);
    if (e == cudaSuccess) count_launch();
    return e;
}

// Whether some outputs of the items overlap.  Then the groups do not: the order in which they write decides.
bool outputs_overlap(const std::vector<BatchItem> &items)
{
    std::vector<std::pair<const float *, const float *>> r;
    r.reserve(2 * items.size());
    for (const BatchItem &b : items) {
        const int64_t px = (int64_t)b.W * b.H;
        r.emplace_back(b.rgb, b.rgb + 3 * px);
        if (b.t_final) r.emplace_back(b.t_final, b.t_final + px);
    }
    std::sort(r.begin(), r.end());
    const float *end = nullptr;
    for (const auto &q : r) {
        if (q.first < end) return true;
        end = q.second;
    }
    return false;
}

// A captured copy reads its source at each replay, so the graph takes the descriptors over and frees them with
// its last instance.  Outside a capture nothing changes hands.
cudaError_t graph_takes(std::unique_ptr<std::vector<BatchItem>> &items, cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamGetCaptureInfo(s, &st, nullptr, &graph, nullptr, nullptr, nullptr);
    if (e != cudaSuccess || st != cudaStreamCaptureStatusActive) return e;
    cudaUserObject_t obj = nullptr;
    e = cudaUserObjectCreate(
        &obj, items.get(), [](void *v) { delete static_cast<std::vector<BatchItem> *>(v); }, 1,
        cudaUserObjectNoDestructorSync);
    if (e != cudaSuccess) return e;
    items.release();
    e = cudaGraphRetainUserObject(graph, obj, 1, cudaGraphUserObjectMove);
    if (e != cudaSuccess) cudaUserObjectRelease(obj, 1);
    return e;
}

}  // namespace

// items: host array of n validated requests; groups by (K, dtype, cell index), stages the
// descriptors in a stream-ordered buffer.
cudaError_t launch_render_batch(const pot_render_item *items, int n, cudaStream_t s, unsigned int *err)
{
    std::vector<int> order(n);
    for (int i = 0; i < n; ++i) order[i] = i;
    auto key = [&](int i) {
        const pot_tree *t = items[i].tree;
        // the frames of a group share their rate (all but tiny boxes have the same): a register less per ray than
        // one rate per item, 8 requests of 256 x 256 207 -> 183 us
        const int tiny = -std::ilogb(walk_frame(t->desc.bbox_size, t->desc.depth).rest);
        return ((t->K * 4 + t->desc.leaf_dtype) * 4 + t->cell_kind) * 64 + tiny;
    };
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return key(a) < key(b); });
    auto owned = std::make_unique<std::vector<BatchItem>>(n);
    std::vector<BatchItem> &desc = *owned;
    std::vector<int> group_start;
    int64_t tiles = 0;
    for (int k = 0; k < n; ++k) {
        const pot_render_item &r = items[order[k]];
        if (k == 0 || key(order[k]) != key(order[k - 1])) {
            group_start.push_back(k);
            tiles = 0;
        }
        const pot_tree *t = r.tree;
        BatchItem &b = desc[k];
        b.child = t->child;
        b.cells = t->cells;
        b.btab = t->btab;
        b.sigma = t->sigma;
        b.sh = t->sh;
        b.codebook = t->codebook;
        b.depth = t->desc.depth;
        b.R = 1 << t->desc.depth;
        for (int a = 0; a < 3; ++a) b.lo[a] = t->desc.bbox_lo[a];
        b.size = t->desc.bbox_size;
        b.frame = walk_frame(t->desc.bbox_size, t->desc.depth);
        for (int c = 0; c < 3; ++c) b.bg[c] = r.bg[c];
        b.gamma = r.gamma;
        b.W = r.cam.width;
        b.H = r.cam.height;
        b.tiles_x = (b.W + kTileW - 1) / kTileW;
        b.by_row = fast_div((uint32_t)b.tiles_x);
        b.tile_begin = tiles;
        b.rgb = r.rgb;
        b.t_final = r.t_final;
        b.cam = r.cam;
        tiles += (int64_t)b.tiles_x * ((b.H + kTileH - 1) / kTileH);
    }
    group_start.push_back(n);
    const int groups = (int)group_start.size() - 1;
    BatchItem *d_items = nullptr;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = graph_takes(owned, s);
    if (e == cudaSuccess) e = scratch_pool(&pool);
    if (e == cudaSuccess)
        e = cudaMallocFromPoolAsync(reinterpret_cast<void **>(&d_items), sizeof(BatchItem) * (size_t)n, pool, s);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(d_items, desc.data(), sizeof(BatchItem) * n, cudaMemcpyHostToDevice, s);
    const bool apart = groups > 1 && !outputs_overlap(desc);
    for (int g = 0; g < groups && e == cudaSuccess; ++g) {
        const int a = group_start[g], b = group_start[g + 1];
        const BatchItem &last = desc[b - 1];
        BatchParams bp;
        bp.items = d_items + a;
        bp.n_items = b - a;
        bp.n_tiles = last.tile_begin + (int64_t)last.tiles_x * ((last.H + kTileH - 1) / kTileH);
        bp.err = err;
        bp.overlaps = g > 0 && apart;
        bp.rate = last.frame.rate;
        const pot_tree *t = items[order[a]].tree;
        const Lookup look = t->cell_kind == POT_CELLS_DENSE   ? kLookDense
                            : t->cell_kind == POT_CELLS_BRICK ? kLookBrick
                                                              : kLookAny;
        const bool need_stack = t->cell_kind == POT_CELLS_NONE;
        switch (t->desc.leaf_dtype) {
        case POT_F32: e = launch_batch_t<float>(bp, t->K, look, need_stack, s); break;
        case POT_F16: e = launch_batch_t<__half>(bp, t->K, look, need_stack, s); break;
        case POT_CB16: e = launch_batch_t<cb16>(bp, t->K, look, need_stack, s); break;
        default: e = launch_batch_t<__nv_bfloat16>(bp, t->K, look, need_stack, s); break;
        }
    }
    cudaFreeAsync(d_items, s);
    return e;
}

}  // namespace pot
