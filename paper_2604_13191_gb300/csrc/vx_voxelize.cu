// vx_voxelize.cu -- level 0 of the pyramid: sparse voxelization of capsules (fiber
// segments) and triangles with 8^3 sub-cell occupancy, mass and second moments.
//
// Pipeline (one stream):
//   prep      per primitive: grid coordinates (Sec. 3.1, P_volume), weights
//   count     up to 32 primitives per warp: conservative voxel test over their bounding boxes, by a
//             record per primitive, its hits kept as ballots (large boxes: a warp each)
//   scan      exclusive offsets of the per-primitive candidate counts
//   emit      (Morton key, primitive id) pairs from the ballots, 32 primitives per warp (those without
//             ballots: a warp each, tested again)
//   sort      stable LSD radix sort by key (Sec. 3.3: samples ordered by block id)
//   heads     segment starts where the key changes (Sec. 3.3)
//   reduce    warp per voxel: exact sub-cell masks (OR over primitives), mass and
//             moment summed in primitive order (Sec. 3.4-3.5, 4.1)
//   finalize  compaction of the non-empty voxels, occupancy counts, S = M / m and
//             the compact SGGX parameters (Eq. compact-sggx)
//
// Arithmetic: every FP32 quantity that decides a bit, and every per-voxel sum, is
// evaluated with the operation order written below and no contraction (the library
// is compiled with -fmad=false); the per-voxel sums run sequentially in primitive
// order so the result does not depend on scheduling.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "vx_internal.cuh"

#include "vx_level0.cuh"

namespace {

// The count pass's ballot store (WS_BALLOTS) in *out and its words per primitive in *stride: 64 (ranges
// of up to 2048 voxels, a capsule of 5 voxels' radius), 32 or 8, the most that takes at most 256 MB and
// that there is memory for; NULL when 8 take more than 256 MB (the emit pass then tests every voxel
// again).  A range's unused words are never touched.  Errors: VX_ERR_OUT_OF_MEMORY without memory for 8.
vx_status window_ballots(vx_context* ctx, uint32_t np, cudaStream_t s, uint32_t** out, uint32_t* stride) {
    *out = nullptr;
    *stride = 0;
    for (uint32_t words : {64u, 32u, 8u}) {
        const size_t bytes = (size_t)np * words * 4;
        if (bytes > ((size_t)256 << 20)) continue;
        const vx_status st = vx_ws_ensure(ctx, WS_BALLOTS, bytes, s);
        if (st == VX_ERR_OUT_OF_MEMORY && words > 8) continue;
        VX_TRY(st);
        *out = (uint32_t*)ctx->ws[WS_BALLOTS].p;
        *stride = words;
        break;
    }
    return VX_OK;
}

// Candidate counts and offsets of the primitives over one window (WS_COUNT, WS_OFFS), and
// the hit ballots of their ranges (WS_BALLOTS, see window_ballots); the exact total goes to
// *total.  Synchronises the stream once (twice when a range is too large for the grouped pass).
vx_status count_window(vx_context* ctx, bool fiber, uint32_t np, const Window& win, float4* r0, float4* r1,
                       float4* r2, uint32_t* misc, cudaStream_t s, uint64_t* total) {
    VX_TRY(vx_ws_ensure(ctx, WS_COUNT, (size_t)np * 4, s));
    VX_TRY(vx_ws_ensure(ctx, WS_OFFS, (size_t)np * 4, s));
    uint32_t* cnt = (uint32_t*)ctx->ws[WS_COUNT].p;
    uint32_t* offs = (uint32_t*)ctx->ws[WS_OFFS].p;
    ctx->ballots = nullptr;
    uint32_t* ballots = nullptr;
    uint32_t stride = 0;
    VX_TRY(window_ballots(ctx, np, s, &ballots, &stride));
    ctx->ballots = ballots;
    ctx->ballots_stride = stride;
    ctx->ballots_np = np;
    for (int i = 0; i < 3; ++i) {
        ctx->ballots_win[i] = win.lo[i];
        ctx->ballots_win[3 + i] = win.hi[i];
    }
    unsigned long long* t64 = (unsigned long long*)(misc + 8);
    uint32_t* const flags = misc + 14;   // (zero but for a count pass that has raised some)
    // ranges of [least, most] voxels, 2^lg primitives to a warp, then offsets and totals
    auto pass = [&](int lg, int least, int most, uint32_t* raise) -> vx_status {
        if (fiber)
            VX_LAUNCH(ctx, ST_COUNT, s, k_count<true><<<count_blocks(np, lg), COUNT_WARPS * 32, 0, s>>>(
                                            r0, r1, r2, np, win, lg, least, most, cnt, ctx->ballots, stride, raise));
        else
            VX_LAUNCH(ctx, ST_COUNT, s, k_count<false><<<count_blocks(np, lg), COUNT_WARPS * 32, 0, s>>>(
                                            r0, r1, r2, np, win, lg, least, most, cnt, ctx->ballots, stride, raise));
        bool done = false;
        VX_TRY(vx_scan_u32(ctx, cnt, offs, np, misc + 1, s, t64, vx_pin_of(ctx, misc, 16), &done));
        if (!done) {   // no primitives
            VX_CUDA_TRY(cudaMemsetAsync(t64, 0, 8, s));
            VX_TRY(vx_readback_async(ctx, 0, misc, 64, s));
        }
        VX_CUDA_TRY(cudaStreamSynchronize(s));
        return ((uint32_t*)ctx->host_pin)[0] ? VX_ERR_INVALID_ARG : VX_OK;
    };
    const int lg = count_lanes_log2(np);
    VX_TRY(pass(lg, 0, lg > 0 ? kGroupRange : kAnyRange, flags));
    const uint32_t raised = ((uint32_t*)ctx->host_pin)[14];
    ctx->ballots_unstored = (raised & kCountUnstored) != 0;
    if (raised) VX_CUDA_TRY(cudaMemsetAsync(flags, 0, 4, s));
    if (raised & kCountLarge) VX_TRY(pass(0, kGroupRange + 1, kAnyRange, nullptr));
    *total = ((const uint64_t*)ctx->host_pin)[4];
    return VX_OK;
}

// Candidate pairs of one pass at most (31-bit pair indices).
constexpr int64_t kMaxPassPairs = 0x7fffffffll;

// A window of the grid in the planning of a voxelization: its corner and size (2^lg voxels
// per side) and, once counted, its candidate-pair total.
struct Leaf {
    int lo[3];
    int lg;
    uint64_t pairs;
};

inline Window window_of(const Leaf& w) {
    Window win;
    for (int i = 0; i < 3; ++i) { win.lo[i] = w.lo[i]; win.hi[i] = w.lo[i] + (1 << w.lg) - 1; }
    return win;
}

inline uint64_t key_hi_of(const Leaf& w) {
    return vx_morton3_64((uint32_t)(w.lo[0] >> w.lg), (uint32_t)(w.lo[1] >> w.lg), (uint32_t)(w.lo[2] >> w.lg))
           << (3 * w.lg);
}

// Emit, sort and segment heads of one window whose candidate counts and offsets are in
// WS_COUNT / WS_OFFS (count_window ran on it last) and whose pair total fits 31 bits.  On
// return the sorted keys / primitive ids are in *k0 / *v0, the run starts in WS_STARTS and
// the number of candidate voxels in *nseg.  Synchronises the stream once.
vx_status window_segments(vx_context* ctx, bool fiber, uint32_t np, const Window& win, int bits, uint32_t npairs,
                          float4* r0, float4* r1, float4* r2, uint32_t* misc, cudaStream_t s, uint32_t** k0,
                          uint32_t** v0, uint32_t** k1, uint32_t** v1, uint32_t* nseg) {
    uint32_t* offs = (uint32_t*)ctx->ws[WS_OFFS].p;
    const unsigned cblocks = (unsigned)std::min<size_t>((np + EMIT_WARPS - 1) / EMIT_WARPS, (size_t)vx::kSMs * 64);
    VX_TRY(vx_ws_ensure(ctx, WS_KEYS0, (size_t)npairs * 4, s));
    VX_TRY(vx_ws_ensure(ctx, WS_VALS0, (size_t)npairs * 4, s));
    VX_TRY(vx_ws_ensure(ctx, WS_KEYS1, (size_t)npairs * 4, s));
    VX_TRY(vx_ws_ensure(ctx, WS_VALS1, (size_t)npairs * 4, s));
    *k0 = (uint32_t*)ctx->ws[WS_KEYS0].p;
    *v0 = (uint32_t*)ctx->ws[WS_VALS0].p;
    *k1 = (uint32_t*)ctx->ws[WS_KEYS1].p;
    *v1 = (uint32_t*)ctx->ws[WS_VALS1].p;
    // the ballots the count pass of this window stored, if it stored any
    bool same = ctx->ballots != nullptr && ctx->ballots_np == np;
    for (int i = 0; i < 3; ++i)
        same = same && ctx->ballots_win[i] == win.lo[i] && ctx->ballots_win[3 + i] == win.hi[i];
    if (same) {
        const unsigned eblocks = (unsigned)std::min<size_t>(((size_t)np + 32 * STAGE_WARPS - 1) / (32 * STAGE_WARPS),
                                                            (size_t)vx::kSMs * 6);
        if (fiber)
            VX_LAUNCH(ctx, ST_EMIT, s, k_emit_stored<true><<<eblocks, STAGE_WARPS * 32, 0, s>>>(
                                           r0, r1, r2, np, win, offs, *k0, *v0, ctx->ballots, ctx->ballots_stride));
        else
            VX_LAUNCH(ctx, ST_EMIT, s, k_emit_stored<false><<<eblocks, STAGE_WARPS * 32, 0, s>>>(
                                           r0, r1, r2, np, win, offs, *k0, *v0, ctx->ballots, ctx->ballots_stride));
    }
    if (!same || ctx->ballots_unstored) {
        uint32_t* const ballots = same ? ctx->ballots : nullptr;
        if (fiber)
            VX_LAUNCH(ctx, ST_EMIT, s, k_candidates<true><<<cblocks, EMIT_WARPS * 32, 0, s>>>(
                                           r0, r1, r2, np, win, offs, *k0, *v0, ballots, ctx->ballots_stride, same));
        else
            VX_LAUNCH(ctx, ST_EMIT, s, k_candidates<false><<<cblocks, EMIT_WARPS * 32, 0, s>>>(
                                           r0, r1, r2, np, win, offs, *k0, *v0, ballots, ctx->ballots_stride, same));
    }
    VX_CUDA_TRY(cudaGetLastError());
    VX_TRY(vx_radix_sort_u32(ctx, k0, v0, k1, v1, npairs, 3 * bits, s, misc));
    VX_TRY(vx_ws_ensure(ctx, WS_FLAGS, (size_t)npairs * 4, s));
    VX_TRY(vx_ws_ensure(ctx, WS_STARTS, (size_t)npairs * 4 + 8, s));
    uint32_t* starts = (uint32_t*)ctx->ws[WS_STARTS].p;
    bool done = false;
    VX_TRY(vx_segment_starts(ctx, *k0, npairs, misc + 2, starts, s, vx_pin_of(ctx, misc, 3), &done));
    if (!done) VX_TRY(vx_readback_async(ctx, 0, misc, 12, s));
    VX_CUDA_TRY(cudaStreamSynchronize(s));
    if (((uint32_t*)ctx->host_pin)[0] & 4u) return VX_ERR_TIMEOUT;   // a bounded wait of the sort gave up
    *nseg = ((uint32_t*)ctx->host_pin)[2];
    return VX_OK;
}

// Per-voxel reduction and compaction of one window after window_segments: the non-empty
// voxels are written to `dst`, a level or a view into one at the window's first row, with
// room for at least nseg rows (dst == NULL: a new level block of exactly the window's
// voxels is allocated into *alloc_out).  *nvox receives the window's voxel count.
// Keys are key_hi | the Morton key relative to the window's corner.  Synchronises once.
vx_status window_reduce(vx_context* ctx, bool fiber, uint32_t np, uint32_t nseg, uint64_t key_hi, int res,
                        uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, const Window& win, float4* r0,
                        float4* r1, float4* r2, uint32_t* misc, cudaStream_t s, const vx_level* dst,
                        vx_level* alloc_out, uint32_t* nvox_out) {
    const int bx = win.lo[0], by = win.lo[1], bz = win.lo[2];
    uint32_t* flags = (uint32_t*)ctx->ws[WS_FLAGS].p;
    uint32_t* starts = (uint32_t*)ctx->ws[WS_STARTS].p;
    vx_stage_units(ctx, ST_FINALIZE, nseg);
    // temp outputs per candidate voxel: mask 64 + mass 4 + moment 24 bytes; the sort's
    // alternate buffers are free now and hold the key and the non-empty flag.
    VX_TRY(vx_ws_ensure(ctx, WS_SEG_OUT, (size_t)std::max<uint32_t>(nseg, 1) * (64 + 4 + 24), s));
    char* so = (char*)ctx->ws[WS_SEG_OUT].p;
    SegOut seg;
    seg.mask = (uint64_t*)so;
    seg.moment = (float*)(so + (size_t)nseg * 64);   // 8-byte aligned rows
    seg.mass = (float*)(so + (size_t)nseg * 88);
    seg.key = k1;
    seg.nonzero = v1;
    VX_CUDA_TRY(cudaMemsetAsync(misc + 6, 0, 4, s));
    if (fiber) {
        // resident blocks (7 per SM) taking voxels from a counter
        const unsigned fblocks = (unsigned)std::min<size_t>((nseg + RED_WARPS - 1) / RED_WARPS, (size_t)vx::kSMs * 7);
        VX_LAUNCH(ctx, ST_REDUCE_FIBERS, s, k_reduce_fibers<<<fblocks, RED_WARPS * 32, 0, s>>>(
                                                k0, v0, starts, misc + 2, r0, r1, seg, bx, by, bz, misc + 6));
    } else {
        // resident blocks (5 per SM)
        const unsigned tblocks = (unsigned)std::min<size_t>((nseg + RED_WARPS - 1) / RED_WARPS, (size_t)vx::kSMs * 5);
        VX_LAUNCH(ctx, ST_REDUCE_TRIS, s, k_reduce_tris<<<tblocks, RED_WARPS * 32, 0, s>>>(
                                              k0, v0, starts, misc + 2, r0, r1, r2, seg, bx, by, bz, misc + 6));
    }
    VX_CUDA_TRY(cudaGetLastError());
    // compaction: dst index = exclusive scan of the non-empty flags (the head flags are free)
    bool done = false;
    VX_TRY(vx_scan_u32(ctx, seg.nonzero, flags, nseg, misc + 3, s, nullptr, vx_pin_of(ctx, misc + 3, 1), &done));
    if (!done) VX_TRY(vx_readback_async(ctx, 0, misc + 3, 4, s));
    VX_CUDA_TRY(cudaStreamSynchronize(s));
    const uint32_t nvox = ((uint32_t*)ctx->host_pin)[0];
    *nvox_out = nvox;
    vx_level view;
    if (dst) {
        view = *dst;
    } else {
        VX_TRY(vx_level_alloc(ctx, alloc_out, nvox, 1, 0, res, s));
        view = *alloc_out;
    }
    if (nvox > 0) {
        VX_LAUNCH(ctx, ST_FINALIZE, s, k_finalize<<<grid_for(nseg, FIN_WARPS * 32), FIN_WARPS * 32, 0, s>>>(seg, misc + 2, flags, view, key_hi));
        VX_CUDA_TRY(cudaGetLastError());
    }
    return VX_OK;
}

// The level arrays of L from row `at` on (a view for k_finalize; K = 1 rows).
inline vx_level level_view(const vx_level& L, int64_t at) {
    vx_level v = L;
    v.keys += at;
    v.mask += (size_t)at * 8;
    v.mass += at;
    v.moment += (size_t)at * 6;
    v.occ += at;
    v.occ_proj += (size_t)at * 3;
    v.lobe_count += at;
    v.lobes += (size_t)at * 7 * L.K;
    v.compact += (size_t)at * 6 * L.K;
    return v;
}

// Prepared primitives of one voxelization: records in grid coordinates (WS_REC_A/B/C).
struct Prepared {
    bool fiber;
    uint32_t np;
    int bits_R;
    int R;
    float4 *r0, *r1, *r2;   // r2: triangles' third records (fibers: none)
    uint32_t* misc;
};

vx_status prepare(vx_context* ctx, const vx_primitives* prims, const vx_grid* grid, cudaStream_t s, Prepared* P) {
    const uint32_t R = grid->resolution;
    if (R == 0 || (R & (R - 1)) != 0) return VX_ERR_INVALID_ARG;
    if (R > 2048 || grid->sub_res != 8) return VX_ERR_UNSUPPORTED;
    if (!(grid->voxel_size > 0.0f) || !isfinite(grid->voxel_size)) return VX_ERR_INVALID_ARG;
    if (prims->num_prims < 0 || prims->num_prims > 0xfffffffell) return VX_ERR_CAPACITY;
    const bool fiber = prims->kind == VX_FIBERS;
    if (!fiber && prims->kind != VX_TRIANGLES) return VX_ERR_INVALID_ARG;
    const uint32_t np = (uint32_t)prims->num_prims;
    P->fiber = fiber;
    P->np = np;
    P->R = (int)R;
    P->bits_R = 0;
    while ((1u << P->bits_R) < R) ++P->bits_R;
    P->r0 = P->r1 = P->r2 = nullptr;
    P->misc = nullptr;
    if (np == 0) return VX_OK;
    if (fiber) {
        if (!prims->ctrl || !prims->fiber_offsets || prims->num_fibers <= 0 || prims->num_ctrl < 0)
            return VX_ERR_INVALID_ARG;
        if (((uintptr_t)prims->ctrl & 15) != 0) return VX_ERR_INVALID_ARG;
    } else {
        if (!prims->tri_verts || ((uintptr_t)prims->tri_verts & 15) != 0) return VX_ERR_INVALID_ARG;
    }
    GridDev g;
    g.o[0] = grid->origin[0]; g.o[1] = grid->origin[1]; g.o[2] = grid->origin[2];
    g.s = 1.0f / grid->voxel_size;
    g.R = (int)R;
    VX_TRY(vx_ws_ensure(ctx, WS_REC_A, (size_t)np * 16, s));
    VX_TRY(vx_ws_ensure(ctx, WS_REC_B, (size_t)np * 16, s));
    if (!fiber) VX_TRY(vx_ws_ensure(ctx, WS_REC_C, (size_t)np * 16, s));
    VX_TRY(vx_ws_ensure(ctx, WS_MISC, 256, s));
    uint32_t* misc = (uint32_t*)ctx->ws[WS_MISC].p;   // [0] err, [1] npairs, [2] nseg, [3] nvox, [4] segtotal, [14] count flags, [15] large walks
    VX_CUDA_TRY(cudaMemsetAsync(misc, 0, 64, s));
    float4* r0 = (float4*)ctx->ws[WS_REC_A].p;
    float4* r1 = (float4*)ctx->ws[WS_REC_B].p;
    float4* r2 = fiber ? nullptr : (float4*)ctx->ws[WS_REC_C].p;
    if (fiber) {
        const int64_t F = prims->num_fibers;
        if (F > 0x7fffffff) return VX_ERR_CAPACITY;
        VX_TRY(vx_ws_ensure(ctx, WS_FIBER_START, (size_t)F * 4 + 256, s));
        uint32_t* fs = (uint32_t*)ctx->ws[WS_FIBER_START].p;
        VX_LAUNCH(ctx, ST_PREP, s, k_fiber_seg_counts<<<grid_for((size_t)F, 256), 256, 0, s>>>(prims->fiber_offsets, F, prims->num_ctrl, fs, misc));
        VX_TRY(vx_scan_u32(ctx, fs, fs, (uint32_t)F, misc + 4, s));
        VX_LAUNCH(ctx, ST_PREP, s, k_prep_fibers<<<grid_for(np, 256), 256, 0, s>>>((const float4*)prims->ctrl, prims->num_ctrl, prims->fiber_offsets, fs, F,
                                                         misc + 4, prims->weights, np, g, r0, r1, misc));
    } else {
        VX_LAUNCH(ctx, ST_PREP, s, k_prep_tris<<<grid_for(np, 256), 256, 0, s>>>((const float4*)prims->tri_verts, prims->weights, np, g, r0,
                                                       r1, r2, misc));
    }
    VX_CUDA_TRY(cudaGetLastError());
    vx_stage_units(ctx, ST_PREP, np);
    P->r0 = r0; P->r1 = r1; P->r2 = r2; P->misc = misc;
    return VX_OK;
}

// Windows of the region [lo, lo + 2^lg)^3 in Morton order: a window is split into its
// eight octants while it is wider than 2^max_lg voxels (max_lg <= 10: keys of one pass are
// 30-bit) or holds more candidate pairs than one pass may; octants without pairs are
// dropped.  Each window is counted (one synchronisation); the list holds every window that
// is kept, with its pair total.  VX_ERR_CAPACITY when a single voxel is over the limit.
// *counted (optional) receives the index of the leaf whose counts and offsets are still in
// the workspace (the last window counted was that leaf), or -1.
vx_status plan_windows(vx_context* ctx, const Prepared& P, const int lo[3], int lg, int max_lg, cudaStream_t s,
                       std::vector<Leaf>* leaves, int* counted) {
    if (counted) *counted = -1;
    struct Pending { int lo[3]; int lg; };
    std::vector<Pending> stack;
    stack.push_back(Pending{{lo[0], lo[1], lo[2]}, lg});
    const uint64_t limit = (uint64_t)std::min<int64_t>(ctx->max_pairs, kMaxPassPairs);
    while (!stack.empty()) {
        const Pending w = stack.back();
        stack.pop_back();
        Leaf leaf{{w.lo[0], w.lo[1], w.lo[2]}, w.lg, 0};
        uint64_t total = 0;
        VX_TRY(count_window(ctx, P.fiber, P.np, window_of(leaf), P.r0, P.r1, P.r2, P.misc, s, &total));
        if (counted) *counted = -1;
        if (total == 0) continue;                                 // an empty window adds nothing
        if (w.lg <= max_lg && total <= limit) {
            leaf.pairs = total;
            leaves->push_back(leaf);
            if (counted) *counted = (int)leaves->size() - 1;
            continue;
        }
        if (w.lg == 0) return VX_ERR_CAPACITY;                    // one voxel over the limit
        const int half = 1 << (w.lg - 1);
        for (int o = 7; o >= 0; --o) {                            // pushed in reverse: popped in Morton order
            Pending c;
            c.lg = w.lg - 1;
            c.lo[0] = w.lo[0] + ((o & 1) ? half : 0);
            c.lo[1] = w.lo[1] + ((o & 2) ? half : 0);
            c.lo[2] = w.lo[2] + ((o & 4) ? half : 0);
            stack.push_back(c);
        }
    }
    return VX_OK;
}

// Level 0 of the planned windows (Morton order), as one level block.  One window: its
// pipeline allocates the block.  Several: a first pass counts each window's candidate
// voxels (emit, sort, heads), one block is allocated for their sum, and a second pass
// reduces every window straight into its rows, so that no window is held twice.
// `counted`: index of the leaf whose counts and offsets are in the workspace (or -1).
vx_status voxelize_leaves(vx_context* ctx, const Prepared& P, const std::vector<Leaf>& leaves, int counted,
                          cudaStream_t s, vx_level* out0) {
    const int res = P.R;
    uint32_t *k0, *v0, *k1, *v1;
    for (const Leaf& w : leaves) {
        vx_stage_units(ctx, ST_COUNT, (int64_t)w.pairs);
        vx_stage_units(ctx, ST_EMIT, (int64_t)w.pairs);
        vx_stage_units(ctx, ST_SORT_SCATTER, (int64_t)w.pairs);
        vx_stage_units(ctx, ST_SORT_HIST, (int64_t)w.pairs);
        vx_stage_units(ctx, ST_REDUCE_FIBERS + (P.fiber ? 0 : 1), (int64_t)w.pairs);
    }
    if (leaves.empty()) return vx_level_alloc(ctx, out0, 0, 1, 0, res, s);
    if (leaves.size() == 1) {
        const Leaf& w = leaves[0];
        const Window win = window_of(w);
        uint64_t total = w.pairs;
        if (counted != 0) VX_TRY(count_window(ctx, P.fiber, P.np, win, P.r0, P.r1, P.r2, P.misc, s, &total));
        uint32_t nseg = 0, nvox = 0;
        VX_TRY(window_segments(ctx, P.fiber, P.np, win, w.lg, (uint32_t)total, P.r0, P.r1, P.r2, P.misc, s, &k0, &v0,
                               &k1, &v1, &nseg));
        vx_status st = window_reduce(ctx, P.fiber, P.np, nseg, key_hi_of(w), res, k0, v0, k1, v1, win, P.r0, P.r1,
                                     P.r2, P.misc, s, nullptr, out0, &nvox);
        if (st != VX_OK) vx_level_release(ctx, out0, s);
        return st;
    }
    // pass 1: candidate voxels per window (an upper bound of its voxels)
    std::vector<uint32_t> nsegs(leaves.size());
    int64_t cap = 0;
    for (size_t i = 0; i < leaves.size(); ++i) {
        const Window win = window_of(leaves[i]);
        uint64_t total = leaves[i].pairs;
        if (counted != (int)i) VX_TRY(count_window(ctx, P.fiber, P.np, win, P.r0, P.r1, P.r2, P.misc, s, &total));
        counted = (int)i;
        VX_TRY(window_segments(ctx, P.fiber, P.np, win, leaves[i].lg, (uint32_t)total, P.r0, P.r1, P.r2, P.misc, s,
                               &k0, &v0, &k1, &v1, &nsegs[i]));
        cap += nsegs[i];
    }
    VX_TRY(vx_level_alloc(ctx, out0, cap, 1, 0, res, s));
    // pass 2: every window reduced into its rows
    int64_t at = 0;
    vx_status st = VX_OK;
    for (size_t i = 0; i < leaves.size() && st == VX_OK; ++i) {
        const Window win = window_of(leaves[i]);
        uint64_t total = leaves[i].pairs;
        uint32_t nseg = 0, nvox = 0;
        if (counted != (int)i) st = count_window(ctx, P.fiber, P.np, win, P.r0, P.r1, P.r2, P.misc, s, &total);
        counted = (int)i;
        if (st == VX_OK)
            st = window_segments(ctx, P.fiber, P.np, win, leaves[i].lg, (uint32_t)total, P.r0, P.r1, P.r2, P.misc, s,
                                 &k0, &v0, &k1, &v1, &nseg);
        if (st == VX_OK && nseg != nsegs[i]) st = VX_ERR_CUDA;    // the two passes must agree
        if (st == VX_OK) {
            const vx_level view = level_view(*out0, at);
            st = window_reduce(ctx, P.fiber, P.np, nseg, key_hi_of(leaves[i]), res, k0, v0, k1, v1, win, P.r0, P.r1,
                               P.r2, P.misc, s, &view, nullptr, &nvox);
        }
        at += nvox;
    }
    if (st != VX_OK) {
        vx_level_release(ctx, out0, s);
        return st;
    }
    out0->num_voxels = at;
    return VX_OK;
}

}  // namespace

extern "C" vx_status vx_voxelize(vx_context* ctx, const vx_primitives* prims, const vx_grid* grid,
                                 void* stream, vx_level* out0) {
    if (!ctx || !prims || !grid || !out0) return VX_ERR_INVALID_ARG;
    memset(out0, 0, sizeof(*out0));
    cudaStream_t s = (cudaStream_t)stream;
    ctx->last_stream = s;
    Prepared P;
    VX_TRY(prepare(ctx, prims, grid, s, &P));
    if (P.np == 0) return vx_level_alloc(ctx, out0, 0, 1, 0, P.R, s);
    std::vector<Leaf> leaves;
    const int lo[3] = {0, 0, 0};
    int counted = -1;
    VX_TRY(plan_windows(ctx, P, lo, P.bits_R, 10, s, &leaves, &counted));
    return voxelize_leaves(ctx, P, leaves, counted, s, out0);
}

// Copies row 0 of `src` (one voxel) into row i of `dst` (same K).
static vx_status copy_root(vx_context* ctx, const vx_level& src, const vx_level& dst, int64_t i, cudaStream_t s) {
    const int K = src.K;
    VX_CUDA_TRY(cudaMemcpyAsync(dst.keys + i, src.keys, 8, cudaMemcpyDeviceToDevice, s));
    VX_CUDA_TRY(cudaMemcpyAsync(dst.mask + (size_t)i * 8, src.mask, 64, cudaMemcpyDeviceToDevice, s));
    VX_CUDA_TRY(cudaMemcpyAsync(dst.mass + i, src.mass, 4, cudaMemcpyDeviceToDevice, s));
    VX_CUDA_TRY(cudaMemcpyAsync(dst.moment + (size_t)i * 6, src.moment, 24, cudaMemcpyDeviceToDevice, s));
    VX_CUDA_TRY(cudaMemcpyAsync(dst.occ + i, src.occ, 2, cudaMemcpyDeviceToDevice, s));
    VX_CUDA_TRY(cudaMemcpyAsync(dst.occ_proj + (size_t)i * 3, src.occ_proj, 3, cudaMemcpyDeviceToDevice, s));
    VX_CUDA_TRY(cudaMemcpyAsync(dst.lobe_count + i, src.lobe_count, 1, cudaMemcpyDeviceToDevice, s));
    VX_CUDA_TRY(cudaMemcpyAsync(dst.lobes + (size_t)i * 7 * K, src.lobes, (size_t)28 * K, cudaMemcpyDeviceToDevice, s));
    VX_CUDA_TRY(cudaMemcpyAsync(dst.compact + (size_t)i * 6 * K, src.compact, (size_t)24 * K, cudaMemcpyDeviceToDevice,
                                s));
    return VX_OK;
}

extern "C" vx_status vx_voxelize_lod_windowed(vx_context* ctx, const vx_primitives* prims, const vx_grid* grid,
                                              const vx_lod_params* lod, int window_log2, vx_window_fn on_window,
                                              void* user, void* stream, vx_level* top, int* num_top) {
    if (!ctx || !prims || !grid || !lod || !on_window || !top || !num_top) return VX_ERR_INVALID_ARG;
    *num_top = 0;
    cudaStream_t s = (cudaStream_t)stream;
    ctx->last_stream = s;
    Prepared P;
    VX_TRY(prepare(ctx, prims, grid, s, &P));
    const int L = P.bits_R, w = window_log2;
    if (w < 1 || w > L) return VX_ERR_INVALID_ARG;
    if (lod->num_levels != 0) return VX_ERR_INVALID_ARG;
    if (lod->K < 1 || lod->K > vx::kMaxK) return VX_ERR_UNSUPPORTED;
    if (lod->K > 1 && (!lod->dirs || lod->n_samples < 1 || lod->n_samples > 65536)) return VX_ERR_INVALID_ARG;
    if (lod->merge != 0 && lod->merge != 1) return VX_ERR_INVALID_ARG;
    if (3 * (L - w) > 21) return VX_ERR_UNSUPPORTED;              // at most 2^21 windows
    const int K = lod->K;
    for (int l = 0; l <= L - w; ++l) memset(&top[l], 0, sizeof(vx_level));
    // the window roots (level w) are gathered here, one row per non-empty window
    vx_level roots;
    VX_TRY(vx_level_alloc(ctx, &roots, P.np ? (int64_t)1 << (3 * (L - w)) : 0, K, w, P.R >> w, s));
    vx_status st = VX_OK;
    int64_t nroots = 0;
    std::vector<Leaf> leaves;
    if (P.np) {
        const int lo[3] = {0, 0, 0};
        st = plan_windows(ctx, P, lo, P.bits_R, std::min(w, 10), s, &leaves, nullptr);
    }
    // leaves are in Morton order, so the leaves of one 2^w window are contiguous
    size_t i = 0;
    int64_t index = 0;
    while (st == VX_OK && i < leaves.size()) {
        const int sh = w;
        size_t j = i;
        while (j < leaves.size() && (leaves[j].lo[0] >> sh) == (leaves[i].lo[0] >> sh) &&
               (leaves[j].lo[1] >> sh) == (leaves[i].lo[1] >> sh) && (leaves[j].lo[2] >> sh) == (leaves[i].lo[2] >> sh))
            ++j;
        const std::vector<Leaf> group(leaves.begin() + i, leaves.begin() + j);
        vx_window info;
        for (int a = 0; a < 3; ++a) info.lo[a] = (leaves[i].lo[a] >> sh) << sh;
        info.log2_size = w;
        info.index = index;
        vx_level lv[12];
        memset(lv, 0, sizeof(lv));
        st = voxelize_leaves(ctx, P, group, -1, s, &lv[0]);
        if (st == VX_OK && lv[0].num_voxels > 0) {
            vx_lod_params wp = *lod;
            wp.num_levels = w;
            st = vx_build_lod(ctx, &lv[0], &wp, stream, &lv[1]);
            if (st == VX_OK) st = copy_root(ctx, lv[w], roots, nroots, s);
            if (st == VX_OK) {
                ++nroots;
                ++index;
                vx_level_release(ctx, &lv[w], s);
                // ownership of levels 0 .. w-1 passes to the callee, whatever it returns
                st = on_window(user, &info, lv, w, stream);
            } else {
                for (int l = 0; l <= w; ++l) vx_level_release(ctx, &lv[l], s);
            }
        } else {
            vx_level_release(ctx, &lv[0], s);
        }
        i = j;
    }
    if (st != VX_OK) {
        vx_level_release(ctx, &roots, s);
        return st;
    }
    roots.num_voxels = nroots;
    top[0] = roots;
    if (L > w) {
        vx_lod_params tp = *lod;
        tp.num_levels = L - w;
        st = vx_build_lod(ctx, &roots, &tp, stream, &top[1]);
        if (st != VX_OK) {
            vx_level_release(ctx, &top[0], s);
            return st;
        }
    }
    *num_top = L - w + 1;
    return VX_OK;
}

// =====================================================================================
// Adjoint (vx_backward)
// =====================================================================================
namespace {

// ---- level-0 adjoints: every level's gradient of a voxel's ancestors, summed -------------------
// The ancestor of voxel i at level l is the row of level l that counts the parents starting at or
// before i: key i starts a parent of level l when its bits above 3 l differ from the previous
// key's, so it starts one at every level up to head_level(i).  A warp takes 256 consecutive keys;
// k_adj_counts stores each warp's parents per level, k_adj_scan turns them into offsets, and
// k_adj_bcast ranks its keys by ballots.  The sums are FP64, whose rate bounds the pass, so they are
// taken once per level-1 parent (levels 1 and up, a quarter of the keys) and then once per voxel.
// 1.01 M voxels and 4 coarser levels: 0.116 ms against 0.17 ms when every voxel added every level
// and 0.27 ms for a flag pass, a scan and an update of the sums per level.
constexpr int ADJ_MAX_LEVELS = 11;
constexpr uint32_t ADJ_TILE = 256;   // keys per warp
struct AdjGrads {
    const float* mass[ADJ_MAX_LEVELS + 1];
    const float* moment[ADJ_MAX_LEVELS + 1];
};

// highest level at which key i starts a parent (at most L; 0: none)
__device__ __forceinline__ int head_level(const uint64_t* __restrict__ keys, uint32_t i, uint32_t n, int L) {
    if (i >= n) return 0;
    if (i == 0) return L;
    const uint64_t x = keys[i] ^ keys[i - 1];
    return x ? min((63 - __clzll((long long)x)) / 3, L) : 0;
}

__global__ void __launch_bounds__(256) k_adj_counts(const uint64_t* __restrict__ keys, uint32_t n, int L, uint32_t nw,
                                                    uint32_t* __restrict__ part) {
    const int lane = threadIdx.x & 31;
    const uint32_t w = (blockIdx.x * 256u + threadIdx.x) >> 5;
    if (w >= nw) return;
    uint32_t cnt[ADJ_MAX_LEVELS];
#pragma unroll
    for (int l = 0; l < ADJ_MAX_LEVELS; ++l) cnt[l] = 0;
    for (uint32_t r = 0; r < ADJ_TILE; r += 32) {
        const int h = head_level(keys, w * ADJ_TILE + r + lane, n, L);
#pragma unroll
        for (int l = 0; l < ADJ_MAX_LEVELS; ++l)
            if (l < L) cnt[l] += __popc(__ballot_sync(0xffffffffu, h > l));
    }
#pragma unroll
    for (int l = 0; l < ADJ_MAX_LEVELS; ++l)
        if (l < L && lane == l) part[(size_t)l * nw + w] = cnt[l];
}

// block l: exclusive scan of row l of part[L][nw], in place
__global__ void __launch_bounds__(1024) k_adj_scan(uint32_t* __restrict__ part, uint32_t nw) {
    __shared__ uint32_t ws[32];
    uint32_t* const row = part + (size_t)blockIdx.x * nw;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (uint32_t b = 0; b < nw; b += 1024) {
        const uint32_t i = b + threadIdx.x;
        const uint32_t v = i < nw ? row[i] : 0u;
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) ws[w] = inc;
        __syncthreads();
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const uint32_t t = ws[k];
            before += k < w ? t : 0u;
            total += t;
        }
        if (i < nw) row[i] = carry + before + inc - v;
        carry += total;
        __syncthreads();
    }
}

constexpr int ADJ_BC_WARPS = 4;
__global__ void __launch_bounds__(ADJ_BC_WARPS * 32) k_adj_bcast(const uint64_t* __restrict__ keys, uint32_t n, int L,
                                                                 uint32_t nw, const uint32_t* __restrict__ part,
                                                                 AdjGrads G, double* __restrict__ gm,
                                                                 double* __restrict__ gM) {
    struct Shared {
        double sum[7 * 64];                      // the parents' sums, component-major
        uint32_t row[ADJ_MAX_LEVELS * 64];       // the parents' rows in levels 1 .. L
    };
    __shared__ Shared shared[ADJ_BC_WARPS];
    Shared& sh = shared[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const uint32_t w = blockIdx.x * ADJ_BC_WARPS + (threadIdx.x >> 5);
    if (w >= nw) return;
    uint32_t base[ADJ_MAX_LEVELS];   // parents of level l + 1 before this chunk's keys
#pragma unroll
    for (int l = 0; l < ADJ_MAX_LEVELS; ++l) base[l] = l < L ? part[(size_t)l * nw + w] : 0u;
    for (uint32_t r = 0; r < ADJ_TILE; r += 64) {
        const uint32_t i0 = w * ADJ_TILE + r;
        if (i0 >= n) break;
        uint32_t loc[2] = {0, 0}, first = 0;
        if (L > 0) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const uint32_t i = i0 + 32u * half + lane;
                const int h = head_level(keys, i, n, L);
                uint32_t p[ADJ_MAX_LEVELS];
#pragma unroll
                for (int l = 0; l < ADJ_MAX_LEVELS; ++l) {
                    if (l >= L) break;
                    const uint32_t b = __ballot_sync(0xffffffffu, h > l);
                    p[l] = base[l] + __popc(b & (0xffffffffu >> (31 - lane))) - 1u;   // key i's own start counts
                    base[l] += __popc(b);
                }
                if (half == 0) first = __shfl_sync(0xffffffffu, p[0], 0);
                loc[half] = p[0] - first;
                // a parent's rows from its first key in the chunk
                if (i < n && (h > 0 || (half == 0 && lane == 0))) {
#pragma unroll
                    for (int l = 0; l < ADJ_MAX_LEVELS; ++l) {
                        if (l >= L) break;
                        sh.row[l * 64 + loc[half]] = p[l];
                    }
                }
            }
            __syncwarp();
            const uint32_t parents = base[0] - first;
            for (uint32_t q = lane; q < parents; q += 32) {
                double m = 0.0, M[6] = {0, 0, 0, 0, 0, 0};
                for (int l = 0; l < L; ++l) {
                    const uint32_t p = sh.row[l * 64 + q];
                    const float* g = G.moment[l + 1] + (size_t)p * 6;
                    m += (double)G.mass[l + 1][p];
#pragma unroll
                    for (int c = 0; c < 6; ++c) M[c] += (double)g[c];
                }
                sh.sum[q] = m;
#pragma unroll
                for (int c = 0; c < 6; ++c) sh.sum[(c + 1) * 64 + q] = M[c];
            }
            __syncwarp();
        }
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const uint32_t i = i0 + 32u * half + lane;
            if (i < n) {
                double g[7];
                g[0] = (double)G.mass[0][i];
#pragma unroll
                for (int c = 0; c < 6; ++c) g[c + 1] = (double)G.moment[0][(size_t)i * 6 + c];
                if (L > 0) {
#pragma unroll
                    for (int c = 0; c < 7; ++c) g[c] += sh.sum[c * 64 + loc[half]];
                }
                gm[i] = g[0];
#pragma unroll
                for (int c = 0; c < 6; ++c) gM[(size_t)i * 6 + c] = g[c + 1];
            }
        }
        __syncwarp();   // the sums have been read
    }
}

// gm[n], gM[n][6] from the levels' gradients; part: L * ceil(n / 256) words
cudaError_t adj_broadcast(const uint64_t* keys, uint32_t n, int L, const float* const* mass, const float* const* moment,
                          uint32_t* part, double* gm, double* gM, cudaStream_t s) {
    AdjGrads G;
    for (int l = 0; l <= ADJ_MAX_LEVELS; ++l) {
        G.mass[l] = l <= L ? mass[l] : nullptr;
        G.moment[l] = l <= L ? moment[l] : nullptr;
    }
    const uint32_t nw = (uint32_t)(((uint64_t)n + ADJ_TILE - 1) / ADJ_TILE);
    const unsigned blocks = (nw + 7) / 8;
    if (L > 0) {
        k_adj_counts<<<blocks, 256, 0, s>>>(keys, n, L, nw, part);
        k_adj_scan<<<L, 1024, 0, s>>>(part, nw);
    }
    k_adj_bcast<<<(nw + ADJ_BC_WARPS - 1) / ADJ_BC_WARPS, ADJ_BC_WARPS * 32, 0, s>>>(keys, n, L, nw, part, G, gm, gM);
    return cudaGetLastError();
}
inline size_t adj_part_bytes(uint32_t n, int L) { return ((size_t)n / ADJ_TILE + 1) * std::max(L, 1) * 4; }

// FP64 operations of the adjoint are few per clock (two lanes per SM), so what can run elsewhere
// does: reciprocals and inverse roots start from the special-function unit's approximation and take
// two steps of Newton's iteration (y + y (1 - x y) and y + y (1/2 - x y^2 / 2); relative error below
// 2^-51; no bit-exact contract here), and comparisons of
// doubles whose order is that of their bits as integers run as integers.
__device__ __forceinline__ double d_rcp(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}
__device__ __forceinline__ double d_rsqrt(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = 0.5 * x;
    y = fma(y, fma(-h * y, y, 0.5), y);
    return fma(y, fma(-h * y, y, 0.5), y);
}
// a / b, corrected by its remainder to the correctly rounded quotient of all but a few in 2^27 operands
// (those whose reciprocal is not)
__device__ __forceinline__ double d_div(double a, double b) {
    const double y = d_rcp(b), q = a * y;
    return fma(fma(-q, b, a), y, q);
}

// Per-segment constants of the fiber adjoint (grid units, FP64), in a warp's shared memory with
// the segment's slot fastest: A, d = B - A, 1 / d per component (0 for 0), unit tangent, |d|, r, w,
// 1 / |d|, 1 / r.
constexpr int SEGC = 17;
__device__ __forceinline__ void seg_constants(float4 Af, float4 Bf, double* __restrict__ c, int slot) {
    const double A[3] = {Af.x, Af.y, Af.z};
    const double d[3] = {(double)Bf.x - Af.x, (double)Bf.y - Af.y, (double)Bf.z - Af.z};
    const double d2 = fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2]));
    const bool some = d2 > 0.0;
    const double idn = some ? d_rsqrt(d2) : 0.0;
    const double dn = d2 * idn;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        c[i * 32 + slot] = A[i];
        c[(3 + i) * 32 + slot] = d[i];
        c[(6 + i) * 32 + slot] = d[i] != 0.0 ? d_rcp(d[i]) : 0.0;
        c[(9 + i) * 32 + slot] = d[i] * idn;
    }
    c[12 * 32 + slot] = dn;
    c[13 * 32 + slot] = Af.w;
    c[14 * 32 + slot] = Bf.w;
    // (a segment without length or radius has gradients that are not numbers, as 0 / 0)
    c[15 * 32 + slot] = some ? idn : INFINITY;
    c[16 * 32 + slot] = Af.w != 0.0f ? d_rcp((double)Af.w) : INFINITY;
}

// The part [t0, t1] of segment `slot` inside voxel (vi, vj, vk), and the axes whose planes cut it
// (-1: the segment's own end); false when it is empty.
__device__ __forceinline__ bool seg_clip(const double* __restrict__ c, int slot, int vi, int vj, int vk, double& t0,
                                         double& t1, int& ax0, int& ax1) {
    const int v[3] = {vi, vj, vk};
    t0 = 0.0;
    t1 = 1.0;
    ax0 = ax1 = -1;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double a = c[i * 32 + slot] - v[i], d = c[(3 + i) * 32 + slot], inv = c[(6 + i) * 32 + slot];
        const long long sign = __double_as_longlong(d);
        if ((sign & 0x7fffffffffffffffll) == 0) {
            if (a < 0.0 || a > 1.0) return false;
        } else {
            const double ta = -a * inv, tb = fma(-a, inv, inv);
            const double tn = sign >= 0 ? ta : tb, tf = sign >= 0 ? tb : ta;
            // (t0 >= 0, so a larger tn has the larger bits; once t1 is negative the part is empty,
            // whichever negative value it takes next)
            if (__double_as_longlong(tn) > __double_as_longlong(t0)) { t0 = tn; ax0 = i; }
            if (__double_as_longlong(tf) < __double_as_longlong(t1)) { t1 = tf; ax1 = i; }
        }
    }
    return __double_as_longlong(t1) > __double_as_longlong(t0);
}

// d/d(A, B, r, w) of  w * pi r^2 len * (gm + gM . T(t))  for the part [t0, t1] of segment `slot`
// in one voxel (grid units); out: dA[3], dB[3], dr, dw.  FP64: the end-point terms of a piece that
// crosses a plane almost parallel to it are large and cancel between the two voxels
// sharing the plane, so FP32 would leave an error of a few 1e-6 of their size.
__device__ __forceinline__ void pair_grad(const double* __restrict__ c, int slot, double t0, double t1, int ax0, int ax1,
                                          double gm, const double* gM, double* out) {
    // (no bit-exact contract here: the multiply-adds are fused explicitly)
    const double pi = 3.14159265358979323846;
    const double t[3] = {c[9 * 32 + slot], c[10 * 32 + slot], c[11 * 32 + slot]};
    const double dn = c[12 * 32 + slot], r = c[13 * 32 + slot], w = c[14 * 32 + slot];
    const double len = (t1 - t0) * dn;
    const double pr2 = pi * r * r;
    const double mu = pr2 * len;
    double gt[3];
    gt[0] = fma(2.0 * gM[0], t[0], fma(gM[3], t[1], gM[4] * t[2]));
    gt[1] = fma(gM[3], t[0], fma(2.0 * gM[1], t[1], gM[5] * t[2]));
    gt[2] = fma(gM[4], t[0], fma(gM[5], t[1], 2.0 * gM[2] * t[2]));
    // gm + gM . T(t) = gm + (t . gt) / 2 (T(t) pairs each off-diagonal once)
    const double tg = fma(t[0], gt[0], fma(t[1], gt[1], t[2] * gt[2]));
    const double G = fma(0.5, tg, gm);
    out[7] = mu * G;                     // d/dw
    out[6] = w * (2.0 * mu * c[16 * 32 + slot]) * G;     // d/dr
    // d len / d A, d B: the clipped ends (1 - t_e) A + t_e B move with both endpoints, and an
    // end on a voxel plane also slides along the segment (its t_e depends on the endpoints)
    const double dte = t1 - t0;
    const double f0 = ax0 >= 0 ? dn * c[(6 + ax0) * 32 + slot] : 0.0;
    const double f1 = ax1 >= 0 ? dn * c[(6 + ax1) * 32 + slot] : 0.0;
    const double sA0 = (1.0 - t0) * f0, sB0 = t0 * f0, sA1 = (1.0 - t1) * f1, sB1 = t1 * f1;
    const double kmu = w * pr2 * G;
    const double wmd = w * mu * c[15 * 32 + slot];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        double cA = -dte * t[k], cB = dte * t[k];
        if (ax0 == k) { cA += sA0; cB += sB0; }
        if (ax1 == k) { cA -= sA1; cB -= sB1; }
        const double gd = wmd * fma(-t[k], tg, gt[k]);
        out[k] = fma(kmu, cA, -gd);
        out[3 + k] = fma(kmu, cB, gd);
    }
}

// first index in keys[lo, hi) whose key is >= k (hi when none)
__device__ __forceinline__ uint32_t lower_key(const uint64_t* __restrict__ keys, uint32_t lo, uint32_t hi, uint64_t k) {
    while (lo < hi) {
        const uint32_t mid = lo + ((hi - lo) >> 1);
        if (keys[mid] < k) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Morton key of a voxel of a grid of up to 2048^3
__device__ __forceinline__ uint64_t voxel_key(uint32_t x, uint32_t y, uint32_t z) {
    return (uint64_t)vx_morton3(x, y, z) | ((uint64_t)(x >> 10) << 30) | ((uint64_t)(y >> 10) << 31) |
           ((uint64_t)(z >> 10) << 32);
}

// A voxel of a primitive waiting for its gradient: the primitive's slot in the warp and the voxel.
// A warp's entries wait in a ring of 64: fewer than 32 wait before a turn's pushes, so at most 63 do
// after it, and a push never meets one that waits.  A push may take the slot of one that has been
// read, so a __syncwarp stands between the reads and the next pushes.
constexpr uint32_t ADJ_RING = 64;
__device__ __forceinline__ uint64_t adj_entry(int slot, int x, int y, int z) {
    return ((uint64_t)slot << 36) | ((uint64_t)x << 24) | ((uint64_t)y << 12) | (uint64_t)z;
}

// Lanes walk the voxels that a segment's axis passes through, as a superset of them: slab by slab
// along the axis on which it is longest, and in a slab the box that its part there spans, widened
// by the rounding of the FP32 walk (1e-6 of the coordinates and the grid).
struct SegWalk {
    float A[3], d[3], inv, tol;
    int R, m, i1, i2;               // the slabs' axis and the other two
    int s, s_end, step;
    int lo1, hi1, lo2, hi2, c1, c2;
    bool done;
    __device__ __forceinline__ void slab() {
        for (; s <= s_end; s += step) {
            // the part inside the slab (all of it when the segment lies in one slab)
            float ta = 0.0f, tb = 1.0f;
            const float dm = sel3(m, d[0], d[1], d[2]);
            if (dm != 0.0f) {
                const float am = sel3(m, A[0], A[1], A[2]);
                const float u = ((float)s - tol - am) * inv, v = ((float)(s + 1) + tol - am) * inv;
                ta = fmaxf(fminf(u, v), 0.0f);
                tb = fminf(fmaxf(u, v), 1.0f);
            }
            const float x0 = sel3(i1, A[0], A[1], A[2]), x1 = sel3(i1, d[0], d[1], d[2]);
            const float y0 = sel3(i2, A[0], A[1], A[2]), y1 = sel3(i2, d[0], d[1], d[2]);
            const float xa = x0 + ta * x1, xb = x0 + tb * x1, ya = y0 + ta * y1, yb = y0 + tb * y1;
            lo1 = clampi(floorf(fminf(xa, xb) - tol), 0, R);
            hi1 = clampi(floorf(fmaxf(xa, xb) + tol), -1, R - 1);
            lo2 = clampi(floorf(fminf(ya, yb) - tol), 0, R);
            hi2 = clampi(floorf(fmaxf(ya, yb) + tol), -1, R - 1);
            if (lo1 <= hi1 && lo2 <= hi2) {
                c1 = lo1;
                c2 = lo2;
                return;
            }
        }
        done = true;
    }
    // floor values beyond the grid (or NaN) are brought to its edge
    static __device__ __forceinline__ int clampi(float f, int lo, int hi) {
        return f >= (float)hi ? hi : (f <= (float)lo ? lo : (f != f ? lo : (int)f));
    }
    static __device__ __forceinline__ int longest(float4 a, float4 b) {
        const float e0 = fabsf(b.x - a.x), e1 = fabsf(b.y - a.y), e2 = fabsf(b.z - a.z);
        return e0 >= e1 && e0 >= e2 ? 0 : (e1 >= e2 ? 1 : 2);
    }
    // number of slabs of a segment, and the first: an end on a plane belongs to the slabs on both sides
    // (the rounding of the clip decides which of them holds it)
    static __device__ __forceinline__ int slabs(float4 a, float4 b, int R, int m, int& first) {
        const float am = sel3(m, a.x, a.y, a.z), bm = sel3(m, b.x, b.y, b.z);
        first = clampi(ceilf(fminf(am, bm)) - 1.0f, 0, R);
        return max(clampi(floorf(fmaxf(am, bm)), -1, R - 1) - first + 1, 0);
    }
    static __device__ __forceinline__ int slabs(float4 a, float4 b, int R) {
        int first;
        return slabs(a, b, R, longest(a, b), first);
    }
    __device__ __forceinline__ void start(float4 a, float4 b, int R_, int sub, int step_) {
        R = R_;
        step = step_;
        A[0] = a.x; A[1] = a.y; A[2] = a.z;
        d[0] = b.x - a.x; d[1] = b.y - a.y; d[2] = b.z - a.z;
        m = longest(a, b);
        i1 = m == 0 ? 1 : 0;
        i2 = m == 2 ? 1 : 2;
        const float M = fmaxf(fmax3(fabsf(a.x), fabsf(a.y), fabsf(a.z)), fmax3(fabsf(b.x), fabsf(b.y), fabsf(b.z)));
        tol = 1e-6f * ((M + (float)R) + 1.0f);
        const float dm = sel3(m, d[0], d[1], d[2]);
        inv = dm != 0.0f ? 1.0f / dm : 0.0f;
        int first;
        s_end = slabs(a, b, R, m, first) + first - 1;
        s = first + sub;
        done = false;
        slab();
    }
    __device__ __forceinline__ uint64_t take(int slot) {
        const int x = m == 0 ? s : c1, y = m == 1 ? s : (m == 0 ? c1 : c2), z = m == 2 ? s : c2;
        if (++c2 > hi2) {
            c2 = lo2;
            if (++c1 > hi1) {
                s += step;
                slab();
            }
        }
        return adj_entry(slot, x, y, z);
    }
};

// Gradients of every segment, 32 >> lg segments per warp (2^lg lanes walk one segment's voxels).
// A segment's axis passes through one or two voxels while its radius makes it a candidate of
// twenty, so the voxels come from the axis alone.  They go into a queue of the warp and are taken
// 32 at a time, so that the FP64 work (the bound: 2 operations per clock and SM) runs with full
// lanes whatever the segments' lengths; each segment's terms are added in the order of its walk.
// A launch takes the segments of [least, most] slabs: with fewer than 32 lanes each, one of more than
// kWalkSlabs would keep the others waiting, and goes to a second launch with a warp each (100,000
// segments, 32 of them 200 voxels long: 0.7 ms, 1.9 ms on single lanes).
// 768k segments at 256^3: 0.34 ms (0.44 with IEEE quotients and roots), against 9.8 ms for a warp per
// segment over its candidate pairs (and 0.5 ms to count and emit those).
constexpr int ADJ_WARPS = 4;
constexpr int kWalkSlabs = 64;
__global__ void __launch_bounds__(ADJ_WARPS * 32) k_adjoint_fibers(const float4* __restrict__ ra,
                                                                   const float4* __restrict__ rb, uint32_t np, int R,
                                                                   int lg, int least, int most,
                                                                   const uint64_t* __restrict__ keys0,
                                                                   uint32_t V0, const double* __restrict__ gm,
                                                                   const double* __restrict__ gM,
                                                                   double* __restrict__ seg_grad,
                                                                   float* __restrict__ gw) {
    struct Shared {
        double c[SEGC * 32];
        double acc[8 * 32];
        uint64_t queue[ADJ_RING];
    };
    __shared__ Shared shared[ADJ_WARPS];
    Shared& sh = shared[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, slots = 32 >> lg, slot = lane >> lg, sub = lane & ((1 << lg) - 1);
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t warps = gridDim.x * ADJ_WARPS;
    for (uint64_t p0 = (uint64_t)(blockIdx.x * ADJ_WARPS + (threadIdx.x >> 5)) * slots; p0 < np;
         p0 += (uint64_t)warps * slots) {
        const uint64_t p = p0 + slot;
        __syncwarp();
        SegWalk walk;
        walk.done = true;
        bool mine = false;
        if (p < np) {
            const float4 a = ra[p], b = rb[p];
            const int n = SegWalk::slabs(a, b, R);
            mine = n >= least && n <= most;
            if (mine) {
                if (sub == 0) seg_constants(a, b, sh.c, slot);
                walk.start(a, b, R, sub, 1 << lg);
            }
        }
        const uint32_t owned = __ballot_sync(0xffffffffu, mine);
        if (owned == 0u) continue;
#pragma unroll
        for (int c = 0; c < 8; ++c) sh.acc[c * 32 + lane] = 0.0;
        uint32_t qh = 0, qn = 0;   // the first waiting entry and their number
        for (;;) {
            const bool more = !walk.done;
            const uint32_t bal = __ballot_sync(0xffffffffu, more);
            if (more) sh.queue[(qh + qn + __popc(bal & lt)) % ADJ_RING] = walk.take(slot);
            qn += __popc(bal);
            if (bal != 0u && qn < 32u) continue;
            if (qn == 0u) break;
            __syncwarp();
            // the gradients of up to 32 queued voxels
            const uint32_t taken = min(qn, 32u);
            const bool on = (uint32_t)lane < taken;
            const uint64_t e = on ? sh.queue[(qh + lane) % ADJ_RING] : 0ull;
            const int own = on ? (int)(e >> 36) : 32;
            bool hit = false;
            double g[8];
            if (on) {
                const int x = (int)(e >> 24) & 0xfff, y = (int)(e >> 12) & 0xfff, z = (int)e & 0xfff;
                double t0, t1;
                int ax0, ax1;
                if (seg_clip(sh.c, own, x, y, z, t0, t1, ax0, ax1)) {
                    const uint64_t k = voxel_key((uint32_t)x, (uint32_t)y, (uint32_t)z);
                    const uint32_t v = lower_key(keys0, 0, V0, k);
                    if (v < V0 && keys0[v] == k) {
                        double gMv[6];
#pragma unroll
                        for (int c = 0; c < 6; ++c) gMv[c] = gM[(size_t)v * 6 + c];
                        pair_grad(sh.c, own, t0, t1, ax0, ax1, gm[v], gMv, g);
                        hit = true;
                    }
                }
            }
            // entries of one segment are added one after the other, in queue order
            const uint32_t peers = __match_any_sync(0xffffffffu, hit ? own : 32 + lane);
            const int rank = __popc(peers & lt);
            for (int r = 0; __any_sync(0xffffffffu, hit && rank >= r); ++r) {
                if (hit && rank == r) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) sh.acc[c * 32 + own] += g[c];
                }
                __syncwarp();
            }
            __syncwarp();   // (also orders the reads of the entries before the next pushes)
            qh += taken;
            qn -= taken;
            if (bal == 0u && qn == 0u) break;
        }
        __syncwarp();
        for (int i = lane; i < slots * 8; i += 32)
            if ((owned >> ((i >> 3) << lg)) & 1u) seg_grad[p0 * 8 + i] = sh.acc[(i & 7) * 32 + (i >> 3)];
        if (gw && lane < slots && ((owned >> (lane << lg)) & 1u)) gw[p0 + lane] = (float)sh.acc[7 * 32 + lane];
    }
}

// Lanes per primitive (log2): one when there are primitives for the lanes of 16 warps per SM (the
// kernels' residency is of that order), more for fewer, so that few but long ones are walked
// by many lanes.
inline int adjoint_lanes_log2(uint32_t np) {
    int lg = 0;
    while (lg < 5 && ((uint64_t)np << lg) < (uint64_t)vx::kSMs * 512) ++lg;
    return lg;
}
inline unsigned adjoint_blocks(uint32_t np, int lg, int warps) {
    const uint64_t w = (((uint64_t)np << lg) + 31) / 32;
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((w + warps - 1) / warps, (uint64_t)vx::kSMs * 64));
}

// Sum over the primitives of their counts or, without counts, of the voxels in their ranges (each at
// most 2^31): no window holds more candidate pairs than that.  *large is set when some primitive's walk
// is too long for a share of a warp (see k_adjoint_fibers, k_adjoint_tris).
template <bool FIBER>
__global__ void k_range_bound(const float4* __restrict__ r0, const float4* __restrict__ r1, const float4* __restrict__ r2,
                              uint32_t np, Window R, const uint32_t* __restrict__ cnt,
                              unsigned long long* __restrict__ total, uint32_t* __restrict__ large) {
    unsigned long long acc = 0;
    bool any = false;
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
        const float4 a = r0[p], b = r1[p];
        const Range rg = FIBER ? capsule_range(a, b, R) : tri_range(a, b, r2[p], R);
        acc += cnt ? (unsigned long long)cnt[p] : (unsigned long long)min(rg.total, 0x80000000ll);
        any = any || (FIBER ? SegWalk::slabs(a, b, R.hi[0] + 1) > kWalkSlabs : rg.total > kGroupRange);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0 && acc) atomicAdd(total, acc);
    if (any) *large = 1u;
}

// The gradients of all segments; `large`: some are left to a second launch.
void adjoint_fibers(const float4* r0, const float4* r1, uint32_t np, int R, bool large, const uint64_t* keys0, uint32_t V0,
                    const double* gm, const double* gM, double* seg_grad, float* gw, cudaStream_t s) {
    const int lg = adjoint_lanes_log2(np);
    const bool split = large && lg < 5;
    k_adjoint_fibers<<<adjoint_blocks(np, lg, ADJ_WARPS), ADJ_WARPS * 32, 0, s>>>(
        r0, r1, np, R, lg, 0, split ? kWalkSlabs : kAnyRange, keys0, V0, gm, gM, seg_grad, gw);
    if (split)
        k_adjoint_fibers<<<adjoint_blocks(np, 5, ADJ_WARPS), ADJ_WARPS * 32, 0, s>>>(
            r0, r1, np, R, 5, kWalkSlabs + 1, kAnyRange, keys0, V0, gm, gM, seg_grad, gw);
}

// thread per control point: world-unit gradients from the segment before and after it
__global__ void k_adjoint_ctrl(const int64_t* __restrict__ off, int64_t F, const uint32_t* __restrict__ seg_start,
                               int64_t P, const double* __restrict__ seg_grad, float s, float4* __restrict__ gctrl) {
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= P) return;
    int64_t lo = 0, hi = F;       // last fiber with off[f] <= c
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (off[mid] <= c) lo = mid + 1; else hi = mid;
    }
    const int64_t f = lo - 1;
    float4 g = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (f >= 0 && c < off[f + 1]) {
        const bool has_prev = c > off[f];
        const bool has_next = c + 1 < off[f + 1];
        double px = 0.0, py = 0.0, pz = 0.0, pr = 0.0, nx = 0.0, ny = 0.0, nz = 0.0, nr = 0.0;
        if (has_prev) {
            const double* q = seg_grad + (size_t)(seg_start[f] + (uint32_t)(c - 1 - off[f])) * 8;
            px = q[3]; py = q[4]; pz = q[5]; pr = q[6];
        }
        if (has_next) {
            const double* q = seg_grad + (size_t)(seg_start[f] + (uint32_t)(c - off[f])) * 8;
            nx = q[0]; ny = q[1]; nz = q[2]; nr = q[6];
        }
        g.x = (float)((px + nx) * (double)s);
        g.y = (float)((py + ny) * (double)s);
        g.z = (float)((pz + nz) * (double)s);
        g.w = (float)((pr + nr) * (0.5 * (double)s));
    }
    gctrl[c] = g;
}

// d/d(U0, U1, U2, w) of  w * area(T ∩ voxel) * (gm + gM . T(n))  for one (triangle, voxel)
// pair (grid units, FP64); out[3j + k] = d/dU_j[k], out[9] = d/dw; false when the area is zero.
// The triangle is the image of the reference triangle {s, t >= 0, s + t <= 1} under
// (s, t) -> U0 + s e1 + t e2, so area(T ∩ voxel) = J * A, J = |e1 x e2|, A the area of
// the reference polygon cut out by the six voxel half-planes.  A box constraint
// g(s, t) <= 0 whose value changes by dg when a vertex moves shifts its polygon edge
// outward by -dg / |grad g|, so dA = -sum over the polygon's edges on box planes of
// (edge length / |grad g|) * dg(edge midpoint) (dg is affine in s, t).  Such an edge runs along
// the direction (-e2_k, e1_k), |(e1_k, e2_k)| = |grad g|, so the quotient is its component in
// that direction over |grad g|^2.  The clip decisions are taken on voxel-local coordinates, as the
// forward's clip takes them: a vertex or an edge lying exactly on a voxel plane (a heightfield's
// border row) stays inside, and its derivative is that of the piece it belongs to.
// What decides (the crossings, the area's and the normal's vanishing) is computed with IEEE quotients,
// products and sums, not fused: where vertices lie on voxel planes, rounding takes exact cases back to
// themselves (1 - 3 * fl(1/3) = 0, a * b - b * a = 0), and a fused operation leaves a residue that moves
// an edge from one of two planes to the other, or gives an empty piece an area and a normal: of 323
// triangles with whole coordinates the derivatives of the area over all voxels then missed that of the
// whole for 40 instead of 13.  They cost 0.06 ms of the 1.17 that the mesh below takes.
// Only the planes that some vertex of the triangle lies beyond are clipped against.
// buf: the warp's two polygons, ADJ_POLY doubles (element (poly, vertex, coord) of lane t at
// [((poly * ADJ_VERTS + vertex) * 5 + coord) * 32 + t]); a vertex carries x, y, z (exact for the
// triangle's own vertices) and s, t.
// (six planes cut a triangle into a polygon of at most nine vertices)
constexpr int ADJ_VERTS = 9;
constexpr int ADJ_POLY = 2 * ADJ_VERTS * 5 * 32;
// Called by the whole warp, `on` telling which lanes have a pair: every clip is made by all lanes that
// need one together.
__device__ __forceinline__ bool tri_pair_grad(bool on, const float4 P0, const float4 P1, const float4 P2, int vi, int vj,
                                              int vk, const double* __restrict__ gmp, const double* __restrict__ gMp,
                                              double* __restrict__ buf, double* out) {
    const int lane = threadIdx.x & 31;
    auto at = [&](int poly, int v, int c) -> double& { return buf[((poly * ADJ_VERTS + v) * 5 + c) * 32 + lane]; };
    const int vox[3] = {vi, vj, vk};
    const float U[3][3] = {{P0.x, P0.y, P0.z}, {P1.x, P1.y, P1.z}, {P2.x, P2.y, P2.z}};
    uint32_t need = 0;   // bit 2 k + side: plane k = vox (side 0) or vox + 1 has a vertex beyond it
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (fminf(fminf(U[0][k], U[1][k]), U[2][k]) < (float)vox[k]) need |= 1u << (2 * k);
        if (fmaxf(fmaxf(U[0][k], U[1][k]), U[2][k]) > (float)(vox[k] + 1)) need |= 2u << (2 * k);
#pragma unroll
        for (int v = 0; v < 3; ++v) at(0, v, k) = (double)(U[v][k] + 0.0f) - vox[k];   // (-0 becomes +0)
    }
    at(0, 0, 3) = 0.0; at(0, 0, 4) = 0.0;
    at(0, 1, 3) = 1.0; at(0, 1, 4) = 0.0;
    at(0, 2, 3) = 0.0; at(0, 2, 4) = 1.0;
    // label of the edge i -> i + 1, four bits each: 0 a triangle edge, 1 + plane a voxel plane
    uint64_t lab = 0;
    int n = 3, cur = 0;
    if (!on) need = 0;
    while (__any_sync(0xffffffffu, need != 0u)) {
        const bool work = need != 0u;
        const int c = work ? __ffs(need) - 1 : 0, k = c >> 1;
        need &= need - 1u;
        const bool hi = c & 1;
        // inside x >= 0 (x <= 1), on the bits as integers: the polygon holds no negative zero (the
        // sums below give none from values that are none)
        uint32_t in = 0;
        if (work)
            for (int i = 0; i < n; ++i) {
                const long long x = __double_as_longlong(at(cur, i, k));
                in |= (hi ? x <= 0x3ff0000000000000ll : x >= 0ll) ? 1u << i : 0u;
            }
        __syncwarp();
        const uint32_t whole = (1u << n) - 1u;
        if (work && in == 0u) {
            n = 0;
            need = 0;
        }
        if (work && in != 0u && in != whole) {
            const double bound = hi ? 1.0 : 0.0;
            const int nx = cur ^ 1;
            uint64_t qlab = 0;
            int m = 0;
            // the vertices inside whose predecessor is outside: one, unless rounding has bent the
            // polygon.  Then the part inside is one run, s .. e, and its two crossings are computed
            // together, instead of in every turn of a loop over the edges.
            const uint32_t before = ((in << 1) | (in >> (n - 1))) & whole;   // bit i: vertex i - 1 is inside
            const uint32_t entries = in & ~before;
            const int run = __popc(in);
            if ((entries & (entries - 1u)) == 0u && run + 2 <= ADJ_VERTS) {
                const int s = __ffs(entries) - 1, p = s == 0 ? n - 1 : s - 1;
                const int e = s + run - 1 >= n ? s + run - 1 - n : s + run - 1, f = e + 1 == n ? 0 : e + 1;
                const double x0 = at(cur, p, k), x1 = at(cur, e, k);
                const double l0 = d_div(bound - x0, at(cur, s, k) - x0), l1 = d_div(bound - x1, at(cur, f, k) - x1);
                // the order of the loop below: from vertex 0 on when it is inside, else from the crossing
                // before s
                m = run + 2;
                const int w0 = s == 0 ? m - 1 : (in & 1u ? e + 2 : 0);
                const int w1 = w0 == 0 ? m - 1 : w0 - 1;
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    if (q == k) {
                        at(nx, w0, q) = at(nx, w1, q) = bound;
                    } else if (q > k) {   // (no plane is left on the axes before k)
                        const double a0 = at(cur, p, q), a1 = at(cur, e, q);
                        at(nx, w0, q) = a0 + l0 * (at(cur, s, q) - a0);
                        at(nx, w1, q) = a1 + l1 * (at(cur, f, q) - a1);
                    }
                }
                qlab = (((lab >> (4 * p)) & 15u) << (4 * w0)) | ((uint64_t)(c + 1) << (4 * w1));
                int i = s, w = w0 + 1 == m ? 0 : w0 + 1;
                for (int j = 0; j < run; ++j) {
#pragma unroll
                    for (int q = 0; q < 5; ++q) at(nx, w, q) = at(cur, i, q);
                    qlab |= ((lab >> (4 * i)) & 15u) << (4 * w);
                    i = i + 1 == n ? 0 : i + 1;
                    w = w + 1 == m ? 0 : w + 1;
                }
            } else {
                for (int i = 0; i < n; ++i) {
                    const int j = i + 1 == n ? 0 : i + 1;
                    const bool a = (in >> i) & 1u, b = (in >> j) & 1u;
                    const uint64_t li = (lab >> (4 * i)) & 15u;
                    if (a && m < ADJ_VERTS) {
                        for (int q = 0; q < 5; ++q) at(nx, m, q) = at(cur, i, q);
                        qlab |= li << (4 * m);
                        ++m;
                    }
                    if (a != b && m < ADJ_VERTS) {
                        const double xi = at(cur, i, k), l = d_div(bound - xi, at(cur, j, k) - xi);
                        for (int q = 0; q < 5; ++q) {
                            const double y = at(cur, i, q);
                            at(nx, m, q) = q == k ? bound : y + l * (at(cur, j, q) - y);
                        }
                        qlab |= (a ? (uint64_t)(c + 1) : li) << (4 * m);
                        ++m;
                    }
                }
            }
            n = m;
            lab = qlab;
            cur = nx;
        }
        __syncwarp();
    }
    if (!on || n < 3) return false;
    const double e1[3] = {(double)P1.x - P0.x, (double)P1.y - P0.y, (double)P1.z - P0.z};
    const double e2[3] = {(double)P2.x - P0.x, (double)P2.y - P0.y, (double)P2.z - P0.z};
    double ig2[3];   // 1 / |grad g|^2 per axis (0: the plane's constraint does not vary)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double g2 = fma(e1[k], e1[k], e2[k] * e2[k]);
        ig2[k] = g2 > 0.0 ? d_rcp(g2) : 0.0;
    }
    double A = 0.0;
    double dA[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    double si = at(cur, 0, 3), ti = at(cur, 0, 4);
    const double s0 = si, t0 = ti;
    for (int i = 0; i < n; ++i) {
        const bool last = i + 1 == n;
        const double sj = last ? s0 : at(cur, i + 1, 3), tj = last ? t0 : at(cur, i + 1, 4);
        A = A + (si * tj - sj * ti);
        const int c = (int)((lab >> (4 * i)) & 15u) - 1;
        if (c >= 0) {
            const int k = c >> 1;
            const double a = k == 0 ? e1[0] : (k == 1 ? e1[1] : e1[2]), b = k == 0 ? e2[0] : (k == 1 ? e2[1] : e2[2]);
            const double g = k == 0 ? ig2[0] : (k == 1 ? ig2[1] : ig2[2]);
            const double len = fabs(fma(tj - ti, a, (si - sj) * b)) * g;
            const double f = (c & 1) ? -len : len;
            const double sm = 0.5 * (si + sj), tm = 0.5 * (ti + tj);
            const double d1 = f * sm, d2 = f * tm, d0 = (f - d1) - d2;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (k == q) {
                    dA[0][q] += d0;
                    dA[1][q] += d1;
                    dA[2][q] += d2;
                }
        }
        si = sj;
        ti = tj;
    }
    A *= 0.5;
    const double nr[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
    const double J2 = fma(nr[0], nr[0], fma(nr[1], nr[1], nr[2] * nr[2]));
    if (!(J2 > 0.0) || !(A > 0.0)) return false;
    const double iJ = d_rsqrt(J2), J = J2 * iJ;
    const double nh[3] = {nr[0] * iJ, nr[1] * iJ, nr[2] * iJ};
    const double mu = J * A;
    double gM[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) gM[c] = gMp[c];
    double gt[3];
    gt[0] = fma(2.0 * gM[0], nh[0], fma(gM[3], nh[1], gM[4] * nh[2]));
    gt[1] = fma(gM[3], nh[0], fma(2.0 * gM[1], nh[1], gM[5] * nh[2]));
    gt[2] = fma(gM[4], nh[0], fma(gM[5], nh[1], 2.0 * gM[2] * nh[2]));
    const double ng = fma(nh[0], gt[0], fma(nh[1], gt[1], nh[2] * gt[2]));
    // gm + gM . T(n) = gm + (n . gt) / 2 (T(n) pairs each off-diagonal once)
    const double G = fma(0.5, ng, *gmp);
    // q = d G / d (raw normal)
    const double q[3] = {fma(-nh[0], ng, gt[0]) * iJ, fma(-nh[1], ng, gt[1]) * iJ, fma(-nh[2], ng, gt[2]) * iJ};
    const double w = P0.w;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        // d J / d U_j = (U_j+1 - U_j+2) x nh,  d G / d U_j = (U_j+1 - U_j+2) x q
        const int j1 = (j + 1) % 3, j2 = (j + 2) % 3;
        const double d[3] = {(double)U[j1][0] - U[j2][0], (double)U[j1][1] - U[j2][1], (double)U[j1][2] - U[j2][2]};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
            const double dJ = fma(d[k1], nh[k2], -d[k2] * nh[k1]), dG = fma(d[k1], q[k2], -d[k2] * q[k1]);
            out[3 * j + k] = w * fma(fma(dJ, A, J * dA[j][k]), G, mu * dG);
        }
    }
    out[9] = mu * G;
    return true;
}

// Gradients of every triangle (world units, [T][3] float4 with w = 0, and the weights), 32 >> lg
// triangles per block of one warp: lanes test the voxels of their triangle's box and queue its
// candidates, which are taken 32 at a time so that the FP64 work runs with full lanes; each
// triangle's terms are added in the order in which its lanes found them.  A launch takes the triangles
// whose boxes hold [least, most] voxels: with fewer than 32 lanes each, one of more than kGroupRange
// would keep the others waiting, and goes to a second launch with a warp each (100,000 triangles, 32 of
// them 150 voxels wide: 33 ms, 763 ms on single lanes).  One warp per block: its
// polygons take 23 KB of shared memory, which leaves eight resident per SM, enough for the FP64
// pipe that bounds the kernel (77 % busy).  178,802 triangles at 256^3: 1.17 ms; 1.6 ms with the
// crossings inside a loop over the edges, 1.8 ms with each lane clipping at its own pace, 10.1 ms for
// a warp per triangle (eight pairs in its lanes), six planes and polygons in local memory.
__global__ void __launch_bounds__(32) k_adjoint_tris(const float4* __restrict__ r0, const float4* __restrict__ r1,
                                                     const float4* __restrict__ r2, uint32_t np, Window R, int lg,
                                                     int least, int most, const uint64_t* __restrict__ keys0, uint32_t V0,
                                                     const double* __restrict__ gm, const double* __restrict__ gM,
                                                     float scale, float4* __restrict__ gverts, float* __restrict__ gw) {
    __shared__ double poly[ADJ_POLY];
    __shared__ double acc[10 * 32];
    __shared__ uint64_t queue[ADJ_RING];
    const int lane = threadIdx.x, slots = 32 >> lg, slot = lane >> lg, sub = lane & ((1 << lg) - 1);
    const uint32_t lt = (1u << lane) - 1u;
    for (uint64_t p0 = (uint64_t)blockIdx.x * slots; p0 < np; p0 += (uint64_t)gridDim.x * slots) {
        const uint64_t p = p0 + slot;
        __syncwarp();
        float4 a, b, c;
        Range rg;
        rg.total = 0;
        if (p < np) {
            a = r0[p];
            b = r1[p];
            c = r2[p];
            rg = tri_range(a, b, c, R);
        }
        const bool mine = p < np && capped_total(rg) >= least && capped_total(rg) <= most;
        const uint32_t owned = __ballot_sync(0xffffffffu, mine);
        if (owned == 0u) continue;
        if (!mine) rg.total = 0;
        long long idx = sub;
#pragma unroll
        for (int k = 0; k < 10; ++k) acc[k * 32 + lane] = 0.0;
        uint32_t qh = 0, qn = 0;   // the first waiting entry and their number
        for (;;) {
            bool push = false;
            int x = 0, y = 0, z = 0;
            const bool more = __any_sync(0xffffffffu, idx < rg.total);
            if (idx < rg.total) {
                int ix, iy, iz;
                voxel_of(idx, rg.total, rg, ix, iy, iz);
                x = rg.lo[0] + ix; y = rg.lo[1] + iy; z = rg.lo[2] + iz;
                push = tri_voxel_candidate(a, b, c, x, y, z);
                idx += 1 << lg;
            }
            const uint32_t bal = __ballot_sync(0xffffffffu, push);
            if (push) queue[(qh + qn + __popc(bal & lt)) % ADJ_RING] = adj_entry(slot, x, y, z);
            qn += __popc(bal);
            if (more && qn < 32u) continue;
            if (qn == 0u) break;
            __syncwarp();
            const uint32_t taken = min(qn, 32u);
            const bool on = (uint32_t)lane < taken;
            const uint64_t e = on ? queue[(qh + lane) % ADJ_RING] : 0ull;
            const int own = on ? (int)(e >> 36) : 32;
            double g[10];
            int ex = 0, ey = 0, ez = 0;
            uint32_t v = 0;
            float4 A = make_float4(0, 0, 0, 0), B = A, C = A;
            bool found = false;
            if (on) {
                ex = (int)(e >> 24) & 0xfff, ey = (int)(e >> 12) & 0xfff, ez = (int)e & 0xfff;
                const uint64_t k = voxel_key((uint32_t)ex, (uint32_t)ey, (uint32_t)ez);
                v = lower_key(keys0, 0, V0, k);
                found = v < V0 && keys0[v] == k;
                A = r0[p0 + own];
                B = r1[p0 + own];
                C = r2[p0 + own];
            }
            const bool hit = tri_pair_grad(found, A, B, C, ex, ey, ez, gm + v, gM + (size_t)v * 6, poly, g);
            // entries of one triangle are added one after the other, in queue order
            const uint32_t peers = __match_any_sync(0xffffffffu, hit ? own : 32 + lane);
            const int rank = __popc(peers & lt);
            for (int r = 0; __any_sync(0xffffffffu, hit && rank >= r); ++r) {
                if (hit && rank == r) {
#pragma unroll
                    for (int k = 0; k < 10; ++k) acc[k * 32 + own] += g[k];
                }
                __syncwarp();
            }
            __syncwarp();   // (also orders the reads of the entries before the next pushes)
            qh += taken;
            qn -= taken;
            if (!more && qn == 0u) break;
        }
        __syncwarp();
        for (int i = lane; i < slots * 3; i += 32) {
            const int t = i / 3, j = i - 3 * t;
            if ((owned >> (t << lg)) & 1u)
                gverts[(p0 + t) * 3 + j] =
                    make_float4((float)(acc[(3 * j) * 32 + t] * (double)scale), (float)(acc[(3 * j + 1) * 32 + t] * (double)scale),
                                (float)(acc[(3 * j + 2) * 32 + t] * (double)scale), 0.0f);
        }
        if (gw && lane < slots && ((owned >> (lane << lg)) & 1u)) gw[p0 + lane] = (float)acc[9 * 32 + lane];
    }
}

}  // namespace

extern "C" vx_status vx_backward(vx_context* ctx, const vx_primitives* prims, const vx_grid* grid,
                                 const uint64_t* keys0, int64_t num_voxels0, int num_levels,
                                 const float* const* grad_mass, const float* const* grad_moment, void* stream,
                                 float* grad_ctrl, float* grad_weights) {
    if (!ctx || !prims || !grid || !grad_mass || !grad_moment || !grad_ctrl) return VX_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    ctx->last_stream = s;
    const bool fiber = prims->kind == VX_FIBERS;
    if (!fiber && prims->kind != VX_TRIANGLES) return VX_ERR_INVALID_ARG;
    const uint32_t R = grid->resolution;
    if (R == 0 || (R & (R - 1)) != 0) return VX_ERR_INVALID_ARG;
    if (R > 2048 || grid->sub_res != 8) return VX_ERR_UNSUPPORTED;
    if (num_voxels0 < 0 || num_voxels0 > 0xffffffffll || num_levels < 0 || num_levels > 11) return VX_ERR_INVALID_ARG;
    if ((num_voxels0 > 0 && !keys0) || !(grid->voxel_size > 0.0f) || !isfinite(grid->voxel_size))
        return VX_ERR_INVALID_ARG;
    if (fiber && prims->num_ctrl < 0) return VX_ERR_INVALID_ARG;
    if (prims->num_prims < 0 || prims->num_prims > 0xfffffffell) return VX_ERR_CAPACITY;
    if (((uintptr_t)grad_ctrl & 15) != 0) return VX_ERR_INVALID_ARG;
    if (fiber && (!prims->ctrl || !prims->fiber_offsets || prims->num_fibers <= 0 || ((uintptr_t)prims->ctrl & 15) != 0))
        return VX_ERR_INVALID_ARG;
    if (!fiber && prims->num_prims > 0 && (!prims->tri_verts || ((uintptr_t)prims->tri_verts & 15) != 0))
        return VX_ERR_INVALID_ARG;
    for (int l = 0; l <= num_levels; ++l)
        if (!grad_mass[l] || !grad_moment[l]) return VX_ERR_INVALID_ARG;
    const uint32_t np = (uint32_t)prims->num_prims;
    const uint32_t V0 = (uint32_t)num_voxels0;
    const int64_t P = fiber ? prims->num_ctrl : 3 * (int64_t)np, F = prims->num_fibers;
    GridDev g;
    g.o[0] = grid->origin[0]; g.o[1] = grid->origin[1]; g.o[2] = grid->origin[2];
    g.s = 1.0f / grid->voxel_size;
    g.R = (int)R;
    if (P) VX_CUDA_TRY(cudaMemsetAsync(grad_ctrl, 0, (size_t)P * 16, s));
    if (grad_weights && np) VX_CUDA_TRY(cudaMemsetAsync(grad_weights, 0, (size_t)np * 4, s));
    if (np == 0) return VX_OK;

    // ---- level-0 adjoints (coarse adjoints broadcast down) ------------------------------
    VX_TRY(vx_ws_ensure(ctx, WS_LOD_FLAGS, adj_part_bytes(V0, num_levels), s));
    VX_TRY(vx_ws_ensure(ctx, WS_LOD_TMP, (size_t)std::max<uint32_t>(V0, 1) * 56, s));
    double* gm = (double*)ctx->ws[WS_LOD_TMP].p;
    double* gM = gm + V0;
    if (V0) {
        cudaError_t e = cudaSuccess;
        VX_LAUNCH(ctx, ST_LOD_HEADS, s, e = adj_broadcast(keys0, V0, num_levels, grad_mass, grad_moment,
                                                          (uint32_t*)ctx->ws[WS_LOD_FLAGS].p, gm, gM, s));
        VX_CUDA_TRY(e);
        if (num_levels > 0) ctx->launches[ST_LOD_HEADS] += 2;   // (three kernels in one bracket)
    }
    Prepared Pp;
    VX_TRY(prepare(ctx, prims, grid, s, &Pp));
    float4 *r0 = Pp.r0, *r1 = Pp.r1, *r2 = Pp.r2;
    uint32_t* misc = Pp.misc;
    if (fiber) VX_TRY(vx_ws_ensure(ctx, WS_SEG_OUT, (size_t)np * 64, s));
    double* pgrad = (double*)ctx->ws[WS_SEG_OUT].p;
    // ---- the per-pass pair limit ---------------------------------------------------------
    // The gradients take no pair buffers, but a voxel over the limit is refused as in vx_voxelize.
    // The voxels of the primitives' ranges bound the pairs of any window; only when they pass the
    // limit are the windows counted.
    const Window full = full_window((int)R);
    unsigned long long* t64 = (unsigned long long*)(misc + 8);
    const unsigned bblocks = (unsigned)std::min<size_t>(grid_for(np, 256), (size_t)vx::kSMs * 8);
    if (fiber)
        VX_LAUNCH(ctx, ST_COUNT, s, k_range_bound<true><<<bblocks, 256, 0, s>>>(r0, r1, nullptr, np, full, nullptr, t64,
                                                                              misc + 15));
    else
        VX_LAUNCH(ctx, ST_COUNT, s, k_range_bound<false><<<bblocks, 256, 0, s>>>(r0, r1, r2, np, full, nullptr, t64,
                                                                               misc + 15));
    VX_CUDA_TRY(cudaGetLastError());
    VX_TRY(vx_readback_async(ctx, 0, misc, 64, s));
    VX_CUDA_TRY(cudaStreamSynchronize(s));
    if (((uint32_t*)ctx->host_pin)[0]) return VX_ERR_INVALID_ARG;
    const bool large = ((uint32_t*)ctx->host_pin)[15] != 0;
    if (((const uint64_t*)ctx->host_pin)[4] > (uint64_t)std::min<int64_t>(ctx->max_pairs, kMaxPassPairs)) {
        std::vector<Leaf> leaves;
        const int lo0[3] = {0, 0, 0};
        VX_TRY(plan_windows(ctx, Pp, lo0, Pp.bits_R, 10, s, &leaves, nullptr));
    }
    // ---- gradients ------------------------------------------------------------------------
    const int lg = adjoint_lanes_log2(np);
    const bool split = large && lg < 5;
    if (!fiber) {
        // (no sharing between triangles: no scatter)
        VX_LAUNCH(ctx, ST_REDUCE_TRIS, s, k_adjoint_tris<<<adjoint_blocks(np, lg, 1), 32, 0, s>>>(
                                              r0, r1, r2, np, full, lg, 0, split ? kGroupRange : kAnyRange, keys0, V0, gm,
                                              gM, g.s, (float4*)grad_ctrl, grad_weights));
        if (split)
            VX_LAUNCH(ctx, ST_REDUCE_TRIS, s, k_adjoint_tris<<<adjoint_blocks(np, 5, 1), 32, 0, s>>>(
                                                  r0, r1, r2, np, full, 5, kGroupRange + 1, kAnyRange, keys0, V0, gm, gM,
                                                  g.s, (float4*)grad_ctrl, grad_weights));
        VX_CUDA_TRY(cudaGetLastError());
        return VX_OK;
    }
    VX_LAUNCH(ctx, ST_REDUCE_FIBERS, s, adjoint_fibers(r0, r1, np, (int)R, large, keys0, V0, gm, gM, pgrad, grad_weights, s));
    if (split) ctx->launches[ST_REDUCE_FIBERS] += 1;   // (two kernels in one bracket)
    // per-segment gradients to control points
    uint32_t* fs = (uint32_t*)ctx->ws[WS_FIBER_START].p;
    VX_LAUNCH(ctx, ST_FINALIZE, s, k_adjoint_ctrl<<<grid_for((size_t)P, 256), 256, 0, s>>>(
                                       prims->fiber_offsets, F, fs, P, pgrad, g.s, (float4*)grad_ctrl));
    VX_CUDA_TRY(cudaGetLastError());
    return VX_OK;
}

// =====================================================================================
// vx_backward_noalloc: the adjoint with its scratch in a fixed device array
// =====================================================================================
// For callers that cannot allocate device memory.  The scratch is one file-scope device
// array, sized for the limits below, held by every device that loads the library until
// the process exits.  Host code must not pass the array's name to a kernel (on the host
// it names a host-side stand-in): its device address is fetched once per device with
// cudaGetSymbolAddress and cached.
namespace {

constexpr uint32_t NA_MAX_PRIMS = 1u << 16;    // 65,536 segments
constexpr uint32_t NA_MAX_FIBERS = 1u << 13;   // 8,192 fibers
constexpr uint32_t NA_MAX_PAIRS = 1u << 21;    // 2,097,152 candidate (voxel, segment) pairs
constexpr uint32_t NA_MAX_VOXELS = 1u << 18;   // 262,144 level-0 voxels

constexpr size_t na_al(size_t x) { return (x + 255) & ~size_t(255); }
constexpr size_t NA_RA = 0;
constexpr size_t NA_RB = NA_RA + na_al(16ull * NA_MAX_PRIMS);
constexpr size_t NA_CNT = NA_RB + na_al(16ull * NA_MAX_PRIMS);
constexpr size_t NA_FS = NA_CNT + na_al(4ull * NA_MAX_PRIMS);
constexpr size_t NA_MISC = NA_FS + na_al(4ull * NA_MAX_FIBERS + 4);
constexpr size_t NA_SEG = NA_MISC + 256;
constexpr size_t NA_GM = NA_SEG + na_al(64ull * NA_MAX_PRIMS);
constexpr size_t NA_GMM = NA_GM + na_al(8ull * NA_MAX_VOXELS);
constexpr size_t NA_ADJ = NA_GMM + na_al(48ull * NA_MAX_VOXELS);
constexpr size_t NA_PART = NA_ADJ + na_al(4ull * ADJ_MAX_LEVELS * (NA_MAX_VOXELS / ADJ_TILE + 1));
constexpr size_t NA_BYTES = NA_PART + na_al(4ull * (NA_MAX_VOXELS / 2048 + 64));   // ~21 MB

static __device__ __align__(256) unsigned char g_noalloc_scratch[NA_BYTES];

std::mutex g_na_mutex;
unsigned char* g_na_ptr[256] = {};

// device address of the scratch array on the current device (set up on first use); the
// stream must belong to that device, or the address would be another device's
vx_status na_scratch(cudaStream_t s, unsigned char** out) {
    int dev = 0, sdev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return VX_ERR_CUDA;
    if (cudaStreamGetDevice(s, &sdev) != cudaSuccess) return VX_ERR_INVALID_ARG;
    if (sdev != dev) return VX_ERR_INVALID_ARG;
    if (dev < 0 || dev >= 256) return VX_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return VX_ERR_CUDA;
        g_na_ptr[dev] = (unsigned char*)p;
    }
    *out = g_na_ptr[dev];
    return VX_OK;
}

}  // namespace

#define NA_TRY(expr)                                   \
    do {                                               \
        if ((expr) != cudaSuccess) return VX_ERR_CUDA; \
    } while (0)

extern "C" vx_status vx_backward_noalloc(const vx_primitives* prims, const vx_grid* grid, const uint64_t* keys0,
                                         int64_t num_voxels0, int num_levels, const float* const* grad_mass,
                                         const float* const* grad_moment, void* stream, float* grad_ctrl,
                                         float* grad_weights) {
    if (!prims || !grid || !grad_mass || !grad_moment || !grad_ctrl) return VX_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (prims->kind != VX_FIBERS) return VX_ERR_UNSUPPORTED;
    const uint32_t R = grid->resolution;
    if (R == 0 || (R & (R - 1)) != 0) return VX_ERR_INVALID_ARG;
    if (R > 1024 || grid->sub_res != 8) return VX_ERR_UNSUPPORTED;
    if (num_voxels0 < 0 || num_levels < 0 || num_levels > 11 || prims->num_prims < 0 || prims->num_fibers <= 0 ||
        prims->num_ctrl < 0 || (num_voxels0 > 0 && !keys0) || !(grid->voxel_size > 0.0f) ||
        !isfinite(grid->voxel_size))
        return VX_ERR_INVALID_ARG;
    if (prims->num_prims > (int64_t)NA_MAX_PRIMS || prims->num_fibers > (int64_t)NA_MAX_FIBERS ||
        num_voxels0 > (int64_t)NA_MAX_VOXELS)
        return VX_ERR_CAPACITY;
    if (!prims->ctrl || !prims->fiber_offsets || ((uintptr_t)prims->ctrl & 15) != 0 ||
        ((uintptr_t)grad_ctrl & 15) != 0)
        return VX_ERR_INVALID_ARG;
    for (int l = 0; l <= num_levels; ++l)
        if (!grad_mass[l] || !grad_moment[l]) return VX_ERR_INVALID_ARG;
    unsigned char* base = nullptr;
    VX_TRY(na_scratch(s, &base));
    const uint32_t np = (uint32_t)prims->num_prims;
    const uint32_t V0 = (uint32_t)num_voxels0;
    const int64_t P = prims->num_ctrl, F = prims->num_fibers;
    GridDev g;
    g.o[0] = grid->origin[0]; g.o[1] = grid->origin[1]; g.o[2] = grid->origin[2];
    g.s = 1.0f / grid->voxel_size;
    g.R = (int)R;
    float4* r0 = (float4*)(base + NA_RA);
    float4* r1 = (float4*)(base + NA_RB);
    uint32_t* cnt = (uint32_t*)(base + NA_CNT);
    uint32_t* fs = (uint32_t*)(base + NA_FS);
    uint32_t* misc = (uint32_t*)(base + NA_MISC);
    double* seg_grad = (double*)(base + NA_SEG);
    double* gm = (double*)(base + NA_GM);
    double* gM = (double*)(base + NA_GMM);
    uint32_t* part = (uint32_t*)(base + NA_PART);

    // the array keeps the previous call's contents: clear the counters and error flag
    NA_TRY(cudaMemsetAsync(misc, 0, 64, s));
    if (np == 0) {
        if (P) NA_TRY(cudaMemsetAsync(grad_ctrl, 0, (size_t)P * 16, s));
        return VX_OK;
    }

    // level-0 adjoints (coarse adjoints broadcast down)
    if (V0) NA_TRY(adj_broadcast(keys0, V0, num_levels, grad_mass, grad_moment, (uint32_t*)(base + NA_ADJ), gm, gM, s));
    // candidate pairs (counted for the limit)
    k_fiber_seg_counts<<<grid_for((size_t)F, 256), 256, 0, s>>>(prims->fiber_offsets, F, prims->num_ctrl, fs, misc);
    NA_TRY(vx_scan_u32_scratch(fs, fs, (uint32_t)F, misc + 4, part, s));
    k_prep_fibers<<<grid_for(np, 256), 256, 0, s>>>((const float4*)prims->ctrl, prims->num_ctrl, prims->fiber_offsets, fs, F, misc + 4,
                                                     prims->weights, np, g, r0, r1, misc);
    const int clg = count_lanes_log2(np);
    uint32_t host[16] = {0};
    uint64_t npairs64 = 0;
    // (ranges too large for the grouped launch are counted by a second one)
    for (int turn = 0; turn < 2; ++turn) {
        k_count<true><<<count_blocks(np, turn ? 0 : clg), COUNT_WARPS * 32, 0, s>>>(
            r0, r1, nullptr, np, full_window((int)R), turn ? 0 : clg, turn ? kGroupRange + 1 : 0,
            turn || clg == 0 ? kAnyRange : kGroupRange, cnt, nullptr, 0u, misc + 14);
        // the exact 64-bit total, and whether a walk is long
        NA_TRY(cudaMemsetAsync(misc + 8, 0, 8, s));
        k_range_bound<true><<<(unsigned)std::min<size_t>(grid_for(np, 256), (size_t)vx::kSMs * 8), 256, 0, s>>>(
            r0, r1, nullptr, np, full_window((int)R), cnt, (unsigned long long*)(misc + 8), misc + 15);
        NA_TRY(cudaMemcpyAsync(host, misc, 64, cudaMemcpyDeviceToHost, s));
        NA_TRY(cudaStreamSynchronize(s));
        if (host[0]) return VX_ERR_INVALID_ARG;
        memcpy(&npairs64, host + 8, 8);
        if (!(host[14] & kCountLarge)) break;
    }
    if (npairs64 > NA_MAX_PAIRS) return VX_ERR_CAPACITY;
    // the caller's outputs are written only once every limit has passed
    adjoint_fibers(r0, r1, np, (int)R, host[15] != 0, keys0, V0, gm, gM, seg_grad, grad_weights, s);
    k_adjoint_ctrl<<<grid_for((size_t)P, 256), 256, 0, s>>>(prims->fiber_offsets, F, fs, P, seg_grad, g.s,
                                                             (float4*)grad_ctrl);
    NA_TRY(cudaGetLastError());
    return VX_OK;
}
