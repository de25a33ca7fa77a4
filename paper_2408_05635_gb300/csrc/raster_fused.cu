// raster_fused.cu -- one tracking iteration's compositing in one block per tile: the
// front-to-back walk of Eqs. 2-4 with the fused combined loss (Sec. III-B), then, in the
// same block and from the same registers, the pose-only reverse walk that differentiates
// Eqs. 2-4.
//
// It computes what k_forward<loss> followed by k_backward<pose-only> compute (the same
// footprint code, the same per-warp lists, the same transposed sums; see raster_fwd.cu and
// raster_bwd.cu for the arithmetic), with three differences in how the work is laid out:
//   - each pixel's upstream gradient, final transmittance and last contributor stay in
//     registers between the walks and are not written to the workspace (the pass consumes
//     its gradients itself: a gs_backward after it is refused);
//   - the batch the forward staged last is usually the one the reverse walk starts with
//     (a tile's whole list when it holds at most one batch): it is not staged again, and
//     each warp cuts the list it built for it in the forward instead of building another,
//     and goes on from its forward to its reverse walk without waiting for the other warps;
//   - a tile's reverse walk starts as soon as its own forward ends, so the tiles that end
//     the forward (the longest lists, launched first) overlap the reverse walks of the
//     others instead of leaving SMs idle before a second kernel.
#include "bwd_walk.cuh"
#include "fwd_walk.cuh"
#include "gs_internal.cuh"

namespace gsk {

namespace {

__device__ __forceinline__ float sgnf(float x) { return (float)((x > 0.f) - (x < 0.f)); }

// Stage batch position tid of the tile's sorted list (record r) for both walks.
__device__ __forceinline__ void stage_one(const TrackTileLaunch &L, uint32_t r, float x0, float y0, float4 *sP0,
                                          float4 *sP1, float4 *sC, float4 *sBox, int tid) {
    if (r < rec_slots(L.d)) {
        const Rec rr = L.ws.rec[r];
        const Footprint f = stage_footprint(rr.a, rr.b, x0, y0);
        sP0[tid] = f.p0;
        sP1[tid] = f.p1;
        sC[tid] = make_float4(rr.c.x, rr.c.y, rr.c.z, rr.a.z);
        sBox[tid] = stage_box(rr.b, -f.p0.x, -f.p0.y);
    } else {
        sBox[tid] = make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY);  // empty: never listed
    }
}

}  // namespace

// Four blocks per SM (64 registers a thread): with five (48 registers) the walks spill
// and issue more instructions, and the kernel is slower.
template <int NB, int LW>
__global__ void __launch_bounds__(kTilePix, 4) k_track_tile(TrackTileLaunch L) {
    static_assert(NB % 32 == 0 && NB <= kBatch, "batch depth: a multiple of 32, at most kBatch");
    static_assert(LW >= 3 && (1 << LW) * kPatchH <= kTilePix, "tile width: 8 to 32 pixels");
    griddep_wait();  // the predecessor's results are visible from here on
    griddep_launch_dependents();
    using A = Acc<true>;
    __shared__ float4 sP0[NB], sC[NB], sBox[NB];
    __shared__ float4 sP1[NB];                     // (kuu, lo, -1/(2 kuu), -1/(2 kvv)): the stride of sP0, sC
    __shared__ __align__(16) uint16_t sList[kTilePix / 32][NB];  // byte offsets: 16 x batch position
    __shared__ float sAcc[NB * A::kStride];
    __shared__ __align__(16) float sRows[kTilePix / 32][kWalkFloats<true>];  // the reverse walk's transposed rows
    __shared__ float s_loss[kTilePix / 32];
    __shared__ uint32_t s_last[kTilePix / 32];
    __shared__ uint2 s_fwd[kTilePix / 32], s_rev[kTilePix / 32];
    const uint32_t tile = L.ws.tile_order[blockIdx.x];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const ViewInfo vi = L.ws.views[view_of_tile(L.ws.views, L.d.V, tile)];
    const uint32_t local = tile - vi.tile_base;
    const int tx = (int)(local % (uint32_t)vi.tiles_x), ty = (int)(local / (uint32_t)vi.tiles_x);
    constexpr int kPPR = (1 << LW) / kPatchW;  // 8 x 4 patches per patch row (tile width 2^LW)
    const int pu0 = (warp % kPPR) * kPatchW, pv0 = (warp / kPPR) * kPatchH;
    const int lu = pu0 + (lane & (kPatchW - 1)), lv = pv0 + lane / kPatchW;
    const int px = (tx << LW) + lu, py = (ty << vi.tile_lh) + lv;
    const bool inside = px < vi.width && py < vi.height;
    const float x0 = (float)(tx << LW), y0 = (float)(ty << vi.tile_lh);
    const float2 uv = make_float2((float)lu, (float)lv);  // tile-local pixel centre
    const float pu_lo = (float)pu0, pu_hi = (float)(pu0 + kPatchW - 1);
    const float pv_lo = (float)pv0, pv_hi = (float)(pv0 + kPatchH - 1);
    const Settings &S = L.s;
    const float thr = S.log2_alpha_min;

    uint32_t start;
    const uint32_t n = tile_entries(L.ws, L.d, tile, start);

    // this pixel's targets: loaded once the first batch is staged (below), so their
    // latency (host memory when the frame is read in place) passes during the forward walk
    // (loaded at the start of the block instead, in-place reads made the kernel slower)
    const uint32_t HW = (uint32_t)vi.width * (uint32_t)vi.height;
    const uint32_t p = inside ? (uint32_t)py * (uint32_t)vi.width + (uint32_t)px : 0u;
    const uint32_t gp = vi.pix_base + p;
    float tr = 0.f, tg = 0.f, tb = 0.f, Dt = 0.f, pr = 0.f;
    bool targets_loaded = false;

    // ---------------------------------------------------------------- forward (Eqs. 2-4)
    FwdPixel walk{1.f, 0.f, 0.f, 0.f, 0.f, 0u, 0u, !inside};
    uint32_t n_eval = 0, n_contrib = 0;
    int64_t staged = -1;  // first list entry of the batch now in shared memory (block-uniform)
    int nl_staged = 0;    // length of this warp's list of the staged batch (warp-uniform)
    for (uint32_t b0 = 0; b0 < n; b0 += NB) {
        if (b0 && __syncthreads_count(!walk.done) == 0) break;  // (and all have walked the staged batch)
        const uint32_t idx = b0 + tid;
        if (tid < NB && idx < n) stage_one(L, L.ws.sorted[start + idx], x0, y0, sP0, sP1, sC, sBox, tid);
        staged = b0;
        if (b0 == 0 && tid < NB) {  // the reverse walk's sums (thread tid owns the row of batch position tid)
#pragma unroll
            for (int k = 0; k < A::kValues; ++k) sAcc[tid * A::kStride + k] = 0.f;
        }
        __syncthreads();
        if (!targets_loaded) {
            targets_loaded = true;
            if (inside) {
                const float *trgb = L.t_rgb + 3u * vi.pix_base;
                tr = trgb[p];
                tg = trgb[HW + p];
                tb = trgb[2u * HW + p];
                Dt = L.t_depth[gp];
                if (L.t_prior) pr = L.t_prior[gp];
            }
        }
        const int cnt = (int)min((uint32_t)NB, n - b0);
        if (__any_sync(0xffffffffu, !walk.done)) {
            // (its hits kept where the reverse walk will stage the batch again)
            const int nl = build_patch_list(sBox, sP0, sP1, sList[warp], cnt, lane, thr, pu_lo, pu_hi, pv_lo, pv_hi,
                                            [&](uint32_t hits) {
                                                if (n > (uint32_t)NB) hit_words(L.ws, tile, start, n, warp)[(b0 >> 5) + lane] = hits;
                                            });
            nl_staged = nl;
            if (!walk.done)
                fwd_walk_batch(walk, sList[warp], nl, b0, sP0, sP1, sC, uv, thr, S.alpha_max, S.t_min, n_eval,
                               n_contrib);
        }
    }
    float T = walk.T;
    const float cr = walk.cr, cg = walk.cg, cb = walk.cb, D = walk.D;
    uint32_t last = walk.last;
    const float Sil = 1.f - T;  // Eq. 4 summed: 1 - prod(1 - a_i)
    count_warp(n_eval, n_contrib, s_fwd);

    // ---------------------------------------------------------------- fused loss
    if (!targets_loaded && inside) {  // an empty tile list: no batch was staged
        const float *trgb = L.t_rgb + 3u * vi.pix_base;
        tr = trgb[p];
        tg = trgb[HW + p];
        tb = trgb[2u * HW + p];
        Dt = L.t_depth[gp];
        if (L.t_prior) pr = L.t_prior[gp];
    }
    float g0 = 0.f, g1 = 0.f, g2 = 0.f, gD = 0.f, gS = 0.f, l = 0.f;
    if (inside) {
        const bool valid = Dt > 0.f;
        const bool M = valid && Sil > S.sil_thresh;
        if (M) {
            const float r0 = cr - tr, r1 = cg - tg, r2 = cb - tb;
            l += S.w_rgb * (fabsf(r0) + fabsf(r1) + fabsf(r2));
            g0 = S.w_rgb * sgnf(r0);
            g1 = S.w_rgb * sgnf(r1);
            g2 = S.w_rgb * sgnf(r2);
            const float rd = D - Dt;
            l += S.w_depth * fabsf(rd);
            gD = S.w_depth * sgnf(rd);
            if (L.t_prior) {
                if (pr > 0.f) {
                    const float rp = D - pr;
                    l += S.w_prior * fabsf(rp);
                    gD += S.w_prior * sgnf(rp);
                }
            }
        }
        if (valid) {
            l += S.w_vis * (1.f - Sil);
            gS = -S.w_vis;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    if (lane == 0) s_loss[warp] = l;

    // ---------------------------------------------------------------- reverse walk (pose)
    if (!(g0 != 0.f || g1 != 0.f || g2 != 0.f || gD != 0.f || gS != 0.f)) last = 0;
    // the reverse walk evaluates this pixel's entries in front of its last contributor and
    // differentiates its contributions: the forward's counts up to that entry
    const uint32_t rev_eval = last ? walk.eval_last : 0u, rev_contrib = last ? n_contrib : 0u;
    count_warp(rev_eval, rev_contrib, s_rev);
    const uint32_t wlast = __reduce_max_sync(0xffffffffu, last);  // largest contributor count in the warp
    if (lane == 0) s_last[warp] = wlast;
    const PixUp up{g0, g1, g2, gD, gS};
    float *buf = sRows[warp];
    store_planes<true>(buf, up, lane);
    float GB = 0.f;  // g . (colour, depth, 1) of everything behind, back-to-front
    // From the batch the forward staged last down to the first.  The staged one needs no
    // barrier: each warp goes on from its forward to its reverse walk by itself, so the
    // warps of a tile wait for one another once (before the flush) instead of after each walk.
    for (int64_t b0 = staged; b0 >= 0; b0 -= NB) {
        const bool resident = b0 == staged;
        const uint32_t filled = min((uint32_t)NB, n - (uint32_t)b0);
        uint32_t words = 0;
        if (!resident) {
            // this warp's hits (it kept them for every batch its pixels reached)
            if (lane < NB / 32 && b0 < (int64_t)wlast) words = hit_words(L.ws, tile, start, n, warp)[(b0 >> 5) + lane];
            // (thread tid flushed the row it clears here, and the others walk no more)
            if (tid < filled) stage_one(L, L.ws.sorted[start + (uint32_t)b0 + tid], x0, y0, sP0, sP1, sC, sBox, tid);
            if (tid < NB) {
#pragma unroll
                for (int k = 0; k < A::kValues; ++k) sAcc[tid * A::kStride + k] = 0.f;
            }
            __syncthreads();
        }
        // this warp's list, limited to entries below its largest contributor count
        const int wcnt = (int)max(min((int64_t)filled, (int64_t)wlast - b0), (int64_t)0);
        int nl = 0;
        if (resident) {
            // the list this warp built for the batch in the forward is still in sList, and
            // its entries below wcnt are the list build_patch_list would give for wcnt.  A
            // warp whose pixels had all stopped before this batch kept an older list, but
            // then wlast <= b0 and no entry is below wcnt = 0.
            for (int k = 0; k < nl_staged; k += 32) {
                const bool below = k + lane < nl_staged && (int)sList[warp][k + lane] < wcnt * 16;
                const int m = __popc(__ballot_sync(0xffffffffu, below));
                nl += m;
                if (m < 32) break;
            }
        } else {
            nl = list_from_words(words, sList[warp], wcnt, lane);
        }
        __syncwarp();
        // entries at byte offsets below lim are in front of this pixel's last contributor
        const int lim = (int)max(min((int64_t)last - b0, (int64_t)NB), (int64_t)0) * 16;
        uint32_t unused = 0;
        bwd_walk_batch<true, false>(sList[warp], nl, lim, sP0, sP1, sC, uv, pu_lo, pv_lo, thr, S.alpha_max, up, T, GB,
                                    buf, sAcc, lane, unused, unused);
        __syncthreads();
        uint32_t nmax = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) nmax = max(nmax, s_last[w]);
        if (nmax > (uint32_t)b0 && tid < min(filled, nmax - (uint32_t)b0)) {
            const uint32_t r = L.ws.sorted[start + (uint32_t)b0 + tid];
            if (r < rec_slots(L.d)) flush_acc<true>(sAcc + tid * A::kStride, L.ws.rec[r].b, 1.f, L.ws.rec_grad + r);
        }
    }
    if (staged < 0) __syncthreads();  // an empty list: the barrier before the flush did not run
    if (tid == 0) {
        DF s{0.f, 0.f};
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s = df_add(s, DF{s_loss[w], 0.f});
        L.ws.tile_loss[tile] = df_pack(s);
        count_block(s_fwd, &L.ws.hdr->fwd_evals, &L.ws.hdr->fwd_contrib);
        count_block(s_rev, &L.ws.hdr->bwd_evals, &L.ws.hdr->bwd_contrib);
    }
}

template <int NB, int LW>
cudaError_t launch_track_tile_nb(const TrackTileLaunch &L, cudaStream_t st) {
    return launch_dep(k_track_tile<NB, LW>, dim3(L.d.T), dim3(tile_threads(L.d)), st, L);
}

template <int NB>
cudaError_t launch_track_tile_lw(const TrackTileLaunch &L, cudaStream_t st) {
    switch (tile_lw(L.d)) {
        case 3: return launch_track_tile_nb<NB, 3>(L, st);
        case 4: return launch_track_tile_nb<NB, 4>(L, st);
        case 5: return launch_track_tile_nb<NB, 5>(L, st);
        default: return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}

cudaError_t launch_track_tile(const TrackTileLaunch &L, cudaStream_t st) {
    if (L.d.T == 0) return cudaSuccess;
    if (!L.t_rgb || !L.t_depth) return cudaErrorInvalidValue;
    // one batch depth for both walks; a batch stages at most one Gaussian per thread
    const uint32_t nb = L.d.fwd_batch ? L.d.fwd_batch : (uint32_t)kBatch;
    if (nb > tile_threads(L.d) || (L.d.bwd_batch ? L.d.bwd_batch : (uint32_t)kBatch) != nb)
        return cudaErrorInvalidValue;
    cudaError_t e;
    switch (nb) {
        case 256: e = launch_track_tile_lw<256>(L, st); break;
        case 128: e = launch_track_tile_lw<128>(L, st); break;
        case 64: e = launch_track_tile_lw<64>(L, st); break;
        default: return cudaErrorInvalidValue;
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace gsk
