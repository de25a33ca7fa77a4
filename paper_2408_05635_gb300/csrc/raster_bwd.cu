// raster_bwd.cu -- reverse compositing: per-record screen-space gradients.
//
// Differentiating Eqs. 2-4 for one pixel with upstream g = dL/d(C_r, C_g, C_b, D, S):
// walking the contributors back to front with B_ch the colour of everything behind
// Gaussian i (B <- B + a_i (v_i - B), starting from the zero background) and T_i the
// transmittance in front of it (recovered from the stored final transmittance as
// T_i = T_{i+1} / (1 - a_i)); a_i is re-evaluated with the forward's footprint code,
// bit for bit, so both walks skip exactly the same Gaussians,
//   dL/da_i = T_i sum_ch g_ch (v_ch,i - B_ch),   v = (r, g, b, depth, 1),
//   dL/dc_i = a_i T_i g_C,  dL/dd_i = a_i T_i g_D,
// and through a_i = o G, G = exp(power): dL/do = dL/da G, dL/dpower = dL/da a
// (both zero where a_i is clamped at alpha_max), dpower/dmu' = conic (p - mu'),
// dpower/d(conic a, b, c) = (-dx^2 / 2, -dx dy, -dy^2 / 2).
// Only the scalar g . B enters dL/da, so the walk carries that scalar instead of B:
// g.B <- g.B + a_i (g.v_i - g.B).  The conic is constant per Gaussian, so the pixel sums
// are taken of the moments dp (dx, dy, dx^2, dx dy, dy^2), dp = dL/dpower, and the conic is
// applied once per (tile, Gaussian) when the sums are flushed.
//
// Batches of NB records (64, 128 or 256, the batch depth, picked per context) are staged
// by the first NB threads, from the tile's last contributor backwards.  Each warp owns an
// 8 x 4 patch of the tile and walks, back to front, only the staged Gaussians whose
// footprint can reach alpha_min on the patch (the hits the forward kept) and that precede its
// last contributor.
// Reduction: each warp sums its 32 pixels' terms of eight Gaussians at a time through a
// small shared matrix read transposed (bwd_walk.cuh), adds the sums into a per-batch
// shared-memory accumulator, and the block flushes once per (tile, Gaussian) with vector
// float4 atomics into the record's global accumulator.
// A quarter of a warp's time went to barriers and to the chain of dependent loads at a
// block's start; the view is found by each warp, a one-batch list is staged beside the
// pixels' loads, and a thread owns its batch position up to the flush (two barriers a batch
// instead of three): 1,204 -> 1,139 us on the mapping window, 411 -> 387 on the dense one.
// The lists come from the forward's hit words (8 words a warp and batch instead of 256 tests):
// 1,139 -> 1,083 and 387 -> 358 us, the forward 739 -> 747 (it keeps them for every render,
// since a reverse walk may follow: 113 -> 115 us on 1M at 1200 x 680).
// Lanes whose pixel the Gaussian does not reach take a = 0, which leaves T and g.B
// unchanged and zeroes every term, so the walk has no divergent branch.
#include "gs_internal.cuh"
#include "bwd_walk.cuh"

namespace gsk {

// Four blocks per SM (64 registers a thread: the walk's unrolled steps spill at 48).
// Dynamic shared memory: kWalkFloats per warp.
template <bool POSE, int NB, int LW>
__global__ void __launch_bounds__(kTilePix, 4) k_backward(BackwardLaunch L) {
    static_assert(NB % 32 == 0 && NB <= kBatch, "batch depth: a multiple of 32, at most kBatch");
    static_assert(LW >= 3 && (1 << LW) * kPatchH <= kTilePix, "tile width: 8 to 32 pixels");
    griddep_wait();  // the predecessor's results are visible from here on
    griddep_launch_dependents();
    using A = Acc<POSE>;
    extern __shared__ __align__(16) float sDyn[];
    __shared__ float4 sP0[NB], sC[NB];
    __shared__ float4 sP1[NB];  // (kuu, lo, -, -): the stride of sP0, sC
    __shared__ float sAcc[NB * A::kStride];
    __shared__ __align__(16) uint16_t sList[kTilePix / 32][NB];  // byte offsets: 16 x batch position
    __shared__ uint32_t s_last[kTilePix / 32];
    __shared__ uint2 s_count[kTilePix / 32];
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
    const float pu_lo = (float)pu0, pv_lo = (float)pv0;
    const Settings &S = L.s;
    const float thr = S.log2_alpha_min;
    float *buf = sDyn + warp * kWalkFloats<POSE>;

    uint32_t start;
    const uint32_t n = tile_entries(L.ws, L.d, tile, start);
    // Stages list entry first + tid and clears its sums; returns its record (or ~0u).  Thread
    // tid owns batch position tid from here to the flush of its sums, so neither the flush
    // nor the next batch's staging after it needs a barrier of its own.
    const auto stage = [&](uint32_t first, int cnt) {
        uint32_t r = ~0u;
        if (tid < cnt) {
            r = L.ws.sorted[start + first + tid];
            if (r < rec_slots(L.d)) {
                const Rec rr = L.ws.rec[r];
                const Footprint f = stage_footprint(rr.a, rr.b, x0, y0);
                sP0[tid] = f.p0;
                sP1[tid] = make_float4(f.p1.x, f.p1.y, 0.f, 0.f);
                sC[tid] = make_float4(rr.c.x, rr.c.y, rr.c.z, rr.a.z);
            } else {
                r = ~0u;  // none: the forward kept no hit of it
            }
        }
        if (tid < NB) {
#pragma unroll
            for (int k = 0; k < A::kValues; ++k) sAcc[tid * A::kStride + k] = 0.f;
        }
        return r;
    };
    // a list of one batch is staged before the pixels' last contributors are known, its
    // loads beside theirs
    const bool single = n <= (uint32_t)NB;
    const auto load_words = [&](uint32_t first) {  // this warp's hits of the batch, a word per lane
        return lane < NB / 32 && first + 32u * lane < n ? hit_words(L.ws, tile, start, n, warp)[(first >> 5) + lane] : 0u;
    };
    uint32_t hits = single ? load_words(0u) : 0u;
    uint32_t rec = single ? stage(0u, (int)n) : ~0u;
    const uint32_t HW = (uint32_t)vi.width * (uint32_t)vi.height;
    const uint32_t p = (uint32_t)py * (uint32_t)vi.width + (uint32_t)px;
    const uint32_t gp = vi.pix_base + p;
    float T = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f, gD = 0.f, gS = 0.f;
    uint32_t last = 0;
    if (inside) {
        const float *ur = L.up_rgb + 3u * vi.pix_base;
        const uint32_t nl = L.ws.n_last[gp];
        const float tf = L.ws.t_final[gp];
        g0 = ur[p];
        g1 = ur[HW + p];
        g2 = ur[2u * HW + p];
        gD = L.up_depth[gp];
        gS = L.up_sil[gp];
        if (g0 != 0.f || g1 != 0.f || g2 != 0.f || gD != 0.f || gS != 0.f) {
            last = min(nl, n);
            T = tf;
        }
    }
    const uint32_t wlast = __reduce_max_sync(0xffffffffu, last);  // largest contributor count in the warp
    if (lane == 0) s_last[warp] = wlast;
    const PixUp up{g0, g1, g2, gD, gS};
    store_planes<POSE>(buf, up, lane);
    __syncthreads();
    uint32_t nmax = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) nmax = max(nmax, s_last[w]);
    float GB = 0.f;  // g . (colour, depth, 1) of everything behind, back-to-front
    uint32_t n_eval = 0, n_contrib = 0;

    for (int64_t b0 = nmax ? (int64_t)((nmax - 1) / NB) * NB : -1; b0 >= 0; b0 -= NB) {
        const int cnt = (int)min((uint32_t)NB, nmax - (uint32_t)b0);
        if (!single) {
            hits = load_words((uint32_t)b0);
            rec = stage((uint32_t)b0, cnt);
            __syncthreads();
        }
        // this warp's list, limited to entries below its largest contributor count
        const int wcnt = (int)min((int64_t)cnt, (int64_t)wlast - b0);
        const int nl = list_from_words(hits, sList[warp], wcnt, lane);
        // entries at byte offsets below lim are in front of this pixel's last contributor
        const int lim = (int)max(min((int64_t)last - b0, (int64_t)NB), (int64_t)0) * 16;
        // (asked again for every batch: the answer kept in a register cost spills.  A pose gradient is
        // the sum over all Gaussians: not finite either way)
        if (!POSE && odd_planes(up)) {
            const WalkState w = bwd_walk_odd<POSE>(sList[warp], nl, lim, sP0, sP1, sC, uv, pu_lo, pv_lo, thr, S.alpha_max, up,
                                                   WalkState{T, GB, n_eval, n_contrib}, buf, sAcc, lane);
            T = w.T;
            GB = w.GB;
            n_eval = w.n_eval;
            n_contrib = w.n_contrib;
        } else {
            bwd_walk_batch<POSE, true>(sList[warp], nl, lim, sP0, sP1, sC, uv, pu_lo, pv_lo, thr, S.alpha_max, up, T, GB,
                                       buf, sAcc, lane, n_eval, n_contrib);
        }
        __syncthreads();
        if (tid < cnt && rec != ~0u) {
            const float4 Q = L.ws.rec[rec].b;  // conic
            flush_acc<POSE>(sAcc + tid * A::kStride, Q, POSE ? 1.f : L.ws.rec[rec].a.w, L.ws.rec_grad + rec);
        }
    }
    count_warp(n_eval, n_contrib, s_count);
    __syncthreads();
    if (tid == 0) {
        count_block(s_count, &L.ws.hdr->bwd_evals, &L.ws.hdr->bwd_contrib);
    }
}

// One block per tile, warp_floats floats of dynamic shared memory per warp.
cudaError_t launch_tiles(void (*kernel)(BackwardLaunch), const BackwardLaunch &L, int warp_floats, cudaStream_t st) {
    const uint32_t threads = tile_threads(L.d);
    const size_t smem = (size_t)(threads / 32) * (size_t)warp_floats * sizeof(float);
    // static and dynamic shared memory together may pass the 48 KB a kernel gets unasked
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return e != cudaSuccess ? e : launch_dep_smem(kernel, dim3(L.d.T), dim3(threads), smem, st, L);
}

template <int NB, int LW>
cudaError_t launch_backward_nb(const BackwardLaunch &L, cudaStream_t st) {
    if (L.pose_only)
        return launch_tiles(k_backward<true, NB, LW>, L, kWalkFloats<true>, st);
    else
        return launch_tiles(k_backward<false, NB, LW>, L, kWalkFloats<false>, st);
}

template <int NB>
cudaError_t launch_backward_lw(const BackwardLaunch &L, cudaStream_t st) {
    switch (tile_lw(L.d)) {
        case 3: return launch_backward_nb<NB, 3>(L, st);
        case 4: return launch_backward_nb<NB, 4>(L, st);
        case 5: return launch_backward_nb<NB, 5>(L, st);
        default: return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}

cudaError_t launch_backward(const BackwardLaunch &L, cudaStream_t st) {
    if (L.d.T == 0) return cudaSuccess;
    // a batch stages at most one Gaussian per thread of the tile block
    const uint32_t nb = L.d.bwd_batch ? L.d.bwd_batch : (uint32_t)kBatch;
    if (nb > tile_threads(L.d)) return cudaErrorInvalidValue;
    cudaError_t e;
    switch (L.d.bwd_batch) {
        case 0:
        case 256: e = launch_backward_lw<256>(L, st); break;
        case 128: e = launch_backward_lw<128>(L, st); break;
        case 64: e = launch_backward_lw<64>(L, st); break;
        default: return cudaErrorInvalidValue;
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace gsk
