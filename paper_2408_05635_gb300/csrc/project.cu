// project.cu -- projection of every (Gaussian, view) pair, tile counting and key emission.
//
// k_project follows the projection of the paper: camera-frame mean R x + t (Sec. II-A),
// Sigma = Rg diag(s^2) Rg^T and Sigma' = J W Sigma W^T J^T (covariance formulas written
// in the source of Sec. I), mu' = pi_m(x_c) (Sec. II-A) and the 2-D footprint of Eq. 1.
// The support of a Gaussian is opacity-aware: o exp(-d^2/2) >= alpha_min holds exactly
// for Mahalanobis d^2 <= 2 ln(o / alpha_min), so tiles outside that ellipse can be
// skipped without changing a single pixel.
#include "gs_internal.cuh"

namespace gsk {

// Tile rectangle of a record's support ellipse.  The pixel box is derived from the
// stored conic (Sigma'_xx = c / det, Sigma'_yy = a / det of the conic); the one-pixel
// margin of tile_rect absorbs the error of the fast reciprocal and square root.  Both
// k_project (counting) and k_emit (writing) call exactly this code on the same floats,
// so they enumerate the same tiles.  Returns false when the box misses the image.
__device__ __forceinline__ bool record_rect(const ViewInfo &vi, float4 A, float4 B, int &tx0, int &tx1, int &ty0,
                                            int &ty1) {
    const float detc = diff_of_products(B.x, B.z, B.y, B.y);
    if (!(detc > 0.f)) return false;
    float hx = INFINITY, hy = INFINITY;
    if (B.w < INFINITY) {
        const float idet = __fdividef(1.f, detc);
        const float qx = __fmul_rn(B.w, __fmul_rn(B.z, idet)), qy = __fmul_rn(B.w, __fmul_rn(B.x, idet));
        hx = qx > 0.f ? __fmul_rn(qx, rsqrtf(qx)) : 0.f;
        hy = qy > 0.f ? __fmul_rn(qy, rsqrtf(qy)) : 0.f;
    }
    tile_rect(vi, A.x, A.y, hx, hy, tx0, tx1, ty0, ty1);
    return tx0 <= tx1 && ty0 <= ty1;
}

// The tiles of a block's records (k_project counts them, k_emit writes a key into each).
// Work is handed out by tile rows: the rows of all the block's rectangles are numbered
// through, each thread takes every kBlock-th and walks the row's span of tiles, so a
// Gaussian close to the camera, whose rectangle spans thousands of tiles, and a warp of
// uneven ones are spread over the block.  The tiles are gathered in shared counters over the
// block's own tile box first (neighbouring Gaussians share their tiles: a map along a
// Morton curve or built frame by frame), which leaves one global atomic per tile and block
// instead of one per (record, tile) pair.  Both kernels run this code on the same floats, so
// they enumerate the same tiles.
//
// Before, a lane walked its own record and a warp or extra blocks the large ones, with an
// atomic per pair: what bound both kernels was the atomics' rate and round trips.  8 views
// of 1M Gaussians (29 pairs a record): k_project 185 -> 113 us, k_emit 161 -> 74; one view
// of 1M at 1200 x 680 (10 pairs): 48 -> 29 and 64 -> 38; 2M in FP16 (4.6): 80 -> 63 and 87
// -> 40 (k_emit's times hold its wait for the scan).  Unchanged within a microsecond where
// latency counts (200k, 37k records); footprints a pixel wide (1.8 pairs a record) 57 -> 61 and 61 -> 55 us.
//
// The box pays where records share its tiles.  Where the tiles are many more than the records
// could meet, zeroing and reading them back costs more than an atomic a pair: 1M pixel-sized
// Gaussians in random order at 1200 x 680 (a block's box is the image) took 143 us a projection
// with it, 108 without; of six pixels (6 tiles a rectangle, so 2.1 box tiles a tile) 63 against 78.
// Without it a record's rows are walked as they are, or, where rows are wide, by four or eight
// threads each, whose atomics fall on neighbouring counters: 200k Gaussians of 40 pixels in
// random order at 1920 x 1080 took 1,376 us with a thread a row, 905 with eight (982 with a
// warp a record); of ten pixels 172 and 150 with four.
constexpr int kSoloRows = 4;     // records of no more rows: handing their rows out costs more than walking them
                                 // (1.8 pairs a record: a window of 864 us took 887)
constexpr int kBoxPerTile = 3;   // most tiles of a box per tile of its records' rectangles
// Most tiles of a box, by the shared memory of six blocks an SM; k_emit's is smaller because its
// scattered loads and stores want the L1 that is left (1M two-pixel Gaussians in random order:
// 53 us, and 65 with 4,864; k_project's 58 with either, and 200k of 40 pixels over 4,800 tiles
// 205 -> 52).
constexpr int kProjectBox = 5632;
constexpr int kEmitBox = 3328;

struct RowRec {  // one record's rows
    float4 a;    // mu'_x, mu'_y, b, det
    float4 b;    // aR, Y, X, t
    float ia;
    int tx0, tx1, ty0;
};

struct BinRows {
    RowRec rec[kBlock];
    uint32_t pre[kBlock + 1];  // rows before each record
    int4 warp_box[kWarps];     // first tile column and row, last column and row
    uint4 warp_rows[kWarps];   // rows, the most of one record, tiles of the rectangles
};

template <int TILES>
struct BinSmem : BinRows {
    uint32_t box[TILES];
};

// Posts the warp's rows and tile box (block_box reads them after a barrier).
__device__ __forceinline__ void post_rows(BinRows &sm, bool has, int tx0, int tx1, int ty0, int ty1) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t rows = has ? (uint32_t)(ty1 - ty0 + 1) : 0u;
    const uint32_t sum = __reduce_add_sync(0xffffffffu, rows);
    const int lx = __reduce_min_sync(0xffffffffu, has ? tx0 : 0x7fffffff), hx = __reduce_max_sync(0xffffffffu, has ? tx1 : -1);
    const int ly = __reduce_min_sync(0xffffffffu, has ? ty0 : 0x7fffffff), hy = __reduce_max_sync(0xffffffffu, has ? ty1 : -1);
    const uint32_t most = __reduce_max_sync(0xffffffffu, rows);
    const uint32_t tiles = __reduce_add_sync(0xffffffffu, has ? rows * (uint32_t)(tx1 - tx0 + 1) : 0u);
    if (lane == 31) {
        sm.warp_box[warp] = make_int4(lx, ly, hx, hy);
        sm.warp_rows[warp] = make_uint4(sum, most, tiles, 0u);
    }
}

// Rows of the warp's lanes before this one.
__device__ __forceinline__ uint32_t rows_before(bool has, int ty0, int ty1) {
    const int lane = threadIdx.x & 31;
    const uint32_t rows = has ? (uint32_t)(ty1 - ty0 + 1) : 0u;
    uint32_t incl = rows;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    return incl - rows;
}

struct BlockBox {
    int x, y, w, area;      // first tile, columns, tiles (0: gathered in global memory)
    bool boxed, solo;
    uint32_t before, rows;  // rows of the warps before this one, of the block
    uint32_t lanes;         // threads that share a row (1, 4 or 8)
};

__device__ __forceinline__ BlockBox block_box(const BinRows &sm, int most_tiles) {
    const int warp = threadIdx.x >> 5;
    int4 q = sm.warp_box[0];
    uint4 r = sm.warp_rows[0];
    BlockBox o;
    o.before = warp > 0 ? r.x : 0u;
#pragma unroll
    for (int w = 1; w < kWarps; ++w) {
        const int4 p = sm.warp_box[w];
        const uint4 c = sm.warp_rows[w];
        q = make_int4(min(q.x, p.x), min(q.y, p.y), max(q.z, p.z), max(q.w, p.w));
        o.before += w < warp ? c.x : 0u;
        r = make_uint4(r.x + c.x, max(r.y, c.y), r.z + c.z, 0u);
    }
    o.rows = r.x;
    o.x = q.x;
    o.y = q.y;
    o.w = q.z - q.x + 1;
    const int64_t area = (int64_t)o.w * (q.w - q.y + 1);
    o.boxed = r.x > 0u && area <= min((int64_t)most_tiles, (int64_t)kBoxPerTile * r.z);
    o.area = o.boxed ? (int)area : 0;
    // rows of three tiles on average by four threads, of twelve by eight: 200k Gaussians of ten
    // pixels at 1280 x 720 (rows of 3) 412 -> 338 us with four, of 40 at 3840 x 2160 (28) 4,573
    // with four and 3,225 with eight
    o.lanes = o.boxed || r.z < 3u * r.x ? 1u : (r.z < 12u * r.x ? 4u : 8u);
    o.solo = r.y <= (uint32_t)kSoloRows && o.lanes == 1u;
    return o;
}

__device__ __forceinline__ void put_rows(RowRec &r, float4 A, float4 B, int tx0, int tx1, int ty0) {
    const RowSpan s = row_span_setup(A.x, A.y, B.x, B.y, B.z, B.w);
    r.a = make_float4(s.mx, s.my, s.b, s.det);
    r.b = make_float4(s.aR, s.Y, s.X, s.t);
    r.ia = s.ia;
    r.tx0 = tx0;
    r.tx1 = tx1;
    r.ty0 = ty0;
}

// body(tile row, first tile column, last) for the rows of this thread's own record.
template <class Body>
__device__ __forceinline__ void for_own_rows(const ViewInfo &vi, float4 A, float4 B, int tx0, int tx1, int ty0, int ty1,
                                             Body &&body) {
    const RowSpan s = row_span_setup(A.x, A.y, B.x, B.y, B.z, B.w);
    for (int ty = ty0; ty <= ty1; ++ty) {
        int a0, a1;
        row_span(vi, s, ty, tx0, tx1, a0, a1);
        if (a0 <= a1) body(ty, a0, a1);
    }
}

// body(record, tile row, first tile column, last) for this thread's share of the rows of
// nrec > 0 records, each row taken by `lanes` neighbouring threads.
template <class Body>
__device__ __forceinline__ void for_rows(const BinRows &sm, int nrec, const ViewInfo &vi, uint32_t lanes, Body &&body) {
    const uint32_t rows = sm.pre[nrec];
    for (uint32_t f = threadIdx.x / lanes; f < rows; f += kBlock / lanes) {
        int lo = 0, hi = nrec - 1;  // the last record whose prefix is at most f
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (sm.pre[mid] <= f) lo = mid; else hi = mid - 1;
        }
        const RowRec &r = sm.rec[lo];
        const int ty = r.ty0 + (int)(f - sm.pre[lo]);
        const float4 ra = r.a, rb = r.b;
        const RowSpan s{ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w, r.ia};
        int a0, a1;
        row_span(vi, s, ty, r.tx0, r.tx1, a0, a1);
        if (a0 <= a1) body(lo, ty, a0, a1);
    }
}

struct ViewChunk {
    ViewInfo v[32];
};

// Copies up to 32 views into the device table (block 0) and zeroes `zero_words` 32-bit
// words at `zero` (all blocks, grid-stride): the per-call reset of the flag word, the
// header and the tile counters, folded into the same launch.
__global__ void k_copy_views(ViewInfo *dst, int count, ViewChunk chunk, uint32_t *zero, size_t zero_words) {
    // the projection may be scheduled now: it waits (griddep_wait) for this grid to end
    // before it touches the workspace
    griddep_launch_dependents();
    if (blockIdx.x == 0 && threadIdx.x < count) dst[threadIdx.x] = chunk.v[threadIdx.x];
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < zero_words; i += (size_t)gridDim.x * blockDim.x)
        zero[i] = 0u;
}

cudaError_t launch_upload_views(const ViewInfo *host_views, int V, ViewInfo *dev, void *zero, size_t zero_bytes,
                                cudaStream_t st) {
    constexpr int kThreads = 256;
    for (int base = 0; base < V || (base == 0 && zero_bytes); base += 32) {
        ViewChunk c;
        const int cnt = V - base < 32 ? (V - base > 0 ? V - base : 0) : 32;
        for (int k = 0; k < cnt; ++k) c.v[k] = host_views[base + k];
        const size_t words = base == 0 ? zero_bytes / 4 : 0;
        size_t blocks = (words + 4 * kThreads - 1) / (4 * kThreads);
        blocks = blocks < 1 ? 1 : (blocks > 1024 ? 1024 : blocks);
        k_copy_views<<<(unsigned)blocks, kThreads, 0, st>>>(dev + base, cnt, c, static_cast<uint32_t *>(zero), words);
    }
    return cudaGetLastError();
}

// Exclusive scan of the per-(tile, sub-bucket) counts into list offsets, by one block of
// kScanThreads.  Each pass loads kScanPer contiguous counters per thread in one round
// (and zeroes them for the next projection), scans the per-thread totals across the
// block and writes the offsets.  Since S divides kScanPer, a tile's S counters sit in
// one thread, which also counts the tile's list length into the buckets of the
// longest-first launch order; the lengths stay in registers when one pass covers all
// counters.  Also: the total pair count, the longest list and the number of records.
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 8;
constexpr int kOrderBuckets = kScanThreads;  // list lengths >= kOrderBuckets - 1 share the first bucket

__device__ __forceinline__ uint32_t order_bucket(uint32_t len) {
    return kOrderBuckets - 1 - min(len, (uint32_t)kOrderBuckets - 1);
}

// Exclusive block-wide scan of one value per thread; `total` gets the block sum.  Uses
// warp_sum (kScanThreads / 32 words) and ends with a barrier.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t *warp_sum, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    uint32_t wi = lane < kScanThreads / 32 ? warp_sum[lane] : 0u;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, wi, off);
        if (lane >= off) wi += v;
    }
    const uint32_t prev = __shfl_sync(0xffffffffu, wi, (warp + 31) & 31);
    total = __shfl_sync(0xffffffffu, wi, kScanThreads / 32 - 1);
    __syncthreads();
    return (warp > 0 ? prev : 0u) + incl - x;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(WsPtrs ws, Dims d) {
    griddep_wait();  // the predecessor's results are visible from here on
    griddep_launch_dependents();
    __shared__ uint32_t warp_sum[kScanThreads / 32];
    __shared__ uint32_t s_bucket[kOrderBuckets];
    __shared__ uint32_t s_max;
    __shared__ unsigned long long s_recs;
    const uint32_t TS = d.T * d.S, S = d.S, smask = d.S - 1, sshift = __ffs(d.S) - 1;  // S: 1, 2 or 4
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        s_max = 0;
        s_recs = 0;
    }
    s_bucket[tid] = 0;
    // record counts of the first cells, fetched now so their latency overlaps the scan
    const uint32_t ncell = (uint32_t)d.V * (uint32_t)d.nblk;
    uint32_t cc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t c = (uint32_t)tid + (uint32_t)k * kScanThreads;
        cc[k] = c < ncell ? ws.cell_cnt[c] : 0u;
    }
    __syncthreads();
    const bool one_pass = TS <= (uint32_t)kScanThreads * kScanPer;
    uint32_t len[kScanPer];  // length of the tile whose first counter is j (j % S == 0)
    unsigned long long carry = 0;  // identical in every thread
    uint32_t max_tile = 0;
    for (uint32_t base = 0; base < TS; base += (uint32_t)kScanThreads * kScanPer) {
        const uint32_t i0 = base + (uint32_t)tid * kScanPer;
        uint32_t c[kScanPer];
        if (i0 + kScanPer <= TS) {
            uint4 *q = reinterpret_cast<uint4 *>(ws.tile_cnt + i0);
            const uint4 a = q[0], b = q[1];
            c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w;
            c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
            q[0] = make_uint4(0u, 0u, 0u, 0u);
            q[1] = make_uint4(0u, 0u, 0u, 0u);
        } else {
#pragma unroll
            for (int k = 0; k < kScanPer; ++k) {
                c[k] = i0 + k < TS ? ws.tile_cnt[i0 + k] : 0u;
                if (i0 + k < TS) ws.tile_cnt[i0 + k] = 0u;
            }
        }
        uint32_t mine = 0;
#pragma unroll
        for (int k = 0; k < kScanPer; ++k) mine += c[k];
        uint32_t total;
        const uint32_t excl = block_exclusive_scan(mine, warp_sum, total);
        unsigned long long run = carry + excl;
        uint32_t o[kScanPer];
#pragma unroll
        for (int k = 0; k < kScanPer; ++k) {
            o[k] = (uint32_t)min(run, (unsigned long long)0xffffffffu);
            run += c[k];
        }
        if (i0 + kScanPer <= TS) {  // whole 32-byte rows: two vector stores per array
            const uint4 a = make_uint4(o[0], o[1], o[2], o[3]), b = make_uint4(o[4], o[5], o[6], o[7]);
            reinterpret_cast<uint4 *>(ws.tile_start + i0)[0] = a;
            reinterpret_cast<uint4 *>(ws.tile_start + i0)[1] = b;
            reinterpret_cast<uint4 *>(ws.cursor + i0)[0] = a;
            reinterpret_cast<uint4 *>(ws.cursor + i0)[1] = b;
        } else {
#pragma unroll
            for (int k = 0; k < kScanPer; ++k)
                if (i0 + k < TS) {
                    ws.tile_start[i0 + k] = o[k];
                    ws.cursor[i0 + k] = o[k];
                }
        }
#pragma unroll
        for (int j = 0; j < kScanPer; ++j) {
            len[j] = 0;
            if ((j & smask) == 0 && i0 + j < TS) {
                uint32_t l = c[j];
                if (S > 1) l += c[(j + 1) % kScanPer];
                if (S > 2) l += c[(j + 2) % kScanPer] + c[(j + 3) % kScanPer];
                len[j] = l;
                max_tile = max(max_tile, l);
                atomicAdd(&s_bucket[order_bucket(l)], 1u);
            }
        }
        carry += total;
    }
    if (tid == 0) {
        ws.tile_start[TS] = (uint32_t)min(carry, (unsigned long long)0xffffffffu);
    }
    __syncthreads();
    {  // exclusive scan of the buckets, one bucket per thread
        uint32_t total;
        const uint32_t c = s_bucket[tid];
        const uint32_t excl = block_exclusive_scan(c, warp_sum, total);
        s_bucket[tid] = excl;
    }
    __syncthreads();
    if (one_pass) {
#pragma unroll
        for (int j = 0; j < kScanPer; ++j) {
            const uint32_t i = (uint32_t)tid * kScanPer + (uint32_t)j;
            if ((j & smask) == 0 && i < TS) ws.tile_order[atomicAdd(&s_bucket[order_bucket(len[j])], 1u)] = i >> sshift;
        }
    } else {
        for (uint32_t t = tid; t < d.T; t += kScanThreads) {
            const uint32_t l = ws.tile_start[(t + 1) * S] - ws.tile_start[t * S];
            ws.tile_order[atomicAdd(&s_bucket[order_bucket(l)], 1u)] = t;
        }
    }
    unsigned long long recs = (unsigned long long)cc[0] + cc[1] + cc[2] + cc[3];
    for (uint32_t c = (uint32_t)tid + 4u * kScanThreads; c < ncell; c += kScanThreads) recs += ws.cell_cnt[c];
    max_tile = __reduce_max_sync(0xffffffffu, max_tile);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) recs += __shfl_xor_sync(0xffffffffu, recs, off);
    if (lane == 0) {
        atomicMax(&s_max, max_tile);
        atomicAdd(&s_recs, recs);
    }
    __syncthreads();
    if (tid == 0) {
        ws.hdr->max_tile = s_max;
        ws.hdr->n_rec = s_recs;
        ws.hdr->n_pairs = carry;
        if (carry > d.pair_cap) atomicOr(ws.err, (uint32_t)kErrPairs);
    }
}

// ------------------------------------------------------------ multi-block form of the scan
// For problems with more counters than one block covers in one pass (many views or small
// tiles), three kernels: (1) each block of kMBThreads sums a chunk of kMBChunk counters,
// counts its tiles into kMBuckets launch-order buckets (list length / 16, the longest
// first), and sums a slice of the cells' record counts; (2) one block turns the chunk sums
// and the bucket counts (bucket-major, so a bucket's blocks are consecutive) into
// exclusive offsets, and writes the totals to the header; (3) each block scans its chunk
// again from its offset, writes the list offsets and cursors, zeroes the counters, and
// places its tiles in the launch order from its buckets' offsets.  The per-block arrays
// live in ws.scan_part: sums, longest lists, record counts (NB each), then the bucket
// counts (kMBuckets x NB).

__device__ __forceinline__ uint32_t mb_bucket(uint32_t len) {
    return kMBuckets - 1 - min(len >> 4, (uint32_t)kMBuckets - 1);
}

// Exclusive scan of one value per thread over a block of NT threads (NT / 32 <= 32 warps);
// `total` gets the block sum.  Ends with a barrier.
template <int NT, class T>
__device__ __forceinline__ T block_scan_excl(T x, T *warp_sum, T &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T incl = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const T v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    T wi = lane < NT / 32 ? warp_sum[lane] : T(0);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const T v = __shfl_up_sync(0xffffffffu, wi, off);
        if (lane >= off) wi += v;
    }
    const T prev = __shfl_sync(0xffffffffu, wi, (warp + 31) & 31);
    total = __shfl_sync(0xffffffffu, wi, NT / 32 - 1);
    __syncthreads();
    return (warp > 0 ? prev : T(0)) + incl - x;
}

// This thread's kMBPer counters of chunk position i0 (vector loads where the run is whole).
__device__ __forceinline__ void load_counts(const uint32_t *cnt, uint32_t i0, uint32_t TS, uint32_t (&c)[kMBPer]) {
    if (i0 + kMBPer <= TS) {
        const uint4 *q = reinterpret_cast<const uint4 *>(cnt + i0);
        const uint4 a = q[0], b = q[1];
        c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w;
        c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
    } else {
#pragma unroll
        for (int k = 0; k < kMBPer; ++k) c[k] = i0 + k < TS ? cnt[i0 + k] : 0u;
    }
}

__global__ void __launch_bounds__(kMBThreads) k_scan_part(WsPtrs ws, Dims d) {
    griddep_wait();  // the predecessor's results are visible from here on
    griddep_launch_dependents();
    __shared__ uint32_t s_hist[kMBuckets], s_sum, s_max, s_rec;
    const uint32_t TS = d.T * d.S, smask = d.S - 1, NB = gridDim.x, b = blockIdx.x;
    const int tid = threadIdx.x;
    if (tid < kMBuckets) s_hist[tid] = 0u;
    if (tid == 0) s_sum = s_max = s_rec = 0u;
    __syncthreads();
    uint32_t c[kMBPer];
    const uint32_t i0 = b * kMBChunk + (uint32_t)tid * kMBPer;
    load_counts(ws.tile_cnt, i0, TS, c);
    uint32_t mine = 0, mx = 0;
#pragma unroll
    for (int j = 0; j < kMBPer; ++j) {
        mine += c[j];
        if ((j & smask) == 0 && i0 + j < TS) {  // the S counters of a tile sit in one thread
            uint32_t l = c[j];
            if (d.S > 1) l += c[(j + 1) % kMBPer];
            if (d.S > 2) l += c[(j + 2) % kMBPer] + c[(j + 3) % kMBPer];
            mx = max(mx, l);
            atomicAdd(&s_hist[mb_bucket(l)], 1u);
        }
    }
    const uint32_t ncell = (uint32_t)d.V * (uint32_t)d.nblk, cpb = (ncell + NB - 1) / NB;
    uint32_t rec = 0;
    for (uint32_t k = b * cpb + (uint32_t)tid; k < min(ncell, (b + 1) * cpb); k += kMBThreads) rec += ws.cell_cnt[k];
    mine = __reduce_add_sync(0xffffffffu, mine);
    mx = __reduce_max_sync(0xffffffffu, mx);
    rec = __reduce_add_sync(0xffffffffu, rec);
    if ((tid & 31) == 0) {
        atomicAdd(&s_sum, mine);
        atomicMax(&s_max, mx);
        atomicAdd(&s_rec, rec);
    }
    __syncthreads();
    uint32_t *part = ws.scan_part;
    if (tid == 0) {
        part[b] = s_sum;
        part[NB + b] = s_max;
        part[2 * NB + b] = s_rec;
    }
    if (tid < kMBuckets) part[3 * NB + (uint32_t)tid * NB + b] = s_hist[tid];
}

// In-place exclusive scan of a[0, n) by one block of kScanThreads (each thread a
// contiguous run); returns the total to every thread.  Sums saturate at 2^32 - 1 where
// they are stored.
__device__ __forceinline__ unsigned long long block_scan_array(uint32_t *a, uint32_t n,
                                                               unsigned long long *warp_sum) {
    const uint32_t per = (n + kScanThreads - 1) / kScanThreads, lo = min(n, (uint32_t)threadIdx.x * per),
                   hi = min(n, lo + per);
    unsigned long long sum = 0;
    for (uint32_t i = lo; i < hi; ++i) sum += a[i];
    unsigned long long total;
    unsigned long long run = block_scan_excl<kScanThreads>(sum, warp_sum, total);
    for (uint32_t i = lo; i < hi; ++i) {
        const uint32_t v = a[i];
        a[i] = (uint32_t)min(run, (unsigned long long)0xffffffffu);
        run += v;
    }
    return total;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_top(WsPtrs ws, Dims d) {
    griddep_wait();  // the predecessor's results are visible from here on
    griddep_launch_dependents();
    __shared__ unsigned long long warp_sum[kScanThreads / 32];
    __shared__ uint32_t s_max;
    __shared__ unsigned long long s_rec;
    const uint32_t TS = d.T * d.S, NB = (TS + kMBChunk - 1) / kMBChunk;
    const int tid = threadIdx.x;
    if (tid == 0) {
        s_max = 0u;
        s_rec = 0ull;
    }
    uint32_t *part = ws.scan_part;
    const unsigned long long total = block_scan_array(part, NB, warp_sum);  // chunk offsets
    block_scan_array(part + 3 * NB, kMBuckets * NB, warp_sum);              // launch-order offsets
    uint32_t mx = 0;
    unsigned long long rec = 0;
    for (uint32_t i = (uint32_t)tid; i < NB; i += kScanThreads) {
        mx = max(mx, part[NB + i]);
        rec += part[2 * NB + i];
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) rec += __shfl_xor_sync(0xffffffffu, rec, off);
    if ((tid & 31) == 0) {
        atomicMax(&s_max, mx);
        atomicAdd(&s_rec, rec);
    }
    __syncthreads();
    if (tid == 0) {
        ws.tile_start[TS] = (uint32_t)min(total, (unsigned long long)0xffffffffu);
        ws.hdr->max_tile = s_max;
        ws.hdr->n_rec = s_rec;
        ws.hdr->n_pairs = total;
        if (total > d.pair_cap) atomicOr(ws.err, (uint32_t)kErrPairs);
    }
}

__global__ void __launch_bounds__(kMBThreads) k_scan_write(WsPtrs ws, Dims d) {
    griddep_wait();  // the predecessor's results are visible from here on
    griddep_launch_dependents();
    __shared__ uint32_t warp_sum[kMBThreads / 32], s_pos[kMBuckets];
    const uint32_t TS = d.T * d.S, smask = d.S - 1, sshift = __ffs(d.S) - 1, NB = gridDim.x, b = blockIdx.x;
    const int tid = threadIdx.x;
    const uint32_t *part = ws.scan_part;
    if (tid < kMBuckets) s_pos[tid] = part[3 * NB + (uint32_t)tid * NB + b];
    uint32_t c[kMBPer];
    const uint32_t i0 = b * kMBChunk + (uint32_t)tid * kMBPer;
    load_counts(ws.tile_cnt, i0, TS, c);
    uint32_t mine = 0;
#pragma unroll
    for (int k = 0; k < kMBPer; ++k) mine += c[k];
    uint32_t total;
    const uint32_t excl = block_scan_excl<kMBThreads>(mine, warp_sum, total);  // (ends with a barrier)
    unsigned long long run = (unsigned long long)part[b] + excl;
    uint32_t o[kMBPer];
#pragma unroll
    for (int k = 0; k < kMBPer; ++k) {
        o[k] = (uint32_t)min(run, (unsigned long long)0xffffffffu);
        run += c[k];
    }
    if (i0 + kMBPer <= TS) {  // whole 32-byte rows: two vector stores per array
        const uint4 a = make_uint4(o[0], o[1], o[2], o[3]), e = make_uint4(o[4], o[5], o[6], o[7]);
        reinterpret_cast<uint4 *>(ws.tile_start + i0)[0] = a;
        reinterpret_cast<uint4 *>(ws.tile_start + i0)[1] = e;
        reinterpret_cast<uint4 *>(ws.cursor + i0)[0] = a;
        reinterpret_cast<uint4 *>(ws.cursor + i0)[1] = e;
        reinterpret_cast<uint4 *>(ws.tile_cnt + i0)[0] = make_uint4(0u, 0u, 0u, 0u);
        reinterpret_cast<uint4 *>(ws.tile_cnt + i0)[1] = make_uint4(0u, 0u, 0u, 0u);
    } else {
#pragma unroll
        for (int k = 0; k < kMBPer; ++k)
            if (i0 + k < TS) {
                ws.tile_start[i0 + k] = o[k];
                ws.cursor[i0 + k] = o[k];
                ws.tile_cnt[i0 + k] = 0u;
            }
    }
#pragma unroll
    for (int j = 0; j < kMBPer; ++j) {
        if ((j & smask) == 0 && i0 + j < TS) {
            uint32_t l = c[j];
            if (d.S > 1) l += c[(j + 1) % kMBPer];
            if (d.S > 2) l += c[(j + 2) % kMBPer] + c[(j + 3) % kMBPer];
            ws.tile_order[atomicAdd(&s_pos[mb_bucket(l)], 1u)] = (i0 + (uint32_t)j) >> sshift;
        }
    }
}

// Up to four passes of the one-block scan take less than the three launches of the
// multi-block form.
constexpr uint64_t kMultiBlockScanFrom = 4ull * kScanThreads * kScanPer;

cudaError_t launch_scan_tiles(const WsPtrs &ws, const Dims &d, cudaStream_t st) {
    const uint64_t TS = (uint64_t)d.T * d.S;
    if (TS <= kMultiBlockScanFrom || !ws.scan_part)
        return launch_dep(k_scan_tiles, dim3(1), dim3(kScanThreads), st, ws, d);
    const uint32_t NB = scan_blocks(TS);
    cudaError_t e = launch_dep(k_scan_part, dim3(NB), dim3(kMBThreads), st, ws, d);
    if (e == cudaSuccess) e = launch_dep(k_scan_top, dim3(1), dim3(kScanThreads), st, ws, d);
    if (e == cudaSuccess) e = launch_dep(k_scan_write, dim3(NB), dim3(kMBThreads), st, ws, d);
    return e;
}

template <int DT, bool ISO>
__global__ void __launch_bounds__(kBlock, 6) k_project(ProjectLaunch L) {
    griddep_wait();  // the predecessor's results are visible from here on
    griddep_launch_dependents();
    const int v = blockIdx.y, b = blockIdx.x, tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    __shared__ float sRt[12];
    __shared__ ViewInfo sv;
    __shared__ uint32_t warp_off[kWarps];
    __shared__ BinSmem<kProjectBox> sm;
    const uint32_t cell = (uint32_t)v * (uint32_t)L.d.nblk + (uint32_t)b;
    if (tid == 0) {
        load_pose(L.poses + 7 * v, sRt);
        sv = L.ws.views[v];
    }
    __syncthreads();
    if (b == 0 && tid < 12) L.ws.view_rt[12 * v + tid] = sRt[tid];
    // per-iteration counters start at zero (nothing else touches the header before the scan)
    if (b == 0 && v == 0 && tid < (int)(sizeof(DevHeader) / 8))
        reinterpret_cast<unsigned long long *>(L.ws.hdr)[tid] = 0ull;
    const ViewInfo vi = sv;
    const int64_t i = (int64_t)b * kBlock + tid;
    const Settings &S = L.s;
    float4 A = make_float4(0.f, 0.f, 0.f, 0.f), B = A, C = A;
    bool vis = false;
    int tx0 = 0, tx1 = 0, ty0 = 0, ty1 = 0;
    if (i < L.d.n) {
        const float mx = __ldg(L.g.means + 3 * i), my = __ldg(L.g.means + 3 * i + 1), mz = __ldg(L.g.means + 3 * i + 2);
        const float x = cam_coord(sRt, 0, mx, my, mz);
        const float y = cam_coord(sRt, 1, mx, my, mz);
        const float z = cam_coord(sRt, 2, mx, my, mz);
        bool reach = z > S.z_near;
        if (reach && S.alpha_min > 0.f) {
            // Early reject of a Gaussian whose support cannot reach the image, before the
            // covariance (it pays off when a warp's Gaussians are spatial neighbours, as in a
            // map built frame by frame): Sigma'_xx = |J0 M|^2 + e <= |J0|^2 s_max^2 + e
            // (M = W Rg diag(s), W and Rg orthonormal; J0 the first row of the clamped
            // Jacobian) and the support radius^2 is at most 2 ln(1 / alpha_min).  Widened by
            // 1 % and 3 px, so a Gaussian dropped here would also fail record_rect's box test.
            float lsm;
            if constexpr (ISO) {
                lsm = ld_attr<DT>(L.g.log_scales, i);
            } else {
                lsm = fmaxf(fmaxf(ld_attr<DT>(L.g.log_scales, 3 * i), ld_attr<DT>(L.g.log_scales, 3 * i + 1)),
                            ld_attr<DT>(L.g.log_scales, 3 * i + 2));
            }
            const float sm2 = __expf(2.f * lsm);
            const float iz = __fdividef(1.f, z);
            const float tx = fminf(fmaxf(x * iz, -vi.tan_lim_x), vi.tan_lim_x);
            const float ty = fminf(fmaxf(y * iz, -vi.tan_lim_y), vi.tan_lim_y);
            const float r2 = -2.f * __logf(S.alpha_min);
            const float hx = 1.01f * sqrtf(r2 * (vi.fx * vi.fx * iz * iz * (1.f + tx * tx) * sm2 + S.dilation)) + 3.f;
            const float hy = 1.01f * sqrtf(r2 * (vi.fy * vi.fy * iz * iz * (1.f + ty * ty) * sm2 + S.dilation)) + 3.f;
            const float mu_x = vi.fx * x * iz + vi.cx, mu_y = vi.fy * y * iz + vi.cy;
            reach = mu_x + hx >= 0.f && mu_x - hx <= (float)(vi.width - 1) && mu_y + hy >= 0.f &&
                    mu_y - hy <= (float)(vi.height - 1);
        }
        if (reach) {
            // M = W Rg diag(s): Sigma_c = M M^T (isotropic: M = s W)
            float M[9];
            if constexpr (ISO) {
                const float sc = __expf(ld_attr<DT>(L.g.log_scales, i));
#pragma unroll
                for (int k = 0; k < 9; ++k) M[k] = sRt[k] * sc;
            } else {
                float qw = ld_attr<DT>(L.g.quats, 4 * i), qx = ld_attr<DT>(L.g.quats, 4 * i + 1);
                float qy = ld_attr<DT>(L.g.quats, 4 * i + 2), qz = ld_attr<DT>(L.g.quats, 4 * i + 3);
                const float qq = qw * qw + qx * qx + qy * qy + qz * qz;
                const float qi = qq > 0.f ? rsqrtf(qq) : 0.f;
                qw *= qi; qx *= qi; qy *= qi; qz *= qi;
                float Rg[9];
                quat_to_rot(qw, qx, qy, qz, Rg);
                const float s0 = __expf(ld_attr<DT>(L.g.log_scales, 3 * i));
                const float s1 = __expf(ld_attr<DT>(L.g.log_scales, 3 * i + 1));
                const float s2 = __expf(ld_attr<DT>(L.g.log_scales, 3 * i + 2));
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    M[3 * r + 0] = (sRt[3 * r] * Rg[0] + sRt[3 * r + 1] * Rg[3] + sRt[3 * r + 2] * Rg[6]) * s0;
                    M[3 * r + 1] = (sRt[3 * r] * Rg[1] + sRt[3 * r + 1] * Rg[4] + sRt[3 * r + 2] * Rg[7]) * s1;
                    M[3 * r + 2] = (sRt[3 * r] * Rg[2] + sRt[3 * r + 1] * Rg[5] + sRt[3 * r + 2] * Rg[8]) * s2;
                }
            }
            const float iz = __fdividef(1.f, z);
            // J at the mean's image-plane tangent, clamped to the view's limits
            const float tx = fminf(fmaxf(x * iz, -vi.tan_lim_x), vi.tan_lim_x);
            const float ty = fminf(fmaxf(y * iz, -vi.tan_lim_y), vi.tan_lim_y);
            const float J00 = vi.fx * iz, J02 = -vi.fx * tx * iz;
            const float J11 = vi.fy * iz, J12 = -vi.fy * ty * iz;
            // N = J M, Sigma' = N N^T + dilation I
            float N0[3], N1[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                N0[c] = J00 * M[c] + J02 * M[6 + c];
                N1[c] = J11 * M[3 + c] + J12 * M[6 + c];
            }
            const float S00 = N0[0] * N0[0] + N0[1] * N0[1] + N0[2] * N0[2] + S.dilation;
            const float S01 = N0[0] * N1[0] + N0[1] * N1[1] + N0[2] * N1[2];
            const float S11 = N1[0] * N1[0] + N1[1] * N1[1] + N1[2] * N1[2] + S.dilation;
            // det(N N^T + e I) = |N0 x N1|^2 + e (S00 + S11) - e^2 (Cauchy-Binet): a sum of
            // squares, where S00 S11 - S01^2 cancels catastrophically once the footprint is
            // thin (N0, N1 nearly parallel: a Gaussian seen edge-on or close to the camera)
            const float cx = diff_of_products(N0[1], N1[2], N0[2], N1[1]);
            const float cy = diff_of_products(N0[2], N1[0], N0[0], N1[2]);
            const float cz = diff_of_products(N0[0], N1[1], N0[1], N1[0]);
            const float det = cx * cx + cy * cy + cz * cz + S.dilation * (S00 + S11 - S.dilation);
            if (det > 0.f) {
                const float idet = __fdividef(1.f, det);
                const float o = __fdividef(1.f, 1.f + __expf(-ld_attr<DT>(L.g.logits, i)));
                float dmax2;
                if (S.alpha_min > 0.f)
                    dmax2 = o >= S.alpha_min ? 2.f * __logf(__fdividef(o, S.alpha_min)) : -1.f;
                else
                    dmax2 = INFINITY;
                if (dmax2 >= 0.f) {
                    A = make_float4(vi.fx * x * iz + vi.cx, vi.fy * y * iz + vi.cy, z, o);
                    B = make_float4(S11 * idet, -S01 * idet, S00 * idet, dmax2);
                    C = make_float4(ld_attr<DT>(L.g.rgb, 3 * i), ld_attr<DT>(L.g.rgb, 3 * i + 1),
                                    ld_attr<DT>(L.g.rgb, 3 * i + 2),
                                    __uint_as_float((uint32_t)((int64_t)v * L.d.n + i)));
                    vis = record_rect(vi, A, B, tx0, tx1, ty0, ty1);
                }
            }
        }
    }
    // compaction into this block's cell: visible Gaussians take the first slots, in order
    const uint32_t ballot = __ballot_sync(0xffffffffu, vis);
    if (lane == 0) warp_off[warp] = __popc(ballot);
    post_rows(sm, vis, tx0, tx1, ty0, ty1);
    __syncthreads();
    uint32_t nrec = 0, slot = __popc(ballot & ((1u << lane) - 1u));
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = warp_off[w];
        slot += w < warp ? c : 0u;
        nrec += c;
    }
    if (tid == 0) L.ws.cell_cnt[cell] = nrec;
    if (nrec == 0) return;
    const BlockBox q = block_box(sm, kProjectBox);
    for (int k = tid; k < q.area; k += kBlock) sm.box[k] = 0u;
    const uint32_t before = q.solo ? 0u : rows_before(vis, ty0, ty1);
    if (vis) {
        const uint32_t rec = cell * kCell + slot;
        Rec r;
        r.a = A; r.b = B; r.c = C;
        L.ws.rec[rec] = r;
        RecGrad z;
        z.g0 = z.g1 = z.g2 = make_float4(0.f, 0.f, 0.f, 0.f);
        L.ws.rec_grad[rec] = z;
        if (!q.solo) {
            put_rows(sm.rec[slot], A, B, tx0, tx1, ty0);
            sm.pre[slot] = q.before + before;
        }
    }
    if (q.boxed || !q.solo) {
        if (tid == 0) sm.pre[nrec] = q.rows;
        __syncthreads();
    }
    // pair counts per (tile, sub-bucket of the cell)
    uint32_t *cnt = L.ws.tile_cnt + vi.tile_base * L.d.S + ((uint32_t)b & (L.d.S - 1));
    const int of_row = (int)((uint32_t)tid & (q.lanes - 1u));  // which of the row's threads this is
    const auto count = [&](int ty, int a0, int a1) {
        if (q.boxed) {
            uint32_t *row = sm.box + (ty - q.y) * q.w - q.x;
            for (int tx = a0; tx <= a1; ++tx) atomicAdd(row + tx, 1u);
        } else {
            for (int tx = a0 + of_row; tx <= a1; tx += (int)q.lanes)
                red_add(cnt + (uint32_t)(ty * vi.tiles_x + tx) * L.d.S, 1u);
        }
    };
    if (q.solo) {
        if (vis) for_own_rows(vi, A, B, tx0, tx1, ty0, ty1, count);
    } else {
        for_rows(sm, (int)nrec, vi, q.lanes, [&](int, int ty, int a0, int a1) { count(ty, a0, a1); });
    }
    if (!q.boxed) return;
    __syncthreads();
    for (int k = tid; k < q.area; k += kBlock) {
        const uint32_t c = sm.box[k];
        if (c) red_add(cnt + (uint32_t)((q.y + k / q.w) * vi.tiles_x + q.x + k % q.w) * L.d.S, c);
    }
}

cudaError_t launch_project(const ProjectLaunch &L, cudaStream_t st) {
    dim3 grid(L.d.nblk, L.d.V);
    const bool iso = L.g.quats == nullptr;  // isotropic Gaussians: one log-radius, no rotation
    cudaError_t e;
    switch (L.dtype) {
        case GS_F32:
            if (iso) e = launch_dep(k_project<GS_F32, true>, grid, dim3(kBlock), st, L);
            else e = launch_dep(k_project<GS_F32, false>, grid, dim3(kBlock), st, L);
            break;
        case GS_BF16:
            if (iso) e = launch_dep(k_project<GS_BF16, true>, grid, dim3(kBlock), st, L);
            else e = launch_dep(k_project<GS_BF16, false>, grid, dim3(kBlock), st, L);
            break;
        case GS_F16:
            if (iso) e = launch_dep(k_project<GS_F16, true>, grid, dim3(kBlock), st, L);
            else e = launch_dep(k_project<GS_F16, false>, grid, dim3(kBlock), st, L);
            break;
        default: return cudaErrorInvalidValue;
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Write one (record, tile) pair at its slot: for the per-tile sort the key depth bits << 32 |
// record; for the device-wide radix sort (GS_SCHED_RADIX) the key tile << 32 | depth bits
// with the record as the value.  Depths are positive, so their bits order as unsigned.
__device__ __forceinline__ void put_pair(const WsPtrs &ws, bool radix, uint32_t slot, uint32_t tile, uint32_t depth_bits,
                                         uint32_t rec) {
    if (radix) {
        ws.keys[slot] = ((unsigned long long)tile << 32) | depth_bits;
        ws.sorted[slot] = rec;
    } else {
        ws.keys[slot] = ((unsigned long long)depth_bits << 32) | rec;
    }
}

// One key per (record, tile met): depth bits (positive floats sort as unsigned ints) in
// the high word, the record in the low word, stored at the next free slot of the tile's
// sub-bucket.  One block per cell: the block counts its pairs per tile as k_project did,
// reserves each tile's slots with one atomic, and hands them out from shared memory.
__global__ void __launch_bounds__(kBlock, 6) k_emit(WsPtrs ws, Dims d) {
    // No early griddep_launch_dependents here: the sort's blocks would then be placed while
    // the emission still runs, on whichever SMs free first, and take slots from its own
    // blocks (12 views / 500k Gaussians: a call 2,900 -> 2,969 us; one view of 2M: 1,632 ->
    // 1,709 us).
    griddep_wait();  // the predecessor's results are visible from here on
    const uint32_t cell = blockIdx.x;
    const int nrec = (int)ws.cell_cnt[cell];
    if (nrec == 0) return;
    __shared__ BinSmem<kEmitBox> sm;
    __shared__ uint32_t s_depth[kBlock];
    const int tid = threadIdx.x;
    const int view = (int)(cell / (uint32_t)d.nblk);
    const ViewInfo vi = ws.views[view];
    float4 A = make_float4(0.f, 0.f, 0.f, 0.f), B = A;
    int tx0 = 0, tx1 = 0, ty0 = 0, ty1 = 0;
    bool has = false;
    if (tid < nrec) {
        const Rec &rec = ws.rec[cell * kCell + tid];
        A = rec.a;
        B = rec.b;
        has = record_rect(vi, A, B, tx0, tx1, ty0, ty1);
    }
    post_rows(sm, has, tx0, tx1, ty0, ty1);
    __syncthreads();
    const BlockBox q = block_box(sm, kEmitBox);
    for (int k = tid; k < q.area; k += kBlock) sm.box[k] = 0u;
    const uint32_t before = q.solo ? 0u : rows_before(has, ty0, ty1);
    if (!q.solo && tid < nrec) {
        put_rows(sm.rec[tid], A, B, tx0, tx1, ty0);
        sm.pre[tid] = q.before + before;
        s_depth[tid] = __float_as_uint(A.z);
    }
    if (q.boxed || !q.solo) {
        if (tid == 0) sm.pre[nrec] = q.rows;
        __syncthreads();
    }
    const bool radix = (d.flags & GS_SCHED_RADIX) != 0;
    const uint32_t sub = (cell % (uint32_t)d.nblk) & (d.S - 1), first = cell * kCell;
    const auto bucket_of = [&](int ty, int tx) { return (vi.tile_base + (uint32_t)(ty * vi.tiles_x + tx)) * d.S + sub; };
    if (!q.boxed) {
        const int g = (int)q.lanes, of_row = tid & (g - 1);
        const auto emit = [&](uint32_t depth, uint32_t r, int ty, int a0, int a1) {
            for (int t0 = a0 + of_row; t0 <= a1; t0 += 4 * g) {  // four atomics in flight before the stores
                uint32_t slot[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (t0 + k * g <= a1) slot[k] = atomicAdd(ws.cursor + bucket_of(ty, t0 + k * g), 1u);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (t0 + k * g <= a1) {
                        const uint32_t bucket = bucket_of(ty, t0 + k * g);
                        if (slot[k] < ws.tile_start[bucket + 1] && slot[k] < d.pair_cap)
                            put_pair(ws, radix, slot[k], bucket / d.S, depth, first + r);
                        else
                            atomicOr(ws.err, (uint32_t)kErrPairs);
                    }
            }
        };
        if (!q.solo) {
            for_rows(sm, nrec, vi, q.lanes, [&](int r, int ty, int a0, int a1) { emit(s_depth[r], (uint32_t)r, ty, a0, a1); });
        } else if (has) {
            for_own_rows(vi, A, B, tx0, tx1, ty0, ty1,
                         [&](int ty, int a0, int a1) { emit(__float_as_uint(A.z), (uint32_t)tid, ty, a0, a1); });
        }
        return;
    }
    const auto count = [&](int ty, int a0, int a1) {
        uint32_t *row = sm.box + (ty - q.y) * q.w - q.x;
        for (int tx = a0; tx <= a1; ++tx) atomicAdd(row + tx, 1u);
    };
    uint32_t span[kSoloRows];  // solo: the row's tiles in the box (first | last << 16; empty: 1 | 0)
    if (q.solo) {
#pragma unroll
        for (int k = 0; k < kSoloRows; ++k) span[k] = 1u;
        if (has) {
            const RowSpan s = row_span_setup(A.x, A.y, B.x, B.y, B.z, B.w);
#pragma unroll
            for (int k = 0; k < kSoloRows; ++k)
                if (ty0 + k <= ty1) {
                    int a0, a1;
                    row_span(vi, s, ty0 + k, tx0, tx1, a0, a1);
                    if (a0 <= a1) {
                        span[k] = (uint32_t)(a0 - q.x) | (uint32_t)(a1 - q.x) << 16;
                        count(ty0 + k, a0, a1);
                    }
                }
        }
    } else {
        for_rows(sm, nrec, vi, 1u, [&](int, int ty, int a0, int a1) { count(ty, a0, a1); });
    }
    __syncthreads();
    for (int k0 = tid; k0 < q.area; k0 += 4 * kBlock) {  // counts to first slots, four tiles in flight
        uint32_t c[4], at[4], end[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = k0 + k * kBlock;
            c[k] = i < q.area ? sm.box[i] : 0u;
            if (c[k]) {
                const uint32_t bucket = bucket_of(q.y + i / q.w, q.x + i % q.w);
                at[k] = atomicAdd(ws.cursor + bucket, c[k]);
                end[k] = ws.tile_start[bucket + 1];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (c[k]) {
                sm.box[k0 + k * kBlock] = at[k];
                if (at[k] + c[k] > end[k] || at[k] + c[k] > d.pair_cap) atomicOr(ws.err, (uint32_t)kErrPairs);
                if (at[k] + c[k] > end[k]) sm.box[k0 + k * kBlock] = d.pair_cap;  // never past the tile's slots
            }
    }
    __syncthreads();
    const auto put = [&](uint32_t depth, uint32_t r, int ty, int a0, int a1) {
        uint32_t *row = sm.box + (ty - q.y) * q.w - q.x;
        for (int tx = a0; tx <= a1; ++tx) {
            const uint32_t slot = atomicAdd(row + tx, 1u);
            if (slot < d.pair_cap)
                put_pair(ws, radix, slot, vi.tile_base + (uint32_t)(ty * vi.tiles_x + tx), depth, first + r);
        }
    };
    if (q.solo) {
#pragma unroll
        for (int k = 0; k < kSoloRows; ++k)
            put(__float_as_uint(A.z), (uint32_t)tid, ty0 + k, q.x + (int)(span[k] & 0xffffu), q.x + (int)(span[k] >> 16));
    } else {
        for_rows(sm, nrec, vi, 1u, [&](int r, int ty, int a0, int a1) { put(s_depth[r], (uint32_t)r, ty, a0, a1); });
    }
}

cudaError_t launch_emit(const WsPtrs &ws, const Dims &d, cudaStream_t st) {
    const cudaError_t e = launch_dep(k_emit, dim3((uint32_t)d.V * (uint32_t)d.nblk), dim3(kBlock), st, ws, d);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace gsk
