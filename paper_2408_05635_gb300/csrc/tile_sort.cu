// tile_sort.cu -- the depth order of every tile's list.
//
// Eqs. 2-4 composite the Gaussians of a pixel front to back, so every tile needs its
// entries in ascending camera depth; ties are broken by Gaussian index (the order the
// oracle uses), which the record index already encodes (records are numbered in
// (view, Gaussian) order).  k_emit leaves each tile's 64-bit keys (depth bits << 32 |
// record) in arrival order inside the tile's own slice of the key array, so the sort is
// segmented by construction: one block per tile sorts its slice and writes the record ids,
// in order, to `sorted` for the compositors.
//
// Up to kSortKeys keys: a distribution sort with the keys in registers.  They fall into
// kFine buckets linear in depth between the list's own extremes (a monotone map, so the
// order across buckets is exact); a counter's atomic gives each key its slot in its bucket,
// a scan of the counters the buckets' places; and a key's place inside its bucket is the
// number of smaller keys there (a few: buckets outnumber keys).  Depths so crowded that a
// bucket would hold more than kBucketMax keys take a bitonic network in shared memory.
// Longer slices: a sample sort.  kSortKeys keys at equal strides are sorted as above, every
// eighth is a splitter, the record ids are grouped by the intervals between them, and runs
// of intervals that fit kSortKeys are sorted as above.  The splitters are whole keys, so
// crowded or equal depths spread as evenly as others do.  An interval that holds more than
// kSortKeys (from about 50k keys on a few, beyond 130k most) is put aside and split again by
// samples of its own.  Only where an interval keeps more than seven eighths of its range, which
// takes equal keys (stale ones, after a capacity overflow), does a bitonic network in global
// memory sort the range.  When one long interval, or a list beyond 65,536 keys, sent the whole
// list through the network, a render of 60,000 in one tile of 4,096 took 15.2 ms instead of 5.8,
// of 130,000 34.7 instead of 13.2 (the network inside the compositor, with blocks of 256
// threads: 9.7 and 22.1).
//
// Bound by latency and instruction issue (a list is read once: 15 MB for the window below).
// As a kernel of its own it runs with many small blocks per SM, and leaves the compositors
// without its 16 KB of shared memory; in the compositor's block (runs of 32 by a bitonic
// network, merged pairwise; a network in global memory above 1,024 keys) the sort had cost
// 164 us of k_forward's 928 for 7.4 M keys in 25,800 lists (here 60 us, the compositor 763),
// 52 of 267 us for 1.9 M keys (15 us), 342 of 840 us for 2.2 M keys in 1,200 lists of up
// to 7,306 (88 us) and 5 of 45 us for 0.22 M keys in 1,200 lists (6 us).
#include "gs_internal.cuh"

namespace gsk {

constexpr int kSortKeys = 1024;
template <int NT>
constexpr int kPer = kSortKeys / NT;  // keys per thread of NT
constexpr int kFine = 1024;
constexpr int kBucketMax = 128;            // comparing a fuller bucket's keys would cost more than the network
constexpr int kCoarse = 128;               // intervals of a long list
constexpr int kStride = kSortKeys / kCoarse;
constexpr int kTodo = 256;                 // intervals put aside: those of two levels

typedef unsigned long long Key;

__device__ __forceinline__ void cmp_swap(Key *k, int lo, int hi) {
    const Key a = k[lo], b = k[hi];
    if (a > b) {
        k[lo] = b;
        k[hi] = a;
    }
}

// Ascending bitonic sort of k[0, n) by all threads of the block.  Each merge of size
// `size` starts with a mirrored comparison (lo, size-1-lo) followed by half-cleaners, so
// every compare-exchange puts the smaller key at the lower index and entries >= n can
// be treated as +inf without being stored.
template <int NT>
__device__ __noinline__ void bitonic_sort(Key *k, int n) {
    int P = 1;
    while (P < n) P <<= 1;
    const int pairs = P >> 1;
    for (int size = 2; size <= P; size <<= 1) {
        const int half = size >> 1;
        for (int p = threadIdx.x; p < pairs; p += NT) {
            const int blk = p / half, off = p - blk * half;
            const int lo = blk * size + off, hi = blk * size + size - 1 - off;
            if (hi < n) cmp_swap(k, lo, hi);
        }
        __syncthreads();
        for (int j = half >> 1; j > 0; j >>= 1) {
            for (int p = threadIdx.x; p < pairs; p += NT) {
                const int lo = (p / j) * 2 * j + (p % j), hi = lo + j;
                if (hi < n) cmp_swap(k, lo, hi);
            }
            __syncthreads();
        }
    }
}

template <int NT>
struct SortSmem {
    Key keys[kSortKeys];
    // two 16-bit counters per word: at most kSortKeys keys, so none carries into its neighbour
    uint32_t fine[kFine / 2];
    Key split[kCoarse];
    uint32_t coarse[kCoarse];
    uint32_t lo[NT / 32], hi[NT / 32], sum[NT / 32], mx[NT / 32];
    uint2 todo[kTodo];  // first place and number of keys of the intervals put aside
};

// The block's shared memory, by name in every function that uses it (through a reference it would be
// addressed as any memory).
template <int NT>
__device__ __forceinline__ SortSmem<NT> &sort_smem() {
    __shared__ SortSmem<NT> sm;
    return sm;
}

// Bucket of a depth: linear between the list's extremes.  Rounded subtraction and
// multiplication are monotone, so a smaller depth never lands in a later bucket (equal
// extremes or an infinite depth put everything into the first or the last one).
__device__ __forceinline__ uint32_t depth_bucket(Key key, float first, float scale) {
    return min(__float2uint_rz(__fmul_rn(__fsub_rn(__uint_as_float((uint32_t)(key >> 32)), first), scale)),
               (uint32_t)kFine - 1);
}

// Exclusive prefix over the block of each thread's `sum`, and the block's largest `mx`.
// Contains one barrier.
template <int NT>
__device__ __forceinline__ uint32_t block_prefix(uint32_t sum, uint32_t &mx, SortSmem<NT> &sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 31) {
        sm.sum[warp] = incl;
        sm.mx[warp] = mx;
    }
    __syncthreads();
    uint32_t base = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        base += w < warp ? sm.sum[w] : 0u;
        mx = max(mx, sm.mx[w]);
    }
    return base + incl - sum;
}

// Sort n <= kSortKeys keys, key k of thread tid being number tid + k NT, and
// emit(place, key) each.  Ends with a barrier.
template <int NT, class Emit>
__device__ __forceinline__ void sort_keys(const Key (&key)[kPer<NT>], int n, SortSmem<NT> &sm, Emit &&emit) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // extremes of the depth bits (positive depths order as unsigned)
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int k = 0; k < kPer<NT>; ++k)
        if (tid + k * NT < n) {
            lo = min(lo, (uint32_t)(key[k] >> 32));
            hi = max(hi, (uint32_t)(key[k] >> 32));
        }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
        sm.lo[warp] = lo;
        sm.hi[warp] = hi;
    }
#pragma unroll
    for (int k = 0; k < kFine / 2 / NT; ++k) sm.fine[tid + k * NT] = 0u;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        lo = min(lo, sm.lo[w]);
        hi = max(hi, sm.hi[w]);
    }
    const float first = __uint_as_float(lo), scale = __fdiv_rn((float)kFine, __fsub_rn(__uint_as_float(hi), first));
    uint32_t at[kPer<NT>];  // bucket, and the key's slot in it << 16
#pragma unroll
    for (int k = 0; k < kPer<NT>; ++k)
        if (tid + k * NT < n) {
            const uint32_t b = depth_bucket(key[k], first, scale), sh = (b & 1u) * 16u;
            at[k] = b | ((atomicAdd(&sm.fine[b >> 1], 1u << sh) >> sh) & 0xffffu) << 16;
        }
    __syncthreads();
    // counts to first places, each thread a contiguous run of counters
    constexpr int kWords = kFine / 2 / NT;
    uint32_t w[kWords], sum = 0, mx = 0;
#pragma unroll
    for (int k = 0; k < kWords; ++k) {
        w[k] = sm.fine[tid * kWords + k];
        sum += (w[k] & 0xffffu) + (w[k] >> 16);
        mx = max(mx, max(w[k] & 0xffffu, w[k] >> 16));
    }
    uint32_t run = block_prefix(sum, mx, sm);
    if (mx > (uint32_t)kBucketMax) {
#pragma unroll
        for (int k = 0; k < kPer<NT>; ++k)
            if (tid + k * NT < n) sm.keys[tid + k * NT] = key[k];
        __syncthreads();
        bitonic_sort<NT>(sm.keys, n);
        for (int i = tid; i < n; i += NT) emit((uint32_t)i, sm.keys[i]);
        __syncthreads();
        return;
    }
#pragma unroll
    for (int k = 0; k < kWords; ++k) {
        const uint32_t l = w[k] & 0xffffu;
        sm.fine[tid * kWords + k] = run | (run + l) << 16;
        run += l + (w[k] >> 16);
    }
    __syncthreads();
    const auto first_place = [&](uint32_t b) { return (sm.fine[b >> 1] >> ((b & 1u) * 16u)) & 0xffffu; };
#pragma unroll
    for (int k = 0; k < kPer<NT>; ++k)
        if (tid + k * NT < n) sm.keys[first_place(at[k] & 0xffffu) + (at[k] >> 16)] = key[k];
    __syncthreads();
    // in bucket order, so that neighbouring threads write neighbouring places
    for (int i = tid; i < n; i += NT) {
        const Key x = sm.keys[i];
        const uint32_t b = depth_bucket(x, first, scale), s = first_place(b);
        const uint32_t e = b + 1u < (uint32_t)kFine ? first_place(b + 1u) : (uint32_t)n;
        uint32_t place = s;
        for (uint32_t j = s; j < e; ++j) place += sm.keys[j] < x;
        emit(place, x);
    }
    __syncthreads();
}

// Intervals of a long list's keys: the number of splitters below each (the last sample is
// no splitter).  The searches advance together, so their loads overlap.
template <int PER>
__device__ __forceinline__ void intervals_of(const Key *split, const Key (&key)[PER], uint32_t (&at)[PER]) {
#pragma unroll
    for (int k = 0; k < PER; ++k) at[k] = 0u;
#pragma unroll
    for (uint32_t step = kCoarse / 2; step > 0; step >>= 1)
#pragma unroll
        for (int k = 0; k < PER; ++k) at[k] += split[at[k] + step - 1u] < key[k] ? step : 0u;
}

// The key of a record: its depth, as k_emit wrote it.
__device__ __forceinline__ Key key_of(const Rec *rec, uint32_t slots, uint32_t r) {
    return (Key)(r < slots ? __float_as_uint(rec[r].a.z) : 0u) << 32 | r;
}

// The m > kSortKeys keys of a list's slice from place `base` on: their record ids grouped by sampled
// intervals and sorted in those that fit; the others are put aside after the `waiting` ones there.
// Returns how many wait (more than kTodo: the last ones are not noted).
template <int NT>
__device__ __forceinline__ int sort_level(const Rec *rec, uint32_t slots, const Key *keys, uint32_t *out, int m, uint32_t base,
                                          int waiting, SortSmem<NT> &sm) {
    const int tid = threadIdx.x;
    Key key[kPer<NT>];
#pragma unroll
    for (int k = 0; k < kPer<NT>; ++k)
        key[k] = keys[(uint32_t)((uint64_t)(tid + k * NT) * (uint32_t)m / (uint32_t)kSortKeys)];
    sort_keys(key, kSortKeys, sm, [&](uint32_t place, Key x) {
        if (place % kStride == kStride - 1) sm.split[place / kStride] = x;
    });
    if (tid < kCoarse) sm.coarse[tid] = 0u;
    __syncthreads();
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {  // count, then place
        for (int i = tid; i < m; i += kSortKeys) {
#pragma unroll
            for (int k = 0; k < kPer<NT>; ++k)
                key[k] = keys[min(i + k * NT, m - 1)];
            uint32_t at[kPer<NT>];
            intervals_of(sm.split, key, at);
#pragma unroll
            for (int k = 0; k < kPer<NT>; ++k)
                if (i + k * NT < m) {
                    const uint32_t slot = atomicAdd(&sm.coarse[at[k]], 1u);
                    if (pass) out[slot] = (uint32_t)key[k];
                }
        }
        __syncthreads();
        if (pass == 0) {
            uint32_t mx = tid < kCoarse ? sm.coarse[tid] : 0u;
            const uint32_t first = block_prefix(mx, mx, sm);
            if (tid < kCoarse) sm.coarse[tid] = first;
            __syncthreads();
        }
    }
    // coarse[k] is now the end of interval k: sort as many intervals at a time as fit
    uint32_t done = 0;
    for (int k = 0; done < (uint32_t)m;) {
        int l = k, e = kCoarse;  // the first interval that ends beyond the buffer
        while (l < e) {
            const int mid = (l + e) >> 1;
            if (sm.coarse[mid] <= done + (uint32_t)kSortKeys) l = mid + 1; else e = mid;
        }
        if (l == k) {  // interval k alone is too long
            const uint32_t size = sm.coarse[k] - done;
            if (tid == 0 && waiting < kTodo) sm.todo[waiting] = make_uint2(base + done, size);
            ++waiting;
            done += size;
            ++k;
            continue;
        }
        const int c = (int)(sm.coarse[l - 1] - done);
        uint32_t *to = out + done;
#pragma unroll
        for (int j = 0; j < kPer<NT>; ++j)
            if (tid + j * NT < c) key[j] = key_of(rec, slots, to[tid + j * NT]);
        sort_keys(key, c, sm, [&](uint32_t place, Key x) { to[place] = (uint32_t)x; });
        done += (uint32_t)c;
        k = l;
    }
    return waiting;
}

// The intervals that the first level over a list's n keys put aside, and theirs.  Each is split by
// samples of its own once the keys stand in the intervals' order; where an interval keeps more
// than seven eighths of its range (equal keys), the range goes through the network, so the levels are few
// whatever the keys.  A function of its own: in the kernel's body it cost the lists that need none of it
// (80 bytes of spills a thread; a render of 1M at 1200 x 680, longest list 1,224, 194.7 -> 198.3 us).
template <int NT>
__device__ __noinline__ void sort_waiting(const Rec *rec, uint32_t slots, Key *keys, uint32_t *out, int n, int waiting) {
    SortSmem<NT> &sm = sort_smem<NT>();
    uint32_t base = 0;
    int m = n, before = 0;  // the range just split; [before, waiting): its intervals
    for (;;) {
        __syncthreads();  // (the intervals are noted, and coarse read)
        if (waiting > before) {
            bool split = waiting <= kTodo;
            for (int w = before; split && w < waiting; ++w) split = sm.todo[w].y <= (uint32_t)(m - m / 8);
            if (split) {
                for (int i = threadIdx.x; i < m; i += NT) keys[base + i] = key_of(rec, slots, out[base + i]);
            } else {
                bitonic_sort<NT>(keys + base, m);
                for (int i = threadIdx.x; i < m; i += NT) out[base + i] = (uint32_t)keys[base + i];
                waiting = before;
            }
            __syncthreads();
        }
        if (waiting == 0) return;
        const uint2 next = sm.todo[--waiting];
        base = next.x;
        m = (int)next.y;
        before = waiting;
        waiting = sort_level<NT>(rec, slots, keys + base, out + base, m, base, waiting, sm);
    }
}

// Pair capacity per tile from which lists are taken to be long.  Blocks of 128 threads keep
// more lists in flight (lists of 290 keys: 60 us against 80 with 256 threads; of 385: 40
// against 53), blocks of 256 sort a long list sooner (513 keys on average, up to 1,858: 27
// against 34 us; 1,847, up to 7,306: 88 against 113; 512 threads: 44 and 87).  The capacity
// stands for the keys, which only the device knows when the kernel is launched: with 1.25 pairs
// reserved for one the line is at 513 keys a tile, with 1.05 at 610, and lists between those then
// take the 34 us.
constexpr uint32_t kLongLists = 640;

// One block per tile, the longest lists first.  The key slice is left as it is or permuted, so the sort can be run
// again on it.
template <int NT>
__global__ void __launch_bounds__(NT, 1280 / NT) k_sort_tiles(WsPtrs ws, Dims d) {
    static_assert(kFine / 2 % NT == 0 && kCoarse <= NT, "counters per thread");
    // no early griddep_launch_dependents: the compositor's longest tiles, launched first,
    // would crowd onto the SMs that free first
    griddep_wait();  // the predecessor's results are visible from here on
    SortSmem<NT> &sm = sort_smem<NT>();
    const int tid = threadIdx.x;
    uint32_t start;
    const int n = (int)tile_entries(ws, d, ws.tile_order[blockIdx.x], start);
    if (n == 0) return;
    Key *keys = ws.keys + start;
    uint32_t *out = ws.sorted + start;
    Key key[kPer<NT>];
    if (n <= kSortKeys) {
#pragma unroll
        for (int k = 0; k < kPer<NT>; ++k)
            if (tid + k * NT < n) key[k] = keys[tid + k * NT];
        sort_keys(key, n, sm, [&](uint32_t place, Key x) { out[place] = (uint32_t)x; });
        return;
    }
    const int waiting = sort_level<NT>(ws.rec, rec_slots(d), keys, out, n, 0u, 0, sm);
    if (waiting > 0) sort_waiting<NT>(ws.rec, rec_slots(d), keys, out, n, waiting);
}

cudaError_t launch_sort_tiles(const WsPtrs &ws, const Dims &d, cudaStream_t st) {
    if (d.pair_cap / kLongLists >= d.T) return launch_dep(k_sort_tiles<256>, dim3(d.T), dim3(256), st, ws, d);
    return launch_dep(k_sort_tiles<128>, dim3(d.T), dim3(128), st, ws, d);
}

}  // namespace gsk
