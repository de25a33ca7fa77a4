// metrics.cu -- image-quality sums of a rendered view against its RGB-D observation, the
// quantities behind the evaluation of Sec. IV (PSNR of the colour, the average depth
// error), summed in a fixed order, so repeated calls agree bit for bit.
//
// The call has no scratch memory, so the sums cannot pass between independent blocks; one
// cluster of 16 blocks adds its partials through distributed shared memory instead.  The
// sums are taken on the FP32 pipes: FP64 runs at a sixty-fourth of the FP32 rate here, and in
// FP64 the pass was bound by it (one block: 1,536 us at 640 x 480).  A colour error and its square
// are exact up to the rounding of the square's low part (the difference and its rounding error,
// the square and its rounding error), and a thread, then eight threads, add them in three
// floats, each taking the rounding errors of the one before; everything across groups of eight
// threads is FP64.  The low parts' roundings (2^-49 of a square) have either sign, so a frame's
// sums end within the last FP64 additions' roundings of the exact ones.  The third float is for
// that: with two, the squares of the differences' rounding errors (all positive, below the low
// parts' last bits) were lost, and 640 x 480 sums were up to 46 units of 2^-53 low; FP64 sums in
// one block, a thread adding hundreds of terms, up to 14 off; here 1.9 (six images of noise).
// Errors outside (2^-40, 2^40) take the FP64 path: inside, the squares of eight threads' pixels
// add to less than FP32's 2^128 for up to 2^43 pixels a thread, and a square's rounding error is a
// normal number.  Measured at 640 x 480 (9.8 MB through 16 SMs): 26 us (21 with two floats), bound by
// instruction issue (68 % of the 16 SMs' cycles) and the loads.
#include <cooperative_groups.h>

#include "gs_internal.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kMetricThreads = 1024;
constexpr int kMetricCluster = 16;   // not a portable size: 8 where 16 blocks do not fit together
constexpr int kMetricPortable = 8;

// Error-free transformations (Knuth's TwoSum): a + b = s + e exactly.
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
    const float s = __fadd_rn(a, b), v = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
    return s;
}

// The same for a, b >= 0: Dekker's Fast2Sum on the ordered pair (five instructions for six, two of
// them beside the FP32 pipe).
__device__ __forceinline__ float two_sum_pos(float a, float b, float &e) {
    const float x = fmaxf(a, b), y = fminf(a, b);
    const float s = __fadd_rn(x, y);
    e = __fsub_rn(y, __fsub_rn(s, x));
    return s;
}

// A sum in three floats: the rounding errors of h go to m, those of m to l.
struct Sum3 {
    float h, m, l;
};

// s + (hi + lo + tail): hi >= 0 like h, tail of the size of l.
__device__ __forceinline__ void accumulate(Sum3 &s, float hi, float lo, float tail) {
    float e, f, g;
    s.h = two_sum_pos(s.h, hi, e);
    s.m = two_sum(s.m, e, f);
    s.m = two_sum(s.m, lo, g);
    s.l = __fadd_rn(s.l, __fadd_rn(tail, __fadd_rn(f, g)));
}

// Is the error a - b (rounded: s) in the range where its square's parts are normal FP32
// numbers and any image's sum of such squares is finite?  Exactly zero is.
__device__ __forceinline__ bool plain(float s) {
    const float m = fabsf(s);
    return m < 0x1p40f && (m > 0x1p-40f || m == 0.f);
}

// (s + t)^2 with s + t the exact difference: s^2 = p + q exactly, then 2 s t and t^2.
__device__ __forceinline__ void add_square(Sum3 &sum, float s, float t) {
    const float p = __fmul_rn(s, s), q = __fmaf_rn(s, s, -p);
    accumulate(sum, p, __fmaf_rn(2.f * s, t, q), __fmul_rn(t, t));
}

constexpr int kLanesPer = 8;  // threads whose sums are added before they become FP64
constexpr int kParts = kMetricThreads / kLanesPer;

__global__ void __launch_bounds__(kMetricThreads) k_image_metrics(const float *rgb, const float *depth,
                                                                 const float *rgb_t, const float *depth_t,
                                                                 int64_t P, double *out) {
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ Sum3 s_part[3][kParts];
    __shared__ double s_warp_slow[3][kMetricThreads / 32], s_block[4];
    __shared__ unsigned long long s_cnt;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_cnt = 0ull;
    const int64_t step = (int64_t)gridDim.x * kMetricThreads;  // the grid is one cluster
    Sum3 sum[3] = {};            // squared colour, |depth|, squared depth
    double slow[3] = {};         // the same of errors outside the pairs' range
    bool any_slow = false;
    uint32_t cnt = 0;
    const auto take = [&](const float (&a)[4], const float (&b)[4]) {
        float t;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float s = two_sum(a[c], -b[c], t);
            if (plain(s)) {
                add_square(sum[0], s, t);
            } else {
                const double e = (double)a[c] - (double)b[c];
                slow[0] += e * e;
                any_slow = true;
            }
        }
        if (b[3] > 0.f) {
            const float s = two_sum(a[3], -b[3], t);
            if (plain(s)) {
                accumulate(sum[1], fabsf(s), s < 0.f ? -t : t, 0.f);
                add_square(sum[2], s, t);
            } else {
                const double e = (double)a[3] - (double)b[3];
                slow[1] += fabs(e);
                slow[2] += e * e;
                any_slow = true;
            }
            ++cnt;
        }
    };
    const auto load = [&](int64_t p, float (&a)[4], float (&b)[4]) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            a[c] = rgb[c * P + p];
            b[c] = rgb_t[c * P + p];
        }
        a[3] = depth[p];
        b[3] = depth_t[p];
    };
    int64_t p = (int64_t)blockIdx.x * kMetricThreads + tid;
    while (p < P) {  // two pixels' sixteen loads in flight
        float a0[4], b0[4], a1[4], b1[4];
        const bool two = p + step < P;
        load(p, a0, b0);
        load(two ? p + step : p, a1, b1);
        take(a0, b0);
        if (two) take(a1, b1);
        p += 2 * step;
    }
    // eight threads' sums by shuffles, then FP64 over the block's 128 groups: a warp-wide
    // FP64 instruction takes 16 cycles of the SM however few lanes want it
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int o = 1; o < kLanesPer; o <<= 1) {
            const float h = __shfl_xor_sync(0xffffffffu, sum[k].h, o), m = __shfl_xor_sync(0xffffffffu, sum[k].m, o);
            const float l = __shfl_xor_sync(0xffffffffu, sum[k].l, o);
            accumulate(sum[k], h, m, l);
        }
        if ((lane & (kLanesPer - 1)) == 0) s_part[k][tid / kLanesPer] = sum[k];
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    __syncthreads();  // s_cnt is set
    if (lane == 0) atomicAdd(&s_cnt, (unsigned long long)cnt);
    if (__any_sync(0xffffffffu, any_slow)) {
#pragma unroll
        for (int k = 0; k < 3; ++k)
            for (int o = 16; o > 0; o >>= 1) slow[k] += __shfl_xor_sync(0xffffffffu, slow[k], o);
    }
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < 3; ++k) s_warp_slow[k][warp] = slow[k];
    __syncthreads();
    if (warp < 3) {
        double acc = s_warp_slow[warp][lane];  // kMetricThreads / 32 = 32 warps
        for (int i = lane; i < kParts; i += 32) {
            const Sum3 q = s_part[warp][i];
            acc += (double)q.h + ((double)q.m + (double)q.l);
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) s_block[warp < 2 ? warp : 3] = acc;
    }
    if (tid == 96) s_block[2] = (double)s_cnt;
    cluster.sync();
    if (cluster.block_rank() == 0 && threadIdx.x < 4) {
        double acc = 0.0;
        for (unsigned r = 0; r < cluster.num_blocks(); ++r) acc += *cluster.map_shared_rank(&s_block[threadIdx.x], r);
        out[threadIdx.x] = acc;
    }
    cluster.sync();  // no block leaves while its sums may still be read
}

}  // namespace

extern "C" gs_status gs_image_metrics(const float *rgb, const float *depth, const float *rgb_t, const float *depth_t,
                                      int64_t pixels, double *out, void *stream) {
    if (!rgb || !depth || !rgb_t || !depth_t || !out || pixels < 1) return GS_ERR_INVALID_ARG;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kMetricThreads);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const auto shape = [&](unsigned blocks) {
        cfg.gridDim = dim3(blocks);
        attr[0].val.clusterDim.x = blocks;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    };
    if (cudaFuncSetAttribute(k_image_metrics, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return GS_ERR_CUDA;
    shape(kMetricCluster);
    int fits = 0;
    if (cudaOccupancyMaxActiveClusters(&fits, k_image_metrics, &cfg) != cudaSuccess || fits < 1) {
        cudaGetLastError();
        shape(kMetricPortable);
    }
    if (cudaLaunchKernelEx(&cfg, k_image_metrics, rgb, depth, rgb_t, depth_t, pixels, out) != cudaSuccess)
        return GS_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}
