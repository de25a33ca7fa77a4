// mapping.cu -- the map side of the method: Gaussians made from an RGB-D frame (the first
// frame, Sec. III-A, and the new observations of a keyframe, Sec. III-C), the
// gradient-based update of every Gaussian parameter with the keyframe poses fixed, and
// the removal of Gaussians whose opacity fell away (duplicate removal, Sec. III-C).
//
// All three are HBM-bound passes over flat arrays.  The two that change the number of
// Gaussians are stable compactions in two launches: a block-count pass, then an emit
// pass in which every block sums the counts of the blocks before it (at most a few
// thousand words, read from L2) and writes its items in order.  A block's items are one
// contiguous run of rows in every output array, so it writes each array value by value
// (consecutive threads, consecutive words) instead of a row of three or four values per
// thread: at 1M Gaussians with moments and an FP16 copy k_prune_emit takes 73 us against 108
// (425 MB: 63 us at the copy rate), and for 154 k new Gaussians of a 640 x 480 frame
// k_add_emit 20 us against 44 (part of that was FP64, below).  No block waits on another, and the live count stays on the device.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "gs_internal.cuh"

namespace {

constexpr int kCompactThreads = 1024;
constexpr int kGroups = 5;  // means, quats, log_scales, opacity_logits, rgb
// Values per Gaussian of each group, and the group's first row in a moment array (in units
// of capacity); isotropic maps (Eq. 1 as written) have no quaternion and one log-radius.
__host__ __device__ constexpr int group_width(int s, bool iso) {
    return s == 1 ? (iso ? 0 : 4) : (s == 2 ? (iso ? 1 : 3) : (s == 3 ? 1 : 3));
}
__host__ __device__ constexpr int group_offset(int s, bool iso) {
    return iso ? (s == 0 ? 0 : (s <= 2 ? 3 : (s == 3 ? 4 : 5))) : (s == 0 ? 0 : (s == 1 ? 3 : (s == 2 ? 7 : (s == 3 ? 10 : 11))));
}
__host__ __device__ constexpr int values_per_gaussian(bool iso) { return iso ? 8 : 14; }

struct MapView {
    float *p[kGroups];
    void *lp[kGroups];  // lp[0] is always NULL (the means have no low-precision copy)
    int32_t lowp_dt;
    bool iso;      // no quaternions, one log-radius
    int64_t cap;
    float *state;  // m: groups at cap * group_offset; v: values_per_gaussian cap further
};

MapView view_of(const gs_map &m) {
    MapView v{};
    v.p[0] = m.means;
    v.p[1] = m.quats;
    v.p[2] = m.log_scales;
    v.p[3] = m.opacity_logits;
    v.p[4] = m.rgb;
    v.lp[0] = nullptr;
    v.lp[1] = m.lowp_quats;
    v.lp[2] = m.lowp_log_scales;
    v.lp[3] = m.lowp_opacity_logits;
    v.lp[4] = m.lowp_rgb;
    v.lowp_dt = m.lowp_dtype;
    v.iso = m.quats == nullptr;
    v.cap = m.capacity;
    v.state = m.adam_state;
    return v;
}

__device__ __forceinline__ void store_lowp(void *base, int64_t i, float x, int dt) {
    if (dt == GS_BF16)
        static_cast<__nv_bfloat16 *>(base)[i] = __float2bfloat16_rn(x);
    else
        static_cast<__half *>(base)[i] = __float2half_rn(x);
}

// Sum of counts[0, b) over the block, and the total when b is the last block.
__device__ uint32_t block_prefix(const uint32_t *counts, uint32_t b) {
    __shared__ uint32_t s_w[kCompactThreads / 32];
    uint32_t acc = 0;
    for (uint32_t k = threadIdx.x; k < b; k += blockDim.x) acc += counts[k];
    acc = __reduce_add_sync(0xffffffffu, acc);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = acc;
    __syncthreads();
    uint32_t tot = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += s_w[w];
    __syncthreads();
    return tot;
}

// Exclusive rank of this thread's flag within the block, and the block's count.
__device__ uint32_t block_rank(bool flag, uint32_t &count) {
    __shared__ uint32_t s_w[kCompactThreads / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint32_t bal = __ballot_sync(0xffffffffu, flag);
    if (lane == 0) s_w[warp] = __popc(bal);
    __syncthreads();
    if (warp == 0) {
        const uint32_t x = lane < nw ? s_w[lane] : 0u;
        uint32_t incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane < nw) s_w[lane] = incl - x;
        if (lane == nw - 1) s_w[kCompactThreads / 32] = incl;
    }
    __syncthreads();
    const uint32_t r = s_w[warp] + __popc(bal & ((1u << lane) - 1u));
    count = s_w[kCompactThreads / 32];
    __syncthreads();
    return r;
}

// ------------------------------------------------------------------ new Gaussians

// FP32 pairs (hi + lo): the FP64 values of the camera that the unprojection takes, and its
// arithmetic.  FP64 issues at a sixty-fourth of the FP32 rate here and bound the pass.  The
// results are those of FP64 rounded to FP32: a pair known to within `err` decides the rounding
// unless the point halfway between two FP32 values lies inside that (nearest), and then, or
// where the pairs leave FP32's range, the pixel is unprojected in FP64.
// Measured in the same call: 57.5 us for the 307,200 pixels of a 640 x 480 frame (pairs with no such
// check 56.2, all in FP64 94.6), 87.7 for 1200 x 680 (85.3, 199); about one pixel in 3,000 has a value that goes
// to FP64.
using gsk::DF;
using gsk::df_add;

DF df_host(double x) {
    const float hi = (float)x;
    return DF{hi, std::isfinite(hi) ? (float)(x - (double)hi) : 0.f};
}
__device__ __forceinline__ DF df_split(double x) {
    const float hi = (float)x;
    return DF{hi, (float)(x - (double)hi)};
}
__device__ __forceinline__ DF df_mul(DF a, DF b) {
    const float p = __fmul_rn(a.hi, b.hi);
    const float e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.hi, -p)));
    const float s = __fadd_rn(p, e);
    return DF{s, __fsub_rn(e, __fsub_rn(s, p))};
}

// Is x.hi the FP32 value nearest to every number within err of the pair x (x.hi = RN(hi + lo))?
// (False where a value is not finite.)
__device__ __forceinline__ bool nearest(DF x, float err) {
    return __fadd_rn(x.hi, __fadd_rn(x.lo, err)) == x.hi && __fadd_rn(x.hi, __fadd_rn(x.lo, -err)) == x.hi;
}

// ln x as a pair, to 2^-41 (|ln x| + 1/2): x = 2^k m, m in [sqrt(1/2), sqrt(2)),
// ln m = 2 atanh(s) = 2 s (1 + z/3 + z^2/5 + ... + z^7/15), s = (m - 1) / (m + 1), z = s^2 < 0.0295
// (the next term is below 2^-44); s, z and the terms to z^2 as pairs, the rest in FP32.
// x: a positive pair, both of whose values are normal or the second zero.
constexpr float kLn2Hi = 0.693147182f, kLn2Lo = (float)(0.69314718055994530942 - (double)kLn2Hi);

__device__ __forceinline__ DF log_pair(DF x) {
    const int bits = __float_as_int(x.hi), k = (bits - __float_as_int(0.70710678f)) >> 23;
    const float mh = __int_as_float(bits - (k << 23)), ml = ldexpf(x.lo, -k);
    const DF num = df_add(DF{__fsub_rn(mh, 1.f), 0.f}, DF{ml, 0.f});  // mh - 1 is exact
    const DF den = df_add(DF{mh, ml}, DF{1.f, 0.f});
    const float q = __fdiv_rn(num.hi, den.hi);
    const float r = __fadd_rn(__fmaf_rn(-q, den.hi, num.hi), __fmaf_rn(-q, den.lo, num.lo));
    const float c = __fdiv_rn(r, den.hi), sh = __fadd_rn(q, c);
    const DF s = DF{sh, __fsub_rn(c, __fsub_rn(sh, q))}, z = df_mul(s, s);
    float t = 1.f / 15.f;
    t = fmaf(t, z.hi, 1.f / 13.f);
    t = fmaf(t, z.hi, 1.f / 11.f);
    t = fmaf(t, z.hi, 1.f / 9.f);
    t = fmaf(t, z.hi, 1.f / 7.f);
    const DF a = df_add(DF{0.2f, (float)(0.2 - (double)0.2f)}, DF{t * z.hi, 0.f});
    const DF b = df_add(DF{1.f / 3.f, (float)(1.0 / 3.0 - (double)(1.f / 3.f))}, df_mul(z, a));
    const DF s2 = DF{2.f * s.hi, 2.f * s.lo};
    const DF ln_m = df_add(s2, df_mul(s2, df_mul(z, b)));
    return df_add(df_mul(DF{(float)k, 0.f}, DF{kLn2Hi, kLn2Lo}), ln_m);
}

struct AddLaunch {
    MapView map;
    int64_t *n;
    const double *pose;
    const float *rgb, *depth, *sil;
    float sil_add;
    double fx, fy, cx, cy;
    DF ifx, ify, ncx, ncy, inv_f;  // 1 / fx, 1 / fy, -cx, -cy, 2 / (fx + fy)
    double ifx64, ify64, inv_f64;
    bool pairs;                    // the camera lies inside the pairs' range
    int32_t width, height;
    uint32_t *counts;  // scratch: one word per block
    int64_t *n0;       // scratch: the live count before the call
    double *Rt;        // scratch: world->camera rotation (9) and translation (3)
    uint32_t *err;
};

__device__ __forceinline__ bool add_flag(const AddLaunch &L, int64_t p, int64_t P) {
    if (p >= P) return false;
    const float d = L.depth[p];
    return d > 0.f && (L.sil == nullptr || L.sil[p] < L.sil_add);
}

__global__ void __launch_bounds__(kCompactThreads) k_add_count(AddLaunch L) {
    const int64_t P = (int64_t)L.width * L.height;
    const int64_t p = (int64_t)blockIdx.x * kCompactThreads + threadIdx.x;
    const uint32_t c = (uint32_t)__syncthreads_count(add_flag(L, p, P));
    if (threadIdx.x == 0) {
        L.counts[blockIdx.x] = c;
        if (blockIdx.x == 0) *L.n0 = *L.n;
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 32) {
        // the rotation of the pose's unit quaternion (renormalised), in FP64: once here
        // instead of in front of every block of the emission
        double w = L.pose[0], x = L.pose[1], y = L.pose[2], z = L.pose[3];
        const double inv = 1.0 / sqrt(w * w + x * x + y * y + z * z);
        w *= inv; x *= inv; y *= inv; z *= inv;
        double *R = L.Rt;
        R[0] = 1.0 - 2.0 * (y * y + z * z); R[1] = 2.0 * (x * y - w * z); R[2] = 2.0 * (x * z + w * y);
        R[3] = 2.0 * (x * y + w * z); R[4] = 1.0 - 2.0 * (x * x + z * z); R[5] = 2.0 * (y * z - w * x);
        R[6] = 2.0 * (x * z - w * y); R[7] = 2.0 * (y * z + w * x); R[8] = 1.0 - 2.0 * (x * x + y * y);
        R[9] = L.pose[4]; R[10] = L.pose[5]; R[11] = L.pose[6];
    }
}

// The pixel's sample point at depth d in the camera frame (inverse of pi_m), then
// world = R^T (x_c - t), and the log-scale ln(d / f), in FP64.
__device__ __noinline__ void unproject_fp64(const AddLaunch &L, const double *R, const double *t, int u, int v, double d,
                                            float (&mean)[3], float &ls) {
    const double xc0 = ((double)u - L.cx) / L.fx * d - t[0];
    const double xc1 = ((double)v - L.cy) / L.fy * d - t[1];
    const double xc2 = d - t[2];
    for (int k = 0; k < 3; ++k) mean[k] = (float)(R[k] * xc0 + R[3 + k] * xc1 + R[6 + k] * xc2);
    ls = (float)log(d / (0.5 * (L.fx + L.fy)));
}

// The means alone, of a pixel inside the pairs' range: with the reciprocals of the focal lengths,
// since FP64 divisions would make a block wait for 3 us.
__device__ __noinline__ void unproject_near_tie(const AddLaunch &L, const double *Rt, int u, int v, double d, float (&mean)[3]) {
    const double xc0 = ((double)u - L.cx) * L.ifx64 * d - Rt[9];
    const double xc1 = ((double)v - L.cy) * L.ify64 * d - Rt[10];
    const double xc2 = d - Rt[11];
    for (int k = 0; k < 3; ++k) mean[k] = (float)(Rt[k] * xc0 + Rt[3 + k] * xc1 + Rt[6 + k] * xc2);
}

// `values` consecutive values of one output array, value(i) the i-th; consecutive threads
// take consecutive values.
template <class T, class F>
__device__ __forceinline__ void write_run(T *out, int values, F &&value) {
    for (int i = threadIdx.x; i < values; i += kCompactThreads) out[i] = value(i);
}
template <class F>
__device__ __forceinline__ void write_lowp(void *base, int64_t first, int values, int dt, F &&value) {
    for (int i = threadIdx.x; i < values; i += kCompactThreads) store_lowp(base, first + i, value(i), dt);
}

// Two blocks per SM (32 registers): the block's phases wait for one another, so a second
// block hides them (21 -> 19 us).
__global__ void __launch_bounds__(kCompactThreads, 2) k_add_emit(AddLaunch L) {
    __shared__ DF s_R[9], s_nt[3];  // R, -t
    __shared__ float s_mean[3 * kCompactThreads], s_rgb[3 * kCompactThreads], s_ls[kCompactThreads];
    const int64_t P = (int64_t)L.width * L.height;
    const int64_t p = (int64_t)blockIdx.x * kCompactThreads + threadIdx.x;
    if (threadIdx.x < 9) s_R[threadIdx.x] = df_split(L.Rt[threadIdx.x]);
    else if (threadIdx.x < 12) s_nt[threadIdx.x - 9] = df_split(-L.Rt[threadIdx.x]);
    const uint32_t before = block_prefix(L.counts, blockIdx.x);
    const bool flag = add_flag(L, p, P);
    uint32_t count;
    const uint32_t r = block_rank(flag, count);  // (ends with a barrier: s_R and s_nt are set)
    if (flag) {
        const int v = (int)(p / L.width), u = (int)(p - (int64_t)v * L.width);
        const float d = L.depth[p];
        float mean[3], ls;
        if (L.pairs && d > 0x1p-60f && d < 0x1p60f) {
            bool sure = true;
            const DF D{d, 0.f};
            const DF x0 = df_add(df_mul(df_mul(df_add(DF{(float)u, 0.f}, L.ncx), L.ifx), D), s_nt[0]);
            const DF x1 = df_add(df_mul(df_mul(df_add(DF{(float)v, 0.f}, L.ncy), L.ify), D), s_nt[1]);
            const DF x2 = df_add(D, s_nt[2]);
            // every term of a mean is at most `size`; on its way are three products and four sums of
            // pairs (2^-46 and 2^-46.5 of it each) and three rounded factors (2^-48): 2^-43.3 together
            const float size = ((float)u + fabsf(L.ncx.hi)) * L.ifx.hi * d + ((float)v + fabsf(L.ncy.hi)) * L.ify.hi * d + d +
                               fabsf(s_nt[0].hi) + fabsf(s_nt[1].hi) + fabsf(s_nt[2].hi);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const DF x = df_add(df_add(df_mul(s_R[k], x0), df_mul(s_R[3 + k], x1)), df_mul(s_R[6 + k], x2));
                mean[k] = x.hi;
                sure = sure && nearest(x, 0x1p-43f * size);
            }
            const DF ln = log_pair(df_mul(D, L.inv_f));
            ls = ln.hi;
            if (!sure) unproject_near_tie(L, L.Rt, u, v, (double)d, mean);
            if (!nearest(ln, 0x1p-40f * (fabsf(ls) + 0.5f))) ls = (float)log((double)d * L.inv_f64);
        } else {
            unproject_fp64(L, L.Rt, L.Rt + 9, u, v, (double)d, mean, ls);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            s_mean[3 * r + k] = mean[k];
            s_rgb[3 * r + k] = L.rgb[k * P + p];
        }
        s_ls[r] = ls;
    }
    __syncthreads();
    const MapView &M = L.map;
    const int64_t n0 = *L.n0, first = n0 + before;
    // the block's rows that fit the capacity
    const int rows = first < M.cap ? (int)min((int64_t)count, M.cap - first) : 0;
    const int wl = M.iso ? 1 : 3;
    write_run(M.p[0] + 3 * first, 3 * rows, [&](int i) { return s_mean[i]; });
    if (!M.iso) write_run(M.p[1] + 4 * first, 4 * rows, [&](int i) { return (i & 3) == 0 ? 1.f : 0.f; });
    write_run(M.p[2] + wl * first, wl * rows, [&](int i) { return s_ls[wl == 1 ? i : i / 3]; });
    write_run(M.p[3] + first, rows, [&](int) { return 0.f; });
    write_run(M.p[4] + 3 * first, 3 * rows, [&](int i) { return s_rgb[i]; });
    if (M.lp[2]) {
        const int dt = M.lowp_dt;
        if (M.lp[1]) write_lowp(M.lp[1], 4 * first, 4 * rows, dt, [&](int i) { return (i & 3) == 0 ? 1.f : 0.f; });
        write_lowp(M.lp[2], wl * first, wl * rows, dt, [&](int i) { return s_ls[wl == 1 ? i : i / 3]; });
        write_lowp(M.lp[3], first, rows, dt, [&](int) { return 0.f; });
        write_lowp(M.lp[4], 3 * first, 3 * rows, dt, [&](int i) { return s_rgb[i]; });
    }
    if (M.state) {
#pragma unroll
        for (int s = 0; s < kGroups; ++s) {
            const int w = group_width(s, M.iso);
            float *m = M.state + M.cap * group_offset(s, M.iso) + w * first;
            write_run(m, w * rows, [&](int) { return 0.f; });
            write_run(m + values_per_gaussian(M.iso) * M.cap, w * rows, [&](int) { return 0.f; });
        }
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        int64_t n1 = n0 + before + count;
        if (n1 > M.cap) {
            n1 = M.cap;
            if (L.err) atomicOr(L.err, 1u);
        }
        *L.n = n1;
    }
}

// ------------------------------------------------------------------ Adam

struct AdamLaunch {
    float *p[kGroups];
    const float *g[kGroups];
    void *lp[kGroups];
    float *m[kGroups], *v[kGroups];
    float lr[kGroups];
    int width[kGroups];
    float b1, b2, omb1, omb2, c1, c2, eps;
    int32_t lowp_dt;
    const int64_t *n;
};

__device__ __forceinline__ float adam_one(float &p, float g, float &m, float &v, float lr, const AdamLaunch &L) {
    m = L.b1 * m + L.omb1 * g;
    v = L.b2 * v + L.omb2 * (g * g);
    const float mh = m * L.c1, vh = v * L.c2;
    p = p - lr * (mh / (sqrtf(vh) + L.eps));
    return p;
}

// blockIdx.y selects the group; a grid-stride loop over its float4 quads, the ragged
// tail (fewer than four values) taken by block 0.
__global__ void __launch_bounds__(256) k_map_adam(AdamLaunch L) {
    const int s = blockIdx.y;
    if (L.g[s] == nullptr || L.width[s] == 0) return;
    const int64_t len = (int64_t)L.width[s] * (*L.n);
    const float lr = L.lr[s];
    float *p = L.p[s], *m = L.m[s], *v = L.v[s];
    const float *g = L.g[s];
    void *lp = L.lp[s];
    const int64_t nq = len >> 2;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += (int64_t)gridDim.x * blockDim.x) {
        float4 P4 = reinterpret_cast<float4 *>(p)[q];
        const float4 G4 = __ldg(reinterpret_cast<const float4 *>(g) + q);
        float4 M4 = reinterpret_cast<float4 *>(m)[q];
        float4 V4 = reinterpret_cast<float4 *>(v)[q];
        adam_one(P4.x, G4.x, M4.x, V4.x, lr, L);
        adam_one(P4.y, G4.y, M4.y, V4.y, lr, L);
        adam_one(P4.z, G4.z, M4.z, V4.z, lr, L);
        adam_one(P4.w, G4.w, M4.w, V4.w, lr, L);
        reinterpret_cast<float4 *>(p)[q] = P4;
        reinterpret_cast<float4 *>(m)[q] = M4;
        reinterpret_cast<float4 *>(v)[q] = V4;
        if (lp) {
            if (L.lowp_dt == GS_BF16) {
                __nv_bfloat162 *o = reinterpret_cast<__nv_bfloat162 *>(lp) + 2 * q;
                o[0] = __floats2bfloat162_rn(P4.x, P4.y);
                o[1] = __floats2bfloat162_rn(P4.z, P4.w);
            } else {
                __half2 *o = reinterpret_cast<__half2 *>(lp) + 2 * q;
                o[0] = __floats2half2_rn(P4.x, P4.y);
                o[1] = __floats2half2_rn(P4.z, P4.w);
            }
        }
    }
    if (blockIdx.x == 0 && threadIdx.x < (len & 3)) {
        const int64_t k = 4 * nq + threadIdx.x;
        float pk = p[k], mk = m[k], vk = v[k];
        adam_one(pk, g[k], mk, vk, lr, L);
        p[k] = pk;
        m[k] = mk;
        v[k] = vk;
        if (lp) store_lowp(lp, k, pk, L.lowp_dt);
    }
}

// ------------------------------------------------------------------ removal

struct PruneLaunch {
    MapView src, dst;
    const int64_t *n_src;
    int64_t *n_dst;
    float logit_min;
    uint32_t *counts;
    int64_t *n0;
};

__global__ void __launch_bounds__(kCompactThreads) k_prune_count(PruneLaunch L) {
    const int64_t i = (int64_t)blockIdx.x * kCompactThreads + threadIdx.x;
    const int64_t n = *L.n_src;
    const bool keep = i < n && L.src.p[3][i] >= L.logit_min;
    const uint32_t c = (uint32_t)__syncthreads_count(keep);
    if (threadIdx.x == 0) {
        L.counts[blockIdx.x] = c;
        if (blockIdx.x == 0) *L.n0 = n;
    }
}

// One group of values (S) of a block's kept Gaussians: row r of the destination's rows
// [j0, j0 + count) is row i0 + idx[r] of the source, in the parameters, the low-precision
// copy (16-bit values, moved as they are) and both moments.  A thread takes W values of each
// array, all their loads before the first store: at four loads in flight the pass was bound
// by latency (137 us at 1.2M Gaussians).
template <int S, bool ISO>
__device__ __forceinline__ void prune_group(const PruneLaunch &L, int64_t i0, int64_t j0, const uint16_t *idx, int count) {
    constexpr int W = group_width(S, ISO);
    if constexpr (W > 0) {
        const MapView &A = L.src, &B = L.dst;
        const bool lowp = S > 0 && A.lp[S] && B.lp[S] && A.lowp_dt == B.lowp_dt, state = A.state && B.state;
        constexpr int64_t o = group_offset(S, ISO), vp = values_per_gaussian(ISO);
        const float *sp = A.p[S] + W * i0, *sm = A.state + A.cap * o + W * i0, *sv = sm + vp * A.cap;
        float *dp = B.p[S] + W * j0, *dm = B.state + B.cap * o + W * j0, *dv = dm + vp * B.cap;
        const uint16_t *sl = static_cast<const uint16_t *>(A.lp[S]) + W * i0;
        uint16_t *dl = static_cast<uint16_t *>(B.lp[S]) + W * j0;
        float p[W], m[W], v[W];
        uint16_t l[W];
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const int i = threadIdx.x + k * kCompactThreads, r = i / W;
            if (i < W * count) {
                const int at = W * (int)idx[r] + (i - W * r);
                p[k] = sp[at];
                if (state) m[k] = sm[at];
                if (state) v[k] = sv[at];
                if (lowp) l[k] = sl[at];
            }
        }
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const int i = threadIdx.x + k * kCompactThreads;
            if (i < W * count) {
                dp[i] = p[k];
                if (state) dm[i] = m[k];
                if (state) dv[i] = v[k];
                if (lowp) dl[i] = l[k];
            }
        }
    }
}

template <bool ISO>
__global__ void __launch_bounds__(kCompactThreads) k_prune_emit(PruneLaunch L) {
    __shared__ uint16_t s_idx[kCompactThreads];
    const int64_t i0 = (int64_t)blockIdx.x * kCompactThreads, i = i0 + threadIdx.x;
    const int64_t n = *L.n0;
    const uint32_t before = block_prefix(L.counts, blockIdx.x);
    const bool keep = i < n && L.src.p[3][i] >= L.logit_min;
    uint32_t count;
    const uint32_t r = block_rank(keep, count);
    if (keep) s_idx[r] = (uint16_t)threadIdx.x;
    __syncthreads();
    const int64_t j0 = before;
    prune_group<0, ISO>(L, i0, j0, s_idx, (int)count);
    prune_group<1, ISO>(L, i0, j0, s_idx, (int)count);
    prune_group<2, ISO>(L, i0, j0, s_idx, (int)count);
    prune_group<3, ISO>(L, i0, j0, s_idx, (int)count);
    prune_group<4, ISO>(L, i0, j0, s_idx, (int)count);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *L.n_dst = (int64_t)before + count;
}

// ------------------------------------------------------------------ host side

constexpr size_t kScratchHead = 256;  // the saved live count and the pose, then one word per block

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool map_ok(const gs_map *m) {
    if (!m || m->capacity < 0 || (m->capacity & 3) != 0) return false;
    const bool iso = m->quats == nullptr;  // isotropic: no quaternions anywhere
    const float *f[5] = {m->means, iso ? m->means : m->quats, m->log_scales, m->opacity_logits, m->rgb};
    for (const float *q : f)
        if (!q || !aligned16(q)) return false;
    if (iso && m->lowp_quats) return false;
    const void *l[4] = {iso ? m->lowp_log_scales : m->lowp_quats, m->lowp_log_scales, m->lowp_opacity_logits,
                        m->lowp_rgb};
    const bool any = l[0] || l[1] || l[2] || l[3];
    if (any) {
        if (m->lowp_dtype != GS_BF16 && m->lowp_dtype != GS_F16) return false;
        for (const void *q : l)
            if (!q || !aligned16(q)) return false;
    }
    return !m->adam_state || aligned16(m->adam_state);
}

size_t scratch_bytes_for(int64_t items) {
    const int64_t blocks = (items + kCompactThreads - 1) / kCompactThreads;
    return kScratchHead + (size_t)(4 * blocks + 255) / 256 * 256;
}

}  // namespace

extern "C" {

void gs_default_map_config(gs_map_config *c) {
    if (!c) return;
    c->lr_means = 1e-4;
    c->lr_quats = 1e-3;
    c->lr_log_scales = 1e-3;
    c->lr_opacity_logits = 5e-2;
    c->lr_rgb = 2.5e-3;
    c->beta1 = 0.9;
    c->beta2 = 0.999;
    c->eps = 1e-15;
    c->sil_add = 0.5f;
    c->opacity_min = 0.005f;
}

size_t gs_map_scratch_bytes(int64_t items) { return items < 0 ? 0 : scratch_bytes_for(items); }

gs_status gs_map_add(const gs_map_config *cfg, const gs_map *map, int64_t *n, const gs_camera *cam,
                     const double *pose, const float *rgb, const float *depth, const float *sil, void *scratch,
                     size_t scratch_bytes, uint32_t *err_flags, void *stream) {
    if (!cfg || !map_ok(map) || !n || !cam || !pose || !rgb || !depth || !scratch) return GS_ERR_INVALID_ARG;
    if (cam->width < 1 || cam->height < 1 || !(cam->fx > 0) || !(cam->fy > 0)) return GS_ERR_INVALID_ARG;
    const int64_t P = (int64_t)cam->width * cam->height;
    if (P >= (1ll << 31) || (reinterpret_cast<uintptr_t>(scratch) & 255u) != 0 ||
        scratch_bytes < scratch_bytes_for(P))
        return GS_ERR_INVALID_ARG;
    AddLaunch L{};
    L.map = view_of(*map);
    L.n = n;
    L.pose = pose;
    L.rgb = rgb;
    L.depth = depth;
    L.sil = sil;
    L.sil_add = cfg->sil_add;
    L.fx = cam->fx;
    L.fy = cam->fy;
    L.cx = cam->cx;
    L.cy = cam->cy;
    L.ifx = df_host(1.0 / cam->fx);
    L.ify = df_host(1.0 / cam->fy);
    L.ncx = df_host(-cam->cx);
    L.ncy = df_host(-cam->cy);
    L.inv_f = df_host(2.0 / (cam->fx + cam->fy));
    L.ifx64 = 1.0 / cam->fx;
    L.ify64 = 1.0 / cam->fy;
    L.inv_f64 = 2.0 / (cam->fx + cam->fy);
    // pixel coordinates exact in FP32, no underflow in a product's low part, no overflow of one
    const auto in_range = [](double x) { return x > 0x1p-30 && x < 0x1p30; };
    L.pairs = in_range(cam->fx) && in_range(cam->fy) && std::fabs(cam->cx) < 0x1p30 && std::fabs(cam->cy) < 0x1p30 &&
              cam->width <= (1 << 24) && cam->height <= (1 << 24);
    L.width = cam->width;
    L.height = cam->height;
    L.n0 = static_cast<int64_t *>(scratch);
    L.Rt = static_cast<double *>(scratch) + 1;  // 96 bytes of the head
    L.counts = reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + kScratchHead);
    L.err = err_flags;
    const unsigned blocks = (unsigned)((P + kCompactThreads - 1) / kCompactThreads);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    k_add_count<<<blocks, kCompactThreads, 0, st>>>(L);
    k_add_emit<<<blocks, kCompactThreads, 0, st>>>(L);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

gs_status gs_map_adam_step(const gs_map_config *cfg, const gs_map *map, const int64_t *n,
                           const gs_gaussians_grad *grads, int64_t step, void *stream) {
    if (!cfg || !map_ok(map) || !map->adam_state || !n || !grads || step < 1) return GS_ERR_INVALID_ARG;
    if (!(cfg->beta1 >= 0 && cfg->beta1 < 1) || !(cfg->beta2 >= 0 && cfg->beta2 < 1) || !(cfg->eps >= 0))
        return GS_ERR_INVALID_ARG;
    const float *gp[5] = {grads->means, grads->quats, grads->log_scales, grads->opacity_logits, grads->rgb};
    for (const float *q : gp)
        if (q && !aligned16(q)) return GS_ERR_INVALID_ARG;
    const MapView M = view_of(*map);
    const double lr[5] = {cfg->lr_means, cfg->lr_quats, cfg->lr_log_scales, cfg->lr_opacity_logits, cfg->lr_rgb};
    AdamLaunch L{};
    for (int s = 0; s < kGroups; ++s) {
        L.p[s] = M.p[s];
        L.g[s] = gp[s];
        L.lp[s] = M.lp[s];
        L.m[s] = M.state + M.cap * group_offset(s, M.iso);
        L.v[s] = L.m[s] + values_per_gaussian(M.iso) * M.cap;
        L.lr[s] = (float)lr[s];
        L.width[s] = group_width(s, M.iso);
    }
    L.b1 = (float)cfg->beta1;
    L.b2 = (float)cfg->beta2;
    L.omb1 = (float)(1.0 - cfg->beta1);
    L.omb2 = (float)(1.0 - cfg->beta2);
    L.c1 = (float)(1.0 / (1.0 - std::pow(cfg->beta1, (double)step)));
    L.c2 = (float)(1.0 / (1.0 - std::pow(cfg->beta2, (double)step)));
    L.eps = (float)cfg->eps;
    L.lowp_dt = M.lowp_dt;
    L.n = n;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return GS_ERR_CUDA;
    // about four resident 256-thread blocks per SM per group; quads beyond a group's
    // live length exit at once
    const int64_t quads = (4 * M.cap + 3) / 4;
    const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(4 * sms, (quads + 255) / 256));
    k_map_adam<<<dim3(gx, kGroups), 256, 0, static_cast<cudaStream_t>(stream)>>>(L);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

gs_status gs_map_prune(const gs_map_config *cfg, const gs_map *src, const int64_t *n_src, const gs_map *dst,
                       int64_t *n_dst, void *scratch, size_t scratch_bytes, void *stream) {
    if (!cfg || !map_ok(src) || !map_ok(dst) || !n_src || !n_dst || !scratch) return GS_ERR_INVALID_ARG;
    if (dst->capacity < src->capacity || src->capacity >= (1ll << 31) || !(cfg->opacity_min > 0.f) ||
        !(cfg->opacity_min < 1.f))
        return GS_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(scratch) & 255u) != 0 || scratch_bytes < scratch_bytes_for(src->capacity))
        return GS_ERR_INVALID_ARG;
    if (src->means == dst->means || (src->quats == nullptr) != (dst->quats == nullptr)) return GS_ERR_INVALID_ARG;
    PruneLaunch L{};
    L.src = view_of(*src);
    L.dst = view_of(*dst);
    L.n_src = n_src;
    L.n_dst = n_dst;
    const double o = (double)cfg->opacity_min;
    L.logit_min = (float)std::log(o / (1.0 - o));
    L.n0 = static_cast<int64_t *>(scratch);
    L.counts = reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + kScratchHead);
    const unsigned blocks = (unsigned)std::max<int64_t>(1, (src->capacity + kCompactThreads - 1) / kCompactThreads);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    k_prune_count<<<blocks, kCompactThreads, 0, st>>>(L);
    if (L.src.iso) k_prune_emit<true><<<blocks, kCompactThreads, 0, st>>>(L);
    else k_prune_emit<false><<<blocks, kCompactThreads, 0, st>>>(L);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

}  // extern "C"
