// msssim.cu -- multi-scale structural similarity (Wang, Simoncelli and Bovik, 2003) of a
// rendered colour image against its observation, the image-quality measure of Sec. IV.
//
// Three launches.  k_pyramid makes the four coarser scales by 2 x 2 average pooling.
// k_ssim_terms takes the local statistics of every scale and channel at once: a window
// position's moments under the 11 x 11 Gaussian window (sigma 1.5) are centred on the window's
// middle pixel so that the variances do not cancel in FP32.  Every position has its own centre,
// so they are taken position by position: 121 taps of nine FP32 operations, and that
// arithmetic bounds the kernel.  (Row moments about a pixel of the row, shifted to the
// window's middle while the rows are added, would be separable; not built.)  A thread takes two positions eight rows apart in
// the two lanes of FP32 pair instructions, from a shared tile that stores the two rows
// interleaved.  The term itself, (2 cov + C2) / (var + var + C2), and its sum are double-float
// on the FP32 pipes (about 46 bits): in FP64 they took longer than the window.
// k_ssim_finish sums the blocks' partials in a fixed order and combines the scales with the
// published exponents.  At 640 x 480: 5 + 58 + 14 us, the first and the last partly
// overlapped (the window kernel keeps the FMA pipes 76 % busy); fifteen launches with the
// moments read from L1 and the terms in FP64 took 230 us, 56 of them one thread's powers.
#include <algorithm>
#include <cmath>

#include "gs_internal.cuh"

namespace {

using gsk::DF;
using gsk::df_add;
using gsk::df_shfl_xor;

constexpr int kWin = 11;
constexpr int kScales = 5;
constexpr int kSsimThreads = 256;
constexpr int kTileW = 32, kHalfH = 8, kTileH = 2 * kHalfH;  // window positions per block
constexpr int kTapW = kTileW + kWin - 1, kTapH = kHalfH + kWin - 1;
static_assert(kTileW * kHalfH == kSsimThreads, "one thread per pair of positions");
constexpr double kC1 = 0.01 * 0.01, kC2 = 0.03 * 0.03;

struct Window {
    float g[kWin];  // the normalised 1-D Gaussian (sigma 1.5); the 2-D window is its outer product
};
struct Weights {
    double b[kScales];  // published scale exponents
};

struct Level {
    const float *x, *y;  // 3 planes each, w x h
    int w, h;
    int first, tiles_x;  // the scale's first block per channel and its blocks per row
};
struct Pyramid {
    Level l[kScales];
    int blocks;  // blocks per channel over all scales
};

// 2 x 2 average pooling of both images' three planes through all scales (odd last rows /
// columns dropped at each): a block makes 16 x 16 pixels of the second scale and what
// follows from them.  blockIdx.x: such blocks, tiles_x per row; blockIdx.y = image * 3 + channel.
__global__ void __launch_bounds__(256) k_pyramid(Pyramid P, int tiles_x) {
    gsk::griddep_launch_dependents();  // the first scale's terms need no pyramid
    __shared__ float s[2][16][16];
    const int ch = blockIdx.y % 3, second = blockIdx.y / 3;
    const int bx = blockIdx.x % tiles_x, by = blockIdx.x / tiles_x;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    int cur = 0;
    for (int j = 1; j < kScales; ++j) {
        const int n = 16 >> (j - 1);  // pixels of scale j per block and axis
        const Level &D = P.l[j];
        const int px = bx * n + tx, py = by * n + ty;
        if (tx < n && ty < n && px < D.w && py < D.h) {
            float a, b, c, d;  // (0, 0), (1, 0), (0, 1), (1, 1) as (row, column)
            if (j == 1) {
                const Level &S = P.l[0];
                const float *in = (second ? S.y : S.x) + (int64_t)ch * S.w * S.h + (int64_t)(2 * py) * S.w + 2 * px;
                a = in[0];
                b = in[S.w];
                c = in[1];
                d = in[S.w + 1];
            } else {
                a = s[cur][2 * ty][2 * tx];
                b = s[cur][2 * ty + 1][2 * tx];
                c = s[cur][2 * ty][2 * tx + 1];
                d = s[cur][2 * ty + 1][2 * tx + 1];
            }
            const float v = 0.25f * ((a + b) + (c + d));
            const_cast<float *>(second ? D.y : D.x)[(int64_t)ch * D.w * D.h + (int64_t)py * D.w + px] = v;
            s[cur ^ 1][ty][tx] = v;
        }
        cur ^= 1;
        __syncthreads();
    }
}

// a b - c exactly rounded to a pair: the product's rounding error by an FMA, the
// difference's by TwoSum.
__device__ __forceinline__ DF df_minus_product(float c, float a, float b) {
    const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p);
    const float s = __fsub_rn(c, p), v = __fsub_rn(s, c);
    const float r = __fsub_rn(__fsub_rn(c, __fsub_rn(s, v)), __fadd_rn(p, v));
    return df_add(DF{s, r}, DF{-e, 0.f});
}

__device__ __forceinline__ DF df_of(double x) {
    const float hi = (float)x;
    return DF{hi, isfinite(hi) ? (float)(x - (double)hi) : 0.f};
}

// a / b to about 46 bits: the FP32 quotient and the correction from its exact remainder.
__device__ __forceinline__ DF df_div(DF a, DF b) {
    const float q = __fdiv_rn(a.hi, b.hi);
    const float r = __fadd_rn(__fmaf_rn(-q, b.hi, a.hi), __fmaf_rn(-q, b.lo, a.lo));
    const float c = __fdividef(r, b.hi), s = __fadd_rn(q, c);
    return DF{s, __fsub_rn(c, __fsub_rn(s, q))};
}

// Contrast-structure term of a position from its shifted moments (variances and covariance
// do not depend on the shift).
__device__ __forceinline__ DF cs_term(float sx, float sy, float sxx, float syy, float sxy) {
    if (!(sxx < 0x1p100f && syy < 0x1p100f)) {  // not finite, or products beyond FP32
        const double vx = (double)sxx - (double)sx * sx, vy = (double)syy - (double)sy * sy;
        const double cxy = (double)sxy - (double)sx * sy;
        return df_of((2.0 * cxy + kC2) / (vx + vy + kC2));
    }
    const DF c2 = DF{(float)kC2, (float)(kC2 - (double)(float)kC2)};
    const DF cov = df_minus_product(sxy, sx, sy);
    const DF num = df_add(DF{2.f * cov.hi, 2.f * cov.lo}, c2);
    const DF den = df_add(df_add(df_minus_product(sxx, sx, sx), df_minus_product(syy, sy, sy)), c2);
    return df_div(num, den);
}

// Terms of every scale: blockIdx.x = block over the scales, blockIdx.y = channel;
// partials[(channel * blocks + block) * 2 + {0, 1}] = sums of l (coarsest scale only: the
// others' are not used) and cs over the block's window positions.
__global__ void __launch_bounds__(kSsimThreads) k_ssim_terms(Pyramid P, Window W, double *partials) {
    __shared__ float2 sx2[kTapH][kTapW], sy2[kTapH][kTapW];  // rows r and r + kHalfH of the tile
    const int ch = blockIdx.y, block = blockIdx.x;
    int j = kScales - 1;
    while (j > 0 && block < P.l[j].first) --j;
    // the first scale reads the caller's images only: its blocks overlap the pyramid (which
    // began after everything before it in the stream had ended)
    if (j > 0) gsk::griddep_wait();
    gsk::griddep_launch_dependents();
    const Level L = P.l[j];
    const int ow = L.w - kWin + 1, oh = L.h - kWin + 1;
    const int t = block - L.first, bx = t % L.tiles_x * kTileW, by = t / L.tiles_x * kTileH;
    const float *X = L.x + (int64_t)ch * L.w * L.h, *Y = L.y + (int64_t)ch * L.w * L.h;
    for (int k = threadIdx.x; k < kTapH * kTapW; k += kSsimThreads) {
        const int r = k / kTapW, c = k - r * kTapW;
        const int px = min(bx + c, L.w - 1);  // clamped pixels belong to no valid position
        const int64_t a = (int64_t)min(by + r, L.h - 1) * L.w + px, b = (int64_t)min(by + r + kHalfH, L.h - 1) * L.w + px;
        sx2[r][c] = make_float2(X[a], X[b]);
        sy2[r][c] = make_float2(Y[a], Y[b]);
    }
    __syncthreads();
    const int tx = threadIdx.x % kTileW, ty = threadIdx.x / kTileW;
    const float2 mx = sx2[ty + kWin / 2][tx + kWin / 2], my = sy2[ty + kWin / 2][tx + kWin / 2];
    const float2 ncx = make_float2(-mx.x, -mx.y), ncy = make_float2(-my.x, -my.y);
    const float2 zero = make_float2(0.f, 0.f);
    float2 sx = zero, sy = zero, sxx = zero, syy = zero, sxy = zero;
#pragma unroll 1
    for (int i = 0; i < kWin; ++i) {
        float2 rx = zero, ry = zero, rxx = zero, ryy = zero, rxy = zero;
#pragma unroll
        for (int q = 0; q < kWin; ++q) {
            const float2 w = make_float2(W.g[q], W.g[q]);
            const float2 a = __fadd2_rn(sx2[ty + i][tx + q], ncx), b = __fadd2_rn(sy2[ty + i][tx + q], ncy);
            const float2 wa = __fmul2_rn(w, a), wb = __fmul2_rn(w, b);
            rx = __ffma2_rn(w, a, rx);
            ry = __ffma2_rn(w, b, ry);
            rxx = __ffma2_rn(wa, a, rxx);
            ryy = __ffma2_rn(wb, b, ryy);
            rxy = __ffma2_rn(wa, b, rxy);
        }
        const float2 w = make_float2(W.g[i], W.g[i]);
        sx = __ffma2_rn(w, rx, sx);
        sy = __ffma2_rn(w, ry, sy);
        sxx = __ffma2_rn(w, rxx, sxx);
        syy = __ffma2_rn(w, ryy, syy);
        sxy = __ffma2_rn(w, rxy, sxy);
    }
    DF cs{0.f, 0.f};
    double l = 0.0;
    const bool in0 = bx + tx < ow && by + ty < oh, in1 = bx + tx < ow && by + ty + kHalfH < oh;
    if (in0) cs = cs_term(sx.x, sy.x, sxx.x, syy.x, sxy.x);
    if (in1) cs = df_add(cs, cs_term(sx.y, sy.y, sxx.y, syy.y, sxy.y));
    if (j == kScales - 1) {
        const auto lum = [](float cx, float cy, float ax, float ay) {
            const double ux = (double)cx + ax, uy = (double)cy + ay;
            return (2.0 * ux * uy + kC1) / (ux * ux + uy * uy + kC1);
        };
        if (in0) l += lum(mx.x, my.x, sx.x, sy.x);
        if (in1) l += lum(mx.y, my.y, sx.y, sy.y);
    }
    __shared__ double s[2][kSsimThreads / 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) cs = df_add(cs, df_shfl_xor(cs, off));
    if (j == kScales - 1)
        for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    if ((threadIdx.x & 31) == 0) {
        s[0][threadIdx.x >> 5] = l;
        s[1][threadIdx.x >> 5] = (double)cs.hi + (double)cs.lo;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double acc = 0.0;
        for (int w = 0; w < kSsimThreads / 32; ++w) acc += s[threadIdx.x][w];
        partials[((int64_t)ch * P.blocks + block) * 2 + threadIdx.x] = acc;
    }
}

// The means of the terms, their powers, and out[1 + ch] = l_5^b5 prod_j max(cs_j, 0)^bj per
// channel, out[0] = their mean.  One block: warp j * 3 + ch sums a scale's partials of a
// channel, then one warp takes all powers, a lane each (a warp-wide FP64 instruction
// occupies the SM's FP64 pipe for 16 cycles whatever its active lanes: 18 warps with one
// power each took 21 us).
constexpr int kFinishWarps = 3 * kScales;

__global__ void __launch_bounds__(32 * kFinishWarps) k_ssim_finish(Pyramid P, Weights B, const double *partials,
                                                                  double *out) {
    gsk::griddep_wait();
    __shared__ double s_mean[kFinishWarps + 3];  // contrast-structure by j * 3 + ch, then luminance by ch
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = warp / 3, ch = warp % 3;
    const bool coarsest = j == kScales - 1;
    {
        const Level &L = P.l[j];
        const int end = j + 1 < kScales ? P.l[j + 1].first : P.blocks;
        const double count = (double)((int64_t)(L.w - kWin + 1) * (L.h - kWin + 1));
        const double2 *part = reinterpret_cast<const double2 *>(partials) + (int64_t)ch * P.blocks;
        double l = 0.0, cs = 0.0;
        for (int b0 = L.first; b0 < end; b0 += 8 * 32) {
            double2 q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int b = b0 + 32 * k + lane;
                q[k] = b < end ? part[b] : make_double2(0.0, 0.0);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (b0 + 32 * k < end) cs += q[k].y;
                if (coarsest) l += q[k].x;
            }
        }
        for (int off = 16; off > 0; off >>= 1) {
            cs += __shfl_xor_sync(0xffffffffu, cs, off);
            if (coarsest) l += __shfl_xor_sync(0xffffffffu, l, off);
        }
        if (lane == 0) {
            s_mean[warp] = cs / count;
            if (coarsest) s_mean[kFinishWarps + ch] = l / count;
        }
    }
    __syncthreads();
    if (threadIdx.x < kFinishWarps + 3)
        s_mean[threadIdx.x] = pow(fmax(s_mean[threadIdx.x], 0.0), B.b[min((int)threadIdx.x / 3, kScales - 1)]);
    __syncthreads();
    if (threadIdx.x == 0) {
        double mean = 0.0;
        for (int c = 0; c < 3; ++c) {
            double v = 1.0;
            for (int k = 0; k <= kScales; ++k) v *= s_mean[k * 3 + c];
            out[1 + c] = v;
            mean += v;
        }
        out[0] = mean / 3.0;
    }
}

constexpr size_t align256(size_t b) { return (b + 255) / 256 * 256; }

size_t scratch_layout(int W, int H, size_t *pyr_bytes, size_t *part_bytes) {
    size_t pyr = 0;
    int w = W, h = H;
    for (int j = 1; j < kScales; ++j) {
        w /= 2;
        h /= 2;
        pyr += align256(2 * 3 * (size_t)w * h * sizeof(float));
    }
    const int64_t ow = W - kWin + 1, oh = H - kWin + 1;
    // room for one partial per 256 positions of the first scale; the blocks of all scales
    // (512 positions each) are fewer
    const int64_t nblk = (ow * oh + 255) / 256;
    const size_t part = align256((size_t)3 * nblk * 2 * sizeof(double));
    *pyr_bytes = pyr;
    *part_bytes = part;
    return pyr + part + align256(kScales * 3 * 2 * sizeof(double));
}

}  // namespace

extern "C" {

size_t gs_msssim_scratch_bytes(int32_t width, int32_t height) {
    if (width < 1 || height < 1) return 0;
    size_t a, b;
    return scratch_layout(width, height, &a, &b);
}

gs_status gs_msssim(const float *rgb, const float *rgb_t, int32_t width, int32_t height, double *out, void *scratch,
                    size_t scratch_bytes, void *stream) {
    if (!rgb || !rgb_t || !out || !scratch) return GS_ERR_INVALID_ARG;
    // the coarsest scale (1/16) must still hold one 11 x 11 window
    if (width < 16 * kWin || height < 16 * kWin || (int64_t)width * height >= (1ll << 31)) return GS_ERR_INVALID_ARG;
    size_t pyr, part;
    const size_t need = scratch_layout(width, height, &pyr, &part);
    if (scratch_bytes < need || (reinterpret_cast<uintptr_t>(scratch) & 255u) != 0) return GS_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Window win;
    {
        double sum = 0.0, gd[kWin];
        for (int i = 0; i < kWin; ++i) {
            const double x = i - (kWin - 1) / 2.0;
            gd[i] = std::exp(-x * x / (2.0 * 1.5 * 1.5));
            sum += gd[i];
        }
        for (int i = 0; i < kWin; ++i) win.g[i] = (float)(gd[i] / sum);
    }
    const Weights wts{{0.0448, 0.2856, 0.3001, 0.2363, 0.1333}};
    char *base = static_cast<char *>(scratch);
    double *partials = reinterpret_cast<double *>(base + pyr);
    Pyramid P;
    size_t off = 0;
    int blocks = 0, w = width, h = height;
    for (int j = 0; j < kScales; ++j) {
        const float *x = rgb, *y = rgb_t;
        if (j > 0) {
            w /= 2;
            h /= 2;
            x = reinterpret_cast<const float *>(base + off);
            y = x + (size_t)3 * w * h;
            off += align256(2 * 3 * (size_t)w * h * sizeof(float));
        }
        const int tx = (w - kWin + kTileW) / kTileW, ty = (h - kWin + kTileH) / kTileH;
        P.l[j] = Level{x, y, w, h, blocks, tx};
        blocks += tx * ty;
    }
    P.blocks = blocks;
    if ((size_t)3 * blocks * 2 * sizeof(double) > part) return GS_ERR_INVALID_ARG;
    const Level &half = P.l[1];
    const int px = (half.w + 15) / 16, py = (half.h + 15) / 16;
    k_pyramid<<<dim3((unsigned)(px * py), 6), 256, 0, st>>>(P, px);
    if (gsk::launch_dep(k_ssim_terms, dim3(blocks, 3), dim3(kSsimThreads), st, P, win, partials) != cudaSuccess)
        return GS_ERR_CUDA;
    if (gsk::launch_dep(k_ssim_finish, dim3(1), dim3(32 * kFinishWarps), st, P, wts, (const double *)partials, out) !=
        cudaSuccess)
        return GS_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

}  // extern "C"
