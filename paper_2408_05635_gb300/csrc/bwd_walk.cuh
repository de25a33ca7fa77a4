// bwd_walk.cuh -- the per-pixel step of the reverse compositing walk (differentiating
// Eqs. 2-4) and the sums over a warp's pixels, shared by k_backward and the fused
// tracking kernel.
//
// A warp owns an 8 x 4 patch, one pixel per lane, and walks its list back to front; the walk
// is bound by instruction issue.  Every (pixel, Gaussian) step yields two values,
// dp = dL/dpower and the weight w = a T; a Gaussian's gradient needs their sums over the
// patch (dp times 1, dx, dy, dx^2, dx dy, dy^2; w times the upstream planes).  Summing
// across lanes with shuffles issued about 30 instructions per entry for the pose's six sums
// and 75 for all ten.  Instead the warp stores dp and w of eight entries as rows of a small
// shared matrix and reads it transposed: lane (row v, entry k) sums the eight pixels of
// patch row v for entry k in registers (dx is the entry's own, dy one number per row), and
// two exchange rounds add the four rows; the walk itself has no exchange left, so its steps
// are independent but for T and g.B.  Rows are 36 floats apart: the stores (32 consecutive
// floats) and the transposed 16-byte loads (eight lanes, eight rows: banks 4k..4k+3) are
// free of conflicts.  Eight rows a warp is what fits four blocks per SM beside the staged
// batch.  Measured on the 640 x 480 / 200k tracking frame: the fused kernel 85.7 M -> 67.0 M
// warp instructions, 107 -> 85 us in ncu (of the 67 M: 10.5 M these sums, 22.9 M the walk's
// steps, 18.6 M the forward walk, 13.6 M sort, staging, lists and loss); the mapping
// window's full walk (8 x 1200 x 680, 1M Gaussians) 2,374 -> 1,202 us.
#pragma once

#include "gs_internal.cuh"

namespace gsk {

constexpr int kRedRows = 8;     // entries per transposed sum
constexpr int kRedStride = 36;  // floats between rows
constexpr int kRedFloats = 2 * kRedRows * kRedStride;  // dp rows, then w rows
// Per warp: the rows, then the upstream planes of its pixels (g_D; the full walk g_r, g_g, g_b too).
template <bool POSE>
constexpr int kWalkFloats = kRedFloats + (POSE ? 32 : 4 * 32);

// Slots of a staged Gaussian's row in the shared accumulator.  Pose only: 0, 1 sum dp dx,
// dp dy; 2 sum w g_D; 3..5 sum dp dx^2, dp dx dy, dp dy^2.  All parameters: 0, 1 the same;
// 2 sum w g_D; 3 sum dp (the opacity's: dL/da a where a is not clamped); 4 sum w g_r;
// 5..7 the second moments; 8, 9 sum w g_g, w g_b.  Odd strides spread rows over the banks.
template <bool POSE>
struct Acc {
    static constexpr int kValues = POSE ? 6 : 10;
    static constexpr int kStride = kValues + 1;
    static constexpr int kHalf = kValues / 2;
};

// One pixel's upstream gradient.
struct PixUp {
    float r, g, b, D, S;
};

// One back-to-front step for this lane's pixel: updates T and g.B and returns dp = dL/dpower
// (zero where the alpha is clamped) and w = a T, both zero where c is false.
__device__ __forceinline__ float2 bwd_step(bool c, const PolyEval &pe, float4 Cc, const PixUp &g, float amax, float &T,
                                           float &GB) {
    const float araw = ex2_approx(pe.poly);
    const float a = c ? fminf(amax, araw) : 0.f;
    const float gv = fmaf(g.r, Cc.x, fmaf(g.g, Cc.y, fmaf(g.b, Cc.z, fmaf(g.D, Cc.w, g.S))));
    const float diff = gv - GB;
    if (c) {
        T = T * rcp_approx(1.f - a);  // transmittance in front of this Gaussian
        GB = fmaf(a, diff, GB);
    }
    const float dalpha = T * diff;
    return make_float2(c && araw < amax ? dalpha * a : 0.f, a * T);
}

__device__ __forceinline__ float sum2(float2 a) { return a.x + a.y; }
__device__ __forceinline__ float2 lo2(const float4 &q) { return make_float2(q.x, q.y); }
__device__ __forceinline__ float2 hi2(const float4 &q) { return make_float2(q.z, q.w); }
__device__ __forceinline__ float dot8(const float4 &a0, const float4 &a1, const float4 &b0, const float4 &b1) {
    return sum2(__ffma2_rn(hi2(a1), hi2(b1), __ffma2_rn(lo2(a1), lo2(b1), __ffma2_rn(hi2(a0), hi2(b0), __fmul2_rn(lo2(a0), lo2(b0))))));
}

// The same of weights a and a plane b that may hold infinities and NaN, which only a weight that is
// not zero brings in.
__device__ __forceinline__ float dot8_met(const float4 &a0, const float4 &a1, const float4 &b0, const float4 &b1) {
    const auto met = [](const float4 &a, const float4 &b) {
        return make_float4(a.x != 0.f ? b.x : 0.f, a.y != 0.f ? b.y : 0.f, a.z != 0.f ? b.z : 0.f, a.w != 0.f ? b.w : 0.f);
    };
    return dot8(a0, a1, met(a0, b0), met(a1, b1));
}

// Sums of the rows [0, m) of `buf` (m <= kRedRows) over the warp's patch, added to the
// accumulator rows of their batch positions.  Lane (v = lane / 8, k = lane mod 8) takes patch
// row v of entry k; off: the entry's byte offset (any valid one for k >= m).  (pu, pv): the
// patch origin.  ODD: a plane may hold values that are not finite.  The caller's stores to buf
// are complete (__syncwarp) and it does not store again before another __syncwarp.
template <bool POSE, bool ODD>
__device__ __forceinline__ void reduce_rows(const float *buf, int m, int off, const float4 *sP0, float pu, float pv,
                                            float *sAcc, int lane) {
    using A = Acc<POSE>;
    const int k = lane & (kRedRows - 1), row = lane >> 3;
    const float4 *dq = reinterpret_cast<const float4 *>(buf + k * kRedStride + row * kPatchW);
    const float4 *wq = reinterpret_cast<const float4 *>(buf + (kRedRows + k) * kRedStride + row * kPatchW);
    const float4 d0 = dq[0], d1 = dq[1], w0 = wq[0], w1 = wq[1];
    const float2 c = *reinterpret_cast<const float2 *>(&at_off(sP0, off));  // (-cu, -cv)
    // dx, dy rounded as eval_poly rounds them: pixel coordinate (exact) less centre
    const float dy = (pv + (float)row) + c.y;
    const float2 p2 = make_float2(pu, pu), c2 = make_float2(c.x, c.x);
    const float2 x0 = __fadd2_rn(__fadd2_rn(p2, make_float2(0.f, 1.f)), c2);
    const float2 x1 = __fadd2_rn(__fadd2_rn(p2, make_float2(2.f, 3.f)), c2);
    const float2 x2 = __fadd2_rn(__fadd2_rn(p2, make_float2(4.f, 5.f)), c2);
    const float2 x3 = __fadd2_rn(__fadd2_rn(p2, make_float2(6.f, 7.f)), c2);
    const float2 t0 = __fmul2_rn(lo2(d0), x0), t1 = __fmul2_rn(hi2(d0), x1);
    const float2 t2 = __fmul2_rn(lo2(d1), x2), t3 = __fmul2_rn(hi2(d1), x3);
    const float R0 = sum2(__fadd2_rn(__fadd2_rn(lo2(d0), hi2(d0)), __fadd2_rn(lo2(d1), hi2(d1))));
    const float R1 = sum2(__fadd2_rn(__fadd2_rn(t0, t1), __fadd2_rn(t2, t3)));
    const float R2 = sum2(__ffma2_rn(t3, x3, __ffma2_rn(t2, x2, __ffma2_rn(t1, x1, __fmul2_rn(t0, x0)))));
    const float Y = dy * R0;
    float a[A::kHalf], b[A::kHalf];  // the halves' values, in slot order
    a[0] = R1;
    a[1] = Y;
    b[0] = R2;
    b[1] = dy * R1;
    b[2] = dy * Y;
    const float4 *pq = reinterpret_cast<const float4 *>(buf + kRedFloats + row * kPatchW);
    const auto plane = [&](int i) { return ODD ? dot8_met(w0, w1, pq[i], pq[i + 1]) : dot8(w0, w1, pq[i], pq[i + 1]); };
    a[2] = plane(0);
    if constexpr (!POSE) {
        a[3] = R0;
        a[4] = plane(8);
        b[3] = plane(16);
        b[4] = plane(24);
    }
    // the four rows of an entry: lanes with bit 4 set take the second half of the values,
    // then neighbours over bit 3 exchange in pairs (an odd last value is summed by both)
    const bool h = (lane & 16) != 0, q = (lane & 8) != 0;
#pragma unroll
    for (int i = 0; i < A::kHalf; ++i) a[i] = (h ? b[i] : a[i]) + __shfl_xor_sync(0xffffffffu, h ? a[i] : b[i], 16);
    float *acc = sAcc + (off >> 4) * A::kStride + (h ? A::kHalf : 0);
#pragma unroll
    for (int i = 0; i + 1 < A::kHalf; i += 2) {
        const float s = (q ? a[i + 1] : a[i]) + __shfl_xor_sync(0xffffffffu, q ? a[i] : a[i + 1], 8);
        if (k < m && s != 0.f) atomicAdd(acc + i + (q ? 1 : 0), s);
    }
    const float s = a[A::kHalf - 1] + __shfl_xor_sync(0xffffffffu, a[A::kHalf - 1], 8);
    if (k < m && !q && s != 0.f) atomicAdd(acc + A::kHalf - 1, s);
}

// The reverse walk of the warp over list entries [0, nl) (byte offsets, ascending), back to
// front: entries below lim are in front of this pixel's last contributor.  COUNT: n_eval and
// n_contrib count the footprints evaluated and differentiated.  ODD: as for reduce_rows.  The topmost nl mod 8
// entries go first, so the other groups of eight are aligned in the list (one load each).
template <bool POSE, bool COUNT, bool ODD = false>
__device__ __forceinline__ void bwd_walk_batch(const uint16_t *list, int nl, int lim, const float4 *sP0,
                                               const float4 *sP1, const float4 *sC, float2 uv, float pu, float pv,
                                               float thr, float amax, const PixUp &g, float &T, float &GB, float *buf,
                                               float *sAcc, int lane, uint32_t &n_eval, uint32_t &n_contrib) {
    const auto step = [&](int j, int r) {
        const PolyEval pe = eval_poly(uv, at_off(sP0, j), p1_at(sP1, j));
        const bool live = j < lim, c = live && pe.poly >= thr;
        if constexpr (COUNT) {
            n_eval += live;
            n_contrib += c;
        }
        const float2 dw = bwd_step(c, pe, at_off(sC, j), g, amax, T, GB);
        buf[r * kRedStride + lane] = dw.x;
        buf[(kRedRows + r) * kRedStride + lane] = dw.y;
    };
    const auto sums = [&](int e, int m) {  // of the entries [e, e + m) just stored
        __syncwarp();
        const int k = lane & (kRedRows - 1);
        reduce_rows<POSE, ODD>(buf, m, (int)list[e + (k < m ? k : 0)], sP0, pu, pv, sAcc, lane);
        __syncwarp();
    };
    int e = nl & ~(kRedRows - 1);
    const int m = nl - e;
    if (m) {
        for (int r = m - 1; r >= 0; --r) step((int)list[e + r], r);
        sums(e, m);
    }
    for (e -= kRedRows; e >= 0; e -= kRedRows) {
        const uint4 q = *reinterpret_cast<const uint4 *>(list + e);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int r = kRedRows - 1; r >= 0; --r) step((int)((r & 1) ? w[r >> 1] >> 16 : w[r >> 1] & 0xffffu), r);
        sums(e, kRedRows);
    }
}

// This lane's pixel's upstream planes, read by reduce_rows.
template <bool POSE>
__device__ __forceinline__ void store_planes(float *buf, const PixUp &g, int lane) {
    buf[kRedFloats + lane] = g.D;
    if constexpr (!POSE) {
        buf[kRedFloats + 32 + lane] = g.r;
        buf[kRedFloats + 64 + lane] = g.g;
        buf[kRedFloats + 96 + lane] = g.b;
    }
}

// Does a plane of the warp hold a value that is not finite (0 times which is not 0)?
__device__ __forceinline__ bool odd_planes(const PixUp &g) {
    return __any_sync(0xffffffffu, fmaf(0.f, g.r, fmaf(0.f, g.g, fmaf(0.f, g.b, 0.f * g.D))) != 0.f);
}

// The walk of a warp with such planes: a pixel whose upstream gradient is an infinity or a NaN
// then reaches the Gaussians it sees and no others.  A function of its own: as a choice inside
// the walk it cost every warp 2 to 3 % (8 views of 1200 x 680: 2,190 -> 2,251 us; this way 2,204).
struct WalkState {
    float T, GB;
    uint32_t n_eval, n_contrib;
};
template <bool POSE>
__device__ __noinline__ WalkState bwd_walk_odd(const uint16_t *list, int nl, int lim, const float4 *sP0, const float4 *sP1,
                                               const float4 *sC, float2 uv, float pu, float pv, float thr, float amax,
                                               PixUp g, WalkState s, float *buf, float *sAcc, int lane) {
    bwd_walk_batch<POSE, true, true>(list, nl, lim, sP0, sP1, sC, uv, pu, pv, thr, amax, g, s.T, s.GB, buf, sAcc, lane,
                                     s.n_eval, s.n_contrib);
    return s;
}

// Apply the conic Q to a Gaussian's sums over the tile and add them to its record's global
// accumulator (o: its opacity, for the full walk).
template <bool POSE>
__device__ __forceinline__ void flush_acc(const float *m, float4 Q, float o, RecGrad *out) {
    constexpr int s = Acc<POSE>::kHalf;  // first second moment
    const float4 v0 = make_float4(Q.x * m[0] + Q.y * m[1], Q.y * m[0] + Q.z * m[1], m[2], POSE ? 0.f : m[3] / o);
    const float4 v1 = make_float4(-0.5f * m[s], -m[s + 1], -0.5f * m[s + 2], 0.f);
    if (v0.x != 0.f || v0.y != 0.f || v0.z != 0.f || v0.w != 0.f) atomicAdd(&out->g0, v0);
    if (v1.x != 0.f || v1.y != 0.f || v1.z != 0.f) atomicAdd(&out->g1, v1);
    if constexpr (!POSE) {
        const float4 v2 = make_float4(m[4], m[8], m[9], 0.f);
        if (v2.x != 0.f || v2.y != 0.f || v2.z != 0.f) atomicAdd(&out->g2, v2);
    }
}

}  // namespace gsk
