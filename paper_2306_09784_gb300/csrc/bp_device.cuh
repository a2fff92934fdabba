// Device helpers shared by the backprojection kernels (backproject.cu,
// backproject_pairs.cu): single-instruction math, the FP32 differential range
// and the interpolate-rotate-accumulate step of one update.
#pragma once

#include "sar_internal.h"

namespace sar {
namespace {

constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23: adding it (rounding down) floors to an integer
constexpr uint32_t kMagicBits = 0x4B400000u;
// Truncation bound of the expansion loop, in bins of the index.
constexpr double kExpansionTolBins = 2e-6;

// Per-block loop choice, OR-reduced over the CTA's FP64 tasks.
constexpr int kFlagExact = 1;    // the expansion loop cannot take the block
constexpr int kFlagOffAxis = 2;  // some Rx offset has a y component

template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(dst), "l"(src), "n"(BYTES),
                 "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ float4 lds128(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(addr)
                 : "memory");
    return v;
}

// Single MUFU operations (flush-to-zero, no special-case fix-up sequences).
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void sincos_approx(float x, float &s, float &c) {
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(x));
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(c) : "f"(x));
}

// FP64 square root of x >= 0 from an FP32 reciprocal-square-root seed and one
// Newton step on the residual x - r^2 (relative error ~1e-14, below what the
// index and phase need).  Non-finite or negative x gives NaN.
__device__ __forceinline__ double sqrt_fp64(double x) {
    // outside the seed's range: tiny -> 0, huge stays huge (rejected later as
    // beyond the maximum range), negative or NaN -> NaN
    const float xf = (float)x;
    if (!(xf >= 1e-30f && xf <= 1e30f))
        return x >= 0.0 ? (x < 1e-30 ? 0.0 : x) : __longlong_as_double(0x7ff8000000000000ll);
    const double y = (double)rsqrt_approx(xf);
    const double r = x * y;
    return fma(0.5 * y, fma(-r, r, x), r);
}

// Differential range d - R for a point at offset (dx, dy) from the tile
// reference, given w = (reference - antenna).xy, R ~ |w| and R^2 in
// w4 = (wx, wy, R, R^2).  Exact identity: d^2 = R^2 + 2 num with
// num = w.delta + |delta|^2 / 2.  With y = rsqrt(s), s = R^2 + 2 num, the first
// guess e = s y - R is refined by one Newton step on the residual
// r = num - e (R + e / 2) = (d^2 - (R + e)^2) / 2, giving e + r y.  Relative
// FP32 error of each term, never an absolute error of order ulp(R).
// `y` returns the reciprocal distance.
__device__ __forceinline__ float range_delta(float4 w, float dx, float dy, float hd2, float &y) {
    const float num = fmaf(w.x, dx, fmaf(w.y, dy, hd2));
    const float s = fmaf(2.0f, num, w.w);
    y = rsqrt_approx(s);
    const float e = fmaf(s, y, -w.z);
    const float t = fmaf(0.5f, e, w.z);
    const float r = fmaf(-e, t, num);
    return fmaf(r, y, e);
}

// OR of the threads' flag bits into a shared slot (one atomic per warp).
__device__ __forceinline__ void or_flags(int *slot, int bits) {
    const int w = (int)__reduce_or_sync(0xffffffffu, (unsigned)bits);
    if ((threadIdx.x & 31) == 0 && w) atomicOr(slot, w);
}

// floor(n / d) for 0 <= n, n d < 2^32, from mul = ceil(2^32 / d).
__device__ __forceinline__ int fast_div(int n, unsigned long long mul) {
    return (int)(((unsigned long long)(unsigned)n * mul) >> 32);
}

// One update: with f the fractional part of idx and g = kappa f, interpolate
// entry (A, D) as A + g D and accumulate it times exp(j g).  tm = 1.5 2^23 +
// floor(idx) exactly; kapm = kappa 1.5 2^23 is exact, so fma(-kappa, tm, kapm)
// = -kappa floor(idx) with one rounding, and g = fma(idx, kappa, that) with
// one more (absolute error ~ ulp(kappa L), a few 1e-4 rad at most).
__device__ __forceinline__ void accumulate(float idx, uint32_t ac, float kap, float kapm, float &acc_re,
                                           float &acc_im) {
    const float tm = __fadd_rd(idx, kMagic);
    const float g = fmaf(idx, kap, fmaf(-kap, tm, kapm));
    const float4 e = lds128((__float_as_uint(tm) << 4) + ac);
    const float vre = fmaf(g, e.z, e.x);
    const float vim = fmaf(g, e.w, e.y);
    float sn, cs;
    sincos_approx(g, sn, cs);
    acc_re = fmaf(vre, cs, acc_re);
    acc_im = fmaf(vre, sn, acc_im);
    acc_re = fmaf(-vim, sn, acc_re);
    acc_im = fmaf(vim, cs, acc_im);
}

// Blackwell's packed FP32 pairs: one instruction issues two FP32 operations,
// each rounded as its scalar form.  Pixels 2h and 2h + 1 of a thread share
// each pair, which cuts the pixel loop's instruction count by a fifth (the
// loop is issue-bound; the FMA pipe does the same work).
__device__ __forceinline__ float2 ffma2(float2 x, float2 y, float2 z) { return __ffma2_rn(x, y, z); }
__device__ __forceinline__ float2 fmul2(float2 x, float2 y) { return __fmul2_rn(x, y); }
__device__ __forceinline__ float2 bcast(float v) { return make_float2(v, v); }

// accumulate() for the pixel pair (2h, 2h + 1) of one pulse and Rx.  The
// imaginary part is kept as two sums, sum vre sn in acc_im and
// sum (-vim) cs in acc_imb (subtracted by the caller), so that every packed
// product has operands of the sign they are computed with; -vim itself comes
// from one scalar FMA with negated operands.
__device__ __forceinline__ void accumulate2(float2 idx, uint32_t ac, float2 kap, float2 nkap, float2 kapm,
                                            float (&acc_re)[kPxPerThread], float (&acc_im)[kPxPerThread],
                                            float (&acc_imb)[kPxPerThread], int h) {
    const float2 tm = __fadd2_rd(idx, bcast(kMagic));
    const float2 g = ffma2(idx, kap, ffma2(nkap, tm, kapm));
    const float4 e0 = lds128((__float_as_uint(tm.x) << 4) + ac);
    const float4 e1 = lds128((__float_as_uint(tm.y) << 4) + ac);
    const float2 vre = make_float2(fmaf(g.x, e0.z, e0.x), fmaf(g.y, e1.z, e1.x));
    const float2 vimn = make_float2(fmaf(-g.x, e0.w, -e0.y), fmaf(-g.y, e1.w, -e1.y));
    float2 sn, cs;
    sincos_approx(g.x, sn.x, cs.x);
    sincos_approx(g.y, sn.y, cs.y);
    float2 re = make_float2(acc_re[2 * h], acc_re[2 * h + 1]);
    float2 im = make_float2(acc_im[2 * h], acc_im[2 * h + 1]);
    float2 imb = make_float2(acc_imb[2 * h], acc_imb[2 * h + 1]);
    re = ffma2(vre, cs, re);
    im = ffma2(vre, sn, im);
    re = ffma2(vimn, sn, re);
    imb = ffma2(vimn, cs, imb);
    acc_re[2 * h] = re.x;
    acc_re[2 * h + 1] = re.y;
    acc_im[2 * h] = im.x;
    acc_im[2 * h + 1] = im.y;
    acc_imb[2 * h] = imb.x;
    acc_imb[2 * h + 1] = imb.y;
}

// Arrival of a warp that has just written its CTA's share of a split tile (its
// 128 pixels) to `partial`.  The last of the tile's CTAs to arrive gets the sum
// of all shares, in CTA order, and true.  arr.count: [n_tiles][8] counters that
// this launch finds at zero (arr.base = 0), or that it raises to its own base,
// above every count of an earlier call: nothing an earlier call left behind
// (one that gave up, or calls that overlapped) reaches this one.
__device__ __forceinline__ bool sum_split_tile(const BpArgs &a, const BpArrivals &arr, int tile,
                                               float (&acc_re)[kPxPerThread], float (&acc_im)[kPxPerThread]) {
    __threadfence();
    __syncwarp();
    const long long PB = a.blocks_per_tile, ua = (long long)tile * PB, ub = ua + PB - 1;
    const int ia = (int)(((ua + 1) * a.G - 1) / a.units), ib = (int)(((ub + 1) * a.G - 1) / a.units);
    int n = 0;
    if ((threadIdx.x & 31) == 0) {
        unsigned long long *count = arr.count + tile * (kBpThreads / 32) + (threadIdx.x >> 5);
        if (arr.base) atomicMax(count, arr.base);
        n = (int)(atomicAdd(count, 1ull) - arr.base);
    }
    n = __shfl_sync(0xffffffffu, n, 0);
    if (n != ib - ia) return false;
    __threadfence();
#pragma unroll
    for (int j = 0; j < kPxPerThread; ++j) acc_re[j] = acc_im[j] = 0.f;
    // CTA ia may have begun in an earlier tile; the others begin in this one
    long long at = (long long)ia * a.seg_max + (tile - (int)((long long)ia * a.units / a.G / PB));
#pragma unroll 4
    for (int i = ia; i <= ib; ++i) {
        const float2 *part = a.partial + at * kTilePx + threadIdx.x;
        at = (long long)(i + 1) * a.seg_max;
#pragma unroll
        for (int j = 0; j < kPxPerThread; ++j) {
            const float2 v = __ldcg(part + j * kBpThreads);
            acc_re[j] += v.x;
            acc_im[j] += v.y;
        }
    }
    return true;
}

}  // namespace
}  // namespace sar
