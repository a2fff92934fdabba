// Per-pixel Doppler index offsets f_doppler(p) of Alg. 2 (paper Sec. III-D):
// the velocity terms of Alg. 1 (lines 5, 8, 9 and the f0 v / c part of line
// 11), evaluated once per reconstruction point from the average vehicle
// velocity over the chirp sequence instead of per (chirp, antenna):
//   vbar = mean_m vel(m),  qt = mean_m q_tx(m),  qr = mean_{m,n} q_rx(m, n),
//   f_doppler(p) = -(f0 / c) (<p - qt, vbar> / |p - qt| + <p - qr, vbar> / |p - qr|) N_fft / fs,
// the rate of change of the two-way path (a platform closing on p shortens
// it) times f0 / c, in bins of the range transform.
//
// Two kernels: a few CTAs sum positions and velocities in FP64; then one thread
// per pixel slot of the plan's tiles (positions = FP64 tile reference + FP32 offset)
// writes its offset at the pixel's image index.  Both read device memory only
// (graph-capturable).
#include "sar_internal.h"

namespace sar {
namespace {

// Partial sums by kMeanCtas CTAs of 256 threads: one CTA is bound by its SM's
// two FP64 lanes (the adds and the warp reductions of 1024 chirps x 8 Rx take
// 15 us there) and by one load in flight.
constexpr int kMeanThreads = 256;

// (e . v) / |e| in FP64: 1 / |e| from an FP32 reciprocal square root and two
// Newton steps, as accurate as hypot and a division (the first leaves 2^-45: up
// to 2.5e-14, which shows where the two antennas' terms cancel).  The FP64 pipe
// has two lanes per SM: hypot and a division took ~100 of its operations per
// distance, this takes 16.  A point on the antenna's mean position has no radial
// direction: 0 there.
__device__ __forceinline__ double radial(double ex, double ey, double vx, double vy) {
    const double d2 = fma(ex, ex, ey * ey), dot = fma(ex, vx, ey * vy);
    const float f = (float)d2;
    if (!(f >= 1e-30f && f <= 1e30f)) {  // beyond the seed's range, zero or not finite
        const double n = hypot(ex, ey);
        return n > 0 ? dot / n : 0.0;
    }
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
    const double y0 = (double)y;
    const double y1 = fma(0.5 * y0, fma(-d2 * y0, y0, 1.0), y0);
    return dot * fma(0.5 * y1, fma(-d2 * y1, y1, 1.0), y1);
}

// sums[cta][0..5]: this CTA's share of the sums of (q_tx.x, q_tx.y, q_rx.x,
// q_rx.y, vel.x, vel.y).
__global__ void __launch_bounds__(kMeanThreads) doppler_sums_kernel(const double *__restrict__ q_tx,
                                                                    const double *__restrict__ q_rx,
                                                                    const double *__restrict__ vel, int M, int R,
                                                                    double *__restrict__ sums) {
    __shared__ double part[6][kMeanThreads / 32];
    double s[6] = {0, 0, 0, 0, 0, 0};
    const int first = blockIdx.x * kMeanThreads + threadIdx.x, step = kMeanCtas * kMeanThreads;
#pragma unroll 4
    for (int m = first; m < M; m += step) {
        s[0] += q_tx[2 * m];
        s[1] += q_tx[2 * m + 1];
        s[4] += vel[2 * m];
        s[5] += vel[2 * m + 1];
    }
    const long long nr = (long long)M * R;
#pragma unroll 4
    for (long long i = first; i < nr; i += step) {
        s[2] += q_rx[2 * i];
        s[3] += q_rx[2 * i + 1];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        double v = s[c];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) part[c][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        double v = 0;
        for (int w = 0; w < kMeanThreads / 32; ++w) v += part[threadIdx.x][w];
        sums[blockIdx.x * 6 + threadIdx.x] = v;
    }
}

__global__ void __launch_bounds__(256) doppler_offsets_kernel(const TileInfo *__restrict__ tiles,
                                                               const float2 *__restrict__ pix,
                                                               const int *__restrict__ out_idx, long long slots,
                                                               const double *__restrict__ sums, int M, long long nr,
                                                               double scale, float *__restrict__ fd) {
    __shared__ double means[6];  // (qt.x, qt.y, qr.x, qr.y, vbar.x, vbar.y)
    if (threadIdx.x < 6) {
        const int c = threadIdx.x;
        double v = 0;
#pragma unroll
        for (int k = 0; k < kMeanCtas; ++k) v += sums[k * 6 + c];
        means[c] = v / ((c == 2 || c == 3) ? (double)nr : (double)M);
    }
    __syncthreads();
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= slots) return;
    const int o = out_idx[s];
    if (o < 0) return;
    const TileInfo ti = tiles[s / kTilePx];
    const float2 d = pix[s];
    const double x = ti.x + (double)d.x, y = ti.y + (double)d.y;
    const double ex = x - means[0], ey = y - means[1];
    const double gx = x - means[2], gy = y - means[3];
    const double vx = means[4], vy = means[5];
    const double v_tx = radial(ex, ey, vx, vy);
    const double v_rx = radial(gx, gy, vx, vy);
    fd[o] = (float)(-(v_tx + v_rx) * scale);
}

}  // namespace

cudaError_t launch_doppler_offsets(const DopplerArgs &a, cudaStream_t s) {
    doppler_sums_kernel<<<kMeanCtas, kMeanThreads, 0, s>>>(a.q_tx, a.q_rx, a.vel, a.M, a.R, a.sums);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long slots = (long long)a.n_tiles * kTilePx;
    if (slots == 0) return cudaSuccess;
    doppler_offsets_kernel<<<(unsigned)((slots + 255) / 256), 256, 0, s>>>(a.tiles, a.pix, a.out_idx, slots,
                                                                            a.sums, a.M, (long long)a.M * a.R, a.scale, a.fd);
    return cudaGetLastError();
}

}  // namespace sar
