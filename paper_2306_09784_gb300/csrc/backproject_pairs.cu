// Backprojection (paper Alg. 2) from interpolation pairs: the single-request
// path of sar_backproject and sar_form_image_host.  The arithmetic of an
// update is that of backproject.cu (the same FP64 references, window starts,
// index and phase roundings); what differs is how the pixel loop is fed.
//
//  * backproject.cu copies each tile's raw samples to shared memory and turns
//    them into (A, D) pairs there, once per tile: on a 512 x 512 frame with
//    FP32 profiles that is 22 % of all shared-memory wavefronts and 8 % of the
//    instructions.  Here expand_pairs_kernel makes the pairs once per call in
//    global memory (16 bytes a bin, L2-resident for ordinary frames), and a
//    tile's window of a profile row is one bulk copy that reports to an
//    mbarrier: no conversion or raw buffer in the CTA, and shared-memory
//    wavefronts fall from 5.7 to 4.3 per 32 updates.  Copies as cp.async of
//    16-byte entries were 1-2 % slower on frames and 15 % on point lists.
//  * What bounds it: the packed FMA, MUFU and shared-memory pipes at 57-62 %
//    each of the time and instruction issue at 61 %, as in backproject.cu.
//    With the expansion, against the copying kernel: 512 x 512 x 1024 x 4 FP32
//    frame 0.86 -> 0.79 ms; 1024 x 1024 x 2048 x 4 FP16 6.42 -> 6.14 ms;
//    165 000 polar points x 1024 x 8 with Doppler offsets 6.07 -> 2.44 ms.
//  * The window is cut to the bins the tile can reach: its own radius and the
//    call's largest Rx offset (reduced by the expansion kernel) instead of
//    the plan-wide length, which a point list's widest run of 1024 points
//    sets.  Window starts, and so every rounding, stay those of the plan-wide
//    window; only the bins before and after the reachable ones are not staged.
//    The pulses per pipeline block follow from the tile's window (as many as
//    fit).
//  * Work is split across CTAs in units of kPairUnit pulses.  A tile shared by
//    several CTAs is summed, in CTA order, by whichever warp arrives last for
//    its 128 pixels: no second launch.
//  * expand_pairs_kernel also takes the Rx offsets (FP64 differences) of a
//    call out of the per-tile stage, so that only the Tx references are FP64
//    there.
//  * Which loop a pulse takes (expansion or exact) is decided as in
//    backproject.cu, per aligned run of its pulse block, so that images do not
//    depend on how blocks are cut here.
#include <cuda_fp16.h>

#include <algorithm>

#include "bp_device.cuh"
#include "sar_internal.h"

namespace sar {
namespace {

// Full barriers of the two table slots, exact-loop bits of the three Tx slots,
// stall bits.
constexpr unsigned kHeaderBytes = 32;
constexpr int kWarps = kBpThreads / 32;
// Slack (bins) on both ends of a staged window: the FP32 index differs from
// the real one by a few 1e-5 bins at most.
constexpr float kWindowSlack = 0.02f;

__device__ __forceinline__ void mbar_init(uint32_t bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait of a whole warp (its lanes stay together): false if the phase
// has not completed after `polls` polls.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int polls) {
    for (int i = 0; i < polls; ++i)
        if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
    return false;
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// Shared memory of one tile: `slots` tables of Mt x R windows of Lt entries,
// three slots of Tx records and two of Rx records.
struct PairLayout {
    int Mt, slots, Lt, s0;
    uint32_t table, txr, rxa, txc, rxb, txo;
};

// Bytes of the records of one pulse.
__host__ __device__ constexpr unsigned pair_const_bytes(int R) { return 3u * 28u + 2u * 24u * (unsigned)R; }

// PU: pulses the pixel loop unrolls together (blocks are multiples of it
// where they can be).
__device__ __forceinline__ PairLayout pair_layout(const BpPairArgs &pa, const TileInfo &ti, int n_pulses, int PU) {
    const BpArgs &a = pa.b;
    PairLayout l;
    const float a1 = a.a1f, rho = (float)ti.rho;
    const float omax = __uint_as_float(pa.call[0]);
    const float o = fminf(omax, ti.o_allow);
    // reachable indices: [a1 (o_allow - o) + G, a1 (o_allow + o) + 4 a1 rho
    // + 2 fd_max + G + 1] in the expansion loop (window start at klo_off),
    // [G, 4 a1 rho + 2 fd_max + G + 1] in the exact loop
    const float span = 4.0f * a1 * rho + 2.0f * a.fd_max + (float)(kGuardBins + 1) + kWindowSlack;
    l.s0 = (int)floorf(a1 * (ti.o_allow - o) + (float)kGuardBins - kWindowSlack);
    const int last = (int)floorf(a1 * (ti.o_allow + o) + span);
    l.Lt = min(max(last - l.s0 + 1, (int)floorf(span) + 1), a.L);
    const unsigned win = (unsigned)(a.R * l.Lt) * 16u;
    const unsigned cap = pa.smem_bytes - kHeaderBytes, cst = pair_const_bytes(a.R);
    l.slots = 2;
    int fit = (int)(cap / (2u * win + cst));
    if (fit < 1) {  // a wide run of points: one table, no copy ahead
        l.slots = 1;
        fit = (int)(cap / (win + cst));
    }
    fit = min(fit, pa.mb_cap);
    if (fit > PU) fit -= fit % PU;
    // equal blocks
    const int nb = (n_pulses + fit - 1) / fit;
    int mt = (n_pulses + nb - 1) / nb;
    mt = (mt + PU - 1) / PU * PU;
    l.Mt = max(1, min(mt, fit));
    l.table = kHeaderBytes;
    l.txr = l.table + (unsigned)(l.slots * l.Mt) * win;
    l.rxa = l.txr + 3u * l.Mt * 16u;
    l.txc = l.rxa + 2u * l.Mt * a.R * 16u;
    l.rxb = l.txc + 3u * l.Mt * 8u;
    l.txo = l.rxb + 2u * l.Mt * a.R * 8u;
    return l;
}

struct PairSmem {
    unsigned char *base;
    uint32_t addr;
    PairLayout l;
    // Tx records of slot s (b % 3): float4 (wx, wy, R, R^2), int2 (index
    // constant bits, k_lo)
    __device__ float4 *txr(int s) const { return reinterpret_cast<float4 *>(base + l.txr) + s * l.Mt; }
    __device__ int2 *txc(int s) const { return reinterpret_cast<int2 *>(base + l.txc) + s * l.Mt; }
    // largest |o|^2 that the pulse's window and loop choice cover
    __device__ float *txo(int s) const { return reinterpret_cast<float *>(base + l.txo) + s * l.Mt; }
    // Rx records of slot t (b % 2).  Expansion loop: (o_x / 2, -c / 2) and
    // o_y / 2; exact loop: (wx, wy, R, R^2) and (index constant bits, k_lo)
    __device__ float4 *rxa(int t, int R) const { return reinterpret_cast<float4 *>(base + l.rxa) + t * l.Mt * R; }
    __device__ int2 *rxb(int t, int R) const { return reinterpret_cast<int2 *>(base + l.rxb) + t * l.Mt * R; }
    // per Tx slot: bit j set where run j of the block takes the exact loop
    __device__ unsigned *exact(int s) const { return reinterpret_cast<unsigned *>(base) + 4 + s; }
    // bit b & 1 set: a wait of block b ran out (two bits, so that a warp already
    // in the next block cannot change what the others read of this one)
    __device__ volatile int *stall() const { return reinterpret_cast<volatile int *>(base) + 7; }
    __device__ uint32_t bar(int t) const { return addr + 8u * t; }
    // first byte of window w of table slot t
    __device__ uint32_t win(int t, int R, int w) const {
        return addr + l.table + (uint32_t)((t * l.Mt * R + w) * l.Lt) * 16u;
    }
};

// Whether a pulse whose Tx offset from the tile reference is (wx, wy) and
// whose largest squared Rx offset is o2 is outside the expansion loop's reach
// (prep_block's criteria in backproject.cu: every one is monotone in the Rx
// offset).  Non-finite geometry is.
__device__ __forceinline__ bool pulse_exact(const TileInfo &ti, float tol2, float wx, float wy, float o2) {
    const float rho = (float)ti.rho;
    const float rt = hypotf(wx, wy);
    const float oa = sqrtf(o2);
    const float dmin = rt - rho;
    return !(rt > 2.0f * rho + oa + 1e-3f && rt < (float)kMaxRange && oa <= ti.o_allow && o2 * oa <= tol2 * dmin * dmin);
}

// FP64 stage of pulses [m0, m0 + np) into Tx slot s: the values of prep_block
// in backproject.cu, one lane per pulse of warp w0.  The loop choice is made
// per run of Mb aligned pulses (run 0 is the one that holds m0); pulses of the
// first and last run outside [m0, m0 + np) are judged by the next warp.  w0
// moves with the block, so that no one warp is always late.
__device__ __forceinline__ void prep_tx(const BpPairArgs &pa, const PairSmem &sm, const TileInfo &ti, int m0, int np,
                                        int s, int w0) {
    const BpArgs &a = pa.b;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int role = (warp - w0) & (kWarps - 1);
    if (role > 1) return;
    const int run0 = fast_div(m0, pa.div_blk);
    const float tol2 = (float)(kExpansionTolBins * 2.0 / a.a1);
    unsigned bits = 0;
    if (role == 0) {
        if (lane < np) {
            const int m = m0 + lane;
            const double2 qt = reinterpret_cast<const double2 *>(a.q_tx)[m];
            const float o2 = pa.o2max[m];
            const double wx = ti.x - qt.x, wy = ti.y - qt.y;
            const double r2 = fma(wx, wx, wy * wy);
            const double r_tx = sqrt_fp64(r2);
            const float r_f = (float)r_tx;
            float4 t4 = make_float4(0.f, 0.f, 1.f, 1.f);
            int2 c = make_int2(0, -(1 << 30));
            bool exact = true;
            if (r_f < (float)kMaxRange) {  // false for NaN and inf
                t4 = make_float4((float)wx, (float)wy, r_f, (float)r2);
                const int k_lo = __double2int_rd(fma(2.0 * a.a1, r_tx, -(double)ti.klo_off)) - kGuardBins;
                c = make_int2(__float_as_int((float)fma(2.0 * a.a1, r_tx, -(double)k_lo)), k_lo);
                exact = pulse_exact(ti, tol2, t4.x, t4.y, o2) || !(sqrtf(o2) <= __uint_as_float(pa.call[0]));
            }
            sm.txr(s)[lane] = t4;
            sm.txc(s)[lane] = c;
            sm.txo(s)[lane] = o2;
            if (exact) bits = 1u << (fast_div(m, pa.div_blk) - run0);
        }
    } else {
        const int lo = run0 * a.Mb, last = fast_div(m0 + np - 1, pa.div_blk);
        const int hi = min((last + 1) * a.Mb, a.M);
        const int n_lo = m0 - lo, n = n_lo + hi - (m0 + np);
        for (int i = lane; i < n; i += 32) {
            const int m = i < n_lo ? lo + i : m0 + np + i - n_lo;
            const double2 qt = reinterpret_cast<const double2 *>(a.q_tx)[m];
            if (pulse_exact(ti, tol2, (float)(ti.x - qt.x), (float)(ti.y - qt.y), pa.o2max[m]))
                bits |= 1u << (i < n_lo ? 0 : last - run0);
        }
    }
    bits = __reduce_or_sync(0xffffffffu, bits);
    if (lane == 0 && bits) atomicOr(sm.exact(s), bits);
}

// Run of pulse m0 + p within its block, whose run 0 holds m0.
__device__ __forceinline__ int run_of(const BpPairArgs &pa, int m0, int p) {
    return fast_div(m0 + p, pa.div_blk) - fast_div(m0, pa.div_blk);
}

// Rx records of pulses [m0, m0 + np) (Tx slot s) into slot t: the expansion
// loop's FP32 coefficients, or for pulses on the exact loop the FP64 Rx
// reference range, window start and index (prep_exact in backproject.cu).
// The offsets of the expansion loop come from memory that every call of the plan
// writes.  Calls are ordered, but a replayed graph's are ordered by the caller;
// so that a mistake there spoils an image and no more, an offset that the
// pulse's window and loop choice do not cover is dropped and flagged.
template <bool MULTI, int RG>
__device__ __forceinline__ void prep_rx(const BpPairArgs &pa, const PairSmem &sm, const TileInfo &ti, int m0, int np,
                                        int s, int t, unsigned exact) {
    const BpArgs &a = pa.b;
    const int R = MULTI ? a.R : RG;
    const float4 *txr = sm.txr(s);
    float4 *rxa = sm.rxa(t, R);
    int2 *rxb = sm.rxb(t, R);
    const float *txo = sm.txo(s);
    const bool axis = !pa.call[1];
    for (int task = threadIdx.x; task < np * R; task += kBpThreads) {
        const int p = MULTI ? fast_div(task, a.div_r) : task / RG;
        const long long row = (long long)m0 * R + task;
        if (!exact || !((exact >> run_of(pa, m0, p)) & 1u)) {
            const float4 t4 = txr[p];
            float4 g = pa.rx[row];  // (o_x, o_y, |o|^2, |o|^2 or infinite off the x axis)
            if (!((axis ? g.w : g.z) <= txo[p])) {
                g = make_float4(0.f, 0.f, 0.f, 0.f);
                atomicOr(a.err, kErrGeometry);
            }
            const float cexp = fmaf(0.5f, g.z, -fmaf(t4.x, g.x, t4.y * g.y));
            // halved so that the pixel loop gets -a / 2 directly
            rxa[task] = make_float4(0.5f * g.x, -0.5f * cexp, 0.f, 0.f);
            rxb[task] = make_int2(__float_as_int(0.5f * g.y), 0);
            continue;
        }
        const double2 qt = reinterpret_cast<const double2 *>(a.q_tx)[m0 + p];
        const double2 qr = reinterpret_cast<const double2 *>(a.q_rx)[row];
        const double wtx = ti.x - qt.x, wty = ti.y - qt.y;
        const double wrx = ti.x - qr.x, wry = ti.y - qr.y;
        const double r_tx = sqrt_fp64(wtx * wtx + wty * wty);
        const double r_rx = sqrt_fp64(wrx * wrx + wry * wry);
        const double d0 = r_tx + r_rx;
        const bool ok_tx = isfinite(r_tx) && r_tx < kMaxRange;
        const bool ok_rx = isfinite(r_rx) && r_rx < kMaxRange;
        rxa[task] = ok_rx ? make_float4((float)wrx, (float)wry, (float)r_rx, (float)(r_rx * r_rx))
                          : make_float4(0.f, 0.f, 1.f, 1.f);
        int2 c = make_int2(__float_as_int((float)kGuardBins), -(1 << 30));
        if (ok_tx && ok_rx) {
            const int k_lo = (int)floor(a.a1 * (d0 - 2.0 * ti.rho) - (double)a.fd_max) - kGuardBins;
            c = make_int2(__float_as_int((float)(a.a1 * d0 - (double)k_lo)), k_lo);
        } else {
            atomicOr(a.err, kErrGeometry);
        }
        rxb[task] = c;
    }
}

// Copies of the windows of pulses [m0, m0 + np) (Tx slot s, Rx slot rt) into
// table slot t: one bulk copy per window, or up to three where it leaves
// [crop_lo, crop_hi), whose outside reads zeros.  The windows go round the
// warps: a warp's copies are issued one after another.
template <bool MULTI, int RG>
__device__ __forceinline__ void stage_windows(const BpPairArgs &pa, const PairSmem &sm, int m0, int np, int s, int t,
                                              int rt, unsigned exact) {
    const BpArgs &a = pa.b;
    const int R = MULTI ? a.R : RG;
    const int nw = np * R, Lt = sm.l.Lt;
    const uint32_t bar = sm.bar(t);
    if (threadIdx.x == 0) mbar_expect(bar, (uint32_t)(nw * Lt) * 16u);
    for (int w = (threadIdx.x & 31) * kWarps + (threadIdx.x >> 5); w < nw; w += kBpThreads) {
        const int p = MULTI ? fast_div(w, a.div_r) : w / RG;
        const bool ex = exact && ((exact >> run_of(pa, m0, p)) & 1u);
        const int k0 = ex ? sm.rxb(rt, R)[w].y : sm.txc(s)[p].y + sm.l.s0;
        const uint32_t dst = sm.win(t, R, w);
        const float4 *row = pa.pairs + ((long long)m0 * R + w) * a.n_bins;
        const int lo = max(k0, a.crop_lo), hi = min(k0 + Lt, a.crop_hi);
        if (lo >= hi) {
            bulk_copy(dst, pa.zero, (uint32_t)Lt * 16u, bar);
            continue;
        }
        const uint32_t nl = (uint32_t)(lo - k0), nm = (uint32_t)(hi - lo), nr = (uint32_t)Lt - nl - nm;
        if (nl) bulk_copy(dst, pa.zero, nl * 16u, bar);
        bulk_copy(dst + nl * 16u, row + (lo - a.crop_lo), nm * 16u, bar);
        if (nr) bulk_copy(dst + (nl + nm) * 16u, pa.zero, nr * 16u, bar);
    }
}

// PU pulses of the expansion loop (see expand_pulses in backproject.cu); ac:
// table address constant of the first pulse's first window, step: bytes per
// window.  The two constants of a (pulse, Rx) are one 8-byte load (two
// shared-memory wavefronts); the address constant is arithmetic.
template <int RG, bool MULTI, int PU, bool FD, bool AXIS>
__device__ __forceinline__ void expand_pairs(const BpArgs &a, const float4 *txr, const int2 *txc, const float4 *rxa,
                                             const int2 *rxb, uint32_t ac, uint32_t step,
                                             const float (&dx)[kPxPerThread], const float (&dy)[kPxPerThread],
                                             const float (&hd2)[kPxPerThread], const float (&fdi)[kPxPerThread],
                                             float (&acc_re)[kPxPerThread], float (&acc_im)[kPxPerThread]) {
    constexpr int H = kPxPerThread / 2;
    const int R = MULTI ? a.R : RG;
    const float two_a1 = 2.0f * a.a1f;
    const float2 kap = bcast(a.kappa), nkap = bcast(-a.kappa), kapm = bcast(a.kappa_magic);
    float2 u[PU][H], nay[PU][H], nkk[PU][H];
    float acc_imb[kPxPerThread];
#pragma unroll
    for (int j = 0; j < kPxPerThread; ++j) acc_imb[j] = 0.f;
#pragma unroll
    for (int q = 0; q < PU; ++q) {
        const float4 t4 = txr[q];
        const float cidx = __int_as_float(txc[q].x);
#pragma unroll
        for (int h = 0; h < H; ++h) {
            float2 y;
            const float2 dt = make_float2(range_delta(t4, dx[2 * h], dy[2 * h], hd2[2 * h], y.x),
                                          range_delta(t4, dx[2 * h + 1], dy[2 * h + 1], hd2[2 * h + 1], y.y));
            const float2 c2 = FD ? make_float2(cidx + fdi[2 * h], cidx + fdi[2 * h + 1]) : bcast(cidx);
            u[q][h] = ffma2(bcast(two_a1), dt, c2);
            nay[q][h] = fmul2(bcast(-two_a1), y);
            nkk[q][h] = fmul2(nay[q][h], fmul2(y, y));
        }
    }
    for (int r0 = 0; r0 < R; r0 += RG) {
#pragma unroll
        for (int q = 0; q < PU; ++q) {
#pragma unroll
            for (int rr = 0; rr < RG; ++rr) {
                const int w = q * R + r0 + rr;
                const float2 o2 = *reinterpret_cast<const float2 *>(rxa + w);
                const float4 o4 = make_float4(o2.x, o2.x, o2.y, o2.y);
                const float oy = AXIS ? 0.f : __int_as_float(rxb[w].x);
                const uint32_t acw = ac + (uint32_t)w * step;
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    // v = -a / 2; with nay = -2 a1 / d and nkk = -2 a1 / d^3,
                    // a1 (d_rx - d_tx) = v (v nkk + nay)
                    const float2 dx2 = make_float2(dx[2 * h], dx[2 * h + 1]);
                    const float2 ox = make_float2(o4.x, o4.y), cc = make_float2(o4.z, o4.w);
                    const float2 v = AXIS ? ffma2(ox, dx2, cc)
                                          : ffma2(ox, dx2,
                                                  ffma2(bcast(oy), make_float2(dy[2 * h], dy[2 * h + 1]), cc));
                    const float2 idx = ffma2(v, ffma2(v, nkk[q][h], nay[q][h]), u[q][h]);
                    accumulate2(idx, acw, kap, nkap, kapm, acc_re, acc_im, acc_imb, h);
                }
            }
        }
        if (!MULTI) break;
    }
#pragma unroll
    for (int j = 0; j < kPxPerThread; ++j) acc_im[j] -= acc_imb[j];
}

template <int RG, bool MULTI>
__host__ __device__ constexpr int pulse_unroll() {
    return MULTI ? 1 : RG >= 3 ? 2 : 4 / RG;
}

// Pulses [p, pe) of a block on the expansion loop.
template <int RG, bool MULTI, bool FD, bool AXIS>
__device__ __forceinline__ void run_expand(const BpArgs &a, const PairSmem &sm, int p, int pe, int s, int t, int rt,
                                           const float (&dx)[kPxPerThread], const float (&dy)[kPxPerThread],
                                           const float (&hd2)[kPxPerThread], const float (&fdi)[kPxPerThread],
                                           float (&acc_re)[kPxPerThread], float (&acc_im)[kPxPerThread]) {
    constexpr int PU = pulse_unroll<RG, MULTI>();
    const int R = MULTI ? a.R : RG;
    const float4 *txr = sm.txr(s);
    const int2 *txc = sm.txc(s);
    const float4 *rxa = sm.rxa(rt, R);
    const int2 *rxb = sm.rxb(rt, R);
    const uint32_t step = (uint32_t)sm.l.Lt * 16u;
    uint32_t ac = sm.win(t, R, p * R) - (uint32_t)sm.l.s0 * 16u - kMagicBits * 16u;
    if (PU > 1) {
        for (; p + PU <= pe; p += PU, ac += PU * R * step)
            expand_pairs<RG, MULTI, PU, FD, AXIS>(a, txr + p, txc + p, rxa + p * R, rxb + p * R, ac, step, dx, dy, hd2, fdi, acc_re,
                                                  acc_im);
    }
    for (; p < pe; ++p, ac += R * step)
        expand_pairs<RG, MULTI, 1, FD, AXIS>(a, txr + p, txc + p, rxa + p * R, rxb + p * R, ac, step, dx, dy, hd2, fdi, acc_re,
                                             acc_im);
}

// range_delta for a pixel pair, the same roundings in packed instructions
// (-t is formed exactly, so that r = num - e t is one FMA).
__device__ __forceinline__ float2 range_delta2(float4 w, float2 dx, float2 dy, float2 hd2) {
    const float2 num = ffma2(bcast(w.x), dx, ffma2(bcast(w.y), dy, hd2));
    const float2 s = ffma2(bcast(2.0f), num, bcast(w.w));
    const float2 y = make_float2(rsqrt_approx(s.x), rsqrt_approx(s.y));
    const float2 e = ffma2(s, y, bcast(-w.z));
    const float2 nt = ffma2(bcast(-0.5f), e, bcast(-w.z));
    const float2 r = ffma2(e, nt, num);
    return ffma2(r, y, e);
}

// Pulses [p, pe) of a stage on the exact loop: every distance from its own
// rsqrt and Newton step, the index clamped into the staged window.  Bound by
// MUFU (one rsqrt, sine and cosine per update); the rest is packed by pixel
// pairs like the expansion loop.
template <int RG, bool FD>
__device__ __forceinline__ void run_exact(const BpArgs &a, const PairSmem &sm, int p, int pe, int s, int t, int rt,
                                          const float (&dx)[kPxPerThread], const float (&dy)[kPxPerThread],
                                          const float (&hd2)[kPxPerThread], const float (&fdi)[kPxPerThread],
                                          float (&acc_re)[kPxPerThread], float (&acc_im)[kPxPerThread]) {
    constexpr int H = kPxPerThread / 2;
    const int R = a.R;
    const float4 *txr = sm.txr(s);
    const float4 *rxa = sm.rxa(rt, R);
    const int2 *rxb = sm.rxb(rt, R);
    const float2 kap = bcast(a.kappa), nkap = bcast(-a.kappa), kapm = bcast(a.kappa_magic);
    // valid indices stay kWindowSlack below Lt (see pair_layout)
    const float lmax = (float)sm.l.Lt - 1e-3f;
    const uint32_t step = (uint32_t)sm.l.Lt * 16u;
    uint32_t ac = sm.win(t, R, p * R) - kMagicBits * 16u;
    auto pair = [](const float (&v)[kPxPerThread], int h) { return make_float2(v[2 * h], v[2 * h + 1]); };
    for (; p < pe; ++p) {
        const float4 t4 = txr[p];
        float2 dt[H];
        float acc_imb[kPxPerThread];
#pragma unroll
        for (int h = 0; h < H; ++h) dt[h] = range_delta2(t4, pair(dx, h), pair(dy, h), pair(hd2, h));
#pragma unroll
        for (int j = 0; j < kPxPerThread; ++j) acc_imb[j] = 0.f;
        for (int r0 = 0; r0 < R; r0 += RG, ac += RG * step) {
#pragma unroll
            for (int rr = 0; rr < RG; ++rr) {
                const int w = p * R + r0 + rr;
                const float4 q4 = rxa[w];
                const float idx0 = __int_as_float(rxb[w].x);
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    const float2 drx = range_delta2(q4, pair(dx, h), pair(dy, h), pair(hd2, h));
                    float2 idx = ffma2(bcast(a.a1f), __fadd2_rn(dt[h], drx), bcast(idx0));
                    if (FD) idx = make_float2(idx.x + fdi[2 * h], idx.y + fdi[2 * h + 1]);
                    idx.x = fminf(fmaxf(idx.x, 0.0f), lmax);
                    idx.y = fminf(fmaxf(idx.y, 0.0f), lmax);
                    accumulate2(idx, ac + rr * step, kap, nkap, kapm, acc_re, acc_im, acc_imb, h);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kPxPerThread; ++j) acc_im[j] -= acc_imb[j];
    }
}

// Pulses [m_begin, m_end) of one tile, from the pixel load to the output
// write (see process_segment in backproject.cu).  slot: this CTA's partial
// sums of a tile it has only a part of (whole == false).
template <int RG, bool MULTI, bool FD>
__device__ __forceinline__ bool pair_segment(const BpPairArgs &pa, PairSmem &sm, uint32_t &phase, int tile, int m_begin,
                                             int m_end, int slot, bool whole) {
    const BpArgs &a = pa.b;
    const TileInfo &ti = a.tiles[tile];
    const int *oidx = a.out_idx + (long long)tile * kTilePx + threadIdx.x;
    float dx[kPxPerThread], dy[kPxPerThread], hd2[kPxPerThread], fdi[kPxPerThread];
    float acc_re[kPxPerThread], acc_im[kPxPerThread];
#pragma unroll
    for (int j = 0; j < kPxPerThread; ++j) {
        const float2 d = a.pix[(long long)tile * kTilePx + threadIdx.x + j * kBpThreads];
        dx[j] = d.x;
        dy[j] = d.y;
        hd2[j] = 0.5f * fmaf(d.x, d.x, d.y * d.y);
        fdi[j] = 0.f;
        const int o = FD ? oidx[j * kBpThreads] : -1;
        if (FD && o >= 0) {
            // out-of-bound offsets: left out of this call and flagged
            const float f = a.fdopp[o];
            if (fabsf(f) <= a.fd_max)
                fdi[j] = f;
            else
                atomicOr(a.err, kErrDopplerBound);
        }
        acc_re[j] = 0.f;
        acc_im[j] = 0.f;
    }
    sm.l = pair_layout(pa, ti, m_end - m_begin, pulse_unroll<RG, MULTI>());
    const bool axis = !pa.call[1];
    const int Mt = sm.l.Mt, slots = sm.l.slots;
    const int nb = (m_end - m_begin + Mt - 1) / Mt;
    auto start = [&](int b) { return m_begin + b * Mt; };
    auto count = [&](int b) { return min(Mt, m_end - m_begin - b * Mt); };

    // Pipeline: Tx records two blocks ahead, Rx records and window copies one
    // block ahead, one barrier per block.  The exact-loop bits of a Tx slot
    // are cleared at the end of the iteration that computes its block.
    prep_tx(pa, sm, ti, start(0), count(0), 0, 0);
    if (nb > 1) prep_tx(pa, sm, ti, start(1), count(1), 1, 2);
    // the previous tile's records may lie where bulk copies write now
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncthreads();
    unsigned x_cur = *sm.exact(0), x_next = nb > 1 ? *sm.exact(1) : 0;
    if (!x_cur) stage_windows<MULTI, RG>(pa, sm, start(0), count(0), 0, 0, 0, 0);
    prep_rx<MULTI, RG>(pa, sm, ti, start(0), count(0), 0, 0, x_cur);
    if (x_cur) {  // window starts of the exact loop come from its Rx records
        __syncthreads();
        stage_windows<MULTI, RG>(pa, sm, start(0), count(0), 0, 0, 0, x_cur);
    }
    __syncthreads();
    int s = 0, t = 0, rt = 0;  // Tx slot b % 3, table slot b % slots, Rx slot b % 2
    for (int b = 0; b < nb; ++b) {
        const int s1 = s == 2 ? 0 : s + 1, s2 = s == 0 ? 2 : s - 1;
        const int t1 = slots == 2 ? t ^ 1 : 0, rt1 = rt ^ 1;
        const bool more = b + 1 < nb;
        if (more) {
            if (slots == 2 && !x_next) stage_windows<MULTI, RG>(pa, sm, start(b + 1), count(b + 1), s1, t1, rt1, 0);
            if (b + 2 < nb) prep_tx(pa, sm, ti, start(b + 2), count(b + 2), s2, 2 * b + 4);
            prep_rx<MULTI, RG>(pa, sm, ti, start(b + 1), count(b + 1), s1, rt1, x_next);
            if (slots == 2 && x_next) {  // block-uniform
                __syncthreads();
                stage_windows<MULTI, RG>(pa, sm, start(b + 1), count(b + 1), s1, t1, rt1, x_next);
            }
        }
        if (!mbar_wait(sm.bar(t), (phase >> t) & 1u, pa.polls)) {
            *sm.stall() = 1 << (b & 1);
            atomicOr(a.err, kErrStall);
        }
        phase ^= 1u << t;
        const int m0 = start(b), np = count(b);
        for (int p = 0; p < np;) {
            int pe = np;
            bool exact = false;
            if (x_cur) {  // block-uniform: the run that holds pulse p
                const int r = run_of(pa, m0, p);
                exact = (x_cur >> r) & 1u;
                pe = min(np, (fast_div(m0, pa.div_blk) + r + 1) * a.Mb - m0);
            }
            if (exact)
                run_exact<RG, FD>(a, sm, p, pe, s, t, rt, dx, dy, hd2, fdi, acc_re, acc_im);
            else if (axis)
                run_expand<RG, MULTI, FD, true>(a, sm, p, pe, s, t, rt, dx, dy, hd2, fdi, acc_re, acc_im);
            else
                run_expand<RG, MULTI, FD, false>(a, sm, p, pe, s, t, rt, dx, dy, hd2, fdi, acc_re, acc_im);
            p = pe;
        }
        if (threadIdx.x == 0) *sm.exact(s) = 0;  // free for block b + 3
        __syncthreads();
        if ((*sm.stall() >> (b & 1)) & 1) {
            // the call gives up and is flagged; this CTA's remaining work is
            // left out.  Its copies in flight write into its shared memory, so
            // they are waited for (bounded) before it goes away.
            mbar_wait(sm.bar(t), ((phase >> t) & 1u) ^ 1u, kWaitPolls);
            if (more && slots == 2) mbar_wait(sm.bar(t1), (phase >> t1) & 1u, kWaitPolls);
            return false;
        }
        if (slots == 1 && more) stage_windows<MULTI, RG>(pa, sm, start(b + 1), count(b + 1), s1, t1, rt1, x_next);
        x_cur = x_next;
        x_next = b + 2 < nb ? *sm.exact(s2) : 0;
        s = s1;
        t = t1;
        rt = rt1;
    }

    if (FD) {
        // the Doppler offset moved the index, not the phase: undo its share
#pragma unroll
        for (int j = 0; j < kPxPerThread; ++j) {
            float cyc = a.beta * fdi[j];
            cyc -= rintf(cyc);
            float sn, cs;
            sincospif(-2.0f * a.sign * cyc, &sn, &cs);
            float re = acc_re[j] * cs - acc_im[j] * sn;
            float im = acc_re[j] * sn + acc_im[j] * cs;
            const int o = oidx[j * kBpThreads];
            if (o >= 0 && !(fabsf(a.fdopp[o]) <= a.fd_max)) re = im = 0.f;
            acc_re[j] = re;
            acc_im[j] = im;
        }
    }

    if (!whole) {
        // this CTA's share of a split tile; the last warp to arrive for these
        // 128 pixels adds all shares
        float2 *dst = a.partial + (long long)slot * kTilePx + threadIdx.x;
#pragma unroll
        for (int j = 0; j < kPxPerThread; ++j) __stcg(dst + j * kBpThreads, make_float2(acc_re[j], acc_im[j]));
        if (!sum_split_tile(a, pa.arrived, tile, acc_re, acc_im)) return true;
    }
#pragma unroll
    for (int j = 0; j < kPxPerThread; ++j) {
        const int o = oidx[j * kBpThreads];
        if (o < 0) continue;
        float2 v = make_float2(acc_re[j], acc_im[j]);
        if (a.accumulate) {
            const float2 prev = a.image[o];
            v.x += prev.x;
            v.y += prev.y;
        }
        a.image[o] = v;
        if (a.image_out) a.image_out[o] = v;
    }
    return true;
}

// MULTI: more Rx channels than one group (otherwise R == RG, known at compile
// time).  MINB: CTAs per SM the register budget is sized for.
template <int RG, bool MULTI, bool FD, int MINB>
__global__ void __launch_bounds__(kBpThreads, MINB)
    backproject_pairs_kernel(const __grid_constant__ BpPairArgs pa) {
    extern __shared__ __align__(128) unsigned char smem_bpp[];
    const BpArgs &a = pa.b;
    PairSmem sm;
    sm.base = smem_bpp;
    sm.addr = (uint32_t)__cvta_generic_to_shared(smem_bpp);
    if (threadIdx.x == 0) {
        mbar_init(sm.bar(0));
        mbar_init(sm.bar(1));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (threadIdx.x < 4) reinterpret_cast<int *>(smem_bpp)[4 + threadIdx.x] = 0;  // exact-loop bits, stall bits
    __syncthreads();
    uint32_t phase = 0;
    const long long u0 = (long long)blockIdx.x * a.units / a.G;
    const long long u1 = (long long)(blockIdx.x + 1) * a.units / a.G;
    const int PB = a.blocks_per_tile;
    const int t_first = (int)(u0 / PB);
    long long u = u0;
    while (u < u1) {
        const int tile = (int)(u / PB);
        const int b0 = (int)(u - (long long)tile * PB);
        const int b1 = (int)min((long long)PB, (long long)b0 + (u1 - u));
        if (!pair_segment<RG, MULTI, FD>(pa, sm, phase, tile, b0 * kPairUnit, min(a.M, b1 * kPairUnit),
                                         (int)blockIdx.x * a.seg_max + (tile - t_first), b0 == 0 && b1 == PB))
            return;
        u += b1 - b0;
    }
}

// (A, D) pairs of every profile row: A = S_k, D = (S_{k+1} exp(-sign j 2 pi
// beta) - S_k) / kappa (see convert_block in backproject.cu); one warp per
// row, 16 bytes written per bin.  The warp of a pulse's first row also takes
// the pulse's Rx offsets o = q_rx - q_tx (FP64 differences, FP32 values), their
// largest square, and into call[0], call[1] (zero before the launch) the FP32
// bits of the call's largest |o| and whether any o has a y component.  The
// launch also zeroes the arrival counters of the call's split tiles.
template <bool FP16>
__global__ void __launch_bounds__(256) expand_pairs_kernel(ExpandArgs e) {
    for (int i = blockIdx.x * 256 + threadIdx.x; i < e.n_arrived; i += gridDim.x * 256) e.arrived[i] = 0;
    __shared__ unsigned call_sh[2];
    if (threadIdx.x < 2) call_sh[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = blockIdx.x * 8 + warp;
    if (row < e.rows) {
        const int m = row / e.R;
        if (row == m * e.R) {
            const double2 qt = reinterpret_cast<const double2 *>(e.q_tx)[m];
            float o2max = 0.f;
            bool off = false;
            for (int r = lane; r < e.R; r += 32) {
                const double2 qr = reinterpret_cast<const double2 *>(e.q_rx)[row + r];
                const float ox = (float)(qr.x - qt.x), oy = (float)(qr.y - qt.y);
                const float o2 = fmaf(ox, ox, oy * oy);
                e.rx[row + r] = make_float4(ox, oy, o2, fabsf(oy) <= 1e-9f ? o2 : INFINITY);
                o2max = fmaxf(o2max, o2 < INFINITY ? o2 : INFINITY);  // NaN: out of the expansion loop's reach
                off |= !(fabsf(oy) <= 1e-9f);
            }
            o2max = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(o2max)));  // o2 >= 0
            off = __any_sync(0xffffffffu, off);
            if (lane == 0) {
                e.o2max[m] = o2max;
                atomicMax(call_sh, __float_as_uint(sqrtf(o2max) * 1.000001f));  // may be infinite
                if (off) call_sh[1] = 1;
            }
        }
        const float sc = FP16 ? __ldg(e.scales + row) : 1.0f;
        const float2 *s32 = reinterpret_cast<const float2 *>(e.prof) + (long long)row * e.n_bins;
        const __half2 *s16 = reinterpret_cast<const __half2 *>(e.prof) + (long long)row * e.n_bins;
        float4 *dst = e.pairs + (long long)row * e.n_bins;
        auto load = [&](int i) {
            if (!FP16) return s32[i];
            const float2 f = __half22float2(s16[i]);
            return make_float2(f.x * sc, f.y * sc);
        };
#pragma unroll 4
        for (int i = lane; i < e.n_bins - 1; i += 32) {
            const float2 s0 = load(i), s1 = load(i + 1);
            const float dre = fmaf(s1.x, e.cb_k.x, fmaf(-s1.y, e.cb_k.y, -s0.x * e.inv_kappa));
            const float dim = fmaf(s1.x, e.cb_k.y, fmaf(s1.y, e.cb_k.x, -s0.y * e.inv_kappa));
            dst[i] = make_float4(s0.x, s0.y, dre, dim);
        }
    }
    __syncthreads();
    if (threadIdx.x < 2) atomicMax(e.call + threadIdx.x, call_sh[threadIdx.x]);
}

template <int RG, bool MULTI>
void *pair_kernel(bool fd, int minb) {
    if (fd) return minb == 3 ? (void *)backproject_pairs_kernel<RG, MULTI, true, 3>
                             : (void *)backproject_pairs_kernel<RG, MULTI, true, 2>;
    return minb == 3 ? (void *)backproject_pairs_kernel<RG, MULTI, false, 3>
                     : (void *)backproject_pairs_kernel<RG, MULTI, false, 2>;
}

void *select_pair_kernel(int rg, bool multi, bool fd, int minb) {
    switch (rg) {
        case 1: return multi ? pair_kernel<1, true>(fd, minb) : pair_kernel<1, false>(fd, minb);
        case 2: return multi ? pair_kernel<2, true>(fd, minb) : pair_kernel<2, false>(fd, minb);
        case 3: return multi ? pair_kernel<3, true>(fd, minb) : pair_kernel<3, false>(fd, minb);
        case 4: return multi ? pair_kernel<4, true>(fd, minb) : pair_kernel<4, false>(fd, minb);
    }
    return nullptr;
}

}  // namespace

// Shared memory that holds one pulse of R windows of L entries in one table.
size_t bp_pairs_min_smem(int R, int L) {
    return kHeaderBytes + (size_t)R * L * 16 + pair_const_bytes(R);
}

cudaError_t bp_pairs_prepare(int rg, int R, size_t smem, int minb, int *ctas_per_sm) {
    *ctas_per_sm = 0;
    for (int fd = 0; fd < 2; ++fd) {
        void *k = select_pair_kernel(rg, R > rg, fd != 0, minb);
        if (!k) return cudaErrorInvalidValue;
        // process-wide attribute shared by all plans: raised to the most any may use
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kBpThreads, smem);
        if (e != cudaSuccess) return e;
        *ctas_per_sm = fd ? std::min(*ctas_per_sm, n) : n;
    }
    return cudaSuccess;
}

cudaError_t launch_backproject_pairs(const BpPairArgs &pa, const ExpandArgs &e, const BpLaunch &l, cudaStream_t s) {
    if (pa.b.units == 0) return cudaSuccess;
    void *k = select_pair_kernel(l.rg, pa.b.R > l.rg, pa.b.fdopp != nullptr, l.minb);
    if (!k) return cudaErrorInvalidValue;
    const unsigned blocks = (unsigned)((e.rows + 7) / 8);
    if (l.fp16)
        expand_pairs_kernel<true><<<blocks, 256, 0, s>>>(e);
    else
        expand_pairs_kernel<false><<<blocks, 256, 0, s>>>(e);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    BpPairArgs args = pa;
    void *params[] = {&args};
    return cudaLaunchKernel(k, dim3(args.b.G), dim3(kBpThreads), params, l.smem, s);
}

}  // namespace sar
