// channelize_correct_impl.cuh -- kernels and launch templates of the fused
// F-stage; compiled once per sample format (channelize_correct_ci16.cu,
// _ci8.cu, _ci4.cu, in parallel), dispatched by channelize_correct.cu.
#pragma once
//
// The F-stage and the delay/bandpass correction in one
// pass: raw int16/int8 samples in, corrected operands in the X-stage layout
// out, with no channelised intermediate in HBM.
//
// Paper, Sec. "Signal processing with GPU kernels": FIR and FFT channelise
// each subband, then fine delay compensation and bandpass correction end the
// per-station processing and transpose on write-back so the correlator reads
// all stations of a channel together. The paper runs these as separate
// kernels through device memory; fusing them removes the write and re-read of
// the channelised block (8 + 8 bytes per complex sample).
//
// The FIR and FFT are those of ppf.cu (register sliding-window FIR, two-pass
// in-register FFT). After FFT pass 2 each output X(n, p, s, k) is multiplied
// by bandpass(n, k) * gain(n, p) * exp(i phi), phi = phi0(n, k) + s * step(n, k)
// (phi0 reduced mod 2 pi and step formed in FP64 by the phase-table kernel,
// as in fx_correct); exp(i phi) is evaluated in FP32 after a reduction to
// [-pi, pi] with a two-constant Cody-Waite split of 2 pi, then __sincosf
// (absolute error about 4e-7 on that interval), once per (station, channel,
// spectrum) and shared by the two pols.
//
// Kernels (all write zeros for spectra past the block's end):
//   ppf_correct_ws_kernel     C = 16, 64, every output form: FIR and FFT on
//                             separate warps, pass 2 with lane = transform row
//                             so a warp store is one 256-byte run of the FP32
//                             spectrum-blocked layout [SB][C][ceil16(S)/16][N][16][2]
//                             or 2 inputs x 16 spectra of a planar plane;
//   ppf_correct_ws256_kernel  C = 256: one CTA per (station, pol), pass 2 with
//                             a thread per two spectra.
// Planar outputs are [SB][C][planes][I_pad][S_pad] (FP16/BF16 x operand_scale,
// hi/lo FP16, or FP32 for the TF32-split X-stage); planar_pad zeroes what the
// F-stage does not write (inputs I..I_pad, spectra past the last round).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "fft_reg.cuh"
#include "internal.h"
#include "ppf_common.cuh"

namespace fxi {
namespace {

using namespace ppf;

// OUT: 1 FP32 spectrum-blocked, 2 FP16 planar, 3 BF16 planar, 4 split FP16 planar, 5 FP32 planar.
// two values as 16-bit operands (OUT 3 BF16, else FP16), the first in the low half
template <int OUT>
__device__ __forceinline__ unsigned pack16(float a, float b)
{
    if constexpr (OUT == 3) {
        const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<const unsigned *>(&v);
    } else {
        const __half2 v = __floats2half2_rn(a, b);
        return *reinterpret_cast<const unsigned *>(&v);
    }
}

// lo parts of split FP16: x - hi rounded to FP16, hi = pack16's halves
__device__ __forceinline__ unsigned pack16_lo(float a, float b, unsigned hi)
{
    const float2 h = __half22float2(*reinterpret_cast<const __half2 *>(&hi));
    return pack16<4>(a - h.x, b - h.y);
}

// Two adjacent spectra of one (channel, input) into the planar planes, o = the
// offset of the first in plane 0 (OUT 2 FP16, 3 BF16, 4 split FP16, 5 FP32).
template <int OUT>
__device__ __forceinline__ void store_planar(void *corr, long long o, long long pstride, float2 ya, float2 yb)
{
    if constexpr (OUT == 5) {
        float *out = reinterpret_cast<float *>(corr) + o;
        *reinterpret_cast<float2 *>(out) = make_float2(ya.x, yb.x);
        *reinterpret_cast<float2 *>(out + pstride) = make_float2(ya.y, yb.y);
    } else {
        unsigned short *out = reinterpret_cast<unsigned short *>(corr) + o;
        const unsigned re = pack16<OUT>(ya.x, yb.x), im = pack16<OUT>(ya.y, yb.y);
        *reinterpret_cast<unsigned *>(out) = re;
        *reinterpret_cast<unsigned *>(out + pstride) = im;
        if constexpr (OUT == 4) {
            *reinterpret_cast<unsigned *>(out + 2 * pstride) = pack16_lo(ya.x, yb.x, re);
            *reinterpret_cast<unsigned *>(out + 3 * pstride) = pack16_lo(ya.y, yb.y, im);
        }
    }
}

// ---------------------------------------------------------------------------
// Warp-specialised fused kernel, FP32 output (C = 16, 64). As ppf_ws_kernel:
// 128 FIR threads (NPC = 64 / C stations) and 128 FFT threads per CTA, FIR
// round b -> rows u[b & 1] -> FULL[b & 1]; FFT round b -> EMPTY[b & 1] for FIR
// round b + 2. Three further choices keep the shared-memory/L1 pipe (which
// also carries the global stores) below saturation:
//  * rows are input-major (row = input * 16 + spectrum, each input's 16 rows
//    offset by 8 entries so the FIR stores of the two pols use different banks);
//    pass 1 (R lanes per row, as in ppf_ws_kernel) writes its results
//    transposed, P1[k1][n2][row] with row stride NTR + 16/R (conflict free),
//    over u[b & 1] once every FFT thread has read its rows (barrier FFT);
//  * pass 2 runs with lane = row: a warp takes (group of 32 rows, k1) items,
//    so each output store of a warp is one station's 16 spectra x 2 pols of
//    one channel, 256 contiguous bytes of the spectrum-blocked layout;
//  * the FIR threads, which have the lighter share of the work, multiply
//    their FIR output by the input's complex gain x operand scale (the FFT is
//    linear, so this equals multiplying its output) and tabulate
//    bandpass x exp(i phi) x flag per (station, channel, spectrum) of their
//    round into a double-buffered table (one __sincosf per owner and round,
//    then rotations by exp(2 i step)); the FFT threads multiply each output
//    by that one factor.
template <int C>
struct FusedWsCfg {
    static constexpr int R = PpfCfg<C>::R;
    static constexpr int NPC = 64 / C;
    static constexpr int NF = NPC * C * kPols;           // 128 FIR threads, 128 FFT threads
    static constexpr int IC = NPC * kPols;               // inputs of a CTA
    static constexpr int NTR = IC * kRound;              // rows per round
    static constexpr int ROW = PpfCfg<C>::ROW;
    static constexpr int PADG = 8;                       // float2 offset per input (16 rows)
    static constexpr int USZ = NTR * ROW + IC * PADG;    // one row buffer
    static constexpr int RS = NTR + 16 / R;              // P1 row stride
    static constexpr int EJ = kRound + 2;                // phase table: 16 spectra + pad (even: 16-byte pairs)
    static constexpr int ESZ = NPC * C * EJ;             // one phase-table buffer
    static constexpr int ITEMS = (NTR / 32) * (R / 2);   // pass-2 items (row group, pair of k1)
    static_assert(C == 16 || C == 64, "warp-specialised fused kernel: C = 16 or 64");
    static_assert(R * R * RS <= USZ, "P1 fits over the row buffer");
    static_assert(ITEMS % 4 == 0 && NTR % 32 == 0, "four FFT warps share the pass-2 items");
};

template <int C, typename TIn>
constexpr size_t fused_ws_smem_bytes()
{
    using W = FusedWsCfg<C>;
    return (size_t)C * sizeof(float2) + 2ull * kRound * W::NPC * C * kPols * sizeof(TIn) +
           (2ull * W::USZ + 2ull * W::ESZ) * sizeof(float2) + 16;   // + 2 mbarriers
}

// CTAs per SM the shared memory allows: 3 at C = 64, 2 at C = 16 (four stations' rows)
template <int C, typename TIn>
constexpr int fused_ws_ctas()
{
    return 3 * (fused_ws_smem_bytes<C, TIn>() + 1024) <= 228 * 1024 ? 3 : 2;
}


// OUT: 1 FP32 spectrum-blocked, 2 FP16 / 3 BF16 / 4 split
// FP16 / 5 FP32 planar ([SB][C][planes][I_pad][s_out], x scale for 2-4).
template <int C, int T, typename TIn, int OUT>
__global__ void __launch_bounds__(2 * FusedWsCfg<C>::NF, fused_ws_ctas<C, TIn>())
ppf_correct_ws_kernel(const TIn *__restrict__ raw, void *__restrict__ corr, const float *__restrict__ taps,
                      const float2 *__restrict__ twiddle, const float2 *__restrict__ phase,
                      const float *__restrict__ bandpass, const float2 *__restrict__ gains, int N, int S, int I_pad,
                      int s_out, float scale, int rounds_per_cta, const float *__restrict__ flags, int s_base,
                      int s_end, int *__restrict__ status, long long budget, int no_loads)
{
    using W = FusedWsCfg<C>;
    constexpr int R = W::R, NPC = W::NPC, NF = W::NF, ROW = W::ROW, PADG = W::PADG, USZ = W::USZ;
    constexpr int RS = W::RS, EJ = W::EJ, ESZ = W::ESZ;
    constexpr int ROW_BYTES = C * kPols * (int)sizeof(TIn);
    constexpr int BUF_BYTES = kRound * NPC * ROW_BYTES;
    constexpr int ALL = 2 * NF;
    static_assert(ROW_BYTES % 16 == 0, "rows must be whole 16-byte chunks");
    static_assert(2 * (fused_ws_smem_bytes<C, TIn>() + 1024) <= 228 * 1024, "at least two CTAs per SM");

    extern __shared__ __align__(16) unsigned char smem[];
    float2 *tw = reinterpret_cast<float2 *>(smem);
    unsigned char *inbuf = smem + C * sizeof(float2);
    float2 *u = reinterpret_cast<float2 *>(inbuf + 2 * BUF_BYTES);   // [2][USZ]
    float2 *et = u + 2 * USZ;                                         // [2][NPC][C][EJ]
    // raw-row mbarriers (one station per CTA: its rows arrive by bulk copy)
    const unsigned rbar = tc::smem_u32(et + 2 * ESZ);

    const int tid = threadIdx.x;
    const int sb = blockIdx.z;
    const int n0 = blockIdx.x * NPC;                // station groups fastest
    const int s0 = s_base + blockIdx.y * rounds_per_cta * kRound;
    const int rows_total = S + T - 1;
    const long long L = (long long)rows_total * C;
    const int nrounds = min(rounds_per_cta, (s_end - s0 + kRound - 1) / kRound);
    auto rowp = [&](float2 *uq, int r) { return uq + r * ROW + (r / kRound) * PADG; };

    for (int i = tid; i < C; i += ALL) tw[i] = twiddle[i];
    if constexpr (NPC == 1) {
        if (tid == 0) {
            tc::mbar_init(rbar, 1);
            tc::mbar_init(rbar + 8, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    }
    __syncthreads();

    if (tid < NF) {
        // ---------------- FIR threads: (station nl, channel c, pol p) ----------------
        // one station (C = 64): thread 0 moves each round's raw rows (one
        // contiguous run) with a bulk copy completing on rbar[buf]; several
        // stations (C = 16): 16-byte cp.async by all FIR threads
        const unsigned char *rows0 = reinterpret_cast<const unsigned char *>(raw) +
                                     (((long long)sb * N + n0) * L) * kPols * sizeof(TIn);
        auto issue = [&](int buf, int r0, int nrows) {
            if (tid == 0 && !no_loads) {            // no_loads: failure-detection test hook
                const int nv = max(0, min(nrows, rows_total - r0));
                bulk_rows_issue(inbuf + buf * BUF_BYTES, rows0 + (long long)r0 * ROW_BYTES,
                                (unsigned)(nv * ROW_BYTES), rbar + 8u * buf);
            }
        };
        auto stage = [&](int buf, int r0, int nrows) {
            const int chunks = nrows * ROW_BYTES / 16;
            for (int q = tid; q < NPC * chunks; q += NF) {
                const int st = q / chunks, ch = q - st * chunks;
                const int n = n0 + st;
                const int row_in = (ch * 16) / ROW_BYTES;
                const int byte_in_row = (ch * 16) - row_in * ROW_BYTES;
                unsigned char *dst = inbuf + buf * BUF_BYTES + (row_in * NPC + st) * ROW_BYTES + byte_in_row;
                const bool ok = (n < N) && (r0 + row_in < rows_total);
                const unsigned char *src = reinterpret_cast<const unsigned char *>(raw);
                if (ok) src += ((((long long)sb * N + n) * L + (long long)r0 * C) * kPols) * sizeof(TIn) + ch * 16;
                cp_async16(dst, src, ok ? 16 : 0);
            }
        };
        const int p = tid % kPols;
        const int c = (tid / kPols) % C;
        const int nl = tid / (kPols * C);
        // phase-table role: (station, channel) = tid mod NPC*C, spectra j0, j0 + 2, ...
        constexpr int OWN = NPC * C;                // = NF / 2
        const int own_nc = tid % OWN, own_j0 = tid / OWN;
        const int own_n = min(n0 + own_nc / C, N - 1);
        const float2 pst = phase[((long long)sb * N + own_n) * C + own_nc % C];   // (phi0, step)
        float sn2, cs2;
        sincosf(2.f * pst.y, &sn2, &cs2);           // exp(2 i step): this owner's spectra are 2 apart
        const float bpo = bandpass ? bandpass[(long long)own_n * C + own_nc % C] : 1.f;
        const int n_fir = min(n0 + nl, N - 1);
        const float2 gg = gains ? gains[n_fir * kPols + p] : make_float2(1.f, 0.f);
        const float2 gsc = make_float2(gg.x * scale, gg.y * scale);
        const float2 rot2 = make_float2(cs2, sn2);
        float2 h[T];
#pragma unroll
        for (int k = 0; k < T; ++k) h[k] = make_float2(taps[k * C + c], taps[k * C + c]);

        if constexpr (NPC == 1) {
            issue(1, s0, T - 1);                        // history rows: buffer 1, phase 0
            issue(0, s0 + T - 1, kRound);               // round 0: buffer 0, phase 0
            raw_wait(rbar + 8, 0, status, budget);
        } else {
            stage(1, s0, T - 1);
            cp_async_commit();
            stage(0, s0 + T - 1, kRound);
            cp_async_commit();
            cp_async_wait<1>();
            named_bar_sync(kBarRaw, NF);
        }
        float2 win[T];
        const TIn *in1 = reinterpret_cast<const TIn *>(inbuf + BUF_BYTES);
#pragma unroll
        for (int k = 0; k < T - 1; ++k) win[k] = to_f2(in1[k * NF + tid]);
        win[T - 1] = make_float2(0.f, 0.f);
        named_bar_sync(kBarRaw, NF);
        if constexpr (NPC == 1) {
            if (tid == 0) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (nrounds > 1) issue(1, s0 + T - 1 + kRound, kRound);    // round 1: buffer 1, phase 1
        } else {
            if (nrounds > 1) stage(1, s0 + T - 1 + kRound, kRound);
            cp_async_commit();
        }

        for (int b = 0; b < nrounds; ++b) {
            const int q = b & 1;
            const int sr = s0 + b * kRound;
            if constexpr (NPC == 1) {
                raw_wait(rbar + 8u * q, (unsigned)(((b + q) / 2) & 1), status, budget);   // round b's rows
            } else {
                cp_async_wait<1>();
                named_bar_sync(kBarRaw, NF);            // raw rows of round b are in
            }
            if (b >= 2) named_bar_sync(kBarEmpty + q, ALL);   // FFT threads are done with u[q], et[q]
            const TIn *in = reinterpret_cast<const TIn *>(inbuf + q * BUF_BYTES);
            float2 *uq = u + q * USZ;
            float2 *fo = rowp(uq, (nl * kPols + p) * kRound) + c;
            // four outputs at a time (four independent FMA chains); tap k of
            // output j takes the sample loaded at output j + k - (T - 1), so the
            // group's new samples stay in t[] until its outputs are formed
#pragma unroll
            for (int j0 = 0; j0 < kRound; j0 += 4) {
                float2 t[4], acc[4];
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    t[qq] = to_f2(in[(j0 + qq) * NF + tid]);
                    acc[qq] = make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int k = 0; k < T; ++k)
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq)
                        acc[qq] = __ffma2_rn(h[k], k >= T - 1 - qq ? t[qq + k - (T - 1)] : win[(j0 + qq + k) % T],
                                             acc[qq]);
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    fo[(j0 + qq) * ROW] = cmul(acc[qq], gsc);   // row (input, spectrum), times gain x scale
                    win[(T - 1 + j0 + qq) % T] = t[qq];
                }
            }
            // exp(i phi) x flag of this round: phi = phi0 + s step reduced to
            // [-pi, pi] (two-constant Cody-Waite split of 2 pi), then __sincosf
            // exp(i phi) at this owner's first spectrum of the round (re-anchored
            // every round), then rotations by exp(2 i step) for the next ones
            float2 *eq = et + q * ESZ + own_nc * EJ;
            float2 e;
            {
                const float phi = fmaf((float)(sr + own_j0), pst.y, pst.x);
                const float kq = rintf(phi * 0.15915494309189535f);
                float r = fmaf(-kq, 6.28125f, phi);
                r = fmaf(-kq, 1.9353071795864769e-3f, r);
                __sincosf(r, &e.y, &e.x);
                e.x *= bpo;
                e.y *= bpo;
            }
#pragma unroll
            for (int qq = 0; qq < kRound / 2; ++qq) {
                const int j = own_j0 + 2 * qq;
                const float fw = flags ? flags[(long long)own_n * S + min(sr + j, S - 1)] : 1.f;
                eq[j] = make_float2(e.x * fw, e.y * fw);
                e = cmul(e, rot2);
            }
            named_bar_arrive(kBarFull + q, ALL);
            named_bar_sync(kBarRaw, NF);                // every FIR thread has read raw buffer q
            if constexpr (NPC == 1) {
                if (tid == 0) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (b + 2 < nrounds) issue(q, s0 + T - 1 + (b + 2) * kRound, kRound);
            } else {
                if (b + 2 < nrounds) stage(q, s0 + T - 1 + (b + 2) * kRound, kRound);
                cp_async_commit();
            }
        }
        if constexpr (NPC != 1) cp_async_wait<0>();
    } else {
        // ---------------- FFT threads ----------------
        const int t = tid - NF;
        const int warp = t / 32, lane = t % 32;
        float2 twr[R];                              // W_C^(n2 k1), n2 = t mod R
#pragma unroll
        for (int k1 = 1; k1 < R; ++k1) twr[k1] = tw[(t % R) * k1];
        const int NB = s_out / kRound;
        const int I = N * kPols;
        constexpr int P1ITERS = W::NTR * R / NF;
        for (int b = 0; b < nrounds; ++b) {
            const int q = b & 1;
            const int sr = s0 + b * kRound;
            float2 *uq = u + q * USZ;
            const float2 *eq = et + q * ESZ;
            named_bar_sync(kBarFull + q, ALL);          // FIR round b is in u[q], et[q]
            // pass 1: R-point FFTs over n1 (stride R), times W_C^(n2 k1)
            float2 v1[P1ITERS][R];
#pragma unroll
            for (int it = 0; it < P1ITERS; ++it) {
                const int task = it * NF + t;
                const float2 *row = rowp(uq, task / R);
#pragma unroll
                for (int n1 = 0; n1 < R; ++n1) v1[it][n1] = row[R * n1 + task % R];
                fft_reg<R>(v1[it]);
#pragma unroll
                for (int k1 = 1; k1 < R; ++k1) v1[it][k1] = cmul(v1[it][k1], twr[k1]);
            }
            named_bar_sync(kBarFft, NF);                // every FFT thread has read its rows of u[q]
#pragma unroll
            for (int it = 0; it < P1ITERS; ++it) {
                const int task = it * NF + t;
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) uq[(k1 * R + task % R) * RS + task / R] = v1[it][k1];
            }
            named_bar_sync(kBarFft, NF);                // P1 complete
            // pass 2: a half-warp per k1 (two k1 per item), each lane two adjacent
            // rows (input il, spectra j and j + 1), so the rows and the phase
            // factors come in 16-byte loads and the planar stores go out in pairs
#pragma unroll
            for (int it = 0; it < W::ITEMS / 4; ++it) {
                const int item = warp + 4 * it;
                const int g = item / (R / 2), k1 = 2 * (item % (R / 2)) + lane / 16;
                const int r = 32 * g + 2 * (lane % 16);
                const int il = r / kRound, j = r % kRound;
                float2 va[R], vb[R];
#pragma unroll
                for (int m = 0; m < R; ++m) {
                    const float4 w = *reinterpret_cast<const float4 *>(uq + (k1 * R + m) * RS + r);
                    va[m] = make_float2(w.x, w.y);
                    vb[m] = make_float2(w.z, w.w);
                }
                fft_reg<R>(va);
                fft_reg<R>(vb);
                const float2 *e = eq + ((il / kPols) * C) * EJ + j;
#pragma unroll
                for (int k2 = 0; k2 < R; ++k2) {
                    const int kout = k1 + R * ((k2 + R / 2) % R);
                    const float4 f = *reinterpret_cast<const float4 *>(e + kout * EJ);
                    va[k2] = cmul(va[k2], make_float2(f.x, f.y));
                    vb[k2] = cmul(vb[k2], make_float2(f.z, f.w));
                }
                if (it == W::ITEMS / 4 - 1 && b + 2 < nrounds) named_bar_arrive(kBarEmpty + q, ALL);
                const int s = sr + j, i = 2 * n0 + il;
                if (sr + kRound > s_end) {                  // only in the block's last round
#pragma unroll
                    for (int k2 = 0; k2 < R; ++k2) {
                        if (s >= s_end) va[k2] = make_float2(0.f, 0.f);
                        if (s + 1 >= s_end) vb[k2] = make_float2(0.f, 0.f);
                    }
                }
                if (i < I) {
                    if constexpr (OUT == 1) {
                        // one warp store = one station's 16 spectra x 2 pols of two channels
                        float2 *out = reinterpret_cast<float2 *>(corr) +
                                      ((((long long)sb * C) * NB + (sr - s_base) / kRound) * N + (i >> 1)) *
                                          (2 * kRound) + j * 2 + (i & 1);
                        const long long kstride = (long long)NB * N * (2 * kRound);
#pragma unroll
                        for (int k2 = 0; k2 < R; ++k2) {
                            const int kout = k1 + R * ((k2 + R / 2) % R);
                            out[kout * kstride] = va[k2];
                            out[kout * kstride + 2] = vb[k2];
                        }
                    } else {
                        // planar: one warp store = 2 inputs x 16 spectra of two (channel, plane)
                        constexpr int planes = OUT == 4 ? 4 : 2;
                        const long long pstride = (long long)I_pad * s_out;
                        const long long base = (long long)sb * C * planes * pstride + (long long)i * s_out + (s - s_base);
#pragma unroll
                        for (int k2 = 0; k2 < R; ++k2) {
                            const int kout = k1 + R * ((k2 + R / 2) % R);
                            const float2 ya = va[k2], yb = vb[k2];
                            const long long o = base + (long long)kout * planes * pstride;
                            store_planar<OUT>(corr, o, pstride, ya, yb);
                        }
                    }
                }
            }
        }
    }
}

// Zero the padding of the planar layout that the fused kernel does not cover:
// inputs [I, I_pad) and spectra [S16, s_out) of every (subband, channel, plane),
// one plane per block in 16-byte stores. Bound by the bytes written: a plane's
// padded inputs are one contiguous run (rows are in_row 16-byte words), the
// padded spectra `gap` words at the end of each other row. 50 stations, 6144
// channels, 700 spectra, split FP16 (415 MB of zeros): 59 us; a 64-thread block
// per row, most of them with nothing to write, took 1382 us.
__global__ void __launch_bounds__(256) planar_pad_kernel(uint4 *__restrict__ corr, int I, int I_pad, int in_row, int gap)
{
    uint4 *plane = corr + (long long)blockIdx.x * I_pad * in_row;
    const int tail = (I_pad - I) * in_row;
    for (int q = threadIdx.x; q < tail; q += blockDim.x) plane[(long long)I * in_row + q] = make_uint4(0, 0, 0, 0);
    for (int q = threadIdx.x; q < I * gap; q += blockDim.x) {
        const int row = q / gap;
        plane[(long long)row * in_row + (in_row - gap) + (q - row * gap)] = make_uint4(0, 0, 0, 0);
    }
}

// ---------------------------------------------------------------------------
// Warp-specialised fused kernel for C = 256:
// one CTA per (station, pol) and SM, 256 FIR threads (one channel each) and 256
// FFT threads in two groups of 128. A round's rows (16 spectra of one input) fit
// twice in shared memory at this channel count only per input; the CTAs of a
// station's two pols are neighbours in the grid and read the same raw rows (the
// second read mostly from L2). FIR round b -> u[b % NB] -> FULL[b % NB]; FFT group
// g takes the rounds b = g mod 2 with its own named barrier, so two rounds are in
// FFT at once.
//
// What bounds it: the FMA pipe with the register reads of its packed FMAs. The
// FIR alone (16 warps, nothing else running) takes 2.0 ms of the 8-bit case below,
// 0.64 of the pipe's rate in every instruction order tried, and the FFT's adds and
// multiplies 1.4 ms at full rate, 3.4 ms together; more warps (20, 24) gain
// nothing. So the design saves instructions and shared-memory traffic:
//  * FP32 and split FP16: the phase factors come from the channel axis. f_k is
//    linear in k, so for a spectrum s exp(i phi(k, s)) = e(k1, s) r(s)^m for
//    k = k1 + 128 + 16 m: the FIR threads put one anchor e (16 x 16 per round,
//    each the gain, flag and scale times one sine and cosine) into a table, the
//    phase-table kernel has left r(s) = exp(2 pi i (fs / 16) tau(s)) per station
//    and spectrum, and an FFT thread steps from its anchor up and down eight
//    channels each in registers.
//  * FP16 and BF16 (TIME): one factor per channel and spectrum, an anchor per
//    channel and round rotated along time by the channel's FIR thread. The two
//    ways differ by 3e-7, as little as either from the exact factor, but in a
//    16-bit operand that flips a rounding now and then, and a beam voltage, which
//    averages nothing, then moves by a unit of the operand (4e-5 normwise in
//    BF16): what users of these precisions have stored would no longer come out
//    again. It costs a 37 KB table per buffer, hence two row buffers, and 4.38 ms
//    instead of 4.01 in the 8-bit case below. The chain of rotations stands beside
//    the second half of the FIR, and the table is freed after the row buffer (in
//    one piece before the FIR, and freed with it: 4.47 ms).
//  * pass 1 (row = 16 lanes) writes its results transposed, P1[k1][n2][row] over
//    u[g] after the group's barrier; in pass 2 a thread takes two adjacent
//    spectra of one k1, so P1 rows come in 16-byte loads and planar values leave
//    in pairs (a warp store is 4 x 32 bytes of rows, FP32 4 x 64).
//  * strides: FIR rows 264 (two rows' halves fall on both halves of the banks in
//    pass 1), P1 rows 18 (even, for the 16-byte loads; eight n2 x two rows of a
//    store on distinct banks).
// 64 stations, 61 subbands of int8, 768 spectra, before this form -> now: FP32
// planes 4.44 -> 4.13 ms (3.7 TB/s of raw rows and operands), FP16 4.45 -> 4.38
// ms,
// spectrum-blocked FP32 10.97 -> 4.86 ms (FIR and FFT alternating on the same
// threads of a CTA for both pols). With
// anchors, two row buffers instead of four took 4.34 for 4.16 ms, four FIR
// outputs at a time instead of eight 4.16 for 4.01.
template <int OUT>
struct Ws256 {
    static constexpr bool TIME = OUT == 2 || OUT == 3;              // factors along time (16-bit operands)
    static constexpr int C = 256, R = 16;
    static constexpr int NF = C, NG = 128;              // FIR threads; FFT threads of a group
    static constexpr int ALL = NF + 2 * NG;
    static constexpr int ROW = C + 8;                   // FIR row stride (float2)
    static constexpr int RS = kRound + 2;               // P1 row stride
    static constexpr int USZ = R * R * RS > kRound * ROW ? R * R * RS : kRound * ROW;   // one buffer: 16 rows, then P1
    static constexpr int TW = R + 2;                    // twiddle row: [n2][k1], even
    static constexpr int EJ = kRound + 2;               // row of a factor table (even, conflict-free in 16 bytes)
    static constexpr int ESZ = TIME ? C * EJ : R * kRound;   // factors [channel][spectrum], or anchors [k1][spectrum]
    static constexpr int NB = TIME ? 2 : 4;             // row buffers
};

template <typename TIn, int OUT>
constexpr size_t ws256_smem_bytes()
{
    using W = Ws256<OUT>;
    return 2ull * kRound * W::C * kPols * sizeof(TIn) +
           ((size_t)W::NB * (W::USZ + W::ESZ) + (size_t)W::R * W::TW) * sizeof(float2) + W::C * sizeof(float2) + 16;   // + 2 mbarriers
}

__device__ __forceinline__ float2 conj2(float2 a) { return make_float2(a.x, -a.y); }

template <int T, typename TIn, int OUT>
__global__ void __launch_bounds__(Ws256<OUT>::ALL, 1)
ppf_correct_ws256_kernel(const TIn *__restrict__ raw, void *__restrict__ corr, const float *__restrict__ taps,
                         const float2 *__restrict__ twiddle, const float2 *__restrict__ phase,
                         const float2 *__restrict__ ratio, const float *__restrict__ bandpass,
                         const float2 *__restrict__ gains, int N, int S, int I_pad, int s_out, float scale,
                         int rounds_per_cta, const float *__restrict__ flags, int s_base, int s_end,
                         int *__restrict__ status, long long budget, int no_loads)
{
    using W = Ws256<OUT>;
    constexpr int C = W::C, R = W::R, NF = W::NF, ROW = W::ROW, USZ = W::USZ, RS = W::RS, TW = W::TW, ESZ = W::ESZ;
    constexpr bool TIME = W::TIME;
    constexpr int EJ = W::EJ;
    constexpr int ROW_BYTES = C * kPols * (int)sizeof(TIn);     // one raw time row of the station (both pols)
    constexpr int BUF_BYTES = kRound * ROW_BYTES;
    constexpr int NG = W::NG;
    constexpr int HAND = NF + NG;               // FULL / EMPTY: the FIR threads and one FFT group
    static_assert(ROW_BYTES % 16 == 0, "rows must be whole 16-byte chunks");
    static_assert(ws256_smem_bytes<TIn, OUT>() <= 227 * 1024, "one CTA per SM");

    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char *inbuf = smem;
    float2 *u = reinterpret_cast<float2 *>(inbuf + 2 * BUF_BYTES);   // [NB][USZ]
    float2 *et = u + W::NB * USZ;                                     // [NB][ESZ] factors or anchors
    float2 *tw = et + W::NB * ESZ;                                        // [n2][TW] W_C^(n2 k1)
    float2 *bpt = tw + R * TW;                                        // [k1][k2] bandpass of output k2, twice
    const unsigned rbar = tc::smem_u32(bpt + C);                      // raw-row mbarriers [2]
    const int tid = threadIdx.x;
    const int sb = blockIdx.z;
    const int n = blockIdx.x / kPols, p = blockIdx.x % kPols;       // (station, pol) fastest
    const int s0 = s_base + blockIdx.y * rounds_per_cta * kRound;
    const int rows_total = S + T - 1;
    const long long L = (long long)rows_total * C;
    const int nrounds = min(rounds_per_cta, (s_end - s0 + kRound - 1) / kRound);

    if (tid < C) {
        const int hi = tid / R, lo = tid % R;
        tw[hi * TW + lo] = twiddle[hi * lo];
        const float bp = bandpass ? bandpass[(long long)n * C + hi + R * ((lo + R / 2) % R)] : 1.f;
        bpt[tid] = make_float2(bp, bp);
    }
    if (tid == 0) {
        tc::mbar_init(rbar, 1);
        tc::mbar_init(rbar + 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    if (tid < NF) {
        // ---------------- FIR threads: channel c of input (n, p) ----------------
        // the station's raw rows of a round are one contiguous run: thread 0
        // moves it with a bulk copy completing on rbar[buf]
        const unsigned char *rows0 = reinterpret_cast<const unsigned char *>(raw) +
                                     (((long long)sb * N + n) * L) * kPols * sizeof(TIn);
        auto issue = [&](int buf, int r0, int nrows) {
            if (tid == 0 && !no_loads) {            // no_loads: failure-detection test hook
                const int nv = max(0, min(nrows, rows_total - r0));
                bulk_rows_issue(inbuf + buf * BUF_BYTES, rows0 + (long long)r0 * ROW_BYTES,
                                (unsigned)(nv * ROW_BYTES), rbar + 8u * buf);
            }
        };
        const int c = tid;
        // anchor role: channel k1 + 128 (k1 = c / 16) of spectrum c % 16 of a round
        const int aj = c % kRound;
        // (with factors along time: channel c, from the round's first spectrum on)
        const float2 pst = phase[((long long)sb * N + n) * C + (TIME ? c : C / 2 + c / kRound)];   // (phi0, step)
        const float2 gg = gains ? gains[n * kPols + p] : make_float2(1.f, 0.f);
        const float bpc = TIME && bandpass ? bandpass[(long long)n * C + c] : 1.f;
        const float2 gsc = make_float2(bpc * gg.x * scale, bpc * gg.y * scale);
        float2 rot = make_float2(1.f, 0.f);
        if constexpr (TIME) sincosf(pst.y, &rot.y, &rot.x);          // exp(i step)
        float2 h[T];
#pragma unroll
        for (int k = 0; k < T; ++k) h[k] = make_float2(taps[k * C + c], taps[k * C + c]);

        issue(1, s0, T - 1);                            // history rows: buffer 1, phase 0
        issue(0, s0 + T - 1, kRound);                   // round 0: buffer 0, phase 0
        raw_wait(rbar + 8, 0, status, budget);
        float2 win[T];
        const TIn *in1 = reinterpret_cast<const TIn *>(inbuf + BUF_BYTES);
#pragma unroll
        for (int k = 0; k < T - 1; ++k) win[k] = to_f2(in1[k * C * kPols + c * kPols + p]);
        win[T - 1] = make_float2(0.f, 0.f);
        named_bar_sync(kBarRaw, NF);
        if (tid == 0) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (nrounds > 1) issue(1, s0 + T - 1 + kRound, kRound);     // round 1: buffer 1, phase 1

        for (int b = 0; b < nrounds; ++b) {
            const int q = b & 1, ub = b % W::NB;
            const int sr = s0 + b * kRound;
            raw_wait(rbar + 8u * q, (unsigned)(((b + q) / 2) & 1), status, budget);   // round b's rows
            // anchor of this round: phi reduced to [-pi, pi] (two-constant Cody-Waite
            // split of 2 pi), sine and cosine, times gain, scale and flag. FX_F32 takes
            // sincosf: with __sincosf the eight steps from the anchor would leave the
            // block further from FP64 than one __sincosf per channel did (20 stations
            // x 700 spectra 3.28e-7, with anchors 3.44e-7, so 3.01e-7), and it is no slower
            // (the 8-bit case above 5.02 -> 4.86 ms)
            float2 e;
            {
                const float phi = fmaf((float)(TIME ? sr : sr + aj), pst.y, pst.x);
                const float kq = rintf(phi * 0.15915494309189535f);
                float r = fmaf(-kq, 6.28125f, phi);
                r = fmaf(-kq, 1.9353071795864769e-3f, r);
                if constexpr (OUT == 1) sincosf(r, &e.y, &e.x);
                else __sincosf(r, &e.y, &e.x);
            }
            e = cmul(gsc, e);
            if (!TIME && flags) {
                const float fw = flags[(long long)n * S + min(sr + aj, S - 1)];
                e = make_float2(e.x * fw, e.y * fw);
            }
            if (b >= W::NB) named_bar_sync(kBar256Empty + ub, HAND);
            if constexpr (!TIME) et[ub * ESZ + c] = e;
            const TIn *in = reinterpret_cast<const TIn *>(inbuf + q * BUF_BYTES);
            float2 *uq = u + ub * USZ;
            // eight outputs at a time, each sample's products one after the other: 4.01 ms
            // of the 8-bit case against 4.17 with four at a time tap by tap (the order
            // decides what the packed FMAs' operand reads can share: in a loop of nothing
            // else they run at 0.67 of the pipe's rate with no operand shared by neighbours,
            // 0.89 with the sample shared)
            constexpr int QN = 8;
#pragma unroll
            for (int j0 = 0; j0 < kRound; j0 += QN) {
                if constexpr (TIME) {
                    // the factors along time beside the second half's FMAs; their table is
                    // free later than the row buffer
                    if (j0 == QN) {
                        if (b >= W::NB) named_bar_sync(kBar256EmptyF + ub, HAND);
                        float4 *eq = reinterpret_cast<float4 *>(et + ub * ESZ + c * EJ);
#pragma unroll
                        for (int j = 0; j < kRound; j += 2) {
                            const float2 e1 = cmul(e, rot);
                            eq[j / 2] = make_float4(e.x, e.y, e1.x, e1.y);
                            e = cmul(e1, rot);
                        }
                    }
                }
                float2 t[QN], acc[QN];
#pragma unroll
                for (int qq = 0; qq < QN; ++qq) {
                    t[qq] = to_f2(in[(j0 + qq) * C * kPols + c * kPols + p]);
                    acc[qq] = make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int m = 0; m < T + QN - 1; ++m)
#pragma unroll
                    for (int qq = 0; qq < QN; ++qq) {
                        const int k = m - qq;                 // tap k of output qq meets sample m
                        if (k >= 0 && k < T)
                            acc[qq] = __ffma2_rn(h[k], m >= T - 1 ? t[m - (T - 1)] : win[(j0 + m) % T], acc[qq]);
                    }
#pragma unroll
                for (int qq = 0; qq < QN; ++qq) {
                    uq[(j0 + qq) * ROW + c] = acc[qq];
                    win[(T - 1 + j0 + qq) % T] = t[qq];
                }
            }
            if (TIME && flags) {
                float2 *eq = et + ub * ESZ + c * EJ;
                for (int j = 0; j < kRound; ++j) {
                    const float fw = flags[(long long)n * S + min(sr + j, S - 1)];
                    eq[j] = make_float2(eq[j].x * fw, eq[j].y * fw);
                }
            }
            named_bar_arrive(kBar256Full + ub, HAND);
            named_bar_sync(kBarRaw, NF);                // every FIR thread has read raw buffer q
            if (tid == 0) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (b + 2 < nrounds) issue(q, s0 + T - 1 + (b + 2) * kRound, kRound);
        }
    } else {
        // ---------------- FFT threads: group g takes rounds b = g mod 2 ----------------
        const int t = tid - NF;
        const int g = t / NG, tg = t % NG;
        const int bar_fft = kBar256Fft + g;
        constexpr int planes = OUT == 4 ? 4 : 2;
        const long long pstride = (long long)I_pad * s_out;
        const int i = n * kPols + p;
        const int S16 = (S + kRound - 1) / kRound * kRound;
        // pass 1: column n2, rows tr0 and tr0 + 8; pass 2: k1, spectra jp and jp + 1
        const int n2 = (tg % 32) / 2, tr0 = 2 * (tg / 32) + (tg & 1);
        const int k1 = tg / 8, jp = 2 * (tg % 8);
        for (int b = g; b < nrounds; b += 2) {
            const int q = b % W::NB;
            const int sr = s0 + b * kRound;
            float2 *uq = u + q * USZ;
            float4 rr = make_float4(1.f, 0.f, 1.f, 0.f);
            if constexpr (!TIME) rr = *reinterpret_cast<const float4 *>(ratio + (long long)n * S16 + sr + jp);
            named_bar_sync(kBar256Full + q, HAND);
            float2 v[2][R];
#pragma unroll
            for (int it = 0; it < 2; ++it)
#pragma unroll
                for (int n1 = 0; n1 < R; ++n1) v[it][n1] = uq[(tr0 + 8 * it) * ROW + R * n1 + n2];
#pragma unroll
            for (int it = 0; it < 2; ++it) fft_reg<R>(v[it]);
#pragma unroll
            for (int kk = 0; kk < R; kk += 2) {
                const float4 w = *reinterpret_cast<const float4 *>(tw + n2 * TW + kk);
#pragma unroll
                for (int it = 0; it < 2; ++it) {
                    if (kk) v[it][kk] = cmul(v[it][kk], make_float2(w.x, w.y));
                    v[it][kk + 1] = cmul(v[it][kk + 1], make_float2(w.z, w.w));
                }
            }
            named_bar_sync(bar_fft, NG);                // every thread of the group has read u[q]
#pragma unroll
            for (int it = 0; it < 2; ++it)
#pragma unroll
                for (int kk = 0; kk < R; ++kk) uq[(kk * R + n2) * RS + tr0 + 8 * it] = v[it][kk];
            named_bar_sync(bar_fft, NG);                // P1 complete
#pragma unroll
            for (int m = 0; m < R; ++m) {
                const float4 w = *reinterpret_cast<const float4 *>(uq + (k1 * R + m) * RS + jp);
                v[0][m] = make_float2(w.x, w.y);
                v[1][m] = make_float2(w.z, w.w);
            }
            if constexpr (TIME) {
                if (b + W::NB < nrounds) named_bar_arrive(kBar256Empty + q, HAND);
#pragma unroll
                for (int it = 0; it < 2; ++it) fft_reg<R>(v[it]);
#pragma unroll
                for (int k2 = 0; k2 < R; ++k2) {
                    const int kout = k1 + R * ((k2 + R / 2) % R);
                    const float4 f = *reinterpret_cast<const float4 *>(et + q * ESZ + kout * EJ + jp);
                    v[0][k2] = cmul(v[0][k2], make_float2(f.x, f.y));
                    v[1][k2] = cmul(v[1][k2], make_float2(f.z, f.w));
                }
                if (b + W::NB < nrounds) named_bar_arrive(kBar256EmptyF + q, HAND);
            } else {
                const float4 ee = *reinterpret_cast<const float4 *>(et + q * ESZ + k1 * kRound + jp);
                if (b + W::NB < nrounds) named_bar_arrive(kBar256Empty + q, HAND);
#pragma unroll
                for (int it = 0; it < 2; ++it) fft_reg<R>(v[it]);
                // output k2 is channel k1 + 128 + 16 k2 for k2 < 8 and k1 + 128 + 16 (k2 - 16) above
                float2 r[2] = {make_float2(rr.x, rr.y), make_float2(rr.z, rr.w)};
                float2 up[2] = {make_float2(ee.x, ee.y), make_float2(ee.z, ee.w)}, dn[2];
#pragma unroll
                for (int it = 0; it < 2; ++it) dn[it] = cmul(up[it], conj2(r[it]));
#pragma unroll
                for (int k2 = 0; k2 < R / 2; k2 += 2) {
                    const float4 bu = *reinterpret_cast<const float4 *>(bpt + k1 * R + k2);
                    const float4 bd = *reinterpret_cast<const float4 *>(bpt + k1 * R + R - 2 - k2);
                    const float2 fu[2] = {make_float2(bu.x, bu.y), make_float2(bu.z, bu.w)};
                    const float2 fd[2] = {make_float2(bd.z, bd.w), make_float2(bd.x, bd.y)};
#pragma unroll
                    for (int qq = 0; qq < 2; ++qq) {
                        const int ku = k2 + qq, kd = R - 1 - ku;
#pragma unroll
                        for (int it = 0; it < 2; ++it) {
                            v[it][ku] = cmul(__fmul2_rn(v[it][ku], fu[qq]), up[it]);
                            v[it][kd] = cmul(__fmul2_rn(v[it][kd], fd[qq]), dn[it]);
                            up[it] = cmul(up[it], r[it]);
                            dn[it] = cmul(dn[it], conj2(r[it]));
                        }
                    }
                }
            }
            const int s = sr + jp;
            if (sr + kRound > s_end) {                         // only in the block's last round
#pragma unroll
                for (int k2 = 0; k2 < R; ++k2) {
                    if (s >= s_end) v[0][k2] = make_float2(0.f, 0.f);
                    if (s + 1 >= s_end) v[1][k2] = make_float2(0.f, 0.f);
                }
            }
            if constexpr (OUT == 1) {
                // Spectrum-blocked: the 16 spectra of a channel are every other 8 bytes
                // of a 256-byte run (the other pol's CTA fills the rest in L2). The
                // lanes of an even and of the next odd k1 swap a spectrum each, so a
                // store holds all 16 spectra of one channel, both values of each sector
                // at once.
                const bool odd = k1 & 1;
                const long long kstride = (long long)(s_out / kRound) * N * (2 * kRound);
                float2 *out = reinterpret_cast<float2 *>(corr) +
                              ((long long)sb * C + (k1 & ~1)) * kstride +
                              ((long long)((sr - s_base) / kRound) * N + n) * (2 * kRound) + (jp + odd) * 2 + p;
#pragma unroll
                for (int k2 = 0; k2 < R; ++k2) {
                    const float2 mine = odd ? v[1][k2] : v[0][k2], give = odd ? v[0][k2] : v[1][k2];
                    const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, 8),
                                                   __shfl_xor_sync(0xffffffffu, give.y, 8));
                    float2 *o = out + (long long)(R * ((k2 + R / 2) % R)) * kstride;
                    o[0] = odd ? got : mine;
                    o[kstride] = odd ? mine : got;
                }
            } else {
                const long long base = (long long)sb * C * planes * pstride + (long long)i * s_out + (s - s_base);
#pragma unroll
                for (int k2 = 0; k2 < R; ++k2) {
                    const int kout = k1 + R * ((k2 + R / 2) % R);
                    store_planar<OUT>(corr, base + (long long)kout * planes * pstride, pstride, v[0][k2], v[1][k2]);
                }
            }
        }
    }
}

// Zeros of the planar layout outside what the F-stage wrote: inputs [I, I_pad)
// and spectra [S16, s_out) of every (subband, channel, plane).
cudaError_t planar_pad(const Handle &h, void *corr, int out, int S16, int s_out, cudaStream_t st)
{
    if (h.I_pad <= h.I && s_out <= S16) return cudaSuccess;
    const long long planes = (long long)h.p.n_subbands * h.p.n_channels * (out == 4 ? 4 : 2);
    // S16 and s_out are multiples of 16 values, so rows and gaps are whole 16-byte words
    const int per = out == 5 ? 4 : 8;
    if (planes > 0x7fffffffLL || (long long)h.I_pad * (s_out / per) > 0x7fffffffLL)
        return cudaErrorInvalidConfiguration;
    planar_pad_kernel<<<(unsigned)planes, 256, 0, st>>>(reinterpret_cast<uint4 *>(corr), h.I, h.I_pad, s_out / per,
                                                         max(s_out - S16, 0) / per);
    return cudaGetLastError();
}

template <int C, int T, typename TIn, int OUT>
cudaError_t launch_t(const Handle &h, const void *raw, void *corr, const float *bandpass, const float2 *gains,
                     const float *flags, const FWindow *win, cudaStream_t st)
{
    const int N = h.p.n_stations, S = h.p.n_spectra, SB = h.p.n_subbands;
    // spectra [s_base, s_end) into an output whose spectrum stride is s_out
    const int s_base = win ? win->s_base : 0;
    const int s_end = win ? win->s_end : S;
    // FP32: the spectrum-blocked layout, s_out a multiple of 16 (ceil16(S) by default)
    const int s_out = win ? win->s_out : (OUT == 1 ? (S + kRound - 1) / kRound * kRound : h.S_pad);
    if (s_base % kRound != 0 || s_end > S || s_base >= s_end || s_end - s_base > s_out ||
        (OUT == 1 && s_out % kRound != 0))
        return cudaErrorInvalidValue;
    const int rounds_total = (s_end - s_base + kRound - 1) / kRound;
    const float scale = (OUT == 1 || OUT == 5) ? 1.f : h.operand_scale;
    if constexpr (C == 16 || C == 64) {
        using W = FusedWsCfg<C>;
        const int sg = (N + W::NPC - 1) / W::NPC;
        // long runs amortise the T-1 history rows each CTA filters first; shorten
        // them only while the grid would be under ~5 waves
        int rpc = 64;
        while (rpc > 1 && (long long)((rounds_total + rpc - 1) / rpc) * sg * SB < 152LL * 16) rpc /= 2;
        dim3 grid(sg, (rounds_total + rpc - 1) / rpc, SB);
        if (grid.x > 0x7fffffffu || grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
        constexpr size_t smem = fused_ws_smem_bytes<C, TIn>();
        auto kern = ppf_correct_ws_kernel<C, T, TIn, OUT>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid, 2 * W::NF, smem, st>>>(reinterpret_cast<const TIn *>(raw), corr, h.d_taps, h.d_twiddle,
                                            h.d_phase, bandpass, gains, N, S, h.I_pad, s_out, scale, rpc, flags,
                                            s_base, s_end, h.d_status, h.tc_timeout_cycles, h.tc_test_no_tma);
        e = cudaGetLastError();
        if (e != cudaSuccess || OUT == 1) return e;
        return planar_pad(h, corr, OUT, rounds_total * kRound, s_out, st);
    } else {
        static_assert(C == 256, "16, 64 or 256 channels");
        // one CTA per (station, pol) and SM; long runs of rounds amortise the
        // prologue, shortened only while the grid would be under ~4 waves
        int rpc = 64;
        while (rpc > 1 && (long long)((rounds_total + rpc - 1) / rpc) * N * kPols * SB < 152LL * 4) rpc /= 2;
        dim3 grid(N * kPols, (rounds_total + rpc - 1) / rpc, SB);
        if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
        constexpr size_t smem = ws256_smem_bytes<TIn, OUT>();
        auto kern = ppf_correct_ws256_kernel<T, TIn, OUT>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid, Ws256<OUT>::ALL, smem, st>>>(reinterpret_cast<const TIn *>(raw), corr, h.d_taps, h.d_twiddle,
                                                h.d_phase, h.d_ratio, bandpass, gains, N, S, h.I_pad, s_out, scale, rpc, flags,
                                                s_base, s_end, h.d_status, h.tc_timeout_cycles,
                                                h.tc_test_no_tma);
        e = cudaGetLastError();
        if (e != cudaSuccess || OUT == 1) return e;
        return planar_pad(h, corr, OUT, rounds_total * kRound, s_out, st);
    }
}

template <int C, int T, typename TIn>
cudaError_t launch_out(const Handle &h, const void *raw, void *corr, const float *bp, const float2 *g, const float *fl,
                       const FWindow *w, cudaStream_t st)
{
    switch (h.p.precision) {
    case FX_F32: return launch_t<C, T, TIn, 1>(h, raw, corr, bp, g, fl, w, st);
    case FX_F16: return launch_t<C, T, TIn, 2>(h, raw, corr, bp, g, fl, w, st);
    case FX_BF16: return launch_t<C, T, TIn, 3>(h, raw, corr, bp, g, fl, w, st);
    case FX_TF32_SPLIT: return launch_t<C, T, TIn, 5>(h, raw, corr, bp, g, fl, w, st);
    default: return launch_t<C, T, TIn, 4>(h, raw, corr, bp, g, fl, w, st);
    }
}

template <int C, typename TIn>
cudaError_t launch_taps(const Handle &h, const void *raw, void *corr, const float *bp, const float2 *g,
                        const float *fl, const FWindow *w, cudaStream_t st)
{
    switch (h.p.n_taps) {
    case 4: return launch_out<C, 4, TIn>(h, raw, corr, bp, g, fl, w, st);
    case 8: return launch_out<C, 8, TIn>(h, raw, corr, bp, g, fl, w, st);
    case 16: return launch_out<C, 16, TIn>(h, raw, corr, bp, g, fl, w, st);
    default: return cudaErrorInvalidValue;
    }
}

template <typename TIn>
cudaError_t launch_fmt(const Handle &h, const void *raw, void *corr, const float *bp, const float2 *g, const float *fl,
                       const FWindow *w, cudaStream_t st)
{
    switch (h.p.n_channels) {
    case 16: return launch_taps<16, TIn>(h, raw, corr, bp, g, fl, w, st);
    case 64: return launch_taps<64, TIn>(h, raw, corr, bp, g, fl, w, st);
    case 256: return launch_taps<256, TIn>(h, raw, corr, bp, g, fl, w, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace fxi
