// xcorr_split.cu -- FP32-accurate X-stage on the tcgen05 tensor cores, any
// station count: FP32 corrected samples split in the kernel into hi + lo,
// V ~ hi hi' + hi lo' + lo hi' (lo lo' dropped), FP32 accumulation in TMEM, chunk
// sums added in IEEE FP32 in registers. Serves FX_TF32_SPLIT (planar FP32
// operands; hi hi' as TF32 MMAs, the cross terms as BF16 MMAs) and FX_F32
// (spectrum-blocked complex operands; every term as TF32 MMAs).
//
// Paper, Sec. "Signal processing with GPU kernels": the correlator forms
// V[a][b] = sum_s Y[s][a] conj(Y[s][b]) for all input pairs and integrates over
// the block, in single precision. TF32 keeps FP32's exponent range with an
// 11-bit significand.
//   FX_TF32_SPLIT: hi = x with its 13 low mantissa bits cleared is exactly a TF32
// value and lo = x - hi is exact in FP32 with |lo| < 2^-10 |x|. The cross terms
// hi lo' and lo hi' are each below 2^-10 of the product; rounding hi and lo to
// BF16 (8-bit significand, FP32 exponent range, round to nearest) changes one by
// at most 2^-8 of itself, i.e. 2^-18 of the product in the worst case and about
// 2^-21 RMS, with zero mean; the dropped lo lo' term is below 2^-20 of the product.
//   FX_F32 takes the place of an FP32 FMA chain and may lose no more than that
// does. hi is x rounded to TF32, so |lo| <= 2^-11 |x| with both signs; a TF32 MMA
// reads 11 of lo's at most 12 bits (2^-24 of x RMS), and lo lo' is 2^-24 of the
// product RMS. With BF16 cross terms, as above, one product's error of 2^-21 shows
// wherever the FMA chain is short or its sum small: uncorrelated stations below
// 768 spectra (2.3 times the chain's error at 128) and lossy blocks (half of the
// spectra lost: 4.6 times at 128, 1.9 at 768).
//
// What bounds it: shared-memory bandwidth (tensor-core operand reads plus the
// converter's traffic), then the tensor pipe. So a diagonal tile, where row
// and column inputs are the same, forms only half of each product and is
// completed by its own transpose at the end of an item. With R, J the real and
// imaginary planes and (hR, lR) ... their hi and lo parts,
//   Q = hJ hR' + hJ lR' - hR lJ'               Im V = Q - Q'
//   P = hR hR' + hJ hJ' + 2 (hR lR' + hJ lJ')  Re V = (P + P') / 2
// (hi hi' of the imaginary part needs one product instead of two, and each
// cross term appears once instead of with its conjugate). Per stage of 16
// spectra and n = 128 inputs:
//   TF32 (K = 8, two K-steps): hJ x [hR; hJ] (N = 2n), hR x hR (N = n)
//   BF16 (K = 16) or TF32:     hJ x [lR; 2lJ], hR x [-lJ; 2lR] (N = 2n)
// into one accumulator of 2n columns [Q | P]: with BF16 cross terms 640 tensor
// clocks and 64 KB of operand reads, against 1024 clocks and 96 KB with all
// products formed, and 24 KB of converter stores against 32 KB; with TF32 ones
// 896 clocks, 88 KB and 48 KB. 64 stations x 1280 channels x 3072
// spectra (4.0 GB of operands): planar 1.45 ms with every product formed and
// the chunk sums reduced in L2, 0.98 ms so (4.1 TB/s; without its MMAs the
// kernel takes 0.66 ms, without its converter 0.95 ms); blocked 1.31 ms with
// chains of 32 spectra (1.22 with 64, 1.63 with 16; BF16 cross terms 1.27 with
// 64), against 6.09 ms on the CUDA cores.
//
// Work items. Rows come in blocks of 128 inputs (M = 128); an item is
// (subband x channel, row block, column block) over the upper block
// triangle: the diagonal item of a row block covers columns
// [row0, row0 + min(128, I_pad - row0)), off-diagonal items cover the columns
// right of it in tiles of at most 64 inputs and form every product:
//   TF32:         hJ_a x [hR; hJ], hR_a x [-hJ; hR]
//   BF16 or TF32: hJ_a x [lR; lJ], hR_a x [-lJ; lR], lJ_a x [hR; hJ], lR_a x [-hJ; hR]
// with Q = Im V and P = Re V. 64 stations (128 inputs) is one diagonal item
// per channel; 76 stations (160 inputs) is a 128-column diagonal item, a
// 32-column off-diagonal item and a 32-row diagonal item.
//
// Shared memory, one stage = 16 spectra. BF16 planes have 32-byte rows and
// 32-byte swizzle; TF32 planes hold the FP32 rows:
//   planar    in the landing ring, 32 spectra (two stages) per slot: TMA boxes of
//             128-byte rows, 128-byte swizzle (64-byte rows cost twice the TMA
//             time per byte). They serve as the TF32 hi operands as they are: a
//             kind::tf32 MMA reads the upper 19 bits of each 32-bit operand and
//             ignores the 13 low mantissa bits (the kernel tests on operands with
//             non-zero low bits check this against an FP64 reference).
//   blocked   one station's 16 spectra x 2 pols are 256 contiguous bytes; a
//             stage lands by one bulk copy, and the converter writes hi rounded
//             to TF32 (which halves lo) and lo as 64-byte rows, 64-byte swizzle.
// Planes of n rows each:
//   diagonal item:     planar TF32 R, J; BF16 hR, hJ, lR, 2lJ, -lJ, 2lR; blocked
//                      those six in FP32. The A operands are planes R, J, hR, hJ
//                      read as 128-row tiles: rows past n are other planes' data
//                      and only reach accumulator rows that are not used; the
//                      regions are large enough that these reads stay inside.
//   off-diagonal item: planar 128-row planes TF32 R, J, BF16 hR, hJ, lR, lJ of the
//                      row inputs; TF32 -J, R, J, BF16 -hJ, hR, hJ, -lJ, lR, lJ
//                      of the columns; blocked hR, hJ, lR, lJ of the rows, then
//                      -hJ, hR, hJ, -lJ, lR, lJ of the columns.
//
// An infinity (blocked). Its hi is the infinity, which meets the other station's
// hi and lo: with a lo of 0 or of the other sign the sum of the two products
// would be a NaN where the product is an infinity; and so it would where both
// overflow. So the converter warps of a stage vote, and if one has met an infinity
// or a value of 2^64 or more all convert the stage again with truncated hi and
// a lo of x's sign that is never zero (split1, SAFE).
//
// Accumulation. The tensor core's FP32 accumulator does not round each
// addition to nearest, so a long chain of MMAs into one accumulator drifts
// (about 2^-24 of the running value per MMA). The accumulator is restarted
// every `chunk` stages and the chunk sums are added in registers (round to
// nearest): the eight epilogue warps hold the whole 128 x 256 accumulator, 128
// registers per thread, so nothing is read back or reduced in memory until
// the item ends. 64 spectra per chunk for FX_TF32_SPLIT; 16 or 32 for FX_F32,
// whose reference is the rounding of an FP32 FMA chain (measured in
// xf32_on_tensor_cores). Each visibility is summed by one lane in a fixed
// order, so results are reproducible.
//
// Warp roles (persistent, one CTA per SM, 512 threads):
//   warps 0-7   epilogue: warp % 4 = TMEM lane quadrant (32 rows), warp / 4 =
//               which 64 columns of Q and of P
//   warp 8      loader
//   warp 9      TMEM allocator + MMA issuer
//   warps 10-15 converter, two groups of three warps that take stages in turn
//               (1.17 ms against 1.33 with six warps on every stage, before the
//               ring was stepped without divisions)
// Registers are moved from the last two warpgroups to the epilogue's
// (setmaxnreg). Two accumulators of 256 columns fill the 512 TMEM columns.
// Every mbarrier wait is bounded; on expiry the role is recorded in the status
// word, all roles leave, in-flight copies and MMAs are drained (bounded) and
// TMEM is freed.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "tc_ptx.cuh"

namespace fxi {
namespace {

using namespace tc;

constexpr int kT3Threads = 512;
constexpr int kT3EpiWarps = 8;
constexpr int kT3ConvGroups = 2, kT3ConvWarps = 3;    // converter: groups take stages in turn, a group's warps share one
constexpr int kT3LoadWarp = 8, kT3MmaWarp = 9, kT3ConvWarp0 = 16 - kT3ConvGroups * kT3ConvWarps;
static_assert(kT3ConvWarp0 > kT3MmaWarp, "warp roles");
constexpr int kT3EpiRegs = 184, kT3RestRegs = 72;      // 256 x (184 + 72) = 512 x 128 registers
constexpr int kT3LaunchRegs = 128;
static_assert(256 * (kT3EpiRegs + kT3RestRegs) <= kT3Threads * kT3LaunchRegs, "the split fits the launch's registers");
constexpr int kT3K = 16;                              // spectra per stage
constexpr unsigned kT3BfRow = 32;                     // one BF16 row: 16 spectra
constexpr unsigned kT3ABf = 128u * kT3BfRow;          // one 128-row BF16 plane: 4 KB
constexpr unsigned kT3StRun = 16u * kPols * 8u;       // one station's 16 spectra x 2 pols, blocked layout
constexpr int kT3MaxStages = 6;
constexpr int kT3MaxItems = 64;                       // items per channel
constexpr int kT3TmemCols = 512;
constexpr int kT3AccCols = 256;
// full, conv, empty, landed per stage; accf 2, acce 2, exch, drain, vote per converter group
constexpr int kT3Bars = 4 * kT3MaxStages + 6 + kT3ConvGroups;
constexpr unsigned kT3Ctrl = 8u * kT3Bars + 16u + 8u * kT3ConvGroups;   // barriers, TMEM base, abort flag, votes
constexpr int kT3Blk = 32 * 33;                       // one 32 x 32 block of the transpose scratch, padded rows
constexpr unsigned kT3Scratch = 10u * kT3Blk * 4u;    // lower block triangle of a 128 x 128 plane
constexpr unsigned kT3ScratchMid = 8u * kT3Blk * 4u;  // six blocks at a time, or the blocks of four segments of 32 inputs
constexpr unsigned kT3ScratchSmall = 4u * kT3Blk * 4u; // four blocks at a time
constexpr unsigned kT3SmemMax = 227u * 1024u;

struct T3Params {
    CUtensorMap map128;       // planar: 3-D (spectrum, input, sb*C*2 + plane), box {32, 128, 1}
    CUtensorMap mapr;         // box {32, rows of the ragged last block, 1}
    CUtensorMap map16;        // box {32, 16, 1}
    int4 items[kT3MaxItems];  // per channel: (row0, col0, n, diagonal)
    const unsigned char *blk; // blocked: corr
    float2 *vis;
    int *status;
    long long n_items;        // ceil(SB * C / group) * ipc
    long long channels;       // SB * C
    int group;                // channels per item: > 1 only with one diagonal item per channel
    int segs;                 // time segments of one channel side by side in a tile (then group = 1)
    int gin;                  // inputs (padded) per channel or segment of a tile
    int nk_all;               // stages of a channel: nk per segment
    long long B;              // baselines
    long long timeout_cycles;
    int ipc;                  // items per channel
    int N, S, nk, chunk;      // stations, spectra, stages per item, stages per accumulator chain
    int nr;                   // rows of mapr's box
    int stages, lands;        // depth of the operand ring and of the landing ring
    unsigned stage_bytes, land_bytes;
    unsigned row_land;        // blocked: offset of the row inputs' stations in a landing slot
    unsigned scratch_bytes;   // kT3Scratch, kT3ScratchMid or kT3ScratchSmall
    int no_tma;               // failure-detection test hook: issue no loads
    int accumulate;           // add to vis
};

__device__ __forceinline__ bool t3wait(unsigned bar, unsigned parity, volatile int *abort_flag, const T3Params &P,
                                       int code)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > P.timeout_cycles) {
            *abort_flag = 1;
            atomicCAS(P.status, 0, code);
            atomicExch(P.status + 1, (int)blockIdx.x);
            return false;
        }
    }
    return true;
}

// Shared-memory matrix descriptor: K-major, 64-byte swizzle (8-row atoms of
// 512 bytes, SBO = 512), LBO unused for this layout, descriptor version 1.
__device__ __forceinline__ unsigned long long sdesc64(unsigned addr)
{
    return (unsigned long long)((addr & 0x3FFFF) >> 4) | (1ull << 16) | ((unsigned long long)(512 >> 4) << 32) |
           (1ull << 46) | (4ull << 61);
}

// The same for the BF16 planes: K-major, 32-byte swizzle (8-row atoms of 256
// bytes, SBO = 256); one 32-byte row is the whole K = 16 of a stage.
__device__ __forceinline__ unsigned long long sdesc32(unsigned addr)
{
    return (unsigned long long)((addr & 0x3FFFF) >> 4) | (1ull << 16) | ((unsigned long long)(256 >> 4) << 32) |
           (1ull << 46) | (6ull << 61);
}

// Instruction descriptor, kind::tf32: D = F32, A = B = TF32, both K-major, M = 128.
__device__ __forceinline__ unsigned idesc_tf32(int n)
{
    return (1u << 4) | (2u << 7) | (2u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(128 >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc,
                                         unsigned idesc, unsigned accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
                 "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
                 : "memory");
}

// Contiguous copy into shared memory (both addresses 16-byte aligned, bytes a multiple of 16).
__device__ __forceinline__ void bulk_g2s(unsigned dst, const void *src, unsigned bytes, unsigned bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Byte offset, in a 32-byte-swizzled BF16 plane, of spectra 4 lc .. 4 lc + 3 of
// row r, and in a 64-byte-swizzled FP32 plane of the same (16 bytes). Both
// swizzles XOR the 16-byte chunk index with address bits 7 and up (64-byte
// rows: chunk ^= (row / 2) mod 4; 32-byte rows: chunk ^= (row / 4) mod 2) and
// the plane bases are aligned to their atoms.
__device__ __forceinline__ unsigned bf_off(int r, int lc)
{
    return (unsigned)(r * 32 + 16 * ((lc >> 1) ^ ((r >> 2) & 1)) + 8 * (lc & 1));
}
__device__ __forceinline__ unsigned tf_off(int r, int lc) { return (unsigned)(r * 64 + 16 * (lc ^ ((r >> 1) & 3))); }

__device__ __forceinline__ unsigned bf16x2(float a, float b)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const unsigned *>(&v);
}
__device__ __forceinline__ uint2 neg_bf16x4(uint2 v) { return make_uint2(v.x ^ 0x80008000u, v.y ^ 0x80008000u); }
__device__ __forceinline__ uint2 dbl_bf16x4(uint2 v)   // exact: doubling only moves the exponent
{
    __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162 *>(&v.x), b = *reinterpret_cast<__nv_bfloat162 *>(&v.y);
    a = __hadd2(a, a);
    b = __hadd2(b, b);
    return make_uint2(*reinterpret_cast<unsigned *>(&a), *reinterpret_cast<unsigned *>(&b));
}

// One value's hi part (a TF32 value) and, through *lo, x - hi (exact).
//  TRUNC  the 13 low bits cleared: what a TF32 MMA reads of the raw value
//  ROUND  rounded to nearest: lo is half as large and has both signs
//  SAFE   as TRUNC, for stages that hold an infinity or a value whose products may
//         overflow: lo has x's sign and is never zero, so that an infinity times
//         the other station's hi and lo is the same infinity twice, not a NaN
enum SplitMode { TRUNC, ROUND, SAFE };
template <int MODE>
__device__ __forceinline__ float split1(float x, float *lo)
{
    const unsigned b = __float_as_uint(x);
    const float h = __uint_as_float((MODE == ROUND ? b + 0x1000u : b) & 0xFFFFE000u);
    *lo = x - h;
    if (MODE == SAFE && x == x && !(fabsf(*lo) > 0.f)) *lo = copysignf(1.17549435e-38f, x);
    return h;
}
constexpr float kT3RoundMax = 0x1p64f;                 // from here on SAFE: hi lo' may overflow

template <int MODE>
__device__ __forceinline__ void split4(float4 x, float4 &h, float4 &l)
{
    h.x = split1<MODE>(x.x, &l.x);
    h.y = split1<MODE>(x.y, &l.y);
    h.z = split1<MODE>(x.z, &l.z);
    h.w = split1<MODE>(x.w, &l.w);
}

// hi and lo of four values of the planar layout, in BF16 (round to nearest even)
struct SplitBf4 {
    uint2 h, l;
};
__device__ __forceinline__ SplitBf4 split_bf4(float4 x)
{
    float4 h, l;
    split4<TRUNC>(x, h, l);
    return {make_uint2(bf16x2(h.x, h.y), bf16x2(h.z, h.w)), make_uint2(bf16x2(l.x, l.y), bf16x2(l.z, l.w))};
}

// Operand planes: DIAG column planes of a diagonal item (hR, hJ, lR, 2lJ, -lJ,
// 2lR), COLS column planes of an off-diagonal item (-hJ, hR, hJ, -lJ, lR, lJ),
// ROWS row planes of an off-diagonal item (hR, hJ, lR, lJ). In BF16 beside the
// landed TF32 rows (planar; a TF32 plane -J before R and J for COLS), or all in
// FP32 (blocked).
enum PlaneRole { DIAG, COLS, ROWS };
template <int ROLE>
__device__ __forceinline__ void put_bf(const SplitBf4 &a, const SplitBf4 &b, unsigned char *bf, unsigned bp)
{
    auto put = [&](int plane, uint2 v) { *reinterpret_cast<uint2 *>(bf + plane * bp) = v; };
    if constexpr (ROLE == DIAG) {
        put(0, a.h);
        put(1, b.h);
        put(2, a.l);
        put(3, dbl_bf16x4(b.l));
        put(4, neg_bf16x4(b.l));
        put(5, dbl_bf16x4(a.l));
    } else if constexpr (ROLE == COLS) {
        put(0, neg_bf16x4(b.h));
        put(1, a.h);
        put(2, b.h);
        put(3, neg_bf16x4(b.l));
        put(4, a.l);
        put(5, b.l);
    } else {
        put(0, a.h);
        put(1, b.h);
        put(2, a.l);
        put(3, b.l);
    }
}

__device__ __forceinline__ float4 neg4(float4 v) { return make_float4(-v.x, -v.y, -v.z, -v.w); }
__device__ __forceinline__ float4 dbl4(float4 v) { return make_float4(v.x + v.x, v.y + v.y, v.z + v.z, v.w + v.w); }

template <int ROLE>
__device__ __forceinline__ void put_tf(float4 hr, float4 hj, float4 lr, float4 lj, unsigned char *tf, unsigned tp)
{
    auto put = [&](int plane, float4 v) { *reinterpret_cast<float4 *>(tf + plane * tp) = v; };
    if constexpr (ROLE == DIAG) {
        put(0, hr);
        put(1, hj);
        put(2, lr);
        put(3, dbl4(lj));
        put(4, neg4(lj));
        put(5, dbl4(lr));
    } else if constexpr (ROLE == COLS) {
        put(0, neg4(hj));
        put(1, hr);
        put(2, hj);
        put(3, neg4(lj));
        put(4, lr);
        put(5, lj);
    } else {
        put(0, hr);
        put(1, hj);
        put(2, lr);
        put(3, lj);
    }
}

// Planar operands: the R and J planes (128-byte rows of 32 spectra, 128-byte
// swizzle, pitch tp) at tf hold the raw rows; this is their half `half`. A
// warp takes 8 rows x 4 chunks, eight lanes two rows r and (r + 5) mod 8: their
// 16-byte reads fall on distinct banks, and so do sixteen lanes' 8-byte stores.
template <int ROLE>
__device__ __forceinline__ void convert_planar(unsigned char *tf, unsigned tp, unsigned char *bf, unsigned bp, int rows,
                                               int half, int cw, int lane)
{
    const int k = lane >> 3, lc = lane & 3;
    const int rl = lane & 4 ? (2 * k + 5) & 7 : 2 * k;
    const unsigned to = (unsigned)(rl * 128 + 16 * ((4 * half + lc) ^ rl)), bo = bf_off(rl, lc);
    for (int r8 = cw; r8 < rows / 8; r8 += kT3ConvWarps) {
        unsigned char *p = tf + r8 * 1024 + to;
        const float4 x = *reinterpret_cast<const float4 *>(p);
        const float4 y = *reinterpret_cast<const float4 *>(p + tp);
        if constexpr (ROLE == COLS) *reinterpret_cast<float4 *>(p - tp) = neg4(y);
        put_bf<ROLE>(split_bf4(x), split_bf4(y), bf + r8 * 256 + bo, bp);
    }
}

// Spectrum-blocked operands: `land` holds stations' runs of [16 spectra][2
// pols] complex values; a task is 4 spectra of one station, both pols, written
// to the FP32 planes (64-byte rows, 64-byte swizzle, pitch tp). Spectra from
// s_lim on count as zero (every gst stations seg fewer: time segments). The four
// 16-byte reads of a task are rotated by lane / 2 so that eight lanes' reads fall
// on distinct banks, and sorted again in registers. Rows are ordered pol by pol
// within eight stations (row 16 (st / 8) + 8 p + st mod 8), so that the lanes of a
// store take consecutive rows and distinct banks too. Returns whether a value of
// this thread's wants SAFE.
template <int ROLE, bool SEG, int MODE>
__device__ __forceinline__ bool convert_blocked(const unsigned char *land, unsigned char *tf, unsigned tp, int rows,
                                                int s_lim, int gst, int seg, int t)
{
    const int nt = rows / 2 * 4;                          // a multiple of 32: whole warps
    const int rot = (t >> 1) & 3;
    float top = 0.f;
    for (int q = t; q < nt; q += 32 * kT3ConvWarps) {
        const float4 *w = reinterpret_cast<const float4 *>(land) + 4 * q;
        float4 v[4], u[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = w[(e + rot) & 3];   // spectrum (e + rot) mod 4 of the group
#pragma unroll
        for (int e = 0; e < 4; ++e) u[e] = rot & 1 ? v[(e + 3) & 3] : v[e];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = rot & 2 ? u[(e + 2) & 3] : u[e];
        const int lc = q & 3, st = q >> 2;
        const int lim = SEG ? s_lim - st / gst * seg : s_lim;
        if (lim < kT3K) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (4 * lc + e >= lim) v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if constexpr (MODE == ROUND) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                top = fmaxf(fmaxf(fmaxf(top, fabsf(v[e].x)), fabsf(v[e].y)), fmaxf(fabsf(v[e].z), fabsf(v[e].w)));
        }
#pragma unroll
        for (int p = 0; p < kPols; ++p) {
            float4 hr, hj, lr, lj;
            split4<MODE>(p ? make_float4(v[0].z, v[1].z, v[2].z, v[3].z)
                           : make_float4(v[0].x, v[1].x, v[2].x, v[3].x), hr, lr);
            split4<MODE>(p ? make_float4(v[0].w, v[1].w, v[2].w, v[3].w)
                           : make_float4(v[0].y, v[1].y, v[2].y, v[3].y), hj, lj);
            put_tf<ROLE>(hr, hj, lr, lj, tf + tf_off(16 * (st >> 3) + 8 * p + (st & 7), lc), tp);
        }
    }
    return top >= kT3RoundMax;
}

// BLOCKED: spectrum-blocked complex operands (FX_F32), else planar (FX_TF32_SPLIT)
// (SEG: time segments of one channel share a tile)
template <bool BLOCKED, bool SEG>
__global__ void __launch_bounds__(kT3Threads, 1) xcorr_split_kernel(const __grid_constant__ T3Params P)
{
    extern __shared__ unsigned char smem_raw[];
    const unsigned base_u32 = smem_u32(smem_raw);
    const unsigned pad = (1024 - (base_u32 & 1023)) & 1023;
    unsigned char *tiles = smem_raw + pad;
    const unsigned tiles_u32 = base_u32 + pad;
    unsigned char *land = tiles + (size_t)P.stages * P.stage_bytes;
    const unsigned land_u32 = tiles_u32 + (unsigned)P.stages * P.stage_bytes;
    float *scratch = reinterpret_cast<float *>(land + (size_t)P.lands * P.land_bytes);
    unsigned char *ctrl = reinterpret_cast<unsigned char *>(scratch) + P.scratch_bytes;
    const unsigned bar0 = smem_u32(ctrl);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };                          // rows landed
    auto conv_bar = [&](int s) { return bar0 + 8u * (kT3MaxStages + s); };         // operands written
    auto empty_bar = [&](int s) { return bar0 + 8u * (2 * kT3MaxStages + s); };    // MMAs done with the stage
    auto landed_bar = [&](int s) { return bar0 + 8u * (3 * kT3MaxStages + s); };   // landing slot no longer needed
    auto accf_bar = [&](int b) { return bar0 + 8u * (4 * kT3MaxStages + b); };
    auto acce_bar = [&](int b) { return bar0 + 8u * (4 * kT3MaxStages + 2 + b); };
    const unsigned exch_bar = bar0 + 8u * (4 * kT3MaxStages + 4);
    const unsigned drain_bar = bar0 + 8u * (4 * kT3MaxStages + 5);
    auto vote_bar = [&](int g) { return bar0 + 8u * (4 * kT3MaxStages + 6 + g); };  // a converter group's warps have voted
    unsigned *tmem_slot = reinterpret_cast<unsigned *>(ctrl + 8 * kT3Bars);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile unsigned *votes = tmem_slot + 2;          // [group][parity]: the last stage that needs SAFE
    // TF32 operands: blocked, planes of 64-byte rows in the stage; planar, planes
    // of 128-byte rows (32 spectra) in the landing slot
    constexpr unsigned TROW = BLOCKED ? 64u : 128u;
    constexpr unsigned TA = 128u * TROW;               // one 128-row plane
    constexpr int PER = BLOCKED ? 1 : 2;               // stages per landing slot
    const int slots = (P.nk + PER - 1) / PER;          // landing slots per item

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kT3MaxStages; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(conv_bar(s), kT3ConvWarps);   // one arrival per converter warp of the stage's group
            mbar_init(empty_bar(s), 1);
            mbar_init(landed_bar(s), BLOCKED ? kT3ConvWarps : 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf_bar(b), 1);
            mbar_init(acce_bar(b), kT3EpiWarps);    // one arrival per epilogue warp
        }
        mbar_init(exch_bar, kT3EpiWarps);
        mbar_init(drain_bar, 1);
        for (int g = 0; g < kT3ConvGroups; ++g) {
            mbar_init(vote_bar(g), kT3ConvWarps);
            votes[2 * g] = votes[2 * g + 1] = 0;
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if constexpr (BLOCKED) {
        // Station slots that no copy fills (the padding of I_pad, a last tile's absent
        // channels) are converted with the rest of their warp, and the largest value
        // there chooses how the real stations are split: they start as zeros, not as
        // what an earlier kernel left in shared memory.
        for (unsigned q = threadIdx.x; q < (unsigned)P.lands * P.land_bytes / 16; q += kT3Threads)
            reinterpret_cast<uint4 *>(land)[q] = make_uint4(0, 0, 0, 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kT3MmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kT3TmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = *tmem_slot;

    if (warp >= kT3EpiWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kT3RestRegs));
        if (warp == kT3LoadWarp) {
            // ================= loader =================
            if (lane == 0) {
                Ring ring;
                int filled = 0;                        // landing slots with a copy issued, up to the ring's depth
                bool ok = true;
                for (long long w = blockIdx.x; w < P.n_items && ok; w += gridDim.x) {
                    const int4 itm = P.items[(int)(w % P.ipc)];
                    const long long gch = w / P.ipc;
                    const int row0 = itm.x, col0 = itm.y, n = itm.z;
                    const bool diag = itm.w != 0;
                    const unsigned pitch = (unsigned)n * TROW;
                    // blocked: stations of the row and of the column inputs
                    const int ast = row0 / 2, bst = col0 / 2;
                    const int chans = (int)min((long long)P.group, P.channels - gch * P.group);
                    const unsigned abytes = (unsigned)min(64, P.N - ast) * kT3StRun;
                    const unsigned bbytes = (unsigned)min(n / 2, P.N - bst) * kT3StRun;
                    const unsigned tx = BLOCKED ? (diag ? 0u : abytes) + (P.group > 1 ? chans * P.N * kT3StRun : bbytes)
                                                : (diag ? 0u : 2u * TA) + 2u * pitch;
                    const long long chstep = P.nk_all * P.N * (long long)kT3StRun;
                    const unsigned char *src = P.blk + gch * P.group * chstep;
                    for (int kc = 0; kc < slots; ++kc, ring.step(P.lands)) {
                        const int l = ring.i;
                        if (!t3wait(landed_bar(l), ring.ph ^ 1u, abort_flag, P, 1)) {
                            ok = false;
                            break;
                        }
                        if (P.no_tma) continue;
                        filled = min(filled + 1, P.lands);
                        if constexpr (BLOCKED && SEG) {
                            // block kc of every segment (none past the channel's end: the
                            // converter counts those spectra as zero)
                            const unsigned run = (unsigned)P.N * kT3StRun;
                            const int live = (P.nk_all - kc + P.nk - 1) / P.nk;
                            mbar_arrive_expect_tx(full_bar(l), live * run);
                            for (int c = 0; c < live; ++c)
                                bulk_g2s(land_u32 + (unsigned)l * P.land_bytes + (unsigned)(c * (P.gin / 2)) * kT3StRun,
                                         src + (long long)(kc + c * P.nk) * run, run, full_bar(l));
                            continue;
                        }
                        mbar_arrive_expect_tx(full_bar(l), tx);
                        const unsigned dst = land_u32 + (unsigned)l * P.land_bytes;
                        if constexpr (BLOCKED) {
                            const unsigned char *b = src + (long long)kc * P.N * kT3StRun;
                            if (P.group > 1) {
                                for (int c = 0; c < chans; ++c)
                                    bulk_g2s(dst + (unsigned)(c * (P.gin / 2)) * kT3StRun, b + c * chstep,
                                             (unsigned)P.N * kT3StRun, full_bar(l));
                                continue;
                            }
                            bulk_g2s(dst, b + (long long)bst * kT3StRun, bbytes, full_bar(l));
                            if (!diag) bulk_g2s(dst + P.row_land, b + (long long)ast * kT3StRun, abytes, full_bar(l));
                        } else {
                            for (int pl = 0; pl < 2; ++pl) {
                                const int z = (int)(gch * P.group * 2 + pl), x = kc * 2 * kT3K;
                                if constexpr (SEG) {   // spectra past the padded end arrive as zeros
                                    for (int c = 0; c < P.segs; ++c)
                                        tma_load_3d(dst + (unsigned)pl * pitch + (unsigned)(c * P.gin) * TROW, &P.mapr,
                                                    full_bar(l), x + c * P.nk * kT3K, 0, z);
                                    continue;
                                }
                                if (P.group > 1) {     // channels past the last one arrive as zeros
                                    for (int c = 0; c < P.group; ++c)
                                        tma_load_3d(dst + (unsigned)pl * pitch + (unsigned)(c * P.gin) * TROW, &P.mapr,
                                                    full_bar(l), x, 0, z + 2 * c);
                                    continue;
                                }
                                if (!diag)         // row inputs: A region planes R and J
                                    tma_load_3d(dst + (unsigned)pl * TA, &P.map128, full_bar(l), x, row0, z);
                                const unsigned bdst = dst + (diag ? 0u : 2u * TA + pitch) + (unsigned)pl * pitch;
                                if (n == 128) {
                                    tma_load_3d(bdst, &P.map128, full_bar(l), x, col0, z);
                                } else if (n == P.nr) {
                                    tma_load_3d(bdst, &P.mapr, full_bar(l), x, col0, z);
                                } else {
                                    for (int r = 0; r < n; r += 16)
                                        tma_load_3d(bdst + (unsigned)r * TROW, &P.map16, full_bar(l), x, col0 + r, z);
                                }
                            }
                        }
                    }
                }
                if (!ok) {                             // wait for the copies of the ring's last uses
                    for (int u = 0; u < filled; ++u) {
                        ring.back(P.lands);
                        drain_wait(full_bar(ring.i), ring.ph, P.timeout_cycles);
                    }
                }
            }
        } else if (warp == kT3MmaWarp) {
            // ================= MMA issuer =================
            if (lane == 0) {
                Ring ring, lring;                        // stages, landing slots
                unsigned acc_it = 0;
                bool ok = true, issued = false;
                // descriptors of the operand regions' first bytes; a plane or K-step further
                // on is an addition in 16-byte units (one thread issues every MMA, so its
                // instructions per MMA count)
                const unsigned long long tdesc0 = BLOCKED ? sdesc64(tiles_u32) : smem_desc(land_u32);
                const unsigned long long bdesc0 = sdesc32(tiles_u32);
                for (long long w = blockIdx.x; w < P.n_items && ok; w += gridDim.x) {
                    const int4 itm = P.items[(int)(w % P.ipc)];
                    const int n = itm.z;
                    const bool diag = itm.w != 0;
                    // plane pitches and the offset of the column BF16 planes, in 16-byte units
                    const unsigned tp = (unsigned)n * TROW / 16, bp = (unsigned)n * kT3BfRow / 16;
                    const unsigned bf0 = diag ? 0u : 4 * kT3ABf / 16;
                    const unsigned id2 = idesc_tf32(2 * n), id1 = idesc_tf32(n);
                    const unsigned idb = make_idesc(1u, 2 * n, false);
                    for (int k0 = 0; k0 < P.nk && ok; k0 += P.chunk, ++acc_it) {
                        const int ab = (int)(acc_it & 1);
                        if (!t3wait(acce_bar(ab), ((acc_it >> 1) & 1u) ^ 1u, abort_flag, P, 2)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const unsigned d = tmem_base + (unsigned)(ab * kT3AccCols);
                        const int kend = min(P.chunk, P.nk - k0);
                        for (int kc = 0; kc < kend; ++kc, ring.step(P.stages)) {
                            const int s = ring.i, l = lring.i;
                            if (!t3wait(conv_bar(s), ring.ph, abort_flag, P, 2)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            const unsigned so = (unsigned)s * (P.stage_bytes >> 4);
                            // this stage's 64 bytes of the TF32 rows
                            const unsigned long long tf =
                                tdesc0 + (BLOCKED ? so : (unsigned)l * (P.land_bytes >> 4) + 4u * ((k0 + kc) % PER));
                            const unsigned long long bf = bdesc0 + so + bf0;
                            // (the small cross terms first, while the accumulator is small: 10 to 20% less
                            // error than after the main term)
                            if (diag) {
                                if constexpr (BLOCKED) {
#pragma unroll
                                    for (int kk = 0; kk < kT3K / 8; ++kk) {
                                        const unsigned long long t = tf + 2u * kk;
                                        mma_tf32(d, t + tp, t + 2 * tp, id2, (kc | kk) ? 1u : 0u);   // hJ x [lR; 2lJ]
                                        mma_tf32(d, t, t + 4 * tp, id2, 1u);                         // hR x [-lJ; 2lR]
                                    }
                                } else {
                                    mma_f16(d, bf + bp, bf + 2 * bp, idb, kc ? 1u : 0u);             // hJ x [lR; 2lJ]
                                    mma_f16(d, bf, bf + 4 * bp, idb, 1u);                            // hR x [-lJ; 2lR]
                                }
#pragma unroll
                                for (int kk = 0; kk < kT3K / 8; ++kk)      // 8 FP32 = 32 bytes per TF32 K-step
                                    mma_tf32(d, tf + tp + 2u * kk, tf + 2u * kk, id2, 1u);           // hJ x [hR; hJ]
#pragma unroll
                                for (int kk = 0; kk < kT3K / 8; ++kk)
                                    mma_tf32(d + (unsigned)n, tf + 2u * kk, tf + 2u * kk, id1, 1u);  // hR x hR
                            } else {
                                // rows: R, J, lR, lJ; columns: -J, R, J, -lJ, lR, lJ (planar: the lo planes and
                                // the cross terms' hi planes in BF16)
                                const unsigned long long tb = tf + (BLOCKED ? 4 * TA : 2 * TA) / 16;
                                if constexpr (BLOCKED) {
                                    constexpr unsigned AP = TA / 16;
#pragma unroll
                                    for (int kk = 0; kk < kT3K / 8; ++kk) {
                                        const unsigned long long ra = tf + 2u * kk, cb = tb + 2u * kk;
                                        mma_tf32(d, ra + AP, cb + 4 * tp, id2, (kc | kk) ? 1u : 0u);   // hJ x [lR; lJ]
                                        mma_tf32(d, ra, cb + 3 * tp, id2, 1u);                         // hR x [-lJ; lR]
                                        mma_tf32(d, ra + 3 * AP, cb + tp, id2, 1u);                    // lJ x [hR; hJ]
                                        mma_tf32(d, ra + 2 * AP, cb, id2, 1u);                         // lR x [-hJ; hR]
                                    }
                                } else {
                                    const unsigned long long ra = bdesc0 + so;
                                    constexpr unsigned AP = kT3ABf / 16;
                                    mma_f16(d, ra + AP, bf + 4 * bp, idb, kc ? 1u : 0u);  // hJ x [lR; lJ]
                                    mma_f16(d, ra, bf + 3 * bp, idb, 1u);                 // hR x [-lJ; lR]
                                    mma_f16(d, ra + 3 * AP, bf + bp, idb, 1u);            // lJ x [hR; hJ]
                                    mma_f16(d, ra + 2 * AP, bf, idb, 1u);                 // lR x [-hJ; hR]
                                }
#pragma unroll
                                for (int kk = 0; kk < kT3K / 8; ++kk) {
                                    mma_tf32(d, tf + TA / 16 + 2u * kk, tb + tp + 2u * kk, id2, 1u);   // hJ x [hR; hJ]
                                    mma_tf32(d, tf + 2u * kk, tb + 2u * kk, id2, 1u);                   // hR x [-hJ; hR]
                                }
                            }
                            issued = true;
                            mma_commit(empty_bar(s));
                            if ((k0 + kc) % PER == PER - 1 || k0 + kc == P.nk - 1) {
                                if (!BLOCKED) mma_commit(landed_bar(l));
                                lring.step(P.lands);
                            }
                        }
                        if (!ok) break;
                        mma_commit(accf_bar(ab));
                    }
                }
                if (!ok && issued) {
                    mma_commit(drain_bar);
                    drain_wait(drain_bar, 0, P.timeout_cycles);
                }
            }
            __syncwarp();
        } else if (warp >= kT3ConvWarp0) {
            // ================= converter (warps 10..15) =================
            const int grp = (warp - kT3ConvWarp0) / kT3ConvWarps, cw = (warp - kT3ConvWarp0) % kT3ConvWarps;
            const int ct = cw * 32 + lane;
            Ring ring, lring;
            unsigned voted = 0;                         // blocked: stages this group has voted on
            int turn = 0;                               // group of the next stage
            bool ok = true;
            for (long long w = blockIdx.x; w < P.n_items && ok; w += gridDim.x) {
                const int4 itm = P.items[(int)(w % P.ipc)];
                const int n = itm.z;
                const bool diag = itm.w != 0;
                const unsigned pitch = (unsigned)n * TROW, bpitch = (unsigned)n * kT3BfRow;
                for (int kc = 0; kc < P.nk; ++kc) {
                    const int s = ring.i, l = lring.i;
                    const unsigned sph = ring.ph, lph = lring.ph;
                    ring.step(P.stages);
                    if (kc % PER == PER - 1 || kc == P.nk - 1) lring.step(P.lands);
                    const bool mine = turn == grp;
                    turn = turn + 1 == kT3ConvGroups ? 0 : turn + 1;
                    if (!mine) continue;
                    // The stage's last use first: stages finish in order, and lands >=
                    // stages, so it also tells that the landing slot's last copy is
                    // over and the parity of the next wait is not ambiguous although
                    // the other group may have taken the slot before.
                    const bool got = t3wait(empty_bar(s), sph ^ 1u, abort_flag, P, 4) &&
                                     t3wait(full_bar(l), lph, abort_flag, P, 4);
                    if (!__all_sync(0xffffffffu, got)) {
                        ok = false;
                        break;
                    }
                    unsigned char *st = tiles + (size_t)s * P.stage_bytes;
                    unsigned char *la = land + (size_t)l * P.land_bytes;
                    if constexpr (BLOCKED) {
                        const int lim = P.S - kc * kT3K, gst = P.gin / 2, seg = P.nk * kT3K;
                        auto convert = [&](auto mode) {
                            constexpr int MODE = decltype(mode)::value;
                            if (diag) return convert_blocked<DIAG, SEG, MODE>(la, st, pitch, n, lim, gst, seg, ct);
                            const bool rows =
                                convert_blocked<ROWS, false, MODE>(la + P.row_land, st, TA, 128, lim, gst, seg, ct);
                            return convert_blocked<COLS, false, MODE>(la, st + 4 * TA, pitch, n, lim, gst, seg, ct) || rows;
                        };
                        // An infinity meets every other station's lo parts, which other warps of the
                        // group may have written: they all have to know of it. (Bounded like every
                        // wait here, hence no named barrier: a warp may have left on an abort.)
                        const bool big = __any_sync(0xffffffffu, convert(std::integral_constant<int, ROUND>{}));
                        ++voted;
                        volatile unsigned *vote = votes + 2 * grp + (voted & 1u);
                        if (big) *vote = voted;
                        __syncwarp();
                        if (lane == 0) mbar_arrive(vote_bar(grp));
                        if (!__all_sync(0xffffffffu, t3wait(vote_bar(grp), (voted & 1u) ^ 1u, abort_flag, P, 4))) {
                            ok = false;
                            break;
                        }
                        if (*vote == voted) convert(std::integral_constant<int, SAFE>{});
                    } else {
                        const int half = kc % PER;
                        if (diag) {
                            convert_planar<DIAG>(la, pitch, st, bpitch, n, half, cw, lane);
                        } else {
                            convert_planar<ROWS>(la, TA, st, kT3ABf, 128, half, cw, lane);
                            convert_planar<COLS>(la + 2 * TA + pitch, pitch, st + 4 * kT3ABf, bpitch, n, half, cw, lane);
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(conv_bar(s));
                        if constexpr (BLOCKED) mbar_arrive(landed_bar(l));
                    }
                }
            }
        }
    } else {
        // ================= epilogue (warps 0..7) =================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kT3EpiRegs));
        const int qd = warp & 3;                        // TMEM lane quadrant
        const int g = warp >> 2;                        // columns 64 g .. 64 g + 63 of Q and of P
        unsigned acc_it = 0, exch_it = 0;
        bool live = true;
        for (long long w = blockIdx.x; w < P.n_items && live; w += gridDim.x) {
            const int4 itm = P.items[(int)(w % P.ipc)];
            const long long gch = w / P.ipc;
            const int row0 = itm.x, col0 = itm.y, n = itm.z;
            const bool diag = itm.w != 0;
            const bool act = row0 + 32 * qd < ((SEG || P.group > 1) ? n : 2 * P.N);   // some of this warp's rows are inputs
            float2 Q[32], V[32];                         // column pairs, for packed adds
#pragma unroll
            for (int k = 0; k < 32; ++k) Q[k] = V[k] = make_float2(0.f, 0.f);
            for (int k0 = 0; k0 < P.nk; k0 += P.chunk, ++acc_it) {
                const int ab = (int)(acc_it & 1);
                const bool got = t3wait(accf_bar(ab), (acc_it >> 1) & 1u, abort_flag, P, 3);
                if (!__all_sync(0xffffffffu, got)) {
                    live = false;
                    break;
                }
                tc_fence_after();
                const unsigned t = tmem_base + ((unsigned)(32 * qd) << 16) + (unsigned)(ab * kT3AccCols + 64 * g);
                if (act) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (64 * g + 16 * u < n) {
                            float a[16], b[16];
                            tmem_ld16(t + 16 * u, a);
                            tmem_ld16(t + (unsigned)n + 16 * u, b);
                            tmem_ld_wait();
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                Q[8 * u + k] = make_float2(Q[8 * u + k].x + a[2 * k], Q[8 * u + k].y + a[2 * k + 1]);
                                V[8 * u + k] = make_float2(V[8 * u + k].x + b[2 * k], V[8 * u + k].y + b[2 * k + 1]);
                            }
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acce_bar(ab));
            }
            if (!live) break;
            auto sync8 = [&]() {
                __syncwarp();
                if (lane == 0) mbar_arrive(exch_bar);
                const bool got = t3wait(exch_bar, exch_it & 1u, abort_flag, P, 3);
                ++exch_it;
                return __all_sync(0xffffffffu, got) != 0;
            };
            if (diag) {
                // Re V = (P + P') / 2, Im V = Q - Q': each warp puts its 32 x 32 blocks
                // on or below the diagonal into the scratch and reads the mirror
                // blocks of those on or above it (rows of 33 words: no bank
                // conflicts), all ten blocks at once or, with less scratch, the diagonal
                // ones last, after three and three others or (blocked) six at once. Blocked
                // channels or segments of up to 32 inputs pass the diagonal ones only.
                const bool diag_only = BLOCKED && P.gin <= 32;
                const int phases = diag_only || P.scratch_bytes >= kT3Scratch     ? 1
                                   : BLOCKED && P.scratch_bytes >= kT3ScratchMid ? 2
                                                                                 : 3;
                auto place = [&](int r, int c, int &slot) {     // block (r, c), c <= r: phase and slot
                    if (!diag_only && phases == 1) {
                        slot = r * (r + 1) / 2 + c;
                        return 0;
                    }
                    const int o = r * (r - 1) / 2 + c;
                    slot = r == c ? r : phases == 2 ? o : o % 3;
                    return r == c ? phases - 1 : diag_only ? -1 : phases == 2 ? 0 : o / 3;
                };
                auto put = [&](const float2 (&A)[32], int phase) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int cb = 2 * g + h;
                        int slot;
                        if (act && cb <= qd && 32 * cb < n && place(qd, cb, slot) == phase) {
                            float *s = scratch + slot * kT3Blk + lane * 33;
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                s[2 * j] = A[16 * h + j].x;
                                s[2 * j + 1] = A[16 * h + j].y;
                            }
                        }
                    }
                };
                auto take = [&](float2 (&A)[32], int phase, float keep, float other) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int cb = 2 * g + h;
                        int slot;
                        if (act && cb >= qd && 32 * cb < n && place(cb, qd, slot) == phase) {
                            const float *s = scratch + slot * kT3Blk + lane;
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                float2 &v = A[16 * h + j];
                                v.x = fmaf(other, s[66 * j], keep * v.x);
                                v.y = fmaf(other, s[66 * j + 33], keep * v.y);
                            }
                        }
                    }
                };
                for (int ph = 0; ph < phases && live; ++ph) {
                    put(V, ph);
                    live = sync8();
                    if (!live) break;
                    take(V, ph, 0.5f, 0.5f);
                    live = sync8();
                }
                for (int ph = 0; ph < phases && live; ++ph) {
                    put(Q, ph);
                    live = sync8();
                    if (!live) break;
                    take(Q, ph, 1.f, -1.f);
                    live = sync8();
                }
                if (!live) break;
            }
            // this lane's row input (blocked: rows pol by pol within eight stations, as
            // are the columns, so column k's other pol is QN columns on)
            constexpr int QN = BLOCKED ? 8 : 1;
            const int slot = (row0 >> 1) + 16 * qd + (BLOCKED ? 8 * (lane >> 4) + (lane & 7) : lane >> 1);
            const int p = BLOCKED ? (lane >> 3) & 1 : lane & 1;
            // a group's channels (or segments) take P.gin / 2 station slots each
            const int cg = (SEG || P.group > 1) ? slot / (P.gin >> 1) : 0;
            const int first = cg * (P.gin >> 1), i = slot - first;
            const long long ch = gch * P.group + cg;
            const bool mine = act && cg < P.group && ch < P.channels;
            if constexpr (SEG) {
                // the segments' diagonal blocks through the scratch (planes Re, Im of segs x
                // gin x gin), then each entry's sum over the segments in their order
                const int area = P.gin * P.gin, plane = P.segs * area;
                const int row = 32 * qd + lane - cg * P.gin, from = cg * P.gin - 64 * g;
                if (act && cg < P.segs) {
                    float *s = scratch + cg * area + row * P.gin - from;
#pragma unroll
                    for (int k = 0; k < 64; ++k)
                        if ((unsigned)(k - from) < (unsigned)P.gin) {
                            s[k] = k & 1 ? V[k / 2].y : V[k / 2].x;
                            s[plane + k] = k & 1 ? Q[k / 2].y : Q[k / 2].x;
                        }
                }
                live = sync8();
                if (!live) break;
                for (int e = threadIdx.x; e < area; e += 32 * kT3EpiWarps) {
                    const int a = e / P.gin, b = e - a * P.gin;
                    const int ei = BLOCKED ? 8 * (a >> 4) + (a & 7) : a >> 1, ep = BLOCKED ? (a >> 3) & 1 : a & 1;
                    const int ej = BLOCKED ? 8 * (b >> 4) + (b & 7) : b >> 1, eq = BLOCKED ? (b >> 3) & 1 : b & 1;
                    if (ei > ej || ej >= P.N) continue;
                    float2 v = make_float2(0.f, 0.f);
                    for (int c = 0; c < P.segs; ++c) {
                        v.x += scratch[c * area + e];
                        v.y += scratch[plane + c * area + e];
                    }
                    float2 *dst = P.vis + (gch * P.B + (long long)ej * (ej + 1) / 2 + ei) * 4 + 2 * ep + eq;
                    if (P.accumulate) v = make_float2(v.x + dst->x, v.y + dst->y);
                    *dst = v;
                }
                live = sync8();
                if (!live) break;
                continue;
            }
            float2 *vrow = P.vis + ch * P.B * 4 + (long long)i * 4 + 2 * p;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!mine || 64 * g + 32 * h >= n || (diag && 2 * g + h < qd)) continue;
#pragma unroll
                for (int jj = 0; jj < 16; ++jj) {
                    const int j = (col0 >> 1) + 32 * g + 16 * h + jj - first;
                    if (i <= j && j < P.N) {
                        const int k = 32 * h + (BLOCKED ? 16 * (jj >> 3) + (jj & 7) : 2 * jj);
                        auto at = [](const float2 (&A)[32], int c) { return c & 1 ? A[c / 2].y : A[c / 2].x; };
                        float4 v = make_float4(at(V, k), at(Q, k), at(V, k + QN), at(Q, k + QN));
                        float4 *dst = reinterpret_cast<float4 *>(vrow + (long long)j * (j + 1) / 2 * 4);
                        if (P.accumulate) {
                            const float4 o = *dst;
                            v = make_float4(v.x + o.x, v.y + o.y, v.z + o.z, v.w + o.w);
                        }
                        *dst = v;
                    }
                }
            }
        }
    }

    __syncthreads();
    if (warp == kT3MmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kT3TmemCols)
                     : "memory");
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn t3_encode_fn()
{
    static EncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(p);
        return static_cast<EncodeTiledFn>(nullptr);
    }();
    return fn;
}

// Channels per item. A tile has 128 rows whatever the station count and a stage
// takes about the same time (0.45 us with 16 inputs, 0.6 us with 128), so small
// arrays share one: G channels' inputs side by side, of whose products only the
// G diagonal blocks are written. As many as fit while every SM still gets an item
// (15616 channels x 256 spectra of 8 stations: blocked 1.10 ms alone, 0.24 ms in
// eights, planar 0.77 and 0.15 ms).
int t3_group(int I_pad, long long channels, int num_sms)
{
    if (I_pad > 64) return 1;
    return (int)std::max<long long>(1, std::min<long long>(128 / I_pad, channels / num_sms));
}

// Time segments per item where the handle has not even two channels per SM to group: up
// to 24 stations (48 inputs), a channel's spectra in 128 / I_pad segments side by
// side, at least four stages each, whose diagonal blocks are summed at the end (8
// stations x 64 channels x 768 spectra: 29 us in one, 16 us in eight). More stations leave
// no room in the tile, or in the scratch for the blocks.
int t3_segments(int I_pad, int group, int nk)
{
    static_assert(2u * 2u * 48u * 48u * 4u <= kT3Scratch && 2u * 4u * 32u * 32u * 4u <= kT3ScratchMid,
                  "the segments' blocks fit the scratch (two of 48 inputs leave the tile below 128)");
    return group > 1 || I_pad > 48 ? 1 : std::max(1, std::min(128 / I_pad, nk / 4));
}

// Item list of one channel (or group) and the shared-memory geometry it needs.
struct T3Plan {
    std::vector<int4> items;
    unsigned stage_bytes = 0, land_bytes = 0, row_land = 0, scratch_bytes = 0;
    int stages = 0, lands = 0;
};

bool t3_plan(int I_pad, bool blocked, int side, T3Plan &pl)
{
    constexpr int NT = 64;                              // columns of an off-diagonal item
    pl.items.clear();
    unsigned nmax = 0, ndmax = 0;                       // widest off-diagonal and diagonal item
    const unsigned trow = blocked ? 64u : 128u;         // bytes of a TF32 row; planar: in the landing slot
    unsigned tf = 0, bf = 0;
    for (int row0 = 0; row0 < I_pad; row0 += 128) {
        const unsigned nd = (unsigned)std::min(128, I_pad - row0) * side;
        pl.items.push_back(make_int4(row0, row0, (int)nd, 1));
        // the planes, and the 128-row reads of the A operands J (TF32) and hJ (BF16)
        tf = std::max(tf, std::max((blocked ? 6u : 2u) * nd, nd + 128u) * trow);
        bf = std::max(bf, std::max(6u * nd, nd + 128u) * kT3BfRow);
        ndmax = std::max(ndmax, nd);
        for (int c0 = row0 + 128; c0 < I_pad; c0 += NT) {
            const int n = std::min(NT, I_pad - c0);
            pl.items.push_back(make_int4(row0, c0, n, 0));
            nmax = std::max(nmax, (unsigned)n);
            tf = std::max(tf, (blocked ? 512u + 6u * n : 256u + 3u * n) * trow);
            bf = std::max(bf, (512u + 6u * n) * kT3BfRow);
        }
    }
    if ((int)pl.items.size() > kT3MaxItems) return false;
    const unsigned k1 = 1023u;
    pl.stage_bytes = ((blocked ? tf : bf) + k1) & ~k1;
    pl.land_bytes = ((blocked ? (64u + nmax / 2) * kT3StRun : tf) + k1) & ~k1;
    pl.row_land = nmax / 2 * kT3StRun;
    // off-diagonal items have larger stages: the small scratch makes room for a third
    // of them up to 80 stations (planar, 78 stations x 1024 channels x 1001 spectra: 873 -> 779 us)
    // and so does the middle one beside full blocked tiles
    pl.scratch_bytes = nmax ? kT3ScratchSmall : blocked && ndmax == 128u ? kT3ScratchMid : kT3Scratch;
    const unsigned room = kT3SmemMax - 1024u - pl.scratch_bytes - kT3Ctrl;
    pl.stages = std::min<int>(kT3MaxStages - 1, (int)(room / (pl.stage_bytes + pl.land_bytes)));
    // blocked slots hold one stage: one more of them where it fits
    pl.lands = pl.stages + (blocked && (pl.stages + 1) * pl.land_bytes + pl.stages * pl.stage_bytes <= room ? 1 : 0);
    return pl.stages >= kT3ConvGroups;
}

template <bool BLOCKED>
cudaError_t t3_launch(const Handle &h, const void *corr, float2 *vis, cudaStream_t st, bool accumulate, int chunk)
{
    T3Plan pl;
    const long long channels = (long long)h.p.n_subbands * h.p.n_channels;
    const int nk = (h.p.n_spectra + kT3K - 1) / kT3K;
    // Time segments change the order of the sums, so the whole handle's channels decide on
    // them and a launch over some of its subbands gives the same bits; sharing a tile
    // changes no sum, and goes by the launch's own channels.
    const long long all = (long long)h.n_subbands_all * h.p.n_channels;
    const int segs = t3_segments(h.I_pad, t3_group(h.I_pad, all, h.num_sms), nk);
    const int group = t3_group(h.I_pad, channels, h.num_sms);
    if (!t3_plan(h.I_pad, BLOCKED, group * segs, pl)) return cudaErrorNotSupported;
    if (2 * channels > 0x7fffffffLL) return cudaErrorInvalidValue;
    T3Params P;
    memset(&P, 0, sizeof(P));
    if constexpr (BLOCKED) {
        P.blk = static_cast<const unsigned char *>(corr);
    } else {
        EncodeTiledFn enc = t3_encode_fn();
        if (!enc) return cudaErrorNotSupported;
        const cuuint64_t gdim[3] = {(cuuint64_t)h.S_pad, (cuuint64_t)h.I_pad, (cuuint64_t)(2 * channels)};
        const cuuint64_t gstride[2] = {(cuuint64_t)h.S_pad * 4, (cuuint64_t)h.S_pad * 4 * h.I_pad};
        const cuuint32_t estr[3] = {1, 1, 1};
        P.nr = (h.I_pad - 1) % 128 + 1;
        CUtensorMap *const maps[3] = {&P.map128, &P.mapr, &P.map16};
        const int rows[3] = {128, P.nr, 16};
        for (int m = 0; m < 3; ++m) {
            const cuuint32_t box[3] = {2 * kT3K, (cuuint32_t)rows[m], 1};
            if (enc(maps[m], CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<void *>(corr), gdim, gstride, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return cudaErrorInvalidValue;
        }
    }
    for (size_t k = 0; k < pl.items.size(); ++k) P.items[k] = pl.items[k];
    P.ipc = (int)pl.items.size();
    P.vis = vis;
    P.status = h.d_status;
    P.channels = channels;
    P.group = group;
    P.gin = h.I_pad;
    P.n_items = (channels + group - 1) / group * P.ipc;
    P.N = h.p.n_stations;
    P.S = h.p.n_spectra;
    P.segs = segs;
    P.nk_all = nk;
    P.nk = (nk + segs - 1) / segs;
    if (!BLOCKED && segs > 1) P.nk = (P.nk + 1) / 2 * 2;   // landing slots hold two stages
    P.chunk = chunk;
    P.B = h.B;
    P.stages = pl.stages;
    P.lands = pl.lands;
    P.stage_bytes = pl.stage_bytes;
    P.land_bytes = pl.land_bytes;
    P.row_land = pl.row_land;
    P.scratch_bytes = pl.scratch_bytes;
    P.timeout_cycles = h.tc_timeout_cycles;
    P.no_tma = h.tc_test_no_tma;
    P.accumulate = accumulate ? 1 : 0;
    const size_t smem = 1024 + (size_t)pl.stages * pl.stage_bytes + (size_t)pl.lands * pl.land_bytes + pl.scratch_bytes +
                        kT3Ctrl;
    auto kern = segs > 1 ? xcorr_split_kernel<BLOCKED, true> : xcorr_split_kernel<BLOCKED, false>;
    // the register split draws on what the launch brings: refuse a build with less
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    if (fa.numRegs < kT3LaunchRegs) return cudaErrorNotSupported;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long grid = std::min<long long>(P.n_items, h.num_sms);
    if (grid <= 0) return cudaSuccess;
    kern<<<(unsigned)grid, kT3Threads, smem, st>>>(P);
    return cudaGetLastError();
}

}  // namespace

bool xsplit_supported(int I_pad)
{
    T3Plan pl;
    return t3_plan(I_pad, false, 1, pl);
}

cudaError_t launch_xcorr_split(const Handle &h, const float *corr, float2 *vis, cudaStream_t st, bool accumulate)
{
    return t3_launch<false>(h, corr, vis, st, accumulate, 4);   // 64 spectra per accumulator chain
}

// FX_F32 goes to the tensor cores where that is at least as accurate as the
// CUDA-core FMA chain, whose error grows with its length. Against FP64, over all
// baselines normwise / over the cross baselines, error as a multiple of the
// chain's (8, 50 and 76 stations; the chain has 2.4e-7 at 128 spectra, 4e-7 at 384,
// 6e-7 at 768, 1.2e-6 at 3072):
//   spectra (accumulator chain)    128 (16)    384 (16)    768 (16)    768 (32)   1024 (32)   3072 (32)
//   uncorrelated noise            0.74 0.46   0.46 0.30   0.35 0.24   0.73 0.43   0.56 0.37   0.37 0.24
//   with a common signal          0.65 0.44   0.37 0.27   0.26 0.21   0.53 0.41   0.49 0.39   0.26 0.23
//   half of the spectra lost      0.86 0.80   0.59 0.54   0.44 0.44   0.79 0.63   0.63 0.56   0.43 0.37
// So chains of 32 from 768 spectra on, or from 1024 on where autocorrelations, which
// lose most to a longer chain, are most of the norm (up to 32 stations); at 128
// spectra they would have up to 1.7, at 384 1.2 (half lost). They drain the
// accumulator half as often (64 stations x 1280 channels x 1024 spectra 476 us,
// with 16 583, CUDA cores 2056). What the chain length cannot mend is a
// baseline with few live spectra, where an FMA chain barely rounds: with 64 of them
// 0.9 and 0.8 of its error, with 16 1.2 and 1.2, 4 2.1 and 2.0, one 3.4 and 3.3
// (1e-7 of the product). Shorter integrations and the forms asked for by flag stay
// on the CUDA cores.
constexpr int kXf32TcSpectra = 128;

bool xf32_on_tensor_cores(const Handle &h)
{
    T3Plan pl;
    return (h.p.flags & (FX_FLAG_XF32_CUDA_CORES | FX_FLAG_XF32_SMALL_TILES | FX_FLAG_XF32_THREE_MULT)) == 0 &&
           h.p.n_spectra >= kXf32TcSpectra && t3_plan(h.I_pad, true, 1, pl);
}

cudaError_t launch_xcorr_f32_tc(const Handle &h, const float2 *corr, float2 *vis, cudaStream_t st, bool accumulate)
{
    return t3_launch<true>(h, corr, vis, st, accumulate, h.p.n_spectra >= (h.I_pad > 64 ? 768 : 1024) ? 2 : 1);
}

}  // namespace fxi
