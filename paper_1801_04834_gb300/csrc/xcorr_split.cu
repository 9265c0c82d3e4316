// xcorr_split.cu -- FP32-accurate X-stage on the tcgen05 tensor cores, any
// station count: FP32 corrected samples split in the kernel into hi + lo,
// V ~ hi hi' + hi lo' + lo hi' (lo lo' dropped), the main term hi hi' as TF32
// MMAs and the cross terms as BF16 MMAs, FP32 accumulation in TMEM, chunk
// sums added in IEEE FP32 in registers. Serves FX_TF32_SPLIT (planar FP32
// operands) and FX_F32 (spectrum-blocked complex operands).
//
// Paper, Sec. "Signal processing with GPU kernels": the correlator forms
// V[a][b] = sum_s Y[s][a] conj(Y[s][b]) for all input pairs and integrates over
// the block, in single precision. TF32 keeps FP32's exponent range with an
// 11-bit significand; hi = x with its 13 low mantissa bits cleared is exactly
// a TF32 value and lo = x - hi is exact in FP32 with |lo| < 2^-10 |x|. The
// cross terms hi lo' and lo hi' are each below 2^-10 of the product, so they
// tolerate BF16 operands: rounding hi and lo to BF16 (8-bit significand, FP32
// exponent range, round to nearest) changes a cross term by at most 2^-8 of
// itself, i.e. 2^-18 of the product in the worst case and about 2^-21 RMS,
// with zero mean; the dropped lo lo' term is below 2^-20 of the product.
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
//   BF16 (K = 16):             hJ x [lR; 2lJ], hR x [-lJ; 2lR] (N = 2n)
// into one accumulator of 2n columns [Q | P]: 640 tensor clocks and 64 KB of
// operand reads, against 1024 clocks and 96 KB with all products formed, and
// 24 KB of converter stores against 32 KB. 64 stations x 1280 channels x 3072
// spectra (4.0 GB of operands): planar 1.45 ms with every product formed and
// the chunk sums reduced in L2, 0.98 ms so (4.1 TB/s; without its MMAs the
// kernel takes 0.66 ms, without its converter 0.95 ms); blocked 1.26 ms,
// against 6.09 ms on the CUDA cores.
//
// Work items. Rows come in blocks of 128 inputs (M = 128); an item is
// (subband x channel, row block, column block) over the upper block
// triangle: the diagonal item of a row block covers columns
// [row0, row0 + min(128, I_pad - row0)), off-diagonal items cover the columns
// right of it in tiles of at most 64 inputs and form every product:
//   TF32: hJ_a x [hR; hJ], hR_a x [-hJ; hR]
//   BF16: hJ_a x [lR; lJ], hR_a x [-lJ; lR], lJ_a x [hR; hJ], lR_a x [-hJ; hR]
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
//             to TF32 (which halves lo) as 64-byte rows, 64-byte swizzle.
// Planes of n rows each:
//   diagonal item:     TF32 R, J; BF16 hR, hJ, lR, 2lJ, -lJ, 2lR. The A operands
//                      are planes R, J, hR, hJ read as 128-row tiles: rows past n
//                      are other planes' data and only reach accumulator rows
//                      that are not used; the regions are large enough that
//                      these reads stay inside.
//   off-diagonal item: 128-row planes TF32 R, J, BF16 hR, hJ, lR, lJ of the row
//                      inputs; TF32 -J, R, J, BF16 -hJ, hR, hJ, -lJ, lR, lJ of
//                      the columns.
//
// Accumulation. The tensor core's FP32 accumulator does not round each
// addition to nearest, so a long chain of MMAs into one accumulator drifts
// (about 2^-24 of the running value per MMA). The accumulator is restarted
// every `chunk` stages and the chunk sums are added in registers (round to
// nearest): the eight epilogue warps hold the whole 128 x 256 accumulator, 128
// registers per thread, so nothing is read back or reduced in memory until
// the item ends. 64 spectra per chunk for FX_TF32_SPLIT; 16 for FX_F32, whose
// reference is the rounding of an FP32 FMA chain (measured in
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
constexpr int kT3Bars = 4 * kT3MaxStages + 6;         // full, conv, empty, landed per stage; accf 2, acce 2, exch, drain
constexpr int kT3Blk = 32 * 33;                       // one 32 x 32 block of the transpose scratch, padded rows
constexpr unsigned kT3Scratch = 10u * kT3Blk * 4u;    // lower block triangle of a 128 x 128 plane
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
    unsigned scratch_bytes;   // kT3Scratch or kT3ScratchSmall
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

// One value's hi part (a TF32 value) and, through *lo, x - hi.
//  TRUNC  the 13 low bits cleared: what a TF32 MMA reads of the raw value
//  ROUND  rounded to nearest: lo is half as large and has both signs
//  SAFE   as TRUNC, and an infinity has no low part (inf - inf would turn its
//         products into NaN); for the values ROUND could carry to infinity
enum SplitMode { TRUNC, ROUND, SAFE };
template <int MODE>
__device__ __forceinline__ float split1(float x, float *lo)
{
    const unsigned b = __float_as_uint(x);
    const float h = __uint_as_float((MODE == ROUND ? b + 0x1000u : b) & 0xFFFFE000u);
    *lo = MODE == SAFE && fabsf(x) == __int_as_float(0x7f800000) ? 0.f : x - h;
    return h;
}
constexpr unsigned kT3RoundMax = 0x7f7f0000u;          // FP32 bits from which SAFE is taken, below
constexpr unsigned kT3BfMax = 0x7f7f8000u;             // those that round to infinity in BF16

// hi and lo parts of four FP32 values: hi in FP32, both in BF16 (round to nearest even)
struct Split4 {
    float4 hf;
    uint2 h, l;
};
template <int MODE>
__device__ __forceinline__ Split4 split4(float4 x)
{
    Split4 r;
    float4 l;
    r.hf.x = split1<MODE>(x.x, &l.x);
    r.hf.y = split1<MODE>(x.y, &l.y);
    r.hf.z = split1<MODE>(x.z, &l.z);
    r.hf.w = split1<MODE>(x.w, &l.w);
    // SAFE: what BF16 would round to infinity takes no part in the cross terms, whose
    // signs are not the product's (inf - inf); the main term carries the infinity
    auto b = [](float h) { return MODE == SAFE && fabsf(h) >= __uint_as_float(kT3BfMax) ? 0.f : h; };
    r.h = make_uint2(bf16x2(b(r.hf.x), b(r.hf.y)), bf16x2(b(r.hf.z), b(r.hf.w)));
    r.l = make_uint2(bf16x2(l.x, l.y), bf16x2(l.z, l.w));
    return r;
}

// Operand planes: DIAG column planes of a diagonal item (BF16 hR, hJ, lR, 2lJ,
// -lJ, 2lR), COLS column planes of an off-diagonal item (BF16 -hJ, hR, hJ, -lJ,
// lR, lJ; a TF32 plane -J before R and J), ROWS row planes of an off-diagonal
// item (BF16 hR, hJ, lR, lJ).
enum PlaneRole { DIAG, COLS, ROWS };
template <int ROLE>
__device__ __forceinline__ void put_bf(const Split4 &a, const Split4 &b, unsigned char *bf, unsigned bp)
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
        put_bf<ROLE>(split4<TRUNC>(x), split4<TRUNC>(y), bf + r8 * 256 + bo, bp);
    }
}

// Spectrum-blocked operands: `land` holds stations' runs of [16 spectra][2
// pols] complex values; a task is 4 spectra of one station, both pols, written
// to the TF32 planes (64-byte rows, 64-byte swizzle, pitch tp) too. Spectra from
// s_lim on count as zero (every gst stations seg fewer: time segments). The four 16-byte reads of a task are rotated by
// lane / 2 so that eight lanes' reads fall on distinct banks, and sorted again
// in registers. Rows are ordered pol by pol within eight stations (row 16 (st /
// 8) + 8 p + st mod 8), so that the lanes of a store take consecutive rows and
// distinct banks too.
template <int ROLE, bool SEG>
__device__ __forceinline__ void convert_blocked(const unsigned char *land, unsigned char *tf, unsigned tp,
                                                unsigned char *bf, unsigned bp, int rows, int s_lim, int gst, int seg, int t)
{
    const int nt = rows / 2 * 4;                          // a multiple of 32: whole warps
    const int rot = (t >> 1) & 3;
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
        float top = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            top = fmaxf(fmaxf(fmaxf(top, fabsf(v[e].x)), fabsf(v[e].y)), fmaxf(fabsf(v[e].z), fabsf(v[e].w)));
        const bool safe = __any_sync(0xffffffffu, top >= __uint_as_float(kT3RoundMax));
        auto put = [&](auto mode) {
            constexpr int MODE = decltype(mode)::value;
#pragma unroll
            for (int p = 0; p < kPols; ++p) {
                const int r = 16 * (st >> 3) + 8 * p + (st & 7);
                const Split4 x = split4<MODE>(p ? make_float4(v[0].z, v[1].z, v[2].z, v[3].z)
                                                : make_float4(v[0].x, v[1].x, v[2].x, v[3].x));
                const Split4 y = split4<MODE>(p ? make_float4(v[0].w, v[1].w, v[2].w, v[3].w)
                                                : make_float4(v[0].y, v[1].y, v[2].y, v[3].y));
                unsigned char *o = tf + tf_off(r, lc);
                *reinterpret_cast<float4 *>(o) = x.hf;
                *reinterpret_cast<float4 *>(o + tp) = y.hf;
                if constexpr (ROLE == COLS) *reinterpret_cast<float4 *>(o - tp) = neg4(y.hf);
                put_bf<ROLE>(x, y, bf + bf_off(r, lc), bp);
            }
        };
        if (safe) put(std::integral_constant<int, SAFE>{});
        else put(std::integral_constant<int, ROUND>{});
    }
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
    unsigned *tmem_slot = reinterpret_cast<unsigned *>(ctrl + 8 * kT3Bars);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
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
                    const unsigned bf0 = BLOCKED ? (diag ? 2 * tp : (2 * TA + 4 * kT3ABf) / 16 + 3 * tp)
                                                 : (diag ? 0u : 4 * kT3ABf / 16);
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
                            if (diag) {
                                // (the small cross terms first, while the accumulator is small: 10% less
                                // error than after the main term)
                                mma_f16(d, bf + bp, bf + 2 * bp, idb, kc ? 1u : 0u);                 // hJ x [lR; 2lJ]
                                mma_f16(d, bf, bf + 4 * bp, idb, 1u);                                // hR x [-lJ; 2lR]
#pragma unroll
                                for (int kk = 0; kk < kT3K / 8; ++kk)      // 8 FP32 = 32 bytes per TF32 K-step
                                    mma_tf32(d, tf + tp + 2u * kk, tf + 2u * kk, id2, 1u);           // hJ x [hR; hJ]
#pragma unroll
                                for (int kk = 0; kk < kT3K / 8; ++kk)
                                    mma_tf32(d + (unsigned)n, tf + 2u * kk, tf + 2u * kk, id1, 1u);  // hR x hR
                            } else {
                                // rows: TF32 R, J, BF16 hR, hJ, lR, lJ; columns: TF32 -J, R, J, BF16 -hJ, hR, hJ, -lJ, lR, lJ
                                const unsigned long long ra = bdesc0 + so + (BLOCKED ? 2 * TA / 16 : 0u);
                                const unsigned long long tb = tf + (BLOCKED ? 2 * TA + 4 * kT3ABf : 2 * TA) / 16;
                                constexpr unsigned AP = kT3ABf / 16;
                                mma_f16(d, ra + AP, bf + 4 * bp, idb, kc ? 1u : 0u);  // hJ x [lR; lJ]
                                mma_f16(d, ra, bf + 3 * bp, idb, 1u);                 // hR x [-lJ; lR]
                                mma_f16(d, ra + 3 * AP, bf + bp, idb, 1u);            // lJ x [hR; hJ]
                                mma_f16(d, ra + 2 * AP, bf, idb, 1u);                 // lR x [-hJ; hR]
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
                        if (diag) {
                            convert_blocked<DIAG, SEG>(la, st, pitch, st + 2 * pitch, bpitch, n, lim, gst, seg, ct);
                        } else {
                            unsigned char *tb = st + 2 * TA + 4 * kT3ABf;
                            convert_blocked<ROWS, false>(la + P.row_land, st, TA, st + 2 * TA, kT3ABf, 128, lim, gst, seg, ct);
                            convert_blocked<COLS, false>(la, tb + pitch, pitch, tb + 3 * pitch, bpitch, n, lim, gst, seg, ct);
                        }
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
                // conflicts), all ten blocks at once or, with the small scratch, in
                // three phases of three, three and the four diagonal ones
                const bool small = P.scratch_bytes < kT3Scratch;
                auto place = [&](int r, int c, int &slot) {     // block (r, c), c <= r: phase and slot
                    if (!small) {
                        slot = r * (r + 1) / 2 + c;
                        return 0;
                    }
                    const int o = r * (r - 1) / 2 + c;
                    slot = r == c ? r : o % 3;
                    return r == c ? 2 : o / 3;
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
                for (int ph = 0; ph < (small ? 3 : 1) && live; ++ph) {
                    put(V, ph);
                    live = sync8();
                    if (!live) break;
                    take(V, ph, 0.5f, 0.5f);
                    live = sync8();
                }
                for (int ph = 0; ph < (small ? 3 : 1) && live; ++ph) {
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
// (15616 channels x 256 spectra of 8 stations: blocked 1.10 ms alone, 0.23 ms in
// eights, planar 0.77 and 0.15 ms).
int t3_group(int I_pad, long long channels, int num_sms)
{
    if (I_pad > 64) return 1;
    return (int)std::max<long long>(1, std::min<long long>(128 / I_pad, channels / num_sms));
}

// Time segments per item where there are not even two channels per SM to group: up
// to 24 stations (48 inputs), a channel's spectra in 128 / I_pad segments side by
// side, at least four stages each, whose diagonal blocks are summed at the end (8
// stations x 64 channels x 768 spectra: 29 us in one, 16 us in eight). More stations leave
// no room in the tile, or in the scratch for the blocks.
int t3_segments(int I_pad, int group, int nk)
{
    static_assert(2u * 2u * 48u * 48u * 4u <= kT3Scratch && 2u * 4u * 32u * 32u * 4u <= kT3Scratch,
                  "the segments' blocks fit the scratch");
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
    unsigned nmax = 0;                                  // widest off-diagonal item
    const unsigned trow = blocked ? 64u : 128u;         // bytes of a TF32 row; planar: in the landing slot
    unsigned tf = 0, bf = 0;
    for (int row0 = 0; row0 < I_pad; row0 += 128) {
        const unsigned nd = (unsigned)std::min(128, I_pad - row0) * side;
        pl.items.push_back(make_int4(row0, row0, (int)nd, 1));
        // the planes, and the 128-row reads of the A operands J (TF32) and hJ (BF16)
        tf = std::max(tf, std::max(2u * nd, nd + 128u) * trow);
        bf = std::max(bf, std::max(6u * nd, nd + 128u) * kT3BfRow);
        for (int c0 = row0 + 128; c0 < I_pad; c0 += NT) {
            const int n = std::min(NT, I_pad - c0);
            pl.items.push_back(make_int4(row0, c0, n, 0));
            nmax = std::max(nmax, (unsigned)n);
            tf = std::max(tf, (256u + 3u * n) * trow);
            bf = std::max(bf, (512u + 6u * n) * kT3BfRow);
        }
    }
    if ((int)pl.items.size() > kT3MaxItems) return false;
    // (blocked: both regions in one stage, BF16 planes right after that item's TF32
    // planes, so a diagonal item's need is below the sum too)
    const unsigned k1 = 1023u;
    pl.stage_bytes = ((blocked ? tf + bf : bf) + k1) & ~k1;
    pl.land_bytes = ((blocked ? (64u + nmax / 2) * kT3StRun : tf) + k1) & ~k1;
    pl.row_land = nmax / 2 * kT3StRun;
    // off-diagonal items have larger stages: the small scratch makes room for a third
    // of them up to 80 stations (78 stations x 1024 channels x 1001 spectra: 873 -> 779 us)
    pl.scratch_bytes = nmax ? kT3ScratchSmall : kT3Scratch;
    const unsigned room = kT3SmemMax - 1024u - pl.scratch_bytes - 8u * kT3Bars - 16u;
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
    const int group = t3_group(h.I_pad, channels, h.num_sms);
    const int nk = (h.p.n_spectra + kT3K - 1) / kT3K;
    const int segs = t3_segments(h.I_pad, group, nk);
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
                        8 * kT3Bars + 16;
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

cudaError_t launch_xcorr_split(const Handle &h, const float *corr, float2 *vis, cudaStream_t st)
{
    return t3_launch<false>(h, corr, vis, st, false, 4);   // 64 spectra per accumulator chain
}

// FX_F32 goes to the tensor cores where that is at least as accurate as the
// CUDA-core FMA chain, whose error grows with its length: against FP64 on
// noise with a common signal (normwise, 2 to 130 stations) the chain has
// 2.4e-7 at 128 spectra, 3.2e-7 at 256, 4.2e-7 at 384, 6.4e-7 at 1024, 8.5e-7 at
// 1536, 1.2e-6 at 3072; the split has 1.6e-7 to 2.4e-7 from 128 spectra on with
// accumulator chains of 16 spectra, 2.5e-7 to 3.3e-7 with 32 and 4.8e-7 to
// 6.9e-7 with 64. Longer chains drain less often (64 stations x 1280 channels
// x 3072 spectra: 1.53 ms with 16, 1.26 ms with 64; CUDA cores 6.09 ms), so the
// longest that stays below the FMA chain is taken. Shorter integrations and the
// forms asked for by flag stay on the CUDA cores.
constexpr int kXf32TcSpectra = 128;

bool xf32_on_tensor_cores(const Handle &h)
{
    T3Plan pl;
    return (h.p.flags & (FX_FLAG_XF32_SMALL_TILES | FX_FLAG_XF32_THREE_MULT)) == 0 &&
           h.p.n_spectra >= kXf32TcSpectra && t3_plan(h.I_pad, true, 1, pl);
}

cudaError_t launch_xcorr_f32_tc(const Handle &h, const float2 *corr, float2 *vis, cudaStream_t st, bool accumulate)
{
    const int S = h.p.n_spectra;
    return t3_launch<true>(h, corr, vis, st, accumulate, S >= 1536 ? 4 : S >= 384 ? 2 : 1);
}

}  // namespace fxi
