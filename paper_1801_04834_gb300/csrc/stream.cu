// stream.cu -- streaming blocks: FIR history kept in the handle, integer-sample
// coarse delay per station, per-baseline counts of valid spectra.
//
// Paper, Sec. "Signal processing with GPU kernels": FIR filter history is
// carried across to the next block. Sec. "Software architecture": the coarse
// (whole-sample) delay is applied by the transpose stage through a circular
// buffer, and lost data is recorded in metadata.
//
// Stream coordinates: t = 0 is the first new sample of the current call, new
// samples are t in [0, S*C), the history holds the hist_len = (T-1)*C +
// max_shift samples before it (zeros before the first call). Station n's
// block is its stream over [-(T-1)*C - d_n, S*C - d_n): the assembled block
// is then an ordinary raw block for the channeliser. After the call the
// history becomes the last hist_len samples of the stream, written to the
// other buffer of a ping-pong pair.
#include "internal.h"

namespace fxi {
namespace {

constexpr int kStatusBadShift = 5;

// One thread writes 16 bytes of a (station, subband)'s block; the source is
// sample-aligned only (the coarse shift), so it is read sample by sample, a
// warp's reads being contiguous all the same. Bound by the bytes moved: 62
// stations x 12 subbands x 3072 spectra of int16 (2.4 GB) 352 us, 6.7 TB/s (one
// sample per thread with a 64-bit division each: 632 us).
template <typename U>
__global__ void __launch_bounds__(256)
stream_assemble_kernel(const U *__restrict__ hist, const U *__restrict__ nw, const int *__restrict__ shift,
                       uint4 *__restrict__ block, int *status, int N, int L, int hist_len, int new_len, int pre,
                       int max_shift)
{
    constexpr int PER = 16 / (int)sizeof(U);
    const int n = blockIdx.y;
    const long long sbn = (long long)blockIdx.z * N + n;
    const int v = blockIdx.x * 256 + threadIdx.x;    // 16-byte word of the row
    if (v >= L / PER) return;
    int d = shift ? shift[n] : 0;
    if (d < 0 || d > max_shift) {
        atomicCAS(status, 0, kStatusBadShift);
        d = d < 0 ? 0 : max_shift;
    }
    const int ts = v * PER - pre - d;                // stream time of the first sample, >= -hist_len
    const U *h = hist + sbn * hist_len + hist_len, *w = nw + sbn * new_len;
    __align__(16) U out[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) out[k] = ts + k < 0 ? h[ts + k] : w[ts + k];
    block[sbn * (L / PER) + v] = *reinterpret_cast<const uint4 *>(out);
}

template <typename U>
__global__ void stream_history_kernel(const U *__restrict__ hist, const U *__restrict__ nw, U *__restrict__ out,
                                      long long total, int hist_len, int new_len)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const long long sbn = idx / hist_len;
    const int j = (int)(idx - sbn * hist_len);
    const int ts = new_len - hist_len + j;          // stream time of history entry j
    out[idx] = ts >= 0 ? nw[sbn * new_len + ts] : hist[sbn * hist_len + hist_len + ts];
}

// counts[b(i,j)] = sum_s w_i(s) w_j(s), one warp per baseline (lanes over the
// spectra: 62 stations x 3072 spectra 15 us; one thread per baseline walking
// the spectra took 238 us)
__global__ void __launch_bounds__(256) baseline_counts_kernel(const float *__restrict__ flags,
                                                              float *__restrict__ counts, int N, int S)
{
    const long long B = (long long)N * (N + 1) / 2;
    const long long b = (long long)blockIdx.x * 8 + threadIdx.x / 32;
    const int lane = threadIdx.x % 32;
    if (b >= B) return;
    if (!flags) {
        if (lane == 0) counts[b] = (float)S;
        return;
    }
    int j = (int)((sqrt(8.0 * (double)b + 1.0) - 1.0) * 0.5);
    while ((long long)j * (j + 1) / 2 > b) --j;
    while ((long long)(j + 1) * (j + 2) / 2 <= b) ++j;
    const int i = (int)(b - (long long)j * (j + 1) / 2);
    const float *wi = flags + (long long)i * S, *wj = flags + (long long)j * S;
    float c = 0.f;
#pragma unroll 4
    for (int s = lane; s < S; s += 32) c = fmaf(wi[s], wj[s], c);
#pragma unroll
    for (int m = 16; m > 0; m /= 2) c += __shfl_xor_sync(0xffffffffu, c, m);
    if (lane == 0) counts[b] = c;
}

template <typename U>
cudaError_t assemble_t(const Handle &h, const void *nw, const int *shift, cudaStream_t st)
{
    const int C = h.p.n_channels, T = h.p.n_taps, S = h.p.n_spectra;
    const int L = (S + T - 1) * C;
    const int words = L / (16 / (int)sizeof(U));     // whole words: L is a multiple of 16 samples
    const dim3 grid((unsigned)((words + 255) / 256), (unsigned)h.p.n_stations, (unsigned)h.p.n_subbands);
    if (grid.z > 65535) return cudaErrorInvalidConfiguration;
    stream_assemble_kernel<U><<<grid, 256, 0, st>>>(
        static_cast<const U *>(h.d_hist[h.hist_cur]), static_cast<const U *>(nw), shift, static_cast<uint4 *>(h.d_block),
        h.d_status, h.p.n_stations, L, h.hist_len, S * C, (T - 1) * C, h.p.max_coarse_shift);
    return cudaGetLastError();
}

template <typename U>
cudaError_t history_t(Handle &h, const void *nw, cudaStream_t st)
{
    const int S = h.p.n_spectra, C = h.p.n_channels;
    const long long total = (long long)h.p.n_subbands * h.p.n_stations * h.hist_len;
    const long long blocks = (total + 255) / 256;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    stream_history_kernel<U><<<(unsigned)blocks, 256, 0, st>>>(static_cast<const U *>(h.d_hist[h.hist_cur]),
                                                               static_cast<const U *>(nw),
                                                               static_cast<U *>(h.d_hist[1 - h.hist_cur]), total,
                                                               h.hist_len, S * C);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) h.hist_cur = 1 - h.hist_cur;
    return e;
}

}  // namespace

int raw_sample_bytes(const Handle &h)
{
    return kPols * (h.p.format == FX_CI16 ? 4 : h.p.format == FX_CI8 ? 2 : 1);
}

cudaError_t launch_stream_assemble(const Handle &h, const void *d_new, const int *shift, cudaStream_t st)
{
    switch (raw_sample_bytes(h)) {
    case 8: return assemble_t<uint2>(h, d_new, shift, st);
    case 4: return assemble_t<unsigned>(h, d_new, shift, st);
    default: return assemble_t<unsigned short>(h, d_new, shift, st);
    }
}

cudaError_t launch_stream_history(Handle &h, const void *d_new, cudaStream_t st)
{
    switch (raw_sample_bytes(h)) {
    case 8: return history_t<uint2>(h, d_new, st);
    case 4: return history_t<unsigned>(h, d_new, st);
    default: return history_t<unsigned short>(h, d_new, st);
    }
}

cudaError_t launch_baseline_counts(const Handle &h, const float *flags, float *counts, cudaStream_t st)
{
    const long long B = h.B;
    baseline_counts_kernel<<<(unsigned)((B + 7) / 8), 256, 0, st>>>(flags, counts, h.p.n_stations,
                                                                        h.p.n_spectra);
    return cudaGetLastError();
}

}  // namespace fxi
