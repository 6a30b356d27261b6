// Input layouts: time-major (SIGPROC-style) 2-bit filterbank data, where each
// time sample's channels follow one another (4 per byte, channel c in bits
// 2(c%4) of byte c/4), turned into the channel-major rows the dedispersion
// kernels read (4 time samples per byte, sample t in bits 2(t%4) of byte
// t/4).  Paper Section 1 describes the 2-bit data; the corner turn only
// moves 2-bit values.
//
// dd_corner_turn_words_kernel: rows and pointers of whole 32-bit words (any
// recorder that pads its samples to words).  A thread takes a 16-channel x
// 16-sample block as 16 words, transposes it in registers, and the CTA's
// blocks meet in shared memory so that every channel row leaves in runs of 64
// bytes or more.
//
// dd_corner_turn_kernel, for any byte stride: a CTA moves a tile of 64
// samples x 64 channels through shared memory.  Thread (group g, quad q) packs the 4 bytes of
// samples 4q..4q+3 for channels 4g..4g+3 into one word, transposes that 4x4
// matrix of 2-bit cells with two masked swaps (cells 6 bits apart inside the
// 2x2 blocks, then blocks 12 bits apart), and so obtains the byte of each of
// the 4 channels holding those 4 samples.
#include "dd_internal.h"

namespace dd {
namespace {

__device__ __forceinline__ uint32_t transpose4x4_2bit(uint32_t w) {
    // cell (s, c) at bit 8s + 2c moves to bit 8c + 2s
    uint32_t t = ((w >> 6) ^ w) & 0x00CC00CCu;
    w ^= t ^ (t << 6);
    t = ((w >> 12) ^ w) & 0x0000F0F0u;
    w ^= t ^ (t << 12);
    return w;
}

__global__ void __launch_bounds__(256) dd_corner_turn_kernel(const uint8_t *__restrict__ tm, long long ld_tm,
                                                             int nchan, long long nsamp, uint8_t *__restrict__ cm,
                                                             long long ld_cm) {
    __shared__ uint8_t in_t[64][17];   // [sample][channel byte], padded
    __shared__ uint8_t out_t[64][17];  // [channel][sample byte], padded
    const long long t0 = (long long)blockIdx.x * 64;
    const int c0 = blockIdx.y * 64;
    const int cb = (nchan + 3) / 4;  // bytes per time sample
    const int tid = threadIdx.x;
    for (int i = tid; i < 64 * 16; i += 256) {
        const int s = i >> 4, b = i & 15;
        const long long t = t0 + s;
        const int byte = c0 / 4 + b;
        in_t[s][b] = (t < nsamp && byte < cb) ? tm[t * ld_tm + byte] : (uint8_t)0;
    }
    __syncthreads();
    {
        const int g = tid & 15, q = tid >> 4;  // channel group (4 channels), sample quad (4 samples)
        const uint32_t w = (uint32_t)in_t[4 * q][g] | ((uint32_t)in_t[4 * q + 1][g] << 8) |
                           ((uint32_t)in_t[4 * q + 2][g] << 16) | ((uint32_t)in_t[4 * q + 3][g] << 24);
        const uint32_t o = transpose4x4_2bit(w);
#pragma unroll
        for (int c = 0; c < 4; ++c) out_t[4 * g + c][q] = (uint8_t)(o >> (8 * c));
    }
    __syncthreads();
    for (int i = tid; i < 64 * 16; i += 256) {
        const int ch = i >> 4, b = i & 15;
        const int c = c0 + ch;
        const long long byte = t0 / 4 + b;
        if (c < nchan && byte < ld_cm) {
            // channels past the band's end were read as zero; samples past nsamp likewise
            cm[(long long)c * ld_cm + byte] = out_t[ch][b];
        }
    }
}

// In-register transpose of a 16 x 16 matrix of 2-bit cells (a[r]: row r, cell
// c in bits 2c): blocks of 8 and 4 cells move by byte permutes, blocks of 2
// and 1 by masked swaps.
__device__ __forceinline__ void transpose16x16_2bit(uint32_t (&a)[16]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t x = a[k], y = a[k + 8];
        a[k] = __byte_perm(x, y, 0x5410);
        a[k + 8] = __byte_perm(x, y, 0x7632);
    }
#pragma unroll
    for (int k = 0; k < 16; ++k)
        if (!(k & 4)) {
            const uint32_t x = a[k], y = a[k + 4];
            a[k] = __byte_perm(x, y, 0x6240);
            a[k + 4] = __byte_perm(x, y, 0x7351);
        }
#pragma unroll
    for (int k = 0; k < 16; ++k)
        if (!(k & 2)) {
            const uint32_t t = ((a[k] >> 4) ^ a[k + 2]) & 0x0F0F0F0Fu;
            a[k + 2] ^= t;
            a[k] ^= t << 4;
        }
#pragma unroll
    for (int k = 0; k < 16; ++k)
        if (!(k & 1)) {
            const uint32_t t = ((a[k] >> 2) ^ a[k + 1]) & 0x33333333u;
            a[k + 1] ^= t;
            a[k] ^= t << 2;
        }
}

// LC lanes of a warp take neighbouring 16-channel words of a sample and 32/LC
// groups of lanes neighbouring 16-sample blocks, so bands narrower than 512
// channels keep every lane busy.
template <int LC>
struct TurnCfg {
    static constexpr int kWarps = 16;
    static constexpr int W = kWarps * 32 / LC;  // 16-sample blocks per CTA
    // words between the k-th channels of neighbouring groups: 16 extra when
    // two rows share a warp's read, so that they fall into different banks
    static constexpr int KS = LC * (W + 1) + (W == 16 ? 16 : 0);
};

// Memory-bound: each byte is read and written once, a sample's row in 4 LC
// byte pieces (128 for bands of 512 channels or more) with 16 loads in flight
// per thread, channel rows in pieces of 4 W bytes.
template <int LC>
__global__ void __launch_bounds__(512) dd_corner_turn_words_kernel(const uint32_t *__restrict__ tm, long long ldw_tm,
                                                                   int nchan, long long nsamp,
                                                                   uint32_t *__restrict__ cm, long long ldw_cm) {
    using C = TurnCfg<LC>;
    __shared__ uint32_t s_t[16 * C::KS];  // [channel in group][group][16-sample block], padded
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l = lane % LC, w = warp * (32 / LC) + lane / LC;
    const int cw = blockIdx.y * LC + l;  // 16-channel word of a sample's row
    const long long wt0 = (long long)blockIdx.x * C::W;
    const long long t = 16 * (wt0 + w);
    uint32_t a[16];
    const bool col = cw < (nchan + 15) / 16;
    const uint32_t *src = tm + t * ldw_tm + cw;
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = col && t + i < nsamp ? __ldcs(src + i * ldw_tm) : 0u;
    transpose16x16_2bit(a);
#pragma unroll
    for (int k = 0; k < 16; ++k) s_t[k * C::KS + l * (C::W + 1) + w] = a[k];
    __syncthreads();
    const int c0 = blockIdx.y * LC * 16;
#pragma unroll 4
    for (int i = threadIdx.x; i < 16 * LC * C::W; i += 512) {
        const int wo = i % C::W, ch = i / C::W;
        const long long o = wt0 + wo;
        if (c0 + ch < nchan && o < ldw_cm)
            __stcs(cm + (long long)(c0 + ch) * ldw_cm + o, s_t[(ch & 15) * C::KS + (ch >> 4) * (C::W + 1) + wo]);
    }
}

template <int LC>
void launch_turn(const uint8_t *tm, size_t ld_tm, int nchan, size_t nsamp, uint8_t *cm, size_t ld_cm,
                 cudaStream_t s) {
    using C = TurnCfg<LC>;
    // whole output rows are written, the padding past nsamp as 0
    const long long words = (long long)(ld_cm / 4);
    const long long nt = (words + C::W - 1) / C::W;
    const dim3 grid((unsigned)nt, (unsigned)(((nchan + 15) / 16 + LC - 1) / LC));
    dd_corner_turn_words_kernel<LC><<<grid, 512, 0, s>>>(reinterpret_cast<const uint32_t *>(tm), (long long)(ld_tm / 4),
                                                         nchan, (long long)nsamp, reinterpret_cast<uint32_t *>(cm),
                                                         words);
}

}  // namespace
}  // namespace dd

using namespace dd;

extern "C" dd_status dd_corner_turn(const uint8_t *d_tm, size_t ld_tm_bytes, int nchan, size_t nsamp, uint8_t *d_cm,
                                    size_t ld_cm_bytes, void *stream) {
    if (!d_tm || !d_cm || nchan <= 0 || nsamp == 0) return fail(DD_ERR_INVALID_ARG, "NULL buffer or empty shape");
    if (ld_tm_bytes < (size_t)(nchan + 3) / 4 || ld_cm_bytes < (nsamp + 3) / 4)
        return fail(DD_ERR_INVALID_ARG, "row strides too short for nchan / nsamp");
    const long long ntile_t = ((long long)nsamp + 63) / 64;
    // output rows are written in whole tiles: cover the padding of the last tile too
    const long long ntile_t_out = ((long long)ld_cm_bytes * 4 + 63) / 64;
    const long long nt = ntile_t > ntile_t_out ? ntile_t : ntile_t_out;
    if (nt > 0x7fffffffLL) return fail(DD_ERR_INVALID_ARG, "gulp too long");
    dim3 grid((unsigned)nt, (unsigned)((nchan + 63) / 64));
    // whole words: the register transpose, with as many lanes across the
    // channels as the band has 16-channel words.  1024 channels x 544752
    // samples (279 MB moved): 231 us with the byte kernel, 49 us (5.7 TB/s)
    // with this one.
    if ((((uintptr_t)d_tm | (uintptr_t)d_cm | ld_tm_bytes | ld_cm_bytes) & 3) == 0 && grid.y <= 65535) {
        const int cw = (nchan + 15) / 16;
        auto launch = cw > 16 ? launch_turn<32> : cw > 8 ? launch_turn<16> : cw > 4 ? launch_turn<8> : launch_turn<4>;
        launch(d_tm, ld_tm_bytes, nchan, nsamp, d_cm, ld_cm_bytes, (cudaStream_t)stream);
        return cuda_fail(cudaGetLastError(), "dd_corner_turn_words_kernel launch");
    }
    dd_corner_turn_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(d_tm, (long long)ld_tm_bytes, nchan,
                                                                  (long long)nsamp, d_cm, (long long)ld_cm_bytes);
    return cuda_fail(cudaGetLastError(), "dd_corner_turn_kernel launch");
}
