// Multibeam coincidence RFI mask (paper Section 2.1): the beams of the
// multibeam receiver act as reference antennas; a sample is interference when
// its total power exceeds k standard deviations in at least min_beams beams
// (the paper's example: 3 sigma in 4 or more of 13), decided independently
// for every sample and written as a boolean mask; masked samples can then be
// replaced, in every beam and channel, by the channel's mean level before
// dedispersion.
//
// Kernels:
//  * dd_zerodm_kernel  -- z_b[t] = sum_c x_b[c][t] for all beams in one
//    launch: 16-byte loads, 2-bit lanes added in nibbles (5 channels) and then
//    byte lanes per 64-channel slice, slices combined in shared memory; sum z and sum z^2 per beam.
//  * dd_rfi_mask_kernel -- per sample, the count of beams with
//    n z - S1 > 0 and (n z - S1)^2 > k^2 (n S2 - S1^2): the test
//    z > mean + k sigma done exactly in integers.
//    The 16-sample words that hold a masked sample join a list.
//  * dd_rfi_apply_kernel -- threads take (listed word, 16 channels, beam) items
//    and rewrite the masked 2-bit lanes with 1 + ((c + t) mod 2).
#include <new>

#include "dd_internal.h"

namespace dd {
namespace {

constexpr int kRfiMaxBeams = 64;

struct BeamPtrs {
    uint8_t *p[kRfiMaxBeams];
};

// A CTA takes 64 kZdGroups samples of one beam (blockIdx.y).  Thread (slice s, group
// g) reads 64 samples (16 bytes) of each of up to 64 channels of its slice.
// Five channels (at most 15) are added in nibbles, even and odd samples apart,
// then widened into byte lanes: acc[4*kw + i] byte j sums sample 16kw + 4j + i
// of the group.  That is 7 integer operations per 16-sample word against 12
// when every word is widened at once (13 beams of 1024 channels x 151536
// samples, 504 MB: 95 us of the 109 us run then, 91 of 102 now); ten loads are in
// flight per thread, and CTAs of 512 samples leave a shorter last wave than 1024
// (104 us).  Bound by how fast DRAM answers: 5.5 TB/s of the copy's 6.8, warps
// wait for loads in 19 of 25 cycles per issue, the ALU pipe is 49 % busy and issue
// slots 29 %; a CTA reads 128 bytes of each row, rows 38 KB apart.  The slices' byte sums meet in shared memory, where thread r
// (group r/16, word kw, lane i) adds its four samples over the slices in
// 16-bit lanes (at most 3 * 21844 < 2^16), then sum z and sum z^2.
constexpr int kZdSlices = 16;  // channel slices per pass (64 channels each)
constexpr int kZdGroups = 8;   // 64-sample groups per CTA

// acc += the 64 samples of each of five channels.
__device__ __forceinline__ void zd_add5(const uint4 *v, uint32_t (&acc)[16]) {
#pragma unroll
    for (int kw = 0; kw < 4; ++kw) {
        uint32_t even = 0, odd = 0;  // nibble k: samples 2k and 2k + 1
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            const uint32_t w = kw == 0 ? v[q].x : kw == 1 ? v[q].y : kw == 2 ? v[q].z : v[q].w;
            even += w & 0x33333333u;
            odd += (w >> 2) & 0x33333333u;
        }
        acc[4 * kw] += even & 0x0F0F0F0Fu;
        acc[4 * kw + 1] += odd & 0x0F0F0F0Fu;
        acc[4 * kw + 2] += (even >> 4) & 0x0F0F0F0Fu;
        acc[4 * kw + 3] += (odd >> 4) & 0x0F0F0F0Fu;
    }
}

__global__ void __launch_bounds__(16 * kZdGroups) dd_zerodm_kernel(const BeamPtrs beams, long long ld_bytes, int nchan,
                                                        long long nsamp, uint32_t *__restrict__ z, long long ldz,
                                                        unsigned long long *__restrict__ stats) {
    __shared__ uint32_t part[kZdSlices][kZdGroups][16];  // [slice][group][4*kw + i]
    const int b = blockIdx.y;
    const uint8_t *in = beams.p[b];
    const int tid = threadIdx.x, g = tid % kZdGroups, sl = tid / kZdGroups;
    const long long t_blk = (long long)blockIdx.x * (64 * kZdGroups);
    const long long byte0 = t_blk / 4 + 16 * g;  // this thread's 16 bytes in every row
    const bool in_row = byte0 < ld_bytes;           // rows cover whole 16-byte groups
    // reducer role: samples t_blk + 64 rg + 16 rkw + 4 j + ri, j = 0..3
    const int rg = tid >> 4, rkw = (tid >> 2) & 3, ri = tid & 3;
    uint32_t lo = 0, hi = 0;  // 16-bit lanes: samples j = 0, 2 (lo) and 1, 3 (hi)
    for (int cs0 = 0; cs0 < nchan; cs0 += 64 * kZdSlices) {
        uint32_t acc[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) acc[q] = 0;
        const int c0 = cs0 + 64 * sl, c1 = min(nchan, c0 + 64);
        if (in_row) {
            const uint8_t *p = in + byte0;
            int c = c0;
            for (; c + 10 <= c1; c += 10) {
                uint4 v[10];
#pragma unroll
                for (int q = 0; q < 10; ++q)
                    v[q] = __ldg(reinterpret_cast<const uint4 *>(p + (long long)(c + q) * ld_bytes));
                zd_add5(v, acc);
                zd_add5(v + 5, acc);
            }
            for (; c < c1; c += 5) {
                uint4 v[5];
#pragma unroll
                for (int q = 0; q < 5; ++q)
                    v[q] = c + q < c1 ? __ldg(reinterpret_cast<const uint4 *>(p + (long long)(c + q) * ld_bytes))
                                      : make_uint4(0, 0, 0, 0);
                zd_add5(v, acc);
            }
        }
#pragma unroll
        for (int q = 0; q < 16; ++q) part[sl][g][q] = acc[q];
        __syncthreads();
#pragma unroll
        for (int s2 = 0; s2 < kZdSlices; ++s2) {
            const uint32_t w = part[s2][rg][4 * rkw + ri];
            lo += w & 0x00FF00FFu;
            hi += (w >> 8) & 0x00FF00FFu;
        }
        __syncthreads();
    }
    const uint32_t v4[4] = {lo & 0xFFFFu, hi & 0xFFFFu, lo >> 16, hi >> 16};
    unsigned long long s1 = 0, s2 = 0;
    uint32_t *zr = z + (long long)b * ldz;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const long long t = t_blk + 64 * rg + 16 * rkw + 4 * j + ri;
        if (t < nsamp) {
            zr[t] = v4[j];
            s1 += v4[j];
            s2 += (unsigned long long)v4[j] * v4[j];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if ((tid & 31) == 0 && (s1 | s2)) {
        atomicAdd(stats + 2 * b, s1);
        atomicAdd(stats + 2 * b + 1, s2);
    }
}

__global__ void __launch_bounds__(256) dd_rfi_mask_kernel(const uint32_t *__restrict__ z, long long ldz, int nbeams,
                                                          long long nsamp, const unsigned long long *__restrict__ stats,
                                                          int k, int min_beams, uint8_t *__restrict__ mask,
                                                          unsigned long long *__restrict__ nmasked,
                                                          unsigned long long *__restrict__ nlist,
                                                          uint2 *__restrict__ list) {
    __shared__ uint32_t s_words[16];  // masked samples of the block's 16-sample words
    __shared__ uint32_t s_zmin[kRfiMaxBeams];  // smallest z of the beam that exceeds
    __shared__ unsigned s_cnt;
    const long long n = nsamp;
    if (threadIdx.x < nbeams) {
        const unsigned long long a = stats[2 * threadIdx.x], q = stats[2 * threadIdx.x + 1];
        // n S2 - S1^2 >= 0 (Cauchy-Schwarz)
        const unsigned __int128 lim = (unsigned __int128)((long long)k * k) *
                                      ((unsigned __int128)n * q - (unsigned __int128)a * a);
        auto exceeds = [&](long long v) {
            const long long dev = n * v - (long long)a;
            return dev > 0 && (unsigned __int128)dev * (unsigned long long)dev > lim;
        };
        // the test is monotone in z: a double estimate of its threshold, then
        // exact steps (one or two); z <= 3 * 21844, so 65533 is never reached
        const double est = ((double)a + sqrt((double)lim)) / (double)n;
        long long v = (long long)fmin(fmax(est, 0.0), 65533.0);
        while (v > 0 && exceeds(v - 1)) --v;
        while (v < 65533 && !exceeds(v)) ++v;
        s_zmin[threadIdx.x] = (uint32_t)v;
    }
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    bool m = false;
    if (t < nsamp) {
        int over = 0;
#pragma unroll 8
        for (int b = 0; b < nbeams; ++b) over += z[(long long)b * ldz + t] >= s_zmin[b];
        m = over >= min_beams;
        mask[t] = (uint8_t)m;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) {
        if (bal) atomicAdd(&s_cnt, (unsigned)__popc(bal));
        s_words[threadIdx.x >> 4] = bal & 0xFFFFu;
        s_words[(threadIdx.x >> 4) + 1] = bal >> 16;
    }
    __syncthreads();
    if (threadIdx.x >= 32 || s_cnt == 0) return;
    if (threadIdx.x == 0) atomicAdd(nmasked, (unsigned long long)s_cnt);
    // words with masked samples join the list in time order within the block:
    // (word, two bits per masked sample)
    const uint32_t bits = threadIdx.x < 16 ? s_words[threadIdx.x] : 0u;
    const unsigned have = __ballot_sync(0xffffffffu, bits != 0);
    unsigned long long pos = 0;
    if (threadIdx.x == 0) pos = atomicAdd(nlist, (unsigned long long)__popc(have));
    pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(have & ((1u << threadIdx.x) - 1u));
    if (bits) {
        uint32_t m2 = (bits | bits << 8) & 0x00FF00FFu;
        m2 = (m2 | m2 << 4) & 0x0F0F0F0Fu;
        m2 = (m2 | m2 << 2) & 0x33333333u;
        m2 = (m2 | m2 << 1) & 0x55555555u;
        list[pos] = make_uint2(blockIdx.x * 16u + threadIdx.x, 3u * m2);
    }
}

// Items (listed word, 16 channels, beam) in that order, so that neighbouring
// threads rewrite neighbouring words of a row, 16 rows in flight per thread.
// A fixed grid: the count is known on the device only, and an empty list
// costs one read.  (One thread per word over all channels took 438 us for 32
// masked words of 13 x 1024 rows; the first run on new data went from 596 to
// 158 us.)
constexpr int kApplyChans = 16;
__global__ void __launch_bounds__(256) dd_rfi_apply_kernel(const BeamPtrs beams, int nbeams, long long ld_bytes,
                                                           int nchan, const unsigned long long *__restrict__ nlist,
                                                           const uint2 *__restrict__ list) {
    const long long nl = (long long)*nlist, ldw = ld_bytes / 4;
    const int nsl = (nchan + kApplyChans - 1) / kApplyChans;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nl * nsl * nbeams;
         i += (long long)gridDim.x * blockDim.x) {
        const long long k = i / nl;
        const uint2 e = list[i - k * nl];
        const int c0 = (int)(k % nsl) * kApplyChans;
        // level 1 + ((c + t) mod 2) at even word starts: 01,10,01,... (even c) or 10,01,... (odd c)
        const uint32_t pat[2] = {0x99999999u & e.y, 0x66666666u & e.y};
        uint32_t *p = reinterpret_cast<uint32_t *>(beams.p[k / nsl]) + (long long)c0 * ldw + e.x;
        uint32_t v[kApplyChans];
#pragma unroll
        for (int c = 0; c < kApplyChans; ++c)
            if (c0 + c < nchan) v[c] = p[c * ldw];
#pragma unroll
        for (int c = 0; c < kApplyChans; ++c)
            if (c0 + c < nchan) p[c * ldw] = (v[c] & ~e.y) | pat[c & 1];
    }
}

struct Rfi {
    int nbeams_max = 0, nchan = 0, sms = 0;
    long long nsamp_max = 0, ldz = 0;
    uint32_t *z = nullptr;                // [nbeams_max][ldz] zero-DM series
    unsigned long long *stats = nullptr;  // [nbeams_max][2]: sum z, sum z^2; then the masked count and the list length
    uint2 *list = nullptr;                // [ceil(nsamp_max/16)] words with masked samples: (word, lanes)
    uint8_t *mask = nullptr;              // [nsamp_max]
    long long nsamp = 0;
    int nbeams = 0;
};

void free_rfi(Rfi *r) {
    if (!r) return;
    cudaFree(r->z);
    cudaFree(r->stats);
    cudaFree(r->mask);
    cudaFree(r->list);
    delete r;
}

}  // namespace
}  // namespace dd

using namespace dd;

extern "C" {

dd_status dd_rfi_create(dd_rfi **out, int nbeams_max, int nchan, size_t nsamp_max) {
    if (!out) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    *out = nullptr;
    if (nbeams_max <= 0 || nbeams_max > kRfiMaxBeams || nchan <= 0 || nchan > 21844 || nsamp_max == 0 ||
        nsamp_max > ((size_t)1 << 31))
        return fail(DD_ERR_INVALID_ARG, "nbeams_max 1..%d, nchan 1..21844, nsamp_max 1..2^31", kRfiMaxBeams);
    Rfi *r = new (std::nothrow) Rfi();
    if (!r) return fail(DD_ERR_NOMEM, "host allocation failed");
    r->nbeams_max = nbeams_max;
    r->nchan = nchan;
    r->nsamp_max = (long long)nsamp_max;
    r->ldz = ((long long)nsamp_max + 15) / 16 * 16;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&r->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMalloc(&r->z, (size_t)nbeams_max * r->ldz * 4);
    if (e == cudaSuccess) e = cudaMalloc(&r->stats, ((size_t)2 * nbeams_max + 2) * 8);
    if (e == cudaSuccess) e = cudaMalloc(&r->mask, (size_t)r->ldz);
    if (e == cudaSuccess) e = cudaMalloc(&r->list, (size_t)(r->ldz / 16) * sizeof(uint2));
    if (e != cudaSuccess) {
        dd_status st = cuda_fail(e, "allocating RFI buffers");
        free_rfi(r);
        return st;
    }
    *out = reinterpret_cast<dd_rfi *>(r);
    return DD_OK;
}

dd_status dd_rfi_run(dd_rfi *rfi, uint8_t *const *d_in, int nbeams, size_t ld_in_bytes, size_t nsamp, int k_sigma,
                     int min_beams, int apply, void *stream) {
    Rfi *r = reinterpret_cast<Rfi *>(rfi);
    if (!r || !d_in) return fail(DD_ERR_INVALID_ARG, "NULL RFI context or beam list");
    if (nbeams <= 0 || nbeams > r->nbeams_max || nsamp == 0 || (long long)nsamp > r->nsamp_max)
        return fail(DD_ERR_INVALID_ARG, "nbeams or nsamp beyond the RFI context's capacity");
    if (ld_in_bytes % 16 != 0 || ld_in_bytes < (nsamp + 3) / 4)
        return fail(DD_ERR_INVALID_ARG, "ld_in_bytes must be a multiple of 16 covering nsamp samples");
    if (k_sigma < 0 || k_sigma > 1000 || min_beams <= 0)
        return fail(DD_ERR_INVALID_ARG, "k_sigma must be 0..1000 and min_beams >= 1");
    BeamPtrs bp{};
    for (int b = 0; b < nbeams; ++b) {
        if (!d_in[b] || ((uintptr_t)d_in[b]) % 16 != 0)
            return fail(DD_ERR_INVALID_ARG, "beam %d input NULL or not 16-byte aligned", b);
        bp.p[b] = d_in[b];
    }
    cudaStream_t st = (cudaStream_t)stream;
    r->nsamp = (long long)nsamp;
    r->nbeams = nbeams;
    DD_CUDA_TRY(cudaMemsetAsync(r->stats, 0, ((size_t)2 * nbeams + 2) * 8, st));
    dd_zerodm_kernel<<<dim3((unsigned)(((long long)nsamp + 64 * kZdGroups - 1) / (64 * kZdGroups)), (unsigned)nbeams),
                       16 * kZdGroups, 0, st>>>(
        bp, (long long)ld_in_bytes, r->nchan, (long long)nsamp, r->z, r->ldz, r->stats);
    dd_rfi_mask_kernel<<<(unsigned)(((long long)nsamp + 255) / 256), 256, 0, st>>>(
        r->z, r->ldz, nbeams, (long long)nsamp, r->stats, k_sigma, min_beams, r->mask, r->stats + 2 * nbeams,
        r->stats + 2 * nbeams + 1, r->list);
    if (apply)
        dd_rfi_apply_kernel<<<4 * r->sms, 256, 0, st>>>(bp, nbeams, (long long)ld_in_bytes, r->nchan,
                                                     r->stats + 2 * nbeams + 1, r->list);
    return cuda_fail(cudaGetLastError(), "RFI kernels");
}

dd_status dd_rfi_result(const dd_rfi *rfi, long long *nmasked, void *stream) {
    const Rfi *r = reinterpret_cast<const Rfi *>(rfi);
    if (!r || !nmasked) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    unsigned long long v = 0;
    DD_CUDA_TRY(cudaMemcpyAsync(&v, r->stats + 2 * r->nbeams, 8, cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    DD_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    *nmasked = (long long)v;
    return DD_OK;
}

dd_status dd_rfi_buffers(const dd_rfi *rfi, const uint32_t **d_zerodm, size_t *ld_zerodm, const uint8_t **d_mask) {
    const Rfi *r = reinterpret_cast<const Rfi *>(rfi);
    if (!r) return fail(DD_ERR_INVALID_ARG, "NULL RFI context");
    if (d_zerodm) *d_zerodm = r->z;
    if (ld_zerodm) *ld_zerodm = (size_t)r->ldz;
    if (d_mask) *d_mask = r->mask;
    return DD_OK;
}

void dd_rfi_destroy(dd_rfi *rfi) { free_rfi(reinterpret_cast<Rfi *>(rfi)); }

}  // extern "C"
