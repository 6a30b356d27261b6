// Candidate classifier: a small CNN over 64x64 DM-time snippets with bfloat16
// weights and activations and float accumulation, trained on the GPU by its
// own forward, backward and AdamW kernels.
//
// Network: four 3x3 convolutions (1->16->32->64->64 channels, zero padding,
// ReLU, 2x2 max pooling), fc 1024->128 (ReLU), fc 128->1 (logit); 191553
// parameters in one flat vector (order and flattening as in include/dd.h).
//
// Numerics: every sum starts from the bias and adds products in increasing
// (input channel, ky, kx) / input order, one thread per output, with fmaf --
// a product of two bfloat16 values is exact in float, so each step rounds
// once and the result equals a plain float sum in that order.  Activations
// after ReLU are rounded to bfloat16 (nearest even); pooling keeps the first
// maximum.  Gradients are float; each convolution weight gradient is a two-stage
// sum (a fixed set of samples per block, then the blocks in order), so training is
// deterministic.  These are CUDA-core kernels (~12.5 M multiply-adds per
// snippet): the fixed summation order is what makes the logits reproducible
// bit for bit, which the tensor cores' internal accumulation order is not.
#include <cuda_bf16.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "dd_internal.h"
#include "tmem.cuh"

namespace dd {
namespace {

constexpr int kConvLayers = 4;
constexpr int kCin[kConvLayers] = {1, 16, 32, 64};
constexpr int kCout[kConvLayers] = {16, 32, 64, 64};
constexpr int kHin[kConvLayers] = {64, 32, 16, 8};
constexpr int kFcIn = 1024, kFcHid = 128;
// Blocks (= partials) of a convolution's weight gradient: two per SM of a GB300.
// A fixed number, so that the order of the sums is the same on every device.
constexpr int kMaxPartials = 304;

struct Layout {
    long long cw[kConvLayers], cb[kConvLayers], f1w, f1b, f2w, f2b, total;
};

constexpr Layout make_layout() {
    Layout L{};
    long long o = 0;
    for (int l = 0; l < kConvLayers; ++l) {
        L.cw[l] = o;
        o += (long long)kCout[l] * kCin[l] * 9;
        L.cb[l] = o;
        o += kCout[l];
    }
    L.f1w = o;
    o += (long long)kFcHid * kFcIn;
    L.f1b = o;
    o += kFcHid;
    L.f2w = o;
    o += kFcHid;
    L.f2b = o;
    o += 1;
    L.total = o;
    return L;
}
// fc1's weights (bfloat16) are read, and their gradients (float) written, 16 bytes at a time
static_assert(make_layout().f1w % 8 == 0 && kFcIn % 8 == 0, "16-byte rows of fc1");

__device__ __forceinline__ float bf2f(uint16_t h) { return __uint_as_float((uint32_t)h << 16); }
__device__ __forceinline__ uint16_t f2bf(float f) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(f));
}

// ---- forward -------------------------------------------------------------------

// Forward convolution + ReLU + pooling, register-tiled and persistent.  A
// thread owns 8 output channels x a 2x4 block of convolution outputs (two
// pooled outputs side by side): per input channel it reads a 4x6 input patch
// and 9x8 weights from shared memory and issues 576 FMAs.  One 512-thread
// block per SM keeps the weights of its COB output channels resident
// ([ci][tap][co], float, copied from a float image) and walks groups
// of SPB snippets; each group's inputs arrive in stages of CIC input channels
// by 4-byte cp.async copies into a ring of NBUF buffers, so the copies of
// the next NBUF - 1 stages overlap the FMAs of this one.
//
// Staged layout of a snippet (bfloat16, row stride RS >= H + 2, RS % 4 == 0):
// two leading zeros, then per channel one zero row followed by its H data rows
// (row data at offsets 0..H-1, zeros at H..RS-1), then one closing zero row.
// Padded coordinate (Y, X), 0 <= Y, X <= H + 1, of channel c sits at element
// 2 + (c(H+1) + Y) RS + X - 1: the left halo is the previous row's last zero,
// the right halo this row's first, the top and bottom halos are zero rows.  A
// thread reads a patch row with two 8-byte loads at offsets 4tx-2 and 4tx+2;
// RS is chosen so the half-warps' loads hit distinct banks.  Buffers are
// zeroed once; copies only ever write data elements.
//
// A halo tap adds w*0 to the sum, which leaves it unchanged (only the sign of
// an exact zero can differ, and the ReLU maps both zeros to +0), so every
// output equals the in-order sum from the bias over (ci, ky, kx) with the
// padded taps skipped.
template <int T, int CI, int CO, int H, int COB, int SPB, int CIC, int RS, int NBUF>
struct ConvFwdCfg {
    static constexpr int HO = H / 2;
    static constexpr int PT = (H / 2) * (H / 4);  // 2x4 pixel tiles per snippet
    static constexpr int CTN = COB / 8;           // 8-channel tiles per block
    static constexpr int TILES = PT * CTN * SPB;  // thread tiles per block
    static constexpr int TPT = TILES / T;  // tiles per thread
    static constexpr int NCB = CO / COB;          // output-channel blocks
    static constexpr int NK = CI / CIC;           // stages per snippet group
    static constexpr int CH = (H + 1) * RS;       // staged elements per channel
    static constexpr int SNIP = (2 + (CIC * (H + 1) + 1) * RS + 7) / 8 * 8;  // staged elements per snippet
    static constexpr int BUF = SPB * SNIP;        // elements per stage buffer
    static constexpr int W_FLOATS = CI * 9 * COB;
    static constexpr int CPS = SPB * CIC * H * H / 2;  // 4-byte copies per stage
    static constexpr size_t SMEM = (size_t)W_FLOATS * 4 + (size_t)NBUF * BUF * 2;
    // blocks per SM: 512 threads of 128 registers, 227 KB of shared memory
    static constexpr int BY_SMEM = (int)(227 * 1024 / (SMEM + 1024));
    static constexpr int RESIDENT = BY_SMEM < 512 / T ? BY_SMEM : 512 / T;
    static_assert(COB % 8 == 0 && CO % COB == 0 && H % 4 == 0 && CI % CIC == 0, "tile shape");
    static_assert(NBUF >= 2 && NBUF <= 4, "stage buffers");
    static_assert(TILES % T == 0 && (TPT == 1 || CIC == CI), "whole tiles per thread");
    static_assert(RS % 4 == 0 && RS >= H + 2, "row stride");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

// Float images of the layers' weights in the staged order, refreshed whenever
// the parameters change: dst[cb][ci][tap][co] = w[cb*COB + co][ci][tap] for
// every output-channel block cb, once for the wide and once for the narrow
// blocks' COB (the first layer has no narrow blocks).  A third image (cob 0) is
// the tensor-core kernels' bfloat16 operand: K-major over k = tap * ci + channel,
// 9 taps padded to 16 when ci = 1.
struct WPrepLayer {
    const uint16_t *w;
    float *dst;
    int ci, cob, count;
};
constexpr int kImages = 3;  // wide, narrow, tensor cores
constexpr int kNoImage = -1;
constexpr int kImageCob[kImages][kConvLayers] = {{16, 32, 64, 64}, {kNoImage, 16, 16, 16}, {0, 0, 0, 0}};
constexpr int kNarrowGroups = 512;  // snippet groups of a wide launch up to which the narrow blocks run
struct WPrepArgs {
    WPrepLayer l[kImages * kConvLayers];
};

__global__ void conv_wprep_kernel(const WPrepArgs a) {
    const WPrepLayer L = a.l[blockIdx.y];
    if (L.cob == 0) {
        const int K = L.ci == 1 ? 16 : 9 * L.ci;
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < L.count; i += gridDim.x * blockDim.x) {
            const int co = i / K, k = i % K, tap = k / L.ci, ci = k % L.ci;
            reinterpret_cast<uint16_t *>(L.dst)[tc::kmajor_offset(co, k, K) / 2] =
                tap < 9 ? L.w[(co * L.ci + ci) * 9 + tap] : (uint16_t)0;
        }
        return;
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < L.count; i += gridDim.x * blockDim.x) {
        const int co = i % L.cob, k = (i / L.cob) % 9, ci = (i / (L.cob * 9)) % L.ci, cb = i / (L.cob * 9 * L.ci);
        L.dst[i] = bf2f(L.w[((cb * L.cob + co) * L.ci + ci) * 9 + k]);
    }
}

__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Two float FMAs in one instruction (fma.rn.f32x2): each half is rounded to
// nearest exactly like fmaf, so pairing output channels changes no result;
// it halves the FMA instructions the schedulers issue.
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float lo_f(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi_f(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }

// acc += the taps of nci input channels: channel i's patch row r at
// xb + i*CH + r*RS (the 8-byte words holding padded columns 4tx-1 .. 4tx+4),
// its weights at wb + i*9*COB.  acc[cp][r][q] holds output channels 2cp (low
// half) and 2cp+1 (high half) of output (r, q) of the thread's 2x4 block.
template <int COB, int CH, int RS>
__device__ __forceinline__ void conv_accumulate(uint64_t (&acc)[4][2][4], const uint16_t *xb, const float *wb,
                                                int nci) {
#pragma unroll 1
    for (int ci = 0; ci < nci; ++ci) {
        uint64_t p[4][6];  // each input value in both halves
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const uint2 a = *reinterpret_cast<const uint2 *>(xb + ci * CH + r * RS);
            const uint2 c = *reinterpret_cast<const uint2 *>(xb + ci * CH + r * RS + 4);
            const float v[6] = {__uint_as_float(a.x & 0xffff0000u), __uint_as_float(a.y << 16),
                                __uint_as_float(a.y & 0xffff0000u), __uint_as_float(c.x << 16),
                                __uint_as_float(c.x & 0xffff0000u), __uint_as_float(c.y << 16)};
#pragma unroll
            for (int k = 0; k < 6; ++k) p[r][k] = pk2(v[k], v[k]);
        }
        const float *wk = wb + ci * 9 * COB;
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) {
                const float4 wa = *reinterpret_cast<const float4 *>(wk + (ky * 3 + kx) * COB);
                const float4 wc = *reinterpret_cast<const float4 *>(wk + (ky * 3 + kx) * COB + 4);
                const uint64_t wv[4] = {pk2(wa.x, wa.y), pk2(wa.z, wa.w), pk2(wc.x, wc.y), pk2(wc.z, wc.w)};
#pragma unroll
                for (int cp = 0; cp < 4; ++cp)
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[cp][r][q] = ffma2(wv[cp], p[r + ky][q + kx], acc[cp][r][q]);
            }
    }
}

// ReLU, bfloat16 rounding and 2x2 max pooling (first maximum) of a thread's
// tile.  ARG: also record which of the four is the first maximum (training
// needs it).  Without ARG the window's float maximum is rounded once: ReLU and
// round-to-nearest are both non-decreasing, so the largest rounded value is
// the rounded largest value (a NaN counts as 0 either way), bit for bit.
template <int CO, int HO, bool ARG>
__device__ __forceinline__ void conv_epilogue(const uint64_t (&acc)[4][2][4], int n, int co_first, int ty, int tx,
                                              uint16_t *__restrict__ pooled, uint8_t *__restrict__ arg) {
    if constexpr (!ARG) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            uint32_t packed = 0;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float m = -INFINITY;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint64_t pr = acc[c / 2][q / 2][2 * j + q % 2];
                    m = fmaxf(m, (c & 1) ? hi_f(pr) : lo_f(pr));  // fmaxf drops NaNs
                }
                packed |= (uint32_t)f2bf(m > 0.0f ? m : 0.0f) << (16 * j);  // ReLU: +0 for -0, 0 and NaN
            }
            const long long o = (((long long)n * CO + co_first + c) * HO + ty) * HO + 2 * tx;
            *reinterpret_cast<uint32_t *>(pooled + o) = packed;
        }
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            uint32_t packed = 0;
            uint32_t args = 0;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                // after the ReLU every value is a non-negative bfloat16 (+0 for
                // x <= 0 or NaN), whose bit patterns order like the values
                uint32_t best = 0;
                int a = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint64_t pr = acc[c / 2][q / 2][2 * j + q % 2];
                    const float x = (c & 1) ? hi_f(pr) : lo_f(pr);
                    const uint32_t r = f2bf(x > 0.0f ? x : 0.0f);
                    if (q == 0 || r > best) {
                        best = r;
                        a = q;
                    }
                }
                packed |= best << (16 * j);
                args |= (uint32_t)a << (8 * j);
            }
            const long long o = (((long long)n * CO + co_first + c) * HO + ty) * HO + 2 * tx;
            *reinterpret_cast<uint32_t *>(pooled + o) = packed;
            *reinterpret_cast<uint16_t *>(arg + o) = (uint16_t)args;
        }
    }
}

template <int T, int CI, int CO, int H, int COB, int SPB, int CIC, int RS, int NBUF, bool ARG>
__global__ void __launch_bounds__(T, 512 / T)
    conv_fwd_kernel(const uint16_t *__restrict__ in, const float *__restrict__ wprep, const uint16_t *__restrict__ b,
                    int N, uint16_t *__restrict__ pooled, uint8_t *__restrict__ arg) {
    using C = ConvFwdCfg<T, CI, CO, H, COB, SPB, CIC, RS, NBUF>;
    constexpr int HO = C::HO;
    extern __shared__ __align__(16) unsigned char smem[];
    float *ws = reinterpret_cast<float *>(smem);
    uint16_t *xs = reinterpret_cast<uint16_t *>(smem + (size_t)C::W_FLOATS * 4);
    const int tid = threadIdx.x;
    // the grid is a multiple of NCB: block i serves channel block i % NCB
    const int cb = blockIdx.x % C::NCB, cta = blockIdx.x / C::NCB, ncta = gridDim.x / C::NCB;
    const int ngroups = (N + SPB - 1) / SPB;
    const int nst = cta < ngroups ? (ngroups - cta + ncta - 1) / ncta * C::NK : 0;
    uint4 *z = reinterpret_cast<uint4 *>(xs);
    for (int i = tid; i < NBUF * C::BUF / 8; i += T) z[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    const float *wsrc = wprep + (size_t)cb * C::W_FLOATS;
    for (int i = tid; i < C::W_FLOATS / 4; i += T) cp_async16(ws + 4 * i, wsrc + 4 * i);
    // stage s: group cta + ncta*(s / NK), input channels [k*CIC, (k+1)*CIC), k = s % NK
    auto issue = [&](int s) {
        const int g = cta + ncta * (s / C::NK), c0 = (s % C::NK) * CIC;
        uint16_t *dst = xs + (s % NBUF) * C::BUF;
#pragma unroll 4
        for (int i = tid; i < C::CPS; i += T) {
            const int x2 = i % (H / 2), y = (i / (H / 2)) % H, cl = (i / (H * H / 2)) % CIC, j = i / (CIC * H * H / 2);
            const int n = g * SPB + j;
            if (n < N)
                cp_async4(dst + j * C::SNIP + 2 + (cl * (H + 1) + y + 1) * RS + 2 * x2,
                          in + (((long long)n * CI + c0 + cl) * H + y) * H + 2 * x2);
        }
    };
    // stages 0 .. NBUF-2 in flight (the weights travel with stage 0)
#pragma unroll
    for (int q = 0; q < NBUF - 1; ++q) {
        if (q < nst) issue(q);
        cp_async_commit();
    }
    uint64_t acc[4][2][4];
#pragma unroll 1
    for (int s = 0; s < nst; ++s) {
        // stage s + NBUF - 1 goes to the buffer stage s - 1 used (released by
        // the barrier that ended iteration s - 1)
        if (s + NBUF - 1 < nst) issue(s + NBUF - 1);
        cp_async_commit();
        cp_async_wait<NBUF - 1>();  // every group but the newest NBUF - 1: stage s is in
        __syncthreads();
        const int k = s % C::NK;
#pragma unroll 1
        for (int q = 0; q < C::TPT; ++q) {  // TPT > 1 only with one stage per group
            const int tile = tid + q * T;
            const int pt = tile % C::PT, ct = (tile / C::PT) % C::CTN, sj = tile / (C::PT * C::CTN);
            const int ty = pt / (H / 4), tx = pt % (H / 4);
            const int cof = cb * COB + ct * 8;
            if (k == 0) {
#pragma unroll
                for (int cp = 0; cp < 4; ++cp) {
                    const uint64_t bias = pk2(bf2f(b[cof + 2 * cp]), bf2f(b[cof + 2 * cp + 1]));
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int qq = 0; qq < 4; ++qq) acc[cp][r][qq] = bias;
                }
            }
            conv_accumulate<COB, C::CH, RS>(acc, xs + (s % NBUF) * C::BUF + sj * C::SNIP + 2 * ty * RS + 4 * tx,
                                            ws + k * CIC * 9 * COB + ct * 8, CIC);
            if (k == C::NK - 1) {
                const int n = (cta + ncta * (s / C::NK)) * SPB + sj;
                if (n < N) conv_epilogue<CO, HO, ARG>(acc, n, cof, ty, tx, pooled, arg);
            }
        }
        __syncthreads();
    }
    cp_async_wait<0>();
}

// fc1, persistent (the fixed-order forward's layout, features [n][64][4][4]):
// block b keeps the weights of OUTS outputs resident as bfloat16 in [i/8][o][8]
// order (a lane's 8 consecutive weights are one 16-byte load, neighbouring
// lanes neighbouring outputs) and walks groups of GROUP snippets, whose
// features are staged as float with the next group's loads in flight in
// registers.  A thread owns one output of GROUP * OUTS / 256 snippets; every
// sum runs over the inputs in increasing order.  Bound by the latency of that
// chain and by shared-memory reads.
constexpr int kFc1Pad = 4;  // floats after a snippet's features: two snippets of a warp in different banks
template <int OUTS, int GROUP>
struct Fc1Cfg {
    static constexpr int SNIPS = 256 / OUTS;     // snippets side by side
    static constexpr int K = GROUP / SNIPS;      // snippets per thread
    static constexpr int XS = kFcIn + kFc1Pad;   // floats per staged snippet
    static constexpr int NB = kFcHid / OUTS;     // output blocks
    static constexpr size_t SMEM = (size_t)OUTS * kFcIn * 2 + (size_t)GROUP * XS * 4;
    static constexpr int RESIDENT = SMEM <= 112 * 1024 ? 2 : 1;
    static_assert(GROUP % SNIPS == 0 && GROUP * kFcIn / 8 % 256 == 0, "tile shape");
};

template <int OUTS, int GROUP>
__global__ void __launch_bounds__(256, (Fc1Cfg<OUTS, GROUP>::RESIDENT))
    fc1_persist_kernel(const uint16_t *__restrict__ feat, const uint16_t *__restrict__ w,
                       const uint16_t *__restrict__ b, int N, uint16_t *__restrict__ h1) {
    using C = Fc1Cfg<OUTS, GROUP>;
    extern __shared__ __align__(16) unsigned char smem[];
    uint4 *ws = reinterpret_cast<uint4 *>(smem);                              // [128][OUTS] x 8 bfloat16
    float *xs = reinterpret_cast<float *>(smem + (size_t)OUTS * kFcIn * 2);  // [GROUP][XS]
    const int tid = threadIdx.x;
    const int ob = blockIdx.x % C::NB * OUTS, cta = blockIdx.x / C::NB, ncta = gridDim.x / C::NB;
    const int o = tid % OUTS, sg = tid / OUTS;
    const int ngroups = (N + GROUP - 1) / GROUP;
    // a group's features: GROUP x 128 uint4
    uint4 nxt[GROUP * kFcIn / 8 / 256];
    auto fetch = [&](int g) {
#pragma unroll
        for (int k = 0; k < GROUP * kFcIn / 8 / 256; ++k) {
            const int e = tid + 256 * k, sn = e / (kFcIn / 8), i8 = e % (kFcIn / 8);
            const int n = g * GROUP + sn;
            nxt[k] = n < N ? __ldg(reinterpret_cast<const uint4 *>(feat + (long long)n * kFcIn) + i8)
                           : make_uint4(0, 0, 0, 0);
        }
    };
    if (cta < ngroups) fetch(cta);
    for (int e = tid; e < OUTS * (kFcIn / 8); e += 256)
        ws[e] = __ldg(reinterpret_cast<const uint4 *>(w + (long long)(ob + e % OUTS) * kFcIn) + e / OUTS);
    const float bias = bf2f(b[ob + o]);
#pragma unroll 1
    for (int g = cta; g < ngroups; g += ncta) {
        __syncthreads();  // the previous group's features are consumed
#pragma unroll
        for (int k = 0; k < GROUP * kFcIn / 8 / 256; ++k) {
            const int e = tid + 256 * k, sn = e / (kFcIn / 8), i8 = e % (kFcIn / 8);
            const uint4 q = nxt[k];
            float4 *dst = reinterpret_cast<float4 *>(xs + sn * C::XS + 8 * i8);
            dst[0] = make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u),
                                 __uint_as_float(q.y << 16), __uint_as_float(q.y & 0xffff0000u));
            dst[1] = make_float4(__uint_as_float(q.z << 16), __uint_as_float(q.z & 0xffff0000u),
                                 __uint_as_float(q.w << 16), __uint_as_float(q.w & 0xffff0000u));
        }
        __syncthreads();
        if (g + ncta < ngroups) fetch(g + ncta);
        float acc[C::K];
#pragma unroll
        for (int k = 0; k < C::K; ++k) acc[k] = bias;
#pragma unroll 4
        for (int i8 = 0; i8 < kFcIn / 8; ++i8) {
            const uint4 wq = ws[i8 * OUTS + o];
            const float wf[8] = {__uint_as_float(wq.x << 16), __uint_as_float(wq.x & 0xffff0000u),
                                 __uint_as_float(wq.y << 16), __uint_as_float(wq.y & 0xffff0000u),
                                 __uint_as_float(wq.z << 16), __uint_as_float(wq.z & 0xffff0000u),
                                 __uint_as_float(wq.w << 16), __uint_as_float(wq.w & 0xffff0000u)};
#pragma unroll
            for (int k = 0; k < C::K; ++k) {
                const float4 xa = *reinterpret_cast<const float4 *>(xs + (sg + C::SNIPS * k) * C::XS + 8 * i8);
                const float4 xc = *reinterpret_cast<const float4 *>(xs + (sg + C::SNIPS * k) * C::XS + 8 * i8 + 4);
                acc[k] = fmaf(wf[0], xa.x, acc[k]);
                acc[k] = fmaf(wf[1], xa.y, acc[k]);
                acc[k] = fmaf(wf[2], xa.z, acc[k]);
                acc[k] = fmaf(wf[3], xa.w, acc[k]);
                acc[k] = fmaf(wf[4], xc.x, acc[k]);
                acc[k] = fmaf(wf[5], xc.y, acc[k]);
                acc[k] = fmaf(wf[6], xc.z, acc[k]);
                acc[k] = fmaf(wf[7], xc.w, acc[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < C::K; ++k) {
            const int n = g * GROUP + sg + C::SNIPS * k;
            if (n < N) h1[(long long)n * kFcHid + ob + o] = f2bf(acc[k] > 0.0f ? acc[k] : 0.0f);
        }
    }
}

// fc2 (128 -> 1): a thread one logit, its hidden row in 16-byte loads (all in
// flight before the in-order sum starts).
__global__ void __launch_bounds__(64) fc2_fwd_kernel(const uint16_t *__restrict__ h1, const uint16_t *__restrict__ w,
                                                     const uint16_t *__restrict__ b, int N, float *__restrict__ z) {
    __shared__ float s_w[kFcHid];
    for (int i = threadIdx.x; i < kFcHid; i += 64) s_w[i] = bf2f(w[i]);
    __syncthreads();
    const int n = blockIdx.x * 64 + threadIdx.x;
    if (n >= N) return;
    const uint4 *row = reinterpret_cast<const uint4 *>(h1 + (long long)n * kFcHid);
    uint4 v[kFcHid / 8];
#pragma unroll
    for (int q = 0; q < kFcHid / 8; ++q) v[q] = __ldg(row + q);
    float acc = bf2f(b[0]);
#pragma unroll
    for (int q = 0; q < kFcHid / 8; ++q) {
        const uint32_t u[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc = fmaf(s_w[8 * q + 2 * i], __uint_as_float(u[i] << 16), acc);
            acc = fmaf(s_w[8 * q + 2 * i + 1], __uint_as_float(u[i] & 0xffff0000u), acc);
        }
    }
    z[n] = acc;
}

// ---- inference forward on the tensor cores -----------------------------------
//
// Implicit-GEMM convolution + ReLU + 2x2 max pooling with tcgen05.  A tile is
// M = 128 pooled outputs; its four window positions q are four accumulators of
// N = CO columns in tensor memory, so pooling is a maximum over registers.  K
// = the 9 taps x CI input channels in (tap, channel) order, 16 per MMA.
//
// No im2col: a snippet's input sits in shared memory as 16-byte cells (8
// channels of one pixel), split by the parities of y and x.  For window
// position q and tap (dy, dx) the input pixels of neighbouring pooled outputs
// are neighbouring cells of one parity plane, so 8 of them are a core matrix
// of the K-major operand where they lie, and a tap is only another start
// address.  Zero cells after each row and before each plane are the padding.
// Narrow images interleave snippets (rows of SUBS of them, cells of XS) so
// that the 16 core matrices of a tile are equally spaced (PITCH).
//
// One unit (UNIT snippets) per step: warp 8 issues its MMAs, the other warps
// fetch the next unit's cells (16-byte cp.async from channel-last memory) and
// turn the previous unit's accumulators into outputs meanwhile.  Bound by the
// MMAs' reads of the 4 KB operand tiles (32 cycles each): the im2col form this
// replaces gathered 9 copies of the input and took 932 / 535 / 293 / 200 us
// for the four layers at 8192 snippets, 131, 121, 76 and 63 us now.  Sums are fp32 in the
// tensor cores' own order, so the logits agree with the fixed-order forward to
// float round-off (the training path keeps the fixed-order kernels above).
// Polls of an MMA-completion mbarrier before a thread gives up (a poll that
// finds the phase incomplete suspends the thread for ~4 us on GB300: ~60 ms,
// against microseconds per tile); after a give-up a thread waits no more.
constexpr uint32_t kTcWaitPolls = 1u << 14;
constexpr int kTcThreads = 288;  // 8 warps of loads and outputs, one issuing MMAs

template <int CI, int CO, int H>
struct ConvTcCfg {
    static constexpr int HO = H / 2, K = 9 * CI, G = CI / 8;
    static constexpr int XS = HO >= 8 ? 1 : 8 / HO;         // snippets interleaved within a row's cells
    static constexpr int PITCH = (HO + 1) * XS;             // cells of a row with its zero cell
    static constexpr int UNIT = HO >= 16 ? 1 : 16 / HO * XS;  // snippets per unit
    static constexpr int SUBS = UNIT / XS;                  // rows interleaved
    static constexpr int YS = PITCH * SUBS;                 // cells from pooled row to pooled row
    static constexpr int LEAD = YS + XS;                    // zero cells before a plane
    static constexpr int PS = LEAD + HO * YS;               // cells of a parity plane
    static constexpr int GS = 4 * PS + 1;                   // cells of a channel group (odd: 8 groups, 8 banks)
    static constexpr int CELLS = G * GS + LEAD;
    static constexpr int TILES = HO * HO * UNIT / 128;
    static constexpr int NBUF = CI == 64 ? 1 : 2;           // input buffers that fit beside the weights
    static constexpr int DCOLS = TILES * 4 * CO;            // accumulator columns of a unit
    static constexpr int B_BYTES = CO * K * 2;
    static constexpr bool FEATURES = HO == 4;               // last layer: [n][co][4][4] for fc1
    static constexpr int OUT_PITCH = CO * HO * HO * 2 + 16; // bytes of a staged snippet of features
    static constexpr int OUT_BYTES = FEATURES ? UNIT * OUT_PITCH : 0;
    static constexpr size_t SMEM = (size_t)NBUF * CELLS * 16 + B_BYTES + OUT_BYTES;
    static constexpr int UNIT_CELLS = UNIT * H * H * G;     // 16-byte copies per unit
    static_assert(SMEM <= 227 * 1024 && 2 * DCOLS == 512, "shared and tensor memory");
    static_assert(TILES * 128 == HO * HO * UNIT && UNIT_CELLS % 256 == 0, "whole tiles");
};

template <int CI, int CO, int H>
__global__ void __launch_bounds__(kTcThreads, 1)
    conv_tc_kernel(const uint16_t *__restrict__ in, const uint16_t *__restrict__ wk, const uint16_t *__restrict__ b,
                   int N, uint16_t *__restrict__ out, unsigned *__restrict__ err) {
    using C = ConvTcCfg<CI, CO, H>;
    constexpr int HO = C::HO;
    extern __shared__ __align__(1024) uint8_t tsm[];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_mbar[2];
    __shared__ float s_bias[CO];
    uint8_t *As = tsm;
    uint8_t *Bs = tsm + (size_t)C::NBUF * C::CELLS * 16;
    uint8_t *Os = Bs + C::B_BYTES;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nunits = (N + C::UNIT - 1) / C::UNIT;
    const int nu = (int)blockIdx.x < nunits ? (nunits - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

    // zero cells once (copies only ever write data cells), weights in MMA order
    for (int i = tid; i < C::NBUF * C::CELLS; i += kTcThreads) reinterpret_cast<uint4 *>(As)[i] = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < C::B_BYTES / 16; i += kTcThreads)
        cp_async16(Bs + 16 * i, reinterpret_cast<const uint4 *>(wk) + i);
    if (tid < CO) s_bias[tid] = bf2f(b[tid]);
    if (warp == 0) tc::tmem_alloc(&s_tmem, 2 * C::DCOLS);
    if (tid == 0) {
        tc::mbar_init(&s_mbar[0], 1);
        tc::mbar_init(&s_mbar[1], 1);
    }
    __syncthreads();
    auto load = [&](int u) {  // unit u of this CTA -> its buffer
        const int s0 = ((int)blockIdx.x + u * (int)gridDim.x) * C::UNIT;
        uint8_t *dst = As + (size_t)(u % C::NBUF) * C::CELLS * 16;
        const uint4 *src = reinterpret_cast<const uint4 *>(in) + (long long)s0 * H * H * C::G;
#pragma unroll 4
        for (int k = 0; k < C::UNIT_CELLS / 256; ++k) {
            const int e = tid + 256 * k;
            const int g = e % C::G, x = (e / C::G) % H, y = (e / (C::G * H)) % H, s = e / (C::G * H * H);
            const int cell = g * C::GS + ((y & 1) * 2 + (x & 1)) * C::PS + C::LEAD + (y >> 1) * C::YS +
                             s / C::XS * C::PITCH + (x >> 1) * C::XS + s % C::XS;
            if (s0 + s < N) cp_async16(dst + 16 * cell, src + e);
        }
    };
    if (warp < 8 && nu > 0) load(0);
    cp_async_wait_all();
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = s_tmem;
    bool ok = true;
    auto wait = [&](int u) {
        if (ok) ok = tc::mbar_wait(&s_mbar[u & 1], (uint32_t)(u >> 1) & 1u, kTcWaitPolls);
    };
    auto issue = [&](int u) {
        const uint64_t a0 = tc::smem_desc(tc::smem_addr(As) + (uint32_t)(u % C::NBUF) * (C::CELLS * 16), C::GS * 16,
                                          C::PITCH * 16);
        const uint64_t b0 = tc::smem_desc(tc::smem_addr(Bs), 128, C::K / 8 * 128);
#pragma unroll
        for (int t = 0; t < C::TILES; ++t)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t d = tmem + (uint32_t)((u & 1) * C::DCOLS + (t * 4 + q) * CO);
#pragma unroll
                for (int tap = 0; tap < 9; ++tap) {
                    const int uy = (q >> 1) + tap / 3 - 1, ux = (q & 1) + tap % 3 - 1;  // -1 .. 2
                    const int yp = uy & 1, xp = ux & 1;
                    const int cell = (yp * 2 + xp) * C::PS + C::LEAD + (uy - yp) / 2 * C::YS + (ux - xp) / 2 * C::XS +
                                     t * 8 * C::XS;
#pragma unroll
                    for (int st = 0; st < CI / 16; ++st)
                        tc::mma_bf16(d, a0 + (uint64_t)(cell + 2 * st * C::GS), b0 + (uint64_t)(16 * (tap * (CI / 16) + st)),
                                     tc::idesc_bf16(128, CO), tap > 0 || st > 0);
                }
            }
        tc::mma_commit(&s_mbar[u & 1]);
    };
    // maximum over the window (bias, ReLU and rounding never decrease, so they
    // follow it), bias, ReLU and rounding of unit u's accumulators: warp w
    // takes rows 32 (w % 4) .. +31 and, with w / 4, one tile or half the channels
    auto epilogue = [&](int u) {
        tc::fence_after_sync();
        const int quad = warp & 3, half = warp >> 2;
        const int m = 32 * quad + lane, grp = m >> 3, e = m & 7;
        const int py = grp / C::SUBS, px = (C::TILES == 2 ? half * 8 : 0) + e / C::XS;
        const int sn = grp % C::SUBS * C::XS + e % C::XS;
        const int n = ((int)blockIdx.x + u * (int)gridDim.x) * C::UNIT + sn;
        const int cb = C::TILES == 2 ? 0 : half * (CO / 2);
        const uint32_t t0 = tmem + (uint32_t)((u & 1) * C::DCOLS + (C::TILES == 2 ? half * 4 * CO : 0) + cb) +
                            ((uint32_t)(32 * quad) << 16);
        static_assert((C::TILES == 2 ? CO : CO / 2) == 32, "32 channels per thread");
#pragma unroll
        for (int c0 = 0; c0 < 32; c0 += 16) {
            float v[4][16];
            tc::tmem_ld4x16(t0 + c0, CO, v);
            uint32_t pk[8];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float a = fmaxf(fmaxf(v[0][i], v[1][i]), fmaxf(v[2][i], v[3][i])) + s_bias[cb + c0 + i];
                const uint32_t r = f2bf(a > 0.0f ? a : 0.0f);
                pk[i / 2] = i % 2 ? pk[i / 2] | r << 16 : r;
            }
            if constexpr (C::FEATURES) {
                uint16_t *o = reinterpret_cast<uint16_t *>(Os + sn * C::OUT_PITCH) + (cb + c0) * HO * HO + py * HO + px;
#pragma unroll
                for (int i = 0; i < 16; ++i) o[i * HO * HO] = (uint16_t)(pk[i / 2] >> (i % 2 * 16));
            } else if (n < N) {
                uint4 *o = reinterpret_cast<uint4 *>(out + (((long long)n * HO + py) * HO + px) * CO + cb + c0);
                o[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                o[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            }
        }
        if constexpr (C::FEATURES) {
            constexpr int Q = CO * HO * HO / 8;  // 16-byte pieces of a snippet
            const int s0 = ((int)blockIdx.x + u * (int)gridDim.x) * C::UNIT;
            asm volatile("bar.sync 1, 256;\n" ::: "memory");
            for (int i = tid; i < C::UNIT * Q; i += 256)
                if (s0 + i / Q < N)
                    reinterpret_cast<uint4 *>(out)[(long long)s0 * Q + i] =
                        *reinterpret_cast<const uint4 *>(Os + i / Q * C::OUT_PITCH + i % Q * 16);
        }
    };
#pragma unroll 1
    for (int u = 0; u < nu; ++u) {
        if (warp == 8) {
            if (lane == 0) issue(u);
            __syncwarp();
        } else if constexpr (C::NBUF == 2) {
            if (u > 0) wait(u - 1);  // frees the other input buffer
            if (u + 1 < nu) load(u + 1);
            if (u > 0) epilogue(u - 1);
        } else {
            if (u > 0) epilogue(u - 1);
            wait(u);
            if (u + 1 < nu) load(u + 1);
        }
        cp_async_wait_all();
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
    }
    if (nu > 0) {
        if (C::NBUF == 2 || warp == 8) wait(nu - 1);
        if (warp < 8) epilogue(nu - 1);
    }
    tc::fence_before_sync();
    if (__syncthreads_or(!ok)) {
        // some completion was not observed: give the last two commits one
        // more short bounded wait before the tensor memory is freed
        for (int k = 1; k <= 2 && nu - k >= 0; ++k)
            tc::mbar_wait(&s_mbar[(nu - k) & 1], (uint32_t)((nu - k) >> 1) & 1u, kTcWaitPolls / 64 + 1);
        tc::fence_before_sync();
        __syncthreads();
    }
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, 2 * C::DCOLS);
    if (!ok && lane == 0) atomicOr(err, 1u);
}

// The first layer (one input channel, 64x64): K = 9 taps padded to 16, built
// per row.  A unit is 4 pooled rows of a snippet = 128 pooled outputs; thread
// (p, qy) builds the rows of output p at window positions (qy, 0) and (qy, 1)
// from 3 x 4 input pixels by byte permutes (three neighbouring words per image
// row, fetched one unit ahead) and stores them as one 16-byte group of 8 taps
// and the ninth tap; the other seven of the second group stay zero.  Bound by
// issue and shared-memory stores; three CTAs per SM hide each other's
// barriers.
struct Conv0Tc {
    static constexpr int A_BYTES = 4 * 128 * 32;  // four window positions
    static constexpr int B_BYTES = 16 * 16 * 2;
    static constexpr int DCOLS = 4 * 16;
};

__global__ void __launch_bounds__(256, 3) conv0_tc_kernel(const uint16_t *__restrict__ in,
                                                          const uint16_t *__restrict__ wk,
                                                          const uint16_t *__restrict__ b, int N,
                                                          uint16_t *__restrict__ out, unsigned *__restrict__ err) {
    using C = Conv0Tc;
    __shared__ __align__(128) uint8_t As[2][C::A_BYTES];
    __shared__ __align__(128) uint8_t Bs[C::B_BYTES];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_mbar[2];
    __shared__ float s_bias[16];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nunits = N * 8;
    const int nu = (int)blockIdx.x < nunits ? (nunits - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    for (int i = tid; i < 2 * C::A_BYTES / 16; i += 256) reinterpret_cast<uint4 *>(As)[i] = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < C::B_BYTES / 16; i += 256)
        reinterpret_cast<uint4 *>(Bs)[i] = __ldg(reinterpret_cast<const uint4 *>(wk) + i);
    if (tid < 16) s_bias[tid] = bf2f(b[tid]);
    if (warp == 0) tc::tmem_alloc(&s_tmem, 2 * C::DCOLS);
    if (tid == 0) {
        tc::mbar_init(&s_mbar[0], 1);
        tc::mbar_init(&s_mbar[1], 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = s_tmem;
    bool ok = true;
    const int p = tid & 127, qy = tid >> 7, px = p & 31;
    uint32_t w[3][3];  // image rows y-1 .. y+1, pixel pairs px-1 .. px+1
    auto fetch = [&](int u) {
        const int unit = (int)blockIdx.x + u * (int)gridDim.x;
        const uint32_t *img = reinterpret_cast<const uint32_t *>(in) + (long long)(unit >> 3) * (64 * 32);
        const int y = 2 * (4 * (unit & 7) + (p >> 5)) + qy;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int yy = y + r - 1;
            const bool row = yy >= 0 && yy < 64;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int xx = px + c - 1;
                w[r][c] = row && xx >= 0 && xx < 32 ? __ldg(img + yy * 32 + xx) : 0u;
            }
        }
    };
    auto build = [&](int u) {
        uint8_t *A = As[u & 1];
        // taps of column x-1, x, x+1: hi of pair 0, lo and hi of pair 1 (x even); both of pair 1, lo of pair 2 (x odd)
        uint8_t *d0 = A + (2 * qy) * 4096 + tc::kmajor_offset(p, 0, 16), *d1 = d0 + 4096;
        *reinterpret_cast<uint4 *>(d0) =
            make_uint4(__byte_perm(w[0][0], w[0][1], 0x5432), __byte_perm(w[0][1], w[1][0], 0x7632), w[1][1],
                       __byte_perm(w[2][0], w[2][1], 0x5432));
        *reinterpret_cast<uint32_t *>(d0 + 128) = w[2][1] >> 16;
        *reinterpret_cast<uint4 *>(d1) = make_uint4(w[0][1], __byte_perm(w[0][2], w[1][1], 0x5410),
                                                    __byte_perm(w[1][1], w[1][2], 0x5432), w[2][1]);
        *reinterpret_cast<uint32_t *>(d1 + 128) = w[2][2] & 0xFFFFu;
    };
    auto epilogue = [&](int u) {
        if (ok) ok = tc::mbar_wait(&s_mbar[u & 1], (uint32_t)(u >> 1) & 1u, kTcWaitPolls);
        tc::fence_after_sync();
        const int quad = warp & 3, cb = (warp >> 2) * 8;
        const int unit = (int)blockIdx.x + u * (int)gridDim.x;
        float v[4][8];
        tc::tmem_ld4x8(tmem + (uint32_t)((u & 1) * C::DCOLS + cb) + ((uint32_t)(32 * quad) << 16), 16, v);
        uint32_t pk[4];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float a = fmaxf(fmaxf(v[0][i], v[1][i]), fmaxf(v[2][i], v[3][i])) + s_bias[cb + i];
            const uint32_t r = f2bf(a > 0.0f ? a : 0.0f);
            pk[i / 2] = i % 2 ? pk[i / 2] | r << 16 : r;
        }
        *reinterpret_cast<uint4 *>(out + ((long long)unit * 128 + 32 * quad + lane) * 16 + cb) =
            make_uint4(pk[0], pk[1], pk[2], pk[3]);
    };
    if (nu > 0) fetch(0);
#pragma unroll 1
    for (int u = 0; u < nu; ++u) {
        build(u);  // its buffer's last MMAs were waited for by the epilogue of unit u - 2
        if (u + 1 < nu) fetch(u + 1);
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (tid == 0) {
            const uint64_t a0 = tc::smem_desc(tc::smem_addr(As[u & 1]), 128, 256);
            const uint64_t b0 = tc::smem_desc(tc::smem_addr(Bs), 128, 256);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                tc::mma_bf16(tmem + (uint32_t)((u & 1) * C::DCOLS + 16 * q), a0 + (uint64_t)(256 * q), b0,
                             tc::idesc_bf16(128, 16), false);
            tc::mma_commit(&s_mbar[u & 1]);
        }
        __syncwarp();
        if (u > 0) epilogue(u - 1);
    }
    if (nu > 0) epilogue(nu - 1);
    tc::fence_before_sync();
    if (__syncthreads_or(!ok)) {
        for (int k = 1; k <= 2 && nu - k >= 0; ++k)
            tc::mbar_wait(&s_mbar[(nu - k) & 1], (uint32_t)((nu - k) >> 1) & 1u, kTcWaitPolls / 64 + 1);
        tc::fence_before_sync();
        __syncthreads();
    }
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, 2 * C::DCOLS);
    if (!ok && lane == 0) atomicOr(err, 1u);
}

// ---- backward ------------------------------------------------------------------

__global__ void __launch_bounds__(1024) bce_kernel(const float *__restrict__ z, const float *__restrict__ y, int N,
                                                   float *__restrict__ dz, float *__restrict__ loss) {
    __shared__ double s[32];
    double acc = 0.0;
    for (int n = threadIdx.x; n < N; n += blockDim.x) {
        const float zn = z[n];
        const float sg = 1.0f / (1.0f + expf(-zn));
        dz[n] = (sg - y[n]) / (float)N;
        const double zd = zn, yd = y[n];
        acc += (zd > 0 ? zd : 0) - zd * yd + log1p(exp(-fabs(zd)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = threadIdx.x < blockDim.x / 32 ? s[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) *loss = (float)(acc / N);
    }
}

// fc2: block 0 sums the weight and bias gradients of fc2 and the bias
// gradient of fc1 over the batch (8 interleaved slices, joined in order); the
// other blocks write dh = dz * w2 where the hidden unit was active.
__global__ void __launch_bounds__(1024) fc2_bwd_kernel(const float *__restrict__ dz, const uint16_t *__restrict__ h1,
                                                       const uint16_t *__restrict__ w2, int N,
                                                       float *__restrict__ g_w2, float *__restrict__ g_b2,
                                                       float *__restrict__ g_b1, float *__restrict__ dh) {
    const int i = threadIdx.x % kFcHid, sl = threadIdx.x / kFcHid;
    const float w = bf2f(w2[i]);
    if (blockIdx.x > 0) {
        for (long long n = (long long)(blockIdx.x - 1) * 8 + sl; n < N; n += (long long)(gridDim.x - 1) * 8)
            dh[n * kFcHid + i] = bf2f(h1[n * kFcHid + i]) > 0.0f ? dz[n] * w : 0.0f;
        return;
    }
    __shared__ float s_w[8][kFcHid], s_b[8][kFcHid], s_z[8];
    float aw = 0.0f, ab = 0.0f, az = 0.0f;
#pragma unroll 8
    for (int n = sl; n < N; n += 8) {
        const float h = bf2f(h1[(long long)n * kFcHid + i]), z = dz[n];
        aw += z * h;
        ab += h > 0.0f ? z * w : 0.0f;
        az += z;
    }
    s_w[sl][i] = aw;
    s_b[sl][i] = ab;
    if (i == 0) s_z[sl] = az;
    __syncthreads();
    if (sl == 0) {
        for (int k = 1; k < 8; ++k) {
            aw += s_w[k][i];
            ab += s_b[k][i];
            az += s_z[k];
        }
        g_w2[i] = aw;
        g_b1[i] = ab;
        if (i == 0) *g_b2 = az;
    }
}

// fc1 weight gradient: a block owns 16 outputs x 64 inputs, a thread one
// output x 4 inputs, the batch staged 32 samples at a time.
__global__ void __launch_bounds__(256) fc1_bwd_w_kernel(const float *__restrict__ dh,
                                                        const uint16_t *__restrict__ feat, int N,
                                                        float *__restrict__ g_w1) {
    __shared__ __align__(16) float s_f[32][64];
    __shared__ float s_d[32][16];
    const int tid = threadIdx.x, i0 = blockIdx.x * 64, o0 = blockIdx.y * 16;
    const int iq = (tid & 15) * 4, o = tid >> 4;
    // this thread's share of a stage: 8 inputs of one sample, 2 values of dh
    const int fn = tid >> 3, fi = (tid & 7) * 8;
    uint4 fv;
    float d0, d1;
    auto fetch = [&](int n0) {
        const int n = n0 + fn, na = n0 + (tid >> 4), nb = na + 16;
        fv = n < N ? __ldg(reinterpret_cast<const uint4 *>(feat + (long long)n * kFcIn + i0 + fi))
                   : make_uint4(0, 0, 0, 0);
        d0 = na < N ? __ldg(dh + (long long)na * kFcHid + o0 + (tid & 15)) : 0.0f;
        d1 = nb < N ? __ldg(dh + (long long)nb * kFcHid + o0 + (tid & 15)) : 0.0f;
    };
    fetch(0);
    float acc[4] = {};
    for (int n0 = 0; n0 < N; n0 += 32) {
        __syncthreads();
        float4 *f4 = reinterpret_cast<float4 *>(&s_f[fn][fi]);
        f4[0] = make_float4(__uint_as_float(fv.x << 16), __uint_as_float(fv.x & 0xffff0000u),
                            __uint_as_float(fv.y << 16), __uint_as_float(fv.y & 0xffff0000u));
        f4[1] = make_float4(__uint_as_float(fv.z << 16), __uint_as_float(fv.z & 0xffff0000u),
                            __uint_as_float(fv.w << 16), __uint_as_float(fv.w & 0xffff0000u));
        s_d[tid >> 4][tid & 15] = d0;
        s_d[(tid >> 4) + 16][tid & 15] = d1;
        __syncthreads();
        if (n0 + 32 < N) fetch(n0 + 32);
#pragma unroll
        for (int n = 0; n < 32; ++n) {
            const float4 f = *reinterpret_cast<const float4 *>(&s_f[n][iq]);
            const float d = s_d[n][o];
            acc[0] = fmaf(d, f.x, acc[0]);
            acc[1] = fmaf(d, f.y, acc[1]);
            acc[2] = fmaf(d, f.z, acc[2]);
            acc[3] = fmaf(d, f.w, acc[3]);
        }
    }
    *reinterpret_cast<float4 *>(g_w1 + (long long)(o0 + o) * kFcIn + i0 + iq) =
        make_float4(acc[0], acc[1], acc[2], acc[3]);
}

// fc1 input gradient: a block owns 16 samples x 64 inputs.
__global__ void __launch_bounds__(256) fc1_bwd_x_kernel(const float *__restrict__ dh, const uint16_t *__restrict__ w1,
                                                        int N, float *__restrict__ dfeat) {
    __shared__ __align__(16) float s_w[kFcHid][64];
    __shared__ float s_d[16][kFcHid];
    const int tid = threadIdx.x, i0 = blockIdx.y * 64, n0 = blockIdx.x * 16;
#pragma unroll
    for (int k = 0; k < kFcHid * 8 / 256; ++k) {
        const int e = tid + 256 * k, o = e >> 3, i8 = (e & 7) * 8;
        const uint4 q = __ldg(reinterpret_cast<const uint4 *>(w1 + (long long)o * kFcIn + i0 + i8));
        float4 *f4 = reinterpret_cast<float4 *>(&s_w[o][i8]);
        f4[0] = make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u),
                            __uint_as_float(q.y << 16), __uint_as_float(q.y & 0xffff0000u));
        f4[1] = make_float4(__uint_as_float(q.z << 16), __uint_as_float(q.z & 0xffff0000u),
                            __uint_as_float(q.w << 16), __uint_as_float(q.w & 0xffff0000u));
    }
#pragma unroll
    for (int k = 0; k < 16 * kFcHid / 256; ++k) {
        const int e = tid + 256 * k, n = n0 + e / kFcHid;
        s_d[e / kFcHid][e % kFcHid] = n < N ? __ldg(dh + (long long)n * kFcHid + e % kFcHid) : 0.0f;
    }
    __syncthreads();
    const int iq = (tid & 15) * 4, r = tid >> 4;
    float acc[4] = {};
#pragma unroll 16
    for (int o = 0; o < kFcHid; ++o) {
        const float4 f = *reinterpret_cast<const float4 *>(&s_w[o][iq]);
        const float d = s_d[r][o];
        acc[0] = fmaf(d, f.x, acc[0]);
        acc[1] = fmaf(d, f.y, acc[1]);
        acc[2] = fmaf(d, f.z, acc[2]);
        acc[3] = fmaf(d, f.w, acc[3]);
    }
    if (n0 + r < N)
        *reinterpret_cast<float4 *>(dfeat + (long long)(n0 + r) * kFcIn + i0 + iq) =
            make_float4(acc[0], acc[1], acc[2], acc[3]);
}

// Gradient of a convolution's pooled output routed to the one position of
// each 2x2 window that pooling kept (0 elsewhere, and 0 where the ReLU cut: a
// dead window).
__device__ __forceinline__ bool live(uint16_t pooled) { return bf2f(pooled) > 0.0f; }
__device__ __forceinline__ float live_grad(float d, uint16_t pooled) { return live(pooled) ? d : 0.0f; }

// Input gradient of a 3x3 convolution: din[n][ci] = sum over (co, taps) of the
// routed output gradient times the flipped weights, a convolution over CO
// channels whose input is expanded to float as it is staged.  FMA-bound like
// the forward kernel and tiled like it: a thread owns 8 input channels x a 2x4
// block of pixels (288 packed FMAs per output channel from a 4x6 patch and 9x8
// weights), a block 16 input channels of SPB samples, so that the 18-37 KB of
// weights and two stages of 8 output channels leave room for several blocks
// per SM.  The next stage's gradients wait in registers.  Sums run over co,
// then the taps.  The one-thread-per-pixel form this replaces read every
// gradient 9 CI times: 4290 us for the three layers at 256 snippets, 153 us
// with this one (3 G multiply-adds: half the packed-FMA rate; 256 blocks leave
// a third of the SMs with one block instead of two).
template <int CI, int CO, int H>
struct ConvBwdXCfg {
    static constexpr int CIB = 16;                    // input channels per block
    static constexpr int COC = 8;                     // output channels per stage
    static constexpr int PT = (H / 2) * (H / 4);      // 2x4 pixel tiles per sample
    static constexpr int THREADS = PT * 2 >= 128 ? PT * 2 : 128;
    static constexpr int SPB = THREADS / (PT * 2);    // samples per block
    // row stride: zeros at H..RS-1 are the right halo and the next row's left
    // one; 24 for H = 16 puts a quarter-warp's two rows into different banks
    static constexpr int RS = H == 16 ? 24 : H + 4;
    static constexpr int CH = (H + 1) * RS;
    static constexpr int SNIP = 4 + (COC * (H + 1) + 1) * RS;  // staged floats per sample
    static constexpr int BUF = SPB * SNIP;
    static constexpr size_t SMEM = (size_t)(CO * 9 * CIB + 2 * BUF) * 4;
    static constexpr int QUADS = SPB * COC * (H / 2) * (H / 8);  // 4-window groups per stage
    static constexpr int QPT = QUADS / THREADS;
    static_assert(QUADS % THREADS == 0 && CO % COC == 0 && CI % CIB == 0 && RS % 4 == 0, "tile shape");
};

template <int CI, int CO, int H>
__global__ void __launch_bounds__((ConvBwdXCfg<CI, CO, H>::THREADS))
    conv_bwd_x_kernel(const float *__restrict__ dpool, const uint16_t *__restrict__ pooled,
                      const uint8_t *__restrict__ arg, const uint16_t *__restrict__ w, int N,
                      float *__restrict__ din) {
    using C = ConvBwdXCfg<CI, CO, H>;
    constexpr int HO = H / 2, CIB = C::CIB, T = C::THREADS;
    extern __shared__ __align__(16) unsigned char smem[];
    float *ws = reinterpret_cast<float *>(smem);  // [co][flipped tap][ci]
    float *gs = ws + CO * 9 * CIB;
    const int tid = threadIdx.x;
    const int ci0 = blockIdx.y * CIB, n0 = blockIdx.x * C::SPB;
    for (int i = tid; i < 2 * C::BUF / 4; i += T) reinterpret_cast<float4 *>(gs)[i] = make_float4(0, 0, 0, 0);
    for (int e = tid; e < CO * CIB * 9; e += T) {
        const int k = e % 9, c = (e / 9) % CIB, co = e / (9 * CIB);
        ws[(co * 9 + 8 - k) * CIB + c] = bf2f(__ldg(w + ((long long)co * CI + ci0 + c) * 9 + k));
    }
    // a stage's 4-window groups: sample j, channel cl, window row yo, windows 4 xq .. 4 xq + 3
    float4 d4[C::QPT];
    uint2 p4[C::QPT];
    uint32_t a4[C::QPT];
    auto fetch = [&](int s) {
#pragma unroll
        for (int k = 0; k < C::QPT; ++k) {
            const int e = tid + k * T;
            const int xq = e % (HO / 4), yo = (e / (HO / 4)) % HO, cl = (e / (HO / 4 * HO)) % C::COC;
            const int n = n0 + e / (HO / 4 * HO * C::COC);
            const long long o = (((long long)n * CO + s * C::COC + cl) * HO + yo) * HO + 4 * xq;
            const bool ok = n < N;
            d4[k] = ok ? __ldg(reinterpret_cast<const float4 *>(dpool + o)) : make_float4(0, 0, 0, 0);
            p4[k] = ok ? __ldg(reinterpret_cast<const uint2 *>(pooled + o)) : make_uint2(0, 0);
            a4[k] = ok ? __ldg(reinterpret_cast<const uint32_t *>(arg + o)) : 0u;
        }
    };
    auto expand = [&](int s) {
#pragma unroll
        for (int k = 0; k < C::QPT; ++k) {
            const int e = tid + k * T;
            const int xq = e % (HO / 4), yo = (e / (HO / 4)) % HO, cl = (e / (HO / 4 * HO)) % C::COC;
            const int j = e / (HO / 4 * HO * C::COC);
            const float g[4] = {live_grad(d4[k].x, (uint16_t)p4[k].x), live_grad(d4[k].y, (uint16_t)(p4[k].x >> 16)),
                                live_grad(d4[k].z, (uint16_t)p4[k].y), live_grad(d4[k].w, (uint16_t)(p4[k].y >> 16))};
            float *dst = gs + (s & 1) * C::BUF + j * C::SNIP + 4 + (cl * (H + 1) + 2 * yo + 1) * C::RS + 8 * xq;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t a = (a4[k] >> (8 * i)) & 0xFFu;
                    v[2 * i] = a == 2 * r ? g[i] : 0.0f;
                    v[2 * i + 1] = a == 2 * r + 1 ? g[i] : 0.0f;
                }
                float4 *d = reinterpret_cast<float4 *>(dst + r * C::RS);
                d[0] = make_float4(v[0], v[1], v[2], v[3]);
                d[1] = make_float4(v[4], v[5], v[6], v[7]);
            }
        }
    };
    const int pt = tid % C::PT, ct = (tid / C::PT) % 2, sj = tid / (2 * C::PT);
    const int ty = pt / (H / 4), tx = pt % (H / 4);
    uint64_t acc[4][2][4];
#pragma unroll
    for (int cp = 0; cp < 4; ++cp)
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[cp][r][q] = 0ull;
    fetch(0);
    __syncthreads();
    expand(0);
    __syncthreads();
    constexpr int NS = CO / C::COC;
#pragma unroll 1
    for (int s = 0; s < NS; ++s) {
        if (s + 1 < NS) fetch(s + 1);
        // padded row Y = 0..H+1 of a channel starts at 4 + (cl(H+1) + Y) RS; patch column 4tx - 1
        const float *xb = gs + (s & 1) * C::BUF + sj * C::SNIP + 4 + 2 * ty * C::RS + 4 * tx;
        const float *wb = ws + s * C::COC * 9 * CIB + ct * 8;
#pragma unroll 1
        for (int cl = 0; cl < C::COC; ++cl) {
            uint64_t p[4][6];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float *row = xb + cl * C::CH + r * C::RS;
                const float l = row[-1], h = row[4];
                const float4 m = *reinterpret_cast<const float4 *>(row);
                const float v[6] = {l, m.x, m.y, m.z, m.w, h};
#pragma unroll
                for (int k = 0; k < 6; ++k) p[r][k] = pk2(v[k], v[k]);
            }
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const float4 wa = *reinterpret_cast<const float4 *>(wb + (cl * 9 + t) * CIB);
                const float4 wc = *reinterpret_cast<const float4 *>(wb + (cl * 9 + t) * CIB + 4);
                const uint64_t wv[4] = {pk2(wa.x, wa.y), pk2(wa.z, wa.w), pk2(wc.x, wc.y), pk2(wc.z, wc.w)};
#pragma unroll
                for (int cp = 0; cp < 4; ++cp)
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            acc[cp][r][q] = ffma2(wv[cp], p[r + t / 3][q + t % 3], acc[cp][r][q]);
            }
        }
        if (s + 1 < NS) expand(s + 1);  // the other buffer: its readers passed the previous barrier
        __syncthreads();
    }
    const int n = n0 + sj;
    if (n >= N) return;
#pragma unroll
    for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = (c & 1) ? hi_f(acc[c / 2][r][q]) : lo_f(acc[c / 2][r][q]);
            *reinterpret_cast<float4 *>(din + (((long long)n * CI + ci0 + ct * 8 + c) * H + 2 * ty + r) * H + 4 * tx) =
                make_float4(v[0], v[1], v[2], v[3]);
        }
}

// Weight gradient of a 3x3 convolution: only one position per 2x2 window
// carries a gradient, so a thread (one output channel, 4 input channels, all 9
// taps: 36 sums) walks the windows of a sample, each a gradient, the position
// that pooling kept and the 3x3 input patch around it: a quarter of the dense
// multiply-adds.  A sample's input sits in shared memory channel-last with a
// zero border (a lane's 4 channels are one 8-byte load, the lanes of one
// output channel consecutive), its (gradient, patch offset) pairs beside it.  In
// a sample with an infinite input (after a ReLU there is no NaN) the patch of a
// dead window is one of zeros past the bottom border, since its gradient of 0
// times infinity would be NaN.  (The 16 -> 32 layer at 256 snippets: 41 us
// without, 42.5 so, 46 with every sample's dead windows there, by bank
// conflicts.)
// A block walks samples blockIdx.x, + gridDim.x, ...; its sums (SL window
// slices joined in order) are one partial, and conv_bwd_w_sum_kernel adds the
// partials in order, so the result is deterministic.  Issue-bound: about 64
// instructions per 36 multiply-adds of a window.  (One thread per weight
// reading the gradients from memory: 4470 us for the four layers at 256
// snippets, 144 us with these and their sums.)
template <int CI, int CO, int H, int COB, int SL>
struct ConvBwdWCfg {
    static constexpr int HO = H / 2, NWIN = HO * HO;
    static constexpr int CQ = CI / 4;                // lanes of one output channel
    static constexpr int THREADS = SL * COB * CQ;
    static constexpr int GS = NWIN + 1;              // padded row of (gradient, offset) pairs
    static constexpr int PIX = CI * 2;               // bytes of a pixel
    static constexpr int ZERO_PATCH = (H + 1) * (H + 2) * PIX;  // rows H+1 (the border) .. H+3, 3 pixels each
    static constexpr int IN_BYTES = (((H + 3) * (H + 2) + 3) * PIX + 15) / 16 * 16;
    static constexpr int RED_BYTES = SL > 1 ? (SL - 1) * COB * CQ * 37 * 4 : 0;  // slices' sums, in the pairs' place
    static constexpr int GP_BYTES = COB * GS * 8;
    static constexpr size_t SMEM = (size_t)IN_BYTES + (GP_BYTES > RED_BYTES ? GP_BYTES : RED_BYTES);
    static constexpr int NW = CO * CI * 9 + CO;
    static_assert(CI % 4 == 0 && CO % COB == 0 && NWIN % SL == 0 && THREADS % 32 == 0, "tile shape");
};

template <int CI, int CO, int H, int COB, int SL>
__global__ void __launch_bounds__((ConvBwdWCfg<CI, CO, H, COB, SL>::THREADS), 2)
    conv_bwd_w_kernel(const float *__restrict__ dpool, const uint16_t *__restrict__ pooled,
                      const uint8_t *__restrict__ arg, const uint16_t *__restrict__ in, int N,
                      float *__restrict__ partial) {
    using C = ConvBwdWCfg<CI, CO, H, COB, SL>;
    constexpr int HO = C::HO, T = C::THREADS;
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char *xin = smem;
    uint2 *gp = reinterpret_cast<uint2 *>(smem + C::IN_BYTES);
    const int tid = threadIdx.x, co0 = blockIdx.y * COB;
    const int cq = tid % C::CQ, co = (tid / C::CQ) % COB, sl = tid / (C::CQ * COB);
    for (int i = tid; i < C::IN_BYTES / 8; i += T) reinterpret_cast<uint2 *>(xin)[i] = make_uint2(0, 0);
    uint64_t acc[9][2];  // taps x two channel pairs
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[t][0] = acc[t][1] = 0ull;
    float bacc = 0.0f;
#pragma unroll 1
    for (int n = blockIdx.x; n < N; n += gridDim.x) {
        __syncthreads();  // zeros written; the previous sample consumed
        uint32_t top = 0;  // largest inputs of even and odd pixels (after the ReLU: none negative)
        // input, channel-last: two neighbouring pixels of 4 channels at a time
#pragma unroll 4
        for (int e = tid; e < C::CQ * H * (H / 2); e += T) {
            const int x2 = e % (H / 2), y = (e / (H / 2)) % H, q = e / (H / 2 * H);
            uint32_t v[4];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                v[c] = __ldg(reinterpret_cast<const uint32_t *>(in + (((long long)n * CI + 4 * q + c) * H + y) * H +
                                                                 2 * x2));
#pragma unroll
            for (int c = 0; c < 4; ++c) top = __vmaxu2(top, v[c]);
            unsigned char *dst = xin + ((y + 1) * (H + 2) + 2 * x2 + 1) * C::PIX + 8 * q;
            *reinterpret_cast<uint2 *>(dst) = make_uint2(__byte_perm(v[0], v[1], 0x5410), __byte_perm(v[2], v[3], 0x5410));
            *reinterpret_cast<uint2 *>(dst + C::PIX) =
                make_uint2(__byte_perm(v[0], v[1], 0x7632), __byte_perm(v[2], v[3], 0x7632));
        }
#pragma unroll 4
        for (int e = tid; e < COB * C::NWIN; e += T) {
            const int k = e % C::NWIN, c = e / C::NWIN;
            const long long o = ((long long)n * CO + co0 + c) * C::NWIN + k;
            const int a = __ldg(arg + o);
            // patch around (2 yo + a/2, 2 xo + a%2): its corner in padded coordinates is that position
            const int off = ((2 * (k / HO) + (a >> 1)) * (H + 2) + 2 * (k % HO) + (a & 1)) * C::PIX;
            gp[c * C::GS + k] = make_uint2(__float_as_uint(live_grad(__ldg(dpool + o), __ldg(pooled + o))), (uint32_t)off);
        }
        if (__syncthreads_or((top & 0xFFFFu) >= 0x7F80u || top >= 0x7F800000u)) {
            for (int e = tid; e < COB * C::NWIN; e += T)
                if (!live(__ldg(pooled + ((long long)n * CO + co0) * C::NWIN + e)))
                    gp[e / C::NWIN * C::GS + e % C::NWIN].y = C::ZERO_PATCH;
            __syncthreads();
        }
        const uint2 *g = gp + co * C::GS + sl * (C::NWIN / SL);
        const unsigned char *xb = xin + 8 * cq;
#pragma unroll 2
        for (int k = 0; k < C::NWIN / SL; ++k) {
            const uint2 e = g[k];
            const float gv = __uint_as_float(e.x);
            const uint64_t g2 = pk2(gv, gv);
            bacc += gv;
            const unsigned char *px = xb + e.y;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const uint2 v = *reinterpret_cast<const uint2 *>(px + ((t / 3) * (H + 2) + t % 3) * C::PIX);
                acc[t][0] = ffma2(g2, pk2(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u)), acc[t][0]);
                acc[t][1] = ffma2(g2, pk2(__uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u)), acc[t][1]);
            }
        }
    }
    float a[37];
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            a[(2 * p) * 9 + t] = lo_f(acc[t][p]);
            a[(2 * p + 1) * 9 + t] = hi_f(acc[t][p]);
        }
    a[36] = bacc;
    if constexpr (SL > 1) {
        float *red = reinterpret_cast<float *>(smem + C::IN_BYTES);
        constexpr int M = COB * C::CQ;  // threads of a slice
        __syncthreads();
        if (sl > 0)
#pragma unroll
            for (int i = 0; i < 37; ++i) red[((sl - 1) * 37 + i) * M + tid % M] = a[i];
        __syncthreads();
        if (sl > 0) return;
        for (int s = 0; s < SL - 1; ++s)
#pragma unroll
            for (int i = 0; i < 37; ++i) a[i] += red[(s * 37 + i) * M + tid];
    }
    // sum i = 9 (channel of the 4) + tap of thread (co, cq): [36][CO][CQ], then the
    // biases, so that neighbouring threads write neighbouring floats (in weight
    // order a store touched 32 sectors and the 64x64 layer took 61 us at 256 snippets, 18 us
    // this way)
    float *dst = partial + (long long)blockIdx.x * C::NW;
#pragma unroll
    for (int i = 0; i < 36; ++i) dst[(i * CO + co0 + co) * C::CQ + cq] = a[i];
    if (cq == 0) dst[CO * CI * 9 + co0 + co] = a[36];
}

// The first layer (one input channel): warp w owns output channel w, its lanes
// the windows of a row, 9 sums each; the sample's image sits in shared memory
// as float with a zero border, past it the zeros that dead windows read (always:
// 22 us at 256 snippets, 25 with their own patches).
__global__ void __launch_bounds__(512) conv0_bwd_w_kernel(const float *__restrict__ dpool,
                                                          const uint16_t *__restrict__ pooled,
                                                          const uint8_t *__restrict__ arg,
                                                          const uint16_t *__restrict__ in, int N,
                                                          float *__restrict__ partial) {
    constexpr int H = 64, HO = 32, CO = 16, RS = H + 2;
    __shared__ float img[(RS + 1) * RS + 3];  // rows H+1 (the border) .. H+3 of zeros, 3 pixels in the last
    const int tid = threadIdx.x, co = tid >> 5, lane = tid & 31;
    for (int i = tid; i < (RS + 1) * RS + 3; i += 512) img[i] = 0.0f;
    float acc[10] = {};  // 9 taps and the bias
#pragma unroll 1
    for (int n = blockIdx.x; n < N; n += gridDim.x) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < H * H / 2 / 512; ++k) {
            const int e = tid + 512 * k, y = e / (H / 2), x2 = e % (H / 2);
            const uint32_t v = __ldg(reinterpret_cast<const uint32_t *>(in + ((long long)n * H + y) * H) + x2);
            float *dst = img + (y + 1) * RS + 2 * x2 + 1;
            dst[0] = __uint_as_float(v << 16);
            dst[1] = __uint_as_float(v & 0xffff0000u);
        }
        __syncthreads();
        const long long o = ((long long)n * CO + co) * HO * HO + lane;
#pragma unroll 4
        for (int yo = 0; yo < HO; ++yo) {
            const int a = __ldg(arg + o + yo * HO);
            const bool on = live(__ldg(pooled + o + yo * HO));
            const float d = __ldg(dpool + o + yo * HO), g = on ? d : 0.0f;
            const float *px = img + (on ? (2 * yo + (a >> 1)) * RS + 2 * lane + (a & 1) : (H + 1) * RS);
#pragma unroll
            for (int t = 0; t < 9; ++t) acc[t] = fmaf(g, px[(t / 3) * RS + t % 3], acc[t]);
            acc[9] += g;
        }
    }
    float *dst = partial + (long long)blockIdx.x * (CO * 9 + CO);
#pragma unroll
    for (int t = 0; t < 10; ++t) {
        float v = acc[t];
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
        if (lane == 0) dst[t < 9 ? co * 9 + t : CO * 9 + co] = v;
    }
}

// Sum the blocks' partials into the weight and bias gradients: 32 weights per
// block, 8 interleaved slices of the partials joined in order.  cocq > 0: the
// weights come as [36][co][cq] (conv_bwd_w_kernel), cocq = CO * CI / 4;
// 0: in weight order.
__global__ void __launch_bounds__(256) conv_bwd_w_sum_kernel(const float *__restrict__ partial, int nparts,
                                                             int nw_weights, int nbias, int cocq,
                                                             float *__restrict__ g_w, float *__restrict__ g_b) {
    __shared__ float s[8][32];
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
    const int wi = blockIdx.x * 32 + lane, nw = nw_weights + nbias;
    float acc = 0.0f;
    if (wi < nw)
#pragma unroll 8
        for (int c = sl; c < nparts; c += 8) acc += __ldg(partial + (long long)c * nw + wi);
    s[sl][lane] = acc;
    __syncthreads();
    if (sl > 0 || wi >= nw) return;
#pragma unroll
    for (int k = 1; k < 8; ++k) acc += s[k][lane];
    if (wi >= nw_weights) g_b[wi - nw_weights] = acc;
    else g_w[cocq > 0 ? wi % cocq * 36 + wi / cocq : wi] = acc;
}

// ---- optimiser -------------------------------------------------------------------

__global__ void adamw_kernel(long long count, float *__restrict__ master, const float *__restrict__ g,
                             float *__restrict__ m, float *__restrict__ v, uint16_t *__restrict__ bf, float lr,
                             float beta1, float beta2, float eps, float wd, float c1, float c2) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    // written without fused multiply-adds so every step rounds like the plain formula
    const float gi = g[i];
    const float mi = __fadd_rn(__fmul_rn(beta1, m[i]), __fmul_rn(__fsub_rn(1.0f, beta1), gi));
    const float vi = __fadd_rn(__fmul_rn(beta2, v[i]), __fmul_rn(__fmul_rn(__fsub_rn(1.0f, beta2), gi), gi));
    m[i] = mi;
    v[i] = vi;
    const float mh = __fdiv_rn(mi, c1), vh = __fdiv_rn(vi, c2);
    const float upd = __fadd_rn(__fdiv_rn(mh, __fadd_rn(__fsqrt_rn(vh), eps)), __fmul_rn(wd, master[i]));
    const float w = __fsub_rn(master[i], __fmul_rn(lr, upd));
    master[i] = w;
    bf[i] = f2bf(w);
}

__global__ void to_bf16_kernel(long long count, const float *__restrict__ master, uint16_t *__restrict__ bf) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) bf[i] = f2bf(master[i]);
}

}  // namespace

struct NN {
    Layout L;
    int max_batch = 0;
    int step = 0;
    float *master = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    uint16_t *bf = nullptr;
    uint16_t *pooled[kConvLayers] = {};
    uint8_t *arg[kConvLayers] = {};
    uint16_t *h1 = nullptr;
    float *z = nullptr, *dz = nullptr, *dh = nullptr, *loss = nullptr, *partial = nullptr;
    float *dpool[kConvLayers] = {};  // gradient w.r.t. each layer's pooled output
    unsigned *tc_err = nullptr;      // tensor-core forward: an MMA completion was not observed
    float *wprep = nullptr;          // float images of the convolution weights in staged order
    int wprep_off[kImages][kConvLayers] = {};
    int nsm = 0;
};

static void free_nn(NN *p) {
    if (!p) return;
    cudaFree(p->master);
    cudaFree(p->grad);
    cudaFree(p->m);
    cudaFree(p->v);
    cudaFree(p->bf);
    for (int l = 0; l < kConvLayers; ++l) {
        cudaFree(p->pooled[l]);
        cudaFree(p->arg[l]);
        cudaFree(p->dpool[l]);
    }
    cudaFree(p->h1);
    cudaFree(p->z);
    cudaFree(p->dz);
    cudaFree(p->dh);
    cudaFree(p->loss);
    cudaFree(p->partial);
    cudaFree(p->tc_err);
    cudaFree(p->wprep);
    delete p;
}

// Refresh the convolutions' float weight images from the bfloat16 parameters.
static void refresh_images(NN *p, cudaStream_t s) {
    WPrepArgs a;
    int most = 0, images = 0;
    for (int i = 0; i < kImages; ++i)
        for (int l = 0; l < kConvLayers; ++l) {
            if (kImageCob[i][l] == kNoImage) continue;
            const int count = (kImageCob[i][l] == 0 && kCin[l] == 1 ? 16 : 9 * kCin[l]) * kCout[l];
            a.l[images++] = {p->bf + p->L.cw[l], p->wprep + p->wprep_off[i][l], kCin[l], kImageCob[i][l], count};
            most = std::max(most, count);
        }
    conv_wprep_kernel<<<dim3((unsigned)((most + 255) / 256), (unsigned)images), 256, 0, s>>>(a);
}

// One convolution layer in the fixed order with the tile parameters given.
template <int T, int CI, int CO, int H, int COB, int SPB, int CIC, int RS, int NBUF>
static dd_status launch_conv_fwd(NN *p, int l, const uint16_t *in, int n, bool with_arg, cudaStream_t s) {
    using C = ConvFwdCfg<T, CI, CO, H, COB, SPB, CIC, RS, NBUF>;
    auto kern = with_arg ? conv_fwd_kernel<T, CI, CO, H, COB, SPB, CIC, RS, NBUF, true>
                         : conv_fwd_kernel<T, CI, CO, H, COB, SPB, CIC, RS, NBUF, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "classifier forward");
    const int groups = (n + SPB - 1) / SPB;
    const int grid = std::max(1, std::min(p->nsm * C::RESIDENT / C::NCB, groups));
    constexpr int image = CI > 1 && COB == 16 ? 1 : 0;  // narrow or wide order
    kern<<<grid * C::NCB, T, C::SMEM, s>>>(in, p->wprep + p->wprep_off[image][l], p->bf + p->L.cb[l], n, p->pooled[l],
                                           p->arg[l]);
    return DD_OK;
}

template <int OUTS, int GROUP>
static dd_status launch_fc1(NN *p, int n, cudaStream_t s) {
    using C = Fc1Cfg<OUTS, GROUP>;
    auto kern = fc1_persist_kernel<OUTS, GROUP>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "classifier forward");
    const int grid = std::max(1, std::min(p->nsm * C::RESIDENT / C::NB, (n + GROUP - 1) / GROUP));
    kern<<<grid * C::NB, 256, C::SMEM, s>>>(p->pooled[3], p->bf + p->L.f1w, p->bf + p->L.f1b, n, p->h1);
    return DD_OK;
}

// The fully connected layers, from the features in pooled[3] to the logits in z.
static dd_status nn_fc(NN *p, int n, cudaStream_t s) {
    // fc1: 16 outputs per block while all blocks of 16 snippets fit one wave of
    // two per SM (12 us against 20 us with 64 outputs at 256 snippets; 74
    // against 56 us at 4096)
    const dd_status st =
        (n + 15) / 16 * (kFcHid / 16) <= 2 * p->nsm ? launch_fc1<16, 16>(p, n, s) : launch_fc1<64, 16>(p, n, s);
    if (st != DD_OK) return st;
    fc2_fwd_kernel<<<(n + 63) / 64, 64, 0, s>>>(p->h1, p->bf + p->L.f2w, p->bf + p->L.f2b, n, p->z);
    return DD_OK;
}

// with_arg: record the pooling argmax of every layer (the backward pass needs it).
static dd_status nn_forward(NN *p, const uint16_t *x, int n, cudaStream_t s, bool with_arg) {
    if (((uintptr_t)x) % 4 != 0) return fail(DD_ERR_INVALID_ARG, "snippets must be 4-byte aligned");
    // Narrow blocks (16 output channels, 128 or 256 threads) when the wide ones
    // (all or 32 output channels, 512 threads) would give an SM no more than
    // about three groups of snippets: with so few, whole SMs idle in the last
    // wave or altogether, where four times as many narrow blocks fill them.
    // Narrow / wide, whole forward: 96 / 207 us at 16 snippets, 170 / 235 at
    // 256, 279 / 332 at 512; past the line the narrow blocks' repeated staging
    // of the inputs costs 1-5 % (3513 / 3355 us at 8192).
    const bool nar1 = n <= kNarrowGroups, nar2 = (n + 1) / 2 <= kNarrowGroups, nar3 = (n + 7) / 8 <= kNarrowGroups;
    // (threads, CI, CO, H, output channels and snippets per block, input
    // channels per stage, row stride, stages)
    dd_status st = launch_conv_fwd<512, 1, 16, 64, 16, 1, 1, 68, 4>(p, 0, x, n, with_arg, s);
    if (st == DD_OK)
        st = nar1 ? launch_conv_fwd<256, 16, 32, 32, 16, 1, 8, 48, 3>(p, 1, p->pooled[0], n, with_arg, s)
                  : launch_conv_fwd<512, 16, 32, 32, 32, 1, 16, 48, 3>(p, 1, p->pooled[0], n, with_arg, s);
    if (st == DD_OK)
        st = nar2 ? launch_conv_fwd<128, 32, 64, 16, 16, 2, 8, 24, 3>(p, 2, p->pooled[1], n, with_arg, s)
                  : launch_conv_fwd<512, 32, 64, 16, 64, 2, 16, 24, 3>(p, 2, p->pooled[1], n, with_arg, s);
    if (st == DD_OK)
        st = nar3 ? launch_conv_fwd<128, 64, 64, 8, 16, 8, 4, 12, 3>(p, 3, p->pooled[2], n, with_arg, s)
                  : launch_conv_fwd<512, 64, 64, 8, 64, 8, 8, 12, 3>(p, 3, p->pooled[2], n, with_arg, s);
    if (st == DD_OK) st = nn_fc(p, n, s);
    if (st != DD_OK) return st;
    return cuda_fail(cudaGetLastError(), "classifier forward");
}

// Inference forward: tensor-core convolutions with channel-last activations
// (stored in the pooled buffers; the last layer writes fc1's order), then the
// fully connected layers.
static dd_status nn_forward_tc(NN *p, const uint16_t *x, int n, cudaStream_t s) {
    const Layout &L = p->L;
    auto wk = [&](int l) { return reinterpret_cast<const uint16_t *>(p->wprep + p->wprep_off[2][l]); };
    conv0_tc_kernel<<<std::min(3 * p->nsm, 8 * n), 256, 0, s>>>(x, wk(0), p->bf + L.cb[0], n, p->pooled[0], p->tc_err);
#define DD_CONV_TC(l, CI, CO, H)                                                                              \
    {                                                                                                         \
        using C = ConvTcCfg<CI, CO, H>;                                                                       \
        auto kern = conv_tc_kernel<CI, CO, H>;                                                                \
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM); \
        if (e != cudaSuccess) return cuda_fail(e, "classifier forward");                                      \
        const int grid = std::min(p->nsm, (n + C::UNIT - 1) / C::UNIT);                                       \
        kern<<<grid, kTcThreads, C::SMEM, s>>>(p->pooled[(l) - 1], wk(l), p->bf + L.cb[l], n, p->pooled[l],   \
                                               p->tc_err);                                                    \
    }
    DD_CONV_TC(1, 16, 32, 32)
    DD_CONV_TC(2, 32, 64, 16)
    DD_CONV_TC(3, 64, 64, 8)
#undef DD_CONV_TC
    dd_status st = nn_fc(p, n, s);
    if (st != DD_OK) return st;
    return cuda_fail(cudaGetLastError(), "classifier forward");
}

}  // namespace dd

using namespace dd;

extern "C" {

dd_status dd_nn_create(dd_nn **out, int max_batch) {
    if (!out || max_batch <= 0 || max_batch > (1 << 16)) return fail(DD_ERR_INVALID_ARG, "max_batch must be 1..65536");
    *out = nullptr;
    NN *p = new (std::nothrow) NN();
    if (!p) return fail(DD_ERR_NOMEM, "host allocation failed");
    p->L = make_layout();
    p->max_batch = max_batch;
    const size_t P = (size_t)p->L.total;
    const size_t nb = (size_t)max_batch;
    cudaError_t e = cudaMalloc(&p->master, P * 4);
    if (e == cudaSuccess) e = cudaMalloc(&p->grad, P * 4);
    if (e == cudaSuccess) e = cudaMalloc(&p->m, P * 4);
    if (e == cudaSuccess) e = cudaMalloc(&p->v, P * 4);
    if (e == cudaSuccess) e = cudaMalloc(&p->bf, P * 2);
    for (int l = 0; l < kConvLayers && e == cudaSuccess; ++l) {
        const size_t cells = nb * kCout[l] * (kHin[l] / 2) * (kHin[l] / 2);
        e = cudaMalloc(&p->pooled[l], cells * 2);
        if (e == cudaSuccess) e = cudaMalloc(&p->arg[l], cells);
        if (e == cudaSuccess) e = cudaMalloc(&p->dpool[l], cells * 4);
    }
    if (e == cudaSuccess) e = cudaMalloc(&p->h1, nb * kFcHid * 2);
    if (e == cudaSuccess) e = cudaMalloc(&p->z, nb * 4);
    if (e == cudaSuccess) e = cudaMalloc(&p->dz, nb * 4);
    if (e == cudaSuccess) e = cudaMalloc(&p->dh, nb * kFcHid * 4);
    if (e == cudaSuccess) e = cudaMalloc(&p->loss, 4);
    size_t part = 0;
    for (int l = 0; l < kConvLayers; ++l) {
        const size_t nw = (size_t)kCout[l] * kCin[l] * 9 + kCout[l];
        part = std::max(part, nw * std::min<size_t>(nb, kMaxPartials));
    }
    if (e == cudaSuccess) e = cudaMalloc(&p->partial, part * 4);
    if (e == cudaSuccess) e = cudaMalloc(&p->tc_err, 4);
    int wtot = 0;
    for (int i = 0; i < kImages; ++i)
        for (int l = 0; l < kConvLayers; ++l) {
            p->wprep_off[i][l] = wtot;
            if (kImageCob[i][l] != kNoImage) wtot += std::max(kCin[l] * 9, 16) * kCout[l];
        }
    if (e == cudaSuccess) e = cudaMalloc(&p->wprep, (size_t)wtot * 4);
    if (e == cudaSuccess) e = cudaMemset(p->wprep, 0, (size_t)wtot * 4);
    if (e == cudaSuccess) e = cudaMemset(p->tc_err, 0, 4);
    if (e == cudaSuccess) {
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&p->nsm, cudaDevAttrMultiProcessorCount, dev);
    }
    if (e == cudaSuccess) e = cudaMemset(p->master, 0, P * 4);
    if (e == cudaSuccess) e = cudaMemset(p->m, 0, P * 4);
    if (e == cudaSuccess) e = cudaMemset(p->v, 0, P * 4);
    if (e == cudaSuccess) e = cudaMemset(p->bf, 0, P * 2);
    if (e == cudaSuccess) e = cudaMemset(p->grad, 0, P * 4);
    if (e != cudaSuccess) {
        dd_status st = cuda_fail(e, "allocating classifier buffers");
        free_nn(p);
        return st;
    }
    *out = reinterpret_cast<dd_nn *>(p);
    return DD_OK;
}

dd_status dd_nn_set_params(dd_nn *nn, const float *h_master) {
    NN *p = reinterpret_cast<NN *>(nn);
    if (!p || !h_master) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    const size_t P = (size_t)p->L.total;
    DD_CUDA_TRY(cudaMemcpy(p->master, h_master, P * 4, cudaMemcpyHostToDevice));
    DD_CUDA_TRY(cudaMemset(p->m, 0, P * 4));
    DD_CUDA_TRY(cudaMemset(p->v, 0, P * 4));
    to_bf16_kernel<<<(unsigned)((P + 255) / 256), 256>>>((long long)P, p->master, p->bf);
    refresh_images(p, nullptr);
    DD_CUDA_TRY(cudaGetLastError());
    DD_CUDA_TRY(cudaDeviceSynchronize());
    p->step = 0;
    return DD_OK;
}

dd_status dd_nn_get_params(const dd_nn *nn, float *h_master) {
    const NN *p = reinterpret_cast<const NN *>(nn);
    if (!p || !h_master) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    DD_CUDA_TRY(cudaDeviceSynchronize());
    DD_CUDA_TRY(cudaMemcpy(h_master, p->master, (size_t)p->L.total * 4, cudaMemcpyDeviceToHost));
    return DD_OK;
}

dd_status dd_nn_forward(dd_nn *nn, const uint16_t *d_x, int n, float *d_logits, void *stream) {
    NN *p = reinterpret_cast<NN *>(nn);
    if (!p || !d_x || n <= 0 || n > p->max_batch) return fail(DD_ERR_INVALID_ARG, "bad classifier forward arguments");
    cudaStream_t s = (cudaStream_t)stream;
    dd_status st = nn_forward(p, d_x, n, s, false);
    if (st != DD_OK) return st;
    if (d_logits) DD_CUDA_TRY(cudaMemcpyAsync(d_logits, p->z, (size_t)n * 4, cudaMemcpyDeviceToDevice, s));
    return DD_OK;
}

dd_status dd_nn_forward_tc(dd_nn *nn, const uint16_t *d_x, int n, float *d_logits, void *stream) {
    NN *p = reinterpret_cast<NN *>(nn);
    if (!p || !d_x || n <= 0 || n > p->max_batch) return fail(DD_ERR_INVALID_ARG, "bad classifier forward arguments");
    if (((uintptr_t)d_x) % 16 != 0) return fail(DD_ERR_INVALID_ARG, "snippets must be 16-byte aligned");
    cudaStream_t s = (cudaStream_t)stream;
    dd_status st = nn_forward_tc(p, d_x, n, s);
    if (st != DD_OK) return st;
    if (d_logits) DD_CUDA_TRY(cudaMemcpyAsync(d_logits, p->z, (size_t)n * 4, cudaMemcpyDeviceToDevice, s));
    return DD_OK;
}

dd_status dd_nn_status(const dd_nn *nn, unsigned *flags) {
    const NN *p = reinterpret_cast<const NN *>(nn);
    if (!p || !flags) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    DD_CUDA_TRY(cudaMemcpy(flags, p->tc_err, 4, cudaMemcpyDeviceToHost));
    return DD_OK;
}

dd_status dd_nn_backward(dd_nn *nn, const uint16_t *d_x, const float *d_labels, int n, void *stream) {
    NN *p = reinterpret_cast<NN *>(nn);
    if (!p || !d_x || !d_labels || n <= 0 || n > p->max_batch)
        return fail(DD_ERR_INVALID_ARG, "bad classifier backward arguments");
    cudaStream_t s = (cudaStream_t)stream;
    dd_status st = nn_forward(p, d_x, n, s, true);
    if (st != DD_OK) return st;
    const Layout &L = p->L;
    float *g = p->grad;
    bce_kernel<<<1, n <= 256 ? 256 : 1024, 0, s>>>(p->z, d_labels, n, p->dz, p->loss);
    fc2_bwd_kernel<<<1 + std::min((n + 7) / 8, 2 * p->nsm), 1024, 0, s>>>(p->dz, p->h1, p->bf + L.f2w, n, g + L.f2w,
                                                                          g + L.f2b, g + L.f1b, p->dh);
    fc1_bwd_w_kernel<<<dim3(kFcIn / 64, kFcHid / 16), 256, 0, s>>>(p->dh, p->pooled[3], n, g + L.f1w);
    fc1_bwd_x_kernel<<<dim3((unsigned)((n + 15) / 16), kFcIn / 64), 256, 0, s>>>(p->dh, p->bf + L.f1w, n, p->dpool[3]);
    const int parts = std::min(n, kMaxPartials);
#define DD_CONV_BWD(l, CI, CO, H, COB, SL)                                                                    \
    {                                                                                                         \
        using CW = ConvBwdWCfg<CI, CO, H, COB, SL>;                                                           \
        using CX = ConvBwdXCfg<CI, CO, H>;                                                                    \
        auto kw = conv_bwd_w_kernel<CI, CO, H, COB, SL>;                                                      \
        auto kx = conv_bwd_x_kernel<CI, CO, H>;                                                               \
        cudaError_t e = cudaFuncSetAttribute(kw, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CW::SMEM); \
        if (e == cudaSuccess)                                                                                 \
            e = cudaFuncSetAttribute(kx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CX::SMEM);         \
        if (e != cudaSuccess) return cuda_fail(e, "classifier backward");                                     \
        const int pw = std::min(n, kMaxPartials / (CO / COB));                                                \
        kw<<<dim3(pw, CO / COB), CW::THREADS, CW::SMEM, s>>>(p->dpool[l], p->pooled[l], p->arg[l],            \
                                                                p->pooled[(l) - 1], n, p->partial);           \
        conv_bwd_w_sum_kernel<<<(CW::NW + 31) / 32, 256, 0, s>>>(p->partial, pw, CO * CI * 9, CO, CO * CW::CQ,  \
                                                                 g + L.cw[l], g + L.cb[l]);                     \
        kx<<<dim3((unsigned)((n + CX::SPB - 1) / CX::SPB), CI / CX::CIB), CX::THREADS, CX::SMEM, s>>>(        \
            p->dpool[l], p->pooled[l], p->arg[l], p->bf + L.cw[l], n, p->dpool[(l) - 1]);                     \
    }
    DD_CONV_BWD(3, 64, 64, 8, 32, 1)
    DD_CONV_BWD(2, 32, 64, 16, 64, 1)
    DD_CONV_BWD(1, 16, 32, 32, 32, 4)
#undef DD_CONV_BWD
    conv0_bwd_w_kernel<<<parts, 512, 0, s>>>(p->dpool[0], p->pooled[0], p->arg[0], d_x, n, p->partial);
    conv_bwd_w_sum_kernel<<<(16 * 9 + 16 + 31) / 32, 256, 0, s>>>(p->partial, parts, 16 * 9, 16, 0, g + L.cw[0],
                                                                  g + L.cb[0]);
    return cuda_fail(cudaGetLastError(), "classifier backward");
}

dd_status dd_nn_get_grads(const dd_nn *nn, float *h_grads, void *stream) {
    const NN *p = reinterpret_cast<const NN *>(nn);
    if (!p || !h_grads) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    DD_CUDA_TRY(cudaMemcpyAsync(h_grads, p->grad, (size_t)p->L.total * 4, cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    DD_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    return DD_OK;
}

dd_status dd_nn_set_grads(dd_nn *nn, const float *h_grads) {
    NN *p = reinterpret_cast<NN *>(nn);
    if (!p || !h_grads) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    DD_CUDA_TRY(cudaMemcpy(p->grad, h_grads, (size_t)p->L.total * 4, cudaMemcpyHostToDevice));
    return DD_OK;
}

dd_status dd_nn_get_loss(const dd_nn *nn, float *h_loss, void *stream) {
    const NN *p = reinterpret_cast<const NN *>(nn);
    if (!p || !h_loss) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    DD_CUDA_TRY(cudaMemcpyAsync(h_loss, p->loss, 4, cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    DD_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    return DD_OK;
}

dd_status dd_nn_adamw(dd_nn *nn, float lr, float beta1, float beta2, float eps, float wd, void *stream) {
    NN *p = reinterpret_cast<NN *>(nn);
    if (!p) return fail(DD_ERR_INVALID_ARG, "NULL classifier");
    if (!(lr >= 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0) || !(wd >= 0))
        return fail(DD_ERR_INVALID_ARG, "bad AdamW hyper-parameters");
    p->step += 1;
    const float c1 = 1.0f - powf(beta1, (float)p->step);
    const float c2 = 1.0f - powf(beta2, (float)p->step);
    const long long P = p->L.total;
    adamw_kernel<<<(unsigned)((P + 255) / 256), 256, 0, (cudaStream_t)stream>>>(P, p->master, p->grad, p->m, p->v,
                                                                                  p->bf, lr, beta1, beta2, eps, wd,
                                                                                  c1, c2);
    refresh_images(p, (cudaStream_t)stream);
    return cuda_fail(cudaGetLastError(), "adamw_kernel launch");
}

dd_status dd_nn_get_state(const dd_nn *nn, float *h_m, float *h_v, uint16_t *h_bf16, int *step) {
    const NN *p = reinterpret_cast<const NN *>(nn);
    if (!p) return fail(DD_ERR_INVALID_ARG, "NULL classifier");
    const size_t P = (size_t)p->L.total;
    DD_CUDA_TRY(cudaDeviceSynchronize());
    if (h_m) DD_CUDA_TRY(cudaMemcpy(h_m, p->m, P * 4, cudaMemcpyDeviceToHost));
    if (h_v) DD_CUDA_TRY(cudaMemcpy(h_v, p->v, P * 4, cudaMemcpyDeviceToHost));
    if (h_bf16) DD_CUDA_TRY(cudaMemcpy(h_bf16, p->bf, P * 2, cudaMemcpyDeviceToHost));
    if (step) *step = p->step;
    return DD_OK;
}

static const char kMagic[8] = {'D', 'D', 'N', 'N', 'C', 'K', 'P', '1'};

dd_status dd_nn_save(const dd_nn *nn, const char *path) {
    const NN *p = reinterpret_cast<const NN *>(nn);
    if (!p || !path) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    const size_t P = (size_t)p->L.total;
    std::vector<float> buf(3 * P);
    DD_CUDA_TRY(cudaDeviceSynchronize());
    DD_CUDA_TRY(cudaMemcpy(buf.data(), p->master, P * 4, cudaMemcpyDeviceToHost));
    DD_CUDA_TRY(cudaMemcpy(buf.data() + P, p->m, P * 4, cudaMemcpyDeviceToHost));
    DD_CUDA_TRY(cudaMemcpy(buf.data() + 2 * P, p->v, P * 4, cudaMemcpyDeviceToHost));
    FILE *f = fopen(path, "wb");
    if (!f) return fail(DD_ERR_INVALID_ARG, "cannot open %s for writing", path);
    const int64_t hdr[2] = {(int64_t)P, (int64_t)p->step};
    bool ok = fwrite(kMagic, 1, 8, f) == 8 && fwrite(hdr, 8, 2, f) == 2 && fwrite(buf.data(), 4, 3 * P, f) == 3 * P;
    ok = (fclose(f) == 0) && ok;
    return ok ? DD_OK : fail(DD_ERR_INTERNAL, "short write to %s", path);
}

dd_status dd_nn_load(dd_nn *nn, const char *path) {
    NN *p = reinterpret_cast<NN *>(nn);
    if (!p || !path) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    const size_t P = (size_t)p->L.total;
    FILE *f = fopen(path, "rb");
    if (!f) return fail(DD_ERR_INVALID_ARG, "cannot open %s", path);
    char magic[8];
    int64_t hdr[2];
    std::vector<float> buf(3 * P);
    bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, kMagic, 8) == 0 && fread(hdr, 8, 2, f) == 2 &&
              hdr[0] == (int64_t)P && fread(buf.data(), 4, 3 * P, f) == 3 * P;
    fclose(f);
    if (!ok) return fail(DD_ERR_INVALID_ARG, "%s is not a classifier checkpoint of %zu parameters", path, P);
    DD_CUDA_TRY(cudaMemcpy(p->master, buf.data(), P * 4, cudaMemcpyHostToDevice));
    DD_CUDA_TRY(cudaMemcpy(p->m, buf.data() + P, P * 4, cudaMemcpyHostToDevice));
    DD_CUDA_TRY(cudaMemcpy(p->v, buf.data() + 2 * P, P * 4, cudaMemcpyHostToDevice));
    to_bf16_kernel<<<(unsigned)((P + 255) / 256), 256>>>((long long)P, p->master, p->bf);
    refresh_images(p, nullptr);
    DD_CUDA_TRY(cudaGetLastError());
    DD_CUDA_TRY(cudaDeviceSynchronize());
    p->step = (int)hdr[1];
    return DD_OK;
}

void dd_nn_destroy(dd_nn *nn) { free_nn(reinterpret_cast<NN *>(nn)); }

}  // extern "C"
