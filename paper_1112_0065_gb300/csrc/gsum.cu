// Channel-group dedispersion (gsum.cuh): its kernels, the rule that chooses
// between it and the tiled kernel, and the launches.
#include <math.h>

#include <vector>

#include "dd_internal.h"
#include "gsum_tables.h"

namespace dd {

using namespace gsum;

namespace {

template <int NP>
__global__ void __launch_bounds__(kThreads, 1)
    dd_gsum_kernel(const __grid_constant__ Args args, const __grid_constant__ CUtensorMap map) {
    extern __shared__ __align__(128) unsigned char gsum_smem[];
    Args a = args;
    a.map = &map;
    init_bars(gsum_smem);
    Phases phase;
    gsum_tile<NP>(a, (int)(blockIdx.x % (unsigned)a.n_dmb), (long long)(blockIdx.x / (unsigned)a.n_dmb), gsum_smem,
                  phase);
}

// Persistent multi-beam form, as tiled::dd_batch_kernel.
template <int NP>
__global__ void __launch_bounds__(kThreads, 1)
    dd_gsum_batch_kernel(const gsum::BatchDesc *__restrict__ desc, unsigned long long *__restrict__ counter) {
    extern __shared__ __align__(128) unsigned char gsum_smem[];
    long long &s_tile = *reinterpret_cast<long long *>(gsum_smem + kTileWord);
    const long long ntiles = desc->ntiles;
    init_bars(gsum_smem);
    // the maps lie in global memory, which the host writes between launches: each
    // thread that issues copies (lane 0 of every warp) fences for itself
    if ((threadIdx.x & 31) == 0)
        for (int b = 0; b < desc->nbeams; ++b) tc::fence_tensormap(&desc->map[b]);
    Phases phase;
    for (;;) {
        if (threadIdx.x == 0) s_tile = (long long)atomicAdd(counter, 1ULL);
        __syncthreads();
        const long long g = s_tile;
        __syncthreads();
        if (g >= ntiles) break;
        int b = 0;
        while (b + 1 < desc->nbeams && g >= desc->tile_start[b + 1]) ++b;
        Args a = desc->beam[b];
        a.map = &desc->map[b];
        const long long local = g - desc->tile_start[b];
        if (!gsum_tile<NP>(a, (int)(local % a.n_dmb), local / a.n_dmb, gsum_smem, phase)) break;
        // the next tile's beam may have another layout, whose copies land where
        // this tile's threads wrote (zero slot, output rows)
        tc::fence_async_smem();
        __syncthreads();
    }
}

}  // namespace

void build_gsum(Plan *p) {
    GsumTable &t = p->gs;
    std::vector<uint32_t> tab;
    std::vector<int32_t> ws;
    try {
        make_tables(p->delays_host.data(), p->nchan, p->ndm, t, tab, ws);
    } catch (...) {  // no host memory for them: the tiled kernel serves the plan
        t.ok = false;
    }
    if (!t.ok || !map_encoder()) return free_gsum(p);
    cudaError_t e = cudaDeviceGetAttribute(&t.sms, cudaDevAttrMultiProcessorCount, p->device);
    if (e == cudaSuccess) e = cudaMalloc(&t.tab, tab.size() * 4);
    if (e == cudaSuccess) e = cudaMalloc(&t.ws, ws.size() * 4);
    if (e == cudaSuccess) e = cudaMemcpy(t.tab, tab.data(), tab.size() * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(t.ws, ws.data(), ws.size() * 4, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {  // no memory for them: the tiled kernel serves the plan
        cudaGetLastError();
        free_gsum(p);
    }
}

void free_gsum(Plan *p) {
    if (p->gs.tab) cudaFree(p->gs.tab);
    if (p->gs.ws) cudaFree(p->gs.ws);
    p->gs = GsumTable();
}

// The rule compares estimates of SM cycles: tiles in waves of one per SM here
// (GsumTable::tile_cycles each), and in half waves on the tiled kernel (two of
// its CTAs, 16 trials x 1536 outputs, share an SM), whose tiles take 9200 + 86
// cycles a channel (98 with 15 bit-planes).  Both fit the measured times within
// 4 % over 20 to 2048 channels, 24 to 1500 trials and 2000 to 131072 outputs,
// and what they leave out, some 8 us of launch and first copies, is the same.
// A gulp too short to fill the waves stays on the tiled kernel, whose tiles are
// smaller; so does one no longer than a gulp on which the autotuner measured the
// tiled kernel faster (longer ones fill the waves better and keep to the rule).  Measured, tiled / here, in us: 1024 channels x 1500 trials x 6208
// outputs 214 / 236, x 10000 267 / 243, x 131072 2778 / 2372; 1024 x 64 x 40000
// 64 / 111, x 131072 165 / 111; 2048 x 700 x 131072 2783 / 2069; 1024 x 1000
// linear trials to DM 1000 (many vectors) x 20000 320 / 390, x 131072 1861 /
// 1799; 96 x 1500 x 131072 531 / 367; 20 x 400 x 6208 13.6 / 14.9, x 10000
// 19.4 / 15.1.
bool use_gsum(const Plan *const *p, const long long *nout, int n) {
    double tiles = 0, work = 0, tiles16 = 0, work16 = 0;
    for (int i = 0; i < n; ++i) {
        const GsumTable &t = p[i]->gs;
        if (!t.ok || nout[i] <= t.tiled_to || gsum_big(p[i]) != gsum_big(p[0])) return false;
        const double m = (double)((nout[i] + kTile - 1) / kTile) * t.n_dmb;
        tiles += m;
        work += m * t.tile_cycles;
        const double m16 = (double)((nout[i] + 1535) / 1536) * ((p[i]->ndm + 15) / 16);
        tiles16 += m16;
        work16 += m16 * (9200.0 + p[i]->nchan * (p[i]->nchan < 2048 ? 86.0 : 98.0));
    }
    const double sms = p[0]->gs.sms;
    return work / tiles * ceil(tiles / sms) < work16 / tiles16 * ceil(tiles16 / sms);
}

dd_status gsum_map(const Plan *p, const uint8_t *d_in, size_t ld_in_bytes, size_t nsamp_in, CUtensorMap *map) {
    const CUresult r = encode_map(d_in, ld_in_bytes, nsamp_in, p->nchan, p->gs.slot, map);
    return r == CUDA_SUCCESS ? DD_OK : fail(DD_ERR_CUDA, "cuTensorMapEncodeTiled: error %d", (int)r);
}

dd_status gsum_args(const Plan *p, size_t nsamp_in, uint32_t *d_out, size_t ld_out, gsum::Args *out) {
    const GsumTable &t = p->gs;
    Args a;
    a.map = nullptr;
    a.tab = t.tab;
    a.ws = t.ws;
    a.nchunks = t.nchunks;
    a.ndm = p->ndm;
    a.n_dmb = t.n_dmb;
    a.slot = t.slot;
    a.nout = (long long)nsamp_in - p->maxdelay;
    a.out = d_out;
    a.ld_out = (long long)ld_out;
    a.poll_limit = tiled::kStagePollLimit;
    const dd_status es = tile_error_word(&a.err);
    if (es != DD_OK) return es;
    *out = a;
    return DD_OK;
}

// Dynamic shared memory of a CTA, for every plan.
size_t gsum_smem() { return kSmem; }

GsumBatchFn gsum_batch_kernel(bool big) { return big ? dd_gsum_batch_kernel<14> : dd_gsum_batch_kernel<12>; }

dd_status launch_gsum(const Plan *p, const uint8_t *d_in, size_t ld_in_bytes, size_t nsamp_in, uint32_t *d_out,
                      size_t ld_out, cudaStream_t stream) {
    Args a;
    dd_status st = gsum_args(p, nsamp_in, d_out, ld_out, &a);
    if (st != DD_OK) return st;
    CUtensorMap map;
    st = gsum_map(p, d_in, ld_in_bytes, nsamp_in, &map);
    if (st != DD_OK) return st;
    const long long nblocks = (a.nout + kTile - 1) / kTile * a.n_dmb;
    if (nblocks > 0x7fffffffLL) return fail(DD_ERR_INVALID_ARG, "gulp too long for one launch");
    auto kern = gsum_big(p) ? dd_gsum_kernel<14> : dd_gsum_kernel<12>;
    DD_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsum_smem()));
    kern<<<(unsigned)nblocks, kThreads, gsum_smem(), stream>>>(a, map);
    return cuda_fail(cudaGetLastError(), "dd_gsum_kernel launch");
}

}  // namespace dd
