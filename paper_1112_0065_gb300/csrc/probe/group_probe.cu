// Probe of the channel-group tile's give-up paths: the tile routine of the
// product library (gsum.cuh) on tables of its own (gsum_tables.h), with one set
// of its mbarriers expecting an arrival that nobody makes.  No fault and no
// endless wait is involved: the copies land normally and every wait is bounded.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "../gsum_tables.h"
#include "dd_probe.h"

namespace dd {
namespace probe {
dd_status report(dd_status s, const char *msg);
}  // namespace probe

namespace {

using namespace gsum;

constexpr int kProbeChan = 64, kProbeVec = 20, kProbeLd = 528;
constexpr int kProbeSamples = kTile + 15;  // the longest delay

__global__ void __launch_bounds__(kThreads, 1)
    group_probe_kernel(const __grid_constant__ Args args, const __grid_constant__ CUtensorMap map, int withheld,
                       int *ret) {
    extern __shared__ __align__(128) unsigned char gsum_smem[];
    Args a = args;
    a.map = &map;
    if (threadIdx.x == 0) {
        uint64_t *bars = reinterpret_cast<uint64_t *>(gsum_smem);
        for (int b = 0; b < 2; ++b) tc::mbar_init(&bars[b], withheld == 1 ? 2 : 1);
        for (int b = 0; b < kBRing; ++b) {
            tc::mbar_init(&bars[2 + b], withheld == 2 ? kWarps + 1 : kWarps);
            tc::mbar_init(&bars[2 + kBRing + b], withheld == 3 ? kWarps + 1 : kWarps);
        }
        tc::fence_mbar_init();
    }
    Phases phase;
    const bool ok = gsum_tile<12>(a, 0, 0, gsum_smem, phase);
    if (threadIdx.x == 0) *ret = ok ? 1 : 0;
}

}  // namespace
}  // namespace dd

extern "C" dd_status dd_probe_group_tile(int withheld, unsigned poll_limit, const uint8_t *h_in, int32_t *h_delays,
                                         uint32_t *h_out, unsigned *h_err) {
    using namespace dd;
    using namespace dd::gsum;
    if (withheld < 0 || withheld > 3 || poll_limit == 0 || poll_limit > (1u << 20) || !h_in || !h_delays || !h_out ||
        !h_err)
        return probe::report(DD_ERR_INVALID_ARG, "withheld 0..3, poll_limit 1..2^20, buffers non-NULL");
    // the last channel of every five lags by one sample more with each trial, up
    // to 15, then the one before it: 20 vectors, more than the pool holds for
    // three chunks
    for (int d = 0; d < kD; ++d)
        for (int c = 0; c < kProbeChan; ++c) {
            const int v = std::min(d, kProbeVec - 1);
            h_delays[d * kProbeChan + c] = c % kG == kG - 1 ? std::min(v, 15) : c % kG == kG - 2 ? std::max(v - 15, 0) : 0;
        }
    GsumTable t;
    std::vector<uint32_t> tab;
    std::vector<int32_t> ws;
    make_tables(h_delays, kProbeChan, kD, t, tab, ws);
    if (!t.ok || t.n_dmb != 1 || !map_encoder()) return probe::report(DD_ERR_INTERNAL, "group tile probe: no tables");
    // chunk 2 has to wait for a chunk before it, else withheld == 3 withholds nothing
    if ((tab[2 * kRecWords + 2] >> 16) >= 2) return probe::report(DD_ERR_INTERNAL, "group tile probe: no wait for a place");
    const size_t in_bytes = (size_t)kProbeChan * kProbeLd, out_bytes = (size_t)kD * kTile * 4;
    const size_t tab_at = in_bytes + out_bytes, ws_at = tab_at + tab.size() * 4, end = (ws_at + ws.size() * 4 + 15) / 16 * 16;
    unsigned char *buf = nullptr;
    cudaError_t e = cudaMalloc(&buf, end + 16);
    if (e != cudaSuccess) return probe::report(DD_ERR_CUDA, "cudaMalloc");
    if (e == cudaSuccess) e = cudaMemcpy(buf, h_in, in_bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(buf + in_bytes, 0xFF, out_bytes);
    if (e == cudaSuccess) e = cudaMemcpy(buf + tab_at, tab.data(), tab.size() * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(buf + ws_at, ws.data(), ws.size() * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(buf + end, 0, 16);
    Args a = {};
    a.tab = reinterpret_cast<uint32_t *>(buf + tab_at);
    a.ws = reinterpret_cast<int32_t *>(buf + ws_at);
    a.nchunks = t.nchunks;
    a.ndm = kD;
    a.n_dmb = 1;
    a.slot = t.slot;
    a.nout = kTile;
    a.out = reinterpret_cast<uint32_t *>(buf + in_bytes);
    a.ld_out = kTile;
    a.err = reinterpret_cast<unsigned *>(buf + end);
    a.poll_limit = poll_limit;
    int *d_ret = reinterpret_cast<int *>(buf + end + 8), ret = -1;
    CUtensorMap map;
    if (e == cudaSuccess && encode_map(buf, kProbeLd, kProbeSamples, kProbeChan, t.slot, &map) != CUDA_SUCCESS)
        e = cudaErrorInvalidValue;
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(group_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e == cudaSuccess) {
        group_probe_kernel<<<1, kThreads, kSmem>>>(a, map, withheld, d_ret);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(h_err, a.err, 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&ret, d_ret, 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(h_out, a.out, out_bytes, cudaMemcpyDeviceToHost);
    cudaFree(buf);
    if (e != cudaSuccess) return probe::report(DD_ERR_CUDA, "group tile probe");
    if (ret != (*h_err & 1u ? 0 : 1)) return probe::report(DD_ERR_INTERNAL, "group tile probe: return value and error word differ");
    return ret ? DD_OK : probe::report(DD_ERR_TIMEOUT, "the tile gave up waiting");
}
