// Host side of the channel-group dedispersion's tile (gsum.cuh): the vectors of
// a delay table, the device tables, and the tensor map of a gulp.
#pragma once

#include <string.h>

#include <algorithm>
#include <atomic>
#include <numeric>
#include <thread>
#include <vector>

#include "dd_internal.h"
#include "gsum.cuh"

namespace dd {
namespace gsum {

// The vectors of one group over one block of trials.
struct Group {
    int nchan = 0;         // channels of the band in it
    int nvec = 0;
    int words = 0;         // words of a vector that some trial reads
    int start[kG] = {};    // first sample of each channel relative to the tile
    uint32_t vec[kD];      // extra delays of channels 1..4, 8 bits each (channel 1 highest), ascending
    uint8_t of[kD];        // vector of each trial
    int off[kD];           // the trial's offset in samples
};

// false: some channel's delay, relative to the group's first, spreads over
// more than one word.
inline bool make_group(const int32_t *delays, int nchan, int ndm, int d0, int c0, Group &g) {
    g.nchan = std::min(kG, nchan - c0);
    const int nd = std::min(kD, ndm - d0);
    const int32_t *first = delays + (size_t)d0 * nchan + c0;
    int lo[kG], rel[kD][kG] = {};
    for (int i = 0; i < kG; ++i) lo[i] = i < g.nchan ? 0x7fffffff : 0;
    for (int j = 0; j < nd; ++j) {
        const int32_t *r = first + (size_t)j * nchan;
        g.off[j] = r[0] - first[0];
        for (int i = 0; i < g.nchan; ++i) {
            rel[j][i] = r[i] - r[0];
            lo[i] = std::min(lo[i], rel[j][i]);
        }
    }
    for (int i = 0; i < kG; ++i) g.start[i] = first[0] + lo[i];
    uint32_t key[kD];
    g.nvec = 0;
    for (int j = 0; j < nd; ++j) {
        key[j] = 0;
        for (int i = 1; i < kG; ++i) {
            const int e = rel[j][i] - lo[i];
            if (e > 15) return false;
            key[j] = key[j] << 8 | (uint32_t)e;
        }
        if (j && key[j] == key[j - 1]) continue;
        uint32_t *end = g.vec + g.nvec, *at = std::lower_bound(g.vec, end, key[j]);
        if (at != end && *at == key[j]) continue;
        memmove(at + 1, at, (size_t)(end - at) * sizeof(uint32_t));
        *at = key[j];
        ++g.nvec;
    }
    for (int j = 0; j < nd; ++j)
        g.of[j] = j && key[j] == key[j - 1] ? g.of[j - 1]
                                            : (uint8_t)(std::lower_bound(g.vec, g.vec + g.nvec, key[j]) - g.vec);
    for (int j = nd; j < kD; ++j) {  // past the last trial: as the last
        g.off[j] = g.off[nd - 1];
        g.of[j] = g.of[nd - 1];
    }
    g.words = (g.off[kD - 1] >> 4) + kHalfWords + 1;  // delays never fall with the trial
    return true;
}

// Dynamic shared memory of a CTA, for every plan: all there is.
constexpr int kSmem = 227 * 1024;

// f(b) for every DM block, on a few threads (1500 trials x 1024 channels: the
// tables took 6 ms of a plan's creation on one); f does not throw.
template <class F>
void each_block(int n, F f) {
    const int want = std::min({8, (int)std::thread::hardware_concurrency(), n / 4});
    std::atomic<int> next{0};
    auto work = [&] {
        for (int b = next++; b < n; b = next++) f(b);
    };
    std::vector<std::thread> threads;
    try {
        for (int k = 1; k < want; ++k) threads.emplace_back(work);
    } catch (...) {  // no more threads: those there are do the work
    }
    work();
    for (std::thread &t : threads) t.join();
}

// Sizes and host tables of the delays [ndm][nchan]; t.ok stays false when they
// do not suit.
inline void make_tables(const int32_t *delays, int nchan, int ndm, GsumTable &t, std::vector<uint32_t> &tab,
                        std::vector<int32_t> &ws) {
    if (nchan < kChunkChans || 3 * nchan >= 1 << 14) return;
    t.n_dmb = (ndm + kD - 1) / kD;
    const int ngroups = (nchan + kG - 1) / kG;
    t.nchunks = ((ngroups + kCG - 1) / kCG + 1) / 2 * 2;
    std::vector<Group> groups((size_t)t.n_dmb * t.nchunks * kCG);
    std::vector<int> from_word((size_t)t.n_dmb * t.nchunks * kParts);  // first staged word of each part
    std::vector<int> most(t.n_dmb, 0);
    std::atomic<bool> suits{true};
    each_block(t.n_dmb, [&](int b) {
        for (int s = 0; s < t.nchunks * kParts && suits; ++s) {
            const size_t k = (size_t)b * t.nchunks * kParts + s;
            int lo = 0x7fffffff, end = 0;
            for (int g = 0; g < kHalfCG && s * kHalfCG + g < ngroups; ++g) {
                Group &x = groups[k * kHalfCG + g];
                if (!make_group(delays, nchan, ndm, b * kD, (s * kHalfCG + g) * kG, x)) {
                    suits = false;
                    return;
                }
                for (int i = 0; i < x.nchan; ++i) {
                    lo = std::min(lo, x.start[i] >> 4);
                    end = std::max(end, (x.start[i] >> 4) + x.words);
                }
            }
            if (s * kHalfCG >= ngroups) continue;
            from_word[k] = lo & ~3;
            most[b] = std::max(most[b], end - from_word[k]);
        }
    });
    if (!suits) return;
    t.slot = (*std::max_element(most.begin(), most.end()) + kHalfWords + 2 + 3) / 4 * 4;
    if (t.slot > 256) return;  // a tensor map's box
    tab.assign((size_t)t.n_dmb * t.nchunks * kRecWords, 0u);
    ws.assign((size_t)t.n_dmb * 2 * kParts, 0);
    // Places in the pool.  First choice for a DM block: each chunk after one of
    // the chunks before it or at the bottom, clear of at least the two before it.
    // Else even chunks at the bottom and odd ones at the top.  Half a vector is
    // padded to 4 cells more than a multiple of 8 where there is room in the DM
    // block: the even and odd words that a quarter-warp stores then fall into
    // different banks.
    const int pool = kSmem - vec_at(t.slot);
    const int nparts = t.nchunks * kParts;
    std::vector<int> need((size_t)t.n_dmb * nparts), half(need.size()), place(need.size());
    std::vector<int> keep((size_t)t.n_dmb * t.nchunks);  // chunks before it that a chunk's place is clear of
    for (int b = 0; b < t.n_dmb; ++b) {
        bool fits = false;
        for (int way = 0; way < 4 && !fits; ++way) {
            const bool pad = !(way & 1), ends = way >= 2;
            long long from[kBRing] = {}, to[kBRing] = {};  // by chunk % kBRing
            fits = true;
            for (int s = 0; s < t.nchunks && fits; ++s) {
                long long bytes[kParts], all = 0;
                for (int q = 0; q < kParts; ++q) {
                    const size_t n = (size_t)b * nparts + s * kParts + q;
                    int nv = 0;
                    need[n] = 0;
                    for (int g = 0; g < kHalfCG; ++g) {
                        need[n] = std::max(need[n], groups[n * kHalfCG + g].words);
                        nv += groups[n * kHalfCG + g].nvec;
                    }
                    half[n] = (need[n] + 1) / 2;
                    while (pad && half[n] && half[n] % 8 != 4) ++half[n];
                    bytes[q] = (long long)nv * half[n] * 32;
                    all += bytes[q];
                }
                // how many of the chunks just before s (kBRing - 1 at most) a place is clear of
                auto clear = [&](long long at) {
                    int w = 0;
                    if (at < 0 || at + all > pool) return 0;
                    for (; w < kBRing - 1 && w < s; ++w)
                        if (at < to[(s - 1 - w) % kBRing] && at + all > from[(s - 1 - w) % kBRing]) return w;
                    return kBRing - 1;
                };
                long long at = ends && (s & 1) ? pool - all : 0;
                int w = clear(at);
                for (int q = 0; q < kBRing - 1 && q < s && !ends; ++q)
                    if (clear(to[(s - 1 - q) % kBRing]) > w) {
                        at = to[(s - 1 - q) % kBRing];
                        w = clear(at);
                    }
                fits = w >= (ends ? 1 : 2);
                keep[(size_t)b * t.nchunks + s] = w;
                from[s % kBRing] = at;
                to[s % kBRing] = at + all;
                for (int q = 0; q < kParts; ++q) {
                    place[(size_t)b * nparts + s * kParts + q] = (int)at;
                    at += bytes[q];
                }
            }
        }
        if (!fits) return;
    }
    std::vector<int> turn(need.size());  // items go round the warps
    for (size_t n = 0, items = 0; n < need.size(); ++n) {
        turn[n] = (int)(items % kWarps);
        items += (size_t)(kHalfCG * need[n] + 31) / 32;
    }
    std::vector<double> alus(t.n_dmb, 0.0);  // ALU instructions of a tile of each DM block
    each_block(t.n_dmb, [&](int b) {
        double alu = 0;
        for (int q = 0; q < 2 * kParts; ++q) ws[(size_t)b * 2 * kParts + q] = from_word[(size_t)b * nparts + q];
        for (int s = 0; s < t.nchunks; ++s) {
            const size_t k = (size_t)b * t.nchunks + s;
            uint32_t *ra = tab.data() + k * kRecWords;
            uint32_t *rb = ra + kAWords;
            for (int part = 0; part < kParts; ++part) {
                const Group *gr = &groups[k * kCG + part * kHalfCG];
                const size_t n = k * kParts + part;
                uint32_t *r = ra + part * kPartWords;
                const int units = (kHalfCG * need[n] + 31) / 32;
                r[0] = (uint32_t)half[n];
                r[1] = (uint32_t)need[n];
                r[3] = s + 2 < t.nchunks ? (uint32_t)from_word[(k + 2) * kParts + part] : 0u;
                r[2] = (uint32_t)units | (uint32_t)turn[n] << 8 | (uint32_t)keep[k] << 16;
                uint32_t at = (uint32_t)(vec_at(t.slot) + place[n]);
                double vwork = 0;
                for (int g = 0; g < kHalfCG; ++g) {
                    const Group &x = gr[g];
                    uint32_t *q = r + 4 + g * kARec;
                    for (int i = 0; i < kG; ++i) {
                        q[i] = i < x.nchan
                                   ? (uint32_t)(raw_at(t.slot, s & 1) + part * raw_bytes(t.slot) +
                                                4 * ((g * kG + i) * t.slot + (x.start[i] >> 4) - from_word[k * kParts + part])) << 5 |
                                         (uint32_t)(2 * (x.start[i] & 15))
                                   : (uint32_t)zero_at(t.slot) << 5;
                    }
                    q[5] = at;
                    q[6] = (uint32_t)x.nvec;
                    for (int v = 0; v < x.nvec; ++v) {
                        const uint32_t e = x.vec[v];
                        const bool fresh = v == 0 || (e >> 16) != (x.vec[v - 1] >> 16);
                        q[8 + 2 * v] = 2 * (e >> 8 & 255) | 2 * (e & 255) << 8 | (fresh ? 0x80u : 0u);
                        q[9 + 2 * v] = 2 * (e >> 24) | 2 * (e >> 16 & 255) << 8;
                        vwork += fresh ? 28 : 20;
                    }
                    for (int j = 0; j < kD; ++j) {
                        uint32_t *e = rb + ((part * kHalfCG + g) * kD + j) * 2;
                        if (x.nchan == 0) {
                            e[0] = (uint32_t)zero_at(t.slot);
                            continue;
                        }
                        const int o = x.off[j] >> 4, h16 = 16 * half[n];
                        e[0] = at + (uint32_t)(x.of[j] * 2 * h16 + ((o & 1) ? h16 : 0) + 16 * (o >> 1));
                        e[1] = (uint32_t)((o & 1) ? 16 - h16 : h16) << 5 | (uint32_t)(2 * (x.off[j] & 15));
                    }
                    at += (uint32_t)(x.nvec * 32 * half[n]);
                }
                alu += kWarps * kDT * kHalfCG * 31.0 + units * (70 + vwork / kHalfCG);
            }
        }
        alus[b] = alu;
    });
    if (pool < kWarps * kHalf * 4) return;  // the finished sums pass through the pool's place
    // two of the ALU's warp instructions a cycle at the 80 % that the kernel reaches
    t.tile_cycles = 0.615 * std::accumulate(alus.begin(), alus.end(), 0.0) / t.n_dmb + 14400;
    t.ok = true;
}

using Encode = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                            const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                            CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, nullptr when it has none.
inline Encode map_encoder() {
    static const Encode encode = [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) !=
                cudaSuccess ||
            found != cudaDriverEntryPointSuccess)
            fn = nullptr;
        return reinterpret_cast<Encode>(fn);
    }();
    return encode;
}

// Tensor map of a gulp's packed rows as words, box = the windows of a part's
// channels; words past the gulp's end read as 0.
inline CUresult encode_map(const uint8_t *d_in, size_t ld_in_bytes, size_t nsamp_in, int nchan, int slot,
                           CUtensorMap *map) {
    const cuuint64_t dim[2] = {(cuuint64_t)((nsamp_in + 15) / 16), (cuuint64_t)nchan};
    const cuuint64_t stride[1] = {(cuuint64_t)ld_in_bytes};
    const cuuint32_t box[2] = {(cuuint32_t)slot, (cuuint32_t)kPartChans}, one[2] = {1, 1};
    return map_encoder()(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<uint8_t *>(d_in), dim, stride, box, one,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

}  // namespace gsum
}  // namespace dd
