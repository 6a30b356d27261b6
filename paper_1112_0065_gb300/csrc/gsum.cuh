// Dedispersion by shared channel-group sums (the single-gulp and the
// persistent multi-beam kernel are in gsum.cu).
//
// Over a block of neighbouring DM trials the delays of five adjacent channels
// relative to the first of them take few distinct combinations: at 1024
// channels and the fine trial grids of a survey, 32 trials share about 8.
// Their sum over those five channels is the same series, only read at another
// offset.  So a CTA (D = 32 trials, 2048 outputs) first forms, for every group
// and every distinct combination (a "vector"), the group's sum as four
// bit-planes in shared memory -- five 2-bit samples sum to at most 15, so no
// bit is wasted -- and every trial then adds the four planes of its vector at
// its own offset: 4 funnel shifts and 8 logic ops per 32 samples and 5
// channels, where adding the channels one by one takes 10 and 20.  The sums
// stay exact.
//
// A plane word holds 16 samples of the tile's first half in its even bits and
// the same 16 positions of the second half (1024 samples later) in its odd
// bits, so that a delay of s samples is a funnel shift by 2 s bits, and two
// words of the packed 2-bit input become the low and the high plane with four
// operations and no transpose.
//
// Bound by the ALU pipe, which the logic ops and the shifts share: 78 % busy at
// 1024 channels x 1500 trials x 131072 outputs, 2373 us against 2780 us for the
// tiled kernel (1.12e9 ALU warp instructions against 1.52e9 at 88 %); the rest
// is the warps' waiting for one another's shares of a chunk.  A barrier a chunk
// took 2739 us, two chunks of slack and smaller chunks 2390, vectors copied
// per channel instead of by tensor maps 80 more.
#pragma once

#include <cuda.h>

#include "dd_internal.h"
#include "tiled_tile.cuh"
#include "tma.cuh"

namespace dd {
namespace gsum {

constexpr int kG = 5;        // channels per group
constexpr int kCG = 4;       // groups per chunk
constexpr int kHalfCG = 2;   // groups per part: one tensor copy, one list of items
constexpr int kParts = kCG / kHalfCG;
constexpr int kPartChans = kG * kHalfCG;
constexpr int kChunkChans = kG * kCG;
constexpr int kWarps = 16;
constexpr int kThreads = 32 * kWarps;
constexpr int kDT = 2;       // trials per warp
constexpr int kD = kWarps * kDT;
constexpr int kHalfWords = 64;            // words of 16 samples per half tile: two per lane
constexpr int kHalf = 16 * kHalfWords;    // samples per half
constexpr int kTile = 2 * kHalf;          // output samples per tile
constexpr int kMaxVec = kD;

// Schedule.  In interval k a warp forms its share of the vectors of chunk k + 1
// (32 words at a time, the shares rotating over the warps) and adds chunk k to
// its two trials.  Warps are not kept in step: one waits for every share of
// chunk k before it adds it, and with a share of its own for the chunks whose
// place in the pool it overwrites to be added by all (where three chunks fit
// the pool that is one interval's slack more), so a warp without a share runs
// ahead of one with.  Stage s (the windows of chunk s, its records) is copied
// when chunk s - 2 is formed.
//
// Table record of chunk s of a DM block, in 32-bit words.  The A part (its
// vectors) has per part (two groups)
//   0     cells of half a vector (its even or odd words)
//   1     words computed per vector
//   2     items of 32 words | first item's warp << 8 | chunks before s that keep their place << 16
//   3     first staged word of the part's channels in chunk s + 2 relative to the tile (a multiple of 4)
// and per group (kARec words each)
//   0..4  per channel (byte offset of its word j = 0 in shared memory << 5) | 2 * (start sample % 16)
//   5     byte offset of vector 0 in shared memory
//   6     number of vectors
//   8..   per vector two words: 2 * (extra delay) of channels 3 and 4 (<< 8), bit 7: channels 1 and 2
//         differ from the previous vector's; and of channels 1 and 2 (<< 8)
// The B part (its trials) has per group and trial two words:
//   0     byte offset of the trial's first cell
//   1     (signed byte distance from there to the cell of the next word << 5) | 2 * (offset % 16)
constexpr int kARec = 8 + 2 * kMaxVec;
constexpr int kPartWords = 4 + kHalfCG * kARec;
constexpr int kAWords = kParts * kPartWords;
constexpr int kBWords = kCG * kD * 2;
constexpr int kRecWords = kAWords + kBWords;
static_assert(kAWords % 4 == 0 && kRecWords % 4 == 0, "16-byte parts");

struct Args {
    const CUtensorMap *map;  // the packed input as 32-bit words, [channel][word]
    const uint32_t *tab;  // [n_dmb][nchunks][kRecWords]
    const int32_t *ws;    // [n_dmb][2][kParts] first staged words of the first two chunks
    int nchunks;          // even; groups past the band are empty
    int ndm;
    int n_dmb;
    int slot;             // staged words per channel, a multiple of 4 (the box of map: slot x kPartChans)
    long long nout;
    uint32_t *out;
    long long ld_out;
    unsigned *err;
    uint32_t poll_limit;
};

constexpr int kBRing = 4;  // B parts, and intervals, that warps may be apart in

// Shared-memory layout in bytes: mbarriers (beside them the persistent kernel's
// tile and the number of stages issued), the two stages' channel windows, a zero
// slot, their A parts, the B parts, the pool of vectors.
constexpr int kTileWord = 112, kStagedWord = 120;
static_assert((2 + 2 * kBRing) * 8 <= kTileWord, "mbarriers");
__host__ __device__ constexpr int raw_bytes(int slot) { return (kPartChans * 4 * slot + 127) / 128 * 128; }
__host__ __device__ constexpr int raw_at(int slot, int b) { return 128 + b * kParts * raw_bytes(slot); }
__host__ __device__ constexpr int zero_at(int slot) { return raw_at(slot, 2); }
__host__ __device__ constexpr int a_at(int slot, int b) { return zero_at(slot) + 4 * slot + b * kAWords * 4; }
__host__ __device__ constexpr int b_at(int slot, int b) { return a_at(slot, 2) + b * kBWords * 4; }
__host__ __device__ constexpr int vec_at(int slot) { return b_at(slot, kBRing); }

using tiled::full_add;

// sum -> p, carry out
__device__ __forceinline__ uint32_t add_into(uint32_t &p, uint32_t a, uint32_t b) {
    uint32_t c;
    full_add(c, p, p, a, b);
    return c;
}

// One word of every vector of a group: the planes of the five channels at the
// group's common start (words j and j + 1 of each), then per vector the
// channels' extra delays and the sum of five 2-bit numbers as four planes.
// Vectors are ordered so that neighbours often share channels 1 and 2, whose
// part of the sum is then kept.  Lanes with store = false form nothing; no lane
// needs another here.
__device__ __forceinline__ void vectors_word(unsigned char *smem, const uint32_t *rec, int j, uint32_t half, bool store) {
    uint32_t lo[kG][2], hi[kG][2];
#pragma unroll
    for (int c = 0; c < kG; ++c) {
        const uint32_t e = rec[c];
        const uint32_t *a = reinterpret_cast<const uint32_t *>(smem + (e >> 5)) + j;
        const uint32_t *b = a + kHalfWords;
        const uint32_t a0 = a[0], a1 = a[1], a2 = a[2], b0 = b[0], b1 = b[1], b2 = b[2];
        const uint32_t x[2] = {__funnelshift_r(a0, a1, e), __funnelshift_r(a1, a2, e)};
        const uint32_t y[2] = {__funnelshift_r(b0, b1, e), __funnelshift_r(b1, b2, e)};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            lo[c][i] = tiled::lop3<0xCA>(0x55555555u, x[i], y[i] << 1);  // first operand selects x over y
            hi[c][i] = tiled::lop3<0xCA>(0x55555555u, x[i] >> 1, y[i]);
        }
    }
    const int nv = store ? (int)rec[6] : 0;  // a lane's own count: those of an item may belong to two groups
    unsigned char *dst = smem + rec[5] + 16u * ((uint32_t)(j >> 1) + ((j & 1) ? half : 0u));
    half *= 32u;
    uint32_t s1 = 0, k1 = 0, s2 = 0, k2 = 0;
    auto one = [&](uint32_t e, uint32_t f, bool live, unsigned char *to) {
        if (e & 0x80u) {
            full_add(k1, s1, lo[0][0], __funnelshift_r(lo[1][0], lo[1][1], f), __funnelshift_r(lo[2][0], lo[2][1], f >> 8));
            full_add(k2, s2, hi[0][0], __funnelshift_r(hi[1][0], hi[1][1], f), __funnelshift_r(hi[2][0], hi[2][1], f >> 8));
        }
        uint32_t p0, p1, p2, p3, ca, cb, cc, t;
        full_add(ca, p0, s1, __funnelshift_r(lo[3][0], lo[3][1], e), __funnelshift_r(lo[4][0], lo[4][1], e >> 8));
        full_add(cb, t, s2, __funnelshift_r(hi[3][0], hi[3][1], e), __funnelshift_r(hi[4][0], hi[4][1], e >> 8));
        full_add(cc, p1, t, k1, ca);
        full_add(p3, p2, k2, cb, cc);
        if (live) *reinterpret_cast<uint4 *>(to) = make_uint4(p0, p1, p2, p3);
    };
    const uint4 *vec = reinterpret_cast<const uint4 *>(rec + 8);
#pragma unroll 1
    for (int v = 0; v < nv; v += 2) {  // a pair past the last vector reads unused words of the record
        const uint4 e = vec[v >> 1];
        one(e.x, e.y, true, dst);
        one(e.z, e.w, v + 1 < nv, dst + half);
        dst += 2u * half;
    }
}

// The four planes of one group at a trial's offset, for a lane's two words.
__device__ __forceinline__ void fetch(const unsigned char *lane_base, uint32_t at, uint32_t e, uint32_t (&v)[2][4]) {
    const unsigned char *p = lane_base + at;
    const uint4 w0 = *reinterpret_cast<const uint4 *>(p);
    const uint4 w1 = *reinterpret_cast<const uint4 *>(p + ((int32_t)e >> 5));
    const uint4 w2 = *reinterpret_cast<const uint4 *>(p + 16);
    v[0][0] = __funnelshift_r(w0.x, w1.x, e);
    v[0][1] = __funnelshift_r(w0.y, w1.y, e);
    v[0][2] = __funnelshift_r(w0.z, w1.z, e);
    v[0][3] = __funnelshift_r(w0.w, w1.w, e);
    v[1][0] = __funnelshift_r(w1.x, w2.x, e);
    v[1][1] = __funnelshift_r(w1.y, w2.y, e);
    v[1][2] = __funnelshift_r(w1.z, w2.z, e);
    v[1][3] = __funnelshift_r(w1.w, w2.w, e);
}

// Transpose the 16 x 32 bit matrix of up to 16 planes: afterwards word r holds
// the value of bit column r in its low half and of column r + 16 in its high
// half.
__device__ __forceinline__ void planes_to_values(uint32_t (&a)[16]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t x = a[k], y = a[k + 8];
        a[k] = __byte_perm(x, y, 0x6240);
        a[k + 8] = __byte_perm(x, y, 0x7351);
    }
    auto swap = [&](int d, uint32_t m) {
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (!(k & d)) {
                const uint32_t x = a[k], y = a[k + d];
                a[k] = tiled::lop3<0xCA>(m, x, y << d);
                a[k + d] = tiled::lop3<0xCA>(m, x >> d, y);
            }
    };
    swap(4, 0x0F0F0F0Fu);
    swap(2, 0x33333333u);
    swap(1, 0x55555555u);
}

// Completions so far of a CTA's mbarriers (number x of a set of n is phase x / n
// of mbarrier x % n): stages and formed chunks, and intervals.  Chunk counts
// are even, so a tile leaves the sets of two at an even count; the sets of four
// keep a running number.
struct Phases {
    uint32_t chunks = 0;  // of the tiles before
};

// Once per CTA, before its first tile; the caller synchronises the block.
__device__ __forceinline__ void init_bars(unsigned char *smem) {
    if (threadIdx.x == 0) {
        uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
        for (int b = 0; b < 2; ++b) tc::mbar_init(&bars[b], 1);  // full: one arrival and the copies' bytes
        for (int b = 0; b < 2 * kBRing; ++b) tc::mbar_init(&bars[2 + b], kWarps);  // formed, spent: one per warp
        tc::fence_mbar_init();
    }
}

// One output tile: DM block dmb x time tile tt.  false (in every thread) when a
// wait ran out of polls: the outputs are then not written, the error word has
// bit 0 set, and the mbarriers serve no further tile.
template <int NP>
__device__ __forceinline__ bool gsum_tile(const Args &a, int dmb, long long tt, unsigned char *smem, Phases &ph) {
    uint64_t *const full = reinterpret_cast<uint64_t *>(smem), *const formed = full + 2, *const spent = formed + kBRing;
    volatile int &staged = *reinterpret_cast<volatile int *>(smem + kStagedWord);  // stages that the tile has issued
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long t0 = tt * kTile;
    const int tw0 = (int)(t0 >> 4);
    const uint32_t *gtab = a.tab + (long long)dmb * a.nchunks * kRecWords;
    for (int i = tid; i < a.slot; i += kThreads) reinterpret_cast<uint32_t *>(smem + zero_at(a.slot))[i] = 0u;
    __syncthreads();

    // stage s into buffer s % 2, by one thread: a tensor copy per part for the
    // windows of its channels (from word ws[part's stride] of the tile; rows past
    // the band and words past the row's end arrive as 0) and one copy for each
    // half of the record.  (A bulk copy per channel cost the issuing warp some 85
    // cycles each.)
    auto stage = [&](int s, const uint32_t *ws, int stride) {
        const int b = s & 1;
        tc::mbar_arrive_expect_tx(&full[b], (uint32_t)(kChunkChans * 4 * a.slot + kRecWords * 4));
#pragma unroll
        for (int q = 0; q < kParts; ++q)
            tc::tensor_copy_g2s(smem + raw_at(a.slot, b) + q * raw_bytes(a.slot), a.map, tw0 + (int)ws[q * stride],
                                s * kChunkChans + q * kPartChans, &full[b]);
        const uint32_t *rec = gtab + (long long)s * kRecWords;
        tc::bulk_copy_g2s(smem + a_at(a.slot, b), rec, kAWords * 4, &full[b]);
        tc::bulk_copy_g2s(smem + b_at(a.slot, s % kBRing), rec + kAWords, kBWords * 4, &full[b]);
        staged = s + 1;
    };
    // A lane whose wait runs out of polls waits no more and skips the work that
    // follows (its sums, and the tile, are then void), but keeps step with its
    // warp.  Lane 0 arrives for the warp, and nowhere any more once it gave up: a
    // phase completes only when every warp's lane 0 came through its waits, so
    // nothing is refilled while another warp reads it, no arrival counts for a
    // later phase, and the other warps run out of polls in their turn.  (The
    // whole warp voting after each wait: 2424 us instead of 2372 for 1024
    // channels x 1500 trials x 131072 outputs.)
    bool ok = true, leader = lane == 0;
    auto wait = [&](uint64_t *bar, uint32_t phase) {
        if (ok) ok = tc::mbar_wait(bar, phase & 1u, a.poll_limit);
        leader = leader && ok;
    };
    // chunk (interval) s of this tile in the sets of kBRing
    auto number = [&](int s) { return ph.chunks + (uint32_t)s; };
    // this warp's share of the vectors of chunk s (an item is 32 words of a part's groups)
    auto form = [&](int s) {
        wait(&full[s & 1], (ph.chunks >> 1) + ((uint32_t)s >> 1));
        const uint32_t *rec = reinterpret_cast<const uint32_t *>(smem + a_at(a.slot, s & 1));
        if (ok) {
#pragma unroll 1
            for (int part = 0; part < kParts; ++part, rec += kPartWords) {
                const uint4 head = *reinterpret_cast<const uint4 *>(rec);
                const int need = (int)head.y, units = (int)(head.z & 255u), keep = (int)(head.z >> 16);
                int u = warp - (int)(head.z >> 8 & 255u);
                u += u < 0 ? kWarps : 0;
                if (u >= units) continue;
                // the latest chunk whose place may be overwritten: those of the tile before
                // are all spent, and so are those before s - 3, as chunk s - 2 is formed
                const int last = s - 1 - keep;
                if (keep < kBRing - 1 && last >= 0) wait(&spent[number(last) % kBRing], number(last) / kBRing);
                if (!ok) break;
                for (; u < units; u += kWarps) {
                    const int i = 32 * u + lane, i1 = min(i, kHalfCG * need - 1);
                    const int g = i1 >= need;
                    vectors_word(smem, rec + 4 + g * kARec, i1 - g * need, head.x, i < kHalfCG * need);
                }
            }
        }
        __syncwarp();
        if (leader) tc::mbar_arrive(&formed[number(s) % kBRing]);
    };

    if (tid == 0)
        for (int s = 0; s < 2; ++s)
            stage(s, reinterpret_cast<const uint32_t *>(a.ws) + (dmb * 2 + s) * kParts, 1);
    form(0);
    uint32_t P[kDT][2][NP], pend[kDT][2][4];
#pragma unroll
    for (int d = 0; d < kDT; ++d)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
#pragma unroll
            for (int k = 0; k < NP; ++k) P[d][i][k] = 0u;
#pragma unroll
            for (int w = 0; w < 4; ++w) pend[d][i][w] = 0u;
        }
    const unsigned char *lane_base = smem + 16 * lane;

#pragma unroll 1
    for (int k = 0; k < a.nchunks; ++k) {
        if (k + 1 < a.nchunks) form(k + 1);
        wait(&formed[number(k) % kBRing], number(k) / kBRing);
        if (ok) {
            if (tid == 32 * (k % kWarps) && k + 2 < a.nchunks)
                stage(k + 2, reinterpret_cast<const uint32_t *>(smem + a_at(a.slot, k & 1)) + 3, kPartWords);
            // the chunk's four groups in a carry-save tree; the trees of two
            // chunks are joined and rippled into the upper planes
            const uint4 *bt = reinterpret_cast<const uint4 *>(smem + b_at(a.slot, k % kBRing)) + warp;
#pragma unroll
            for (int d = 0; d < kDT; ++d) {  // a table cell holds the warp's two trials
                uint32_t q[2][2][4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint4 ea = bt[2 * h * (kD / 2)], eb = bt[(2 * h + 1) * (kD / 2)];
                    uint32_t va[2][4], vb[2][4];
                    fetch(lane_base, d ? ea.z : ea.x, d ? ea.w : ea.y, va);
                    fetch(lane_base, d ? eb.z : eb.x, d ? eb.w : eb.y, vb);
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int w = 0; w < 4; ++w) q[h][i][w] = add_into(P[d][i][w], va[i][w], vb[i][w]);
                }
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int w = 0; w < 4; ++w) q[0][i][w] = add_into(P[d][i][w + 1], q[0][i][w], q[1][i][w]);
                if (k & 1) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        uint32_t c = 0;
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            const uint32_t x = add_into(P[d][i][w + 2], pend[d][i][w], q[0][i][w]);
                            c = add_into(P[d][i][w + 3], x, c);
                        }
#pragma unroll
                        for (int w = 7; w < NP; ++w) {
                            const uint32_t t = P[d][i][w] ^ c;
                            c &= P[d][i][w];
                            P[d][i][w] = t;
                        }
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int w = 0; w < 4; ++w) pend[d][i][w] = q[0][i][w];
                }
            }
        }
        __syncwarp();
        if (leader) tc::mbar_arrive(&spent[number(k) % kBRing]);
    }
    const uint32_t first = ph.chunks;
    ph.chunks += (uint32_t)a.nchunks;
    if (__syncthreads_or(!ok)) {
        // a stage or an interval never completed: record it, give the last two
        // stages' copies one more short bounded wait, and leave the outputs alone
        if (tid == 0) atomicOr(a.err, 1u);
        const uint32_t last = a.poll_limit / 64 + 1;
        for (int s = staged - 2; s < staged; ++s)
            tc::mbar_wait(&full[s & 1], ((first >> 1) + ((uint32_t)s >> 1)) & 1u, last);
        return false;
    }

    // planes -> sums, through shared memory (the pool's place, 4 KB per warp,
    // 16-byte cells in an order free of bank conflicts) so that a warp stores
    // 512 bytes of a row at a time; straight from the lanes every store touched
    // 32 rows of 16 bytes and the end of a tile cost a tenth of it
    uint4 *rows = reinterpret_cast<uint4 *>(smem + vec_at(a.slot) + warp * kHalf * 4);
#pragma unroll
    for (int d = 0; d < kDT; ++d) {
        const int dm = dmb * kD + warp * kDT + d;
        if (dm >= a.ndm) continue;
        uint32_t *orow = a.out + (long long)dm * a.ld_out;
        uint32_t v[2][16];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
#pragma unroll
            for (int k = 0; k < 16; ++k) v[i][k] = k < NP ? P[d][i][k] : 0u;
            planes_to_values(v[i]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // even columns: the first half's samples, odd: the second's
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t s[4];
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const uint32_t x = v[i][2 * ((4 * q + m) % 8) + h];  // samples n and n + 8 share a word
                        s[m] = q < 2 ? x & 0xFFFFu : x >> 16;
                    }
                    rows[(8 * lane + 4 * i + q) ^ (lane & 7)] = make_uint4(s[0], s[1], s[2], s[3]);
                }
            __syncwarp();
#pragma unroll 4
            for (int m = 0; m < kHalf / 128; ++m) {
                const int cell = 32 * m + lane;
                const uint4 s = rows[cell ^ ((cell >> 3) & 7)];
                const long long t = t0 + h * kHalf + 4 * cell;
                if (t + 4 <= a.nout) {
                    *reinterpret_cast<uint4 *>(orow + t) = s;
                } else {
                    if (t < a.nout) orow[t] = s.x;
                    if (t + 1 < a.nout) orow[t + 1] = s.y;
                    if (t + 2 < a.nout) orow[t + 2] = s.z;
                }
            }
            __syncwarp();
        }
    }
    return true;
}

// Work list of the persistent multi-beam kernel, as tiled::BatchDesc.
struct BatchDesc {
    CUtensorMap map[DD_BATCH_MAX_BEAMS];
    Args beam[DD_BATCH_MAX_BEAMS];
    long long tile_start[DD_BATCH_MAX_BEAMS + 1];
    long long ntiles;
    int nbeams;
};

}  // namespace gsum
}  // namespace dd
