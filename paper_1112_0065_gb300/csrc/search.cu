// Search stage after dedispersion (paper Section 2.3): baseline removal,
// boxcar matched filtering over a list of widths, a sigma cut and grouping of
// contiguous above-threshold cells into events, and DM-time snippets around
// each event for the classifier.
//
// Kernels (all exact integer arithmetic up to the S/N division):
//  * dd_median_kernel   every warp follows the lower median of the sliding window
//                    [t-half, t+half) of its own row segment, 32 outputs at a
//                    time; writes y = x - median and adds sum(y^2) to the row
//                    total (int64).
//  * dd_mean_kernel  the paper's running mean instead (an option): x minus the
//                    window mean rounded half up.
//  * dd_mf_kernel       a CTA loads a tile of y plus the widest boxcar's halo,
//                    prefix-sums it in shared memory, and for every sample
//                    decides with integer thresholds whether some width reaches
//                    the S/N cut; hot cells get their best S/N and width and a
//                    bit in the row's hot bitmask.
//  * runs/vunion/compress/group_reduce kernels: 4-connected groups in
//                    (DM, time) from runs of hot cells along time joined across
//                    rows by union-find (roots = smallest run start, so the
//                    result is deterministic); one record per group at its best
//                    cell.
//  * mark/count_marks/scan_chunks/write_marks: the records in (DM, time) order.
//  * dd_snippet_kernel  64 DM rows x 64 bins of w samples around each event, each
//                    bin the S/N of its boxcar, rounded to bfloat16.
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <type_traits>

#include "dd_internal.h"

namespace dd {
namespace {

constexpr int kMaxWidths = 16;
constexpr int kMfThreads = 256;
constexpr int kMfTile = 4096;
constexpr int kCompactThreads = 256;
constexpr int kCompactChunk = 1 << 16;  // cells per compaction chunk
constexpr unsigned kUnionCap = 1u << 22;  // bound on union-find retries per edge

struct DevState {
    unsigned long long nhot;
    unsigned int nroots;
    unsigned int err;  // bit 0: value beyond histogram; bit 2: union cap hit
    unsigned long long nrebuild;  // median histograms recounted from their window
};

struct SearchCfgDev {
    int nw;
    int widths[kMaxWidths];
    unsigned wmask;  // bit j: width 2^j is searched (widths are powers of two <= 1024)
};
constexpr int kPows = 11;  // possible widths 2^0 .. 2^10

// ---------------------------------------------------------------------------
// baseline: sliding lower median by histogram walk
// ---------------------------------------------------------------------------

// A warp takes the lower medians of one row segment, 32 consecutive outputs (one
// per lane) at a time.  It keeps m, a value near the coming medians, how many
// values of the window [t - h, t + h) of the step's first output lie below m and
// how many not above it, and a histogram of the values around m.  Ballots over
// the values that enter and leave with the step's 32 moves give both counts for
// every lane's own window; only where some lane's median is not m does the warp
// walk along the histogram, one pair of ballots per value.
//
// Bound by instruction issue.  One lane per row segment, its histogram in its
// own bank (what this replaces), took about as many instructions, but all of an
// output's bookkeeping was one dependency chain, 8192 outputs and counts long,
// with too few lanes to hide it.  Measured, window 8192: the search of a
// dedispersed gulp of 1500 x 131072 with pulses and interference 2606 us before,
// 1875 now (the medians alone 1496 and 750); searches of noise rows, 700 x 100003:
// 1800 before, 999 now, 16 x 100000: 1126 and 116; 1500 x 40000 with window
// 1000: 1009 and 904; 300 x 20000 with window 128 and steps in the rows: 254 and
// 205.  A bound on the counts by one warp sum before the ballots
// settled two steps in three at window 8192 and cost more than it saved.
constexpr int kMwWarps = 4;    // warps per block, each on its own row segment
constexpr int kMwBins = 256;   // values base .. base + 255 are counted
constexpr int kMwUnroll = 2;   // of the step loop (4: 2457 us instead of 2399 for a search with window 2048)
constexpr int kMwBlocks = 8;   // blocks per SM: 64 registers a thread
constexpr unsigned kMwGroup = 4;  // steps of 32 outputs per group of copies; two groups are on their way

__device__ __forceinline__ void copy_async4(uint32_t *dst, const uint32_t *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Every output of the group of steps from t has its whole window [t - h, t + h)
// in the row, and is one of those up to stop.
__device__ __forceinline__ bool group_inside(unsigned t, unsigned h, unsigned n, unsigned stop) {
    return t >= h && t + 32 * kMwGroup + h <= n && t + 32 * kMwGroup <= stop;
}

// Start copying the values of kMwGroup steps of 32 outputs: x[t], x[t + h] and
// x[t - h] of the lane's outputs, into words 0, 32 and 64 of each step's 96 (a
// lane reads only what it copied itself; values outside the row are not copied).
__device__ __forceinline__ void fetch_group(uint32_t *to, const uint32_t *row, unsigned tg, int lane, unsigned h,
                                            unsigned n, unsigned stop) {
    const unsigned t = tg + (unsigned)lane;
    const uint32_t *p = row + t;
    if (group_inside(tg, h, n, stop)) {
#pragma unroll
        for (int j = 0; j < (int)kMwGroup; ++j) {
            copy_async4(to + 96 * j, p + 32 * j);
            copy_async4(to + 96 * j + 32, p + h + 32 * j);
            copy_async4(to + 96 * j + 64, p - h + 32 * j);
        }
    } else {
#pragma unroll 1
        for (unsigned j = 0; j < kMwGroup; ++j)
            if (t + 32 * j < stop) {
                copy_async4(to + 96 * j, p + 32 * j);
                if (t + 32 * j + h < n) copy_async4(to + 96 * j + 32, p + h + 32 * j);
                if (t + 32 * j >= h) copy_async4(to + 96 * j + 64, row + (t + 32 * j - h));
            }
    }
    copy_commit();
}

// H[bin] += by, if the bin is one.
__device__ __forceinline__ void mw_bump(uint32_t h_addr, int bin, uint32_t by) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.lt.u32 p, %1, %3;\n@p red.shared.add.u32 [%0], %2;\n}" ::"r"(h_addr + 4u * (uint32_t)bin),
        "r"(bin), "r"(by), "n"(kMwBins)
        : "memory");
}

// Histogram of row[lo, hi) (values clipped to top) in kMwBins bins of 2^shift
// values from base; returns the count of values below base.
__device__ __forceinline__ int mw_count(const uint32_t *__restrict__ row, unsigned lo, unsigned hi, uint32_t top,
                                        int base, int shift, uint32_t *H, int lane) {
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kMwBins / 32; ++k) H[32 * k + lane] = 0u;
    __syncwarp();
    int below = 0;
    unsigned i = lo + (unsigned)lane;
    const uint32_t h_addr = (uint32_t)__cvta_generic_to_shared(H);
    auto one = [&](uint32_t v) {
        const int e = (int)min(v, top) - base;
        below -= e >> 31;
        mw_bump(h_addr, e >> shift, 1u);
    };
    for (; i + 7 * 32 < hi; i += 8 * 32) {
        uint32_t v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldg(row + i + 32 * u);
#pragma unroll
        for (int u = 0; u < 8; ++u) one(v[u]);
    }
    for (; i < hi; i += 32) one(__ldg(row + i));
    __syncwarp();
    return __reduce_add_sync(0xffffffffu, below);
}

// Bin of rank r from below values under the first bin: -> false when it lies
// outside; c0 / c1: values under the bin, and under the next.
__device__ __forceinline__ bool mw_find(const uint32_t *H, int lane, int below, int r, int &bin, int &c0, int &c1) {
    constexpr int kPer = kMwBins / 32;
    uint32_t v[kPer];
    int sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        v[k] = H[kPer * lane + k];
        sum += (int)v[k];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    int lo = below + incl - sum;
    const unsigned who = __ballot_sync(0xffffffffu, lo <= r && r < lo + sum);
    if (!who) return false;
    int b = kPer * lane, hi = lo;
#pragma unroll
    for (int k = 0; k < kPer; ++k)
        if (hi <= r) {  // the bin is k or a later one
            lo = hi;
            hi += (int)v[k];
            b = kPer * lane + k;
        }
    const int src = __ffs(who) - 1;
    bin = __shfl_sync(0xffffffffu, b, src);
    c0 = __shfl_sync(0xffffffffu, lo, src);
    c1 = __shfl_sync(0xffffffffu, hi, src);
    return true;
}

__global__ void __launch_bounds__(32 * kMwWarps, kMwBlocks) dd_median_kernel(
    const uint32_t *__restrict__ x, long long ld_x, int ndm, unsigned n, unsigned h, unsigned seg, unsigned nseg,
    uint32_t top, int32_t *__restrict__ y, long long ld_y, unsigned long long *__restrict__ sumsq, DevState *st) {
    __shared__ __align__(16) uint32_t s_hist[kMwWarps][kMwBins];
    __shared__ uint32_t s_ring[kMwWarps][2][kMwGroup][3][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t *const H = s_hist[wid];
    const uint32_t h_addr = (uint32_t)__cvta_generic_to_shared(H);
    const long long g = (long long)blockIdx.x * kMwWarps + wid;
    const int d = (int)(g / nseg);
    if (d >= ndm) return;
    unsigned t0 = (unsigned)(g % nseg) * seg;
    const unsigned t_end = min(n, t0 + seg);
    const uint32_t *const row = x + (long long)d * ld_x;
    int32_t *const yrow = y + (long long)d * ld_y;

    // the first window's median is expected near that of 64 of its values
    int guess;
    {
        const unsigned lo = t0 - min(t0, h);
        const unsigned long long span = min(n, t0 + h) - 1 - lo;
        const uint32_t v0 = min(__ldg(row + lo + (unsigned)(span * (unsigned)lane / 63u)), top);
        const uint32_t v1 = min(__ldg(row + lo + (unsigned)(span * (unsigned)(lane + 32) / 63u)), top);
        int less = 0, same = 0;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
            const uint32_t a = __shfl_sync(0xffffffffu, v0, k), b = __shfl_sync(0xffffffffu, v1, k);
            less += (a < v0) + (b < v0);
            same += (a == v0) + (b == v0);
        }
        // the value of the first half whose rank comes nearest the middle
        const int off = max(0, max(less - 31, 32 - (less + same)));
        const int best = (int)__reduce_min_sync(0xffffffffu, (unsigned)off);
        guess = (int)__shfl_sync(0xffffffffu, v0, __ffs(__ballot_sync(0xffffffffu, off == best)) - 1);
    }
    unsigned long long ssq = 0;
    uint32_t most = 0;
    unsigned builds = 0;

    // One go: the histogram from the window of t0, then steps of 32 outputs
    // until the segment ends or a median lies beyond the bins; the next go
    // starts at that output, with its bins around the median before it (its
    // first output's median is then within the bins).
#pragma unroll 1
    while (t0 < t_end) {
        auto inside = [&](unsigned t) { return group_inside(t, h, n, t_end); };
        auto fetch = [&](unsigned t, int half) {
            fetch_group(&s_ring[wid][half][0][0][lane], row, t, lane, h, n, t_end);
        };
        fetch(t0, 0);
        fetch(t0 + 32 * kMwGroup, 1);

        // state: base = value of the first bin, m = a value near the coming
        // medians, b0 / b1 = values of the window below m / not above it
        int base = max(0, guess - kMwBins / 2), m, b0, b1;
        {
            const unsigned lo = t0 - min(t0, h), hi = min(n, t0 + h);
            const int rank = (int)(hi - lo - 1) >> 1;
            // around the guess; where the median is not there, it is narrowed
            // down from all values (65532 at most), 32 bins at a time
            int shift = 0, at = 0, bin;
            bool narrowing = false;
#pragma unroll 1
            for (;;) {
                const int below = mw_count(row, lo, hi, top, base, shift, H, lane);
                const bool found = mw_find(H, lane, below, rank, bin, b0, b1);
                if (found && shift == 0) break;
                if (!narrowing) {
                    narrowing = true;
                    shift = 11;
                } else {
                    at += bin << shift;
                    shift = shift == 1 ? 0 : shift - 5;
                }
                base = shift ? at : max(0, at - kMwBins / 2);
            }
            m = base + bin;
            ++builds;
        }

        // 32 outputs; FULL: of an inside group.  Returns those before the first
        // whose median lies beyond the bins.
        auto step = [&](auto is_full, unsigned ts, const uint32_t *from) {
            constexpr bool FULL = decltype(is_full)::value;
            const unsigned t = ts + (unsigned)lane;
            const bool act = FULL || t < t_end;
            const uint32_t nc = from[0];
            int vi = (int)min(from[32], top), vo = (int)min(from[64], top);
            if (!FULL) {  // past the row: above every median
                if (t + h >= n) vi = (int)top + 1;
                if (t < h) vo = (int)top + 1;
            }
            // values that enter and leave with the 32 moves: below m, not above it
            const unsigned lt = (1u << lane) - 1u;
            const unsigned i0 = __ballot_sync(0xffffffffu, vi < m), o0 = __ballot_sync(0xffffffffu, vo < m);
            const unsigned i1 = __ballot_sync(0xffffffffu, vi <= m), o1 = __ballot_sync(0xffffffffu, vo <= m);
            // the median's rank (past the row of no use)
            const int r = FULL ? (int)h - 1 : ((int)(min(n, t + h) - (t - min(t, h))) - 1) >> 1;
            // m is the median of all 32?  (Of a window of 8192 noise values nine
            // times in ten.)
            const int c0 = b0 + __popc(i0 & lt) - __popc(o0 & lt), c1 = b1 + __popc(i1 & lt) - __popc(o1 & lt);
            int med = m, to = m, done = 32;
            if (__any_sync(0xffffffffu, act && (c0 > r || c1 <= r))) {
                // values of the window of output t that are below v: (those of
                // the window of ts) + (entered since) - (left since)
                auto since = [&](int v) {
                    return __popc(__ballot_sync(0xffffffffu, vi < v) & lt) -
                           __popc(__ballot_sync(0xffffffffu, vo < v) & lt);
                };
                __syncwarp();
                int v = m + 1, b = b1, c = c1;
                unsigned left;  // lanes whose median is v or above it, below
#pragma unroll 1
                while ((left = __ballot_sync(0xffffffffu, act && c <= r))) {
                    if (v - base >= kMwBins) {
                        done = __ffs(left) - 1;
                        break;
                    }
                    if (c <= r) med = v;
                    b += (int)H[v - base];
                    ++v;
                    c = b + since(v);
                }
                v = m, b = b0, c = c0;
#pragma unroll 1
                while ((left = __ballot_sync(0xffffffffu, act && c > r))) {
                    --v;
                    if (v < base) {
                        done = min(done, __ffs(left) - 1);
                        break;
                    }
                    if (c > r) med = v;
                    b -= (int)H[v - base];
                    c = b + since(v);
                }
                to = __shfl_sync(0xffffffffu, med, 31);
                __syncwarp();
            }
            if (act && lane < done) {
                most = max(most, nc);
                const int yv = (int)min(nc, top) - med;
                yrow[t] = yv;
                ssq += (unsigned long long)((long long)yv * yv);
            }
            if (done < 32) {
                if (done) m = __shfl_sync(0xffffffffu, med, done - 1);
                return done;
            }
            // the window moves on by 32
            mw_bump(h_addr, vi - base, 1u);
            mw_bump(h_addr, vo - base, 0xffffffffu);
            b0 += __popc(i0) - __popc(o0);
            b1 += __popc(i1) - __popc(o1);
            if (m != to) {
                __syncwarp();
                while (m < to) {
                    b0 = b1;
                    ++m;
                    b1 += (int)H[m - base];
                }
                while (m > to) {
                    b1 = b0;
                    --m;
                    b0 -= (int)H[m - base];
                }
                __syncwarp();
            }
            return done;
        };
        int half = 0;
        bool far = false;
#pragma unroll 1
        while (t0 < t_end) {
            copy_wait<1>();
            const uint32_t *from = &s_ring[wid][half][0][0][lane];
            if (inside(t0)) {
#pragma unroll kMwUnroll
                for (unsigned j = 0; j < kMwGroup; ++j) {
                    const int done = step(std::true_type(), t0 + 32 * j, from + 96 * j);
                    if (done < 32) {
                        t0 += 32 * j + (unsigned)done;
                        far = true;
                        break;
                    }
                }
            } else {
#pragma unroll 1
                for (unsigned j = 0; j < kMwGroup && t0 + 32 * j < t_end; ++j) {
                    const int done = step(std::false_type(), t0 + 32 * j, from + 96 * j);
                    if (done < 32) {
                        t0 += 32 * j + (unsigned)done;
                        far = true;
                        break;
                    }
                }
            }
            if (far) break;
            fetch(t0 + 64 * kMwGroup, half);
            half ^= 1;
            t0 += 32 * kMwGroup;
        }
        copy_wait<0>();
        __syncwarp();
        guess = m;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) ssq += __shfl_down_sync(0xffffffffu, ssq, o);
    if (lane == 0) {
        atomicAdd(sumsq + d, ssq);
        if (builds > 1) atomicAdd(&st->nrebuild, (unsigned long long)(builds - 1));
    }
    if (most > top) atomicOr(&st->err, 1u);
}

// Outputs per segment.  A segment takes in its first window at the cost of `first`
// outputs (the medians' histogram 0.15 of one per value, the means' sum 0.05), so
// long ones are cheaper, but the warps have to fill the
// device (32 per SM, half a segment's time lost at the end).  Measured for whole
// searches of 1500 x 131072, h 4096, segments of 2048 / 4096 / 8192 (chosen):
// 2718 / 2576 / 2504 us (40 warps per SM then); 16 x 100000, segments of 256 (chosen) / 4096: 142 / 167.
unsigned row_segment(int sms, int ndm, long long n, double first) {
    unsigned best = 0;
    double least = 0;
    for (unsigned seg = 256; seg <= 32768; seg *= 2) {
        const double warps = (double)ndm * (double)((n + seg - 1) / seg);
        const double cost = (std::max(warps / ((double)sms * kMwBlocks * kMwWarps), 1.0) + 0.5) * (first + seg);
        if (!best || cost < least) {
            best = seg;
            least = cost;
        }
    }
    return best;
}

// ---------------------------------------------------------------------------
// baseline, paper form: running mean (rounded half up)
// ---------------------------------------------------------------------------

// floor(a / m) from inv = floor((2^32 - 1) / m), for a < 2^32 and 1 <= m < 2^17:
// 2^32 / m exceeds inv by 1 at most, so the product's high word is the quotient
// or one less, and the remainder tells.
__device__ __forceinline__ uint32_t udiv_by(uint32_t a, uint32_t m, uint32_t inv) {
    const uint32_t q = __umulhi(a, inv);
    return q + (a - q * m >= m ? 1u : 0u);
}

// y[t] = x[t] - floor((S + floor(m/2)) / m) for the window sum S of its m
// values (= the mean rounded half up; S < 2^32 since m <= 65534 and x <=
// 65532), and the row's sum of y^2.  A warp takes a row segment as in the median
// kernel, one lane per output: S moves by the difference of the value that
// enters and the one that leaves, scanned over the warp.  Nothing but x is read
// and nothing but y written; a block that staged 8192 outputs with both windows'
// values and scanned them in shared memory (what this replaces) read and added
// every value twice: 253 us for 700 x 100003 with window 8192, now 204 (0.56 GB,
// 82 us).  Issue slots are 62 % taken, 64 thread instructions per output; the
// rest is the latency of the scan's five steps, of which a warp has four side by
// side, with 28 warps on an SM.
__global__ void __launch_bounds__(32 * kMwWarps, kMwBlocks) dd_mean_kernel(
    const uint32_t *__restrict__ x, long long ld_x, int ndm, unsigned n, unsigned h, unsigned seg, unsigned nseg,
    uint32_t top, int32_t *__restrict__ y, long long ld_y, unsigned long long *__restrict__ sumsq, DevState *st) {
    __shared__ uint32_t s_ring[kMwWarps][2][kMwGroup][3][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long g = (long long)blockIdx.x * kMwWarps + wid;
    const int d = (int)(g / nseg);
    if (d >= ndm) return;
    unsigned t0 = (unsigned)(g % nseg) * seg;
    const unsigned t_end = min(n, t0 + seg);
    const uint32_t *const row = x + (long long)d * ld_x;
    int32_t *const yrow = y + (long long)d * ld_y;
    fetch_group(&s_ring[wid][0][0][0][lane], row, t0, lane, h, n, t_end);
    fetch_group(&s_ring[wid][1][0][0][lane], row, t0 + 32 * kMwGroup, lane, h, n, t_end);

    // sum of the first window
    uint32_t sum = 0;
    {
        unsigned i = t0 - min(t0, h) + (unsigned)lane;
        const unsigned hi = min(n, t0 + h);
        for (; i + 7 * 32 < hi; i += 8 * 32) {
            uint32_t v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = __ldg(row + i + 32 * u);
#pragma unroll
            for (int u = 0; u < 8; ++u) sum += min(v[u], top);
        }
        for (; i < hi; i += 32) sum += min(__ldg(row + i), top);
        sum = __reduce_add_sync(0xffffffffu, sum);  // below 2^32
    }
    const uint32_t m_full = 2 * h, inv_full = 0xffffffffu / m_full;
    unsigned long long ssq = 0;
    uint32_t most = 0;
    // the outputs of one group; FULL: an inside one
    auto group = [&](auto is_full, const uint32_t *from) {
        constexpr bool FULL = decltype(is_full)::value;
        uint32_t cur[kMwGroup], incl[kMwGroup], own[kMwGroup];
#pragma unroll
        for (int j = 0; j < (int)kMwGroup; ++j) {
            const unsigned t = t0 + 32 * j + (unsigned)lane;
            const bool act = FULL || t < t_end;
            cur[j] = act ? from[96 * j] : 0u;
            own[j] = (FULL || (act && t + h < n) ? min(from[96 * j + 32], top) : 0u) -
                     (FULL || (act && t >= h) ? min(from[96 * j + 64], top) : 0u);
            incl[j] = own[j];
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {  // the four steps' moves, scanned over the warp
            const bool add = lane >= o;
#pragma unroll
            for (int j = 0; j < (int)kMwGroup; ++j) {
                const uint32_t u = __shfl_up_sync(0xffffffffu, incl[j], o);
                if (add) incl[j] += u;
            }
        }
#pragma unroll
        for (int j = 0; j < (int)kMwGroup; ++j) {
            const unsigned t = t0 + 32 * j + (unsigned)lane;
            const uint32_t S = sum + incl[j] - own[j];
            uint32_t mean;
            if (FULL) {
                mean = udiv_by(S + h, m_full, inv_full);
            } else {
                const uint32_t m = t < t_end ? min(n, t + h) - (t - min(t, h)) : 1u;
                mean = udiv_by(S + m / 2, m, 0xffffffffu / m);
            }
            most = max(most, cur[j]);
            const int32_t yv = (int32_t)min(cur[j], top) - (int32_t)mean;
            if (FULL || t < t_end) {
                yrow[t] = yv;
                ssq += (unsigned long long)((long long)yv * yv);
            }
            sum += __shfl_sync(0xffffffffu, incl[j], 31);
        }
    };
    int half = 0;
#pragma unroll 1
    for (; t0 < t_end; t0 += 32 * kMwGroup) {
        copy_wait<1>();
        const uint32_t *from = &s_ring[wid][half][0][0][lane];
        if (group_inside(t0, h, n, t_end))
            group(std::true_type(), from);
        else
            group(std::false_type(), from);
        fetch_group(&s_ring[wid][half][0][0][lane], row, t0 + 64 * kMwGroup, lane, h, n, t_end);
        half ^= 1;
    }
    copy_wait<0>();
#pragma unroll
    for (int o = 16; o; o >>= 1) ssq += __shfl_down_sync(0xffffffffu, ssq, o);
    if (lane == 0 && ssq) atomicAdd(sumsq + d, ssq);
    if (most > top) atomicOr(&st->err, 1u);
}

// ---------------------------------------------------------------------------
// matched filter + sigma cut
// ---------------------------------------------------------------------------

// Per (row, width): the denominator float(sigma*sqrt(w)) and the smallest
// boxcar sum S whose S/N, float(S)/den rounded to nearest, reaches thresh.
// The rounded quotient never decreases as S grows, so a cell is hot exactly
// when some S_w >= T_w, decided with integer compares.
__global__ void dd_thresh_kernel(const unsigned long long *__restrict__ sumsq, long long n, const SearchCfgDev cfg,
                                 float thresh, int ndm, float *__restrict__ den, int32_t *__restrict__ tmin) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ndm * cfg.nw) return;
    const int d = i / cfg.nw, k = i % cfg.nw;
    const unsigned long long ss = sumsq[d];
    const double sigma = sqrt((double)ss / (double)n);
    const float dn = (float)(sigma * sqrt((double)cfg.widths[k]));
    den[i] = dn;
    int32_t T = 0x7fffffff;  // a constant row never reaches the threshold
    if (ss != 0ULL) {
        long long t = (long long)ceil((double)thresh * (double)dn);
        const long long cap = 1LL << 30;
        t = max(-cap, min(cap, t));
        while (t > -cap && (float)(t - 1) / dn >= thresh) --t;
        while (t < cap && !((float)t / dn >= thresh)) ++t;
        T = (int32_t)t;
    }
    tmin[i] = T;
}

// A CTA takes kMfTile samples of one row plus the widest boxcar's halo
// (kMfSpan samples in all), forms the exclusive prefix P in shared memory
// (each thread sums kMfSeg consecutive samples, then a block scan of the
// threads' totals), and tests its cells four at a time: a lane owns four
// consecutive cells, reads P at the cells and at the cells + w with 16-byte
// loads, and compares each boxcar sum S_w = P[t+w] - P[t] with the smallest
// sum reaching the threshold.  That exact test runs only in warps where a bound
// for a lane's four cells says that one may be hot (mf_may_be_hot4), which takes
// a third of its operations and a quarter of its words: a gulp of 1500 x 131072
// with 15 % hot cells 572 us before the bound, 462 now (1.65 GB to read and
// write, 250 us; the rest are the hot cells' S/N over 11 widths).  Hot cells get
// their best S/N and width; the four-cell nibbles of eight lanes form one word
// of the row's hot bitmask.
constexpr int kMfSpan = kMfTile + 1024;       // samples loaded per tile (tile + widest boxcar)
constexpr int kMfSeg = kMfSpan / kMfThreads;  // samples per thread in the scan
static_assert(kMfSeg % 4 == 0 && kMfSeg * kMfThreads == kMfSpan, "scan segments of whole int4s");

// a / b rounded to nearest from y = 1/b rounded to nearest (Markstein's
// correction step): q = a*y, r = a - b*q (exact with one fused multiply-add),
// q + r*y.  Correctly rounded for normal a, b and quotients away from the
// overflow and underflow ranges -- here |a| < 2^31 is an integer and b =
// sigma * sqrt(w) lies far from both.
__device__ __forceinline__ float div_rn(float a, float b, float y) {
    const float q = a * y;
    const float r = fmaf(-q, b, a);
    return fmaf(r, y, q);
}

// Hot flags of the four cells t..t+3: some searched width 2^j has
// P[t+i+2^j] - P[t+i] >= tm[j] (and, outside INSIDE tiles, t+i+2^j <= nrem).
// The widths are compile-time offsets; 1 and 2 come from the registers
// p0 = P[t..t+3], p45 = P[t+4..t+5], the others from 16-byte loads.
// ALLW: all 11 widths are searched (wmask = 0x7FF), so no width test is needed.
template <bool INSIDE, bool ALLW>
__device__ __forceinline__ void mf_test4(const int32_t *P, int t, int nrem, unsigned wmask, const int32_t (&tm)[kPows],
                                         int4 p0, int2 p45, bool &h0, bool &h1, bool &h2, bool &h3) {
    if constexpr (INSIDE) {
        // S - T >= 0 for some width <=> the AND of all S - T has its sign bit
        // clear: one add and half a 3-input AND per (cell, width) instead of a
        // compare.  |S| < 2^27 and |T| <= 2^30 (or T = INT_MAX with S = 0 on a
        // constant row), so S - T does not wrap.
        int32_t a0 = -1, a1 = -1, a2 = -1, a3 = -1;
#pragma unroll
        for (int j = 0; j < kPows; ++j) {
            if (!ALLW && !((wmask >> j) & 1u)) continue;
            int4 pw;
            if (j == 0) pw = make_int4(p0.y, p0.z, p0.w, p45.x);
            else if (j == 1) pw = make_int4(p0.z, p0.w, p45.x, p45.y);
            else pw = *reinterpret_cast<const int4 *>(P + t + (1 << j));
            const int32_t T = tm[j];
            a0 &= pw.x - p0.x - T;
            a1 &= pw.y - p0.y - T;
            a2 &= pw.z - p0.z - T;
            a3 &= pw.w - p0.w - T;
        }
        h0 = a0 >= 0;
        h1 = a1 >= 0;
        h2 = a2 >= 0;
        h3 = a3 >= 0;
    } else {
#pragma unroll
    for (int j = 0; j < kPows; ++j) {
        if (!ALLW && !((wmask >> j) & 1u)) continue;
        const int w = 1 << j;
        int4 pw;
        if (j == 0) pw = make_int4(p0.y, p0.z, p0.w, p45.x);
        else if (j == 1) pw = make_int4(p0.z, p0.w, p45.x, p45.y);
        else pw = *reinterpret_cast<const int4 *>(P + t + w);
        const int32_t T = tm[j];
        h0 |= t + w <= nrem && pw.x - p0.x >= T;
        h1 |= t + 1 + w <= nrem && pw.y - p0.y >= T;
        h2 |= t + 2 + w <= nrem && pw.z - p0.z >= T;
        h3 |= t + 3 + w <= nrem && pw.w - p0.w >= T;
    }
    }
}

// false: none of the four cells t..t+3 is hot (true: one may be).  Widths 1 and
// 2 cell by cell, from the registers; for a wider one the four sums are at most
// the largest of P[t+w..t+w+3] (p4[w / 4]) less the smallest of P[t..t+3]: one
// operation and one word for four cells, and noise hardly ever reaches T with
// it (at w = 4 the bound covers 7 samples, T is 6 sigma of 4).
template <bool ALLW>
__device__ __forceinline__ bool mf_may_be_hot4(const int32_t *p4, unsigned wmask, const int32_t (&tm)[kPows], int4 p0,
                                               int2 p45) {
    int32_t a = -1, wide = -0x7fffffff - 1;
    if (ALLW || (wmask & 1u)) {
        a &= (p0.y - p0.x - tm[0]) & (p0.z - p0.y - tm[0]);
        a &= (p0.w - p0.z - tm[0]) & (p45.x - p0.w - tm[0]);
    }
    if (ALLW || (wmask & 2u)) {
        a &= (p0.z - p0.x - tm[1]) & (p0.w - p0.y - tm[1]);
        a &= (p45.x - p0.z - tm[1]) & (p45.y - p0.w - tm[1]);
    }
#pragma unroll
    for (int j = 2; j < kPows; ++j) {
        if (!ALLW && !((wmask >> j) & 1u)) continue;
        wide = max(wide, p4[(1 << j) / 4] - tm[j]);
    }
    return a >= 0 || wide >= min(min(p0.x, p0.y), min(p0.z, p0.w));
}

template <bool ALLW>
__global__ void __launch_bounds__(kMfThreads) dd_mf_kernel(const int32_t *__restrict__ y, long long ld_y, long long n,
                                                        const unsigned long long *__restrict__ sumsq,
                                                        const SearchCfgDev cfg, float thresh,
                                                        float *__restrict__ best, uint16_t *__restrict__ bestw,
                                                        uint32_t *__restrict__ hotbits, int nwr, DevState *st,
                                                        int32_t *__restrict__ pre, long long *__restrict__ tile_sum,
                                                        int ntiles, const float *__restrict__ den_all,
                                                        const int32_t *__restrict__ tmin_all, int full_map) {
    __shared__ __align__(16) int32_t P[kMfSpan];  // exclusive prefix of the tile's samples
    __shared__ int32_t P4[kMfSpan / 4];           // largest of each four
    // per-width values indexed by log2(width)
    __shared__ float s_den[kPows];
    __shared__ float s_rcp[kPows];  // 1/den rounded to nearest
    __shared__ int32_t s_tmin[kPows];
    __shared__ int32_t s_warp[kMfThreads / 32];
    __shared__ unsigned s_nhot;
    __shared__ unsigned s_nlist;
    __shared__ uint16_t s_list[kMfTile];  // tile cells whose S/N is computed
    const int d = blockIdx.y;
    const long long t0 = (long long)blockIdx.x * kMfTile;
    const int nw = cfg.nw;
    const unsigned wmask = cfg.wmask;
    const int32_t *row = y + (long long)d * ld_y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long ss = sumsq[d];
    if (tid < kPows) {
        const bool has = (wmask >> tid) & 1u;
        const int k = __popc(wmask & ((1u << tid) - 1u));  // index of width 2^tid in the list
        const float dn = has ? den_all[d * nw + k] : 1.0f;
        s_den[tid] = dn;
        s_rcp[tid] = __frcp_rn(dn);
        s_tmin[tid] = has ? tmin_all[d * nw + k] : 0x7fffffff;
    }
    if (tid == 0) {
        s_nhot = 0;
        s_nlist = 0;
    }
    // samples of the row from t0 (0 past its end): every copy in flight at
    // once.  16-byte cp.async when the whole span lies in the row and starts
    // on a 16-byte boundary; else 4-byte ones (a copy past the end reads
    // nothing and writes 0)
    if (t0 + kMfSpan <= n && ((reinterpret_cast<uintptr_t>(row + t0) & 15u) == 0)) {
#pragma unroll
        for (int q = 0; q < kMfSeg / 4; ++q) {
            const int i = 4 * (tid + q * kMfThreads);
            const unsigned dst = (unsigned)__cvta_generic_to_shared(P + i);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(row + t0 + i) : "memory");
        }
    } else {
#pragma unroll
        for (int q = 0; q < kMfSeg; ++q) {
            const int i = tid + q * kMfThreads;
            const bool in = t0 + i < n;
            const unsigned dst = (unsigned)__cvta_generic_to_shared(P + i);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(in ? row + t0 + i : row),
                         "r"(in ? 4 : 0)
                         : "memory");
        }
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    // exclusive prefix: per-thread segment sums, then a block scan of the totals
    int4 v[kMfSeg / 4];
    int32_t tot = 0;
#pragma unroll
    for (int q = 0; q < kMfSeg / 4; ++q) {
        v[q] = *reinterpret_cast<const int4 *>(P + tid * kMfSeg + 4 * q);
        int32_t e0 = tot, e1 = e0 + v[q].x, e2 = e1 + v[q].y, e3 = e2 + v[q].z;
        tot = e3 + v[q].w;
        v[q] = make_int4(e0, e1, e2, e3);
    }
    int32_t incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int32_t off = incl - tot;
    for (int w2 = 0; w2 < warp; ++w2) off += s_warp[w2];
#pragma unroll
    for (int q = 0; q < kMfSeg / 4; ++q)
    {
        const int4 w = make_int4(v[q].x + off, v[q].y + off, v[q].z + off, v[q].w + off);
        *reinterpret_cast<int4 *>(P + tid * kMfSeg + 4 * q) = w;
        P4[tid * (kMfSeg / 4) + q] = max(max(w.x, w.y), max(w.z, w.w));
    }
    __syncthreads();

    int32_t tm[kPows];
#pragma unroll
    for (int j = 0; j < kPows; ++j) tm[j] = s_tmin[j];
    const long long nrem_l = n - t0;  // samples of the row from t0 on
    const int nrem = (int)min((long long)kMfSpan, nrem_l);
    if (tid == 0) tile_sum[(long long)d * ntiles + blockIdx.x] = P[min(kMfTile, nrem)];
    // every cell of the tile and every boxcar lie inside the row
    const bool inside = nrem_l >= (long long)kMfTile + (1 << (31 - __clz(wmask)));
    const long long cbase = (long long)d * n + t0;
#pragma unroll 1
    for (int j = 0; j < kMfTile / (32 * 4 * (kMfThreads / 32)); ++j) {
        const int t = warp * (kMfTile / (kMfThreads / 32)) + j * 128 + lane * 4;  // first of this lane's 4 cells
        const int4 p0 = *reinterpret_cast<const int4 *>(P + t);
        const int2 p45 = *reinterpret_cast<const int2 *>(P + t + 4);
        if (t + 3 < nrem && ((cbase + t) & 3) == 0) {
            *reinterpret_cast<int4 *>(pre + cbase + t) = p0;  // pre comes from cudaMalloc: 16-byte aligned rows of 4
        } else {
            const int32_t pc[4] = {p0.x, p0.y, p0.z, p0.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (t + i < nrem) pre[cbase + t + i] = pc[i];
        }
        const long long tw = t0 + t;  // first cell of the word for lanes 0, 8, 16, 24
        if (!full_map && !__any_sync(0xffffffffu, mf_may_be_hot4<ALLW>(P4 + t / 4, wmask, tm, p0, p45))) {
            if ((lane & 7) == 0 && tw < n) hotbits[(long long)d * nwr + tw / 32] = 0u;
            continue;
        }
        bool h0 = false, h1 = false, h2 = false, h3 = false;
        if (inside)
            mf_test4<true, ALLW>(P, t, nrem, wmask, tm, p0, p45, h0, h1, h2, h3);
        else
            mf_test4<false, ALLW>(P, t, nrem, wmask, tm, p0, p45, h0, h1, h2, h3);
        const bool hc[4] = {h0, h1, h2, h3};
        uint32_t nib = 0, live = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool lv = t + i < nrem;
            live |= (uint32_t)lv << i;
            nib |= (uint32_t)(lv && hc[i]) << i;
        }
        // cells whose S/N is computed (hot ones, or all with full_map) join
        // the tile's list, warp by warp in cell order
        const uint32_t want = full_map ? live : nib;
        if (__any_sync(0xffffffffu, want != 0u)) {
            const int cnt = __popc(want);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            unsigned wbase = 0;
            if (lane == 31) wbase = atomicAdd(&s_nlist, (unsigned)incl);
            unsigned pos = __shfl_sync(0xffffffffu, wbase, 31) + (unsigned)(incl - cnt);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if ((want >> i) & 1u) s_list[pos++] = (uint16_t)(t + i);
        }
        // eight lanes' nibbles make one 32-cell word of the hot bitmask
        uint32_t word = nib << (4 * (lane & 7));
        word |= __shfl_xor_sync(0xffffffffu, word, 1);
        word |= __shfl_xor_sync(0xffffffffu, word, 2);
        word |= __shfl_xor_sync(0xffffffffu, word, 4);
        if ((lane & 7) == 0 && tw < n) {
            hotbits[(long long)d * nwr + tw / 32] = word;
            if (word) atomicAdd(&s_nhot, (unsigned)__popc(word));
        }
    }
    __syncthreads();
    if (tid == 0 && s_nhot) atomicAdd(&st->nhot, (unsigned long long)s_nhot);
    // best S/N and width of the listed cells, one cell per thread.  Listed
    // hot cells skip the widths whose sum stays below the threshold sum: their
    // S/N is below the threshold, so below the cell's best (ties included);
    // the full map computes every width
    const unsigned nl = s_nlist;
#pragma unroll 1
    for (unsigned e = tid; e < nl; e += kMfThreads) {
        const int c = s_list[e];
        float bs = 0.0f;
        int bw = 0;
        const int32_t pi = P[c];
#pragma unroll
        for (int j = 0; j < kPows; ++j) {
            const int32_t S = P[c + (1 << j)] - pi;  // inside the staged span: c + 2^j < 4096 + 1024
            if ((ALLW || ((wmask >> j) & 1u)) && c + (1 << j) <= nrem && (full_map || S >= tm[j])) {
                const float snr = ss == 0 ? 0.0f : div_rn((float)S, s_den[j], s_rcp[j]);
                if (bw == 0 || snr > bs) {
                    bs = snr;
                    bw = 1 << j;
                }
            }
        }
        best[cbase + c] = bw ? bs : -INFINITY;  // no width fits before the row end
        bestw[cbase + c] = (uint16_t)bw;
    }
}

// Per row, exclusive prefix of the tile totals: tile_off[d][i] = sum of tiles < i.
__global__ void dd_tile_scan_kernel(const long long *__restrict__ tile_sum, long long *__restrict__ tile_off, int ndm,
                                 int ntiles) {
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= ndm) return;
    long long acc = 0;
    for (int i = 0; i < ntiles; ++i) {
        tile_off[(long long)d * ntiles + i] = acc;
        acc += tile_sum[(long long)d * ntiles + i];
    }
}

// ---------------------------------------------------------------------------
// grouping: runs of hot cells along time, joined across DM rows
// ---------------------------------------------------------------------------

// hotbits holds, per row, ceil(n/32) words: bit t%32 of word t/32 is set when
// cell (d, t) is hot.  A run is a maximal interval of hot cells in one row and
// its start is the cell where it begins.  The run start of any hot cell
// follows from its word and wl, the last run start before each word: the
// highest run-start bit at or below the cell's bit, else wl of the word.  The
// run starts form a union-find forest in L (entries at run starts only) whose
// roots are the smallest start of each group (deterministic), linked with
// atomicMin.  Two runs in neighbouring rows touch exactly when their
// intervals overlap, and the first column of an overlap is the start of one
// of the two runs, so the rows are joined by visiting only the vertically
// adjacent hot cells that are a run start in either row.
__device__ __forceinline__ uint32_t run_starts(uint32_t m, uint32_t prev_word) {
    return m & ~((m << 1) | (prev_word >> 31));
}

// Run start (cell index) of hot bit b of a word with run-start bits s whose
// bit 0 is cell cw; wl_w = the last run start before the word.
__device__ __forceinline__ int32_t run_start_of(uint32_t s, int b, long long cw, int32_t wl_w) {
    const uint32_t m = s & ((2u << b) - 1u);  // run starts at or below b (b = 31: all)
    return m ? (int32_t)(cw + 31 - __clz(m)) : wl_w;
}

// Per word of row blockIdx.x, the last run start before it (wl), and every
// run start as its own union-find node.  Warp k of the block owns a
// contiguous range of the row's words and walks it 32 words at a time (lane =
// word, coalesced): pass 1 finds the last run start of each range, a scan over
// the warps gives each range the last start before it, and pass 2 writes wl
// from a running max carried across the warp's steps.
__global__ void __launch_bounds__(512) dd_runs_kernel(const uint32_t *__restrict__ hotbits, int nwr, long long n,
                                                      int32_t *__restrict__ L, int32_t *__restrict__ wl) {
    __shared__ int s_warp[16];
    const int d = blockIdx.x;
    const uint32_t *hb = hotbits + (long long)d * nwr;
    const long long cbase = (long long)d * n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (nwr + 16 * 32 - 1) / (16 * 32) * 32;  // words per warp, whole steps of 32
    const int w0 = min(nwr, warp * per), w1 = min(nwr, w0 + per);
    // pass 1: last run start (time index) in the warp's range
    int last = -1;
    for (int wb = w0; wb < w1; wb += 32) {
        const int w = wb + lane;
        if (w < w1) {
            const uint32_t s = run_starts(hb[w], w > 0 ? hb[w - 1] : 0u);
            if (s) last = 32 * w + 31 - __clz(s);
        }
    }
    last = __reduce_max_sync(0xffffffffu, last + 1) - 1;  // as unsigned: -1 -> 0
    if (lane == 0) s_warp[warp] = last;
    __syncthreads();
    int carry = -1;
    for (int k = 0; k < warp; ++k) carry = max(carry, s_warp[k]);
    // pass 2
    int32_t *wrow = wl + (long long)d * nwr;
    for (int wb = w0; wb < w1; wb += 32) {
        const int w = wb + lane;
        uint32_t s = 0;
        if (w < w1) s = run_starts(hb[w], w > 0 ? hb[w - 1] : 0u);
        const int lw = s ? 32 * w + 31 - __clz(s) : -1;
        int incl = lw;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl = max(incl, u);
        }
        int before = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) before = -1;
        if (w < w1) {
            wrow[w] = (int32_t)(cbase + max(carry, before));  // meaningful when bit 0 continues a run
            for (uint32_t q = s; q; q &= q - 1) {
                const int32_t c = (int32_t)(cbase + 32 * w + __ffs(q) - 1);
                L[c] = c;
            }
        }
        carry = max(carry, __shfl_sync(0xffffffffu, incl, 31));
    }
}

// find with path halving: each visited node is pointed at its grandparent.
// Labels only ever move to smaller indices of the same group, so a plain
// store of an ancestor is safe against concurrent links (a linker that loses
// its update sees the changed parent and retries).
__device__ __forceinline__ int32_t find_halving(int32_t *L, int32_t x) {
    int32_t p = __ldcg(L + x);
    while (p != x) {
        const int32_t gp = __ldcg(L + p);
        if (gp != p) __stcg(L + x, gp);
        x = gp;
        p = __ldcg(L + x);
    }
    return x;
}

__device__ void unite(int32_t *L, int32_t a, int32_t b, DevState *st) {
    for (unsigned it = 0; it < kUnionCap; ++it) {
        a = find_halving(L, a);
        b = find_halving(L, b);
        if (a == b) return;
        if (a < b) {
            const int32_t t = a;
            a = b;
            b = t;
        }
        // link the larger root a under b
        const int32_t old = atomicMin(L + a, b);
        if (old == a) return;
        a = old;
    }
    atomicOr(&st->err, 4u);
}

// Join runs of rows d-1 and d that overlap, at the first column of each overlap.
__global__ void dd_vunion_kernel(const uint32_t *__restrict__ hotbits, int nwr, int ndm, long long n, int32_t *L,
                                 const int32_t *__restrict__ wl, DevState *st) {
    // rows on y, words on x: no index division
    for (int d = 1 + blockIdx.y; d < ndm; d += gridDim.y) {
        const uint32_t *h2 = hotbits + (long long)d * nwr, *h1 = h2 - nwr;
        const int32_t *wl2 = wl + (long long)d * nwr, *wl1 = wl2 - nwr;
        for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < nwr; w += gridDim.x * blockDim.x) {
            const uint32_t a2 = h2[w], a1 = h1[w];
            const uint32_t v = a1 & a2;
            if (!v) continue;
            const uint32_t s2 = run_starts(a2, w > 0 ? h2[w - 1] : 0u);
            const uint32_t s1 = run_starts(a1, w > 0 ? h1[w - 1] : 0u);
            const long long cw2 = (long long)d * n + 32LL * w;
            for (uint32_t q = v & (s1 | s2); q; q &= q - 1) {
                const int b = __ffs(q) - 1;
                const int32_t a = run_start_of(s2, b, cw2, wl2[w]);
                const int32_t e = run_start_of(s1, b, cw2 - n, wl1[w]);
                unite(L, a, e, st);
            }
        }
    }
}

// Every run start points straight at its root; roots get compact ids, stored in
// place as -(id + 2), where a search that meets one ends (two passes over the
// bitmask, one for the roots and one for the ids, took 56 us for 1500 x 131072,
// this one 31).
__global__ void dd_compress_kernel(const uint32_t *__restrict__ hotbits, int nwr, int ndm, long long n, int32_t *L,
                                   DevState *st) {
    for (int d = blockIdx.y; d < ndm; d += gridDim.y) {
        const uint32_t *h = hotbits + (long long)d * nwr;
        for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < nwr; w += gridDim.x * blockDim.x) {
            for (uint32_t q = run_starts(h[w], w > 0 ? h[w - 1] : 0u); q; q &= q - 1) {
                const int32_t c = (int32_t)((long long)d * n + 32 * w + __ffs(q) - 1);
                int32_t x = c, p = __ldcg(L + x);
                while (p != x && p >= 0) {
                    x = p;
                    p = __ldcg(L + x);
                }
                L[c] = x != c ? x : -2 - (int32_t)atomicAdd(&st->nroots, 1u);
            }
        }
    }
}

// Group id of a run start: start -> root (one hop after compression).
__device__ __forceinline__ int group_id(const int32_t *L, int32_t start) {
    int32_t v = L[start];
    for (int hop = 0; hop < 1 && v >= 0; ++hop) v = L[v];
    return v <= -2 ? -2 - v : -1;
}

// Per group: the largest (S/N, -cell) key and the number of cells.  A lane
// takes one word; each stretch of consecutive hot bits lies in one run and
// gives one record, and the warp combines records of the same group before
// its atomics.  The stretches' S/N values are read by the whole warp, a stretch
// at a time (four on their way): lane by lane, each its own line of 32 values,
// 3e7 hot cells of 1500 x 131072 took 144 us, now 134, bound by the chain of
// loads from a run start to its group.  (A lane that goes down 4 or 16 rows and
// hands records on when the group changes: 133 and 159 us.)
__global__ void dd_group_reduce_kernel(const uint32_t *__restrict__ hotbits, int nwr, int ndm, long long n,
                                       const int32_t *__restrict__ L, const int32_t *__restrict__ wl,
                                       const float *__restrict__ best, int max_cands,
                                       unsigned long long *__restrict__ key, long long *__restrict__ cnt) {
    const int lane = threadIdx.x & 31;
    // rows on y; a warp takes 32 consecutive words of one row
    for (int d = blockIdx.y; d < ndm; d += gridDim.y)
    for (int w0 = blockIdx.x * blockDim.x + (int)(threadIdx.x & ~31u); w0 < nwr; w0 += gridDim.x * blockDim.x) {
        const int w = w0 + lane;
        const long long k = (long long)d * nwr + w;
        uint32_t q = 0, sq = 0;  // hot bits, run-start bits
        const long long cw = (long long)d * n + 32LL * w;  // cell index of bit 0 of this word
        int32_t wlk = 0;
        if (w < nwr) {
            q = hotbits[k];
            if (q) {
                sq = run_starts(q, w > 0 ? hotbits[k - 1] : 0u);
                wlk = wl[k];
            }
        }
        while (__any_sync(0xffffffffu, q != 0u)) {
            int id = -1;
            unsigned long long kv = 0;
            unsigned cntv = 0;
            int32_t c0 = 0;
            unsigned todo = __ballot_sync(0xffffffffu, q != 0u);
            if (q) {
                const int b0 = __ffs(q) - 1;
                const uint32_t rest = ~(q >> b0);
                const int len = rest ? __ffs(rest) - 1 : 32 - b0;
                q = len >= 32 - b0 ? 0u : q & ~(((1u << len) - 1u) << b0);
                c0 = (int32_t)(cw + b0);
                id = group_id(L, ((sq >> b0) & 1u) ? c0 : wlk);  // a stretch not at a run start begins at bit 0
                if (id >= max_cands) id = -1;
                cntv = (unsigned)len;
            }
            while (todo) {
                constexpr int kAhead = 4;
                uint32_t v[kAhead];
                int src[kAhead];
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    src[u] = todo ? __ffs(todo) - 1 : -1;
                    todo &= todo - 1;
                    const int32_t first = __shfl_sync(0xffffffffu, c0, src[u] & 31);
                    const unsigned cells = __shfl_sync(0xffffffffu, cntv, src[u] & 31);
                    v[u] = src[u] >= 0 && (unsigned)lane < cells ? __float_as_uint(best[(uint32_t)first + lane]) : 0u;
                }
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    // largest S/N (positive: ordered as its bits) first, then the
                    // smallest cell index (lower DM, then earlier time)
                    const uint32_t top = __reduce_max_sync(0xffffffffu, v[u]);
                    const int at = __ffs(__ballot_sync(0xffffffffu, v[u] == top)) - 1;
                    if (lane == src[u]) kv = ((unsigned long long)top << 32) | (0xFFFFFFFFu - (uint32_t)(c0 + at));
                }
            }
            const unsigned peers = __match_any_sync(0xffffffffu, id);
            unsigned long long m = kv;
            unsigned long long tot = 0;
            for (unsigned p = peers; p; p &= p - 1) {
                const int src = __ffs(p) - 1;
                const unsigned long long v = __shfl_sync(peers, kv, src);
                tot += __shfl_sync(peers, cntv, src);
                m = v > m ? v : m;
            }
            if (id >= 0 && lane == __ffs(peers) - 1) {
                atomicMax(key + id, m);
                atomicAdd(reinterpret_cast<unsigned long long *>(cnt + id), tot);
            }
        }
    }
}

// Mark each group's representative cell in a bitmask, and store its group id
// in the (no longer needed) label array.
__global__ void dd_mark_kernel(const unsigned long long *__restrict__ key, int32_t *__restrict__ L,
                               unsigned *__restrict__ marks, const DevState *st, int max_cands) {
    const int nr = (int)min((unsigned)max_cands, st->nroots);
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < nr; id += gridDim.x * blockDim.x) {
        const uint32_t c = 0xFFFFFFFFu - (uint32_t)(key[id] & 0xFFFFFFFFu);
        L[c] = id;
        atomicOr(marks + (c >> 5), 1u << (c & 31));
    }
}

// Ordered compaction of the marked cells (cell order = (DM, time) order):
// per-chunk counts, an exclusive scan over chunks, then an ordered write.  A
// thread owns kCompactWords consecutive words of a chunk.
constexpr int kCompactWords = kCompactChunk / 32 / kCompactThreads;
static_assert(kCompactWords * 32 * kCompactThreads == kCompactChunk, "chunk = threads x words x 32");

__global__ void __launch_bounds__(kCompactThreads) dd_count_marks_kernel(const unsigned *__restrict__ marks,
                                                                         long long nwords,
                                                                         unsigned *__restrict__ chunk_count) {
    __shared__ unsigned s_cnt;
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    const long long w0 = (long long)blockIdx.x * (kCompactChunk / 32) + threadIdx.x * kCompactWords;
    unsigned mine = 0;
#pragma unroll
    for (int i = 0; i < kCompactWords; ++i)
        if (w0 + i < nwords) mine += __popc(marks[w0 + i]);
    if (mine) atomicAdd(&s_cnt, mine);
    __syncthreads();
    if (threadIdx.x == 0) chunk_count[blockIdx.x] = s_cnt;
}

// Exclusive scan of the chunk counts in place, by one CTA, 1024 at a time with
// two barriers each (256 at a time with 16 barriers: 12 us for 3000 chunks).
constexpr int kScanThreads = 1024;
__global__ void __launch_bounds__(kScanThreads) dd_scan_chunks_kernel(unsigned *__restrict__ chunk_count, int nchunks) {
    __shared__ unsigned s_warp[2][kScanThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto warp_scan = [&](unsigned v) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        return v;
    };
    unsigned carry = 0;
    int buf = 0;
    for (int base = 0; base < nchunks; base += kScanThreads) {
        const int i = base + (int)threadIdx.x;
        const unsigned v = i < nchunks ? chunk_count[i] : 0u;
        const unsigned incl = warp_scan(v);
        if (lane == 31) s_warp[buf][warp] = incl;
        __syncthreads();
        // every warp scans the warps' totals; the other buffer is the next round's
        const unsigned totals = warp_scan(s_warp[buf][lane]);
        const unsigned before = __shfl_sync(0xffffffffu, totals, (warp + 31) & 31);
        if (i < nchunks) chunk_count[i] = carry + (warp ? before : 0u) + incl - v;
        carry += __shfl_sync(0xffffffffu, totals, 31);
        buf ^= 1;
    }
}

__global__ void __launch_bounds__(kCompactThreads) dd_write_marks_kernel(
    const unsigned *__restrict__ marks, long long nwords, const uint16_t *__restrict__ bestw,
    const float *__restrict__ best, const int32_t *__restrict__ L, const long long *__restrict__ cnt, long long n,
    int beam, const unsigned *__restrict__ chunk_off, int max_cands, dd_candidate *__restrict__ out) {
    __shared__ unsigned s_warp[kCompactThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long w0 = (long long)blockIdx.x * (kCompactChunk / 32) + threadIdx.x * kCompactWords;
    uint32_t mw[kCompactWords];
    unsigned mine = 0;
#pragma unroll
    for (int i = 0; i < kCompactWords; ++i) {
        mw[i] = w0 + i < nwords ? marks[w0 + i] : 0u;
        mine += __popc(mw[i]);
    }
    // exclusive scan of the threads' counts (thread order = cell order)
    unsigned incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    unsigned pos = chunk_off[blockIdx.x] + incl - mine;
    for (int k = 0; k < warp; ++k) pos += s_warp[k];
#pragma unroll
    for (int i = 0; i < kCompactWords; ++i) {
        for (uint32_t q = mw[i]; q; q &= q - 1) {
            const long long c = (w0 + i) * 32 + __ffs(q) - 1;
            if (pos < (unsigned)max_cands) {
                dd_candidate o;
                o.beam = beam;
                o.d = (int32_t)(c / n);
                o.t = (int32_t)(c % n);
                o.w = bestw[c];
                o.snr = best[c];
                o.score = 0.0f;
                o.ncells = cnt[L[c]];
                out[pos] = o;
            }
            ++pos;
        }
    }
}

// ---------------------------------------------------------------------------
// snippets
// ---------------------------------------------------------------------------

// Row prefix P(t) = sum of y[0..t) from the tile-local prefixes and the tile offsets.
__device__ __forceinline__ long long row_prefix(const int32_t *pre_row, const long long *off_row,
                                                const long long *sum_row, long long n, int ntiles, long long t) {
    if (t <= 0) return 0;
    if (t >= n) return off_row[ntiles - 1] + sum_row[ntiles - 1];
    return off_row[t / kMfTile] + (long long)pre_row[t];
}

__global__ void __launch_bounds__(256) dd_snippet_kernel(const int32_t *__restrict__ pre,
                                                      const long long *__restrict__ tile_off,
                                                      const long long *__restrict__ tile_sum, int ntiles, int ndm,
                                                      long long n, const unsigned long long *__restrict__ sumsq,
                                                      const dd_candidate *__restrict__ cands,
                                                      __nv_bfloat16 *__restrict__ out) {
    __shared__ float s_den[64];  // per snippet row: float(sigma * sqrt(w)), 0 for no data
    const dd_candidate cd = cands[blockIdx.x];
    const int w = cd.w;
    if (threadIdx.x < 64) {
        const int dd = cd.d - 32 + threadIdx.x;
        float den = 0.0f;
        if (dd >= 0 && dd < ndm && sumsq[dd] != 0ULL)
            den = (float)(sqrt((double)sumsq[dd] / (double)n) * sqrt((double)w));
        s_den[threadIdx.x] = den;
    }
    __syncthreads();
    __nv_bfloat16 *o = out + (long long)blockIdx.x * 64 * 64;
    const int lane = threadIdx.x & 31;
    // a warp takes 32 consecutive bins of one row: each lane looks up the
    // prefix at its bin's start and takes its end from the next lane (four
    // rows' lookups in flight at once)
#pragma unroll 4
    for (int i = threadIdx.x; i < 64 * 64; i += blockDim.x) {
        const int r = i >> 6, b = i & 63;
        const int dd = cd.d - 32 + r;
        const float den = s_den[r];  // the same for the whole warp
        float v = 0.0f;
        if (den != 0.0f) {
            const long long s0 = (long long)cd.t + (long long)(b - 32) * w;
            const int32_t *pr = pre + (long long)dd * n;
            const long long *orow = tile_off + (long long)dd * ntiles, *srow = tile_sum + (long long)dd * ntiles;
            const long long p0 = row_prefix(pr, orow, srow, n, ntiles, s0);
            long long p1 = __shfl_down_sync(0xffffffffu, p0, 1);
            if (lane == 31) p1 = row_prefix(pr, orow, srow, n, ntiles, s0 + w);
            v = (float)(p1 - p0) / den;
        }
        o[i] = __float2bfloat16_rn(v);
    }
}

// Snippets straight from y (dd_snippets with caller buffers): each bin sums
// its w samples with warp shuffles.
__global__ void __launch_bounds__(256) dd_snippet_from_y_kernel(const int32_t *__restrict__ y, long long ld_y, int ndm,
                                                      long long n, const unsigned long long *__restrict__ sumsq,
                                                      const dd_candidate *__restrict__ cands,
                                                      __nv_bfloat16 *__restrict__ out) {
    const dd_candidate cd = cands[blockIdx.x];
    const int w = cd.w;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __nv_bfloat16 *o = out + (long long)blockIdx.x * 64 * 64;
    for (int r = warp; r < 64; r += 8) {
        const int dd = cd.d - 32 + r;
        const bool live = dd >= 0 && dd < ndm && sumsq[dd] != 0ULL;
        float den = 1.0f;
        if (live) den = (float)(sqrt((double)sumsq[dd] / (double)n) * sqrt((double)w));
        const int32_t *row = y + (long long)(live ? dd : 0) * ld_y;
        const long long base = (long long)cd.t - 32LL * w;
        // 64 bins of w samples cover [base, base + 64w): read it 32 samples at a time
        long long bin_acc = 0;  // lane 0 keeps the running bin sum when w >= 32
        for (long long s = 0; s < 64LL * w; s += 32) {
            const long long t = base + s + lane;
            long long v = (live && t >= 0 && t < n) ? (long long)row[t] : 0;
            if (w >= 32) {
#pragma unroll
                for (int o2 = 16; o2 > 0; o2 >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o2);
                bin_acc += v;
                if (((s + 32) % w) == 0) {
                    if (lane == 0) {
                        const int b = (int)(s / w);
                        o[r * 64 + b] = __float2bfloat16_rn(live ? (float)bin_acc / den : 0.0f);
                    }
                    bin_acc = 0;
                }
            } else {
                for (int o2 = 1; o2 < w; o2 <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o2);
                if ((lane % w) == 0) {
                    const int b = (int)((s + lane) / w);
                    o[r * 64 + b] = __float2bfloat16_rn(live ? (float)v / den : 0.0f);
                }
            }
        }
    }
}


}  // namespace

struct Search {
    dd_search_config cfg;
    SearchCfgDev dcfg;
    int nbins = 0;
    int sms = 0;
    int32_t *y = nullptr;
    unsigned long long *sumsq = nullptr;
    float *best = nullptr;
    uint16_t *bestw = nullptr;
    int32_t *labels = nullptr;    // union-find forest (entries at run starts only)
    int32_t *wl = nullptr;        // [ndm][ceil(n/32)] last run start before each word
    uint32_t *hotbits = nullptr;  // [ndm][ceil(n/32)] hot-cell bitmask
    unsigned long long *key = nullptr;
    long long *cnt = nullptr;
    dd_candidate *cands = nullptr;
    unsigned *chunk = nullptr;  // per-chunk counts / offsets for the ordered compaction
    int32_t *pre = nullptr;       // tile-local exclusive prefix of y
    unsigned *marks = nullptr;    // representative-cell bitmask
    float *den = nullptr;         // [ndm][nw] S/N denominators
    int32_t *tmin = nullptr;      // [ndm][nw] smallest boxcar sum reaching thresh
    long long *tile_sum = nullptr, *tile_off = nullptr;
    int ntiles = 0;
    size_t nchunks_cap = 0;
    DevState *st = nullptr;
    // last run
    int ndm = 0;
    long long n = 0;
    long long ld_y = 0;
};

static void free_search(Search *s) {
    if (!s) return;
    cudaFree(s->y);
    cudaFree(s->sumsq);
    cudaFree(s->best);
    cudaFree(s->bestw);
    cudaFree(s->labels);
    cudaFree(s->wl);
    cudaFree(s->hotbits);
    cudaFree(s->key);
    cudaFree(s->cnt);
    cudaFree(s->chunk);
    cudaFree(s->pre);
    cudaFree(s->marks);
    cudaFree(s->den);
    cudaFree(s->tmin);
    cudaFree(s->tile_sum);
    cudaFree(s->tile_off);
    cudaFree(s->cands);
    cudaFree(s->st);
    delete s;
}

}  // namespace dd

using namespace dd;

extern "C" {

dd_status dd_search_create(dd_search **out, const dd_search_config *cfg) {
    if (!out || !cfg) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    *out = nullptr;
    const dd_search_config &c = *cfg;
    if (c.ndm_max <= 0 || c.n_max == 0 || c.nchan <= 0 || c.nchan > 21844 || c.half_window <= 0 || c.half_window > 32767 || c.nwidths <= 0 ||
        c.nwidths > kMaxWidths || !(c.thresh > 0) || c.max_cands <= 0 || c.max_cands > DD_SEARCH_MAX_CANDS ||
        c.baseline < 0 || c.baseline > 1)
        return fail(DD_ERR_INVALID_ARG, "bad search configuration");
    if ((double)c.ndm_max * (double)c.n_max >= 2147483647.0)
        return fail(DD_ERR_INVALID_ARG, "ndm_max * n_max must stay below 2^31 (cell indices are int32)");
    for (int k = 0; k < c.nwidths; ++k) {
        const int w = c.widths[k];
        if (w <= 0 || w > 1024 || (w & (w - 1)) || (k > 0 && w <= c.widths[k - 1]))
            return fail(DD_ERR_INVALID_ARG, "widths must be ascending powers of two <= 1024");
    }
    Search *s = new (std::nothrow) Search();
    if (!s) return fail(DD_ERR_NOMEM, "host allocation failed");
    s->cfg = c;
    s->dcfg.nw = c.nwidths;
    for (int k = 0; k < kMaxWidths; ++k) s->dcfg.widths[k] = k < c.nwidths ? c.widths[k] : 0;
    s->dcfg.wmask = 0;
    for (int k = 0; k < c.nwidths; ++k) s->dcfg.wmask |= (unsigned)c.widths[k];
    s->nbins = 3 * c.nchan + 1;
    const size_t cells = (size_t)c.ndm_max * c.n_max;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMalloc(&s->y, cells * 4);
    if (e == cudaSuccess) e = cudaMalloc(&s->sumsq, (size_t)c.ndm_max * 8);
    if (e == cudaSuccess) e = cudaMalloc(&s->best, cells * 4);
    if (e == cudaSuccess) e = cudaMalloc(&s->bestw, cells * 2);
    if (e == cudaSuccess) e = cudaMalloc(&s->labels, cells * 4);
    if (e == cudaSuccess) e = cudaMalloc(&s->hotbits, (size_t)c.ndm_max * ((c.n_max + 31) / 32) * 4);
    if (e == cudaSuccess) e = cudaMalloc(&s->wl, (size_t)c.ndm_max * ((c.n_max + 31) / 32) * 4);
    if (e == cudaSuccess) e = cudaMalloc(&s->key, (size_t)c.max_cands * 8);
    if (e == cudaSuccess) e = cudaMalloc(&s->cnt, (size_t)c.max_cands * 8);
    if (e == cudaSuccess) e = cudaMalloc(&s->cands, (size_t)c.max_cands * sizeof(dd_candidate));
    s->nchunks_cap = (cells + kCompactChunk - 1) / kCompactChunk;
    if (e == cudaSuccess) e = cudaMalloc(&s->chunk, s->nchunks_cap * sizeof(unsigned));
    const size_t tiles_cap = (size_t)c.ndm_max * ((c.n_max + kMfTile - 1) / kMfTile);
    if (e == cudaSuccess) e = cudaMalloc(&s->pre, cells * 4);
    if (e == cudaSuccess) e = cudaMalloc(&s->marks, (cells + 31) / 32 * 4);
    if (e == cudaSuccess) e = cudaMalloc(&s->den, (size_t)c.ndm_max * kMaxWidths * 4);
    if (e == cudaSuccess) e = cudaMalloc(&s->tmin, (size_t)c.ndm_max * kMaxWidths * 4);
    if (e == cudaSuccess) e = cudaMalloc(&s->tile_sum, tiles_cap * 8);
    if (e == cudaSuccess) e = cudaMalloc(&s->tile_off, tiles_cap * 8);
    if (e == cudaSuccess) e = cudaMalloc(&s->st, sizeof(DevState));
    if (e == cudaSuccess) e = cudaMemset(s->st, 0, sizeof(DevState));
    if (e != cudaSuccess) {
        dd_status st = cuda_fail(e, "allocating search buffers");
        free_search(s);
        return st;
    }
    *out = reinterpret_cast<dd_search *>(s);
    return DD_OK;
}

dd_status dd_search_run(dd_search *search, const uint32_t *d_x, size_t ld_x, int ndm, size_t n, int beam,
                        void *stream) {
    Search *s = reinterpret_cast<Search *>(search);
    if (!s || !d_x) return fail(DD_ERR_INVALID_ARG, "NULL search or input");
    if (ndm <= 0 || ndm > s->cfg.ndm_max || n == 0 || n > s->cfg.n_max || ld_x < n)
        return fail(DD_ERR_INVALID_ARG, "ndm/n beyond the search capacity or ld_x < n");
    cudaStream_t st = (cudaStream_t)stream;
    s->ndm = ndm;
    s->n = (long long)n;
    s->ld_y = (long long)n;
    DD_CUDA_TRY(cudaMemsetAsync(s->sumsq, 0, (size_t)ndm * 8, st));
    DD_CUDA_TRY(cudaMemsetAsync(s->st, 0, sizeof(DevState), st));
    DD_CUDA_TRY(cudaMemsetAsync(s->key, 0, (size_t)s->cfg.max_cands * 8, st));
    DD_CUDA_TRY(cudaMemsetAsync(s->cnt, 0, (size_t)s->cfg.max_cands * 8, st));
    // baseline
    const long long h = s->cfg.half_window;
    s->ntiles = (int)((n + kMfTile - 1) / kMfTile);
    if (s->cfg.baseline == 1) {
        const unsigned seg = row_segment(s->sms, ndm, (long long)n, 0.1 * (double)h);
        const unsigned nseg = (unsigned)(((long long)n + seg - 1) / seg);
        dd_mean_kernel<<<(unsigned)(((long long)ndm * nseg + kMwWarps - 1) / kMwWarps), 32 * kMwWarps, 0, st>>>(
            d_x, (long long)ld_x, ndm, (unsigned)n, (unsigned)h, seg, nseg, (uint32_t)(s->nbins - 1), s->y, s->ld_y,
            s->sumsq, s->st);
    } else {
        const unsigned seg = row_segment(s->sms, ndm, (long long)n, 0.3 * (double)h);
        const unsigned nseg = (unsigned)(((long long)n + seg - 1) / seg);
        dd_median_kernel<<<(unsigned)(((long long)ndm * nseg + kMwWarps - 1) / kMwWarps), 32 * kMwWarps, 0, st>>>(
            d_x, (long long)ld_x, ndm, (unsigned)n, (unsigned)h, seg, nseg, (uint32_t)(s->nbins - 1), s->y, s->ld_y,
            s->sumsq, s->st);
    }
    DD_CUDA_TRY(cudaGetLastError());
    // matched filter + sigma cut
    dim3 fg((unsigned)((n + kMfTile - 1) / kMfTile), (unsigned)ndm);
    s->ntiles = (int)((n + kMfTile - 1) / kMfTile);
    dd_thresh_kernel<<<(ndm * s->cfg.nwidths + 127) / 128, 128, 0, st>>>(s->sumsq, (long long)n, s->dcfg,
                                                                        s->cfg.thresh, ndm, s->den, s->tmin);
    const int nwr = (int)((n + 31) / 32);
    if (s->dcfg.wmask == (1u << kPows) - 1u)
        dd_mf_kernel<true><<<fg, kMfThreads, 0, st>>>(s->y, s->ld_y, (long long)n, s->sumsq, s->dcfg, s->cfg.thresh, s->best,
                                             s->bestw, s->hotbits, nwr, s->st, s->pre, s->tile_sum, s->ntiles, s->den,
                                             s->tmin, s->cfg.full_map);
    else
        dd_mf_kernel<false><<<fg, kMfThreads, 0, st>>>(s->y, s->ld_y, (long long)n, s->sumsq, s->dcfg, s->cfg.thresh, s->best,
                                             s->bestw, s->hotbits, nwr, s->st, s->pre, s->tile_sum, s->ntiles, s->den,
                                             s->tmin, s->cfg.full_map);
    DD_CUDA_TRY(cudaGetLastError());
    dd_tile_scan_kernel<<<(ndm + 127) / 128, 128, 0, st>>>(s->tile_sum, s->tile_off, ndm, s->ntiles);
    // grouping
    const int g = s->sms * 8;
    const long long cells = (long long)ndm * (long long)n;
    dd_runs_kernel<<<ndm, 512, 0, st>>>(s->hotbits, nwr, (long long)n, s->labels, s->wl);
    // word kernels: words of a row on x, rows on y
    const dim3 gw((unsigned)std::min((nwr + 255) / 256, 64), (unsigned)std::min(ndm, 4096));
    dd_vunion_kernel<<<gw, 256, 0, st>>>(s->hotbits, nwr, ndm, (long long)n, s->labels, s->wl, s->st);
    dd_compress_kernel<<<gw, 256, 0, st>>>(s->hotbits, nwr, ndm, (long long)n, s->labels, s->st);
    dd_group_reduce_kernel<<<gw, 256, 0, st>>>(s->hotbits, nwr, ndm, (long long)n, s->labels, s->wl, s->best,
                                              s->cfg.max_cands, s->key, s->cnt);
    const long long nwords = (cells + 31) / 32;
    DD_CUDA_TRY(cudaMemsetAsync(s->marks, 0, (size_t)nwords * 4, st));
    dd_mark_kernel<<<g, 256, 0, st>>>(s->key, s->labels, s->marks, s->st, s->cfg.max_cands);
    const int nchunks = (int)((cells + kCompactChunk - 1) / kCompactChunk);
    dd_count_marks_kernel<<<nchunks, kCompactThreads, 0, st>>>(s->marks, nwords, s->chunk);
    dd_scan_chunks_kernel<<<1, kScanThreads, 0, st>>>(s->chunk, nchunks);
    dd_write_marks_kernel<<<nchunks, kCompactThreads, 0, st>>>(s->marks, nwords, s->bestw, s->best, s->labels, s->cnt,
                                                               (long long)n, beam, s->chunk, s->cfg.max_cands,
                                                               s->cands);
    return cuda_fail(cudaGetLastError(), "search kernels");
}

}  // extern "C"

namespace dd {
const unsigned *search_dev_ngroups(const dd_search *search) {
    return &reinterpret_cast<const Search *>(search)->st->nroots;
}
}  // namespace dd

extern "C" {

dd_status dd_search_result(const dd_search *search, long long *nhot, int *ngroups, unsigned *flags, void *stream) {
    const Search *s = reinterpret_cast<const Search *>(search);
    if (!s) return fail(DD_ERR_INVALID_ARG, "NULL search");
    DevState h;
    DD_CUDA_TRY(cudaMemcpyAsync(&h, s->st, sizeof(h), cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    DD_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    if (nhot) *nhot = (long long)h.nhot;
    if (ngroups) *ngroups = (int)h.nroots;
    if (flags) *flags = h.err;
    return DD_OK;
}

dd_status dd_search_stats(const dd_search *search, long long *median_rebuilds, void *stream) {
    const Search *s = reinterpret_cast<const Search *>(search);
    if (!s) return fail(DD_ERR_INVALID_ARG, "NULL search");
    DevState h;
    DD_CUDA_TRY(cudaMemcpyAsync(&h, s->st, sizeof(h), cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    DD_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    if (median_rebuilds) *median_rebuilds = (long long)h.nrebuild;
    return DD_OK;
}

dd_status dd_search_candidates(const dd_search *search, dd_candidate *host_out, int max, int *count, void *stream) {
    const Search *s = reinterpret_cast<const Search *>(search);
    if (!s || !count) return fail(DD_ERR_INVALID_ARG, "NULL search or count");
    int ng = 0;
    dd_status r = dd_search_result(search, nullptr, &ng, nullptr, stream);
    if (r != DD_OK) return r;
    const int avail = std::min(ng, s->cfg.max_cands);
    *count = avail;
    const int k = std::min(avail, max);
    if (k > 0 && host_out) {
        DD_CUDA_TRY(cudaMemcpyAsync(host_out, s->cands, (size_t)k * sizeof(dd_candidate), cudaMemcpyDeviceToHost,
                                    (cudaStream_t)stream));
        DD_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    }
    return DD_OK;
}

dd_status dd_search_device_candidates(const dd_search *search, const dd_candidate **d_cands) {
    const Search *s = reinterpret_cast<const Search *>(search);
    if (!s || !d_cands) return fail(DD_ERR_INVALID_ARG, "NULL argument");
    *d_cands = s->cands;
    return DD_OK;
}

dd_status dd_search_buffers(const dd_search *search, const int32_t **d_y, const int64_t **d_sumsq,
                            const float **d_best, const uint16_t **d_bestw) {
    const Search *s = reinterpret_cast<const Search *>(search);
    if (!s) return fail(DD_ERR_INVALID_ARG, "NULL search");
    if (d_y) *d_y = s->y;
    if (d_sumsq) *d_sumsq = reinterpret_cast<const int64_t *>(s->sumsq);
    if (d_best) *d_best = s->best;
    if (d_bestw) *d_bestw = s->bestw;
    return DD_OK;
}

dd_status dd_snippets(const int32_t *d_y, size_t ld_y, int ndm, size_t n, const int64_t *d_sumsq, int ncand,
                      const dd_candidate *d_cands, uint16_t *d_out, void *stream) {
    if (!d_y || !d_sumsq || !d_cands || !d_out || ndm <= 0 || n == 0 || ld_y < n || ncand < 0)
        return fail(DD_ERR_INVALID_ARG, "bad snippet arguments");
    if (ncand == 0) return DD_OK;
    dd_snippet_from_y_kernel<<<ncand, 256, 0, (cudaStream_t)stream>>>(
        d_y, (long long)ld_y, ndm, (long long)n, reinterpret_cast<const unsigned long long *>(d_sumsq), d_cands,
        reinterpret_cast<__nv_bfloat16 *>(d_out));
    return cuda_fail(cudaGetLastError(), "dd_snippet_kernel launch");
}

dd_status dd_search_snippets(const dd_search *search, int ncand, uint16_t *d_out, void *stream) {
    const Search *s = reinterpret_cast<const Search *>(search);
    if (!s || !d_out || ncand < 0) return fail(DD_ERR_INVALID_ARG, "NULL search or output");
    if (ncand > s->cfg.max_cands) return fail(DD_ERR_INVALID_ARG, "ncand beyond the candidate capacity");
    if (ncand == 0) return DD_OK;
    dd_snippet_kernel<<<ncand, 256, 0, (cudaStream_t)stream>>>(s->pre, s->tile_off, s->tile_sum, s->ntiles, s->ndm,
                                                            s->n, s->sumsq, s->cands,
                                                            reinterpret_cast<__nv_bfloat16 *>(d_out));
    return cuda_fail(cudaGetLastError(), "dd_snippet_kernel launch");
}

void dd_search_destroy(dd_search *search) { free_search(reinterpret_cast<Search *>(search)); }

}  // extern "C"
