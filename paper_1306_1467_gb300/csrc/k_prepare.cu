// One-time preparation kernels: integral images (Sec. 2.1), int32 Haar feature
// values (Sec. 2.2) and the per-feature stable sample order that the round
// search scans (the threshold search of Sec. 2.2-2.3 needs the samples of a
// feature in value order).
#include <limits.h>

#include <type_traits>

#include "vjb_device.cuh"
#include "vjb_haar.cuh"
#include "vjb_integral.cuh"
#include "vjb_internal.cuh"

namespace vjb {

// ---- K1: integral images --------------------------------------------------------
// A CTA takes 32 windows, a lane each.  Output is point-major, ii_t[(y * (w + 1) +
// x) * stride + i], so that the feature kernels read consecutive windows with
// coalesced loads.  ii(x, y) = sum of pixels with x' < x and y' < y (zero first
// row and column): running sums along the rows in shared memory, then down the
// columns, a band of rows at a time (the whole window where it fits).
// ii16 receives the values modulo 2^16 in the same layout (the sort evaluates
// features of small boxes from these).
//
// Bound by its writes for large sets and by the two chains of additions (w and
// h long) for small ones: 10 us at 24x24 / 1,000 (ncu).  One thread per window,
// each pixel after the one above it in memory, took 41 us there and 46 us at
// 15,000.
constexpr int kIntegralThreads = 512;

__global__ void __launch_bounds__(kIntegralThreads)
    k_integral(const uint8_t *__restrict__ px, int n, int h, int w, int band, int32_t *__restrict__ ii_t,
               uint16_t *__restrict__ ii16, int stride) {
    extern __shared__ __align__(16) int32_t sums[];  // [band][w][32], then the carry [w][32], then the pixels
    int32_t *carry = sums + (size_t)band * w * 32;
    uint32_t *tile = reinterpret_cast<uint32_t *>(carry + w * 32);
    const int tstride = tile_stride(band * w);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int i0 = blockIdx.x * kTileWindows, i = i0 + lane;
    const int W1 = w + 1;
    const bool in = i < n;
    auto put = [&](int point, int32_t v) {
        if (in) {
            ii_t[(size_t)point * stride + i] = v;
            if (ii16) ii16[(size_t)point * stride + i] = (uint16_t)v;
        }
    };
    for (int x = warp; x <= w; x += nw) put(x, 0);
    for (int y = 1 + warp; y <= h; y += nw) put(y * W1, 0);
    for (int x = warp; x < w; x += nw) carry[x * 32 + lane] = 0;
    for (int y0 = 0; y0 < h; y0 += band) {
        const int rows = min(band, h - y0);
        stage_pixels(px, i0, n, h * w, y0 * w, rows * w, tile, tstride);
        __syncthreads();
        row_sums(tile, tstride, rows, w, sums, w);
        __syncthreads();
        for (int x = warp; x < w; x += nw) {
            int32_t v = carry[x * 32 + lane];
#pragma unroll 4
            for (int y = 0; y < rows; ++y) {
                v += sums[(y * w + x) * 32 + lane];
                put((y0 + y + 1) * W1 + x + 1, v);
            }
            carry[x * 32 + lane] = v;
        }
        __syncthreads();
    }
}

constexpr size_t kIntegralSmem = 100 * 1024;  // at most: two CTAs an SM

// Once per device, before the first launch: a kernel's limit on shared memory is
// the same for every context and thread, so a launch must not set its own.
cudaError_t set_integral_limits() {
    return cudaFuncSetAttribute(k_integral, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kIntegralSmem);
}

cudaError_t launch_integral(const uint8_t *px, int n, int h, int w, int32_t *ii_t, uint16_t *ii16,
                            int ii_stride, cudaStream_t st) {
    auto bytes = [&](int band) { return ((size_t)band * w * 32 + w * 32 + 32 * tile_stride(band * w)) * 4; };
    int band = h;  // or fewer rows, down to one at a time (up to 255 pixels: 73 KB)
    while (band > 1 && bytes(band) > kIntegralSmem) --band;
    k_integral<<<(n + kTileWindows - 1) / kTileWindows, kIntegralThreads, bytes(band), st>>>(px, n, h, w, band, ii_t,
                                                                                            ii16, ii_stride);
    return cudaGetLastError();
}

// ---- the feature list -------------------------------------------------------------
// A CTA per (type, width, height), whose positions are neighbours in the list and
// start at a closed form of the three.  Filling the list on the host (for its
// length, and again for the copy) took 1.1 ms of adding a 24x24 job to a batch
// (2,287 samples: 4.45 -> 3.34 ms) and 2.1 ms of a first 32x32 table (19.8 ->
// 17.7).
__global__ void k_enumerate(int W, int H, DevFeature *__restrict__ feat) {
    int g = blockIdx.x, t = 0;
    int64_t at = 0;
    for (;; ++t) {
        const HaarBase b = haar_base(t);
        const int sizes = (W / b.w) * (H / b.h);
        if (g < sizes) break;
        g -= sizes;
        at += haar_count(t, W, H);
    }
    const HaarBase b = haar_base(t);
    const int mh = H / b.h, i = g / mh, j = g % mh;  // sizes before this one
    const int fw = (i + 1) * b.w, fh = (j + 1) * b.h, nx = W - fw + 1;
    at += haar_places(W, b.w, i) * haar_places(H, b.h, mh) + nx * haar_places(H, b.h, j);
    for (int p = threadIdx.x; p < nx * (H - fh + 1); p += blockDim.x)
        feat[at + p] = DevFeature{(uint8_t)t, (uint8_t)(p % nx), (uint8_t)(p / nx), (uint8_t)fw, (uint8_t)fh, 0, 0, 0};
}

cudaError_t launch_enumerate(int w, int h, DevFeature *feat, cudaStream_t st) {
    int sizes = 0;
    for (int t = 0; t < 5; ++t) sizes += (w / haar_base(t).w) * (h / haar_base(t).h);
    k_enumerate<<<sizes, 128, 0, st>>>(w, h, feat);
    return cudaGetLastError();
}

// ---- K2: feature values ------------------------------------------------------------
// One CTA per feature; threads stride over windows.  out[(f - f0) * n + i].
__global__ void k_feature_values(const int32_t *__restrict__ ii_t, int stride, int n, int w,
                                 const DevFeature *__restrict__ feat, int64_t f0,
                                 int32_t *__restrict__ out) {
    const DevFeature d = feat[f0 + blockIdx.x];
    int32_t *o = out + (size_t)blockIdx.x * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        o[i] = haar_value(ii_t, stride, w, d.type, d.x, d.y, d.w, d.h, i);
}

cudaError_t launch_feature_values(const int32_t *ii_t, int ii_stride, int n, int w,
                                  const DevFeature *feat, int64_t f0, int64_t nf, int32_t *out,
                                  cudaStream_t st) {
    if (nf <= 0) return cudaSuccess;
    k_feature_values<<<(unsigned)nf, 256, 0, st>>>(ii_t, ii_stride, n, w, feat, f0, out);
    return cudaGetLastError();
}

// ---- K3: segmented stable sort ---------------------------------------------------------
// One 1024-thread CTA per feature row.  The CTA first evaluates its feature on
// every window (the K2 arithmetic, fused here so the int32 values never leave
// the SM), then sorts keys value - min (non-negative) by an LSD radix sort with
// 8-bit digits over only the bits the row's value span needs.  Each pass ranks
// digits stably: items are held in registers in a "warp-striped" layout (warp
// wp, column j, lane l -> position wp*32*IPT + j*32 + l), a warp walks its
// columns in position order and ranks equal digits inside a column, and the
// per-(digit, warp) counts are scanned digit-major.  Equal keys therefore keep
// their order, and since items start in sample order, ties end up ordered by
// sample index.  Output entry = weight word | (value < next value) << 15,
// written in the lane-run row layout; positions n .. npad-1 hold the padding
// word n (weight 0, no flag).
constexpr int kSortThreads = 1024;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kRadix = 256;
constexpr int kHistStride = kSortWarps + 1;  // (digit, warp) counters, padded against bank conflicts
constexpr int kHistWords = kRadix * kHistStride;
// Gather groups of a row with two weight copies (n <= 16352): one per entry
// of a lane run, at most 16384 / 32.  Their masks sit after the histogram and
// the per-thread bank loads (32 bytes each) reuse the histogram space.
constexpr int kMaxGroups = 512;
static_assert(kSortThreads * 32 / 4 <= kHistWords, "histogram space too small for bank loads");

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// End of a row's write (all threads of the CTA): count the row and flag an
// entry before position n whose word lies outside the weight array or is the
// padding word.  The search kernels gather weights through the table without
// bounds checks; the host accepts a table only if no entry was flagged and
// every row was counted.  stat[0]: kFlagBadTable or 0, stat[1]: rows written.
__device__ __forceinline__ void row_written(bool bad, int32_t *stat) {
    const int any_bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        if (any_bad) atomicOr(&stat[0], kFlagBadTable);
        atomicAdd(&stat[1], 1);
    }
}

// Lanes of the warp holding the same BITS-bit digit `d` as this lane: one
// ballot per digit bit, each narrowing the set to the lanes that agree on that
// bit.  On this GPU BITS ballots (four instructions a bit) rank a sort pass
// faster than one __match_any_sync: 29.8 vs 31.7 ms for the 24x24 / 15k
// tables.
template <int BITS>
__device__ __forceinline__ uint32_t digit_peers(uint32_t d) {
    uint32_t eq = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < BITS; ++b) {
        uint32_t m;
        asm("{\n\t.reg .pred p;\n\t"
            "and.b32 %0, %1, %2;\n\t"
            "setp.ne.u32 p, %0, 0;\n\t"
            "vote.sync.ballot.b32 %0, p, 0xffffffff;\n\t"
            "@!p not.b32 %0, %0;\n\t}"
            : "=r"(m)
            : "r"(d), "r"(1u << b));
        eq &= m;
    }
    return eq;
}

// Exclusive scan of one int per thread over the CTA; returns the thread's
// exclusive prefix.  `ws` holds kSortWarps ints.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t *ws) {
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) ws[wp] = inc;
    __syncthreads();
    if (wp == 0) {
        uint32_t t = ws[lane];
        uint32_t ti = t;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, ti, d);
            if (lane >= d) ti += y;
        }
        ws[lane] = ti - t;
    }
    __syncthreads();
    const uint32_t r = ws[wp] + inc - x;
    __syncthreads();
    return r;
}

template <int IPT>
__global__ void __launch_bounds__(kSortThreads, 1)
    k_sort_rows(const int32_t *__restrict__ ii_t, int ii_stride, int w,
                const DevFeature *__restrict__ feat, int64_t f0, WeightLayout L,
                uint16_t *__restrict__ rows, int npad, const int32_t *__restrict__ row_list, int32_t *stat) {
    const int row = row_list ? row_list[blockIdx.x] : (int)blockIdx.x;  // row of the tile
    constexpr int NP = kSortThreads * IPT;
    const int n = L.n;
    extern __shared__ __align__(16) uint8_t smem[];
    uint32_t *skey = reinterpret_cast<uint32_t *>(smem);
    uint32_t *hist = skey + NP;                                            // kHistWords (+ kMaxGroups)
    uint32_t *ws = hist + kHistWords + (IPT <= 16 ? kMaxGroups : 0);        // kSortWarps
    int32_t *mm = reinterpret_cast<int32_t *>(ws + kSortWarps);             // 2
    uint16_t *sidx = reinterpret_cast<uint16_t *>(mm + 2);                  // NP

    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int pos0 = wp * 32 * IPT + lane;
    const DevFeature d = feat[f0 + row];

    // the feature on every window, into shared memory (K2's arithmetic)
    int32_t lo = INT_MAX, hi = INT_MIN;
    for (int p = threadIdx.x; p < n; p += kSortThreads) {
        const int32_t x = haar_value(ii_t, ii_stride, w, d.type, d.x, d.y, d.w, d.h, p);
        skey[p] = static_cast<uint32_t>(x);
        lo = min(lo, x);
        hi = max(hi, x);
    }
    __syncthreads();
    uint32_t key[IPT];
    uint32_t ipk[(IPT + 1) / 2];  // two 16-bit sample indices per register
#pragma unroll
    for (int j = 0; j < IPT; ++j) {
        const int p = pos0 + j * 32;
        key[j] = p < n ? skey[p] : 0u;
    }
#pragma unroll
    for (int s = 16; s; s >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, s));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, s));
    }
    if (threadIdx.x == 0) { mm[0] = INT_MAX; mm[1] = INT_MIN; }
    __syncthreads();
    if (lane == 0) { atomicMin(&mm[0], lo); atomicMax(&mm[1], hi); }
    __syncthreads();
    lo = mm[0];
    hi = mm[1];
    const uint32_t span = static_cast<uint32_t>(hi) - static_cast<uint32_t>(lo);
    const int bits = span ? 32 - __clz(span) : 0;
#pragma unroll
    for (int j = 0; j < IPT; ++j) {
        const int p = pos0 + j * 32;
        // padding items take the all-ones key: they sort after every real item
        key[j] = (p < n) ? key[j] - static_cast<uint32_t>(lo) : 0xffffffffu;
        if (j & 1) ipk[j >> 1] |= static_cast<uint32_t>(p) << 16;
        else ipk[j >> 1] = static_cast<uint32_t>(p) & 0xffffu;
    }

    const uint32_t lt = lanemask_lt();
    for (int shift = 0; shift < bits; shift += 8) {
        for (int k = threadIdx.x; k < kHistWords; k += kSortThreads) hist[k] = 0;
        __syncthreads();
        // count digits per (digit, warp)
#pragma unroll
        for (int j = 0; j < IPT; ++j) {
            const uint32_t dg = (key[j] >> shift) & (kRadix - 1);
            const uint32_t peers = digit_peers<8>(dg);
            if (lane == __ffs(peers) - 1) hist[dg * kHistStride + wp] += __popc(peers);
        }
        __syncthreads();
        // exclusive scan, digit-major then warp: thread t owns 8 consecutive counters
        {
            constexpr int PER = kRadix * kSortWarps / kSortThreads;  // 8
            uint32_t c[PER];
            uint32_t s = 0;
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int lin = threadIdx.x * PER + q;
                c[q] = hist[(lin >> 5) * kHistStride + (lin & 31)];
                s += c[q];
            }
            uint32_t off = block_exclusive_scan(s, ws);
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int lin = threadIdx.x * PER + q;
                hist[(lin >> 5) * kHistStride + (lin & 31)] = off;
                off += c[q];
            }
        }
        __syncthreads();
        // scatter in position order
#pragma unroll
        for (int j = 0; j < IPT; ++j) {
            const uint32_t dg = (key[j] >> shift) & (kRadix - 1);
            const uint32_t peers = digit_peers<8>(dg);
            const uint32_t base = hist[dg * kHistStride + wp];
            __syncwarp();
            if (lane == __ffs(peers) - 1) hist[dg * kHistStride + wp] = base + __popc(peers);
            __syncwarp();
            const uint32_t dst = base + __popc(peers & lt);
            skey[dst] = key[j];
            sidx[dst] = static_cast<uint16_t>((j & 1) ? (ipk[j >> 1] >> 16) : (ipk[j >> 1] & 0xffffu));
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < IPT; ++j) {
            const int p = pos0 + j * 32;
            key[j] = skey[p];
            const uint32_t ix = sidx[p];
            if (j & 1) ipk[j >> 1] = (ipk[j >> 1] & 0xffffu) | (ix << 16);
            else ipk[j >> 1] = ix;
        }
        __syncthreads();
    }
    // make the final order visible in shared memory (also when no pass ran)
#pragma unroll
    for (int j = 0; j < IPT; ++j) {
        const int p = pos0 + j * 32;
        skey[p] = key[j];
        sidx[p] = static_cast<uint16_t>((j & 1) ? (ipk[j >> 1] >> 16) : (ipk[j >> 1] & 0xffffu));
    }
    __syncthreads();
    uint16_t *out = rows + (size_t)row * npad;
    const int run = npad / 32;  // entries per lane run (see phys_of)
    if (L.dual) {
        // With two weight copies, choose per entry which copy the search
        // gathers from.  One gather instruction of the search kernel reads
        // entry r of every lane run: the 32 entries k * run + r, k = 0..31.
        // For each such group, greedily put each entry that has a copy B
        // (samples below L.nb) in the less loaded of its two banks (copy A:
        // i mod 32, copy B: rot(i) mod 32), then let such entries move to a
        // lighter bank.  Bank loads are kept per thread, bank-major so that
        // the threads do not share banks.  The split flags first go into bit 15
        // of the sample indices (n <= 32767), which frees the keys' space for
        // the choices of the 32-item variant.
        for (int p = threadIdx.x; p < n; p += kSortThreads)
            if (p == n - 1 || skey[p] < skey[p + 1]) sidx[p] |= 0x8000u;
        __syncthreads();
        uint32_t *gchoice = IPT <= 16 ? hist + kRadix * kSortWarps : skey;  // one mask per group
        uint8_t *ld = reinterpret_cast<uint8_t *>(hist) + threadIdx.x;
        for (int g = threadIdx.x; g < run; g += kSortThreads) {
#pragma unroll
            for (int b = 0; b < 32; ++b) ld[b * kSortThreads] = 0;
            uint32_t mask = 0;
            bool pad_seen = false;
            for (int k = 0; k < 32; ++k) {
                const int p = k * run + g;
                if (p >= n) {
                    if (!pad_seen) ld[(n & 31) * kSortThreads]++;  // padding: one broadcast read
                    pad_seen = true;
                    continue;
                }
                const int i = sidx[p] & 0x7fff;
                const int ba = i & 31, bb = rot_b(i) & 31;
                if (i < L.nb && ld[bb * kSortThreads] < ld[ba * kSortThreads]) {
                    ld[bb * kSortThreads]++;
                    mask |= 1u << k;
                } else {
                    ld[ba * kSortThreads]++;
                }
            }
            // two passes of single moves: an entry leaves its bank when the
            // other one is at least two entries lighter
            for (int pass = 0; pass < 2; ++pass)
                for (int k = 0; k < 32; ++k) {
                    const int p = k * run + g;
                    if (p >= n) break;
                    const int i = sidx[p] & 0x7fff;
                    if (i >= L.nb) continue;
                    const int ba = i & 31, bb = rot_b(i) & 31;
                    const bool onb = (mask >> k) & 1u;
                    const int cur = onb ? bb : ba, oth = onb ? ba : bb;
                    if (ld[cur * kSortThreads] > ld[oth * kSortThreads] + 1) {
                        ld[cur * kSortThreads]--;
                        ld[oth * kSortThreads]++;
                        mask ^= 1u << k;
                    }
                }
            gchoice[g] = mask;
        }
        __syncthreads();
        bool bad = false;
        for (int P = threadIdx.x; P < npad; P += kSortThreads) {
            const int p = logical_of(P, run);
            uint16_t e;
            if (p < n) {
                const uint32_t x = sidx[p];
                int word = (int)(x & 0x7fffu);
                const int k = (P >> 3) & 31, g = (P >> 8) * kChunkElems + (P & 7);  // p = k * run + g
                if ((gchoice[g] >> k) & 1u) word = L.off_b + rot_b(word);
                bad |= word >= L.words || word == n;
                e = make_entry(word, (x & 0x8000u) != 0, P);
            } else {
                e = make_entry(n, false, P);
            }
            out[P] = e;
        }
        row_written(bad, stat);
        return;
    }
    bool bad = false;
    for (int P = threadIdx.x; P < npad; P += kSortThreads) {
        const int p = logical_of(P, run);
        uint16_t e;
        if (p < n) {
            const bool step = (p == n - 1) || (skey[p] < skey[p + 1]);
            bad |= (int)sidx[p] >= L.words || (int)sidx[p] == n;
            e = make_entry(sidx[p], step, P);
        } else {
            e = make_entry(n, false, P);
        }
        out[P] = e;
    }
    row_written(bad, stat);
}

template <int IPT>
static size_t sort_smem() {
    const size_t hist_words = kHistWords + (IPT <= 16 ? kMaxGroups : 0);
    return (size_t)kSortThreads * IPT * 4 + hist_words * 4 + kSortWarps * 4 + 8 +
           (size_t)kSortThreads * IPT * 2;
}

template <int IPT>
static cudaError_t launch_sort_ipt(const int32_t *ii_t, int ii_stride, int w, const DevFeature *feat,
                                   int64_t f0, int64_t nf, const WeightLayout &L, uint16_t *rows,
                                   int npad, const int32_t *row_list, int32_t *stat, cudaStream_t st) {
    const size_t sm = sort_smem<IPT>();
    cudaError_t e = cudaFuncSetAttribute(k_sort_rows<IPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sm);
    if (e != cudaSuccess) return e;
    k_sort_rows<IPT><<<(unsigned)nf, kSortThreads, sm, st>>>(ii_t, ii_stride, w, feat, f0, L, rows, npad,
                                                            row_list, stat);
    return cudaGetLastError();
}

// ---- K3, packed variant (the one every row goes through first) ---------------------------
// The same stable sort for rows whose items fit one 32-bit word: value - min
// in the high bits above a sample index of ib bits (14 up to 16,384 samples).
// A row whose value span does not fit next to its index is listed for the
// two-word sort above.  Only the value bits are sorted, in passes over digits
// of at most 8 bits, as few and as even as that allows (at least 5 bits: one
// pass up to 8 bits of span, two up to 16); the starting index order and stable
// passes order ties by sample index.
//
// A pass: each warp counts the digits of its items (a contiguous range of
// positions) in counters of its own, the counters become first positions by a
// scan over (digit, warp), and each item takes its place with an atomic add on
// its warp's counter of its digit, 32 items after the 32 before them.  That is
// stable where the lanes of one such add are served in lane order, as this GPU
// does; since nothing promises it, the write checks that the finished row's
// words ascend (a word is value, then sample index, so ascending words are the
// order itself) and a row that fails is listed for the two-word sort, which
// ranks with ballots.
//
// Then the bank choice of the two weight copies and the run-interleaved write,
// one 16-byte chunk per thread.
//
// What bounds it: shared memory (16x16 / 15,000 under ncu: its pipe 74% busy, 37
// wavefronts per 32 items, half of them the atomics' bank conflicts) and the
// barriers between phases that use it unevenly.  Ranking with one ballot per
// digit bit, the form before, was ALU bound at 223 instructions an item.
// Tables in all, then -> with atomics -> with gaps between the finished runs
// (kRunGap) and the samples of one copy placed first -> values eight windows a
// load, counts in batches -> smaller CTAs, and rows whose last runs are short
// chosen and written like whole ones:
//   24x24 / 2,003   6.04 ->  2.90 ->  2.54 ->  2.54 ->  2.27 ms
//   32x32 / 5,003   31.9 ->  20.0 ->  17.1 ->  16.8 ->  15.6
//   24x24 / 10,963  16.4 ->  12.9 ->  12.3 ->  11.6 ->  10.3
//   24x24 / 15,000  20.9 ->  16.1 ->  15.8 ->  15.0 ->  13.8
//   24x24 / 18,300  34.4 ->  26.0 ->  21.9 ->  21.0 ->  19.1
//
// Threads per CTA: few, with as many items each as the registers hold (128
// threads up to 4,096 samples, 256 up to 15,360, 384 with two CTAs an SM up to
// 20,736, then 512).  Every warp has counters of its own to clear and scan, and
// more and smaller CTAs leave other rows to run while one waits at a barrier:
// 256 threads of 40 to 60 items, three CTAs an SM, against 512 of 20 to 30, two:
// 10,000 samples 11.24 -> 9.74 ms, 13,000 13.36 -> 11.9, 15,000 15.0 -> 14.1; 384
// of 48 against 640 of 30: 18,300 21.0 -> 19.0; 512 of 48 and 64 against 1,024 of
// 24 and 32: 24,000 13.3 -> 12.4, 32,766 12.9 -> 12.3.  The other way round costs:
// 512 threads of 16 at 8,000 8.6 against 7.6 ms, 640 of 24 at 15,000 15.6 against
// 15.0; so do too few warps: 128 of 40 at 5,003 17.3 against 16.7 ms, 192 of 40 at
// 7,148 7.14 against 6.91.
//
// Measured and dropped: one pass with a counter per value for spans up to 14
// bits (one warp ranking a row in order waits its turn behind the other CTA's
// warps: 16.9 ms at 15,000); buckets filled in any order and put right by
// counting or by insertion (28.7 ms); predicated atomics for the last warp's
// missing items (the compiler wraps each in a branch: 158 instructions); the
// row filled up to whole groups of 32 items and whole groups skipped (the
// batches' branches cost more registers: 15,000 13.8 -> 14.1, 3,300 3.5 -> 3.75,
// though 4,090 3.83 -> 3.59).
constexpr int kPkDigitBits = 8;
// Words between the 32 lane runs of a finished row in shared memory: runs are a
// multiple of 8 words long, and without a gap the reads of one place in every
// run (the write's 16-byte chunks, the refined groups' entries) meet in a few
// banks, in one when the run is a multiple of 32 (24x24 / 4,096: 4.36 -> 3.65 ms
// with the gap).
constexpr int kRunGap = 4;
constexpr int kPkRadix = 1 << kPkDigitBits;

// Adds to counters in shared memory, as the instructions themselves: the
// ranking depends on one following the other in program order.
__device__ __forceinline__ void shared_add(uint32_t addr, uint32_t x) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(x) : "memory");
}
__device__ __forceinline__ uint32_t shared_take(uint32_t addr) {
    uint32_t old;
    asm volatile("atom.shared.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(addr) : "memory");
    return old;
}

// CTAs an SM by registers: a thread holds its IPT items and about 20 values
// more.  (40 registers for 16 items and 48 for 20 spill a little, outside the
// passes, and are still better than fewer CTAs: 2,003 2.53 -> 2.49 ms, 32x32 /
// 5,003 16.84 -> 16.73.)
constexpr int packed_ctas(int ipt, int th) {
    return 65536 / (th * (ipt <= 16 ? 40 : ipt <= 20 ? 48 : ipt <= 32 ? 64 : ipt <= 48 ? 72 : 80));
}

template <int IPT, int TH>
__global__ void __launch_bounds__(TH, packed_ctas(IPT, TH))
    k_sort_rows_packed(const int32_t *__restrict__ ii_t, const uint16_t *__restrict__ ii16, int ii_stride, int w,
                       const DevFeature *__restrict__ feat, int64_t f0, WeightLayout L,
                       uint16_t *__restrict__ rows, int npad, int32_t *ovf, int32_t *stat) {
    constexpr int NP = TH * IPT;
    constexpr int WARPS = TH / 32;
    constexpr int GROUPS = NP / 32;  // lane-run groups of the longest row
    static_assert(4 * GROUPS <= kPkRadix * WARPS, "counter space too small for the refine list");
    const int n = L.n;
    extern __shared__ __align__(16) uint8_t smem[];
    uint32_t *skey = reinterpret_cast<uint32_t *>(smem);                        // NP items
    // kPkRadix * WARPS counters, from a multiple of a warp's share of them
    uint32_t *hist = skey + NP + 32 * kRunGap;
    hist += ((0u - smem_u32(hist)) & (4u * kPkRadix - 1u)) / 4u;
    uint32_t *gchoice = hist + kPkRadix * WARPS;                                // GROUPS
    uint32_t *ws = gchoice + GROUPS;                                            // kPkRadix / 32
    int32_t *mm = reinterpret_cast<int32_t *>(ws + kPkRadix / 32);              // 2 * WARPS
    uint32_t *spare = reinterpret_cast<uint32_t *>(mm + 2 * WARPS);             // 32

    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int pos0 = wp * 32 * IPT + lane;
    const DevFeature d = feat[f0 + blockIdx.x];

    // the feature on every window (K2's arithmetic), four windows per thread
    // and point.  Boxes of at most kNarrowArea pixels come from the
    // integral images modulo 2^16, eight windows a load and two to a 32-bit
    // word (half the bytes, and the points are added two windows at a time);
    // they are kept as 16-bit offsets from the type's smallest possible value.
    const bool narrow = ii16 && d.w * d.h <= kNarrowArea;
    uint16_t *val16 = reinterpret_cast<uint16_t *>(skey);
    int32_t lo = INT_MAX, hi = INT_MIN;
    if (narrow) {
        uint32_t lo2 = 0xffffffffu, hi2 = 0u;
        haar_rows_narrow<TH>(ii16, ii_stride, w, d.type, d.x, d.y, d.w, d.h, n, [&](int q, uint4 x) {
            const int left = n - 8 * q;  // at least 1
            if (left < 8) {  // past the last sample: repeat the window before, word by word
                auto half = [](uint32_t a) { return (a & 0xffffu) * 0x10001u; };
                if (left == 1) x.x = half(x.x);
                if (left <= 2) x.y = (x.x >> 16) * 0x10001u;
                if (left == 3) x.y = half(x.y);
                if (left <= 4) x.z = (x.y >> 16) * 0x10001u;
                if (left == 5) x.z = half(x.z);
                if (left <= 6) x.w = (x.z >> 16) * 0x10001u;
                if (left == 7) x.w = half(x.w);
            }
            reinterpret_cast<uint4 *>(skey)[q] = x;
            lo2 = __vminu2(__vminu2(lo2, __vminu2(x.x, x.y)), __vminu2(x.z, x.w));
            hi2 = __vmaxu2(__vmaxu2(hi2, __vmaxu2(x.x, x.y)), __vmaxu2(x.z, x.w));
        });
        lo = (int32_t)min(lo2 & 0xffffu, lo2 >> 16);
        hi = (int32_t)max(hi2 & 0xffffu, hi2 >> 16);
    } else {
        haar_rows<TH, int4>(
            ii_t, ii_stride, w, d.type, d.x, d.y, d.w, d.h, n,
            [](int4 a, int4 b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); },
            [&](int q, int4 pos, int4 neg) {
                const int p = 4 * q;
                const int4 x = make_int4(pos.x - neg.x, pos.y - neg.y, pos.z - neg.z, pos.w - neg.w);
                reinterpret_cast<int4 *>(skey)[q] = x;
                lo = min(lo, x.x);
                hi = max(hi, x.x);
                if (p + 1 < n) { lo = min(lo, x.y); hi = max(hi, x.y); }
                if (p + 2 < n) { lo = min(lo, x.z); hi = max(hi, x.z); }
                if (p + 3 < n) { lo = min(lo, x.w); hi = max(hi, x.w); }
            });
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) { mm[2 * wp] = lo; mm[2 * wp + 1] = hi; }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, mm[2 * (lane % WARPS)]);
    hi = __reduce_max_sync(0xffffffffu, mm[2 * (lane % WARPS) + 1]);
    const uint32_t span = static_cast<uint32_t>(hi) - static_cast<uint32_t>(lo);
    const int bits = span ? 32 - __clz(span) : 0;
    // bits of a sample index (at least those the bank choice looks at)
    const int ib = max(10, 32 - __clz((uint32_t)(n - 1)));
    const uint32_t imask = (1u << ib) - 1u;
    if (bits + ib > 32) {  // value and index do not fit one word: the two-word sort takes the row
        if (threadIdx.x == 0) ovf[1 + atomicAdd(ovf, 1)] = (int32_t)blockIdx.x;
        return;
    }
    // items pos0 + 32 j; those from j = mine on lie past the last sample and
    // are not counted or stored
    const int mine = (n - pos0 + 31) >> 5;
    // a warp with samples to the end of its range counts and places all of them;
    // another's lanes past the last sample add to a spare word (a skipped add
    // costs a branch around every one)
    const bool all_mine = (wp + 1) * 32 * IPT <= n;
    const uint32_t spare32 = smem_u32(spare + lane);
    const int passes = max(1, (bits + kPkDigitBits - 1) / kPkDigitBits);
    const int D = max(5, (bits + passes - 1) / passes);
    uint32_t *own = hist + (wp << D);  // this warp's counters, one per digit
    const uint32_t own32 = smem_u32(own);
    const uint32_t dmask = ((1u << D) - 1u) << 2;  // a digit as a byte offset
    // one stable pass over the D-bit digit from bit `shift` of the values, the
    // items in position order from item(j, p)
    const int run = npad / 32;
    auto radix_pass = [&](int shift, auto digit, auto item) {
        const int sh = ib + shift - 2;
        // the last pass leaves the gaps between the runs: position + kRunGap * (position / run)
        const uint32_t per_run = shift + D >= bits ? 0xffffffffu / (uint32_t)run + 1u : 0u;
        for (int k = lane; k < (1 << D); k += 32) own[k] = 0u;
        __syncwarp();
        // (eight items are read, then counted: an item's read would wait for the
        // add before it; tables at 24x24 / 10,963 11.9 -> 11.6 ms)
        auto count = [&](auto whole) {
            constexpr int BATCH = 8;
#pragma unroll
            for (int j0 = 0; j0 < IPT; j0 += BATCH) {
                uint32_t at[BATCH];
#pragma unroll
                for (int u = 0; u < BATCH && j0 + u < IPT; ++u) at[u] = (digit(pos0 + 32 * (j0 + u), sh) & dmask) | own32;
#pragma unroll
                for (int u = 0; u < BATCH && j0 + u < IPT; ++u)
                    shared_add(decltype(whole)::value || j0 + u < mine ? at[u] : spare32, 1u);
            }
        };
        if (all_mine) count(std::true_type{});
        else count(std::false_type{});
        __syncthreads();
        // first positions, by digit, then warp: a thread takes digit q * TH +
        // tid of every warp's counters
        constexpr int ROUNDS = (kPkRadix + TH - 1) / TH;
        uint32_t pre[ROUNDS];
#pragma unroll
        for (int q = 0; q < ROUNDS; ++q) {
            const int dg = q * TH + (int)threadIdx.x;
            if (dg < (1 << D)) {  // uniform over a warp: D >= 5
                uint32_t t = 0u;
#pragma unroll 8
                for (int w = 0; w < WARPS; ++w) t += hist[(w << D) + dg];
                uint32_t inc = t;
#pragma unroll
                for (int dd = 1; dd < 32; dd <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, dd);
                    if (lane >= dd) inc += y;
                }
                if (lane == 31) ws[q * WARPS + wp] = inc;
                pre[q] = inc - t;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < ROUNDS; ++q) {
            const int dg = q * TH + (int)threadIdx.x;
            if (dg < (1 << D)) {
                const int before = q * WARPS + wp;  // at most kPkRadix / 32 - 1
                uint32_t run = pre[q] + __reduce_add_sync(0xffffffffu, lane < before ? ws[lane % (kPkRadix / 32)] : 0u);
#pragma unroll 8
                for (int w = 0; w < WARPS; ++w) {
                    const uint32_t t = hist[(w << D) + dg];
                    hist[(w << D) + dg] = run;
                    run += t;
                }
            }
        }
        // the items again (holding them through the scan costs spills), all
        // read before any is stored
        uint32_t c[IPT];
#pragma unroll
        for (int j = 0; j < IPT; ++j) c[j] = item(pos0 + 32 * j);
        __syncthreads();
        // (adds in batches, so that a store does not wait for its own add alone)
        auto place = [&](auto whole) {
            constexpr int BATCH = 4;
#pragma unroll
            for (int j0 = 0; j0 < IPT; j0 += BATCH) {
                uint32_t to[BATCH];
#pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    const int j = j0 + u;
                    if (j >= IPT) break;
                    const uint32_t at = ((c[j] >> sh) & dmask) | own32;
                    to[u] = shared_take(decltype(whole)::value || j < mine ? at : spare32);
                }
#pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    const int j = j0 + u;
                    if (j < IPT && (decltype(whole)::value || j < mine)) skey[to[u] + kRunGap * __umulhi(to[u], per_run)] = c[j];
                }
            }
        };
        if (all_mine) place(std::true_type{});
        else place(std::false_type{});
        __syncthreads();
    };
    // (a row of one value takes a pass too: every digit 0, the items in order)
    if (narrow)
        radix_pass(
            0, [&](int p, int) { return ((uint32_t)val16[p] - (uint32_t)lo) << 2; },
            [&](int p) { return (((uint32_t)val16[p] - (uint32_t)lo) << ib) + (uint32_t)p; });
    else
        radix_pass(
            0, [&](int p, int) { return (skey[p] - (uint32_t)lo) << 2; },
            [&](int p) { return ((skey[p] - (uint32_t)lo) << ib) + (uint32_t)p; });
    for (int shift = D; shift < bits; shift += D) 
        radix_pass(
            shift, [&](int p, int sh) { return skey[p] >> sh; }, [&](int p) { return skey[p]; });

    uint16_t *out = rows + (size_t)blockIdx.x * npad;
    const int pitch = run + kRunGap;  // from run to run in skey
    if (L.dual) {
        // bank-balanced copy choice per gather group (see k_sort_rows): each
        // entry goes to the less loaded of its two banks, one thread a group.
        // The 32 banks' loads are three masks (banks with at least 1, 2, 3
        // entries).  The groups left with a bank at 3 are listed (in the free
        // counter space) and taken by a warp each, a lane per entry: while an
        // entry of such a bank has its other bank below 2, the first of them
        // moves there.
        uint32_t *rlist = hist;      // (group, masks) of the groups to refine
        auto bank_bits = [&](uint32_t x, uint32_t &a, uint32_t &b) {  // x: a word of skey (its bits 0-9 are the index's)
            a = __funnelshift_l(0u, 1u, x);                    // 1 << (i mod 32)
            b = __funnelshift_l(0u, 1u, x + 13u * (x >> 5));  // 1 << (rot_b(i) mod 32)
        };
        if (threadIdx.x == 0) mm[0] = 0;
        __syncthreads();
        // Of a group's 32 entries every group has `whole`, and those below row
        // position n one more: a loop of that length diverges, and rolled it
        // took as long again as the rest (2,003 samples: tables 2.49 -> 2.33 ms,
        // 32x32 / 5,003 16.7 -> 15.8).
        const int whole = n / run;
        auto choose = [&](auto partial) {
            for (int g = threadIdx.x; g < run; g += TH) {
                uint32_t m1 = 0u, m2 = 0u, m3 = 0u, mask = 0u;
                const uint32_t *first = skey + g;
                const int kend = whole + (whole * run + g < n ? 1 : 0);  // entries k * run + g < n
                auto put = [&](uint32_t to) {
                    m3 |= m2 & to;
                    m2 |= m1 & to;
                    m1 |= to;
                };
                auto entry = [&](int k, bool there) {
                    const uint32_t x = first[k * pitch];
                    uint32_t a, b;
                    bank_bits(x, a, b);
                    if (!there) a = b = 0u;
                    if (decltype(partial)::value && (int)(x & imask) >= L.nb) a = b = 0u;  // placed before
                    // bank b is less loaded if it has no entry and a has one,
                    // or has one and a has two; without branches
                    uint32_t to;
                    asm("{\n\t.reg .pred p, q;\n\t.reg .b32 t;\n\t"
                        "and.b32 t, %2, %4;\n\tsetp.ne.u32 p, t, 0;\n\t"
                        "and.b32 t, %2, %5;\n\tsetp.eq.and.u32 p, t, 0, p;\n\t"
                        "and.b32 t, %3, %4;\n\tsetp.ne.u32 q, t, 0;\n\t"
                        "and.b32 t, %3, %5;\n\tsetp.eq.and.u32 q, t, 0, q;\n\t"
                        "or.pred p, p, q;\n\t"
                        "selp.b32 %0, %5, %4, p;\n\t"
                        "@p or.b32 %1, %1, %6;\n\t}"
                        : "=r"(to), "+r"(mask)
                        : "r"(m1), "r"(m2), "r"(a), "r"(b), "r"(1u << k));
                    put(to);
                };
                // eight entries at a time; past the row's end (position k * run +
                // g, in the last runs only) an entry counts nothing
                auto entries = [&](auto each) {
                    for (int k0 = 0; k0 < 32; k0 += 8) {
                        if (k0 + 8 <= whole) {
#pragma unroll
                            for (int u = 0; u < 8; ++u) each(k0 + u, true);
                        } else {
#pragma unroll
                            for (int u = 0; u < 8; ++u) each(k0 + u, k0 + u < kend);
                        }
                    }
                };
                if (decltype(partial)::value)
                    // the samples with one copy first: those with two fill the gaps
                    entries([&](int k, bool there) {
                        const uint32_t x = first[k * pitch];
                        put(there && (int)(x & imask) >= L.nb ? __funnelshift_l(0u, 1u, x) : 0u);
                    });
                entries(entry);
                if (kend < 32) put(1u << (n & 31));  // the padding word, read as a broadcast
                gchoice[g] = mask;
                // (rows above 20,736 samples: so few entries have two copies that
                // refining buys no search time; 24,000: 5 us for 2.9 ms)
                if (m3 && (NP <= 54 * 384 || !decltype(partial)::value)) {
                    const int q = atomicAdd(&mm[0], 1);
                    reinterpret_cast<uint4 *>(rlist)[q] = make_uint4((uint32_t)g, m1, m2, m3);
                }
            }
        };
        if (L.nb < n) choose(std::true_type{});  // samples from nb on have one copy only
        else choose(std::false_type{});
        __syncthreads();
        const int nref = mm[0];
        // (the next group's words are on their way while this one is taken)
        struct Group {
            int g;
            uint32_t m1, m2, m3, mask, x;
        } cur, next;
        auto fetch = [&](int q, Group &k) {
            if (q >= nref) return;
            const uint4 l = reinterpret_cast<const uint4 *>(rlist)[q];
            k.g = (int)l.x;
            k.m1 = l.y;
            k.m2 = l.z;
            k.m3 = l.w;
            k.mask = gchoice[k.g];
            k.x = skey[lane * pitch + k.g];
        };
        fetch(wp, next);
        for (int q = wp; q < nref; q += WARPS) {
            cur = next;
            fetch(q + WARPS, next);
            uint32_t a, b;
            bank_bits(cur.x, a, b);
            bool onb = (cur.mask >> lane) & 1u;
            const bool can = lane * run + cur.g < n && (int)(cur.x & imask) < L.nb;
            for (;;) {
                const uint32_t now = onb ? b : a, oth = onb ? a : b;
                const uint32_t moves = __ballot_sync(0xffffffffu, can && (cur.m3 & now) && !(cur.m2 & oth));
                if (!moves) break;
                const int first = __ffs(moves) - 1;
                const uint32_t from = __shfl_sync(0xffffffffu, now, first), to = __shfl_sync(0xffffffffu, oth, first);
                cur.m3 &= ~from;
                cur.m2 |= cur.m1 & to;
                cur.m1 |= to;
                cur.mask ^= 1u << first;
                if (lane == first) onb = !onb;
            }
            if (lane == 0) gchoice[cur.g] = cur.mask;
        }
        __syncthreads();
    }
    // the run-interleaved write: one 16-byte chunk (8 entries) per thread;
    // chunk c holds entries t * 8 .. t * 8 + 7 of lane run k (c = t * 32 + k),
    // consecutive positions p0 .. p0 + 7 of the value order
    bool bad = false, unsorted = false;
    for (int c = threadIdx.x; c < npad / kChunkElems; c += TH) {
        const int k = c & 31, t = c >> 5;
        const int p0 = k * run + t * kChunkElems;
        uint32_t cp[kChunkElems + 1];
        const uint32_t *at = skey + k * pitch + t * kChunkElems;
        const uint4 lo4 = *reinterpret_cast<const uint4 *>(at);
        const uint4 hi4 = *reinterpret_cast<const uint4 *>(at + 4);
        cp[0] = lo4.x; cp[1] = lo4.y; cp[2] = lo4.z; cp[3] = lo4.w;
        cp[4] = hi4.x; cp[5] = hi4.y; cp[6] = hi4.z; cp[7] = hi4.w;
        // (the run's last chunk is followed by the next run, past the gap)
        cp[8] = p0 + kChunkElems < n ? at[kChunkElems + (t == run / kChunkElems - 1 ? kRunGap : 0)] : 0u;
        uint32_t gc[kChunkElems] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
        if (L.dual) {
            const uint4 g0 = *reinterpret_cast<const uint4 *>(gchoice + t * kChunkElems);
            const uint4 g1 = *reinterpret_cast<const uint4 *>(gchoice + t * kChunkElems + 4);
            gc[0] = g0.x; gc[1] = g0.y; gc[2] = g0.z; gc[3] = g0.w;
            gc[4] = g1.x; gc[5] = g1.y; gc[6] = g1.z; gc[7] = g1.w;
        }
        uint32_t wv[kChunkElems / 2];
        const uint32_t lanebit = 1u << k;
        if (p0 >= n) {  // padding, at the end of the last lane run: one lane of a warp (2,003: 2.33 -> 2.27 ms)
            const uint32_t two = make_entry(n, false, 0) | make_entry(n, false, 1) << 16;
            wv[0] = wv[1] = wv[2] = wv[3] = two;
        } else if (p0 + kChunkElems < n) {  // the row goes on after the chunk
#pragma unroll
            for (int j = 0; j < kChunkElems; ++j) {
                const uint32_t i = cp[j] & imask;
                const bool tob = (gc[j] & lanebit) != 0u;
                const uint32_t word = tob ? (uint32_t)L.off_b + (uint32_t)rot_b((int)i) : i;
                // words ascend, and two of one value differ below the value bits only
                const uint32_t f = (cp[j] ^ cp[j + 1]) > imask ? (j & 1 ? 0x10000u : 0x8000u) : 0u;
                unsorted |= cp[j] >= cp[j + 1];
                // a sample index in range names a word of the weight array, and not the padding word
                bad |= i >= (uint32_t)(tob ? L.nb : n);
                if (j & 1) wv[j >> 1] |= (word << 17) | f;  // make_entry's two forms
                else wv[j >> 1] = word | f;
            }
        } else {
#pragma unroll
            for (int j = 0; j < kChunkElems; ++j) {
                const int p = p0 + j;
                uint32_t e = make_entry(n, false, j);
                if (p < n) {
                    const uint32_t i = cp[j] & imask;
                    const bool tob = (gc[j] & lanebit) != 0u;
                    const bool last = p == n - 1;
                    unsorted |= !last && cp[j] >= cp[j + 1];
                    bad |= i >= (uint32_t)(tob ? L.nb : n);
                    e = make_entry(tob ? L.off_b + rot_b((int)i) : (int)i, last || (cp[j] ^ cp[j + 1]) > imask, j);
                }
                if (j & 1) wv[j >> 1] |= e << 16;
                else wv[j >> 1] = e;
            }
        }
        reinterpret_cast<uint4 *>(out)[c] = make_uint4(wv[0], wv[1], wv[2], wv[3]);
    }
    if (__syncthreads_or(unsorted)) {  // the two-word sort writes the row again
        if (threadIdx.x == 0) ovf[1 + atomicAdd(ovf, 1)] = (int32_t)blockIdx.x;
        return;
    }
    row_written(bad, stat);
}

template <int IPT, int TH>
static size_t sort_packed_smem() {
    return (size_t)(TH * IPT + 32 * kRunGap + kPkRadix + kPkRadix * (TH / 32) + TH * IPT / 32 + kPkRadix / 32 + 2 * (TH / 32) + 32) * 4;
}

template <int IPT, int TH>
static cudaError_t launch_sort_packed(const int32_t *ii_t, const uint16_t *ii16, int ii_stride, int w,
                                      const DevFeature *feat,
                                      int64_t f0, int64_t nf, const WeightLayout &L, uint16_t *rows,
                                      int npad, int32_t *ovf, int32_t *stat, cudaStream_t st) {
    const size_t sm = sort_packed_smem<IPT, TH>();
    cudaError_t e = cudaFuncSetAttribute(k_sort_rows_packed<IPT, TH>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_sort_rows_packed<IPT, TH><<<(unsigned)nf, TH, sm, st>>>(ii_t, ii16, ii_stride, w, feat, f0, L, rows, npad,
                                                              ovf, stat);
    return cudaGetLastError();
}

// Two-word sort of `nf` rows of the tile (all of them, or those listed).
static cudaError_t launch_sort_wide(const int32_t *ii_t, int ii_stride, int w, const DevFeature *feat,
                                   int64_t f0, int64_t nf, const WeightLayout &L, uint16_t *rows, int npad,
                                   const int32_t *row_list, int32_t *stat, cudaStream_t st) {
    const int n = L.n;
#define VJB_SORT_CASE(I) launch_sort_ipt<I>(ii_t, ii_stride, w, feat, f0, nf, L, rows, npad, row_list, stat, st)
    if (n <= kSortThreads * 1) return VJB_SORT_CASE(1);
    if (n <= kSortThreads * 2) return VJB_SORT_CASE(2);
    if (n <= kSortThreads * 4) return VJB_SORT_CASE(4);
    if (n <= kSortThreads * 8) return VJB_SORT_CASE(8);
    if (n <= kSortThreads * 16) return VJB_SORT_CASE(16);
    return VJB_SORT_CASE(32);
#undef VJB_SORT_CASE
}

// Rows of a tile: the packed sort for every row, then the two-word sort for
// the rows that the packed sort lists: those whose value span and sample index
// do not fit one word (and any it would have written out of order).
// `ii16` (the integral images modulo 2^16, or null) serves the packed sort's
// features of small boxes.  `scratch` (3 + nf ints of device memory): [0] and [1] the table's check
// state (see row_written; zeroed by the caller once per table), [2] the
// tile's listed-row count, then the listed rows.  Waits for the stream when
// it reads the count.
cudaError_t launch_sort_rows(const int32_t *ii_t, const uint16_t *ii16, int ii_stride, int w,
                             const DevFeature *feat, int64_t f0, int64_t nf, const WeightLayout &L, uint16_t *rows,
                             int npad, int32_t *scratch, cudaStream_t st) {
    if (nf <= 0) return cudaSuccess;
    const int n = L.n;
    int32_t *stat = scratch, *ovf = scratch + 2;
    cudaError_t e = cudaMemsetAsync(ovf, 0, sizeof(int32_t), st);
    if (e != cudaSuccess) return e;
    // the variant with the fewest idle items: TH threads of I items
#define VJB_PK_CASE(I, TH) \
    if (n <= (I) * (TH))   \
        e = launch_sort_packed<I, TH>(ii_t, ii16, ii_stride, w, feat, f0, nf, L, rows, npad, ovf, stat, st); \
    else
    VJB_PK_CASE(8, 128)
    VJB_PK_CASE(16, 128)
    VJB_PK_CASE(20, 128)
    VJB_PK_CASE(24, 128)
    VJB_PK_CASE(28, 128)
    VJB_PK_CASE(32, 128)
    VJB_PK_CASE(20, 256)
    VJB_PK_CASE(24, 256)
    VJB_PK_CASE(28, 256)
    VJB_PK_CASE(32, 256)
    VJB_PK_CASE(36, 256)
    VJB_PK_CASE(40, 256)
    VJB_PK_CASE(44, 256)
    VJB_PK_CASE(48, 256)
    VJB_PK_CASE(52, 256)
    VJB_PK_CASE(56, 256)
    VJB_PK_CASE(60, 256)
    VJB_PK_CASE(44, 384)
    VJB_PK_CASE(48, 384)
    VJB_PK_CASE(54, 384)
    VJB_PK_CASE(48, 512)
    VJB_PK_CASE(64, 512)
    e = cudaErrorInvalidValue;
#undef VJB_PK_CASE
    if (e != cudaSuccess) return e;
    int32_t count = 0;
    e = cudaMemcpyAsync(&count, ovf, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess || count == 0) return e;
    return launch_sort_wide(ii_t, ii_stride, w, feat, f0, count, L, rows, npad, ovf + 1, stat, st);
}

}  // namespace vjb
