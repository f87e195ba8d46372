// Per-round search for the least-error decision stump over every Haar feature
// (Sec. 2.3 step 2: eps_t = min over f, p, theta of sum_i w_i |h(x_i) - y_i|).
//
// For one feature, let the samples be taken in value order (the sorted table)
// and let D(s) = sum over the first s samples of v_i, v_i = +w_i for a face and
// -w_i for a non-face.  With T+ and T- the face and non-face weight totals, the
// stump that puts the first s samples "below" the threshold errs by
//     T+ - D(s)   for p = +1 (below is a face),
//     T- + D(s)   for p = -1 (above is a face),
// and only splits between two different values are thresholds (bit 15 of the
// entry before the split; s = 0 is always one).  So the feature's least error
// is min(T+ - max D, T- + min D) over valid splits.
//
// A search is two steps:
//  * k_screen (the hot kernel): streams the whole uint16 table once per round
//    with TMA, gathers v from shared memory, and forms D with FP32 prefix sums.
//    A warp scans one row: lane k walks its own run of the value order (the
//    row layout interleaves 32 runs), summing 16 or 24 entries at a time in
//    FP32 and folding each piece into a compensated (TwoSum) running total; one
//    FP32 warp scan of the 32 run totals per row places every lane's best
//    prefix in the row.  It writes each feature's FP32 error and each CTA's
//    minimum.
//  * the round's tail (k_tail.cu) lists every feature whose screened error is
//    within a margin of the smallest one and scans the listed rows again in
//    double-float (compensated FP32) arithmetic throughout, giving each one's
//    best split, polarity and an error to about 1e-14 relative; the round's
//    stump is the best of them: lowest error, then feature, split, +1 before -1.
//
// Screening error bound (u = 2^-24, sum |v| = T+ + T- = 1 after normalising):
// a piece's partial sums of at most 24 terms err by at most 24u times the
// piece's |v| mass; the compensated run total adds O(u^2); placing the
// piece's extreme on the run total adds 2u |D|; rounding the 32 run totals
// to FP32 adds u, their five-level FP32 scan 5u (each total passes through
// at most five additions, sum |run totals| <= 1), and placing a lane's
// extreme on its run offset u |D|; forming T+- -/+ D in FP32 adds 2u.  So
// |screened - exact| <= 35u.  A margin of 72u (twice 36u) keeps every
// feature that could beat the best one.
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "k_search.cuh"

namespace vjb {

// Dynamic shared memory of k_screen: the weight array at the base, then (from
// the next 1 KiB boundary) the per-warp TMA rings, their mbarriers and the
// per-warp minima.
size_t search_smem_bytes(const SearchShape &s, int words) {
    size_t b = align_up((size_t)words * 4, 16);
    b += 1024;  // alignment of the rings to 1 KiB
    b += (size_t)s.warps * s.stages * s.box_lines * kLineBytes;
    b += (size_t)s.warps * s.stages * 8;
    b += (size_t)s.warps * 4 + 16;
    return b;
}

WeightLayout make_layout(int n, bool allow_dual) {
    WeightLayout L;
    L.n = n;
    const int off_b = (int)align_up((size_t)n + 1, 32);
    // table entries hold 15-bit word offsets: copy B takes what is left of the
    // 32,768 words after copy A, whole 32-sample blocks (all n while n <= 16,351)
    const int room = off_b < 32768 ? (32768 - off_b) / 32 * 32 : 0;
    L.nb = allow_dual ? (n < room ? n : room) : 0;
    L.dual = L.nb > 0 ? 1 : 0;
    L.off_b = L.dual ? off_b : 0;
    L.words = L.dual ? off_b + (int)align_up((size_t)L.nb, 32) : (int)align_up((size_t)n + 1, 4);
    return L;
}

template <int U>
__global__ void __launch_bounds__(U >= 4 ? 384 : (U == 3 ? 512 : 640), 1)
    k_screen(const __grid_constant__ CUtensorMap tmap, const float *__restrict__ v, int words,
             int lines_per_row, int box_lines, int stage_lines, int64_t nfeat,
             int stages, RoundState *rs, float *__restrict__ ferr, float *__restrict__ bmin) {
    if (rs->status != VJB_OK) return;
    extern __shared__ __align__(16) float sv[];  // weights at the base of dynamic shared memory
    const int nw = blockDim.x >> 5;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sv32 = smem_u32(sv);
    const uint32_t stage_bytes = (uint32_t)stage_lines * kLineBytes;  // a multiple of 1 KiB
    const uint32_t ring0 = (uint32_t)align_up(sv32 + (uint32_t)words * 4u, 1024);
    const uint32_t bars0 = ring0 + (uint32_t)nw * stages * stage_bytes;
    float *wbest = reinterpret_cast<float *>(reinterpret_cast<char *>(sv) + (bars0 + nw * stages * 8 - sv32));

    const uint32_t ring_w = ring0 + (uint32_t)warp * stages * stage_bytes;
    const uint32_t bar_w = bars0 + (uint32_t)(warp * stages * 8);
    if (lane == 0) {
        for (int s = 0; s < stages; ++s) mbar_init(bar_w + 8 * s, 1);
        fence_barrier_init();
    }

    // rows gw, gw + G, ... of this warp; feature indices fit int32 (nfeat <
    // 2^31), and so does the warp's chunk count (G >= 152 warps, at most 128
    // chunks per row)
    const int gw = blockIdx.x * nw + warp;
    const int G = gridDim.x * nw;
    const int nf_w = gw < nfeat ? (int)((nfeat - 1 - gw) / G) + 1 : 0;
    const int nc = (lines_per_row + box_lines - 1) / box_lines;
    const int total = nf_w * nc;
    const uint32_t tx = (uint32_t)box_lines * kLineBytes;

    // producer state (lane 0): the next chunk to load, in this warp's order
    int issued = 0, prow = gw, pline = 0, pstage = 0;
    const int last_line = (nc - 1) * box_lines;
    auto issue_next = [&]() {
        if (issued >= total) return;
        const uint32_t bar = bar_w + 8u * (uint32_t)pstage;
        mbar_arrive_expect_tx(bar, tx);
        tma_load_3d(ring_w + (uint32_t)pstage * stage_bytes, &tmap, 0, pline, prow, bar);
        if (pline == last_line) { pline = 0; prow += G; } else { pline += box_lines; }
        if (++pstage == stages) pstage = 0;
        ++issued;
    };
    if (lane == 0)
        for (int s = 0; s < stages; ++s) issue_next();
    __syncwarp();
    // the weights, staged while the first copies of the table are in flight
    stage_weights(sv, v, words);
    __syncthreads();

    const float Tp = (float)rs->t_pos, Tm = (float)rs->t_neg;
    float best = INFINITY;
    int cstage = 0;
    uint32_t cpar = 0;  // consumer ring position and mbarrier phase
    int consumed = 0;
    bool ok = true;
    const int crs_full = box_lines >> 2;                          // chunk rows of a full stage
    const int crs_last = (lines_per_row - (nc - 1) * box_lines) >> 2;  // and of a row's last one
    for (int k = 0; k < nf_w && ok; ++k) {
        const int f = gw + k * G;
        float ahi = 0.f, alo = 0.f, bmx = -INFINITY, bmn = INFINITY;
        // one stage: wait for its copy, scan it, give the slot its next copy
        auto stage_step = [&](auto scan) -> bool {
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar_w + 8u * (uint32_t)cstage, cpar))) return false;
            scan(ring_w + (uint32_t)cstage * stage_bytes);
            __syncwarp();
            if (lane == 0) {
                fence_proxy_async_smem();
                issue_next();
            }
            if (++cstage == stages) { cstage = 0; cpar ^= 1u; }
            ++consumed;
            return true;
        };
        if (U == 3 && crs_full == 6) {
            // the default shape: the full stages in a loop of their own around
            // one call that the compiler schedules apart from the general stage
            // (0.787 -> 0.759 ms at 24x24 / 15k), then the row's last stage
            for (int c = 0; c < nc - 1 && ok; ++c)
                ok = stage_step([&](uint32_t sb) { scan_pieces<2, 3>(sb, 0, lane, sv, ahi, alo, bmx, bmn); });
            if (ok) ok = stage_step([&](uint32_t sb) { scan_stage<U>(sb, crs_last, lane, sv, ahi, alo, bmx, bmn); });
        } else {
            for (int c = 0; c < nc && ok; ++c)
                ok = stage_step([&](uint32_t sb) {
                    scan_stage<U>(sb, c == nc - 1 ? crs_last : crs_full, lane, sv, ahi, alo, bmx, bmn);
                });
        }
        if (!ok) break;
        const float e = finish_row(ahi, alo, bmx, bmn, Tp, Tm, lane);
        if (lane == 0) {
            ferr[f] = e;
            best = fminf(best, e);
        }
    }
    if (!ok) {
        // stop: record the failure and wait (bounded) for this warp's copies in flight
        if (lane == 0) {
            atomicOr(&rs->flags, kFlagWaitTimeout);
            // chunks issued but not consumed sit in the ring from the current stage on
            int st = cstage;
            uint32_t ph = cpar;
            const int pending = issued - consumed;
            for (int s = 0; s < pending; ++s) {
                mbar_wait_bounded(bar_w + 8u * (uint32_t)st, ph, 100000000ull);
                if (++st == stages) { st = 0; ph ^= 1u; }
            }
        }
        __syncwarp();
    }
    if (lane == 0) wbest[warp] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = INFINITY;
        for (int w = 0; w < nw; ++w) m = fminf(m, wbest[w]);
        bmin[blockIdx.x] = m;
    }
}

cudaError_t launch_screen(const CUtensorMap *tmap, const float *v, const WeightLayout &L,
                          int lines_per_row, int box_lines, int64_t nfeat, const SearchShape &shape,
                          int grid, RoundState *rs, float *ferr, float *bmin, cudaStream_t st) {
    const size_t sm = search_smem_bytes(shape, L.words);
    const int threads = shape.warps * 32;
    switch (shape.unroll) {
    case 1:
        k_screen<1><<<grid, threads, sm, st>>>(*tmap, v, L.words, lines_per_row, box_lines,
                                               shape.box_lines, nfeat, shape.stages, rs, ferr, bmin);
        break;
    case 4:
        k_screen<4><<<grid, threads, sm, st>>>(*tmap, v, L.words, lines_per_row, box_lines,
                                               shape.box_lines, nfeat, shape.stages, rs, ferr, bmin);
        break;
    case 3:
        k_screen<3><<<grid, threads, sm, st>>>(*tmap, v, L.words, lines_per_row, box_lines,
                                               shape.box_lines, nfeat, shape.stages, rs, ferr, bmin);
        break;
    default:
        k_screen<2><<<grid, threads, sm, st>>>(*tmap, v, L.words, lines_per_row, box_lines,
                                               shape.box_lines, nfeat, shape.stages, rs, ferr, bmin);
    }
    return cudaGetLastError();
}

cudaError_t set_screen_smem_limit(int bytes) {
    cudaError_t e = cudaFuncSetAttribute(k_screen<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_screen<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_screen<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_screen<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e;
}

int screen_max_warps(int unroll) { return unroll >= 4 ? 12 : (unroll == 3 ? 16 : 20); }

int screen_occupancy(const SearchShape &s, int words) {
    int blocks = 0;
    cudaError_t e;
    const size_t sm = search_smem_bytes(s, words);
    if (s.unroll == 1) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_screen<1>, s.warps * 32, sm);
    else if (s.unroll == 4) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_screen<4>, s.warps * 32, sm);
    else if (s.unroll == 3) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_screen<3>, s.warps * 32, sm);
    else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_screen<2>, s.warps * 32, sm);
    return e == cudaSuccess ? blocks : 0;
}

}  // namespace vjb

namespace vjb {

// ---- allocation-free variant of the search kernel --------------------------------------
// Some callers cannot call cudaMalloc at the moment they want a search: a
// real-time loop whose memory is fixed up front, or a framework that hands all
// device memory to its own pool.  vjb_screen_noalloc serves them: the caller passes the sorted table,
// the signed weights and the outputs, and the only scratch the search needs --
// one (error, feature) partial per CTA plus a completion counter for the
// last-CTA reduction -- lives in the file-scope array below.  Every GPU that
// loads this library holds the array (8.4 KiB) until the process exits, and
// every call shares it.
constexpr int kNoAllocMaxCtas = 1024;
constexpr int kNoAllocWords = 2 * kNoAllocMaxCtas + 64;
constexpr int kNoAllocDone = 2 * kNoAllocMaxCtas;      // completion counter
constexpr int kNoAllocFlags = 2 * kNoAllocMaxCtas + 1; // error flags of the call
static __device__ __align__(256) uint32_t g_noalloc_scratch[kNoAllocWords];

// Stage of the caller's table: 16 lines, 1,024 entries of the value order.
// Lane l takes half a line, 32 neighbouring entries.
constexpr int kNoAllocLines = 16;
constexpr int kNoAllocStage = kNoAllocLines * kLineBytes;
// The weights take the whole 15-bit index range, zero from n on, so that an
// entry above n reads as padding without a clamp at every gather.
constexpr int kNoAllocWeights = 32768;

// Dynamic shared memory of k_screen_noalloc: the TMA rings first (1 KiB
// aligned), then the weights, the mbarriers and the per-warp minima.
static size_t noalloc_smem_bytes(const SearchShape &s) {
    size_t b = 1024;
    b += (size_t)s.warps * s.stages * kNoAllocStage;
    b += (size_t)kNoAllocWeights * 4;
    b += (size_t)s.warps * s.stages * 8;
    b += (size_t)s.warps * 4;
    return b;
}

// Predicated running max/min: update only where `flag` is set (a valid split).
__device__ __forceinline__ void minmax_if(uint32_t flag, float a, float &mx, float &mn) {
    asm("{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %2, 0;\n\t"
        "@p max.f32 %0, %0, %3;\n\t"
        "@p min.f32 %1, %1, %3;\n\t}"
        : "+f"(mx), "+f"(mn)
        : "r"(flag), "f"(a));
}

// One stage of a row.  The lane's 32 entries are two pieces of 16 summed from
// zero side by side; their largest and smallest prefixes at valid splits are
// placed on the row by an FP32 scan of the 32 lanes' totals and the
// compensated sum of the stages before (chi + clo).  Lines past the row's end
// arrive as zeros: no flags, and their sums come after every split of the row.
//
// What bounds it: the shared-memory pipe (81% busy under ncu, ALU 53%).  The
// caller's order is one random gather an entry, 3.5 wavefronts a warp
// instruction, against 2 with the two bank-balanced copies of k_screen; with
// the rest 4.4 wavefronts per 32 entries, 218 us at 16x16 / 15,000 if the pipe
// never waited.  A scan per 1,024 entries instead of per 512, no clamps at the
// gathers, the weights staged behind the first copies and 16 warps instead of
// 8: 452 -> 281 us a call there (3.46 TB/s).  Weights first in shared memory
// (constant gather addresses) were slower, 299 us, and so were entries taken two
// at a time as in k_screen (scan_two), 305 us.
__device__ __forceinline__ void screen_stage_plain(uint32_t sbase, int lane, const float *__restrict__ sv, float &chi,
                                                   float &clo, float &MX, float &MN) {
    // chunk c of line l is stored at chunk c ^ (l mod 8) (128-byte swizzle):
    // eight lanes (four lines) cover all the banks
    const uint32_t line = (uint32_t)lane >> 1, first = ((uint32_t)lane & 1u) * 4u;
    const uint32_t at = sbase + line * kLineBytes;
    uint32_t w[2][8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint4 q = lds128(at + (((first + c) ^ (line & 7u)) << 4));
        uint32_t *x = w[c >> 1] + 4 * (c & 1);
        x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
    }
    float g[2][16];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            g[u][2 * j] = sv[w[u][j] & kIndexMask];
            g[u][2 * j + 1] = sv[(w[u][j] >> 16) & kIndexMask];
        }
    float a[2] = {0.f, 0.f}, mx[2] = {-INFINITY, -INFINITY}, mn[2] = {INFINITY, INFINITY};
#pragma unroll
    for (int j = 0; j < 16; ++j)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            a[u] += g[u][j];
            minmax_if(w[u][j >> 1] & ((j & 1) ? 0x80000000u : 0x8000u), a[u], mx[u], mn[u]);
        }
    const float own = a[0] + a[1];
    float x = own;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    float excl = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0) excl = 0.f;
    const float b0 = chi + (clo + excl), b1 = chi + (clo + (excl + a[0]));
    MX = fmaxf(MX, fmaxf(b0 + mx[0], b1 + mx[1]));
    MN = fminf(MN, fminf(b0 + mn[0], b1 + mn[1]));
    float s, e;
    two_sum(chi, __shfl_sync(0xffffffffu, x, 31), s, e);
    chi = s;
    clo += e;
}

__global__ void __launch_bounds__(512, 1)
    k_screen_noalloc(const __grid_constant__ CUtensorMap tmap, const float *__restrict__ v, int n,
                     int lines_per_row, int box_lines, int64_t nfeat, int stages, float Tp,
                     float Tm, float *__restrict__ ferr, float *__restrict__ best_err,
                     int32_t *__restrict__ best_feature, uint32_t *__restrict__ scratch) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>(align_up(reinterpret_cast<size_t>(smem_raw), 1024));
    const int nw = blockDim.x >> 5;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *rings = base;
    float *sv = reinterpret_cast<float *>(rings + (size_t)nw * stages * kNoAllocStage);
    uint64_t *bars = reinterpret_cast<uint64_t *>(sv + kNoAllocWeights);
    float *wbest = reinterpret_cast<float *>(bars + nw * stages);
    __shared__ int32_t wfeat[16];
    __shared__ bool last_cta;

    const uint32_t ring_w = smem_u32(rings + (size_t)warp * stages * kNoAllocStage);
    const uint32_t bar_w = smem_u32(bars + warp * stages);
    if (lane == 0) {
        for (int s = 0; s < stages; ++s) mbar_init(bar_w + 8 * s, 1);
        fence_barrier_init();
    }
    // rows shorter than a stage: the lines no copy writes hold zeros, as the
    // lines past a longer row's end do
    for (int s = 0; s < stages; ++s)
        for (int i = box_lines * kLineBytes + 16 * lane; i < kNoAllocStage; i += 16 * 32)
            *reinterpret_cast<uint4 *>(rings + (size_t)(warp * stages + s) * kNoAllocStage + i) = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();

    const int64_t gw = (int64_t)blockIdx.x * nw + warp;
    const int64_t G = (int64_t)gridDim.x * nw;
    const int64_t nf_w = gw < nfeat ? (nfeat - 1 - gw) / G + 1 : 0;
    const int nc = (lines_per_row + box_lines - 1) / box_lines;
    const int64_t total = nf_w * nc;
    const uint32_t tx = (uint32_t)box_lines * kLineBytes;
    // producer (lane 0): the next stage to load, in this warp's order
    int64_t issued = 0, prow = gw;
    int pline = 0, pstage = 0;
    auto issue_next = [&]() {
        if (issued >= total) return;
        const uint32_t bar = bar_w + 8u * (uint32_t)pstage;
        mbar_arrive_expect_tx(bar, tx);
        tma_load_3d(ring_w + (uint32_t)pstage * kNoAllocStage, &tmap, 0, pline, (int32_t)prow, bar);
        pline += box_lines;
        if (pline >= lines_per_row) { pline = 0; prow += G; }
        if (++pstage == stages) pstage = 0;
        ++issued;
    };
    if (lane == 0)
        for (int s = 0; s < stages; ++s) issue_next();
    __syncwarp();
    // the weights, staged while the first copies are in flight
    for (int i = threadIdx.x; i < kNoAllocWeights; i += blockDim.x) sv[i] = i < n ? v[i] : 0.f;
    __syncthreads();

    float best = INFINITY;
    int32_t bestf = 0x7fffffff;
    int64_t consumed = 0;
    int cstage = 0;
    uint32_t cpar = 0;
    bool ok = true;
    for (int64_t k = 0; k < nf_w && ok; ++k) {
        const int64_t f = gw + k * G;
        float chi = 0.f, clo = 0.f, MX = 0.f, MN = 0.f;
        for (int c = 0; c < nc; ++c) {
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar_w + 8u * (uint32_t)cstage, cpar))) {
                ok = false;
                break;
            }
            screen_stage_plain(ring_w + (uint32_t)cstage * kNoAllocStage, lane, sv, chi, clo, MX, MN);
            __syncwarp();
            if (lane == 0) {
                fence_proxy_async_smem();
                issue_next();
            }
            if (++cstage == stages) { cstage = 0; cpar ^= 1u; }
            ++consumed;
        }
        if (!ok) break;
        // (a min does not round: the least of the lanes' errors is the row's)
        const float e = float_from_order_key(__reduce_min_sync(0xffffffffu, float_order_key(fminf(Tp - MX, Tm + MN))));
        if (lane == 0) {
            ferr[f] = e;
            if (e < best) { best = e; bestf = (int32_t)f; }
        }
    }
    if (!ok && lane == 0) {
        atomicOr(&scratch[kNoAllocFlags], (uint32_t)kFlagWaitTimeout);
        for (const int64_t pending = issued; consumed < pending; ++consumed) {
            mbar_wait_bounded(bar_w + 8u * (uint32_t)cstage, cpar, 100000000ull);
            if (++cstage == stages) { cstage = 0; cpar ^= 1u; }
        }
    }
    __syncwarp();
    if (lane == 0) { wbest[warp] = best; wfeat[warp] = bestf; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = INFINITY;
        int32_t mf = 0x7fffffff;
        for (int w = 0; w < nw; ++w)
            if (wbest[w] < m || (wbest[w] == m && wfeat[w] < mf)) { m = wbest[w]; mf = wfeat[w]; }
        scratch[blockIdx.x] = __float_as_uint(m);
        scratch[kNoAllocMaxCtas + blockIdx.x] = (uint32_t)mf;
        __threadfence();
        last_cta = atomicAdd(&scratch[kNoAllocDone], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last_cta && threadIdx.x == 0) {
        __threadfence();
        float m = INFINITY;
        int32_t mf = -1;
        for (unsigned b = 0; b < gridDim.x; ++b) {
            const float e = __uint_as_float(((volatile uint32_t *)scratch)[b]);
            const int32_t f = (int32_t)((volatile uint32_t *)scratch)[kNoAllocMaxCtas + b];
            if (e < m || (e == m && f < mf)) { m = e; mf = f; }
        }
        // a wait that gave up leaves rows unscanned: no minimum to report
        const bool failed = ((volatile uint32_t *)scratch)[kNoAllocFlags] != 0u;
        *best_err = failed ? __int_as_float(0x7fc00000) : m;
        *best_feature = failed ? -1 : mf;
        scratch[kNoAllocDone] = 0u;  // the next call starts from zero
    }
}

}  // namespace vjb

namespace {

typedef CUresult (*NoAllocEncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                    const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                    const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct NoAllocDevice {
    bool ready = false;
    uint32_t *scratch = nullptr;  // device address of g_noalloc_scratch on this device
    int num_sms = 0;
    int max_smem = 0;             // dynamic shared memory the kernel may use
};
constexpr int kNoAllocDevices = 64;
NoAllocDevice g_noalloc_dev[kNoAllocDevices];
NoAllocEncodeFn g_noalloc_encode = nullptr;
std::mutex g_noalloc_mu;

}  // namespace

namespace vjb {
int report_error(int code, const char *msg);
}

extern "C" int vjb_screen_noalloc(const uint16_t *rows, const float *v, int32_t n, int32_t npad,
                                  int64_t nfeat, double t_pos, double t_neg, int32_t ctas,
                                  float *feature_err, float *best_err, int32_t *best_feature,
                                  void *cuda_stream) {
    using namespace vjb;
    if (!rows || !v || !feature_err || !best_err || !best_feature)
        return report_error(VJB_EINVAL, "vjb_screen_noalloc: NULL pointer argument");
    if (n < 1 || n > VJB_MAX_SAMPLES)
        return report_error(VJB_EINVAL, "vjb_screen_noalloc: n outside [1, VJB_MAX_SAMPLES]");
    if (npad < n || npad % kLineElems != 0)
        return report_error(VJB_EINVAL, "vjb_screen_noalloc: npad must be >= n and a multiple of 64");
    if (nfeat < 1 || nfeat > 0x7fffffffLL)
        return report_error(VJB_EINVAL, "vjb_screen_noalloc: nfeat outside [1, 2^31 - 1]");
    if ((reinterpret_cast<uintptr_t>(rows) & 15u) != 0)
        return report_error(VJB_EINVAL, "vjb_screen_noalloc: rows must be 16-byte aligned");
    if (!(t_pos >= 0.0) || !(t_neg >= 0.0) || !std::isfinite(t_pos) || !std::isfinite(t_neg))
        return report_error(VJB_EINVAL, "vjb_screen_noalloc: class totals must be finite and >= 0");
    if (ctas < 0 || ctas > kNoAllocMaxCtas)
        return report_error(VJB_EINVAL, "vjb_screen_noalloc: ctas outside [0, 1024] (the scratch array holds 1024 partials)");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocDevices)
        return report_error(VJB_ECUDA, "vjb_screen_noalloc: no usable current device");
    NoAllocDevice &D = g_noalloc_dev[dev];
    {
        // set-up, once per device, with that device current
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!D.ready) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p)
                return report_error(VJB_ECUDA, "vjb_screen_noalloc: cudaGetSymbolAddress of the scratch array failed");
            int optin = 0;
            cudaFuncAttributes fa;
            if (cudaDeviceGetAttribute(&D.num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
                cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
                cudaFuncGetAttributes(&fa, k_screen_noalloc) != cudaSuccess)
                return report_error(VJB_ECUDA, "vjb_screen_noalloc: device attribute query failed");
            // the kernel's own static shared memory comes out of the same per-CTA limit
            D.max_smem = optin - (int)fa.sharedSizeBytes;
            if (cudaFuncSetAttribute(k_screen_noalloc, cudaFuncAttributeMaxDynamicSharedMemorySize, D.max_smem) != cudaSuccess)
                return report_error(VJB_ECUDA, "vjb_screen_noalloc: setting the kernel's shared-memory limit failed");
            if (!g_noalloc_encode) {
                void *fn = nullptr;
                cudaDriverEntryPointQueryResult q;
                if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
                    q != cudaDriverEntryPointSuccess || !fn)
                    return report_error(VJB_ECUDA, "vjb_screen_noalloc: cuTensorMapEncodeTiled unavailable");
                g_noalloc_encode = reinterpret_cast<NoAllocEncodeFn>(fn);
            }
            D.scratch = static_cast<uint32_t *>(p);
            D.ready = true;
        }
    }
    const int grid = ctas ? ctas : std::min(D.num_sms, kNoAllocMaxCtas);
    const SearchShape tries[] = {{16, 3, 1, 1, kNoAllocLines}, {16, 2, 1, 1, kNoAllocLines}, {8, 2, 1, 1, kNoAllocLines}};
    const SearchShape *shape = nullptr;
    for (const auto &s : tries)
        if (noalloc_smem_bytes(s) <= (size_t)D.max_smem) { shape = &s; break; }
    if (!shape) return report_error(VJB_EINVAL, "vjb_screen_noalloc: the weights do not fit shared memory");
    const int lines = npad / kLineElems;
    const int box_lines = std::min(kNoAllocLines, lines);
    CUtensorMap tmap;
    cuuint64_t dims[3] = {(cuuint64_t)kLineElems, (cuuint64_t)lines, (cuuint64_t)nfeat};
    cuuint64_t strides[2] = {(cuuint64_t)kLineBytes, (cuuint64_t)lines * kLineBytes};
    cuuint32_t box[3] = {(cuuint32_t)kLineElems, (cuuint32_t)box_lines, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    if (g_noalloc_encode(&tmap, CU_TENSOR_MAP_DATA_TYPE_UINT16, 3, const_cast<uint16_t *>(rows), dims,
                         strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return report_error(VJB_EINVAL, "vjb_screen_noalloc: the table cannot be described by a tensor map");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // the counter and the flags must start at zero; the partials are all overwritten
    if (cudaMemsetAsync(D.scratch + kNoAllocDone, 0, 2 * sizeof(uint32_t), st) != cudaSuccess)
        return report_error(VJB_ECUDA, "vjb_screen_noalloc: clearing the scratch counter failed");
    k_screen_noalloc<<<grid, shape->warps * 32, noalloc_smem_bytes(*shape), st>>>(
        tmap, v, n, lines, box_lines, nfeat, shape->stages, (float)t_pos, (float)t_neg, feature_err,
        best_err, best_feature, D.scratch);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return report_error(VJB_ECUDA, cudaGetErrorString(e));
    return VJB_OK;
}
