// The strong classifier of Sec. 2.3 (the final hypothesis) applied to windows:
//     C(x) = 1  iff  sum_t alpha_t h_t(x) >= 1/2 sum_t alpha_t,
// h_t(x) = 1 iff p_t f_t(x) < p_t theta_t.  Every window's alpha_t are added in
// FP64 in stump order, so its score does not depend on the launch shape.
#include <math.h>

#include "vjb_device.cuh"
#include "vjb_haar.cuh"
#include "vjb_integral.cuh"
#include "vjb_internal.cuh"

namespace vjb {

constexpr int kClassifyThreads = 256;
constexpr int kClassifyStage = 256;  // stumps per shared-memory block

__device__ __forceinline__ bool stump_says(const ClassStump &c, int32_t v) {
    return c.polarity > 0 ? (v < c.threshold) : (v > c.threshold);
}

// From the windows' pixels: a CTA forms the integral images of 32 windows in
// shared memory (a lane each), its warps evaluate the stumps, 128 at a time, to
// one word of 32 answers a stump, and one warp adds the alphas in order while
// the others go on with the next 128.  The feature corners are shared-memory
// reads without bank conflicts, and nothing but the pixels is read from memory.
//
// What bounds it: the chain of FP64 additions for a few windows, the FP64 unit
// (a warp-wide addition holds it for about 16 cycles) for many.  24x24 windows,
// 200 stumps (ncu): 18 us for 200 windows and 302 us for 150,001; integral images
// through memory and one thread per window took 154 and 380 us.
constexpr int kFusedThreads = 512;
constexpr int kFusedStage = 128;  // stumps at a time

__host__ __device__ __forceinline__ size_t classify_words(int h, int w) {
    return (size_t)(h + 1) * (w + 1) * 32 + (size_t)32 * tile_stride(h * w);
}

__global__ void __launch_bounds__(kFusedThreads)
    k_classify_windows(const uint8_t *__restrict__ px, int n, int h, int w, const ClassStump *__restrict__ stumps, int T,
                       double half_alpha, uint8_t *__restrict__ labels, double *__restrict__ scores) {
    extern __shared__ __align__(16) int32_t ii[];  // [point][32], then the pixels
    __shared__ ClassStump sst[3][kFusedStage];
    __shared__ uint32_t says[2][kFusedStage];
    const int W1 = w + 1;
    uint32_t *tile = reinterpret_cast<uint32_t *>(ii + (size_t)(h + 1) * W1 * 32);
    const int tstride = tile_stride(h * w);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int i0 = blockIdx.x * kTileWindows, i = i0 + lane;
    stage_pixels(px, i0, n, h * w, 0, h * w, tile, tstride);
    for (int x = warp; x <= w; x += nw) ii[x * 32 + lane] = 0;
    for (int y = 1 + warp; y <= h; y += nw) ii[y * W1 * 32 + lane] = 0;
    auto stage_stumps = [&](int t0, int buf) {
        const int m = min(kFusedStage, T - t0);
        for (int k = threadIdx.x; k < m; k += blockDim.x) sst[buf][k] = stumps[t0 + k];
    };
    stage_stumps(0, 0);
    __syncthreads();
    row_sums(tile, tstride, h, w, ii + (W1 + 1) * 32, W1);
    __syncthreads();
    for (int x = 1 + warp; x <= w; x += nw) {
        int32_t v = 0;
#pragma unroll 4
        for (int y = 1; y <= h; ++y) {
            v += ii[(y * W1 + x) * 32 + lane];
            ii[(y * W1 + x) * 32 + lane] = v;
        }
    }
    __syncthreads();
    double s = 0.0;  // warp 0: lane's window
    // Part q of the stumps is held in sst[q mod 3] and its answers in says[q mod
    // 2]: while warp 0 adds up part q, the others evaluate part q + 1 and stage
    // part q + 2, and they wait for it before they go further.
    for (int q = 0, t0 = 0; t0 < T; ++q, t0 += kFusedStage) {
        const int m = min(kFusedStage, T - t0);
        const ClassStump *st = sst[q % 3];
        uint32_t *word = says[q & 1];
        for (int k = warp; k < m; k += nw) {
            const ClassStump c = st[k];
            int32_t pos, neg;
            haar_sums<int32_t>(
                c.f.type, c.f.x, c.f.y, c.f.w, c.f.h, [&](int x, int y) { return ii[(y * W1 + x) * 32 + lane]; },
                [](int32_t a, int32_t b) { return a + b; }, pos, neg);
            const uint32_t yes = __ballot_sync(0xffffffffu, stump_says(c, pos - neg));
            if (lane == 0) word[k] = yes;
        }
        stage_stumps(t0 + kFusedStage, (q + 1) % 3);
        __syncthreads();
        if (warp == 0) {
#pragma unroll 8
            for (int k = 0; k < m; ++k) s += (word[k] >> lane) & 1u ? st[k].alpha : 0.0;
        }
    }
    if (warp == 0 && i < n) {
        labels[i] = s >= half_alpha ? 1 : 0;
        if (scores) scores[i] = s;
    }
}

// Once per device, before the first launch (as set_integral_limits): what a CTA
// may have in all, `max_smem`, less what the kernel holds anyway.
cudaError_t set_classify_limits(int max_smem) {
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, k_classify_windows);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_classify_windows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                max_smem - (int)fa.sharedSizeBytes);
}

bool classify_fits(int h, int w) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, k_classify_windows) != cudaSuccess) return false;
    return classify_words(h, w) * 4 <= (size_t)fa.maxDynamicSharedSizeBytes;
}

cudaError_t launch_classify_windows(const uint8_t *px, int n, int h, int w, const ClassStump *stumps, int T,
                                    double half_alpha, uint8_t *labels, double *scores, cudaStream_t st) {
    const size_t sm = classify_words(h, w) * 4;
    k_classify_windows<<<(n + kTileWindows - 1) / kTileWindows, kFusedThreads, sm, st>>>(px, n, h, w, stumps, T,
                                                                                        half_alpha, labels, scores);
    return cudaGetLastError();
}

// Windows whose integral images do not fit shared memory (from about 40x40
// on): one thread per window, integral images through memory.
__global__ void __launch_bounds__(kClassifyThreads)
    k_strong_classify(const int32_t *__restrict__ ii_t, int ii_stride, int n, int win_w,
                      const ClassStump *__restrict__ stumps, int T, double half_alpha, uint8_t *__restrict__ labels, double *__restrict__ scores) {
    __shared__ ClassStump sst[kClassifyStage];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double s = 0.0;
    for (int t0 = 0; t0 < T; t0 += kClassifyStage) {
        const int m = min(kClassifyStage, T - t0);
        __syncthreads();
        for (int k = threadIdx.x; k < m; k += blockDim.x) sst[k] = stumps[t0 + k];
        __syncthreads();
        if (i < n)
            for (int k = 0; k < m; ++k) {
                const ClassStump &c = sst[k];
                const int32_t v = haar_value(ii_t, ii_stride, win_w, c.f.type, c.f.x, c.f.y, c.f.w, c.f.h, i);
                if (stump_says(c, v)) s += c.alpha;
            }
    }
    if (i < n) {
        labels[i] = s >= half_alpha ? 1 : 0;
        if (scores) scores[i] = s;
    }
}

cudaError_t launch_strong_classify(const int32_t *ii_t, int ii_stride, int n, int win_w, const ClassStump *stumps, int T,
                                   double half_alpha, uint8_t *labels, double *scores, cudaStream_t st) {
    const int grid = (n + kClassifyThreads - 1) / kClassifyThreads;
    k_strong_classify<<<grid, kClassifyThreads, 0, st>>>(ii_t, ii_stride, n, win_w, stumps, T, half_alpha, labels, scores);
    return cudaGetLastError();
}

}  // namespace vjb
