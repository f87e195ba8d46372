// Integral images of 32 windows in shared memory (Sec. 2.1), a lane per
// window: the pieces that the preparation's integral kernel and the
// classifier share.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vjb {

constexpr int kTileWindows = 32;

// Words from one window's pixels to the next in shared memory: odd, so that
// the 32 lanes' bytes at one offset sit in 32 banks.
__host__ __device__ __forceinline__ int tile_stride(int bytes) { return ((bytes + 3) >> 2) | 1; }

// Pixels [off, off + len) of windows i0 .. i0 + 31 (those below n) into
// `tile`, a warp per window: whole words where every window's part starts on
// one (px is a device allocation), else bytes.
__device__ __forceinline__ void stage_pixels(const uint8_t *__restrict__ px, int i0, int n, int hw, int off, int len,
                                             uint32_t *tile, int stride) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int count = min(kTileWindows, n - i0);
    if (((hw | off | len) & 3) == 0) {
        for (int i = warp; i < count; i += nw) {
            const uint32_t *src = reinterpret_cast<const uint32_t *>(px + (size_t)(i0 + i) * hw + off);
            for (int k = lane; k < len >> 2; k += 32) tile[i * stride + k] = __ldg(src + k);
        }
    } else {
        for (int i = warp; i < count; i += nw) {
            const uint8_t *src = px + (size_t)(i0 + i) * hw + off;
            uint8_t *dst = reinterpret_cast<uint8_t *>(tile + i * stride);
            for (int k = lane; k < len; k += 32) dst[k] = __ldg(src + k);
        }
    }
}

// Running sums along `rows` rows of w staged pixels, a warp per row, to
// sums[(y * pitch + x) * 32 + lane].
__device__ __forceinline__ void row_sums(const uint32_t *tile, int stride, int rows, int w, int32_t *sums, int pitch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint8_t *mine = reinterpret_cast<const uint8_t *>(tile + lane * stride);
    for (int y = warp; y < rows; y += nw) {
        int32_t s = 0;
#pragma unroll 4
        for (int x = 0; x < w; ++x) {
            s += mine[y * w + x];
            sums[(y * pitch + x) * 32 + lane] = s;
        }
    }
}

}  // namespace vjb
