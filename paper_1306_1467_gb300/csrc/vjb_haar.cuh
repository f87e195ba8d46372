// Haar feature values (Sec. 2.1-2.2) from the point-major integral images:
// one window, four windows per load, and the narrow-box form from the
// integral images modulo 2^16.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "vjb.h"

namespace vjb {

// Haar feature value from integral images stored point-major: point (px, py)
// of sample i is at ii_t[(py * (w + 1) + px) * stride + i].  Rectangle sums use
// the four corners of Sec. 2.1 (4 + 1 - (2 + 3)); the combination per type is
// the dark-minus-white reading documented in vjb.h.
__device__ __forceinline__ int32_t haar_value(const int32_t *__restrict__ ii_t, int stride,
                                              int w, int type, int x, int y, int fw, int fh,
                                              int i) {
    const int W1 = w + 1;
    auto P = [&](int px, int py) -> int32_t { return __ldg(ii_t + (size_t)(py * W1 + px) * stride + i); };
    auto R = [&](int rx, int ry, int rw, int rh) -> int32_t {
        return P(rx + rw, ry + rh) + P(rx, ry) - (P(rx + rw, ry) + P(rx, ry + rh));
    };
    switch (type) {
    case VJB_HAAR_2H: {
        const int a = fw >> 1;
        return R(x + a, y, a, fh) - R(x, y, a, fh);
    }
    case VJB_HAAR_2V: {
        const int b = fh >> 1;
        return R(x, y + b, fw, b) - R(x, y, fw, b);
    }
    case VJB_HAAR_3H: {
        const int a = fw / 3;
        return R(x + a, y, a, fh) - R(x, y, a, fh) - R(x + 2 * a, y, a, fh);
    }
    case VJB_HAAR_3V: {
        const int b = fh / 3;
        return R(x, y + b, fw, b) - R(x, y, fw, b) - R(x, y + 2 * b, fw, b);
    }
    default: {
        const int a = fw >> 1, b = fh >> 1;
        return R(x + a, y, a, b) + R(x, y + b, a, b) - R(x, y, a, b) - R(x + a, y + b, a, b);
    }
    }
}

// A feature's value as sums of integral-image points: the points added and
// those subtracted (`pos`, `neg`), from a loader P(px, py) of the points and
// an adder.  With C0, C1, ... the point columns (or rows) at the rectangles'
// edges, two rectangles give C0 - 2 C1 + C2 and three C0 - 2 C1 + 2 C2 - C3,
// bottom minus top (right minus left); four give -(x) (y) of two such pairs.
template <class V, class Load, class Add>
__device__ __forceinline__ void haar_sums(int type, int x, int y, int fw, int fh, Load P, Add add, V &pos, V &neg) {
    auto twice = [&](V a) { return add(a, a); };
    switch (type) {
    case VJB_HAAR_2H: {
        const int a = fw >> 1, b = y + fh;
        pos = add(add(P(x, b), P(x + fw, b)), twice(P(x + a, y)));
        neg = add(add(P(x, y), P(x + fw, y)), twice(P(x + a, b)));
        break;
    }
    case VJB_HAAR_2V: {
        const int a = fh >> 1, r = x + fw;
        pos = add(add(P(r, y), P(r, y + fh)), twice(P(x, y + a)));
        neg = add(add(P(x, y), P(x, y + fh)), twice(P(r, y + a)));
        break;
    }
    case VJB_HAAR_3H: {
        const int a = fw / 3, b = y + fh;
        pos = add(add(P(x, b), P(x + fw, y)), twice(add(P(x + 2 * a, b), P(x + a, y))));
        neg = add(add(P(x, y), P(x + fw, b)), twice(add(P(x + 2 * a, y), P(x + a, b))));
        break;
    }
    case VJB_HAAR_3V: {
        const int a = fh / 3, r = x + fw;
        pos = add(add(P(r, y), P(x, y + fh)), twice(add(P(r, y + 2 * a), P(x, y + a))));
        neg = add(add(P(x, y), P(r, y + fh)), twice(add(P(x, y + 2 * a), P(r, y + a))));
        break;
    }
    default: {
        const int a = fw >> 1, b = fh >> 1, r = x + fw, t = y + fh;
        pos = twice(add(add(P(x + a, y), P(x + a, t)), add(P(x, y + b), P(r, y + b))));
        neg = add(add(add(P(x, y), P(r, y)), add(P(x, t), P(r, t))), twice(twice(P(x + a, y + b))));
        break;
    }
    }
}

// haar_value for the four windows i .. i + 3 (i a multiple of 4, the row
// stride a multiple of 4): one 16-byte load per corner.
__device__ __forceinline__ int4 haar_value4(const int32_t *__restrict__ ii_t, int stride, int w, int type,
                                            int x, int y, int fw, int fh, int i) {
    const int W1 = w + 1;
    int4 p, q;
    haar_sums<int4>(
        type, x, y, fw, fh,
        [&](int px, int py) { return __ldg(reinterpret_cast<const int4 *>(ii_t + (size_t)(py * W1 + px) * stride + i)); },
        [](int4 a, int4 b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }, p, q);
    return make_int4(p.x - q.x, p.y - q.y, p.z - q.z, p.w - q.w);
}

// Area of a feature's subtracted rectangles: its value lies in
// [-255 * neg, 255 * (fw * fh - neg)], a range 255 * fw * fh wide (the
// rectangles tile the fw x fh box; pixels are 0..255).
__device__ __forceinline__ int haar_neg_area(int type, int fw, int fh) {
    switch (type) {
    case VJB_HAAR_3H: return 2 * (fw / 3) * fh;
    case VJB_HAAR_3V: return 2 * fw * (fh / 3);
    default: return fw * fh / 2;  // 2H (fw even), 2V (fh even), four-rectangle (both even)
    }
}

// Largest box (fw * fh) whose values span at most 2^16 integers: 255 * 257 =
// 65535.
constexpr int kNarrowArea = 257;

// Two 16-bit sums in one word.
__device__ __forceinline__ uint32_t add16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("add.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// A feature with fw * fh <= kNarrowArea on the four windows i .. i + 3 (i and
// the row stride multiples of 4) from the integral images modulo 2^16 (ii16,
// same layout): one 8-byte load per corner, two windows to a word.  The corner
// combination is exact modulo 2^16, and the value is the one integer of its
// residue class in [-255 * neg, -255 * neg + 65535]; returned are the four
// values' offsets from the lower end of that range, 16 bits each.
__device__ __forceinline__ uint2 haar_offsets4(const uint16_t *__restrict__ ii16, int stride, int w, int type,
                                               int x, int y, int fw, int fh, int i) {
    const int W1 = w + 1;
    uint2 p, q;
    haar_sums<uint2>(
        type, x, y, fw, fh,
        [&](int px, int py) { return __ldg(reinterpret_cast<const uint2 *>(ii16 + (size_t)(py * W1 + px) * stride + i)); },
        [](uint2 a, uint2 b) { return make_uint2(add16x2(a.x, b.x), add16x2(a.y, b.y)); }, p, q);
    // p - q + 255 neg, the subtraction as ~q + 1
    const uint32_t up = ((uint32_t)(255 * haar_neg_area(type, fw, fh) + 1) & 0xffffu) * 0x10001u;
    return make_uint2(add16x2(add16x2(p.x, up), ~q.x), add16x2(add16x2(p.y, up), ~q.y));
}

}  // namespace vjb
