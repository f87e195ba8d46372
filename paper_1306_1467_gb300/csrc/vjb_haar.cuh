// Haar feature values (Sec. 2.1-2.2) from the point-major integral images:
// one window, all windows of a row, several a load, and the narrow-box form
// from the integral images modulo 2^16.
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

// A feature on every window of a CTA, a load's worth of windows a thread and
// step: calls each(q, pos, neg) for q = threadIdx.x, + TH, ... up to the last
// window, with haar_sums' two sums for the windows from q times that many on.
// Q is the type of a load along a point's line (the row stride is a multiple of
// 32 windows), `add` the adder on it.
//
// Along the split axis the points lie `s` apart on a near and, `t` further, a
// far line: two rectangles are far - near with 1, -2, 1, three with 1, -2, 2, -1
// and four the product of two such pairs.  The type is looked at and the points
// are placed once, outside the loop (32-bit places: 64-bit pointers spill, 15.4
// against 16.0 ms of tables at 24x24 / 15,000), and eight 16-bit windows a load
// instead of four halve the loads and addresses (15.4 -> 15.1 ms).
template <int TH, class Q, class T, class Add, class Each>
__device__ __forceinline__ void haar_rows(const T *__restrict__ ii, int stride, int w, int type, int x, int y, int fw,
                                          int fh, int n, Add add, Each each) {
    constexpr uint32_t kWin = sizeof(Q) / sizeof(T);
    const int W1 = w + 1;
    const Q *const o = reinterpret_cast<const Q *>(ii + (size_t)(y * W1 + x) * stride);
    const uint32_t line = (uint32_t)stride / kWin;  // places from the first point fit 32 bits: 256 * 256 lines of 8,192
    auto twice = [&](Q a) { return add(a, a); };
    auto along = [&](auto sums) {
        for (uint32_t q = threadIdx.x; kWin * q < (uint32_t)n; q += TH) sums(q, [&](uint32_t at) { return __ldg(o + (at + q)); });
    };
    if (type == VJB_HAAR_4) {
        const uint32_t s = line * (fw >> 1), t = line * W1 * (fh >> 1);
        const uint32_t c1 = s + 2 * t, c3 = t + 2 * s, e1 = 2 * s, e2 = 2 * t, e3 = e1 + e2, m = s + t;
        along([&](uint32_t q, auto P) {
            const Q pos = twice(add(add(P(s), P(c1)), add(P(t), P(c3))));
            const Q neg = add(add(add(P(0u), P(e1)), add(P(e2), P(e3))), twice(twice(P(m))));
            each((int)q, pos, neg);
        });
        return;
    }
    const bool across = type == VJB_HAAR_2H || type == VJB_HAAR_3H;
    const bool two = type == VJB_HAAR_2H || type == VJB_HAAR_2V;
    const int parts = two ? 2 : 3;
    const uint32_t s = line * (across ? fw / parts : W1 * (fh / parts)), t = line * (across ? W1 * fh : fw);
    const uint32_t n2 = 2 * s, f1 = t + s, f2 = f1 + s;
    if (two) {
        along([&](uint32_t q, auto P) {
            const Q pos = add(add(P(t), P(f2)), twice(P(s)));
            const Q neg = add(add(P(0u), P(n2)), twice(P(f1)));
            each((int)q, pos, neg);
        });
    } else {
        const uint32_t n3 = n2 + s, f3 = f2 + s;
        along([&](uint32_t q, auto P) {
            const Q pos = add(add(P(t), P(n3)), twice(add(P(f2), P(s))));
            const Q neg = add(add(P(0u), P(f3)), twice(add(P(n2), P(f1))));
            each((int)q, pos, neg);
        });
    }
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

// A feature with fw * fh <= kNarrowArea on every window, from the integral
// images modulo 2^16 (ii16, same layout): one 16-byte load per point, two windows
// to a word.  The combination of the points is exact modulo 2^16, and the value
// is the one integer of its residue class in [-255 * neg, -255 * neg + 65535];
// each(q, x) gets the eight values' offsets from the lower end of that range, 16
// bits each.
template <int TH, class Each>
__device__ __forceinline__ void haar_rows_narrow(const uint16_t *__restrict__ ii16, int stride, int w, int type, int x,
                                                 int y, int fw, int fh, int n, Each each) {
    // p - q + 255 neg, the subtraction as ~q + 1
    const uint32_t up = ((uint32_t)(255 * haar_neg_area(type, fw, fh) + 1) & 0xffffu) * 0x10001u;
    auto fin = [&](uint32_t p, uint32_t q) { return add16x2(add16x2(p, up), ~q); };
    haar_rows<TH, uint4>(
        ii16, stride, w, type, x, y, fw, fh, n,
        [](uint4 a, uint4 b) {
            return make_uint4(add16x2(a.x, b.x), add16x2(a.y, b.y), add16x2(a.z, b.z), add16x2(a.w, b.w));
        },
        [&](int k, uint4 p, uint4 q) { each(k, make_uint4(fin(p.x, q.x), fin(p.y, q.y), fin(p.z, q.z), fin(p.w, q.w))); });
}

}  // namespace vjb
