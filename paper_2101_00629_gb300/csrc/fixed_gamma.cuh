// FP64-grade covariance kernel values in 64-bit fixed point.
//
// GB300 issues 1.6 FP64 FMAs per clock and SM but 64 32-bit integer
// multiply-adds and 128 logic or add operations, so one FP64 operation costs
// as much as about eighty 32-bit ones. Evaluating exp(-t) and the distance in
// 64-bit integers therefore takes a tenth of the time of the FP64 formula at
// a smaller error: arguments carry 53 to 55 fraction bits whatever their
// size (an FP64 argument t has a rounding error of t 2^-53, which the
// exponential turns into a relative one), and the exponential itself is good
// to 2^-56.
//
// Coordinates are held as x s 2^Q modulo 2^64, s the scale that turns a
// distance into a base-2 exponent (log2(e) / L for the exponential kernels,
// sqrt(log2 e) / L for the Gaussian, ...). Differences of such numbers are
// right whenever the true difference fits, whatever the offset of the domain.
// Every function here also compiles for the host, where its error is tested.
#pragma once

#include <cmath>
#include <cstdint>

#include "../../include/kl.h"

namespace kl {
namespace fx {

// Fraction bits of the coordinates (kCoord) and of the exponent t (kArg).
// A coordinate difference is a signed 64-bit number: it is right for
// |difference| < 64 (Gauss) or 256. kMaxArg keeps each difference and the
// exponent in range, with room for the rounding of the bounds: Gauss t < 2048,
// |difference| <= sqrt(1000); separable exponential t < 512, |difference| <= t;
// Euclidean ones |difference| < 128 (the norm scales three squares to 62 bits).
template <int KIND>
struct Format {
    static constexpr int kCoord = KIND == KL_KERNEL_GAUSS ? 57 : 55;
    static constexpr int kArg = KIND == KL_KERNEL_GAUSS ? 53 : 55;
    // largest exponent the fixed-point evaluation takes
    static constexpr float kMaxArg = KIND == KL_KERNEL_GAUSS ? 1000.0f : KIND == KL_KERNEL_EXP_SEP ? 250.0f : 120.0f;
};

__host__ __device__ inline uint32_t mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return uint32_t((uint64_t(a) * b) >> 32);
#endif
}
__host__ __device__ inline uint64_t mulwide(uint32_t a, uint32_t b) { return uint64_t(a) * b; }
// a b + c, one multiply-add each
__host__ __device__ inline uint64_t madwide(uint32_t a, uint32_t b, uint64_t c) {
#ifdef __CUDA_ARCH__
    uint64_t d;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return uint64_t(a) * b + c;
#endif
}
__host__ __device__ inline int64_t madwide_s(int32_t a, int32_t b, int64_t c) {
#ifdef __CUDA_ARCH__
    int64_t d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return int64_t(a) * b + c;
#endif
}
// high half of a 64 x 64-bit product, up to two units low
__host__ __device__ inline uint64_t mulhi64(uint64_t a, uint64_t b) {
    const uint32_t ah = uint32_t(a >> 32), bh = uint32_t(b >> 32);
    return madwide(ah, bh, mulhi32(ah, uint32_t(b))) + mulhi32(uint32_t(a), bh);
}

// 2^-(i / 2048) in units of 2^-63, i = 0..2047: products of the eleven
// factors 2^-(2^b / 2048), rounded to 64 bits (error of a product below
// 2^-60).
struct Exp2Table {
    uint64_t v[2048];
    static constexpr uint64_t mulhi(uint64_t a, uint64_t b) {
        const uint64_t al = a & 0xffffffffu, ah = a >> 32, bl = b & 0xffffffffu, bh = b >> 32;
        const uint64_t m = ah * bl + ((al * bl) >> 32);
        const uint64_t n = al * bh + (m & 0xffffffffu);
        return ah * bh + (m >> 32) + ((n + 0x80000000u) >> 32);
    }
    constexpr Exp2Table() : v{} {
        constexpr uint64_t f[11] = {0xffe9d2b2f7db2756ull, 0xffd3a751c0f7e10cull, 0xffa756521c8daed2ull,
                                    0xff4ecb59511ec8a5ull, 0xfe9e115c7b8f884cull, 0xfd3e0c0cf486c175ull,
                                    0xfa83b2db722a033aull, 0xf5257d152486cc2cull, 0xeac0c6e7dd24392full,
                                    0xd744fccad69d6af4ull, 0xb504f333f9de6484ull};
        for (int i = 0; i < 2048; ++i) {
            uint64_t t = uint64_t(1) << 63;
            for (int b = 0; b < 11; ++b)
                if (i >> b & 1) t = mulhi(t, f[b]);
            v[i] = t;
        }
    }
};

// 2^-frac(t) in units of 2^-63 and n = floor(t) for t with Q fraction bits:
// the table gives the leading 11 fraction bits, the cubic that
// Chebyshev-economises 1 - 2^-r on [0, 2^-11] (error 2^-57.7) the rest.
template <int Q>
__host__ __device__ __forceinline__ uint64_t exp2_neg(uint64_t t, const uint64_t* tab, uint32_t& n) {
    const uint32_t th = uint32_t(t >> 32), tl = uint32_t(t);
    n = th >> (Q - 32);
    const uint64_t T = tab[(th >> (Q - 43)) & 2047u];
    const uint32_t r = uint32_t(t >> (Q - 43));        // 2^-43
    const uint32_t rl = tl & ((1u << (Q - 43)) - 1u);  // 2^-Q, what r leaves
    const uint32_t v = 0xf5fdefcbu - (mulhi32(r, 0xe34e6d62u) >> 13);  // c2 - c3 r, 2^-34
    const uint32_t w = mulhi32(r, v);                                  // 2^-45
    // c1 r - w r, 2^-75
    uint64_t p = madwide(r, 0xb17217f7u, mulhi32(r, 0xd180aefeu));
    p = madwide(rl, Q == 55 ? 0xb1721u : 0x2c5c86u, p);
    p -= mulwide(r, w) >> 13;
    return T - (mulhi64(T, p) >> 11);
}

// |a - b| (one unit low where a < b)
__host__ __device__ __forceinline__ uint64_t absdiff(uint64_t a, uint64_t b) {
    const int64_t d = int64_t(a - b);
    return uint64_t(d ^ (d >> 63));
}

// sqrt(x^2 + y^2 + z^2) of fixed-point numbers below 2^62, same units, error
// about one unit: the sum of squares of the numbers shifted up to 62 bits, an
// approximate reciprocal square root in FP32 and two Newton corrections with
// exact integer residuals.
__host__ __device__ __forceinline__ uint64_t norm3(uint64_t x, uint64_t y, uint64_t z) {
    const uint32_t top = uint32_t((x | y | z) >> 32);
    if (top == 0) {  // closer than 2^-23: the squares are exact in FP64
        const double dx = double(x), dy = double(y), dz = double(z);
        return uint64_t(sqrt(dx * dx + dy * dy + dz * dz) + 0.5);
    }
#ifdef __CUDA_ARCH__
    const int sh = __clz(int(top)) - 2;
#else
    const int sh = __builtin_clz(top) - 2;
#endif
    x <<= sh;
    y <<= sh;
    z <<= sh;
    const uint32_t xh = uint32_t(x >> 32), yh = uint32_t(y >> 32), zh = uint32_t(z >> 32);
    // the sum of squares in units of 2^64: high parts and twice the cross
    // terms (the squares of the low parts are below one unit)
    const uint64_t C = madwide(xh, uint32_t(x), madwide(yh, uint32_t(y), mulwide(zh, uint32_t(z))));
    const uint64_t R = madwide(xh, xh, madwide(yh, yh, madwide(zh, zh, C >> 31)));  // in [2^58, 2^62)
    const float f = float(uint32_t(R >> 32));
#ifdef __CUDA_ARCH__
    float g;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(g) : "f"(f));
#else
    const float g = float(1.0 / std::sqrt(double(f)) * (1.0 + 1e-7));  // as inexact as the device's
#endif
    // r0 = sqrt(R) to 22 bits
    const uint32_t r0 = uint32_t(int(f * g * 128.0f + 0.5f)) << 9;
    const int64_t e = int64_t(R - mulwide(r0, r0));
    // sqrt(R) - r0 = e / (2 r0), in units of 2^-13
    const int32_t c = int32_t(float(int32_t(e >> 11)) * (g * 128.0f));
    // (R - (r0 + c 2^-13)^2) 2^26, exact modulo 2^64 and small
    const int64_t e1 = madwide_s(c, -c, int64_t((uint64_t(e) << 26) - (uint64_t(int64_t(int32_t(r0)) * c) << 14)));
    const int32_t c2 = int32_t(float(int32_t(e1 >> 18)) * (g * 128.0f));  // 2^-32
    const uint64_t r = (uint64_t(r0) << 32) + uint64_t(int64_t(c) * (1 << 19)) + uint64_t(int64_t(c2));
    return r >> sh;
}

// The exponent t (kArg fraction bits) of a pair; for Matern-3/2 the kernel is
// (1 + t ln 2) 2^-t.
template <int KIND>
__host__ __device__ __forceinline__ uint64_t exponent(uint64_t x, uint64_t y, uint64_t z) {
    if (KIND == KL_KERNEL_EXP_SEP) return x + y + z;
    if (KIND == KL_KERNEL_GAUSS) {
        // 2^-114 units -> 2^-53: drop 61 bits of the sum of squares
        const uint32_t xh = uint32_t(x >> 32), yh = uint32_t(y >> 32), zh = uint32_t(z >> 32);
        const uint32_t xl = uint32_t(x), yl = uint32_t(y), zl = uint32_t(z);
        const uint64_t H = madwide(xh, xh, madwide(yh, yh, mulwide(zh, zh)));
        const uint64_t L = mulwide((mulhi32(xl, xl) >> 2) + (mulhi32(yl, yl) >> 2) + (mulhi32(zl, zl) >> 2), 2u);
        const uint64_t C = madwide(xh, xl, madwide(yh, yl, madwide(zh, zl, L)));
        return (H << 3) + (C >> 28);
    }
    return norm3(x, y, z);
}

// 1 + t ln 2 (Matern-3/2), same units as t
__host__ __device__ __forceinline__ uint64_t matern_factor(uint64_t t) {
    const uint32_t th = uint32_t(t >> 32), tl = uint32_t(t);
    return madwide(th, 0xb17217f7u, (uint64_t(1) << 55) + mulhi32(th, 0xd1cf79acu)) + mulhi32(tl, 0xb17217f7u);
}

// E 2^-63 2^-n as FP64 (n < 1000)
__host__ __device__ __forceinline__ double to_double(uint64_t E, uint32_t n) {
    const uint64_t b = ((E + 512) >> 10) + (uint64_t(1021u - n) << 52);
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double d;
    __builtin_memcpy(&d, &b, 8);
    return d;
#endif
}

// x sm 2^se 2^Q modulo 2^64 (rounded towards minus infinity) for finite x
template <int Q>
__host__ __device__ inline uint64_t to_fixed(double x, uint64_t sm, int se) {
    uint64_t b;
#ifdef __CUDA_ARCH__
    b = uint64_t(__double_as_longlong(x));
#else
    __builtin_memcpy(&b, &x, 8);
#endif
    const int ef = int(b >> 52) & 2047;
    const uint64_t m = (b & 0xfffffffffffffull) | (ef ? uint64_t(1) << 52 : 0);
    // 128-bit product hi:lo
#ifdef __CUDA_ARCH__
    const uint64_t hi = __umul64hi(m, sm), lo = m * sm;
#else
    const unsigned __int128 pr = (unsigned __int128)m * sm;
    const uint64_t hi = uint64_t(pr >> 64), lo = uint64_t(pr);
#endif
    const int s = (ef ? ef : 1) - 1075 + se + Q;  // left shift of hi:lo
    uint64_t v;
    if (s >= 0) v = s < 64 ? lo << s : 0;
    else if (s > -64) v = (lo >> -s) | (hi << (64 + s));
    else v = s > -128 ? hi >> (-s - 64) : 0;
    return b >> 63 ? 0 - v : v;
}

}  // namespace fx
}  // namespace kl
