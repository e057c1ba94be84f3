// f64_int.cuh -- double-precision exp(-a^2) and division on the integer pipes.
//
// GB300 issues one double-precision warp instruction per SM quarter every 64
// cycles or so (1.0 TFLOP/s), and an exponential or a division is a chain of
// ten to twenty of them.  Both are evaluated here in 64-bit fixed point
// instead (largest errors measured: 0.66 ulp below |a| = 8 and 0.64 ulp, rms
// 0.294 and 0.291 where rounding alone gives 0.289), at about 85 and 45 issue
// slots, while the double-precision pipe works on the elimination.
// A 64-bit product's high half is three 32 x 32 -> 64 multiply-adds (the
// low halves' product is dropped: an error below two units of the result).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace mgx {

// 2^(j/1024), j = 0..1023, in Q1.62, from integer square roots of two.
struct Exp2Table {
    uint64_t v[1024];
    constexpr Exp2Table() : v() {
        uint64_t root[10] = {};  // 2^(2^-k), k = 10..1, in Q1.62
        unsigned __int128 x = (unsigned __int128)1 << 125;  // 2 in Q.124
        for (int k = 1; k <= 10; ++k) {
            uint64_t r = 0;  // floor(sqrt(x))
            for (int b = 62; b >= 0; --b) {
                const uint64_t t = r | (uint64_t(1) << b);
                if ((unsigned __int128)t * t <= x) r = t;
            }
            root[10 - k] = r;
            x = (unsigned __int128)r << 62;
        }
        for (int j = 0; j < 1024; ++j) {
            uint64_t p = uint64_t(1) << 62;
            for (int b = 0; b < 10; ++b)
                if (j >> b & 1) p = uint64_t(((unsigned __int128)p * root[b] + ((unsigned __int128)1 << 61)) >> 62);
            v[j] = p;
        }
    }
};

__host__ __device__ __forceinline__ uint32_t mul_hi32(uint32_t a, uint32_t b) {
    return uint32_t((uint64_t(a) * b) >> 32);
}

// High half of a b for a, b < 2^63, low by at most two units.
__host__ __device__ __forceinline__ uint64_t mul_hi63(uint64_t a, uint64_t b) {
    const uint32_t ah = uint32_t(a >> 32), al = uint32_t(a), bh = uint32_t(b >> 32), bl = uint32_t(b);
    uint64_t t = uint64_t(ah) * bl;
    t += uint64_t(al) * bh;
    return uint64_t(ah) * bh + (t >> 32);
}

__host__ __device__ __forceinline__ double bits_double(uint64_t b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double d;
    memcpy(&d, &b, 8);
    return d;
#endif
}

__host__ __device__ __forceinline__ uint64_t double_bits(double d) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(d);
#else
    uint64_t b;
    memcpy(&b, &d, 8);
    return b;
#endif
}

// 2^(-a^2) for |a| = A / 2^57 (Q7.57); 0 from |a| = 31 on (2^-961).
// a^2 = n + f; 2^(-a^2) = 2^-(n+1) 2^(1-f), 1 - f = j/1024 + r: the table's
// 2^(j/1024) times 1 + p(r), p the Taylor polynomial of 2^r - 1 to degree four
// (r < 2^-10: the next term is below 2^-59).  a^2 carries 56 fraction bits
// below |a| = 8 and 52 above, where g < 2^-64.
__host__ __device__ __forceinline__ double exp2_neg_sq(uint64_t A, const uint64_t *tab) {
    if (A >= (uint64_t(31) << 57)) return 0.0;
    const bool small = A < (uint64_t(1) << 60);
    const uint64_t M = A << (small ? 3 : 1);   // |a| / 8 or / 32 in Q0.63
    const uint64_t Y = mul_hi63(M, M);         // a^2 / 64 or / 1024 in Q0.62
    const uint32_t n = uint32_t(Y >> (small ? 56 : 52));
    const uint64_t F = ~(Y << (small ? 8 : 12));  // 1 - f in Q0.64 (less 2^-64)
    const uint64_t T = tab[F >> 54];
    const uint64_t R = (F << 9) & 0x7fffffffffffffffull;  // 2^10 r in Q0.63
    const uint32_t Rh = uint32_t(R >> 31);
    // ln2^k / k! 2^(-10 (k-1)) for k = 4..1, scaled by 2^24, 2^24, 2^12, 1
    const uint32_t v = mul_hi32(Rh, 645462u) + 3814213304u;
    const uint64_t q = ((uint64_t(Rh) * v) >> 13) + 8862793787191474850ull;     // Q0.63
    const uint64_t s = (mul_hi63(R, q) >> 11) + 6393154322601327830ull;        // Q0.63
    const uint64_t m = T + (mul_hi63(T, mul_hi63(R, s)) >> 8);  // Q1.62
    return bits_double(((m + 512) >> 10) + (uint64_t(1021 - n) << 52));
}

// |alpha + u gamma| in Q7.57: alpha in Q6.57, gamma < 62 as gamma 2^(57 + sh) with
// sh in its lowest three bits, u in Q0.63.  For alpha in (-63, 33) the sum is below
// 95; from 64 on it is taken for a negative one of magnitude 128 less it, above 33,
// where the profile is 0 all the same (exp2_neg_sq).
__host__ __device__ __forceinline__ uint64_t arg_magnitude(uint64_t alpha, uint64_t g, uint64_t u) {
    const uint64_t v = alpha + ((mul_hi63(u, g) << 1) >> (g & 7));
    return v >> 63 ? 0 - v : v;
}

// log2 x for x >= 0 from its exponent and first 20 fraction bits, low by less
// than 2^-18 for a normal x; an upper bound for a subnormal one and for 0.
__host__ __device__ __forceinline__ float log2_bits(double x) {
    const uint32_t hi = uint32_t(double_bits(x) >> 32), mb = 0x3f800000u | (hi & 0xfffffu) << 3;
#ifdef __CUDA_ARCH__
    const float f = __log2f(__uint_as_float(mb));
#else
    float m;
    memcpy(&m, &mb, 4);
    const float f = log2f(m);
#endif
    return float(int(hi >> 20) - 1023) + f;
}

// The |a| from which a line (centre values c0, e0) leaves the continuum's cc and
// ec as they are, bit for bit: a product below half an ulp, at least 2^-54 of
// them, rounds away, and 2^(-a^2) is taken as 0 from |a| = 31 on.  From exponents,
// so that the values' units do not matter.
__host__ __device__ __forceinline__ float far_profile(double cc, double ec, double c0, double e0) {
    constexpr uint64_t kNormal = uint64_t(1) << 52;
    if (double_bits(cc) < kNormal || (e0 > 0.0 && double_bits(ec) < kNormal)) return 31.f;
    float x = log2_bits(c0) - log2_bits(cc);
    if (e0 > 0.0) x = fmaxf(x, log2_bits(e0) - log2_bits(ec));
    return fminf(sqrtf(fmaxf(54.1f + x, 0.f)) * 1.0001f + 1e-3f, 31.f);
}

// 1 / x and 1 / sqrt x as the device approximates them (documented within 1 and 2
// ulp).  On the host, for the tests, the rounded values moved by MGX_HOST_ULPS.
#ifndef MGX_HOST_ULPS
#define MGX_HOST_ULPS 0
#endif
__host__ __device__ __forceinline__ float moved(float r, int ulps) {
    uint32_t b;
    memcpy(&b, &r, 4);
    b += uint32_t(ulps);
    memcpy(&r, &b, 4);
    return r;
}

__host__ __device__ __forceinline__ float rcp_approx(float x) {
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return moved(1.0f / x, MGX_HOST_ULPS);
#endif
}

__host__ __device__ __forceinline__ float rsqrt_approx(float x) {
#ifdef __CUDA_ARCH__
    return rsqrtf(x);
#else
    return moved(float(1.0 / sqrt(double(x))), 2 * MGX_HOST_ULPS);
#endif
}

// sqrt(a) for a >= 0 within 0.51 ulp; outside the range of the single-precision
// root the library's.
__host__ __device__ __forceinline__ double root(double a) {
    if (!(a > 1e-36 && a < 1e36)) return sqrt(a);
    const double y = double(rsqrt_approx(float(a)));  // 2^-21.4
    double s = a * y;
    const double h = 0.5 * y;
    s = fma(fma(-s, s, a), h, s);         // 2^-42
    return fma(fma(-s, s, a), h, s);
}

// e / t for finite e >= 0, t > 0: the mantissas' quotient from a
// single-precision reciprocal and one fixed-point correction with its square.
__host__ __device__ __forceinline__ double div_pos(double e, double t) {
    const uint64_t be = double_bits(e), bt = double_bits(t);
    const int xe = int(be >> 52), xt = int(bt >> 52), ex = xe - xt;
    if (xe == 0 || xt == 0 || ex > 1000 || ex < -1000) return e / t;  // zero, subnormal or far out
    const uint64_t hid = uint64_t(1) << 62, man = hid - 1;
    const uint64_t me = ((be << 10) & man) | hid, mt = ((bt << 10) & man) | hid;  // Q1.62
    const uint32_t tb = 0x3f800000u | (uint32_t(bt >> 29) & 0x7fffffu);
    // the reciprocal of t's leading bits, lowered by 2^-21 so that 1 - t x is not negative
    float x;
    memcpy(&x, &tb, 4);
    const uint32_t X = uint32_t(rcp_approx(x) * 2147482624.0f);  // Q1.31
    const uint64_t tx = uint64_t(uint32_t(mt >> 32)) * X + mul_hi32(uint32_t(mt), X);  // t x in Q2.61
    const uint64_t qe = uint64_t(uint32_t(me >> 32)) * X + mul_hi32(uint32_t(me), X);
    uint64_t d = (uint64_t(1) << 61) - tx;  // 1 - t x in [0, 2^-20)
    const uint32_t dh = uint32_t(d >> 25);
    d += (dh * dh) >> 11;                   // its square (the cube is below 2^-60)
    const uint64_t s = qe + (mul_hi63(qe, d << 21) >> 18);  // Q2.61, in (1/2, 2)
    const bool low = s < (uint64_t(1) << 61);
    const uint64_t s2 = low ? s << 1 : s;
    return bits_double(((s2 + 256) >> 9) + (uint64_t(int64_t(1022 + ex - int(low))) << 52));
}

// x in [0, 2) in Q1.62, rounded down.
__host__ __device__ __forceinline__ uint64_t to_q62(double x) {
    const uint64_t b = double_bits(x);
    const uint32_t s = 1023u - uint32_t(b >> 52);
    const uint64_t m = ((b << 10) & ((uint64_t(1) << 62) - 1)) | (uint64_t(1) << 62);
    return s < 64u ? m >> s : 0;
}

// v 2^-62 for v in [2^59, 2^62], to the nearest double (halves up).
__host__ __device__ __forceinline__ double from_q62(uint64_t v) {
#ifdef __CUDA_ARCH__
    const int sh = __clzll((long long)v) - 1;
#else
    const int sh = __builtin_clzll(v) - 1;
#endif
    return bits_double((((v << sh) + 512) >> 10) + (uint64_t(1022 - sh) << 52));
}

// v 2^-61 for v below 2^63, to the nearest double (0 for 0).
__host__ __device__ __forceinline__ double from_q61(uint64_t v) {
#ifdef __CUDA_ARCH__
    return __ull2double_rn(v) * 0x1p-61;
#else
    return double(v) * 0x1p-61;
#endif
}

// Conversions and a halving that the FP64 pipe would take 77 cycles for: a
// non-negative float as a double, half a non-negative double, and D in Q0.62
// as the nearest float.
__host__ __device__ __forceinline__ double widen(float x) {
#ifdef __CUDA_ARCH__
    const uint32_t b = __float_as_uint(x);
    return b >= 0x00800000u ? __hiloint2double(int((b >> 3) + 0x38000000u), int(b << 29)) : double(x);
#else
    return double(x);
#endif
}

__host__ __device__ __forceinline__ double halve(double x) {
    const uint64_t b = double_bits(x);
    return b >= (uint64_t(2) << 52) ? bits_double(b - (uint64_t(1) << 52)) : x * 0.5;
}

__host__ __device__ __forceinline__ float narrow_q62(uint64_t D) {
    const uint32_t top = uint32_t(D >> 31) | uint32_t((D & 0x7fffffffu) != 0);  // Q.31, sticky
    return float(top) * 4.656612873077393e-10f;                                // 2^-31
}

// b D as the nearest float, D in Q0.62, b a double in [0, 2).
__host__ __device__ __forceinline__ float narrow_product(double b, uint64_t D) {
    const uint64_t bits = double_bits(b);
    const uint32_t e = uint32_t(bits >> 52);
    if (e < 930u) return float(b * from_q62(D));  // below 2^-93, where the scale below is no normal float
    const uint64_t m = ((bits << 10) & ((uint64_t(1) << 62) - 1)) | (uint64_t(1) << 62);
    const uint64_t p = mul_hi63(m, D);            // b D 2^(1023 - e) in Q.60, at least 2^58
    const uint32_t top = uint32_t(p >> 29) | uint32_t((p & 0x1fffffffu) != 0);  // Q.31, sticky
#ifdef __CUDA_ARCH__
    return float(top) * __uint_as_float((e - 927u) << 23);  // 2^(e - 1023 - 31)
#else
    return float(double(top) * bits_double(uint64_t(e - 31u) << 52));
#endif
}

// One pivot of the scaled elimination in fixed point: with Y = D Fh of the row
// before (Q2.61), the increment t < 1 (Q1.62) and b < 1, its mean with the one
// before (Q2.61):  Fh = b + Y,  D = 1 / (1 + t Fh) (returned, Q0.62),  Y = D Fh.
// For Y < 2 on entry Fh is below 3 and 1 + t Fh below 4, which is what the
// formats hold.  The scaled quantities are of order one, so 59 fraction bits are
// more than a double's 53; the reciprocal is a single-precision one with one
// correction and its square.
__host__ __device__ __forceinline__ uint64_t pivot_q(uint64_t t, uint64_t b, uint64_t &Y) {
    const uint64_t F = b + Y;
    const uint64_t den = (uint64_t(1) << 59) + mul_hi63(t, F);  // Q4.59, in [1, 4)
    const uint32_t top = uint32_t(den >> 30);                   // Q2.29
    const uint32_t X = uint32_t(rcp_approx(float(top)) * 1152920954851033088.0f);  // Q0.31, low by up to 2^-20
    const uint64_t dx = uint64_t(uint32_t(den >> 32)) * X + mul_hi32(uint32_t(den), X);  // den X in Q.58
    uint64_t d = (uint64_t(1) << 58) - dx;  // 1 - den X in [0, 2^-20.5)
    const uint32_t dh = uint32_t((d + (1u << 21)) >> 22);
    d += (dh * dh) >> 14;                   // its square (the cube is below 2^-61)
    const uint64_t D = (uint64_t(X) << 31) + (mul_hi63(uint64_t(X) << 31, d << 23) >> 17);
    Y = mul_hi63(F, D) << 2;
    return D;
}

// Y of the pivots as they carry it: Q2.61 below 2, else the double's own bits
// with the sign bit set.  With increments up to 1 alone Y stays below 1.12
// (Y + t / 2 does not pass sqrt(1 + t^2 / 4) for the largest t); a thick cell
// followed by a thin one leaves half the thick one's increment.
__host__ __device__ __forceinline__ uint64_t hold_y(double y) {
    const uint64_t b = double_bits(y);
    return b < (uint64_t(1024) << 52) ? to_q62(y) >> 1 : b | (uint64_t(1) << 63);
}

__host__ __device__ __forceinline__ double held_y(uint64_t Y) {
    return Y >> 63 ? bits_double(Y & ~(uint64_t(1) << 63)) : from_q61(Y);
}

// One pivot for any increment dt >= 0 and mean increment dtb: D and dtb D as the
// nearest floats, Y updated.  In fixed point where its formats hold the operands;
// else (cells thicker than dtau_max <= 1 lets through, and the thin ones behind
// them) in double precision.
__host__ __device__ __forceinline__ void pivot(double dt, double dtb, uint64_t &Y, float &D, float &bD) {
    constexpr uint32_t kOne = 0x3ff00000u;
    if (uint32_t(double_bits(dt) >> 32) < kOne && uint32_t(double_bits(dtb) >> 32) < kOne && Y < (uint64_t(1) << 62)) {
        const uint64_t q = pivot_q(to_q62(dt), to_q62(dtb) >> 1, Y);
        D = narrow_q62(q);
        bD = narrow_product(dtb, q);
    } else {
        const double F = dtb + held_y(Y), d = div_pos(1.0, 1.0 + dt * F);
        D = float(d);
        bD = float(dtb * d);
        Y = hold_y(d * F);
    }
}

}  // namespace mgx
