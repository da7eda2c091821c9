// Rate functions of the Hodgkin-Huxley gates (textbook rates, V in mV) from the
// membrane potential on the fixed-point grid 2^-46, |V| < 256, in integer
// arithmetic.
//
// Why: GB300 retires 1.9 FP64 instructions per clock and SM against 7.2 unsigned
// 64 x 64 high products and about 60 32-bit integer instructions.  Six
// exponentials and three divisions in FP64 were 70 of the slope's 105 FP64
// instructions, and the FP64 pipe bound the stage; here the six rates take none.
//
// Method.  A positive value is (m, e) = m 2^(e - 63), 2^63 <= m < 2^64 (about 62
// good bits).  Two exponentials suffice, by Tang's (1989) table-driven method on
// t = -(V + 65)/tau log2(e): 2^t = 2^k 2^(j/256) 2^f with f in [0, 2^-8) and the
// degree-5 Taylor polynomial of 2^f (the next term is below 2^-60):
//   E80 = exp(-(V + 65)/80)  and  E18 = exp(-(V + 65)/18);
// then E20 = E80^4 and E10 = E20^2 by squaring, and exp(-(V + 40)/10),
// exp(-(V + 35)/10), exp(-(V + 55)/10) are E10 times constants.  Reciprocals: an
// FP32 seed (23 bits) and two Newton steps.  Relative error of every rate below
// 2^-56 (a host model of the same integer steps against 60-digit arithmetic, V in
// (-256, 256)), and below 2^-52 for alpha_m, alpha_n next to the series branch,
// where 1 - exp(-x) cancels (FP64 had 2^-50 there).
#pragma once
#include "fastmath.cuh"

namespace simk {

struct UFloat { // m 2^(e - 63)
    uint64_t m;
    int e;
};

// Constants (derived in 60-digit decimal arithmetic).
constexpr uint64_t kLog2e80 = 0x93bb62877cdff3c9ull; // log2(e)/80 2^69
constexpr uint64_t kLog2e18 = 0xa42589ebe01547c3ull; // log2(e)/18 2^67
constexpr uint64_t kEx1 = 0xb17217f7d1cf79acull;     // ln 2 2^64
constexpr uint64_t kEx2 = 0x0f5fdeffc162c754ull;     // ln^2 2 / 2 2^62
constexpr uint32_t kEx3 = 0xe35846b8u;               // ln^3 2 / 6 2^36
constexpr uint32_t kEx4 = 0x9d955b7eu;               // ln^4 2 / 24 2^38
constexpr uint32_t kEx5 = 0xaec3ff3cu;               // ln^5 2 / 120 2^41

// 2^t for t on the grid 2^-G (|t| < 64).
template <int G> __device__ __forceinline__ UFloat uf_exp2(int64_t t, const MathTables &T)
{
    const int64_t k = t >> (G - 8);
    const uint64_t F = (uint64_t)t << (72 - G); // f 2^72
    const uint64_t f2 = __umul64hi(F, F);       // f^2 2^80
    const uint32_t fh = (uint32_t)(F >> 32), f2h = (uint32_t)(f2 >> 32), f3 = __umulhi(fh, f2h); // f 2^40, f^2 2^48, f^3 2^56
    const uint64_t g = kEx2 + (((uint64_t)fh * kEx3) >> 14) + (((uint64_t)f2h * kEx4) >> 24) +
                       (((uint64_t)f3 * kEx5) >> 35);                           // (2^f - 1 - f ln 2) / f^2, 2^62
    const uint64_t em1 = __umul64hi(F, kEx1) + (__umul64hi(f2, g << 1) >> 7);    // (2^f - 1) 2^72
    const uint64_t tj = __ldg(T.exp2q + ((int)k & (kExp2Tab - 1)));              // 2^(j/256) 2^63
    return UFloat{tj + (__umul64hi(tj, em1) >> 8), (int)(k >> 8)};
}

__device__ __forceinline__ UFloat uf_mul(const UFloat &a, const UFloat &b)
{
    const uint64_t h = __umul64hi(a.m, b.m); // [2^62, 2^64)
    const bool top = (int64_t)h < 0;
    return UFloat{top ? h : h << 1, a.e + b.e + (top ? 1 : 0)};
}

// x 2^(e - 63), x > 0, normalised.
__device__ __forceinline__ UFloat uf_norm(uint64_t x, int e)
{
    const int lz = __clzll((long long)x);
    return UFloat{x << lz, e - lz};
}

// |1 - a| (a != 1; the caller keeps |1 - a| well above the grid) and 1 + a.
__device__ __forceinline__ UFloat uf_one_minus(const UFloat &a)
{
    const uint64_t one = 1ull << 63;
    return a.e < 0 ? uf_norm(one - (a.m >> min(-a.e, 63)), 0) : uf_norm(a.m - (one >> min(a.e, 63)), a.e);
}
__device__ __forceinline__ UFloat uf_one_plus(const UFloat &a)
{
    const uint64_t half = 1ull << 62;
    return a.e < 0 ? uf_norm(half + (a.m >> min(1 - a.e, 63)), 1) : uf_norm((a.m >> 1) + (half >> min(a.e, 62)), a.e + 1);
}

// 1 / a: y = 2^126 / m in (2^62, 2^63] from an FP32 seed of m's top 24 bits, two
// Newton steps y += y (2^62 - (m y >> 64)) 2^-62.
__device__ __forceinline__ UFloat uf_rcp(const UFloat &a)
{
    float s;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(__uint_as_float(0x3F800000u | ((uint32_t)(a.m >> 40) & 0x7FFFFFu))));
    const uint32_t sb = min(__float_as_uint(s), 0x3F7FFFFFu); // below 1
    uint64_t y = (uint64_t)(0x800000u | (sb & 0x7FFFFFu)) << 39;
#pragma unroll
    for (int k = 0; k < 2; ++k)
        y += (uint64_t)mulhi_su((int64_t)(((1ull << 62) - __umul64hi(a.m, y)) << 2), y);
    y = (int64_t)y < 0 ? (1ull << 63) - 1 : y; // m = 2^63
    return UFloat{y << 1, -a.e - 1};
}

// Nearest double (the values here lie far inside its exponent range).  The rounding bit is
// added after the shift: m + 1024 wraps for m within 1024 of 2^64, where the carry has to
// reach the exponent.
__device__ __forceinline__ double uf_double(const UFloat &a)
{
    return __longlong_as_double((long long)(((uint64_t)(int64_t)(a.e + 1022) << 52) + (a.m >> 11) + ((a.m >> 10) & 1)));
}

struct HHRates {
    double am, bm, ah, bh, an, bn;
};

// x / (1 - e^-x) for small |x|: 1 + x/2 + x^2/12 - x^4/720 + x^6/30240 - x^8/1209600.
__device__ __forceinline__ double hh_ratio_series(double x)
{
    const double z = x * x;
    const double p = fma(z, fma(z, fma(z, -1.0 / 1209600.0, 1.0 / 30240.0), -1.0 / 720.0), 1.0 / 12.0);
    return fma(x, 0.5, fma(z, p, 1.0));
}

// q = V 2^46, |q| < 2^54.
__device__ __forceinline__ HHRates hh_rates(int64_t q, const MathTables &T)
{
    const int64_t w = (q + (65ll << 46)) << 8;
    const UFloat e80 = uf_exp2<59>(-mulhi_su(w, kLog2e80), T), e18 = uf_exp2<57>(-mulhi_su(w, kLog2e18), T);
    const UFloat e40 = uf_mul(e80, e80), e20 = uf_mul(e40, e40), e10 = uf_mul(e20, e20);
    HHRates r;
    r.bm = uf_double(UFloat{e18.m, e18.e + 2});                                     // 4 exp(-(V + 65)/18)
    r.ah = uf_double(uf_mul(e20, UFloat{0x8f5c28f5c28f5c29ull, -4}));               // 0.07 exp(-(V + 65)/20)
    r.bn = uf_double(UFloat{e80.m, e80.e - 3});                                     // exp(-(V + 65)/80) / 8
    r.bh = uf_double(uf_rcp(uf_one_plus(uf_mul(e10, UFloat{0xa0af2dfb7d882f97ull, 4})))); // 1 / (1 + e^3 E10)
    // alpha_m = x / (1 - e^-x), x = (V + 40)/10; alpha_n = 0.1 z / (1 - e^-z), z = (V + 55)/10:
    // |x| on 2^-58, |0.1 z| on 2^-61; the series for |x| < 2^-4
    const int64_t v40 = q + (40ll << 46), v55 = q + (55ll << 46);
    const uint64_t a40 = (uint64_t)(v40 < 0 ? -v40 : v40), a55 = (uint64_t)(v55 < 0 ? -v55 : v55);
    constexpr uint64_t kNear = 5ull << 43; // 0.625 mV
    if (a40 >= kNear) {
        const UFloat x = uf_norm(__umul64hi(a40 << 9, 0xcccccccccccccccdull), 5); // 0.8 2^64
        r.am = uf_double(uf_mul(x, uf_rcp(uf_one_minus(uf_mul(e10, UFloat{0xc2eb7ec98f05d8eaull, 3}))))); // e^2.5 E10
    } else {
        r.am = hh_ratio_series(ll2double_scaled(v40, 46) * 0.1);
    }
    if (a55 >= kNear) {
        const UFloat x = uf_norm(__umul64hi(a55 << 9, 0xa3d70a3d70a3d70aull), 2); // 0.64 2^64
        r.an = uf_double(uf_mul(x, uf_rcp(uf_one_minus(uf_mul(e10, UFloat{0xadf85458a2bb4a9bull, 1}))))); // e E10
    } else {
        r.an = 0.1 * hh_ratio_series(ll2double_scaled(v55, 46) * 0.1);
    }
    return r;
}

} // namespace simk
