// Elementary functions of the node right-hand sides with few FP64 instructions.
//
// GB300 retires about 2 FP64 lanes per clock per SM, against 64 lanes of 32-bit
// integer arithmetic and 128 of FP32.  The routines below keep every FP64
// instruction that the result's accuracy needs and move the rest to the
// integer and FP32 pipes; sin and cos need none at all.  The Hodgkin-Huxley rates
// take the integer forms of exp and the quotients in hh_rates.cuh; exp and 1/d here
// serve sim_math_eval.
//
// Methods (textbook; constants derived for this code from pi and ln 2 in
// high-precision arithmetic):
//   sin/cos  fixed_sincos, in integer arithmetic only: additive range
//            reduction by pi/2048 (Cody & Waite 1980), t = |x| * 2048/pi from one
//            unsigned 64 x 64 high product of |x| 2^55 and 512/pi 2^56 (grid
//            2^-45); k = floor t, r = (t - k) pi/2048 >= 0; Taylor polynomials
//            sin r = r - r^3 (1/6 - r^2/120) and cos r - 1 = -r^2/2 + r^4/24
//            (first omitted terms below 2^-65), whose small terms take 32 x 32
//            products; the angle-addition formula around the table point
//            j pi/2048 of the first quadrant, j = k mod 1024 (the "accurate table"
//            approach of Tang and Gal): S_j + C_j sin r + S_j (cos r - 1) and
//            C_j - S_j sin r + C_j (cos r - 1), (S_j, C_j) on the grid 2^-62, then
//            k / 1024 quarter turns.  Every factor is non-negative, so that no
//            product needs a sign correction.  The result is sin and cos on the
//            grid 2^-62, of magnitude at most 2^62, within 2^-53.6 of the true
//            values for |x| < 256 (a host model of the same integer steps was
//            checked against long double sinl/cosl over 2 * 10^7 arguments and the
//            reduction edges: worst error 7.2e-17, set by the grid of t); that
//            grid is what the exact window sums consume.
//            |x| >= 256, Inf and NaN use the library routine.
//   exp      Tang (1989) table-driven method: x = (64 m + j) ln2/64 + r,
//            exp(x) = 2^m 2^(j/64) exp(r), degree-5 Taylor polynomial for
//            exp(r) - 1, |r| <= ~ln2/128.  8 FP64 instructions.
//   1/d      FP32 hardware reciprocal as the seed, then two Newton steps
//            y <- y + y (1 - d y) in FP64.  4 FP64 instructions, error <= 1 ulp.
// Accuracy is checked on the GPU against the C library (see the tests).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

namespace simk {

// Tables (host-filled at handle creation; see sim_api.cu).
constexpr int kSinTab = 1024;  // sin/cos(j pi/2048), j in [0, 1024)
constexpr int kExpTab = 64;    // 2^(j/64), j in [0, 64)
constexpr int kExp2Tab = 256;  // 2^(j/256), j in [0, 256)

struct MathTables {
    const ulonglong2 *sincos_q; // (sin, cos) of j*pi/2048 on the grid 2^-62 (fill_math_tables)
    const double *exp2j;       // 2^(j/64)
    const unsigned long long *exp2q; // 2^(j/256) rounded onto the grid 2^-63
};

// The tables as one block of 64-bit words (host-filled in long double, uploaded
// once per network or device): sincos_q (2 kSinTab uint64), exp2j (kExpTab
// doubles), exp2q (kExp2Tab uint64).
constexpr int kMathTableWords = 2 * kSinTab + kExpTab + kExp2Tab;
__host__ __device__ inline MathTables math_tables_at(const void *block)
{
    const double *d = static_cast<const double *>(block);
    return MathTables{reinterpret_cast<const ulonglong2 *>(d), d + 2 * kSinTab,
                      reinterpret_cast<const unsigned long long *>(d + 2 * kSinTab + kExpTab)};
}

// |x| as a float by truncating the mantissa (integer instructions; |x| must be
// inside the float exponent range, which every caller checks first).
__device__ __forceinline__ float dbl_to_flt_trunc(double x)
{
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const uint32_t hi = (uint32_t)(b >> 32);
    const int e = (int)((hi >> 20) & 0x7FF);
    if (e < 1023 - 126) return 0.0f;
    if (e > 1023 + 127) return __uint_as_float((hi & 0x80000000u) | 0x7F800000u); // Inf (also for NaN)
    const uint32_t mant = ((hi & 0xFFFFFu) << 3) | (uint32_t)((b >> 29) & 7u);
    return __uint_as_float((hi & 0x80000000u) | ((uint32_t)(e - 1023 + 127) << 23) | mant);
}

// Exact double of a 32-bit integer (integer instructions only).
__device__ __forceinline__ double int_to_dbl(int k)
{
    if (k == 0) return 0.0;
    const uint64_t sign = k < 0 ? (1ull << 63) : 0ull;
    const uint32_t a = (uint32_t)(k < 0 ? -k : k);
    const int lz = __clz((int)a);
    const uint64_t mant = ((uint64_t)a << (lz + 21)) & 0xFFFFFFFFFFFFFull; // drop the leading one
    const uint64_t ex = (uint64_t)(1023 + 31 - lz);
    return __longlong_as_double((long long)(sign | (ex << 52) | mant));
}

// Nearest integer to xf * scale in FP32 (1.5 * 2^23 rounding constant).
__device__ __forceinline__ int round_scaled(float xf, float scale)
{
    const float t = fmaf(xf, scale, 12582912.0f);
    return __float_as_int(t) - 0x4B400000;
}

// Constants of fixed_sincos (derived from pi in 60-digit arithmetic).
constexpr uint64_t kPio512Inv56 = 0xa2f9836e4e44152aull; // round(512/pi * 2^56)
constexpr uint64_t kPio2048Q73 = 0xc90fdaa22168c235ull;  // round(pi/2048 * 2^73)
constexpr uint32_t kSixthQ34 = 2863311531u;               // round(2^34 / 6)
constexpr uint32_t kInv120Q16 = 546u;                     // round(2^16 / 120)
constexpr uint32_t kInv24Q28 = 11184811u;                 // round(2^28 / 24)

// a b / 2^64 from three 32 x 32 products, the low words' product left out: the
// exact floor or one less.  a <= 2^63 and b <= 2^63, so that the sum of the middle
// products stays below 2^64.  (On GB300 a 32 x 32 + 64 multiply-add retires at half
// rate, and the exact high product takes four and their carries.)
__device__ __forceinline__ uint64_t umulhi_near(uint64_t a, uint64_t b)
{
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return (uint64_t)ah * bh + (((uint64_t)ah * bl + (uint64_t)al * bh) >> 32);
}

// A signed factor v in [-2^62, 2^62] moved to [0, 2^63] for an unsigned product:
// with a constant b that is a multiple of 4, floor(v b / 2^64) is the high product
// of biased62(v) and b less b / 4 (one addition in the high word, against a compare,
// two selects and a 64-bit subtraction in mulhi_su).
__device__ __forceinline__ uint64_t biased62(int64_t v)
{
    return (uint64_t)v + (1ull << 62);
}

// floor(a b / 2^64) for signed a and unsigned b: the unsigned high product of
// a's two's-complement bits, less b when a is negative.
__device__ __forceinline__ int64_t mulhi_su(int64_t a, uint64_t b)
{
    return (int64_t)(__umul64hi((uint64_t)a, b) - (a < 0 ? b : 0ull));
}

// floor(a b / 2^64) for signed a and b, from the unsigned high product.
__device__ __forceinline__ int64_t mulhi_ss(int64_t a, int64_t b)
{
    uint64_t h = __umul64hi((uint64_t)a, (uint64_t)b);
    h -= a < 0 ? (uint64_t)b : 0ull;
    h -= b < 0 ? (uint64_t)a : 0ull;
    return (int64_t)h;
}

// sin x and cos x on the grid 2^-62 (s62, c62 in [-2^62, 2^62]), absolute
// error below 2^-53.6.  Integer instructions only on the fast path |x| < 256;
// beyond it, and for Inf and NaN, the library routine (ok = false for a
// non-finite x).
//   X = |x| 2^55 (truncated), t = X (512/pi) 2^-64: |x| 2048/pi on the grid 2^-45,
//   k = floor t, r = (t - k) pi/2048 in [0, pi/2048);
//   sin r = r - r^3 (1/6 - r^2/120) and 1 - cos r = r^2/2 - r^4/24, the small
//   terms from 32 x 32 products of the top words;
//   the angle-addition formula around the table point j pi/2048, j = k mod 1024;
//   quarter turns by k / 1024.
// Against a table over the half turn, r rounded to nearest and signed factors (33
// wide multiplies and four sign corrections; here 26 and none) a Kuramoto ring of
// 10^6 nodes takes 98 us per RK4 step in place of 104, a 101^3 cube 151 of 160.
__device__ __forceinline__ void fixed_sincos(double x, const MathTables &T, int64_t &s62, int64_t &c62, bool &ok)
{
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF);
    if (e >= 1023 + 8) {
        double s, c;
        sincos(x, &s, &c);
        s62 = to_fixed(s, 62, 1, ok);
        c62 = to_fixed(c, 62, 1, ok);
        return;
    }
    const uint64_t m = ((b << 10) & ((1ull << 62) - 1)) | (1ull << 62); // significand 2^62
    const uint64_t t = __umul64hi(m >> min(1030 - e, 63), kPio512Inv56); // |x| 2048/pi 2^45
    const uint32_t k = (uint32_t)(t >> 45);
    const uint64_t g = t << 19; // t - k on the grid 2^-64
    const uint32_t gh = (uint32_t)(g >> 32), gl = (uint32_t)g;
    constexpr uint32_t ph = (uint32_t)(kPio2048Q73 >> 32), pl = (uint32_t)kPio2048Q73;
    const uint64_t u = (uint64_t)gh * pl; // r 2^73, the product of the low words left out
    const uint64_t R = (uint64_t)gh * ph + (u >> 32) + (((uint64_t)gl * ph + (uint32_t)u) >> 32);
    const uint32_t rh = (uint32_t)(R >> 32);
    const uint64_t z = (uint64_t)rh * rh + (((uint64_t)rh * (uint32_t)R) >> 31); // r^2 2^82
    const uint32_t zh = (uint32_t)(z >> 32);                                     // r^2 2^50
    const uint32_t v59 = __umulhi(rh, zh);                                       // r^3 2^59
    const uint32_t u34 = kSixthQ34 - __umulhi(zh, kInv120Q16);                   // (1/6 - r^2/120) 2^34
    const uint64_t sr = (R >> 9) - (((uint64_t)v59 * u34) >> 29);                // sin r 2^64
    const uint64_t cm = (z >> 19) - __umulhi(__umulhi(zh, zh), kInv24Q28);       // (1 - cos r) 2^64
    const ulonglong2 tq = __ldg(T.sincos_q + (k & (kSinTab - 1)));               // (S_j, C_j) 2^62
    const int64_t s1 = (int64_t)(tq.x - umulhi_near(tq.x, cm) + umulhi_near(tq.y, sr));
    const int64_t c1 = (int64_t)(tq.y - umulhi_near(tq.y, cm) - umulhi_near(tq.x, sr));
    const bool odd = k & kSinTab;
    const int64_t s = odd ? c1 : s1, c = odd ? s1 : c1;
    s62 = ((k << 20) ^ (uint32_t)(b >> 32)) >> 31 ? -s : s; // k's half-turn bit and the sign of x
    c62 = (k ^ (k << 1)) & (2 * kSinTab) ? -c : c;          // quarter turns 1 and 2
}

// v 2^-62 rounded onto the coarser grid 2^-F (F <= 61), half up.
__device__ __forceinline__ int64_t q62_to(int64_t v, int F)
{
    const int sh = 62 - F;
    return (v + (1ll << (sh - 1))) >> sh;
}

// sin and cos as doubles, correctly rounded from fixed_sincos's values on the
// grid 2^-62 (NaN for an infinite or NaN x).
__device__ __forceinline__ void fast_sincos(double x, const MathTables &T, double &s, double &c)
{
    int64_t s62, c62;
    bool ok = true;
    fixed_sincos(x, T, s62, c62, ok);
    if (!ok) {
        s = c = x - x;
        return;
    }
    s = fixed_to_double(s62, 62);
    c = fixed_to_double(c62, 62);
}

// ln2/64 = L1 + L2 + L3 (L1, L2 rounded to 32 significant bits; two parts are
// enough here because |k| < 2^16).
constexpr double kLn2o64_1 = 0x1.62e42ffp-7;
constexpr double kLn2o64_2 = -0x1.718432a2p-41;
constexpr double kLn2o64_3 = 0x1.3c7673007e5edp-75;
constexpr float k64oLn2 = 92.3324814f;

__device__ __forceinline__ double fast_exp(double x, const MathTables &T)
{
    const float xf = dbl_to_flt_trunc(x);
    if (!(fabsf(xf) < 700.0f)) return exp(x);
    const int k = round_scaled(xf, k64oLn2);
    const double dk = int_to_dbl(k);
    double r = fma(-dk, kLn2o64_1, x);
    r = fma(-dk, kLn2o64_2, r);
    // exp(r) - 1 = r + r^2 (1/2 + r (1/6 + r (1/24 + r/120)))   (|r| <= 0.0055)
    double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    q = fma(r, q, 1.0 / 6.0);
    q = fma(r, q, 0.5);
    const double em1 = fma(r * r, q, r);
    const double tj = __ldg(T.exp2j + (k & (kExpTab - 1)));
    const double v = fma(tj, em1, tj);
    // times 2^m, m = floor(k / 64): add m to the exponent field
    const int m = k >> 6;
    return __longlong_as_double(__double_as_longlong(v) + ((long long)m << 52));
}

// 1/d for finite d with |d| in [2^-120, 2^120] (else the IEEE division).
__device__ __forceinline__ double fast_rcp(double d)
{
    const float df = dbl_to_flt_trunc(d);
    const float af = fabsf(df);
    if (!(af > 1e-36f && af < 1e36f)) return 1.0 / d;
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(df));
    // the seed as a double: float bits widened by integer instructions
    const uint32_t fb = __float_as_uint(yf);
    const uint64_t db = ((uint64_t)(fb & 0x80000000u) << 32) |
                        ((uint64_t)(((fb >> 23) & 0xFFu) - 127 + 1023) << 52) | ((uint64_t)(fb & 0x7FFFFFu) << 29);
    double y = __longlong_as_double((long long)db);
    double e = fma(-d, y, 1.0);
    y = fma(y, e, y);
    e = fma(-d, y, 1.0);
    return fma(y, e, y);
}

// x / (1 - exp(-x)), with its limit 1 at x = 0 (the Hodgkin-Huxley rate form).
// |x| < 0.1: the series 1 + x/2 + x^2/12 - x^4/720 + x^6/30240 - x^8/1209600
// (Bernoulli numbers; the next term is below 2^-58).  Otherwise x * (1/(1 - e^-x)).
__device__ __forceinline__ double fast_x_over_1mexp(double x, const MathTables &T)
{
    const float xf = dbl_to_flt_trunc(x);
    if (fabsf(xf) < 0.1f) {
        const double z = x * x;
        const double p = fma(z, fma(z, fma(z, -1.0 / 1209600.0, 1.0 / 30240.0), -1.0 / 720.0), 1.0 / 12.0);
        return fma(x, 0.5, fma(z, p, 1.0));
    }
    return x * fast_rcp(1.0 - fast_exp(-x, T));
}

} // namespace simk
