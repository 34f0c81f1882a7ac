// mcg_fixed.cuh -- log, square root, cosine and sine of the double-precision
// walk's normals, in 64-bit integers.
//
// GB300 does 1.6 double-precision operations a clock and SM, and the library's
// log, sqrt and sincos take some 110 of them per step: 6 us of latency and nine
// tenths of the plain walk's throughput.  Its integer units do 64 32-bit
// operations a clock, so the functions are evaluated here on 64-bit integers,
// to about 2^-62 of their range (apart, to 2^-57 of themselves where they are
// small: u1 next to 1, angles next to an axis), and rounded to double precision
// where the problem states a double; the radius is then within 0.9 units in the
// last place, cosine and sine within 1.6 of those of the rounded angle:
//
//   u1 = (w + 1/2) 2^-32 exactly, L = -ln u1 = e ln 2 + ln c_i - ln(1 + y),
//     u1 = v 2^-e, v in [1/2, 1), c_i a 16-bit reciprocal of v's 1/512
//     interval (1 for the last, so that small L keep their leading digits),
//     y = v c_i - 1 exactly, |y| <= 2^-9; ln(1 + y) by its series to y^6;
//   sqrt(2 L): the hardware's reciprocal root and two corrections by the exact
//     remainder N - S^2;
//   cos, sin of a = 2 pi u2 (rounded, as a double): quadrant, the angle in the
//     middle of one of 256 parts of it (table) and the rest theta,
//     |theta| <= 2^-8.3, by their series to theta^6, put together by the
//     addition theorems.
//
// The tables are computed at compile time from the same series.  Compiles for
// the host as well, where the functions are compared with 60-digit values.
// Digits for the small values cost the full walk 5 % (28.7 -> 27.2 steps/ns).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mcg {
namespace fx {

constexpr uint64_t kLn2 = 0xB17217F7D1CF79ACull;      // ln 2, units of 2^-64
constexpr uint64_t kHalfPi57 = 0x03243F6A8885A309ull;  // pi / 2, units of 2^-57
constexpr uint64_t kTwoPi50 = 0x001921FB54442D18ull;   // the double nearest 2 pi, units of 2^-50
constexpr uint64_t kPi1024 = 0x00C90FDAA22168C2ull;    // pi / 1024, units of 2^-64 ...
constexpr uint32_t kPi1024Low = 0x34C4C662u;           // ... and its next 32 bits

// High word of the 128-bit product, by 32-bit halves (constant expressions).
constexpr uint64_t mulhi_c(uint64_t a, uint64_t b)
{
    const uint64_t a0 = (uint32_t)a, a1 = a >> 32, b0 = (uint32_t)b, b1 = b >> 32;
    const uint64_t m = a1 * b0 + (a0 * b0 >> 32), n = a0 * b1 + (uint32_t)m;
    return a1 * b1 + (m >> 32) + (n >> 32);
}

struct Tables {
    uint64_t ln_c[256];    // units of 2^-64
    int64_t cos_sin[512];  // cos, sin of (j + 1/2) pi / 512, units of 2^-63
    uint32_t c[256];       // units of 2^-15

    constexpr Tables() : ln_c(), cos_sin(), c()
    {
        for (int i = 0; i < 256; ++i) {
            // 2^15 / v for v = (512 + 2 i + 1) / 1024, rounded
            const uint32_t den = 512u + 2u * (uint32_t)i + 1u;
            c[i] = i == 255 ? 1u << 15 : (uint32_t)(((1u << 26) / den + 1u) >> 1);
            // ln c = 2 atanh s = 2 (s + s^3 / 3 + ...), s = (c - 1) / (c + 1)
            const uint64_t num = c[i] - (1u << 15), d = c[i] + (1u << 15);
            const uint64_t q = (num << 32) / d, s = (q << 32) | ((((num << 32) % d) << 32) / d);
            const uint64_t s2 = mulhi_c(s, s);
            uint64_t p = s, sum = 0;
            for (uint64_t k = 1; p != 0; k += 2) {
                sum += p / k;
                p = mulhi_c(p, s2);
            }
            ln_c[i] = 2 * sum;
        }
        for (int j = 0; j < 128; ++j) {  // up to pi / 4 by the series, the rest mirrored
            const uint64_t x = kHalfPi57 / 512 * (2 * j + 1) * 128 + (kHalfPi57 % 512) * (2 * j + 1) * 128 / 512;
            const uint64_t x2 = mulhi_c(x, x);
            uint64_t even = ~0ull >> 1, odd = x >> 1, ce = even, so = odd;
            for (uint64_t k = 1; even != 0; ++k) {  // units of 2^-63
                even = mulhi_c(even, x2) / ((2 * k - 1) * (2 * k));
                odd = mulhi_c(odd, x2) / ((2 * k) * (2 * k + 1));
                ce = (k & 1) ? ce - even : ce + even;
                so = (k & 1) ? so - odd : so + odd;
            }
            cos_sin[2 * j] = cos_sin[2 * (255 - j) + 1] = (int64_t)ce;
            cos_sin[2 * j + 1] = cos_sin[2 * (255 - j)] = (int64_t)so;
        }
    }
};

static __device__ const Tables g_tables{};

// 32 by 32 bits; high word of a 64 by 64 bit product without the carry from
// the lowest words (at most 2 units low); a^2 likewise.
__host__ __device__ __forceinline__ uint64_t mul32(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
__host__ __device__ __forceinline__ uint64_t mulhi(uint64_t a, uint64_t b)
{
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32), b0 = (uint32_t)b, b1 = (uint32_t)(b >> 32);
    const uint64_t m = mul32(a1, b0), n = mul32(a0, b1) + (uint32_t)m;
    return mul32(a1, b1) + (m >> 32) + (n >> 32);
}
// (the same, up to 3 units low)
__host__ __device__ __forceinline__ uint64_t mulhi3(uint64_t a, uint64_t b)
{
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32), b0 = (uint32_t)b, b1 = (uint32_t)(b >> 32);
    return mul32(a1, b1) + (mul32(a1, b0) >> 32) + (mul32(a0, b1) >> 32);
}
__host__ __device__ __forceinline__ uint64_t sqrhi(uint64_t a)
{
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32);
    return mul32(a1, a1) + (mul32(a0, a1) >> 31);
}
__host__ __device__ __forceinline__ int clz64(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}
__host__ __device__ __forceinline__ float rsqrt_seed(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / __builtin_sqrtf(x);
#endif
}

// The same number as neg_log's for y = 1 - u1 <= 2^-9 (units of 2^-64): from
// fixed digits its leading ones would be missing, 2.9e-11 of the radius at
// u1 = 1 - 2^-33.  Here y (1 + y/2 + y^2 A), y with all its digits.  (A call, as
// it is rare: one u1 in 512.)
struct Scaled {
    uint64_t N;
    int E;
};
static __host__ __device__ __noinline__ Scaled neg_log_near_one(uint64_t y)
{
    const uint32_t ys = (uint32_t)(y >> 24);  // units of 2^-40
    const uint64_t y2 = sqrhi(y);
    const uint32_t B = 0x40000000u + (uint32_t)(mul32(ys, 0x33333333u) >> 40) +
                       (uint32_t)(mul32((uint32_t)(y2 >> 16), 0x2AAAAAABu) >> 48);  // 1/4 + y/5 + y^2/6
    const uint64_t q = (y >> 1) + mulhi3(y2, 0x5555555555555555ull + (mul32(ys, B) >> 8));
    const int z = clz64(y);
    const uint64_t n = y << z, N = n + mulhi3(n, q);
    return N < n ? Scaled{N >> 1 | 1ull << 63, 1 - z} : Scaled{N, -z};
}

// -ln((w + 1/2) 2^-32) = N 2^(E - 64), N in [2^63, 2^64)
__host__ __device__ __forceinline__ void neg_log(const Tables& T, uint32_t w, uint64_t& N, int& E)
{
    const uint64_t m = 2ull * w + 1ull;  // u1 = m 2^-33
    const int z = clz64(m);
    const uint64_t V = m << z;           // v, units of 2^-64
    const uint32_t e = (uint32_t)z - 31u;
    const uint32_t i = (uint32_t)(V >> 55) & 255u;
    if (i == 255u && e == 0u) {
        const Scaled L = neg_log_near_one(0ull - V);
        N = L.N;
        E = L.E;
        return;
    }
    // y = v c - 1 exactly (33 by 17 bits), units of 2^-64: sign and size
    const uint32_t c = T.c[i];
    const int64_t y48 = (int64_t)(((V >> 63) * c << 32) + mul32((uint32_t)(V >> 31), c) - (1ull << 48));
    const bool neg = y48 < 0;
    const uint64_t y = (uint64_t)(neg ? -y48 : y48) << 16;
    // ln(1 + y) = y - y^2/2 + y^3 A, A = 1/3 - y B, B = 1/4 - y/5 + y^2/6; 32
    // bits of B do (y^4 B < 2^-38), for A they would leave 2^-58
    const uint32_t ys = (uint32_t)(y >> 24);           // units of 2^-40
    const uint64_t y2 = sqrhi(y);
    const uint32_t y5 = (uint32_t)(mul32(ys, 0x33333333u) >> 40), y6 = (uint32_t)(mul32((uint32_t)(y2 >> 16), 0x2AAAAAABu) >> 48);
    const uint32_t B = 0x40000000u + (neg ? y5 : 0u - y5) + y6;
    const uint64_t yB = mul32(ys, B) >> 8;
    const uint64_t y3A = mulhi3(y2, mulhi3(y, 0x5555555555555555ull + (neg ? yB : 0ull - yB)));
    const int64_t odd = (int64_t)(y + y3A);
    const int64_t ln1 = (neg ? -odd : odd) - (int64_t)(y2 >> 1);
    // e ln 2 + ln c - ln1, integer part in hi
    uint64_t lo = e * kLn2;
    uint32_t hi = (uint32_t)((mul32(e, (uint32_t)(kLn2 >> 32)) + (mul32(e, (uint32_t)kLn2) >> 32)) >> 32);
    lo += T.ln_c[i];
    hi += lo < T.ln_c[i] ? 1u : 0u;
    const uint64_t before = lo;
    lo -= (uint64_t)ln1;
    hi -= (before < (uint64_t)ln1 ? 1u : 0u) + (uint32_t)(ln1 >> 63);
    if (hi) {
        E = 64 - clz64((uint64_t)hi);
        N = ((uint64_t)hi << (64 - E)) | (lo >> E);
    } else {
        E = -clz64(lo);
        N = lo << -E;
    }
}

// sqrt(N 2^(E - 64)) = S 2^(H - 64)
__host__ __device__ __forceinline__ uint64_t root(uint64_t N, int E, int& H)
{
    if (E & 1) {
        N >>= 1;
        ++E;
    }
    H = E >> 1;
    const float x = (float)(uint32_t)(N >> 32) * 0x1p-32f;  // [1/4, 1]
    const float y = fminf(rsqrt_seed(x), 1.9999998f);
    const uint32_t s0 = (uint32_t)(fminf(x * y, 0.99999994f) * 0x1p32f), Y = (uint32_t)(y * 0x1p31f);
    const uint64_t s1 = (uint64_t)s0 << 32;
    // remainder / (2 root): to 30 of its 43 bits, then what that left to all
    const int64_t d1 = ((int64_t)(int32_t)((int64_t)(N - mul32(s0, s0)) >> 14) * (int64_t)(Y >> 1)) >> 17;
    uint64_t s = s1 + (uint64_t)d1;
    if (d1 > 0 && s < s1) s = ~0ull;
    const int64_t d2 = ((int64_t)(int32_t)(N - sqrhi(s)) * (int64_t)(Y >> 1)) >> 31;
    const uint64_t t = s + (uint64_t)d2;
    return d2 > 0 && t < s ? ~0ull : t;
}

// cos, sin of the double a = 2 pi (w + 1/2) 2^-32, units of 2^-63; returns a
__host__ __device__ __forceinline__ uint64_t cos_sin(const Tables& T, uint32_t w, int64_t& co, int64_t& si)
{
    // a rounded to 53 bits, units of 2^-61 (finer digits of a small a are lost)
    const uint64_t p0 = (uint64_t)(uint32_t)kTwoPi50 * w, p1 = (kTwoPi50 >> 32) * w + (p0 >> 32);
    const uint64_t lo = (p1 << 33) | (p0 & 0xFFFFFFFFu) << 1, sum = lo + kTwoPi50;
    const uint64_t hi = (p1 >> 31) + (sum < lo ? 1u : 0u);  // 2 pi (2 w + 1), units of 2^-83
    uint64_t a = hi << 42 | sum >> 22;
    const int drop = 11 - clz64(a | 1u);
    if (drop > 0) a = (a + (1ull << (drop - 1))) & ~((1ull << drop) - 1ull);
    // the middle of its part of a quadrant, and the rest
    const uint32_t part = 2u * (w >> 22) + 1u, j = (w >> 22) & 255u;
    const int64_t th = (int64_t)((a << 3) - (part * kPi1024 + (mul32(part, kPi1024Low) >> 32)));
    const bool neg = th < 0;
    const uint64_t t = (uint64_t)(neg ? -th : th), t2 = sqrhi(t);
    const uint32_t th2 = (uint32_t)(t2 >> 32), tm2 = (uint32_t)(t2 >> 16);  // units of 2^-32, 2^-48
    // sin t = t - t W, W = t2 (1/6 - t2/120); 1 - cos t = t2/2 - t2^2/24 + t2^3/720
    const uint64_t W = mulhi3(t2, 0x2AAAAAAAAAAAAAABull - (mul32(tm2, 35791394u) >> 16));
    const uint64_t st = t - mulhi3(t, W);
    const uint32_t t4 = (uint32_t)(mul32(tm2, tm2) >> 32), t6 = (uint32_t)(mul32(t4, th2) >> 32);
    const uint64_t m = (t2 >> 1) - (mul32(t4, 178956971u) >> 32) + (mul32(t6, 5965232u) >> 32);
    const uint64_t C = (uint64_t)T.cos_sin[2 * j], S = (uint64_t)T.cos_sin[2 * j + 1];
    const int64_t Ss = (int64_t)mulhi(S, st), Cs = (int64_t)mulhi(C, st);
    int64_t cq = (int64_t)(C - mulhi(C, m)) - (neg ? -Ss : Ss), sq = (int64_t)(S - mulhi(S, m)) + (neg ? -Cs : Cs);
    // (next to an axis the rounding can carry a 1 past the largest integer)
    if ((int32_t)(cq >> 32) < -0x40000000) cq = 0x7FFFFFFFFFFFFFFFll;
    if ((int32_t)(sq >> 32) < -0x40000000) sq = 0x7FFFFFFFFFFFFFFFll;
    const bool swap = (w >> 30) & 1u;                 // quadrants 1, 3
    co = swap ? sq : cq;
    si = swap ? cq : sq;
    if (((w >> 30) + 1u) & 2u) co = -co;              // quadrants 1, 2
    if (w >> 31) si = -si;                            // quadrants 2, 3
    return a;
}

__host__ __device__ __forceinline__ double to_double(int64_t v)
{
#ifdef __CUDA_ARCH__
    return __ll2double_rn(v);
#else
    return (double)v;
#endif
}

// Next to an axis (2^20 of w, |a - k pi/2| <= 2^-9.3) the digits of cos_sin's
// units leave the smaller of the two with an error of up to 4e-11 of itself.
// There it is, but for its sign, sin d = d (1 - d^2/6 + d^4/120), d = a - k pi/2
// to 96 digits.  In units of 2^-63.  (A call, as it is rare: one w in 512.)
constexpr uint32_t kAxis = 1u << 20;
static __host__ __device__ __noinline__ double near_axis(uint32_t w, uint64_t a)
{
    const uint32_t k = (w + kAxis) >> 30, last = w >> 31 & (k == 0u);  // axis 0 .. 3, or the first again: 4
    uint64_t h, l;                                                     // d, units of 2^-96
    bool neg = false;
    if (k + last != 0u) {
        // k pi / 2 (hexadecimal 1.921FB54442D18469898CC517 each)
        const uint64_t kh = k == 1u ? 0x1921FB544ull : (k == 2u ? 0x3243F6A88ull : (k == 3u ? 0x4B65F1FCCull : 0x6487ED511ull));
        const uint64_t kl = k == 1u ? 0x42D18469898CC517ull
                                    : (k == 2u ? 0x85A308D313198A2Eull
                                               : (k == 3u ? 0xC8748D3C9CA64F45ull : 0x0B4611A62633145Cull));
        h = a >> 29;
        l = a << 35;
        neg = h < kh || (h == kh && l < kl);
        const uint64_t sh = neg ? h : kh, sl = neg ? l : kl;
        h = neg ? kh : h;
        l = neg ? kl : l;
        h -= sh + (l < sl ? 1u : 0u);
        l -= sl;
    } else {
        // a itself, from 2 pi (2 w + 1) in units of 2^-83: to 53 bits, ties to even
        const uint64_t m = 2ull * w + 1ull, p = mul32((uint32_t)kTwoPi50, (uint32_t)m);
        const uint64_t q = mul32((uint32_t)(kTwoPi50 >> 32), (uint32_t)m) + (p >> 32);
        h = q >> 32;
        l = q << 32 | (uint32_t)p;
        const int drop = (h ? 128 - clz64(h) : 64 - clz64(l)) - 53;  // at most 21
        if (drop > 0) {
            const uint64_t half = 1ull << (drop - 1), rest = l & (2ull * half - 1ull);
            l -= rest;
            if (rest > half || (rest == half && (l >> drop & 1u))) {
                l += 2ull * half;
                h += l == 0ull ? 1u : 0u;
            }
        }
        h = h << 13 | l >> 51;
        l <<= 13;
    }
    const uint64_t t = h << 32 | l >> 32, t2 = sqrhi(t);
    const uint64_t W = mulhi3(t2, 0x2AAAAAAAAAAAAAABull) - (mul32((uint32_t)(t2 >> 16), (uint32_t)(t2 >> 16)) >> 32) / 120u;
    const int z = h ? clz64(h) : 64 + clz64(l);  // d = m 2^(-32 - z)
    const uint64_t m = z < 64 ? h << z | l >> (64 - z) : l << (z - 64);
    const int64_t s = (int64_t)((m - mulhi3(m, W)) >> 1);
    // sin d at axes 0, 3 (there the cosine) and 4, -sin d at 1 (the cosine), 2
    const double v = to_double((k == 1u || k == 2u) != neg ? -s : s);
    int64_t bits;
#ifdef __CUDA_ARCH__
    bits = __double_as_longlong(v);
#else
    __builtin_memcpy(&bits, &v, 8);
#endif
    bits += (int64_t)(32 - z) << 52;  // times 2^(32 - z)
#ifdef __CUDA_ARCH__
    return __longlong_as_double(bits);
#else
    double r;
    __builtin_memcpy(&r, &bits, 8);
    return r;
#endif
}

// The normals' parts as the problem states them in doubles: r = sqrt(-2 ln u1)
// (the logarithm and the root rounded), cosine c and sine s of a; r comes scaled
// by 2^-63 to the unit of the others, which are given as integers too; rf is r in
// single precision.
__host__ __device__ __forceinline__ void polar64(const Tables& T, uint32_t w1, uint32_t w2, double& r, float& rf,
                                                 int64_t& co, int64_t& si, double& c, double& s)
{
    uint64_t N;
    int E, H;
    neg_log(T, w1, N, E);
    uint64_t m = (N >> 11) + ((N >> 10) & 1u);  // 53 bits (2^53 at most)
    E += (int)(m >> 53);
    m <<= 11 - (int)(m >> 53);
    const uint64_t S = root(m, E + 1, H);
    // (the leading bit adds one to the exponent field)
    const uint64_t bits = ((uint64_t)(H + 1021 - 63) << 52) + (S >> 11) + ((S >> 10) & 1u);
    const uint32_t fbits = ((uint32_t)(H + 125) << 23) + (uint32_t)(S >> 40);
#ifdef __CUDA_ARCH__
    r = __longlong_as_double((long long)bits);
    rf = __uint_as_float(fbits);
#else
    __builtin_memcpy(&r, &bits, 8);
    __builtin_memcpy(&rf, &fbits, 4);
#endif
    const uint64_t a = cos_sin(T, w2, co, si);
    c = to_double(co);
    s = to_double(si);
    if (((w2 + kAxis) & 0x3FFFFFFFu) < 2u * kAxis) {
        const double v = near_axis(w2, a);
        if ((w2 + kAxis) >> 30 & 1u) c = v;
        else s = v;
    }
}

}  // namespace fx
}  // namespace mcg
