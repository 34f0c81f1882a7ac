// mcg_cell.cuh -- the field of a homogeneous box cell seen from a distance,
// as a series about its centre: with half-widths h and d the vector from the
// field point to the centre, the mean of 1 / |d + delta| over the cell is
//
//   f(d) = 1 / r + sum_n P_2n(d) / r^(4n + 1),   r = |d|,
//   P_2n / r^(4n + 1) = sum_(i+j+k=n) h_x^2i h_y^2j h_z^2k /
//                       ((2i+1)! (2j+1)! (2k+1)!)  d^(2i,2j,2k) (1 / r),
//
// the Taylor series of 1 / r averaged term by term.  P_2n is a homogeneous
// harmonic polynomial of degree 2n in the squares X, Y, Z of d's coordinates.
// Kept up to n = 4 (the field; n = 5 next to its near zone) or 5 (the tables):
// the relative remainder of n <= 4 for a cube is 4e-10 at four sides and 7e-12 at
// six (compared with 14^3-point Gauss quadrature for four cell shapes, the cube
// the worst); that of n <= 5 is 1e-8 at two sides, 1e-10 at three, 4e-12 at four
// (against the closed form in 40 digits).
// Along a row of cells (Y, Z fixed) every P_2n is a short polynomial in X.
#pragma once
#include <cuda_runtime.h>

namespace mcg {

constexpr int kSeriesOrders = 5;
constexpr int kSeriesTerms = 3 + 6 + 10 + 15 + 21;

// Coefficients of P_2, P_4, .. P_10 in that order, each with its monomials
// X^a Y^b Z^c by falling a, then falling b (host; mcg_field.cu).
void cell_series(const double h[3], double out[kSeriesTerms]);

// A number as an unevaluated sum of two single-precision ones.
struct Pair {
    float h, l;
};

__device__ __forceinline__ Pair pair_of(double v)
{
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}
__device__ __forceinline__ Pair mul(Pair a, Pair b)
{
    const float h = __fmul_rn(a.h, b.h);
    return {h, fmaf(a.h, b.l, fmaf(a.l, b.h, __fmaf_rn(a.h, b.h, -h)))};
}
__device__ __forceinline__ Pair add(Pair a, Pair b)
{
    const float h = __fadd_rn(a.h, b.h), t = __fsub_rn(h, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(h, t)), __fsub_rn(b.h, t));
    return {h, e + (a.l + b.l)};
}
// The same number, its leading part the nearest float.
__device__ __forceinline__ Pair rounded(Pair a)
{
    const float h = __fadd_rn(a.h, a.l);
    return {h, __fsub_rn(a.l, __fsub_rn(h, a.h))};
}
// a + b, |a| >= |b|
__device__ __forceinline__ Pair add_small(Pair a, Pair b)
{
    const float h = __fadd_rn(a.h, b.h);
    return {h, __fsub_rn(b.h, __fsub_rn(h, a.h)) + (a.l + b.l)};
}

// A row's polynomials in X: f's correction terms and, for df/dz = d_z (...),
// the derivatives by Z.
struct SeriesRow {
    float c4[2], c6[3], c8[4], c10[5];  // coefficients of X^(n-1) .. X^0 (X^n is the row's constant)
    float d4, d6[2], d8[3];             // of dP/dZ below its leading constant
};

__device__ __forceinline__ SeriesRow series_row(const float* p, float Y, float Z)
{
    const float *q4 = p + 3, *q6 = p + 9, *q8 = p + 19, *q10 = p + 34;
    SeriesRow r;
    r.c4[0] = fmaf(q4[1], Y, q4[2] * Z);
    r.c4[1] = fmaf(fmaf(q4[3], Y, q4[4] * Z), Y, q4[5] * Z * Z);
    r.c6[0] = fmaf(q6[1], Y, q6[2] * Z);
    r.c6[1] = fmaf(fmaf(q6[3], Y, q6[4] * Z), Y, q6[5] * Z * Z);
    r.c6[2] = fmaf(fmaf(fmaf(q6[6], Y, q6[7] * Z), Y, q6[8] * Z * Z), Y, q6[9] * Z * Z * Z);
    r.c8[0] = fmaf(q8[1], Y, q8[2] * Z);
    r.c8[1] = fmaf(fmaf(q8[3], Y, q8[4] * Z), Y, q8[5] * Z * Z);
    r.c8[2] = fmaf(fmaf(fmaf(q8[6], Y, q8[7] * Z), Y, q8[8] * Z * Z), Y, q8[9] * Z * Z * Z);
    r.c8[3] = fmaf(fmaf(fmaf(fmaf(q8[10], Y, q8[11] * Z), Y, q8[12] * Z * Z), Y, q8[13] * Z * Z * Z), Y,
                   q8[14] * Z * Z * Z * Z);
    const float Z2 = Z * Z, Z4 = Z2 * Z2;
    r.c10[0] = fmaf(q10[1], Y, q10[2] * Z);
    r.c10[1] = fmaf(fmaf(q10[3], Y, q10[4] * Z), Y, q10[5] * Z2);
    r.c10[2] = fmaf(fmaf(fmaf(q10[6], Y, q10[7] * Z), Y, q10[8] * Z2), Y, q10[9] * Z2 * Z);
    r.c10[3] = fmaf(fmaf(fmaf(fmaf(q10[10], Y, q10[11] * Z), Y, q10[12] * Z2), Y, q10[13] * Z2 * Z), Y, q10[14] * Z4);
    r.c10[4] = fmaf(fmaf(fmaf(fmaf(fmaf(q10[15], Y, q10[16] * Z), Y, q10[17] * Z2), Y, q10[18] * Z2 * Z), Y,
                         q10[19] * Z4), Y, q10[20] * Z4 * Z);
    r.d4 = fmaf(q4[4], Y, 2.0f * q4[5] * Z);
    r.d6[0] = fmaf(q6[4], Y, 2.0f * q6[5] * Z);
    r.d6[1] = fmaf(fmaf(q6[7], Y, 2.0f * q6[8] * Z), Y, 3.0f * q6[9] * Z * Z);
    r.d8[0] = fmaf(q8[4], Y, 2.0f * q8[5] * Z);
    r.d8[1] = fmaf(fmaf(q8[7], Y, 2.0f * q8[8] * Z), Y, 3.0f * q8[9] * Z * Z);
    r.d8[2] = fmaf(fmaf(fmaf(q8[11], Y, 2.0f * q8[12] * Z), Y, 3.0f * q8[13] * Z * Z), Y, 4.0f * q8[14] * Z * Z * Z);
    return r;
}

// P_4, P_6, P_8 and the value, the sum over them of P_2n y^(4n+1), y = 1 / r, in
// single precision: the terms are at most 5e-5 of 1 / r from four cell sides.
__device__ __forceinline__ void series_polys(const float* p, const SeriesRow& r, float X, float& P4, float& P6,
                                             float& P8)
{
    P4 = fmaf(fmaf(p[3], X, r.c4[0]), X, r.c4[1]);
    P6 = fmaf(fmaf(fmaf(p[9], X, r.c6[0]), X, r.c6[1]), X, r.c6[2]);
    P8 = fmaf(fmaf(fmaf(fmaf(p[19], X, r.c8[0]), X, r.c8[1]), X, r.c8[2]), X, r.c8[3]);
}

__device__ __forceinline__ float series_value(float P4, float P6, float P8, float y, float y2)
{
    const float y4 = y2 * y2;
    return y4 * y4 * y * fmaf(y4, fmaf(y4, P8, P6), P4);
}

// P_10, and P_10 y^21.
__device__ __forceinline__ float series_p10(const float* p, const SeriesRow& r, float X)
{
    return fmaf(fmaf(fmaf(fmaf(fmaf(p[34], X, r.c10[0]), X, r.c10[1]), X, r.c10[2]), X, r.c10[3]), X, r.c10[4]);
}
__device__ __forceinline__ float series_tenth(const float* p, const SeriesRow& r, float X, float y, float y2)
{
    const float y4 = y2 * y2, y8 = y4 * y4;
    return y8 * y8 * y4 * y * series_p10(p, r, X);
}

// The same terms (n = 2, 3, 4) of (df/dz) / d_z: 2 dP_2n/dZ y^(4n+1) - (4n+1) P_2n y^(4n+3);
// n = 3 and 4 by y^13.
__device__ __forceinline__ float slope_rest(const float* p, const SeriesRow& r, float X, float P6, float P8, float y2)
{
    const float D6 = fmaf(fmaf(p[11], X, r.d6[0]), X, r.d6[1]);
    const float D8 = fmaf(fmaf(fmaf(p[21], X, r.d8[0]), X, r.d8[1]), X, r.d8[2]);
    const float t6 = fmaf(-13.0f * y2, P6, 2.0f * D6), t8 = fmaf(-17.0f * y2, P8, 2.0f * D8);
    return fmaf(y2 * y2, t8, t6);
}
__device__ __forceinline__ float series_slope(const float* p, const SeriesRow& r, float X, float P4, float P6,
                                              float P8, float y, float y2)
{
    const float D4 = fmaf(p[5], X, r.d4);
    const float t4 = fmaf(-9.0f * y2, P4, 2.0f * D4);
    const float y4 = y2 * y2;
    return y4 * y4 * y * fmaf(y4, slope_rest(p, r, X, P6, P8, y2), t4);
}

// P_2 y^5, the second-order term of a cell that is not a cube (P_2 = 0 for
// one), up to 2e-3 of 1 / r at six sides and of one sign over whole regions:
// as a pair.  p0: P_2's coefficient of X, c: the row's rest.
__device__ __forceinline__ Pair series_second(Pair p0, Pair c, Pair X, Pair y, Pair y2, Pair& P2, Pair& y5)
{
    P2 = add(mul(p0, X), c);
    y5 = mul(mul(y2, y2), y);
    return mul(P2, y5);
}

// 1 / sqrt(s) as a pair, relative error below 2^-45: the
// hardware root (22 bits) and one third-order step whose residual
// 1 - s y^2 is formed exactly in two pieces.
// Also y^2 as a pair.
__device__ __forceinline__ Pair rsqrt_pair(Pair s, Pair& y2)
{
    Pair y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.h) : "f"(s.h));
    y2.h = __fmul_rn(y.h, y.h);
    y2.l = __fmaf_rn(y.h, y.h, -y2.h);
    float e = fmaf(-s.h, y2.h, 1.0f);
    e = fmaf(-s.h, y2.l, e);
    e = fmaf(-s.l, y2.h, e);
    y.l = y.h * e * fmaf(0.375f, e, 0.5f);
    y2.l = fmaf(2.0f * y.h, y.l, y2.l);
    return y;
}

// What series_value and series_slope lack of a cell's own terms, in single
// precision: the digits of P_4's (as pairs; p4: its coefficients), and P_10's.
__device__ __forceinline__ void series_lacks(const float* p, const Pair* p4, Pair X, Pair Y, Pair Z, float& f, float& g)
{
    const SeriesRow r = series_row(p, Y.h, Z.h);
    Pair y2;
    const Pair y = rsqrt_pair(add(X, rounded(add(Y, Z))), y2);
    float P4, P6, P8;
    series_polys(p, r, X.h, P4, P6, P8);
    const float v = series_value(P4, P6, P8, y.h, y2.h), s = series_slope(p, r, X.h, P4, P6, P8, y.h, y2.h);
    const float y4 = y2.h * y2.h, y13 = y4 * y4 * y4 * y.h;
    const float v68 = y13 * fmaf(y4, P8, P6), s68 = y13 * slope_rest(p, r, X.h, P6, P8, y2.h);
    // P_10 and 2 dP_10/dZ - 21 P_10 y^2, of the direction: homogeneous of degree 5 and
    // 4, so that no power above y^13 is formed (in a long grid y is 100 and more)
    const float x1 = X.h * y2.h, y1 = Y.h * y2.h, z1 = Z.h * y2.h, z2 = z1 * z1, z3 = z2 * z1;
    const SeriesRow u = series_row(p, y1, z1);
    const float* q = p + 34;
    const float d3 = fmaf(q[4], y1, 2.0f * q[5] * z1);
    const float d2 = fmaf(fmaf(q[7], y1, 2.0f * q[8] * z1), y1, 3.0f * q[9] * z2);
    const float d1 = fmaf(fmaf(fmaf(q[11], y1, 2.0f * q[12] * z1), y1, 3.0f * q[13] * z2), y1, 4.0f * q[14] * z3);
    const float d0 = fmaf(fmaf(fmaf(fmaf(q[16], y1, 2.0f * q[17] * z1), y1, 3.0f * q[18] * z2), y1,
                               4.0f * q[19] * z3), y1, 5.0f * q[20] * z2 * z2);
    const float D10 = fmaf(fmaf(fmaf(fmaf(q[2], x1, d3), x1, d2), x1, d1), x1, d0);
    const float P10 = series_p10(p, u, x1);
    const float v10 = y4 * y4 * y2.h * y.h * P10, s10 = y13 * fmaf(-21.0f, P10, 2.0f * D10);
    // P_4 and 2 dP_4/dZ - 9 P_4 y^2
    const Pair a = add(mul(p4[1], Y), mul(p4[2], Z));
    const Pair b = add(mul(add(mul(p4[3], Y), mul(p4[4], Z)), Y), mul(mul(p4[5], Z), Z));
    const Pair P = add(mul(add(mul(p4[0], X), a), X), b);
    const Pair D = add(add(mul(p4[2], X), mul(p4[4], Y)), mul({2.0f, 0.0f}, mul(p4[5], Z)));
    const Pair u4 = mul(y2, y2), u9 = mul(mul(u4, u4), y);
    const Pair V = mul(P, u9), S = mul(add(mul({2.0f, 0.0f}, D), mul({-9.0f, 0.0f}, mul(P, y2))), u9);
    f = ((V.h - v) + v68) + (V.l + v10);
    g = ((S.h - s) + s68) + (S.l + s10);
}

// sum += v without losing the rounding of the leading parts.
__device__ __forceinline__ void accumulate(Pair& sum, Pair v)
{
    const Pair r = add({sum.h, 0.0f}, {v.h, 0.0f});
    sum.h = r.h;
    sum.l += r.l + v.l;
}

}  // namespace mcg
