// mcg_field.cu -- the exact potential Phi and vertical gravity dPhi/dz of the
// density models at arbitrary points: the closed forms the walk's estimates
// are checked against (the paper compares its stochastic solution with the
// analytic prism field, Sec. 4.2, and with a finite-element solution).
//
//  * sphere: -G M / r outside, -G M (3 a^2 - r^2) / (2 a^3) inside;
//  * prism : Nagy's corner function F summed over the eight corners,
//            Phi = -G rho [[[F]]], dPhi/dz = G rho [[[dF/dz]]];
//  * voxel : the sum of the voxels' prism fields.  Cells near the point are
//            summed by grid node: every node is a corner of up to eight cells,
//            each adding its density with the corner's sign, so
//              Phi(x) = -G sum_nodes w_n F(n - x),  w_n = sum_cells s rho,
//            one corner-function evaluation per node instead of eight per
//            cell, in double precision.  All other cells use the series of
//            mcg_cell.cuh, its leading term in pairs of single-precision
//            numbers.
#include <algorithm>
#include <cmath>
#include <cstring>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "mcg_cell.cuh"
#include "mcg_device.cuh"
#include "mcg_internal.h"

namespace mcg {

namespace {

struct FieldParams {
    int32_t kind;
    double G, rho0;
    double c[3], a;           // sphere
    double lo[3], hi[3];      // prism
    const float* grid;        // voxel grid, x fastest
    int32_t nx, ny, nz;
    double org[3], sp[3];
    double series[kSeriesTerms];  // cell_series of a cell
    double near;              // cells with a centre within this of the point (per axis) are summed by node
    const double* x;          // points, n x 3
    int64_t n;
    double* phi;
    double* gz;
};

__device__ __forceinline__ void neumaier(double& s, double& c, double v)
{
    const double t = s + v;
    if (fabs(s) >= fabs(v)) c += (s - t) + v;
    else c += (v - t) + s;
    s = t;
}

// F(x, y, z) and dF/dz of the prism corner function (Nagy):
//   F     = xy ln(z+r) + yz ln(x+r) + zx ln(y+r)
//           - x^2/2 atan(yz/(xr)) - y^2/2 atan(zx/(yr)) - z^2/2 atan(xy/(zr)),
//   dF/dz = x ln(y+r) + y ln(x+r) - z atan(xy/(zr)),
// a term whose polynomial prefactor is 0 taken as its limit 0; the two share
// their logarithms and the z arctangent.
__device__ __forceinline__ void corner_f_dfdz(double x, double y, double z, double& F, double& D)
{
    F = 0.0;
    D = 0.0;
    const double r = sqrt(x * x + y * y + z * z);
    if (r == 0.0) return;
    const double lx = (y != 0.0) ? log_tr(x, y, z, r) : 0.0;   // ln(x + r)
    const double ly = (x != 0.0) ? log_tr(y, z, x, r) : 0.0;   // ln(y + r)
    if (x * y != 0.0) F += x * y * log_tr(z, x, y, r);
    if (y * z != 0.0) F += y * z * lx;
    if (z * x != 0.0) F += z * x * ly;
    if (x != 0.0) F -= 0.5 * x * x * atan(y * z / (x * r));
    if (y != 0.0) F -= 0.5 * y * y * atan(z * x / (y * r));
    if (x != 0.0) D += x * ly;
    if (y != 0.0) D += y * lx;
    if (z != 0.0) {
        const double az = atan(x * y / (z * r));
        F -= 0.5 * z * z * az;
        D -= z * az;
    }
}

// Closed forms of the sphere and the prism, one thread per point.
__global__ void field_closed_kernel(const FieldParams P)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    const double* x = P.x + 3 * i;
    double phi = 0.0, gz = 0.0;   // no density: no field
    if (P.kind == MCG_RHO_SPHERE) {
        const double dx = x[0] - P.c[0], dy = x[1] - P.c[1], dz = x[2] - P.c[2];
        const double r = sqrt(dx * dx + dy * dy + dz * dz);
        const double M = 4.0 / 3.0 * 3.14159265358979323846 * P.a * P.a * P.a * P.rho0;
        if (r >= P.a) {
            phi = -P.G * M / r;
            gz = P.G * M * dz / (r * r * r);
        } else {
            phi = -P.G * M * (3.0 * P.a * P.a - r * r) / (2.0 * P.a * P.a * P.a);
            gz = P.G * M * dz / (P.a * P.a * P.a);
        }
    } else if (P.kind == MCG_RHO_PRISM) {
        double sf = 0.0, sd = 0.0;
        for (int c = 0; c < 8; ++c) {
            const int ci = c & 1, cj = (c >> 1) & 1, ck = (c >> 2) & 1;
            double F, D;
            corner_f_dfdz((ci ? P.hi[0] : P.lo[0]) - x[0], (cj ? P.hi[1] : P.lo[1]) - x[1],
                          (ck ? P.hi[2] : P.lo[2]) - x[2], F, D);
            const bool neg = ((3 - ci - cj - ck) & 1) != 0;   // sign flips with every lower limit
            sf += neg ? -F : F;
            sd += neg ? -D : D;
        }
        phi = -P.G * P.rho0 * sf;
        gz = P.G * P.rho0 * sd;
    }
    if (P.phi) P.phi[i] = phi;
    if (P.gz) P.gz[i] = gz;
}

// ---------------------------------------------------------------------------
// Voxel model.  A cluster of blocks per point (one block where there are
// many points).  What bounds it: GB300 does 1.6 double-precision operations a
// clock and SM against 128 single-precision ones, and a corner function takes
// about 390 of them, so the sum over every node of a 128 x 128 x 64 grid
// spent 0.9 ms a point and SM-wave in the double-precision pipe (231 ms for
// 256 points).  Only the cells within kNearCells sides of the point need it;
// the others take ~95 single-precision instructions: a thread runs a row of
// cells (its Y, Z polynomials in registers), 16 columns of 256 rows at a time
// through shared memory so that the grid is read in whole sectors.  What the
// single-precision terms of the far cells next to the near ones lack (P_4's
// digits, P_10) is added for them apart, in pairs.  Now 2.6 ms (one point
// 0.30 ms; flat 16 x 128 x 64 cells 9.6 ms).  Error, in units of the cells' own
// terms added up, against 64-bit mantissas (nine grids, points on, in and
// around them): 1e-13 at most, for df/dz (all nodes in doubles: 3e-12; without
// the rim: 5e-13).
// ---------------------------------------------------------------------------
constexpr int kFieldThreads = 256;
constexpr int kFieldCols = 16;
constexpr double kNearCells = 6.0, kRimCells = 8.0;

// The rim: far cells up to kRimCells sides from the point, next to the near ones, and
// what their single-precision terms lack: beyond, 1e-12 of a cell's df/dz.  (A
// call, and its set-up after the loop over all cells: that loop lost 4 to 6 %
// with either in its way.)
struct Rim {
    int first[3], count[3];  // cells along each axis, the near ones lo .. hi - 1 among them
    int lo[3], hi[3];
    Pair d0[3], step[3];     // the first cell's centre, and from cell to cell
};
__device__ __noinline__ float2 rim_sum(const float* grid, int nx, int ny, const Rim& R, const float* sp, const Pair* sp4,
                                       int64_t from, int stride)
{
    const int64_t cells = (int64_t)R.count[0] * R.count[1] * R.count[2];
    float2 sum = {0.0f, 0.0f};
    for (int64_t q = from; q < cells; q += stride) {
        const int64_t row = q / R.count[0];
        const int c[3] = {(int)(q - row * R.count[0]), (int)(row % R.count[1]), (int)(row / R.count[1])};
        const int ix = R.first[0] + c[0], iy = R.first[1] + c[1], iz = R.first[2] + c[2];
        if (ix >= R.lo[0] && ix < R.hi[0] && iy >= R.lo[1] && iy < R.hi[1] && iz >= R.lo[2] && iz < R.hi[2]) continue;
        const float rho = __ldg(grid + ix + (int64_t)nx * (iy + (int64_t)ny * iz));
        Pair d[3], sq[3];
        for (int k = 0; k < 3; ++k) {
            d[k] = add(R.d0[k], mul({(float)c[k], 0.0f}, R.step[k]));
            sq[k] = rounded(mul(d[k], d[k]));
        }
        float f, g;
        series_lacks(sp, sp4, sq[0], sq[1], sq[2], f, g);
        sum.x = fmaf(rho, f, sum.x);
        sum.y = fmaf(rho * d[2].h, g, sum.y);
    }
    return sum;
}

template <bool CUBE>
__global__ void __launch_bounds__(kFieldThreads, 2) field_voxel_kernel(const FieldParams P)
{
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int parts = (int)cluster.num_blocks(), part = (int)cluster.block_rank();
    __shared__ float tile[kFieldThreads][kFieldCols + 1];
    __shared__ Pair sx[kFieldCols];     // X of the tile's columns
    __shared__ Pair sp4[6];  
    __shared__ Rim rim;
    __shared__ float sp[kSeriesTerms];   // the series for lengths in units of L
    __shared__ double red[2][kFieldThreads / 32], total[2];
    const int64_t i = blockIdx.x / parts;
    const int t = threadIdx.x;
    const double x[3] = {P.x[3 * i], P.x[3 * i + 1], P.x[3 * i + 2]};
    const int n[3] = {P.nx, P.ny, P.nz};
    // the near cells, and the unit of length: the geometric mean of the
    // nearest and the farthest distance keeps r^8 and r^-17 within range
    int lo[3], hi[3];  // near cells lo .. hi - 1 along each axis
    double out2 = 0.0, far2 = 0.0;
    for (int k = 0; k < 3; ++k) {
        const double a = (x[k] - P.org[k]) / P.sp[k], w = P.near / P.sp[k];
        lo[k] = (int)fmin(fmax(ceil(a - w - 0.5), 0.0), (double)n[k]);
        hi[k] = (int)fmin(fmax(floor(a + w - 0.5) + 1.0, 0.0), (double)n[k]);
        const double g0 = P.org[k] - x[k], g1 = g0 + n[k] * P.sp[k];
        const double o = fmax(fmax(g0, -g1), 0.0), f = fmax(fabs(g0), fabs(g1));
        out2 += o * o;
        far2 += f * f;
    }
    const bool none_near = lo[0] >= hi[0] || lo[1] >= hi[1] || lo[2] >= hi[2];
    if (none_near)
        for (int k = 0; k < 3; ++k) lo[k] = hi[k] = 0;
    const double L = sqrt(fmax(sqrt(out2), P.near) * sqrt(far2)), invL = 1.0 / L;
    if (t < kSeriesTerms) {
        const double q = invL * invL, q2 = q * q;
        const double v = P.series[t] * (t < 3 ? q : t < 9 ? q2 : t < 19 ? q2 * q : t < 34 ? q2 * q2 : q2 * q2 * q);
        sp[t] = (float)v;
        if (t >= 3 && t < 9) sp4[t - 3] = pair_of(v);
    }

    // far cells: sum of rho f and of rho (df/dz), lengths in units of L
    double phi = 0.0, gz = 0.0;
    const int64_t rows = (int64_t)P.ny * P.nz;
    const Pair p2x = pair_of(P.series[0] * invL * invL), p2z2 = pair_of(2.0 * P.series[2] * invL * invL);
    for (int64_t r0 = (int64_t)part * kFieldThreads; r0 < rows; r0 += (int64_t)parts * kFieldThreads) {
        const int64_t row = r0 + t;
        const int iy = (int)(row % P.ny), iz = (int)(row / P.ny);
        const double dy = (P.org[1] + (iy + 0.5) * P.sp[1] - x[1]) * invL,
                     dz = (P.org[2] + (iz + 0.5) * P.sp[2] - x[2]) * invL;
        const Pair yz = pair_of(dy * dy + dz * dz);
        const Pair c2 = pair_of((P.series[1] * dy * dy + P.series[2] * dz * dz) * invL * invL);
        SeriesRow sr;
        Pair fs = {0.f, 0.f}, gs = {0.f, 0.f};  // the row's sums
        for (int c0 = 0; c0 < P.nx; c0 += kFieldCols) {
            __syncthreads();
            for (int e = t; e < kFieldThreads * kFieldCols; e += kFieldThreads) {
                const int er = e / kFieldCols, ec = e % kFieldCols;
                const int64_t rr = r0 + er;
                const int ix = c0 + ec;
                float v = 0.f;
                if (rr < rows && ix < P.nx) {
                    const int jy = (int)(rr % P.ny), jz = (int)(rr / P.ny);
                    const bool near = ix >= lo[0] && ix < hi[0] && jy >= lo[1] && jy < hi[1] && jz >= lo[2] && jz < hi[2];
                    if (!near) v = __ldg(P.grid + rr * P.nx + ix);
                }
                tile[er][ec] = v;
            }
            if (t < kFieldCols) {
                const double dx = (P.org[0] + (c0 + t + 0.5) * P.sp[0] - x[0]) * invL, X = dx * dx;
                sx[t] = pair_of(X);
            }
            __syncthreads();
            if (c0 == 0) sr = series_row(sp, (float)(dy * dy), (float)(dz * dz));
            const int cols = P.nx - c0 < kFieldCols ? P.nx - c0 : kFieldCols;
#pragma unroll 2
            for (int c = 0; c < cols; ++c) {
                const float rho = tile[t][c];
                if (rho == 0.0f) continue;  // (near, outside the grid, or empty)
                const Pair X = sx[c];
                Pair y2;
                const Pair y = rsqrt_pair(add(X, yz), y2);
                float P4, P6, P8;
                series_polys(sp, sr, X.h, P4, P6, P8);
                Pair f = {y.h, y.l + series_value(P4, P6, P8, y.h, y2.h)};
                const Pair y3 = mul(y, y2);
                Pair g = {-y3.h, series_slope(sp, sr, X.h, P4, P6, P8, y.h, y2.h) - y3.l};
                if constexpr (!CUBE) {
                    Pair P2, y5;
                    const Pair v = series_second(p2x, c2, X, y, y2, P2, y5);
                    f = add_small(f, v);
                    // 2 dP_2/dZ y^5 - 5 P_2 y^7
                    const Pair w = mul(mul(P2, y2), {-5.0f, 0.0f});
                    g = add_small(g, mul(add(p2z2, w), y5));
                }
                accumulate(fs, mul({rho, 0.0f}, f));
                accumulate(gs, mul({rho, 0.0f}, g));
            }
        }
        phi += (double)fs.h + (double)fs.l;
        gz += dz * ((double)gs.h + (double)gs.l);
    }
    if (t >= 64 && t < 67) {  // (a thread per axis: all of them would wait for the double-precision pipe)
        const int k = t - 64, nk = k == 0 ? P.nx : (k == 1 ? P.ny : P.nz);
        const double xk = P.x[3 * i + k], a = (xk - P.org[k]) / P.sp[k], w = P.near * (kRimCells / kNearCells) / P.sp[k];
        const int first = (int)fmin(fmax(ceil(a - w - 0.5), 0.0), (double)nk);
        rim.first[k] = first;
        rim.count[k] = max((int)fmin(fmax(floor(a + w - 0.5) + 1.0, 0.0), (double)nk) - first, 0);
        rim.lo[k] = k == 0 ? lo[0] : (k == 1 ? lo[1] : lo[2]);
        rim.hi[k] = k == 0 ? hi[0] : (k == 1 ? hi[1] : hi[2]);
        rim.d0[k] = pair_of((P.org[k] + (first + 0.5) * P.sp[k] - xk) * invL);
        rim.step[k] = pair_of(P.sp[k] * invL);
    }
    __syncthreads();  // (sp: a block may have had no rows)
    {
        const float2 lacks = rim_sum(P.grid, P.nx, P.ny, rim, sp, sp4, part * kFieldThreads + t, parts * kFieldThreads);
        phi += (double)lacks.x;
        gz += (double)lacks.y;
    }
    const double V = P.sp[0] * P.sp[1] * P.sp[2];
    phi *= V * invL;
    gz *= V * invL * invL;

    // near cells: their nodes lo .. hi, each with the weight of the near
    // cells it belongs to (upper corner, sign +, of the cell before it along
    // an axis, lower corner, sign -, of its own)
    if (!none_near) {
        const int mx = hi[0] - lo[0] + 1, my = hi[1] - lo[1] + 1, mz = hi[2] - lo[2] + 1;
        const int64_t nodes = (int64_t)mx * my * mz;
        double sf = 0.0, cf = 0.0, sd = 0.0, cd = 0.0;
        for (int64_t q = (int64_t)part * kFieldThreads + t; q < nodes; q += (int64_t)parts * kFieldThreads) {
            const int a = lo[0] + (int)(q % mx), b = lo[1] + (int)((q / mx) % my), c = lo[2] + (int)(q / ((int64_t)mx * my));
            double w = 0.0;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int di = m & 1, dj = (m >> 1) & 1, dk = (m >> 2) & 1;
                const int ci = a - 1 + di, cj = b - 1 + dj, ck = c - 1 + dk;
                double v = 0.0;
                if (ci >= lo[0] && ci < hi[0] && cj >= lo[1] && cj < hi[1] && ck >= lo[2] && ck < hi[2])
                    v = (double)__ldg(P.grid + ci + (int64_t)P.nx * (cj + (int64_t)P.ny * ck));
                w += ((di + dj + dk) & 1) ? -v : v;
            }
            if (w == 0.0) continue;
            double F, D;
            corner_f_dfdz(P.org[0] + a * P.sp[0] - x[0], P.org[1] + b * P.sp[1] - x[1], P.org[2] + c * P.sp[2] - x[2],
                          F, D);
            neumaier(sf, cf, w * F);
            neumaier(sd, cd, w * D);
        }
        phi += sf + cf;
        gz += sd + cd;
    }

    // block sums, then the cluster's, in a fixed order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        phi += __shfl_xor_sync(0xffffffffu, phi, o);
        gz += __shfl_xor_sync(0xffffffffu, gz, o);
    }
    if ((t & 31) == 0) {
        red[0][t >> 5] = phi;
        red[1][t >> 5] = gz;
    }
    __syncthreads();
    if (t < 2) {
        double v = 0.0;
        for (int w = 0; w < kFieldThreads / 32; ++w) v += red[t][w];
        total[t] = v;
    }
    cluster.sync();
    if (part == 0 && t < 2) {
        double v = 0.0;
        for (int b = 0; b < parts; ++b) v += *cluster.map_shared_rank(&total[t], b);
        if (t == 0 && P.phi) P.phi[i] = -P.G * v;
        if (t == 1 && P.gz) P.gz[i] = P.G * v;
    }
    cluster.sync();  // the other blocks' shared memory stays until it has been read
}

// The walks' own density samplers at given points and their two copies
// (x, y, z + h), (x, y, z - h), out[3 i + c]: the mixed walk's single-
// precision sampler on the point taken relative to the domain centre (the
// walk's frame), or the plain walk's double-precision sampler.
template <int RHO>
__global__ void density_f32_kernel(const WalkParams P, const double* __restrict__ x, int64_t n,
                                   double* __restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float wx = (float)(x[3 * i] - P.cen[0]), wy = (float)(x[3 * i + 1] - P.cen[1]),
                wz = (float)(x[3 * i + 2] - P.cen[2]);
    float a, b, c;
    rho3_f32<RHO>(P, model_of(P), wx, wy, wz, P.h_f, a, b, c);
    out[3 * i] = a;
    out[3 * i + 1] = b;
    out[3 * i + 2] = c;
}

__global__ void density_f64_kernel(const WalkParams P, const double* __restrict__ x, int64_t n,
                                   double* __restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double off[3] = {0.0, P.h, -P.h};
    for (int c = 0; c < 3; ++c) {
        const double X[3] = {x[3 * i], x[3 * i + 1], __dadd_rn(x[3 * i + 2], off[c])};
        out[3 * i + c] = rho_f64(P, model_of(P), X);
    }
}

// The integer polynomials d^(2i,2j,2k) (1 / r) r^(4n+1), n = i + j + k: one
// derivative at a time, d_x (P / r^m) = (r^2 d_x P - m x P) / r^(m+2).
struct DerivativeTable {
    // [n-1][index of (i, j, k)][index of the monomial], both by falling first
    // and second exponent
    double c[kSeriesOrders][21][21];
    DerivativeTable()
    {
        constexpr int N = 2 * kSeriesOrders + 1;  // exponents 0 .. 10
        auto at = [](int a, int b, int c) { return (a * N + b) * N + c; };
        std::memset(c, 0, sizeof(c));
        for (int n = 1; n <= kSeriesOrders; ++n)
            for (int i = n, e = 0; i >= 0; --i)
                for (int j = n - i; j >= 0; --j, ++e) {
                    const int order[3] = {2 * i, 2 * j, 2 * (n - i - j)};
                    double P[N * N * N] = {};
                    P[0] = 1.0;
                    int m = 1, deg = 0;
                    for (int ax = 0; ax < 3; ++ax)
                        for (int d = 0; d < order[ax]; ++d, m += 2, ++deg) {
                            double Q[N * N * N] = {};
                            for (int a = 0; a <= deg; ++a)
                                for (int b = 0; a + b <= deg; ++b) {
                                    const int x[3] = {a, b, deg - a - b};
                                    const double v = P[at(x[0], x[1], x[2])];
                                    if (v == 0.0) continue;
                                    int y[3] = {x[0], x[1], x[2]};
                                    ++y[ax];
                                    Q[at(y[0], y[1], y[2])] -= m * v;
                                    if (x[ax] == 0) continue;
                                    for (int k = 0; k < 3; ++k) {
                                        int z[3] = {x[0], x[1], x[2]};
                                        --z[ax];
                                        z[k] += 2;
                                        Q[at(z[0], z[1], z[2])] += x[ax] * v;
                                    }
                                }
                            std::memcpy(P, Q, sizeof(P));
                        }
                    for (int a = n, q = 0; a >= 0; --a)
                        for (int b = n - a; b >= 0; --b, ++q) c[n - 1][e][q] = P[at(2 * a, 2 * b, 2 * (n - a - b))];
                }
    }
};

}  // namespace

void cell_series(const double h[3], double out[kSeriesTerms])
{
    static const DerivativeTable T;
    const double fact[kSeriesOrders + 1] = {1.0, 6.0, 120.0, 5040.0, 362880.0, 39916800.0};  // (2i + 1)!
    double* o = out;
    for (int n = 1; n <= kSeriesOrders; ++n) {
        const int terms = (n + 1) * (n + 2) / 2;
        for (int q = 0; q < terms; ++q) o[q] = 0.0;
        for (int i = n, e = 0; i >= 0; --i)
            for (int j = n - i; j >= 0; --j, ++e) {
                const int k = n - i - j;
                const double w = std::pow(h[0], 2 * i) * std::pow(h[1], 2 * j) * std::pow(h[2], 2 * k) /
                                 (fact[i] * fact[j] * fact[k]);
                for (int q = 0; q < terms; ++q) o[q] += w * T.c[n - 1][e][q];
            }
        o += terms;
    }
}

void preload_field_kernels()
{
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, (const void*)field_closed_kernel) != cudaSuccess) cudaGetLastError();
    if (cudaFuncGetAttributes(&a, (const void*)field_voxel_kernel<true>) != cudaSuccess) cudaGetLastError();
    if (cudaFuncGetAttributes(&a, (const void*)field_voxel_kernel<false>) != cudaSuccess) cudaGetLastError();
    const void* fns[6] = {(const void*)density_f64_kernel,           (const void*)density_f32_kernel<MCG_RHO_NONE>,
                          (const void*)density_f32_kernel<MCG_RHO_SPHERE>, (const void*)density_f32_kernel<MCG_RHO_PRISM>,
                          (const void*)density_f32_kernel<MCG_RHO_VOXEL>,  (const void*)density_f32_kernel<kRhoVoxelPacked>};
    for (const void* f : fns)
        if (cudaFuncGetAttributes(&a, f) != cudaSuccess) cudaGetLastError();
}

}  // namespace mcg

using namespace mcg;

extern "C" int mcg_field(const mcg_density* density, const double* points_dev, int64_t n, double* phi_dev,
                         double* gz_dev, void* stream)
{
    if (!density) return set_error(MCG_ERR_ARG, "null density");
    if (n < 0) return set_error(MCG_ERR_ARG, "n must be non-negative");
    if (n == 0 || (!phi_dev && !gz_dev)) return MCG_OK;
    if (!points_dev) return set_error(MCG_ERR_ARG, "null points");
    if (!std::isfinite(density->G)) return set_error(MCG_ERR_ARG, "G must be finite");
    preload_kernels();
    FieldParams P;
    std::memset(&P, 0, sizeof(P));
    P.kind = density->kind;
    P.G = density->G;
    P.rho0 = density->rho0;
    P.x = points_dev;
    P.n = n;
    P.phi = phi_dev;
    P.gz = gz_dev;
    cudaStream_t st = (cudaStream_t)stream;
    switch (density->kind) {
    case MCG_RHO_NONE:
    case MCG_RHO_SPHERE:
    case MCG_RHO_PRISM: {
        for (int k = 0; k < 3; ++k) {
            P.c[k] = density->center[k];
            P.lo[k] = density->lo[k];
            P.hi[k] = density->hi[k];
        }
        P.a = density->radius;
        if (density->kind == MCG_RHO_SPHERE && !(density->radius > 0.0))
            return set_error(MCG_ERR_ARG, "sphere radius must be positive");
        const int64_t blocks = (n + 127) / 128;
        if (blocks > 2147483647LL) return set_error(MCG_ERR_ARG, "too many points");
        field_closed_kernel<<<(unsigned)blocks, 128, 0, st>>>(P);
        break;
    }
    case MCG_RHO_VOXEL: {
        if (!density->grid) return set_error(MCG_ERR_ARG, "voxel grid pointer is null");
        if (density->nx <= 0 || density->ny <= 0 || density->nz <= 0 || density->nx >= 65535 ||
            density->ny >= 65535 || density->nz >= 65535)
            return set_error(MCG_ERR_ARG, "voxel dims must be in [1, 65534]");
        if (n > 2147483647LL) return set_error(MCG_ERR_ARG, "too many points");
        P.grid = density->grid;
        P.nx = (int32_t)density->nx;
        P.ny = (int32_t)density->ny;
        P.nz = (int32_t)density->nz;
        for (int k = 0; k < 3; ++k) {
            if (!(density->spacing[k] > 0.0)) return set_error(MCG_ERR_ARG, "voxel spacing must be positive");
            P.org[k] = density->origin[k];
            P.sp[k] = density->spacing[k];
        }
        const double half[3] = {0.5 * P.sp[0], 0.5 * P.sp[1], 0.5 * P.sp[2]};
        cell_series(half, P.series);
        P.near = kNearCells * std::max(P.sp[0], std::max(P.sp[1], P.sp[2]));
        // few points: a cluster of eight blocks each, so that they fill the SMs.
        // (128 x 128 x 64 cells, eight blocks against one: 1 point 0.29 and 1.97
        // ms, 96 1.11 and 2.04, 256 2.58 and 2.54, 320 3.3 and 4.9, 1024 9.8 and
        // 9.8, 2048 19.5 and 17.2; a grid of 40 x 50 x 20, where the near zone
        // weighs more: 1 point 0.09 and 0.31, 96 0.38 and 0.32, 256 0.87 and 0.53)
        const unsigned parts = n < 2048 ? 8u : 1u;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)n * parts);
        cfg.blockDim = dim3(kFieldThreads);
        cfg.stream = st;
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = parts;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        const bool cube = P.series[0] == 0.0 && P.series[1] == 0.0 && P.series[2] == 0.0;
        // (its error, if any, is read and cleared below)
        if (cube) cudaLaunchKernelEx(&cfg, field_voxel_kernel<true>, P);
        else cudaLaunchKernelEx(&cfg, field_voxel_kernel<false>, P);
        break;
    }
    default:
        return set_error(MCG_ERR_ARG, "unknown density kind %d", density->kind);
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? MCG_OK : set_error(MCG_ERR_CUDA, "field kernel launch: %s", cudaGetErrorString(e));
}

extern "C" int mcg_density_at(const mcg_domain* domain, const mcg_density* density, double h, int32_t precision,
                              const double* points_dev, int64_t n, double* out_dev, void* stream)
{
    if (!domain || !density) return set_error(MCG_ERR_ARG, "null domain or density");
    if (precision != MCG_FP64 && precision != MCG_MIXED) return set_error(MCG_ERR_ARG, "bad precision");
    if (!(h >= 0.0) || !std::isfinite(h)) return set_error(MCG_ERR_ARG, "h must be finite and non-negative");
    if (n < 0) return set_error(MCG_ERR_ARG, "n must be non-negative");
    mcg_boundary zero;
    std::memset(&zero, 0, sizeof(zero));
    zero.kind = MCG_G_ZERO;
    mcg_options o;
    mcg_options_default(&o);
    o.h = h;
    o.crn_gz = 1;
    o.precision = precision;
    WalkParams P;
    const int rc = make_params(domain, density, &zero, 1.0, 0, &o, P);
    if (rc) return rc;
    if (n == 0) return MCG_OK;
    if (!points_dev || !out_dev) return set_error(MCG_ERR_ARG, "null device buffer");
    if (n > 2147483647LL * 128LL) return set_error(MCG_ERR_ARG, "too many points");
    preload_kernels();
    const unsigned blocks = (unsigned)((n + 127) / 128);
    cudaStream_t st = (cudaStream_t)stream;
    if (precision == MCG_FP64) {
        density_f64_kernel<<<blocks, 128, 0, st>>>(P, points_dev, n, out_dev);
    } else {
        const int kind = (P.rho_kind == MCG_RHO_VOXEL && P.zq) ? kRhoVoxelPacked : P.rho_kind;
        switch (kind) {
        case MCG_RHO_SPHERE: density_f32_kernel<MCG_RHO_SPHERE><<<blocks, 128, 0, st>>>(P, points_dev, n, out_dev); break;
        case MCG_RHO_PRISM: density_f32_kernel<MCG_RHO_PRISM><<<blocks, 128, 0, st>>>(P, points_dev, n, out_dev); break;
        case MCG_RHO_VOXEL: density_f32_kernel<MCG_RHO_VOXEL><<<blocks, 128, 0, st>>>(P, points_dev, n, out_dev); break;
        case kRhoVoxelPacked:
            density_f32_kernel<kRhoVoxelPacked><<<blocks, 128, 0, st>>>(P, points_dev, n, out_dev);
            break;
        default: density_f32_kernel<MCG_RHO_NONE><<<blocks, 128, 0, st>>>(P, points_dev, n, out_dev); break;
        }
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? MCG_OK : set_error(MCG_ERR_CUDA, "density kernel launch: %s", cudaGetErrorString(e));
}
