// mcg_setup.cu -- set-up of the heterogeneous model, run once per model
// outside the walk: the Gaussian-random-field density grid and the boundary
// tables of the Dirichlet data (the potential of the voxel model on the six
// faces of the box, by prism summation).
#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "mcg_cell.cuh"
#include "mcg_device.cuh"
#include "mcg_internal.h"

namespace mcg {

namespace {

constexpr int kMaxTaps = 63;

struct Taps {
    double w[kMaxTaps];
    int R;
};

// White noise: voxels 4q..4q+3 take the two Box-Muller pairs of Philox
// counter (q, 0, 0, 1).
__global__ void grf_noise_kernel(uint32_t k0, uint32_t k1, int64_t n, double* __restrict__ a)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (4 * q >= n) return;
    const uint4 w = philox4x32_10(make_uint4((uint32_t)q, 0u, 0u, 1u), k0, k1);
    double z[4];
    box_muller_f64(w.x, w.y, z[0], z[1]);
    box_muller_f64(w.z, w.w, z[2], z[3]);
    for (int j = 0; j < 4; ++j)
        if (4 * q + j < n) a[4 * q + j] = z[j];
}

// One separable pass of the Gaussian filter along an axis of length L and
// stride st, zero outside the grid, taps summed from -R to R.
__global__ void grf_smooth_kernel(const double* __restrict__ a, double* __restrict__ b, int64_t n, int64_t L,
                                  int64_t st, const Taps T)
{
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const int64_t coord = (v / st) % L;
    double acc = 0.0;
    for (int m = -T.R; m <= T.R; ++m) {
        const int64_t c2 = coord + m;
        if (c2 < 0 || c2 >= L) continue;
        acc = __dadd_rn(acc, __dmul_rn(T.w[m + T.R], a[v + m * st]));
    }
    b[v] = acc;
}

// Mean and population standard deviation of a, in two passes of
// `blocks` blocks: strided Neumaier partial sums per thread, a pairwise tree
// per block into part[block]; whoever needs the total adds the blocks'
// sums in order.  (One block alone took 4.5 ms for 128 x 128 x 64 voxels: an SM
// does 1.6 double-precision additions a clock.)
__device__ void neumaier_add(double& s, double& c, double x)
{
    const double t = s + x;
    if (fabs(s) >= fabs(x)) c += (s - t) + x;
    else c += (x - t) + s;
    s = t;
}

constexpr int kMomentThreads = 256;

__device__ double in_order(const double* part, int blocks)
{
    double s = 0.0, c = 0.0;
    for (int b = 0; b < blocks; ++b) neumaier_add(s, c, part[b]);
    return s + c;
}

// MEAN: sum of a.  Otherwise sum of (a - mean)^2, the mean from `means`.
template <bool MEAN>
__global__ void __launch_bounds__(kMomentThreads) grf_moments_kernel(const double* __restrict__ a, int64_t n,
                                                                     const double* __restrict__ means,
                                                                     double* __restrict__ part)
{
    __shared__ double sh[kMomentThreads];
    const int t = threadIdx.x;
    double mean = 0.0;
    if (!MEAN) {
        if (t == 0) sh[0] = in_order(means, gridDim.x) / (double)n;
        __syncthreads();
        mean = sh[0];
        __syncthreads();
    }
    double s = 0.0, c = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kMomentThreads + t; i < n; i += (int64_t)gridDim.x * kMomentThreads) {
        const double d = MEAN ? a[i] : (a[i] - mean) * (a[i] - mean);
        neumaier_add(s, c, d);
    }
    sh[t] = s + c;
    __syncthreads();
    for (int k = kMomentThreads / 2; k > 0; k >>= 1) {
        if (t < k) sh[t] += sh[t + k];
        __syncthreads();
    }
    if (t == 0) part[blockIdx.x] = sh[0];
}

__global__ void grf_transform_kernel(const double* __restrict__ a, int64_t n, const double* __restrict__ means,
                                     const double* __restrict__ squares, int blocks, double amp,
                                     float* __restrict__ grid)
{
    __shared__ double mom[2];
    if (threadIdx.x == 0) mom[0] = in_order(means, blocks) / (double)n;
    if (threadIdx.x == 32) mom[1] = sqrt(in_order(squares, blocks) / (double)n);
    __syncthreads();
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const double Z = (a[v] - mom[0]) / mom[1];
        grid[v] = (float)(amp * (exp(Z) - 1.0));
    }
}

// ---------------------------------------------------------------------------
// Boundary tables.
// ---------------------------------------------------------------------------
struct TableParams {
    double lo[3], hi[3];
    int32_t nu, nv;
    const float* grid;
    int32_t nx, ny, nz;
    double org[3], sp[3];
    double vol;              // cell volume
    double near2;            // squared radius of the exact (near) zone
    double unit;             // longest side of a cell
    double core_least;       // half-width of the core of a small near zone
    double second[3];        // cell_series for lengths in units of `unit`: its order 2 ...
    float series[kSeriesTerms];  // ... and all of it in single precision
    double G;
    float* out;
};

constexpr int kTableThreads = 256;
constexpr int kTableWarps = kTableThreads / 32;
constexpr int kRowsPerTile = 8;
// Cells of the near zone up to kCoreSides of the longest side from the node,
// along every axis, are summed by grid node (exact), the rest by the series of
// mcg_cell.cuh, whose remainder is 4e-12 of the cell's own term there: without
// P_10 (1e-8) one table value in a thousand rounded to its neighbour.  A smaller
// zone's core is the box inside it, down to core_least: three sides (1e-10), or
// 2.25 for cells of 1 : 0.6 and longer (at most 9e-10; with three, 128 x 24 x 64
// cells and a zone of four diagonals took 10.3 ms for 6 x 21^2 nodes instead of
// 4.9).  Below that the core stays as large and each of its cells is asked
// whether it is near.
constexpr double kCoreSides = 4.0, kCoreLeast = 3.0, kCoreLeastLong = 2.25, kLong = 0.6;
// Beyond 2048 sides P_4 .. P_10 add less than 1e-15 of the cell's term (0.015 y^4,
// below the pairs' 3e-14), and powers of coordinates counted in sides overflow
// from 1.6e4 sides on (inf times an underflown y^20 is no number).
constexpr float kSeriesEnds = 1.0f / 2048.0f;

__device__ __forceinline__ void node_position(const TableParams& T, int64_t node, double x[3])
{
    const int64_t per_face = (int64_t)T.nu * T.nv;
    const int f = (int)(node / per_face);
    const int64_t r = node % per_face;
    const int iu = (int)(r % T.nu), iv = (int)(r / T.nu);
    const int k = f >> 1;
    const int a = (k == 0) ? 1 : 0, b = (k == 2) ? 1 : 2;
    x[k] = (f & 1) ? T.hi[k] : T.lo[k];
    x[a] = T.lo[a] + (T.hi[a] - T.lo[a]) * (double)iu / (double)(T.nu - 1);
    x[b] = T.lo[b] + (T.hi[b] - T.lo[b]) * (double)iv / (double)(T.nv - 1);
}

// Offset of a cell's centre along an axis, and the squared distance (rounded
// alike wherever a cell is asked whether it is near).
__device__ __forceinline__ double cell_offset(const TableParams& T, int k, int i, double x)
{
    return __dadd_rn(__fma_rn((double)i + 0.5, T.sp[k], T.org[k]), -x);
}
__device__ __forceinline__ double square_sum(double a, double b2) { return __fma_rn(a, a, b2); }

// Point-mass far field for every voxel (single-precision terms, summed per
// row in single precision and per row into double), then, for voxels whose
// centre lies within the near radius, their own potential in place of the
// point mass.  Writes Phi = -G sum.
//
// A block takes 32 NPL nodes (NPL per lane); its warps, and with few nodes the
// blocks of its cluster, split the rows of the grid between them.  What
// bounds it: the reciprocal root of each voxel and node (16 a clock and SM,
// 22 ms for 6 x 128^2 nodes over 128 x 128 x 64 voxels).  Before, a thread
// summed a node alone (486 nodes: 179 ms, on two SMs) and the near zone was
// exact prisms in double precision throughout (6 x 128^2 nodes: 342 of 377 ms,
// ~690 prisms a node of 8 corners; the pipe does 1.6 operations a clock and
// SM).  Now 0.5 and 37 ms, 25 of them the point masses, with the same values
// to the last bit (twelve grids and zones).
template <int NPL>
__global__ void __launch_bounds__(kTableThreads, 2) tables_kernel(const TableParams T)
{
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int parts = (int)cluster.num_blocks(), part = (int)cluster.block_rank();
    __shared__ float4 rho_s[kTableWarps][kRowsPerTile][32];
    __shared__ float4 cx_s[32];                     // voxel-centre x offsets, (float)ix * sx
    __shared__ double sum_s[kTableWarps][32 * NPL];
    __shared__ double total_s[32 * NPL];
    const int64_t nodes = 6ll * T.nu * T.nv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t first = (int64_t)(blockIdx.x / parts) * (32 * NPL);
    const float sx = (float)T.sp[0], sy = (float)T.sp[1], sz = (float)T.sp[2];
    // (a column past the grid has no density: far away, so that its term is 0)
    for (int i = threadIdx.x; i < 128; i += kTableThreads) ((float*)cx_s)[i] = i < T.nx ? (float)i * sx : 1e18f;
    __syncthreads();
    float px[NPL], py[NPL], pz[NPL];
    double acc[NPL];
#pragma unroll
    for (int j = 0; j < NPL; ++j) {
        const int64_t node = first + 32 * j + lane;
        double x[3];
        node_position(T, node < nodes ? node : nodes - 1, x);
        // node relative to the first voxel centre, single precision
        px[j] = (float)(x[0] - (T.org[0] + 0.5 * T.sp[0]));
        py[j] = (float)(x[1] - (T.org[1] + 0.5 * T.sp[1]));
        pz[j] = (float)(x[2] - (T.org[2] + 0.5 * T.sp[2]));
        acc[j] = 0.0;
    }
    const int rows = T.ny * T.nz, quads = (T.nx + 3) / 4;
    const int stride = kTableWarps * parts * kRowsPerTile;
    for (int r0 = (part * kTableWarps + warp) * kRowsPerTile; r0 < rows; r0 += stride) {
        __syncwarp();
        for (int rr = 0; rr < kRowsPerTile; ++rr)
            for (int ix = lane; ix < 4 * quads; ix += 32)
                ((float*)rho_s[warp][rr])[ix] =
                    (r0 + rr < rows && ix < T.nx) ? __ldg(T.grid + (int64_t)(r0 + rr) * T.nx + ix) : 0.0f;
        __syncwarp();
        for (int rr = 0; rr < kRowsPerTile && r0 + rr < rows; ++rr) {
            const int row = r0 + rr;
            float dyz2[NPL], sum[NPL];
#pragma unroll
            for (int j = 0; j < NPL; ++j) {
                const float dy = (float)(row % T.ny) * sy - py[j];
                const float dz = (float)(row / T.ny) * sz - pz[j];
                dyz2[j] = fmaf(dy, dy, dz * dz);
                sum[j] = 0.0f;
            }
#pragma unroll 2
            for (int q = 0; q < quads; ++q) {
                const float4 r4 = rho_s[warp][rr][q], c4 = cx_s[q];
                const float rv[4] = {r4.x, r4.y, r4.z, r4.w}, cv[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int j = 0; j < NPL; ++j) {
                        const float dx = cv[e] - px[j];
                        float y;
                        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(fmaf(dx, dx, dyz2[j])));
                        sum[j] = fmaf(rv[e], y, sum[j]);
                    }
            }
#pragma unroll
            for (int j = 0; j < NPL; ++j) acc[j] += (double)sum[j];
        }
    }
    // near zone: the voxel's own potential minus the point mass already
    // counted; the rows of the zone's box go round the warps
    const double R = sqrt(T.near2), inv = 1.0 / T.unit, inv2 = inv * inv;
    const int n[3] = {T.nx, T.ny, T.nz};
#pragma unroll
    for (int j = 0; j < NPL; ++j) {
        const int64_t node = first + 32 * j + lane;
        double x[3];
        node_position(T, node < nodes ? node : nodes - 1, x);
        acc[j] *= T.vol;
        int ilo[3], ihi[3];
        for (int k = 0; k < 3; ++k) {
            const double a = fmin(fmax(floor((x[k] - R - T.org[k]) / T.sp[k]), 0.0), (double)n[k]);
            const double b = fmin(fmax(floor((x[k] + R - T.org[k]) / T.sp[k]), -1.0), (double)(n[k] - 1));
            ilo[k] = (int)a;
            ihi[k] = (int)b;
        }
        if (ilo[0] > ihi[0] || ilo[1] > ihi[1] || ilo[2] > ihi[2]) continue;
        // the core: a box of cells inside the near zone (its half-width is below
        // R / sqrt 3), or of cells to be asked
        const bool whole = R * 0.57 >= T.core_least;
        const double core = whole ? fmin(kCoreSides * T.unit, R * 0.57) : fmin(T.core_least, R);
        int clo[3], chi[3];
        for (int k = 0; k < 3; ++k) {
            const double a = (x[k] - T.org[k]) / T.sp[k], w = core / T.sp[k];
            clo[k] = (int)fmin(fmax(ceil(a - w - 0.5), 0.0), (double)n[k]);
            chi[k] = (int)fmin(fmax(floor(a + w - 0.5) + 1.0, 0.0), (double)n[k]);
        }
        const int wy = ihi[1] - ilo[1] + 1, box_rows = wy * (ihi[2] - ilo[2] + 1);
        for (int q = part * kTableWarps + warp; q < box_rows; q += kTableWarps * parts) {
            const int iy = ilo[1] + q % wy, iz = ilo[2] + q / wy;
            const double cy = cell_offset(T, 1, iy, x[1]), cz = cell_offset(T, 2, iz, x[2]);
            const double cyz = square_sum(cy, __dmul_rn(cz, cz));
            if (cyz >= T.near2) continue;
            const bool core_row = iy >= clo[1] && iy < chi[1] && iz >= clo[2] && iz < chi[2];
            const double Y = cy * cy * inv2, Z = cz * cz * inv2;
            const SeriesRow sr = series_row(T.series, (float)Y, (float)Z);
            const Pair p2x = pair_of(T.second[0]), c2 = pair_of(T.second[1] * Y + T.second[2] * Z);
            const float dy = (float)iy * sy - py[j], dz = (float)iz * sz - pz[j];
            for (int ix = ilo[0]; ix <= ihi[0]; ++ix) {
                const double cx = cell_offset(T, 0, ix, x[0]);
                const double d2 = square_sum(cx, cyz);
                if (d2 >= T.near2) continue;
                const float rho = __ldg(T.grid + ((int64_t)iz * T.ny + iy) * T.nx + ix);
                if (rho == 0.0f) continue;
                const float dx = ((const float*)cx_s)[ix] - px[j];
                float pm;
                asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(pm) : "f"(fmaf(dx, dx, fmaf(dy, dy, dz * dz))));
                if (core_row && ix >= clo[0] && ix < chi[0]) {
                    acc[j] -= T.vol * (double)(rho * pm);  // its own potential: the core's node sum
                } else {
                    const Pair X = pair_of(cx * cx * inv2);
                    Pair y2, P2, y5;
                    const Pair y = rsqrt_pair(pair_of(d2 * inv2), y2);
                    const Pair v = series_second(p2x, c2, X, y, y2, P2, y5);
                    float higher = 0.0f;
                    if (y.h > kSeriesEnds) {
                        float P4, P6, P8;
                        series_polys(T.series, sr, X.h, P4, P6, P8);
                        higher = series_value(P4, P6, P8, y.h, y2.h) + series_tenth(T.series, sr, X.h, y.h, y2.h);
                    }
                    const Pair f = add_small({y.h, y.l + higher}, v);
                    acc[j] += T.vol * ((double)rho * (((double)f.h + (double)f.l) * inv) - (double)(rho * pm));
                }
            }
        }
        // the core's nodes, each with the weight of the core cells it belongs
        // to (upper corner, sign +, of the cell before it along an axis,
        // lower corner, sign -, of its own)
        const int mx = chi[0] - clo[0] + 1, my = chi[1] - clo[1] + 1, mz = chi[2] - clo[2] + 1;
        if (mx <= 1 || my <= 1 || mz <= 1) continue;
        for (int q = part * kTableWarps + warp; q < mx * my * mz; q += kTableWarps * parts) {
            const int a = clo[0] + q % mx, b = clo[1] + q / mx % my, c = clo[2] + q / (mx * my);
            double w = 0.0;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int ci = a - 1 + (m & 1), cj = b - 1 + ((m >> 1) & 1), ck = c - 1 + (m >> 2);
                double v = 0.0;
                bool in = ci >= clo[0] && ci < chi[0] && cj >= clo[1] && cj < chi[1] && ck >= clo[2] && ck < chi[2];
                if (!whole) {
                    const double cz = cell_offset(T, 2, ck, x[2]);
                    const double cyz = square_sum(cell_offset(T, 1, cj, x[1]), __dmul_rn(cz, cz));
                    in = in && square_sum(cell_offset(T, 0, ci, x[0]), cyz) < T.near2;
                }
                if (in) v = (double)__ldg(T.grid + ((int64_t)ck * T.ny + cj) * T.nx + ci);
                w += ((m ^ (m >> 1) ^ (m >> 2)) & 1) ? -v : v;
            }
            if (w != 0.0)
                acc[j] += w * prism_corner(T.org[0] + a * T.sp[0] - x[0], T.org[1] + b * T.sp[1] - x[1],
                                           T.org[2] + c * T.sp[2] - x[2]);
        }
    }
    // the warps' sums, then the cluster's, in order
#pragma unroll
    for (int j = 0; j < NPL; ++j) sum_s[warp][32 * j + lane] = acc[j];
    __syncthreads();
    const int t = threadIdx.x;
    if (t < 32 * NPL) {
        double v = 0.0;
        for (int w = 0; w < kTableWarps; ++w) v += sum_s[w][t];
        total_s[t] = v;
    }
    cluster.sync();
    if (part == 0 && t < 32 * NPL && first + t < nodes) {
        double v = 0.0;
        for (int b = 0; b < parts; ++b) v += *cluster.map_shared_rank(&total_s[t], b);
        T.out[first + t] = (float)(-T.G * v);
    }
    cluster.sync();  // the other blocks' shared memory stays until it has been read
}

// Packed voxel grid: entry (iz + 1, iy, ix) = layers iz-1, iz, iz+1 of
// column (ix, iy), 0 outside the grid, for iz = -1 .. nz.
__global__ void voxel_pack_kernel(const float* __restrict__ g, int nx, int ny, int nz, float4* __restrict__ out)
{
    const int64_t n = (int64_t)nx * ny * (nz + 2);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int ix = (int)(e % nx), iy = (int)((e / nx) % ny), iz = (int)(e / ((int64_t)nx * ny)) - 1;
    const int64_t col = (int64_t)iy * nx + ix, plane = (int64_t)nx * ny;
    float v[3];
    for (int d = 0; d < 3; ++d) {
        const int k = iz - 1 + d;
        v[d] = (k >= 0 && k < nz) ? g[col + plane * k] : 0.0f;
    }
    out[e] = make_float4(v[0], v[1], v[2], 0.0f);
}

// Packed tables: entry (f, iv, iu) = the corners (iu, iv), (iu+1, iv),
// (iu, iv+1), (iu+1, iv+1) of cell (iu, iv) of face f.
__global__ void table_pack_kernel(const float* __restrict__ t, int nu, int nv, float4* __restrict__ out)
{
    const int64_t cells = (int64_t)(nu - 1) * (nv - 1);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 6 * cells) return;
    const int f = (int)(e / cells);
    const int64_t r = e % cells;
    const int iu = (int)(r % (nu - 1)), iv = (int)(r / (nu - 1));
    const float* row = t + (int64_t)f * nu * nv + (int64_t)iv * nu + iu;
    out[e] = make_float4(row[0], row[1], row[nu], row[nu + 1]);
}

}  // namespace

int voxel_pack(const mcg_density* rho, float* out, cudaStream_t st)
{
    if (!rho || !out) return set_error(MCG_ERR_ARG, "null argument");
    if (rho->kind != MCG_RHO_VOXEL || !rho->grid) return set_error(MCG_ERR_ARG, "voxel_pack needs a voxel density");
    if (rho->nx <= 0 || rho->ny <= 0 || rho->nz <= 0) return set_error(MCG_ERR_ARG, "voxel dims must be positive");
    if ((double)rho->nx * (double)rho->ny * (double)(rho->nz + 2) >= 2147483647.0)
        return set_error(MCG_ERR_ARG, "voxel grid too large to pack");
    if ((uintptr_t)out % 16 != 0) return set_error(MCG_ERR_ARG, "packed grid must be 16-byte aligned");
    const int64_t n = rho->nx * rho->ny * (rho->nz + 2);
    voxel_pack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(rho->grid, (int)rho->nx, (int)rho->ny,
                                                                      (int)rho->nz, (float4*)out);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? MCG_OK : set_error(MCG_ERR_CUDA, "voxel pack kernel: %s", cudaGetErrorString(e));
}

int table_pack(const mcg_boundary* b, float* out, cudaStream_t st)
{
    if (!b || !out) return set_error(MCG_ERR_ARG, "null argument");
    if (b->kind != MCG_G_TABLE || !b->faces || b->nu < 2 || b->nv < 2)
        return set_error(MCG_ERR_ARG, "table_pack needs tables with nu, nv >= 2");
    if ((uintptr_t)out % 16 != 0) return set_error(MCG_ERR_ARG, "packed tables must be 16-byte aligned");
    const int64_t n = 6ll * (b->nu - 1) * (b->nv - 1);
    if (n >= 2147483647LL) return set_error(MCG_ERR_ARG, "tables too large to pack");
    table_pack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(b->faces, b->nu, b->nv, (float4*)out);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? MCG_OK : set_error(MCG_ERR_CUDA, "table pack kernel: %s", cudaGetErrorString(e));
}

int grf_density(uint64_t seed, int64_t nx, int64_t ny, int64_t nz, double sigma_vox, double amp, float* grid_out,
                double* work, cudaStream_t st)
{
    if (nx <= 0 || ny <= 0 || nz <= 0) return set_error(MCG_ERR_ARG, "grid dims must be positive");
    if (!(sigma_vox > 0.0) || !std::isfinite(sigma_vox)) return set_error(MCG_ERR_ARG, "sigma_vox must be positive");
    const int R = (int)std::ceil(3.0 * sigma_vox);
    if (2 * R + 1 > kMaxTaps) return set_error(MCG_ERR_ARG, "sigma_vox too large (at most %d taps)", kMaxTaps);
    if (!grid_out || !work) return set_error(MCG_ERR_ARG, "null device buffer");
    const int64_t n = nx * ny * nz;
    Taps T;
    T.R = R;
    double wsum = 0.0;
    for (int m = -R; m <= R; ++m) {
        T.w[m + R] = std::exp(-(double)m * (double)m / (2.0 * sigma_vox * sigma_vox));
        wsum += T.w[m + R];
    }
    for (int m = 0; m <= 2 * R; ++m) T.w[m] /= wsum;
    double* a = work;
    double* b = work + n;
    double* mom = work + 2 * n;
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const int64_t q = (n + 3) / 4;
    grf_noise_kernel<<<(unsigned)((q + 255) / 256), 256, 0, st>>>(k0, k1, n, a);
    const int64_t dims[3] = {nx, ny, nz}, strides[3] = {1, nx, nx * ny};
    for (int axis = 0; axis < 3; ++axis) {
        grf_smooth_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, b, n, dims[axis], strides[axis], T);
        double* t = a;
        a = b;
        b = t;
    }
    // the blocks' sums go behind the filter's spare buffer's start, or, for a
    // grid too small to lend one, into the 32 doubles behind both
    const int blocks = (int)std::min<int64_t>(64, (n + 4095) / 4096);
    double* part = blocks > 8 ? b : mom;
    grf_moments_kernel<true><<<blocks, kMomentThreads, 0, st>>>(a, n, nullptr, part);
    grf_moments_kernel<false><<<blocks, kMomentThreads, 0, st>>>(a, n, part, part + blocks);
    const int64_t tb = std::min<int64_t>((n + 255) / 256, 1024);
    grf_transform_kernel<<<(unsigned)tb, 256, 0, st>>>(a, n, part, part + blocks, blocks, amp, grid_out);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? MCG_OK : set_error(MCG_ERR_CUDA, "grf kernels: %s", cudaGetErrorString(e));
}

int boundary_tables(const mcg_domain* d, const mcg_density* rho, int32_t nu, int32_t nv, double near_cells,
                    float* faces_out, cudaStream_t st)
{
    if (!d || !rho || !faces_out) return set_error(MCG_ERR_ARG, "null argument");
    if (rho->kind != MCG_RHO_VOXEL || !rho->grid) return set_error(MCG_ERR_ARG, "tables need a voxel density");
    if (nu < 2 || nv < 2) return set_error(MCG_ERR_ARG, "tables need nu, nv >= 2");
    if (rho->nx <= 0 || rho->nx > 128 || rho->ny <= 0 || rho->nz <= 0)
        return set_error(MCG_ERR_ARG, "table generation supports 1 <= nx <= 128 cells along x");
    if (!(near_cells >= 0.0)) return set_error(MCG_ERR_ARG, "near_cells must be >= 0");
    TableParams T;
    for (int k = 0; k < 3; ++k) {
        if (!(d->lo[k] < d->hi[k])) return set_error(MCG_ERR_ARG, "domain lo >= hi");
        if (!(rho->spacing[k] > 0.0)) return set_error(MCG_ERR_ARG, "voxel spacing must be positive");
        T.lo[k] = d->lo[k];
        T.hi[k] = d->hi[k];
        T.org[k] = rho->origin[k];
        T.sp[k] = rho->spacing[k];
    }
    T.nu = nu;
    T.nv = nv;
    T.grid = rho->grid;
    T.nx = (int32_t)rho->nx;
    T.ny = (int32_t)rho->ny;
    T.nz = (int32_t)rho->nz;
    T.vol = T.sp[0] * T.sp[1] * T.sp[2];
    const double diag = std::sqrt(T.sp[0] * T.sp[0] + T.sp[1] * T.sp[1] + T.sp[2] * T.sp[2]);
    T.near2 = (near_cells * diag) * (near_cells * diag);
    T.G = rho->G;
    T.out = faces_out;
    const int64_t nodes = 6ll * nu * nv;
    T.unit = std::max(T.sp[0], std::max(T.sp[1], T.sp[2]));
    const double second = T.sp[0] + T.sp[1] + T.sp[2] - T.unit - std::min(T.sp[0], std::min(T.sp[1], T.sp[2]));
    T.core_least = (second > kLong * T.unit ? kCoreLeast : kCoreLeastLong) * T.unit;
    const double half[3] = {0.5 * T.sp[0] / T.unit, 0.5 * T.sp[1] / T.unit, 0.5 * T.sp[2] / T.unit};
    double series[kSeriesTerms];
    cell_series(half, series);
    for (int i = 0; i < 3; ++i) T.second[i] = series[i];
    for (int i = 0; i < kSeriesTerms; ++i) T.series[i] = (float)series[i];
    // two nodes a lane share each density read; with few nodes one, and a
    // cluster of eight blocks for each 32 of them, so that they fill the SMs.
    // (128 x 128 x 64 cells; one node a lane in 1 and 8 blocks, two in 1 and 8:
    // 486 nodes 3.4, 0.53, 6.0, 0.85 ms; 14406 8.9, 7.0, 9.7, 6.7; 25350 11.2,
    // 11.3, 12.2, 10.6; 39366 16.8, 17.8, 17.7, 16.8; 60000 24.8, 26.9, 24.4, 25.6;
    // 98304 38.1, 43.0, 37.3, 40.2)
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool many = nodes >= 64ll * 4 * sms;
    const int64_t per = many ? 64 : 32, groups = (nodes + per - 1) / per;
    const unsigned parts = groups >= 4ll * sms ? 1u : 8u;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)groups * parts);
    cfg.blockDim = dim3(kTableThreads);
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = parts;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (many) cudaLaunchKernelEx(&cfg, tables_kernel<2>, T);
    else cudaLaunchKernelEx(&cfg, tables_kernel<1>, T);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? MCG_OK : set_error(MCG_ERR_CUDA, "tables kernel: %s", cudaGetErrorString(e));
}

}  // namespace mcg
