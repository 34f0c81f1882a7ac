// mcg_walk64.cu -- the double-precision walk (Sec. 2.3 of the paper, steps 1-4).
//
// Increments, positions and exits are doubles, rounded operation by operation
// (no contraction), so a path agrees with a plain double-precision evaluation
// to the last bits of log, sqrt, cos and sin; the source integral is a sum over
// the walk's points (exact counts where the density is rho0 or 0, else lane by
// lane), closed at the exit.  GB300 does 1.6 double-precision operations a clock
// and SM, and a step evaluated in doubles throughout took 166, 6.6 us for a
// lane.  What is left of them: the products that make an increment (3 a normal)
// and the additions that move the walk.  The functions are evaluated in 64-bit
// integers (mcg_fixed.cuh), and the tests of a point (inside Omega, in the
// density's support, in which cell) in single precision, with doubles where that
// is too close to call.
//
// A warp holds G <= 8 walks and k = 32 / G lanes share each: a lane makes the
// increments of one four-step block, a lane per walk and coordinate adds them
// up in order through shared memory, then each lane tests its own block.
//
// What bounds it: with the GPU full the double-precision pipe (busy 71 % of
// the time: 64 operations of a block's 3100 instructions a lane) and the
// integer pipes beside it (issue 58 %): 27.3 steps/ns against 3.2 for the plain
// evaluation (ore body, capped walks).  With few walks the chain of additions
// and a block's dependent integers: 88 ns a step for a lone walk over the ore
// body, most of its blocks far from it (6270 before).  Walks of the sphere, 8 x 2000 paths: 17.7 -> 0.91 ms; ore body at
// 10 m steps, 30 x 256 paths: 106.7 -> 2.06 ms.
#include <cmath>

#include <cuda_runtime.h>

#include "mcg_device.cuh"
#include "mcg_fixed.cuh"
#include "mcg_internal.h"
#include "mcg_walk.cuh"

namespace mcg {

namespace {

constexpr int kSlots = 16;          // walks a warp holds: live, and ended ones waiting for their evaluation
constexpr unsigned kLiveMax = 8;    // live ones at most (with 4, a full launch 22.4 steps/ns instead of 27.3,
                                    // 8 x 2000 paths of the sphere 0.81 ms instead of 0.91)
constexpr int kBatch = 10;          // walks evaluated at once: 30 copies on 32 lanes (5 and 8: no difference
                                    // beyond the runs' own)
constexpr int kMoveRow = 33;        // double2 per row of the moves

// How near to a face, or (squared) to a sphere, single precision does not
// decide: a point is known to about 4e-7 of the domain's largest half-width.
struct Near {
    float sd;           // step scale
    float face, sphere, ball;
    float cell[3];      // voxel faces, in cells
};

// The plain tests, in doubles.
__device__ __noinline__ bool inside_exact(const WalkParams& P, double x, double y, double z)
{
    if (P.ball) {
        const double dx = __dadd_rn(x, -P.cen[0]), dy = __dadd_rn(y, -P.cen[1]), dz = __dadd_rn(z, -P.cen[2]);
        return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)) < P.R2;
    }
    return x > P.lo[0] && x < P.hi[0] && y > P.lo[1] && y < P.hi[1] && z > P.lo[2] && z < P.hi[2];
}
// Support of a density that is rho0 or 0 (the tests of rho_f64).
__device__ __noinline__ bool support_exact(const WalkParams& P, double x, double y, double z)
{
    if (P.rho_kind == MCG_RHO_PRISM)
        return x >= P.plo[0] && x < P.phi[0] && y >= P.plo[1] && y < P.phi[1] && z >= P.plo[2] && z < P.phi[2];
    const double dx = __dadd_rn(x, -P.sc[0]), dy = __dadd_rn(y, -P.sc[1]), dz = __dadd_rn(z, -P.sc[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)) < P.srad2;
}
__device__ __noinline__ double rho_exact(const WalkParams& P, const ModelRef& M, double x, double y, double z)
{
    const double X[3] = {x, y, z};
    return rho_f64(P, M, X);
}
__device__ __forceinline__ double copy_z(const WalkParams& P, int c, double z)
{
    return __dadd_rn(z, c == 0 ? 0.0 : (c == 1 ? P.h : -P.h));
}

// Copies of a point strictly inside Omega: f its position in single precision
// relative to the domain's centre, W(k) its coordinates in doubles.
template <bool CRN, typename Point>
__device__ __forceinline__ unsigned inside64(const WalkParams& P, const Near& T, const float f[3], Point W)
{
    unsigned in = 0u, close = 0u;
    const float q = P.ball ? fmaf(f[0], f[0], f[1] * f[1]) - P.R2_f : fmaxf(fabsf(f[0]) - P.half_f[0], fabsf(f[1]) - P.half_f[1]);
    const float near = P.ball ? T.ball : T.face;
#pragma unroll
    for (int c = 0; c < (CRN ? 3 : 1); ++c) {
        const float z = c == 0 ? f[2] : (c == 1 ? f[2] + P.h_f : f[2] - P.h_f);
        const float d = P.ball ? fmaf(z, z, q) : fmaxf(q, fabsf(z) - P.half_f[2]);
        if (d < 0.0f) in |= 1u << c;
        if (fabsf(d) <= near) close |= 1u << c;
    }
    while (close) {
        const int c = __ffs(close) - 1;
        close &= close - 1u;
        in = (in & ~(1u << c)) | (inside_exact(P, W(0), W(1), copy_z(P, c, W(2))) ? 1u << c : 0u);
    }
    return in;
}

// Copies in the support of a density that is rho0 or 0.
template <int RHO, bool CRN, typename Point>
__device__ __forceinline__ unsigned support64(const WalkParams& P, const Near& T, const float f[3], Point W)
{
    unsigned in = 0u, close = 0u;
    const float x = f[0] - P.sc_f[0], y = f[1] - P.sc_f[1];
    const float q = RHO == MCG_RHO_SPHERE
                        ? fmaf(x, x, y * y) - P.srad2_f
                        : fmaxf(fmaxf(P.plo_f[0] - f[0], f[0] - P.phi_f[0]), fmaxf(P.plo_f[1] - f[1], f[1] - P.phi_f[1]));
#pragma unroll
    for (int c = 0; c < (CRN ? 3 : 1); ++c) {
        const float z = c == 0 ? f[2] : (c == 1 ? f[2] + P.h_f : f[2] - P.h_f), zs = z - P.sc_f[2];
        const float d = RHO == MCG_RHO_SPHERE ? fmaf(zs, zs, q) : fmaxf(q, fmaxf(P.plo_f[2] - z, z - P.phi_f[2]));
        if (d < 0.0f) in |= 1u << c;
        if (fabsf(d) <= (RHO == MCG_RHO_SPHERE ? T.sphere : T.face)) close |= 1u << c;
    }
    while (close) {
        const int c = __ffs(close) - 1;
        close &= close - 1u;
        in = (in & ~(1u << c)) | (support_exact(P, W(0), W(1), copy_z(P, c, W(2))) ? 1u << c : 0u);
    }
    return in;
}

// Voxel densities of the copies.
template <bool CRN, typename Point>
__device__ __forceinline__ void voxel64(const WalkParams& P, const Near& T, const ModelRef& M, const float f[3],
                                        Point W, double rho[3])
{
    const float tx = (f[0] - P.org_f[0]) * P.inv_sp_f[0], ty = (f[1] - P.org_f[1]) * P.inv_sp_f[1],
                tz = (f[2] - P.org_f[2]) * P.inv_sp_f[2];
    const bool in = tx >= 0.f && tx < (float)P.nx && ty >= 0.f && ty < (float)P.ny;
    const bool xy_close = fabsf(tx - rintf(tx)) <= T.cell[0] || fabsf(ty - rintf(ty)) <= T.cell[1];
    const unsigned col = in ? (unsigned)(int)tx + (unsigned)P.nx * (unsigned)(int)ty : 0u;
    unsigned close = 0u;
#pragma unroll
    for (int c = 0; c < (CRN ? 3 : 1); ++c) {
        const float z = c == 0 ? tz : (c == 1 ? tz + P.hz_f : tz - P.hz_f);
        rho[c] = 0.0;
        if (xy_close || fabsf(z - rintf(z)) <= T.cell[2]) close |= 1u << c;
        else if (in && z >= 0.f && z < (float)P.nz)
            rho[c] = (double)__ldg(M.grid + (col + (unsigned)(P.nx * P.ny) * (unsigned)(int)z));
    }
    while (close) {
        const int c = __ffs(close) - 1;
        close &= close - 1u;
        const double v = rho_exact(P, M, W(0), W(1), copy_z(P, c, W(2)));
        if (c == 0) rho[0] = v;
        if (c == 1) rho[1] = v;
        if (c == 2) rho[2] = v;
    }
}

// ---------------------------------------------------------------------------
// Brownian-bridge exit test of an inside step X -> Y (the paper's Remark on
// exit-time estimation, after Gobet): the bridge crosses the plane of a face
// at distances d_X, d_Y with probability exp(-2 d_X d_Y / sd^2); with the
// faces taken as independent the step exits with probability
// 1 - prod (1 - p_face).  One uniform per RNG-step n: Philox counter
// (n / 4, p, s, 2), word n % 4, shared by the copies.  Returns the face with
// the largest p (2k lower, 2k+1 upper) if the step exits, else -1.
// ---------------------------------------------------------------------------
__device__ __noinline__ int bridge_face_f64(const WalkParams& P, const double* X, const double* Y, uint32_t s,
                                            uint32_t p, uint32_t n)
{
    double q = 1.0, pmax = -1.0;
    int kmax = -1;
    for (int f = 0; f < 6; ++f) {
        const int k = f >> 1;
        const double dX = (f & 1) ? __dadd_rn(P.hi[k], -X[k]) : __dadd_rn(X[k], -P.lo[k]);
        const double dY = (f & 1) ? __dadd_rn(P.hi[k], -Y[k]) : __dadd_rn(Y[k], -P.lo[k]);
        const double pk = exp(__ddiv_rn(__dmul_rn(__dmul_rn(-2.0, dX), dY), __dmul_rn(P.sd, P.sd)));
        q = __dmul_rn(q, __dadd_rn(1.0, -pk));
        if (pk > pmax) {
            pmax = pk;
            kmax = f;
        }
    }
    const uint4 w = philox4x32_10(make_uint4(n >> 2, p, s, 2u), P.key0, P.key1);
    const uint32_t word = (n & 3u) == 0u ? w.x : (n & 3u) == 1u ? w.y : (n & 3u) == 2u ? w.z : w.w;
    return (u01_f64(word) < 1.0 - q) ? kmax : -1;
}

__device__ __forceinline__ void write_path(const WalkParams& P, int32_t* status, unsigned long long item, double u0,
                                           double up, double um, int64_t steps)
{
    const double d = P.crn ? (up - um) / (2.0 * P.h) : kNaN;
    P.pp_u[item] = u0;
    P.pp_d[item] = d;
    P.pp_steps[item] = steps;
    const bool bad = !isfinite(u0) || (P.crn && !isfinite(d));
    if (bad) atomicOr(status, 1 << MCG_ERR_NONFINITE);
}

// A walk of the warp and the exits of its copies (a copy's last point inside
// Omega, its increment and first point outside, its source sum, and the face
// of a bridge exit or -1); the evaluation leaves the exit point in `X` and u
// in `sum`.
struct Exit {
    double X[3], dW[3], Y[3];
    double sum;
    int32_t face, pad;
};
struct Walk {
    double w[3];
    unsigned long long acc[3];  // half points of the support, or a double's bits
    unsigned long long item, steps;
    uint32_t s, p, blk, alive, k0, k1;
    int32_t seg;
    uint32_t pad;
    Exit exit[3];
};

// Increment of step m of the block whose first counter is c: the same numbers
// as the block's, for a copy's exit.
__device__ __noinline__ void step_of(const fx::Tables& tables, double sd, uint4 c, uint32_t k0, uint32_t k1, int m,
                                     double dW[3])
{
    for (int q = 0; q < 3; ++q) {
        const int j = 3 * m + q;  // normal of the block
        uint4 ctr = c;
        ctr.x += (uint32_t)(j >> 2);
        const uint4 v = philox4x32_10(ctr, k0, k1);
        double rd;
        float rf;
        int64_t co, si;
        double cs, sn;
        fx::polar64(tables, (j & 2) ? v.z : v.x, (j & 2) ? v.w : v.y, rd, rf, co, si, cs, sn);
        dW[q] = __dmul_rn(sd, __dmul_rn(rd, (j & 1) ? sn : cs));
    }
}

// u and d of the ended walks in `mask`, 10 at a time: a lane per copy clips
// the exit step, closes the trapezoid and (but for the prism's closed form)
// reads g; the closed form takes a lane per corner, four copies at a time.
template <int RHO, bool CRN, bool SEG>
__device__ __noinline__ void evaluate(const WalkParams& P, Walk* walks, unsigned mask)
{
    constexpr int NC = CRN ? 3 : 1;
    const int lane = threadIdx.x & 31;
    while (mask) {
        const int n = __popc(mask) < kBatch ? __popc(mask) : kBatch;
        const int j = lane / NC, c = lane % NC;
        Walk* w = nullptr;
        int32_t* status = P.status;
        if (j < n) {
            w = walks + __fns(mask, 0, j + 1);
            ModelRef M = model_of(P);
            if constexpr (SEG) {
                M = model_of(P.seg[w->seg]);
                status = P.seg[w->seg].status;
            }
            Exit& e = w->exit[c];
            const double *X = e.X, *dW = e.dW, *Y = e.Y;
            double xs[3] = {Y[0], Y[1], Y[2]};
            double theta = 1.0;
            int face = e.face;
            if (face >= 0) {  // the bridge left Omega: on this face below Y after a full step
                xs[face >> 1] = (face & 1) ? P.hi[face >> 1] : P.lo[face >> 1];
            } else if (P.clip && P.ball) {
                const double q[3] = {__dadd_rn(X[0], -P.cen[0]), __dadd_rn(X[1], -P.cen[1]),
                                     __dadd_rn(X[2], -P.cen[2])};
                theta = ball_theta(q, dW, P.R2);
                for (int k = 0; k < 3; ++k) xs[k] = __dadd_rn(X[k], __dmul_rn(theta, dW[k]));
            } else if (P.clip) {
                int at = -1;
                double tmin = __longlong_as_double(0x7ff0000000000000LL), wall = 0.0;
                for (int k = 0; k < 3; ++k) {
                    double b;
                    if (Y[k] <= P.lo[k]) b = P.lo[k];
                    else if (Y[k] >= P.hi[k]) b = P.hi[k];
                    else continue;
                    const double t = __ddiv_rn(__dadd_rn(b, -X[k]), dW[k]);
                    if (t < tmin) {
                        tmin = t;
                        at = k;
                        wall = b;
                    }
                }
                theta = at < 0 ? kNaN : fmin(fmax(tmin, 0.0), 1.0);
                for (int k = 0; k < 3; ++k) xs[k] = __dadd_rn(X[k], __dmul_rn(theta, dW[k]));
                if (at >= 0) {
                    xs[at] = wall;
                    face = 2 * at + (wall == P.hi[at] ? 1 : 0);
                }
            }
            // the trapezoid: `sum` holds rho_0 / 2 and every inside point after it
            double I = 0.0;
            if constexpr (RHO != MCG_RHO_NONE) {
                const double rp = rho_f64(P, M, X), r = rho_f64(P, M, xs);
                I = __dadd_rn(__dmul_rn(P.dt, __dadd_rn(e.sum, -0.5 * rp)),
                              __dmul_rn(__dmul_rn(__dmul_rn(0.5, __dadd_rn(rp, r)), theta), P.dt));
            }
            const double g = P.g_kind == MCG_G_PRISM ? 0.0 : boundary_value(P, M, face, xs);
            for (int k = 0; k < 3; ++k) e.X[k] = xs[k];
            e.sum = P.g_kind == MCG_G_PRISM ? __dmul_rn(P.two_pi_G, I) : __dadd_rn(g, -__dmul_rn(P.two_pi_G, I));
        }
        __syncwarp();
        if (P.g_kind == MCG_G_PRISM) {
            for (int r0 = 0; r0 < n * NC; r0 += 4) {
                const int r = r0 + (lane >> 3) < n * NC ? r0 + (lane >> 3) : n * NC - 1;
                Exit& e = walks[__fns(mask, 0, r / NC + 1)].exit[r % NC];
                const double* x = e.X;
                const int i = lane & 1, jj = (lane >> 1) & 1, k = (lane >> 2) & 1;
                const double f = prism_corner((i ? P.phi[0] : P.plo[0]) - x[0], (jj ? P.phi[1] : P.plo[1]) - x[1],
                                              (k ? P.phi[2] : P.plo[2]) - x[2]);
                double s = 0.0;  // the corners in the order of prism_potential
                for (int q = 0; q < 8; ++q) {
                    const double v = __shfl_sync(kFull, f, (lane & 24) + q);
                    s += ((3 - (q & 1) - ((q >> 1) & 1) - (q >> 2)) & 1) ? -v : v;
                }
                if ((lane & 7) == 0 && r0 + (lane >> 3) < n * NC) e.sum = __dadd_rn(-P.G * P.rho0 * s, -e.sum);
            }
            __syncwarp();
        }
        if (j < n && c == 0)
            write_path(P, status, w->item, w->exit[0].sum, CRN ? w->exit[1].sum : 0.0, CRN ? w->exit[2].sum : 0.0,
                       (int64_t)w->steps);
        __syncwarp();
        for (int i = 0; i < n; ++i) mask &= mask - 1u;
    }
}

template <int RHO, bool CRN, bool SEG>
__global__ void __launch_bounds__(128, 4) walk64_kernel(const WalkParams P, const Near T)
{
    constexpr int NC = CRN ? 3 : 1;
    __shared__ fx::Tables tables;
    __shared__ Walk sh_walk[4][kSlots];
    __shared__ double2 sh_move[4][6 * kMoveRow];  // increments, then positions (rows 2 c, 2 c + 1: coordinate c)
    __shared__ float sh_df[4][12][32];            // the increments in single precision
    for (int i = threadIdx.x; i < (int)(sizeof(fx::Tables) / 4); i += blockDim.x)
        ((uint32_t*)&tables)[i] = ((const uint32_t*)&fx::g_tables)[i];
    __syncthreads();
    Walk* walks = sh_walk[threadIdx.x >> 5];
    double2* move = sh_move[threadIdx.x >> 5];
    float(*df)[32] = sh_df[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    unsigned livem = 0u, donem = 0u;  // slots: live walks, walks to evaluate
    bool drained = false;
    unsigned round = 0u;

    for (;;) {
        if ((++round & 15u) == 0u && cancelled(P)) {
            if (lane == 0) atomicOr(P.status, 1 << MCG_ERR_CANCELLED);
            if (lane < kSlots && (livem >> lane & 1u)) {  // these walks give no result
                const Walk& w = walks[lane];
                P.pp_u[w.item] = kNaN;
                P.pp_d[w.item] = kNaN;
                P.pp_steps[w.item] = (int64_t)w.steps + (int64_t)__popc(w.alive) * 4 * (int64_t)w.blk;
            }
            livem = 0u;
            drained = true;
        }
        const unsigned live = (unsigned)__popc(livem);
        if (!drained && live < (unsigned)P.quota) {
            const unsigned want = (unsigned)P.quota - live;
            if ((unsigned)(kSlots - __popc(livem | donem)) < want) {
                evaluate<RHO, CRN, SEG>(P, walks, donem);
                donem = 0u;
            }
            unsigned long long base = 0ull;
            if (lane == 0) base = atomicAdd(P.counter, (unsigned long long)want);
            base = __shfl_sync(kFull, base, 0);
            drained = base + want >= P.total;
            const unsigned long long item = base + (unsigned)lane;
            unsigned slot = 0u;
            bool start = lane < (int)want && item < P.total;
            if (start) {
                slot = __fns(~(livem | donem), 0, lane + 1);
                Walk& w = walks[slot];
                const double* st = P.stations;
                unsigned long long local = item, N = (unsigned long long)P.N, p0 = (unsigned long long)P.p0;
                int32_t* status = P.status;
                w.k0 = P.key0;
                w.k1 = P.key1;
                ModelRef M = model_of(P);
                if constexpr (SEG) {
                    w.seg = find_seg(P, item);
                    const WalkSeg& g = P.seg[w.seg];
                    local = item - g.begin;
                    N = (unsigned long long)g.N;
                    p0 = (unsigned long long)g.p0;
                    st = g.stations;
                    status = g.status;
                    w.k0 = g.key0;
                    w.k1 = g.key1;
                    M = model_of(g);
                }
                const uint32_t s = (uint32_t)(local / N);
                start = station_ok(P, st, status, s, item);
                if (start) {
                    w.s = s;
                    w.p = (uint32_t)(p0 + local % N);
                    w.item = item;
                    w.steps = 0ull;
                    w.blk = 0u;
                    w.alive = CRN ? 7u : 1u;
                    for (int k = 0; k < 3; ++k) w.w[k] = st[3 * s + k];
                    for (int c = 0; c < NC; ++c) {
                        const double X[3] = {w.w[0], w.w[1], __dadd_rn(w.w[2], c == 0 ? 0.0 : (c == 1 ? P.h : -P.h))};
                        if constexpr (kTwoValued<RHO>) w.acc[c] = support_exact(P, X[0], X[1], X[2]) ? 1u : 0u;
                        else w.acc[c] = (unsigned long long)__double_as_longlong(0.5 * rho_f64(P, M, X));
                    }
                }
            }
            livem |= __reduce_or_sync(kFull, start ? 1u << slot : 0u);
            __syncwarp();
        }
        if (livem == 0u) {
            if (!drained) continue;
            evaluate<RHO, CRN, SEG>(P, walks, donem);
            break;
        }

        // G live walks, k lanes each (a power of two)
        const int G = __popc(livem), k = G == 1 ? 32 : (G == 2 ? 16 : (G <= 4 ? 8 : 4));
        const bool mine = lane / k < G;
        const int g = mine ? lane / k : G - 1, l = lane & (k - 1);
        const int slot = (int)__fns(livem, 0, g + 1);
        const unsigned gmask = (k == 32 ? kFull : ((1u << k) - 1u)) << (lane & ~(k - 1));
        // the chain's walk and coordinate of this lane
        const int chain = lane % 3, chain_g = lane / 3;
        Walk& cw = walks[chain_g < G ? (int)__fns(livem, 0, chain_g + 1) : slot];
        Walk& w = walks[slot];
        const uint32_t gs = w.s, gp = w.p, gk0 = SEG ? w.k0 : P.key0, gk1 = SEG ? w.k1 : P.key1;
        uint32_t gblk = w.blk;
        unsigned gal = w.alive;
        ModelRef M = model_of(P);
        if constexpr (SEG) M = model_of(P.seg[w.seg]);
        const int64_t cap_blk = cap_block(P);
        unsigned n_in[3] = {0u, 0u, 0u};        // this lane's points of the support ...
        double r_in[3] = {0.0, 0.0, 0.0};       // ... or densities, not yet in the walk's sums
        auto add_up = [&]() {
            if constexpr (kTwoValued<RHO>) {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if (n_in[c]) atomicAdd(&w.acc[c], 2ull * n_in[c]);
                    n_in[c] = 0u;
                }
            } else if constexpr (RHO == MCG_RHO_VOXEL) {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    double v = r_in[c];
                    for (int d = k >> 1; d > 0; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
                    if (mine && l == 0)
                        w.acc[c] = (unsigned long long)__double_as_longlong(__longlong_as_double((long long)w.acc[c]) + v);
                    r_in[c] = 0.0;
                }
            }
            __syncwarp();
        };
        // increment j of this lane's block
        auto put = [&](uint32_t j, double d, float d_f) {
            const uint32_t m = (j * 11u) >> 5, c = j - 3u * m;
            ((double*)&move[(2u * c + (m >> 1)) * kMoveRow + lane])[m & 1u] = d;
            df[j][lane] = d_f;
        };
        // coordinate c of the position after step m of this lane's block
        auto after = [&](int m, int c) -> double {
            return ((const double*)&move[(2 * c + (m >> 1)) * kMoveRow + lane])[m & 1];
        };
        bool ended = false, capped = false;
        for (int r = 0; r < 16; ++r) {
            int kk = k;
            if ((int64_t)gblk + kk > cap_blk) kk = (int)(cap_blk - (int64_t)gblk);
            const bool act = mine && l < kk;
            const uint32_t myblk = gblk + (uint32_t)l;
            // the block's increments, a Philox call at a time (unrolled over all
            // six pairs, the body left the warps waiting for the instruction
            // cache)
            float reach = 0.0f;  // -(sum of the radii)
#pragma unroll 1
            for (uint32_t i = 0; i < 3; ++i) {
                uint4 v = philox4x32_10(make_uint4(3u * myblk + i, gp, gs, 0u), gk0, gk1);
#pragma unroll
                for (uint32_t q = 0; q < 2; ++q) {  // (two at once: a lone walk waits for each)
                    double rd;
                    float rf;
                    int64_t co, si;
                    double cs, sn;
                    fx::polar64(tables, v.x, v.y, rd, rf, co, si, cs, sn);
                    v.x = v.z;
                    v.y = v.w;
                    rf *= T.sd;
                    reach -= rf;
                    const uint32_t j = 4u * i + 2u * q;  // normals j, j + 1: coordinate j % 3 of step j / 3
                    put(j, __dmul_rn(P.sd, __dmul_rn(rd, cs)), rf * ((float)(int32_t)(co >> 32) * 0x1p-31f));
                    put(j + 1u, __dmul_rn(P.sd, __dmul_rn(rd, sn)), rf * ((float)(int32_t)(si >> 32) * 0x1p-31f));
                }
            }
            double W0[3] = {w.w[0], w.w[1], w.w[2]};  // before the block (of the round, for its first)
            __syncwarp();
            if (chain_g < G) {
                double x = cw.w[chain];
                double2* a = move + 2 * chain * kMoveRow + chain_g * k;
                double2* b = a + kMoveRow;
                double2 p = a[0], q = b[0];
                for (int i = 0; i < k; ++i) {
                    const int n = i + 1 < k ? i + 1 : i;
                    const double2 pn = a[n], qn = b[n];
                    x = p.x = __dadd_rn(x, p.x);
                    x = p.y = __dadd_rn(x, p.y);
                    x = q.x = __dadd_rn(x, q.x);
                    x = q.y = __dadd_rn(x, q.y);
                    a[i] = p;
                    b[i] = q;
                    p = pn;
                    q = qn;
                }
            }
            __syncwarp();
            if (l > 0)
                for (int c = 0; c < 3; ++c) W0[c] = move[(2 * c + 1) * kMoveRow + lane - 1].y;
            float f[3];
            for (int c = 0; c < 3; ++c) f[c] = (float)(W0[c] - P.cen[c]);
            const float nr[6] = {reach, 0.f, 0.f, 0.f, 0.f, 0.f};
            bool inside, quiet;
            if (P.ball) block_bounds<RHO, true>(P, f[0], f[1], f[2], nr, inside, quiet);
            else block_bounds<RHO, false>(P, f[0], f[1], f[2], nr, inside, quiet);
            const bool all_inside = __all_sync(kFull, inside || !act);
            if (!__all_sync(kFull, quiet || !act)) {
                unsigned la = act ? gal : 0u, out = 0u, om = 0u, of = 0u;
                unsigned n[3] = {0u, 0u, 0u};
                double rs[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
                for (int m = 0; m < 4; ++m) {
                    for (int c = 0; c < 3; ++c) f[c] += df[3 * m + c][lane];
                    auto W = [&](int c) { return after(m, c); };
                    if (!all_inside && la) {
                        const unsigned gone = la & ~inside64<CRN>(P, T, f, W);
                        out |= gone;
                        la &= ~gone;
#pragma unroll
                        for (int c = 0; c < NC; ++c)
                            if (gone & (1u << c)) om |= (unsigned)m << (2 * c);
                        if (!SEG && P.bridge) {
#pragma unroll 1
                            for (int c = 0; c < NC; ++c) {
                                if (!(la & (1u << c))) continue;
                                double X[3], Y[3];
                                for (int i = 0; i < 3; ++i) {
                                    X[i] = m == 0 ? W0[i] : after(m - 1, i);
                                    Y[i] = after(m, i);
                                }
                                X[2] = copy_z(P, c, X[2]);
                                Y[2] = copy_z(P, c, Y[2]);
                                const int fb = bridge_face_f64(P, X, Y, gs, gp, 4u * myblk + (uint32_t)m);
                                if (fb < 0) continue;
                                out |= 1u << c;
                                la &= ~(1u << c);
                                om |= (unsigned)m << (2 * c);
                                of |= (unsigned)(fb + 1) << (3 * c);
                            }
                        }
                    }
                    if (la) {
                        if constexpr (kTwoValued<RHO>) {
                            const unsigned in = la & support64<RHO, CRN>(P, T, f, W);
#pragma unroll
                            for (int c = 0; c < NC; ++c) n[c] += (in >> c) & 1u;
                        } else if constexpr (RHO == MCG_RHO_VOXEL) {
                            double v[3];
                            voxel64<CRN>(P, T, M, f, W, v);
#pragma unroll
                            for (int c = 0; c < NC; ++c)
                                if (la & (1u << c)) rs[c] += v[c];
                        }
                    }
                }
                int first[3] = {32, 32, 32};  // the lane of the round in which each copy leaves
                const bool any_out = __any_sync(kFull, out != 0u);
                if (any_out) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const unsigned b = __ballot_sync(kFull, (out >> c) & 1u) & gmask;
                        if (b) first[c] = __ffs(b) - 1;
                    }
                }
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (lane <= first[c]) {
                        n_in[c] += n[c];
                        if constexpr (RHO == MCG_RHO_VOXEL) r_in[c] += rs[c];
                    }
                if (any_out) {
                    add_up();
                    unsigned left = 0u;
#pragma unroll
                    for (int c = 0; c < NC; ++c) left |= first[c] < 32 ? 1u << c : 0u;
#pragma unroll 1
                    for (int c = 0; c < NC; ++c) {
                        if (!mine || lane != (c == 0 ? first[0] : (c == 1 ? first[1] : first[2]))) continue;
                        const int m = (int)((om >> (2 * c)) & 3u);
                        Exit& e = w.exit[c];
                        for (int i = 0; i < 3; ++i) {
                            e.X[i] = m == 0 ? W0[i] : after(m - 1, i);
                            e.Y[i] = after(m, i);
                        }
                        e.X[2] = copy_z(P, c, e.X[2]);
                        e.Y[2] = copy_z(P, c, e.Y[2]);
                        // (the moves' place holds positions now)
                        step_of(tables, P.sd, make_uint4(3u * myblk, gp, gs, 0u), gk0, gk1, m, e.dW);
                        e.face = (int)((of >> (3 * c)) & 7u) - 1;
                        if constexpr (kTwoValued<RHO>)  // (0 for any rho0 where the walk never met the body)
                            e.sum = w.acc[c] ? 0.5 * P.rho0 * (double)(long long)w.acc[c] : 0.0;
                        else e.sum = __longlong_as_double((long long)w.acc[c]);
                        atomicAdd(&w.steps, (unsigned long long)nstep_of(myblk, m));
                    }
                    gal &= ~left;
                }
            }
            __syncwarp();
            if (act && l == kk - 1)
                for (int c = 0; c < 3; ++c) w.w[c] = move[(2 * c + 1) * kMoveRow + lane].y;
            __syncwarp();
            gblk += (uint32_t)kk;
            if (mine && gal == 0u) ended = true;
            else if (mine && (int64_t)gblk >= cap_blk) ended = capped = true;
            if (__any_sync(kFull, ended)) break;  // regroup the others, or take new walks
        }
        add_up();
        if (mine && l == 0) {
            w.blk = gblk;
            w.alive = gal;
            if (capped) {
                atomicOr(SEG ? P.seg[w.seg].status : P.status, 1 << MCG_ERR_STEP_CAP);
                P.pp_u[w.item] = kNaN;
                P.pp_d[w.item] = kNaN;
                P.pp_steps[w.item] = (int64_t)w.steps + (int64_t)__popc(gal) * 4 * (int64_t)gblk;
            }
        }
        const unsigned end = __reduce_or_sync(kFull, ended ? 1u << slot : 0u);
        donem |= end & ~__reduce_or_sync(kFull, capped ? 1u << slot : 0u);
        livem &= ~end;
        __syncwarp();
        if (__popc(donem) >= kBatch) {
            evaluate<RHO, CRN, SEG>(P, walks, donem);
            donem = 0u;
        }
    }
}

Near make_near(const WalkParams& P)
{
    Near T = {};
    double R = 0.0;
    for (int k = 0; k < 3; ++k) R = std::fmax(R, 0.5 * (P.hi[k] - P.lo[k]));
    // a float step's position: 4 additions and a product, each within 2^-24 of
    // the walk's reach (the domain and one step beyond it)
    const double reach = R + P.h + 7.0 * P.sd, err = 2e-6 * reach;
    T.sd = std::nextafter((float)P.sd, INFINITY);
    T.face = (float)err;
    T.ball = (float)(4.0 * err * reach);
    T.sphere = (float)(4.0 * err * (P.srad + err));
    if (P.rho_kind == MCG_RHO_SPHERE)
        for (int k = 0; k < 3; ++k)
            if (!(std::fabs(P.sc[k] - P.cen[k]) < 2.0 * reach) || !(P.srad < 4.0 * reach)) T.sphere = INFINITY;
    if (P.rho_kind == MCG_RHO_VOXEL)
        for (int k = 0; k < 3; ++k)
            T.cell[k] = (float)(2.0 * (err + 2e-7 * std::fabs(P.org[k] - P.cen[k])) / P.sp[k]);
    return T;
}

template <int RHO>
const void* fn(bool crn, bool seg)
{
    if (seg) return crn ? (const void*)walk64_kernel<RHO, true, true> : (const void*)walk64_kernel<RHO, false, true>;
    return crn ? (const void*)walk64_kernel<RHO, true, false> : (const void*)walk64_kernel<RHO, false, false>;
}

}  // namespace

const void* walk64_fn(int rho_kind, bool crn, bool seg)
{
    switch (rho_kind) {
    case MCG_RHO_SPHERE: return fn<MCG_RHO_SPHERE>(crn, seg);
    case MCG_RHO_PRISM: return fn<MCG_RHO_PRISM>(crn, seg);
    case MCG_RHO_VOXEL: return fn<MCG_RHO_VOXEL>(crn, seg);
    default: return fn<MCG_RHO_NONE>(crn, seg);
    }
}

cudaError_t launch_walk64(const WalkParams& P0, int block, int blocks, cudaStream_t st)
{
    WalkParams P = P0;
    // walks per warp: spread over all resident warps, at most kLiveMax each
    // (more only share the lanes differently)
    const long long per_block = block / 32;
    const long long per_warp = (long long)(P.total / (unsigned long long)(blocks * per_block));
    P.quota = (int32_t)(per_warp < 1 ? 1 : per_warp > (long long)kLiveMax ? kLiveMax : per_warp);
    const long long need = (long long)((P.total + (unsigned long long)per_block - 1ull) / (unsigned long long)per_block);
    const int grid = need < (long long)blocks ? (int)need : blocks;
    Near T = make_near(P);
    void* args[2] = {&P, &T};
    cudaLaunchKernel(walk64_fn(P.rho_kind, P.crn != 0, P.seg != nullptr), dim3((unsigned)(grid > 0 ? grid : 1)),
                     dim3((unsigned)block), args, 0, st);
    return cudaGetLastError();
}

void preload_walk64_kernels()
{
    for (int kind : {MCG_RHO_NONE, MCG_RHO_SPHERE, MCG_RHO_PRISM, MCG_RHO_VOXEL})
        for (int q = 0; q < 4; ++q) {
            cudaFuncAttributes a;
            if (cudaFuncGetAttributes(&a, walk64_fn(kind, q & 1, q & 2)) != cudaSuccess) cudaGetLastError();
        }
}

}  // namespace mcg
