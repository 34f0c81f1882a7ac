// mcg_walk.cuh -- what the mixed walk (mcg_walk.cu) and the double-precision
// walk (mcg_walk64.cu) share: claiming work, cancellation, the conservative
// tests of a block and the exit geometry.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "mcg_device.cuh"
#include "mcg_internal.h"

namespace mcg {

constexpr unsigned kFull = 0xffffffffu;
constexpr double kNaN = __builtin_nan("");

// Claims new items for free lanes of this warp while it holds fewer than
// `quota` walks.  Returns true on the lanes that got one (in `item`); sets
// the warp-uniform `drained` once the work list has no more.
__device__ __forceinline__ bool refill(const WalkParams& P, bool busy, unsigned quota, bool& drained,
                                       unsigned long long& item)
{
    const unsigned freem = __ballot_sync(kFull, !busy);
    const unsigned live = 32u - (unsigned)__popc(freem);
    if (drained || live >= quota) return false;
    const int lane = threadIdx.x & 31;
    const unsigned rank = (unsigned)__popc(freem & ((1u << lane) - 1u));
    const bool want = !busy && rank < quota - live;
    const unsigned wantm = __ballot_sync(kFull, want);
    const int leader = __ffs(wantm) - 1;
    unsigned long long base = 0ull;
    if (lane == leader) base = atomicAdd(P.counter, (unsigned long long)__popc(wantm));
    base = __shfl_sync(kFull, base, leader);
    drained = base + (unsigned long long)__popc(wantm) >= P.total;
    item = base + rank;  // the wanting lanes are the first of the free ones
    return want && item < P.total;
}

// A station whose walk copies are not all strictly inside Omega gets NaN
// and the MCG_ERR_ARG bit (mcgrav_solve rejects such stations up front).
__device__ __forceinline__ bool station_ok(const WalkParams& P, const double* stations, int32_t* status, uint32_t s,
                                           unsigned long long item)
{
    const double x = stations[3 * s], y = stations[3 * s + 1], z = stations[3 * s + 2];
    bool ok;
    if (P.ball) {
        const double dx = x - P.cen[0], dy = y - P.cen[1], dz = z - P.cen[2];
        const double q = dx * dx + dy * dy;
        ok = q + dz * dz < P.R2 && q + (dz + P.h) * (dz + P.h) < P.R2 && q + (dz - P.h) * (dz - P.h) < P.R2;
    } else {
        ok = x > P.lo[0] && x < P.hi[0] && y > P.lo[1] && y < P.hi[1] && z - P.h > P.lo[2] && z + P.h < P.hi[2] &&
             z > P.lo[2] && z < P.hi[2];
    }
    if (!ok) {
        P.pp_u[item] = kNaN;
        P.pp_d[item] = kNaN;
        P.pp_steps[item] = 0;  // no completion flag: the mixed walk's exit kernel writes NaN too
        atomicOr(status, 1 << MCG_ERR_ARG);
    }
    return ok;
}

__device__ __forceinline__ int64_t nstep_of(uint32_t blk, int m) { return 4 * (int64_t)blk + m + 1; }

// The block at whose end a live walk has reached the step cap (max_steps may be
// the largest integer: no rounding up by an addition).
__device__ __forceinline__ int64_t cap_block(const WalkParams& P) { return P.max_steps / 4 + (P.max_steps % 4 != 0); }

// The cancel flag may live in host-mapped or device memory and is written
// by the host while the kernel runs: read it with a system-scope relaxed
// load so the write is observed whatever caches the line.
__device__ __forceinline__ bool cancelled(const WalkParams& P)
{
    int c = 0;
    if ((threadIdx.x & 31) == 0 && P.cancel != nullptr)
        asm volatile("ld.relaxed.sys.global.s32 %0, [%1];" : "=r"(c) : "l"((const void*)P.cancel) : "memory");
    return __shfl_sync(kFull, c, 0) != 0;
}

// A density that is rho0 or 0: its source sum is rho0 times a count of
// points, kept exactly (a single-precision count of whole and half points in
// registers, half points as a 64-bit integer beyond it), so no double
// precision is needed before the exit and the sum does not depend on the
// order of its terms.
template <int RHO>
constexpr bool kTwoValued = RHO == MCG_RHO_PRISM || RHO == MCG_RHO_SPHERE;
template <int RHO>
constexpr bool kVoxel = RHO == MCG_RHO_VOXEL || RHO == kRhoVoxelPacked;

// Conservative tests of a four-step block.  No coordinate moves by more than
// -(nr[0] + ... + nr[5]) over the block, so if that bound keeps every copy inside the conservative box
// (ball) -- `inside` -- the block needs no exit test, and if it also stays
// outside the density's support box -- `quiet` -- only the position changes.
// The boxes' margin, 1e-5 of the domain, is some twenty times the
// single-precision rounding of the bound and of the four moves.
template <int RHO, bool BALL>
__device__ __forceinline__ void block_bounds(const WalkParams& P, float x, float y, float z, const float nr[6],
                                             bool& inside, bool& quiet)
{
    const float rs = ((nr[0] + nr[1]) + (nr[2] + nr[3])) + (nr[4] + nr[5]);  // <= 0
    const float ax = fabsf(x) - rs, ay = fabsf(y) - rs, az = fabsf(z) - rs;
    if (BALL) inside = fmaf(ax, ax, fmaf(ay, ay, az * az)) < P.in_r2_f;
    else inside = ax < P.in_f[0] && ay < P.in_f[1] && az < P.in_f[2];
    quiet = inside;
    if constexpr (kTwoValued<RHO>)
        quiet = inside && (fabsf(x - P.far_c[0]) + rs > P.far_h[0] || fabsf(y - P.far_c[1]) + rs > P.far_h[1] ||
                           fabsf(z - P.far_c[2]) + rs > P.far_h[2]);
    else if constexpr (kVoxel<RHO>)
        quiet = false;
}

// Fraction theta in [0, 1] of the step X -> X + dW (coordinates relative to
// the ball centre) at which the segment leaves the ball of radius R: the
// positive root of |X + theta dW|^2 = R^2 in the form without cancellation.
__device__ __forceinline__ double ball_theta(const double* q, const double* dW, double R2)
{
    double a = 0.0, b = 0.0, c = -R2;
    for (int k = 0; k < 3; ++k) {
        a = __dadd_rn(a, __dmul_rn(dW[k], dW[k]));
        b = __dadd_rn(b, __dmul_rn(__dmul_rn(2.0, q[k]), dW[k]));
        c = __dadd_rn(c, __dmul_rn(q[k], q[k]));
    }
    const double D = __dadd_rn(__dmul_rn(b, b), -__dmul_rn(__dmul_rn(4.0, a), c));
    const double t = (b >= 0.0) ? __ddiv_rn(__dmul_rn(-2.0, c), __dadd_rn(b, __dsqrt_rn(D)))
                                : __ddiv_rn(__dadd_rn(-b, __dsqrt_rn(D)), __dmul_rn(2.0, a));
    return fmin(fmax(t, 0.0), 1.0);
}

}  // namespace mcg
