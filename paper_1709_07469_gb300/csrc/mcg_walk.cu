// mcg_walk.cu -- the mixed walk (Sec. 2.3 of the paper, steps 1-4) and the
// launch of either walk (the double-precision one is in mcg_walk64.cu).
//
// The kernel is persistent: every warp keeps up to 32 walks in flight and, as
// walks exit, refills the free lanes from a global work counter with one
// warp-aggregated atomic (__ballot_sync / __shfl_sync), so lanes do not idle
// behind the long exit-time tail.  A lane owns one path (station s, path p)
// and its common-random-number copies x0, x0 + h e_z, x0 - h e_z, which share
// every Gaussian increment.  Random numbers come four steps at a time: three
// Philox4x32-10 calls -> twelve normals -> four Euler-Maruyama steps.
//
//  * walk_mixed_kernel: single-precision stepping, random-number transform
//    and density lookup; the source integral keeps single-precision partial
//    sums over at most 64 steps which are flushed into a double accumulator
//    (an exact count where the density is rho0 or 0);
//    the exit-segment clip, the boundary value and the per-path estimate are
//    double precision and run in exit_mixed_kernel.  Where a warp has few
//    walks (small launches, the exit-time tail) its lanes share them.
//
// Launch shape: 128 threads, at least MCG_MIXED_MINB blocks per SM (the
// register bound that gave the best rate; the grid is sized from the
// occupancy the compiled kernel actually gets).
#include <type_traits>

#include <cuda_runtime.h>

#include "mcg_device.cuh"
#include "mcg_internal.h"
#include "mcg_walk.cuh"

namespace mcg {

namespace {

#ifndef MCG_MIXED_MINB
#define MCG_MIXED_MINB 5
#endif

// ---------------------------------------------------------------------------
// Bounded wait on a hand-over slot (failure-detection hook).  Walks stay in
// the warp that claimed them: once the work list is used up a warp runs the
// walks it has left as strips (below), which is faster than handing them to
// other warps (prism ore body, 30 x 8192 paths: 162 ms against 190 ms; voxel
// survey, 256 x 512: 5.8 against 11.6 ms).  mcg_options.fault_unpublished
// starts a launch with slots of the hand-over pool reserved and never
// published, as by a warp that died between the two; a warp without walks
// claims one, waits a bounded time for its ready flag and reports
// MCG_ERR_TIMEOUT.  pool_ctr[0]: slots reserved, [1]: slots claimed.
// ---------------------------------------------------------------------------
constexpr int kReadySpin = 1 << 20;                   // bounded wait for a ready flag (~0.1 s)

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* a)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* a)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
    return v;
}

// One thread: claims a reserved slot, if there is one, and waits for it.
__device__ __forceinline__ void pool_wait(const WalkParams& P)
{
    const unsigned long long c = ld_acquire_u64(P.pool_ctr + 1);
    if (c >= ld_acquire_u64(P.pool_ctr) || atomicCAS(P.pool_ctr + 1, c, c + 1ull) != c) return;
    uint32_t ready = 0u;
    for (int i = 0; i < kReadySpin && !ready; ++i) {
        ready = ld_acquire_u32(P.pool_ready + c);
        if (!ready) __nanosleep(64);
    }
    if (!ready) atomicOr(P.status, 1 << MCG_ERR_TIMEOUT);
}

// Mixed walk exit (run by exit_mixed_kernel, one thread per path, so the
// double-precision work is convergent): X, Y relative to the box centre in
// single precision as the walk computed them; the walk's sum acc (flushed +
// partial) is S = rho_0 / 2 + sum_{n=1}^{N-1} rho_n, so the trapezoid integral
// over the inside steps is dt (S - rho_{N-1} / 2).
__device__ __forceinline__ double exit_mixed(const WalkParams& P, const ModelRef& M, const float* Xf, const float* Yf,
                                             double acc, float rp)
{
    double X[3], dW[3], xs[3];
    for (int k = 0; k < 3; ++k) {
        X[k] = (double)Xf[k];
        dW[k] = (double)Yf[k] - (double)Xf[k];
    }
    double theta = 1.0;
    int face = -1;
    if (P.clip && P.ball) {
        theta = ball_theta(X, dW, P.R2);
        for (int k = 0; k < 3; ++k) xs[k] = P.cen[k] + (X[k] + theta * dW[k]);
    } else if (P.clip) {
        int kstar = -1;
        double tmin = __longlong_as_double(0x7ff0000000000000LL);
        for (int k = 0; k < 3; ++k) {
            if (!(fabsf(Yf[k]) >= P.half_f[k])) continue;  // the test that ended the walk
            const double b = (Yf[k] > 0.f ? P.hi[k] : P.lo[k]) - P.cen[k];
            const double t = (b - X[k]) / dW[k];
            if (t < tmin) {
                tmin = t;
                kstar = k;
            }
        }
        if (kstar < 0) return kNaN;
        theta = fmin(fmax(tmin, 0.0), 1.0);
        for (int k = 0; k < 3; ++k) xs[k] = P.cen[k] + (X[k] + theta * dW[k]);
        const bool upper = Yf[kstar] > 0.f;
        xs[kstar] = upper ? P.hi[kstar] : P.lo[kstar];
        face = 2 * kstar + (upper ? 1 : 0);
    } else {
        for (int k = 0; k < 3; ++k) xs[k] = P.cen[k] + (double)Yf[k];
    }
    const double r = rho_f64(P, M, xs);
    const double rpd = (double)rp;
    const double I = P.dt * (acc - 0.5 * rpd) + 0.5 * theta * P.dt * (rpd + r);
    return boundary_value<true>(P, M, face, xs) - P.two_pi_G * I;
}

// Exit record of copy c of item `item` (record c * total + item of frec):
// 32 bytes, written as two 16-byte stores that fill one sector -- X (the walk
// position before the exit step, copy 0's coordinates; copy c adds its z
// offset), Y (the copy's first point not strictly inside Omega) and the
// source sum (a double's bits or, where the density is rho0 or 0, a count of
// half points: recorded_sum).  rho at X is not stored:
// exit_mixed_kernel evaluates the same single-precision density function at
// the same X, which gives the walk's value bit for bit.  The record is valid
// once the item's step count carries kDoneFlag.
__device__ __forceinline__ void put_exit(const WalkParams& P, int c, unsigned long long item, float x0, float x1,
                                         float x2, float y0, float y1, float y2, unsigned long long acc)
{
    float4* r = (float4*)P.frec + 2 * ((size_t)c * P.total + item);
    r[0] = make_float4(x0, x1, x2, y0);
    r[1] = make_float4(y1, y2, __uint_as_float((unsigned)acc), __uint_as_float((unsigned)(acc >> 32)));
}

// Source sum of a copy, for its exit record: `held` is the flushed part (a
// double's bits, or a count of half points), `part` the single-precision part
// since.  The exit kernel turns a count into a sum: the double-precision
// product, taken here, costs the step loop its pipe even where no lane exits
// (bulk rate 1.043 -> 1.050e12 path-steps/s on the prism ore body).
template <int RHO>
__device__ __forceinline__ unsigned long long source_sum(unsigned long long held, float part)
{
    if constexpr (RHO == MCG_RHO_NONE)
        return 0ull;
    else if constexpr (kTwoValued<RHO>)
        return held + (unsigned long long)(unsigned)(2.0f * part);
    else
        return (unsigned long long)__double_as_longlong(__longlong_as_double((long long)held) + (double)part);
}
template <int RHO>
__device__ __forceinline__ double recorded_sum(const WalkParams& P, unsigned long long acc)
{
    if constexpr (kTwoValued<RHO>)
        return acc ? (double)P.rho0_f * (0.5 * (double)(long long)acc) : 0.0;  // (0 for any rho0)
    else
        return __longlong_as_double((long long)acc);
}

// The flushed part with `part` added (the same sum as source_sum's: a count since
// the last flush is below 2^22, so the width it is converted in does not matter).
template <int RHO>
__device__ __forceinline__ unsigned long long flushed(unsigned long long held, float part)
{
    if constexpr (kTwoValued<RHO>)
        return held + (unsigned long long)(2.0f * part);
    else
        return (unsigned long long)__double_as_longlong(__longlong_as_double((long long)held) + (double)part);
}

// Single-precision bridge test of the copies `cand` for step m of block blk
// (walk position (wx, wy, wz) -> (nx, ny, nz), box-centre coordinates, copy c
// shifted by +h, -h in z).  Returns the mask of copies that exit and, 3 bits
// per copy, their faces.
__device__ __noinline__ unsigned bridge_exits_f32(const WalkParams& P, unsigned cand, float wx, float wy, float wz,
                                                  float nx, float ny, float nz, float hf, uint32_t s, uint32_t p,
                                                  uint32_t blk, int m, unsigned* faces)
{
    const uint4 w = philox4x32_10(make_uint4(blk, p, s, 2u), P.key0, P.key1);
    const uint32_t word = m == 0 ? w.x : m == 1 ? w.y : m == 2 ? w.z : w.w;
    const float U = u01_f32(word);
    const float hx = P.half_f[0], hy = P.half_f[1], hz = P.half_f[2], K = P.bridge_k_f;
    const float pxy[4] = {__expf(K * (wx + hx) * (nx + hx)), __expf(K * (hx - wx) * (hx - nx)),
                          __expf(K * (wy + hy) * (ny + hy)), __expf(K * (hy - wy) * (hy - ny))};
    float qxy = 1.0f, pbest = -1.0f;
    int fbest = -1;
    for (int f = 0; f < 4; ++f) {
        qxy *= 1.0f - pxy[f];
        if (pxy[f] > pbest) {
            pbest = pxy[f];
            fbest = f;
        }
    }
    unsigned out = 0u, fb = 0u;
    for (int c = 0; c < 3; ++c) {
        if (!(cand & (1u << c))) continue;
        const float off = c == 0 ? 0.0f : (c == 1 ? hf : -hf);
        const float zX = wz + off, zY = nz + off;
        const float plo = __expf(K * (zX + hz) * (zY + hz)), phi = __expf(K * (hz - zX) * (hz - zY));
        const float q = qxy * (1.0f - plo) * (1.0f - phi);
        if (U < 1.0f - q) {
            int f = fbest;
            float pb = pbest;
            if (plo > pb) {
                pb = plo;
                f = 4;
            }
            if (phi > pb) f = 5;
            out |= 1u << c;
            fb |= (unsigned)f << (3 * c);
        }
    }
    *faces = fb;
    return out;
}

// ---------------------------------------------------------------------------
// Mixed-precision walk: single-precision stepping and no double-precision
// arithmetic in the step loop.  A warp works in one of two ways:
//
//  * lanes (more than kStripMax walks live): a lane steps a walk of its own;
//    the three common-random-number copies are updated branch-free, exits
//    (rare) take a side branch that writes an exit record, which
//    exit_mixed_kernel turns into per-path values.  Up to 16 blocks (64
//    steps) between refills;
//  * strips (at most kStripMax walks live: a small launch, or the exit-time
//    tail of a large one): k = 32 / walks lanes share a walk.  The random
//    numbers of different blocks do not depend on one another, so each lane
//    makes those of one block; only the positions form a serial chain, one
//    fused multiply-add per coordinate and step, which a lane per coordinate
//    runs through shared memory; then each lane tests and sums its own block.
//
// Both take the same steps in the same arithmetic, so a walk's numbers do not
// depend on how it was run (but for the rounding of a voxel grid's sums, which
// are flushed where the warp regroups).  What bounds them, on the prism ore body (1 m
// steps): a walk alone takes 115 ns a step as a lane (the block's dependent
// generator, logarithm and root, ~950 cycles) and 7 ns as a strip of 32 (that
// once per 32 blocks, and the chain, 16 cycles a block); with the GPU full,
// lanes run 340 steps/ns, strips 240 (k = 2) to 190 (k = 16), as the chain
// idles most lanes, so a full warp runs lanes.  Solves that this shortens:
// 30 x 256 paths 178 -> 16 ms, 30 x 8192 paths 333 -> 150 ms.  The price: the
// strips' registers leave a full launch 20 warps per SM instead of 24, 1.6 %
// where a second stream hides the tail anyway (30 x 131072 paths a step).
// ---------------------------------------------------------------------------
constexpr unsigned kStripMax = 16;
constexpr int kStripRow = 33;  // float4 per row: rows of one block column fall into different banks

// Copies strictly inside Omega at the walk position (x, y, z): bit c for copy c.
template <bool CRN, bool BALL>
__device__ __forceinline__ unsigned copies_inside(const WalkParams& P, float x, float y, float z, float hf)
{
    unsigned ins;
    if (BALL) {
        // (explicit rounding: lanes and strips must take the same decisions)
        const float q = __fmaf_rn(x, x, __fmul_rn(y, y));
        const float zb = z + hf, zc = z - hf;
        ins = (__fmaf_rn(z, z, q) < P.R2_f) ? 1u : 0u;
        if (CRN) {
            ins |= (__fmaf_rn(zb, zb, q) < P.R2_f) ? 2u : 0u;
            ins |= (__fmaf_rn(zc, zc, q) < P.R2_f) ? 4u : 0u;
        }
    } else {
        const bool inxy = fabsf(x) < P.half_f[0] && fabsf(y) < P.half_f[1];
        ins = (inxy && fabsf(z) < P.half_f[2]) ? 1u : 0u;
        if (CRN) {
            ins |= (inxy && fabsf(z + hf) < P.half_f[2]) ? 2u : 0u;
            ins |= (inxy && fabsf(z - hf) < P.half_f[2]) ? 4u : 0u;
        }
    }
    return ins;
}

// Y of copy c for a bridge exit on face f below the step's end (x, y, z).
__device__ __forceinline__ void bridge_point(const WalkParams& P, int c, int f, float x, float y, float z, float hf,
                                             float out[3])
{
    out[0] = x;
    out[1] = y;
    out[2] = z + (c == 0 ? 0.0f : (c == 1 ? hf : -hf));
    const float b = (f & 1) ? P.half_f[f >> 1] : -P.half_f[f >> 1];
    if ((f >> 1) == 0) out[0] = b;
    else if ((f >> 1) == 1) out[1] = b;
    else out[2] = b;
}

// The moves of block `blk` of walk (s, p) to column `lane` of the strip:
// per coordinate four steps to a float4, radii in rows 0-2, cosines or sines
// in rows 3-5.  Returns minus the sum of the radii.
__device__ __forceinline__ float strip_moves(float4* strip, int lane, uint32_t s, uint32_t p, uint32_t blk, uint32_t k0,
                                             uint32_t k1, float lnscale)
{
    float nr[6], cs[12];
    polar12_f32(s, p, blk, k0, k1, lnscale, nr, cs);
    strip[0 * kStripRow + lane] = make_float4(nr[0], nr[1], nr[3], nr[4]);
    strip[1 * kStripRow + lane] = make_float4(nr[0], nr[2], nr[3], nr[5]);
    strip[2 * kStripRow + lane] = make_float4(nr[1], nr[2], nr[4], nr[5]);
    strip[3 * kStripRow + lane] = make_float4(cs[0], cs[3], cs[6], cs[9]);
    strip[4 * kStripRow + lane] = make_float4(cs[1], cs[4], cs[7], cs[10]);
    strip[5 * kStripRow + lane] = make_float4(cs[2], cs[5], cs[8], cs[11]);
    return ((nr[0] + nr[1]) + (nr[2] + nr[3])) + (nr[4] + nr[5]);
}

// SEG: a multi-request launch (the segment table maps each item to its
// request); each lane then carries its walk's generator key and model array,
// and keeps the segment index with the walk's other cold state.
template <int RHO, bool CRN, bool BRIDGE, bool BALL, bool SEG>
__global__ void __launch_bounds__(128, MCG_MIXED_MINB) walk_mixed_kernel(const WalkParams P)
{
    static_assert(!(SEG && (BRIDGE || BALL)), "multi-request launches use the box without the bridge test");
    constexpr int NC = CRN ? 3 : 1;
    // Per-walk state touched only at refills, exits and flushes lives in
    // shared memory (one slot per thread); the step loop keeps the position,
    // the partial sums, the path indices and the live-copy mask in registers.
    __shared__ unsigned long long sh_acc[3][128];  // flushed sums per copy (source_sum)
    __shared__ unsigned long long sh_item[128];    // work item of the walk
    __shared__ unsigned long long sh_steps[128];   // EM steps of the copies that have exited
    __shared__ int sh_seg[SEG ? 128 : 1];          // segment of the walk (multi-request launch)
    // strips: the blocks' increments, then densities; the walks' positions and
    // the blocks' last ones; per copy the counts (two-valued) or running sums
    __shared__ float4 sh_strip[4][6 * kStripRow];
    __shared__ float sh_base[4][3 * kStripMax];
    __shared__ float sh_end[4][3 * kStripRow];
    using Part = std::conditional_t<kTwoValued<RHO>, unsigned, float>;  // half points, or a running sum
    __shared__ Part sh_part[RHO == MCG_RHO_NONE ? 1 : 3][128];
    __shared__ int sh_own[4][kStripMax];  // slot of the g-th live walk
    const int t = threadIdx.x;
    bool busy = false, drained = false;
    uint32_t s = 0u, p = 0u, blk = 0u;
    float wx = 0.f, wy = 0.f, wz = 0.f;
    float S0 = 0.f, S1 = 0.f, S2 = 0.f;  // single-precision partial sums (two-valued density: counts)
    unsigned alive = 0u;
    const float hf = CRN ? P.h_f : 0.0f;
    unsigned round = 0u;
    const int lane = t & 31;
    const unsigned lanes_below = (1u << lane) - 1u;
    bool stop = false;  // cancelled: take no more work of any kind
    uint32_t k0 = P.key0, k1 = P.key1;  // generator key of the lane's walk
    ModelRef M = model_of(P);           // model arrays of the lane's walk
    // the lane's walk now belongs to the request of launch item `it`
    auto adopt = [&](unsigned long long it) {
        if constexpr (SEG) {
            const int gi = find_seg(P, it);
            const WalkSeg& g = P.seg[gi];
            k0 = g.key0;
            k1 = g.key1;
            M = model_of(g);
            sh_seg[t] = gi;
        }
    };
    auto flush = [&]() {
        if constexpr (RHO != MCG_RHO_NONE) {
            sh_acc[0][t] = flushed<RHO>(sh_acc[0][t], S0);
            S0 = 0.f;
            if (CRN) {
                sh_acc[1][t] = flushed<RHO>(sh_acc[1][t], S1);
                sh_acc[2][t] = flushed<RHO>(sh_acc[2][t], S2);
                S1 = S2 = 0.f;
            }
        }
    };

    for (;;) {
        if ((++round & 15u) == 0u && cancelled(P)) {
            // walks in flight and unclaimed items give no result
            if (lane == 0) atomicOr(P.status, 1 << MCG_ERR_CANCELLED);
            if (busy) {
                const unsigned long long it = sh_item[t];  // (no completion flag: NaN)
                P.pp_steps[it] = (long long)sh_steps[t] + (long long)__popc(alive) * 4 * (long long)blk;
            }
            busy = false;
            drained = true;
            stop = true;
        }
        unsigned long long item = 0ull;
        bool start = refill(P, busy, (unsigned)P.quota, drained, item);
        const double* st = P.stations;
        if (start) {
            unsigned long long local = item, N = (unsigned long long)P.N, p0 = (unsigned long long)P.p0;
            int32_t* status = P.status;
            if constexpr (SEG) {
                adopt(item);
                const WalkSeg& g = P.seg[sh_seg[t]];
                local = item - g.begin;
                N = (unsigned long long)g.N;
                p0 = (unsigned long long)g.p0;
                st = g.stations;
                status = g.status;
            }
            s = (uint32_t)(local / N);
            p = (uint32_t)(p0 + local % N);
            start = station_ok(P, st, status, s, item);
        }
        if (start) {
            wx = (float)(st[3 * s + 0] - P.cen[0]);
            wy = (float)(st[3 * s + 1] - P.cen[1]);
            wz = (float)(st[3 * s + 2] - P.cen[2]);
            if constexpr (kTwoValued<RHO>) {
                const unsigned in = support3_f32<RHO>(P, wx, wy, wz, hf);
                S0 = (in & 1u) ? 0.5f : 0.0f;
                S1 = (in & 2u) ? 0.5f : 0.0f;
                S2 = (in & 4u) ? 0.5f : 0.0f;
            } else {
                float r0, r1, r2;
                rho3_f32<RHO>(P, SEG ? M : model_of(P), wx, wy, wz, hf, r0, r1, r2);
                S0 = 0.5f * r0;
                S1 = 0.5f * r1;
                S2 = 0.5f * r2;
            }
            sh_acc[0][t] = sh_acc[1][t] = sh_acc[2][t] = 0ull;
            sh_item[t] = item;
            sh_steps[t] = 0ull;
            alive = CRN ? 7u : 1u;
            blk = 0u;
            busy = true;
        }
        const unsigned livem = __ballot_sync(kFull, busy);
        if (livem == 0u) {
            if (!drained) continue;  // (every claimed station lay outside Omega)
            if (P.fault_unpublished && P.pool && !stop && lane == 0) pool_wait(P);
            break;
        }

        if (__popc(livem) <= (int)kStripMax) {
            // ----------------------------------------------------------------
            // Strips.  Group g of k lanes runs the g-th live walk; what the
            // group's lanes share is held alike in all of them.
            // ----------------------------------------------------------------
            const int G = __popc(livem), k = 32 / G, ks = k;
            const int g = lane / k < G ? lane / k : G - 1;
            const bool mine = lane / k < G;          // this lane belongs to a group
            const int l = lane - g * k;              // its block of the group's round
            float4* const strip = sh_strip[t >> 5];
            float* base = sh_base[t >> 5];
            const int* own = sh_own[t >> 5];
            const int rank = __popc(livem & lanes_below);
            // the counts move as half points, the running sums as they are
            auto part_of = [](float v) -> Part { return kTwoValued<RHO> ? (Part)(2.0f * v) : (Part)v; };
            auto value_of = [](Part v) -> float { return kTwoValued<RHO> ? 0.5f * (float)v : (float)v; };
            if (busy) {
                sh_own[t >> 5][rank] = t;
                base[3 * rank] = wx;
                base[3 * rank + 1] = wy;
                base[3 * rank + 2] = wz;
                if constexpr (RHO != MCG_RHO_NONE) {
                    sh_part[0][t] = part_of(S0);
                    if (CRN) {
                        sh_part[1][t] = part_of(S1);
                        sh_part[2][t] = part_of(S2);
                    }
                }
            }
            __syncwarp();
            const int slot = own[g], owner = slot & 31;
            const unsigned gmask = (k == 32 ? kFull : ((1u << k) - 1u)) << (g * k);
            const uint32_t gs = __shfl_sync(kFull, s, owner), gp = __shfl_sync(kFull, p, owner);
            uint32_t gblk = __shfl_sync(kFull, blk, owner);
            unsigned gal = __shfl_sync(kFull, alive, owner);
            uint32_t gk0 = k0, gk1 = k1;
            ModelRef gM = M;
            if constexpr (SEG) {
                gk0 = __shfl_sync(kFull, k0, owner);
                gk1 = __shfl_sync(kFull, k1, owner);
                gM.grid = (const float*)__shfl_sync(kFull, (unsigned long long)M.grid, owner);
                gM.zq = (const float4*)__shfl_sync(kFull, (unsigned long long)M.zq, owner);
            }
            unsigned N0 = 0u, N1 = 0u, N2 = 0u;  // this lane's points of the support, not yet in sh_part
            auto add_counts = [&]() {
                if (N0) atomicAdd((unsigned*)&sh_part[0][slot], 2u * N0);
                if (CRN && N1) atomicAdd((unsigned*)&sh_part[1][slot], 2u * N1);
                if (CRN && N2) atomicAdd((unsigned*)&sh_part[2][slot], 2u * N2);
                N0 = N1 = N2 = 0u;
                __syncwarp();
            };
            const uint32_t flushed_at = gblk;  // (the last regrouping)
            const int64_t cap_blk = cap_block(P);
            const bool near_cap = __any_sync(kFull, (int64_t)gblk + 16 * k >= cap_blk);
            bool ended = false;  // the group's walk is complete or capped
            // The chain of one coordinate of a walk from x, the four positions
            // of each block in the place of its radii; two blocks at a time,
            // the next two loaded meanwhile.
            auto run_chain = [&](int q, float x) {
                float4* rr = strip + (q % 3) * kStripRow + (q / 3) * k;
                const float4* cc = rr + 3 * kStripRow;
                auto four = [&x](const float4& a, const float4& b) {
                    float4 y;
                    x = y.x = fmaf(a.x, b.x, x);
                    x = y.y = fmaf(a.y, b.y, x);
                    x = y.z = fmaf(a.z, b.z, x);
                    x = y.w = fmaf(a.w, b.w, x);
                    return y;
                };
                float4 a0 = rr[0], b0 = cc[0], a1 = rr[1], b1 = cc[1];  // k >= 2
                int i = 0;
#pragma unroll 2
                for (; i + 4 <= k; i += 2) {
                    const float4 a2 = rr[i + 2], b2 = cc[i + 2], a3 = rr[i + 3], b3 = cc[i + 3];
                    rr[i] = four(a0, b0);
                    rr[i + 1] = four(a1, b1);
                    a0 = a2;
                    b0 = b2;
                    a1 = a3;
                    b1 = b3;
                }
                rr[i] = four(a0, b0);
                rr[i + 1] = four(a1, b1);
                if (i + 2 < k) rr[i + 2] = four(rr[i + 2], cc[i + 2]);  // k odd
            };
            // A lone walk waits for its chain: only each block's last position
            // is left (its lane repeats the four moves), as a store of all four
            // holds the registers of its operands, and the operands are
            // loaded three blocks ahead.  With the rounds compiled for it alone,
            // 7.2 ns a step against 9.8.
            auto run_lone_chain = [&](float x) {
                const float4 *rr = strip + lane * kStripRow, *cc = rr + 3 * kStripRow;
                float* e = sh_end[t >> 5] + lane * kStripRow;
                float4 a[3], b[3];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    a[j] = rr[j];
                    b[j] = cc[j];
                }
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const float4 &u = a[i % 3], &v = b[i % 3];
                    e[i] = x = fmaf(u.w, v.w, fmaf(u.z, v.z, fmaf(u.y, v.y, fmaf(u.x, v.x, x))));
                    if (i + 3 < 32) {
                        a[i % 3] = rr[i + 3];
                        b[i % 3] = cc[i + 3];
                    }
                }
            };
            // (compiled twice: for a lone walk, and for several)
            auto rounds = [&](auto lone) {
            for (int r = 0; r < 16; ++r) {
                // blocks of this round: up to k, not past the cap, and for a
                // density that is summed in single precision not past the
                // next flush (16 blocks after the last)
                constexpr bool LONE = decltype(lone)::value;
                const int k = LONE ? 32 : ks;
                int kk = k;
                if constexpr (kVoxel<RHO>) kk = min(kk, 16 - (int)((gblk - flushed_at) & 15u));
                if ((int64_t)gblk + kk > cap_blk) kk = (int)(cap_blk - (int64_t)gblk);
                const bool act = mine && l < kk;
                const float rs = strip_moves(strip, lane, gs, gp, gblk + (uint32_t)l, SEG ? gk0 : P.key0,
                                             SEG ? gk1 : P.key1, P.lnscale_f);
                __syncwarp();
                const float3 w0 = make_float3(base[3 * g], base[3 * g + 1], base[3 * g + 2]);  // before the round
                if constexpr (LONE) {
                    if (lane < 3) run_lone_chain(base[lane]);
                } else {
                    for (int q = lane; q < 3 * G; q += 32) run_chain(q, base[q]);
                }
                __syncwarp();
                float px[5], py[5], pz[5];
                if constexpr (LONE) {
                    const float* e = sh_end[t >> 5];
                    auto four = [&](int c, float x, float* p) {
                        const float4 a = strip[c * kStripRow + lane], b = strip[(c + 3) * kStripRow + lane];
                        p[0] = lane > 0 ? e[c * kStripRow + lane - 1] : x;
                        p[1] = fmaf(a.x, b.x, p[0]);
                        p[2] = fmaf(a.y, b.y, p[1]);
                        p[3] = fmaf(a.z, b.z, p[2]);
                        p[4] = fmaf(a.w, b.w, p[3]);
                    };
                    four(0, w0.x, px);
                    four(1, w0.y, py);
                    four(2, w0.z, pz);
                } else {
                    auto four = [&](int c, float x, float* p) {
                        const float4 a = strip[c * kStripRow + lane];
                        const float before = __shfl_up_sync(kFull, a.w, 1);
                        p[0] = l > 0 ? before : x;
                        p[1] = a.x;
                        p[2] = a.y;
                        p[3] = a.z;
                        p[4] = a.w;
                    };
                    four(0, w0.x, px);
                    four(1, w0.y, py);
                    four(2, w0.z, pz);
                }
                if (act && l == kk - 1) {  // (the others have read it before the chain)
                    base[3 * g] = px[4];
                    base[3 * g + 1] = py[4];
                    base[3 * g + 2] = pz[4];
                }
                bool inside, quiet;
                const float reach[6] = {rs, 0.f, 0.f, 0.f, 0.f, 0.f};
                block_bounds<RHO, BALL>(P, px[0], py[0], pz[0], reach, inside, quiet);
                bool any_out = false;
                if (!__all_sync(kFull, quiet || !act)) {
                    const bool all_inside = __all_sync(kFull, inside || !act);
                    const uint32_t myblk = gblk + (uint32_t)l;
                    unsigned la = act ? gal : 0u;  // copies live at this point of the block
                    unsigned out = 0u;             // copies that leave in this block ...
                    unsigned om = 0u, of = 0u;     // ... their step (2 bits each); bridge face + 1 (3 bits each)
                    unsigned n0 = 0u, n1 = 0u, n2 = 0u;  // points of the density's support (two-valued)
                    float rv[4][3];
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        if (!all_inside) {
                            const unsigned ins = copies_inside<CRN, BALL>(P, px[m + 1], py[m + 1], pz[m + 1], hf);
                            const unsigned gone = la & ~ins;
                            if (gone) {
                                out |= gone;
#pragma unroll
                                for (int c = 0; c < NC; ++c)
                                    if (gone & (1u << c)) om |= (unsigned)m << (2 * c);
                                la &= ins;
                            }
                            if (BRIDGE && la) {
                                unsigned faces = 0u;
                                const unsigned bx = bridge_exits_f32(P, la, px[m], py[m], pz[m], px[m + 1], py[m + 1],
                                                                     pz[m + 1], hf, gs, gp, myblk, m, &faces);
                                if (bx) {
                                    out |= bx;
                                    la &= ~bx;
#pragma unroll
                                    for (int c = 0; c < NC; ++c)
                                        if (bx & (1u << c)) {
                                            om |= (unsigned)m << (2 * c);
                                            of |= (((faces >> (3 * c)) & 7u) + 1u) << (3 * c);
                                        }
                                }
                            }
                        }
                        if constexpr (kTwoValued<RHO>) {
                            const unsigned in = la & support3_f32<RHO>(P, px[m + 1], py[m + 1], pz[m + 1], hf);
                            n0 += in & 1u;
                            n1 += (in >> 1) & 1u;
                            n2 += in >> 2;
                        } else if constexpr (kVoxel<RHO>) {
                            rho3_f32<RHO>(P, SEG ? gM : model_of(P), px[m + 1], py[m + 1], pz[m + 1], hf, rv[m][0],
                                          rv[m][1], rv[m][2]);
                        }
                    }
                    // the first block of the round in which each copy leaves
                    int first[3] = {32, 32, 32};
                    any_out = __any_sync(kFull, out != 0u);
                    if (any_out) {
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            const unsigned b = __ballot_sync(kFull, (out >> c) & 1u) & gmask;
                            if (b) first[c] = __ffs(b) - 1;
                        }
                    }
                    float pre[3] = {0.f, 0.f, 0.f};  // single-precision sums before this block (voxel)
                    if constexpr (kTwoValued<RHO>) {
                        // counts up to the exit; exact, so the order does not matter
                        if (lane <= first[0]) N0 += n0;
                        if (CRN && lane <= first[1]) N1 += n1;
                        if (CRN && lane <= first[2]) N2 += n2;
                        if (any_out) add_counts();
                    } else if constexpr (kVoxel<RHO>) {
                        // the same order of additions as a lane's: a chain
                        // over the round's blocks, lane q copy q % NC of walk q / NC
#pragma unroll
                        for (int c = 0; c < NC; ++c)
                            strip[(3 + c) * kStripRow + lane] =
                                act ? make_float4(rv[0][c], rv[1][c], rv[2][c], rv[3][c]) : make_float4(0.f, 0.f, 0.f, 0.f);
                        __syncwarp();
                        for (int q = lane; q < NC * G; q += 32) {
                            const int gq = q / NC, c = q % NC;
                            Part* part = &sh_part[c][own[gq]];
                            float S = value_of(*part);
                            float4* rr = strip + c * kStripRow + gq * k;
                            for (int i = 0; i < k; ++i) {
                                const float4 v = rr[3 * kStripRow + i];
                                rr[i].x = S;
                                S += v.x;
                                S += v.y;
                                S += v.z;
                                S += v.w;
                            }
                            *part = part_of(S);
                        }
                        __syncwarp();
#pragma unroll
                        for (int c = 0; c < NC; ++c) pre[c] = strip[c * kStripRow + lane].x;
                    }
                    if (any_out) {
                        const unsigned left = (first[0] < 32 ? 1u : 0u) | (first[1] < 32 ? 2u : 0u) |
                                              (first[2] < 32 ? 4u : 0u);
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            if (!mine || lane != first[c]) continue;
                            const unsigned m = (om >> (2 * c)) & 3u;
                            float x = 0.f, y = 0.f, z = 0.f, e[3] = {0.f, 0.f, 0.f}, ez = 0.f;
                            float part = pre[c];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                if (i == (int)m) {
                                    x = px[i];
                                    y = py[i];
                                    z = pz[i];
                                    e[0] = px[i + 1];
                                    e[1] = py[i + 1];
                                    ez = pz[i + 1];
                                }
                                if constexpr (kVoxel<RHO>)
                                    if (i < (int)m) part += rv[i][c];
                            }
                            if constexpr (kTwoValued<RHO>) part = value_of(sh_part[c][slot]);
                            e[2] = c == 0 ? ez : (c == 1 ? ez + hf : ez - hf);
                            if constexpr (BRIDGE) {
                                const int f = (int)((of >> (3 * c)) & 7u) - 1;
                                if (f >= 0) bridge_point(P, c, f, e[0], e[1], ez, hf, e);
                            }
                            put_exit(P, c, sh_item[slot], x, y, z, e[0], e[1], e[2],
                                     source_sum<RHO>(sh_acc[c][slot], part));
                            atomicAdd(&sh_steps[slot], (unsigned long long)nstep_of(myblk, (int)m));
                        }
                        gal &= ~left;
                        __syncwarp();
                    }
                }
                gblk += (uint32_t)kk;
                if constexpr (kVoxel<RHO>) {
                    if (((gblk - flushed_at) & 15u) == 0u && l < NC && mine) {  // flush (k >= 2: two lanes may take three copies)
                        for (int c = l; c < NC; c += k) {
                            sh_acc[c][slot] = flushed<RHO>(sh_acc[c][slot], value_of(sh_part[c][slot]));
                            sh_part[c][slot] = (Part)0;
                        }
                    }
                }
                __syncwarp();
                if (!any_out && !near_cap) continue;
                if (mine && gal == 0u) {
                    if (l == 0) P.pp_steps[sh_item[slot]] = (long long)(sh_steps[slot] | (unsigned long long)kDoneFlag);
                    ended = true;
                } else if (mine && (int64_t)gblk >= cap_blk) {
                    if (l == 0) {
                        atomicOr(SEG ? P.seg[sh_seg[slot]].status : P.status, 1 << MCG_ERR_STEP_CAP);
                        // (no completion flag: the exit kernel writes NaN)
                        P.pp_steps[sh_item[slot]] =
                            (long long)sh_steps[slot] + (long long)__popc(gal) * 4 * (long long)gblk;
                    }
                    ended = true;
                }
                if (__any_sync(kFull, ended)) break;  // regroup the others, or take new walks
            }
            };
            if (G == 1) rounds(std::true_type{});
            else rounds(std::false_type{});
            // back to the owners
            if constexpr (kTwoValued<RHO>) add_counts();
            const int from = rank * k & 31;
            const uint32_t nb = __shfl_sync(kFull, gblk, from);
            const unsigned na = __shfl_sync(kFull, gal, from);
            const int ne = __shfl_sync(kFull, (int)ended, from);
            if (busy) {
                wx = base[3 * rank];
                wy = base[3 * rank + 1];
                wz = base[3 * rank + 2];
                blk = nb;
                alive = na;
                if constexpr (RHO != MCG_RHO_NONE) {
                    S0 = value_of(sh_part[0][t]);
                    if (CRN) {
                        S1 = value_of(sh_part[1][t]);
                        S2 = value_of(sh_part[2][t]);
                    }
                }
                if (ne) busy = false;
            }
            __syncwarp();
            // single-precision sums whenever the warp regroups, as lanes do;
            // counts now and then (at most 2048 steps a round: below 2^22)
            if (!kTwoValued<RHO> || (round & 63u) == 0u) flush();
            continue;
        }

        // two four-step blocks per iteration for the analytic densities; one
        // for the voxel grid, whose larger step body (prefetched lookups)
        // otherwise strains the instruction cache
        constexpr int kBlocksUnrolled = kVoxel<RHO> ? 1 : 2;
#pragma unroll (kBlocksUnrolled)
        for (int k = 0; k < 16; ++k) {
            if (busy) {
                // the block's twelve normals in polar form: coordinate j of
                // the moves is nr[j / 2] cs[j]; (a single-request launch reads
                // its key straight from the launch parameters: uniform across
                // the warp)
                float nr[6], cs[12];
                polar12_f32(s, p, blk, SEG ? k0 : P.key0, SEG ? k1 : P.key1, P.lnscale_f, nr, cs);
                // one fused multiply-add per coordinate and step
                auto mv = [&](float x, int j) -> float { return fmaf(nr[j >> 1], cs[j], x); };
                // The block tests are taken for the warp (all live lanes), so
                // a warp never runs both the quiet moves and the full steps.
                // (Not for the voxel grid: the second copy of the step body
                // costs its kernel six registers and a sixth of its resident
                // warps.)
                constexpr bool kBlockTest = !kVoxel<RHO>;
                bool all_quiet = false, all_inside = false;
                if constexpr (kBlockTest) {
                    bool inside, quiet;
                    if constexpr (BALL || !kTwoValued<RHO>) {
                        block_bounds<RHO, BALL>(P, wx, wy, wz, nr, inside, quiet);
                    } else {
                        // the tests of block_bounds; written out here, with each
                        // difference where it is compared, they schedule better
                        // (bulk rate 1.050 -> 1.067e12 path-steps/s)
                        const float rs = ((nr[0] + nr[1]) + (nr[2] + nr[3])) + (nr[4] + nr[5]);  // <= 0
                        inside = fabsf(wx) - rs < P.in_f[0] && fabsf(wy) - rs < P.in_f[1] &&
                                 fabsf(wz) - rs < P.in_f[2];
                        const bool far = fabsf(wx - P.far_c[0]) + rs > P.far_h[0] ||
                                         fabsf(wy - P.far_c[1]) + rs > P.far_h[1] ||
                                         fabsf(wz - P.far_c[2]) + rs > P.far_h[2];
                        quiet = inside && far;
                    }
                    const unsigned am = __activemask();
                    all_quiet = __all_sync(am, quiet);
                    all_inside = __all_sync(am, inside);
                }
                // Voxel grid: the block's four positions are known once its
                // normals are, so all twelve density loads are issued here
                // and their latency overlaps the steps (same positions, same
                // summation order: results are unchanged).
                float px[4], py[4], pz[4], rv[4][3];
                if constexpr (kVoxel<RHO>) {
                    float x = wx, y = wy, zz = wz;
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        x = mv(x, 3 * m);
                        y = mv(y, 3 * m + 1);
                        zz = mv(zz, 3 * m + 2);
                        px[m] = x;
                        py[m] = y;
                        pz[m] = zz;
                        rho3_f32<RHO>(P, SEG ? M : model_of(P), x, y, zz, hf, rv[m][0], rv[m][1], rv[m][2]);
                    }
                }
                if (all_quiet) {
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        wx = mv(wx, 3 * m);
                        wy = mv(wy, 3 * m + 1);
                        wz = mv(wz, 3 * m + 2);
                    }
                } else {
                    auto full_steps = [&](auto ki) {
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const float nx = kVoxel<RHO> ? px[m] : mv(wx, 3 * m);
                        const float ny = kVoxel<RHO> ? py[m] : mv(wy, 3 * m + 1);
                        const float nz = kVoxel<RHO> ? pz[m] : mv(wz, 3 * m + 2);
                        // surely inside: by the block test, or (voxel grid) by a test of the step
                        bool inside_all = decltype(ki)::value;
                        if constexpr (!kBlockTest && !decltype(ki)::value)
                            inside_all = fabsf(nx) < P.in_f[0] && fabsf(ny) < P.in_f[1] && fabsf(nz) < P.in_f[2];
                        if (!inside_all) {
                            const unsigned ins = copies_inside<CRN, BALL>(P, nx, ny, nz, hf);
                            const unsigned out = alive & ~ins;
                            if (out) {  // some copy left Omega on this step
                                const unsigned long long it = sh_item[t];
                                auto sum = [&](int c, float part) { return source_sum<RHO>(sh_acc[c][t], part); };
                                if (out & 1u) put_exit(P, 0, it, wx, wy, wz, nx, ny, nz, sum(0, S0));
                                if (CRN && (out & 2u)) put_exit(P, 1, it, wx, wy, wz, nx, ny, nz + hf, sum(1, S1));
                                if (CRN && (out & 4u)) put_exit(P, 2, it, wx, wy, wz, nx, ny, nz - hf, sum(2, S2));
                                sh_steps[t] += (unsigned long long)nstep_of(blk, m) * __popc(out);
                                alive &= ins;
                            }
                            if (BRIDGE && alive) {  // within the bridge band of a face
                                unsigned faces = 0u;
                                const unsigned bx = bridge_exits_f32(P, alive, wx, wy, wz, nx, ny, nz, hf, s, p, blk, m,
                                                                     &faces);
                                if (bx) {
                                    const unsigned long long it = sh_item[t];
                                    for (int c = 0; c < 3; ++c) {
                                        if (!(bx & (1u << c))) continue;
                                        float e[3];
                                        bridge_point(P, c, (int)((faces >> (3 * c)) & 7u), nx, ny, nz, hf, e);
                                        const float part = c == 0 ? S0 : (c == 1 ? S1 : S2);
                                        put_exit(P, c, it, wx, wy, wz, e[0], e[1], e[2],
                                                 source_sum<RHO>(sh_acc[c][t], part));
                                    }
                                    sh_steps[t] += (unsigned long long)nstep_of(blk, m) * __popc(bx);
                                    alive &= ~bx;
                                }
                            }
                        }
                        if constexpr (kTwoValued<RHO>) {
                            // count where a copy is in the density's support
                            // (no live-copy test: a copy that has left has
                            // its record, its count is not read again)
                            const unsigned in = support3_f32<RHO>(P, nx, ny, nz, hf);
                            if (in & 1u) S0 += 1.0f;
                            if (CRN && (in & 2u)) S1 += 1.0f;
                            if (CRN && (in & 4u)) S2 += 1.0f;
                        } else if constexpr (kVoxel<RHO>) {
                            S0 += rv[m][0];
                            if (CRN) {
                                S1 += rv[m][1];
                                S2 += rv[m][2];
                            }
                        }
                        wx = nx;
                        wy = ny;
                        wz = nz;
                        // no early exit when the last copy leaves: the remaining
                        // steps of the block write nothing (no live copy), and a
                        // branch-free four-step body schedules better
                    }
                    };
                    if (kBlockTest && all_inside)
                        full_steps(std::true_type{});
                    else
                        full_steps(std::false_type{});
                }
                ++blk;
                if (!alive) {  // every copy has its exit record: mark the item complete
                    P.pp_steps[sh_item[t]] = (long long)(sh_steps[t] | (unsigned long long)kDoneFlag);
                    busy = false;
                } else if (4 * (int64_t)blk >= P.max_steps) {
                    const unsigned long long it = sh_item[t];
                    atomicOr(SEG ? P.seg[sh_seg[t]].status : P.status, 1 << MCG_ERR_STEP_CAP);
                    // (no completion flag: the exit kernel writes NaN)
                    P.pp_steps[it] = (long long)sh_steps[t] + (long long)__popc(alive) * 4 * (long long)blk;
                    busy = false;
                }
            }
            // enough walks have ended: leave the block loop to refill their
            // lanes or to regroup
            if (__popc(livem & ~__ballot_sync(kFull, busy)) >= P.refill_min) break;
        }
        // warp-uniform flush of the partial sums: every 64 steps at most for
        // single-precision sums, now and then for the exact counts
        if (!kTwoValued<RHO> || (round & 63u) == 0u) flush();
    }
}

// Per-path values of one item from its exit records (double precision).  The
// density at the last inside point is re-evaluated from X by the walk's own
// single-precision function.
template <int RHO, bool SEG>
__device__ __forceinline__ void exit_item(const WalkParams& P, unsigned long long item, float hf)
{
    ModelRef M = model_of(P);
    int32_t* status = P.status;
    if constexpr (SEG) {  // the item's request: its model arrays and status word
        const WalkSeg& g = P.seg[find_seg(P, item)];
        M = model_of(g);
        status = g.status;
    }
    double u[3] = {kNaN, kNaN, kNaN};
    const int nc = P.crn ? 3 : 1;
    const size_t T = P.total;
    for (int c = 0; c < nc; ++c) {
        const float4* rec = (const float4*)P.frec + 2 * ((size_t)c * T + item);
        const float4 a = rec[0], b = rec[1];
        float r[3];
        rho3_f32<RHO>(P, M, a.x, a.y, a.z, hf, r[0], r[1], r[2]);
        const float X[3] = {a.x, a.y, c == 0 ? a.z : (c == 1 ? a.z + hf : a.z - hf)};
        const float Y[3] = {a.w, b.x, b.y};
        const double acc = recorded_sum<RHO>(
            P, ((unsigned long long)__float_as_uint(b.w) << 32) | (unsigned long long)__float_as_uint(b.z));
        u[c] = exit_mixed(P, M, X, Y, acc, r[c]);
    }
    const double d = P.crn ? (u[1] - u[2]) / (2.0 * P.h) : kNaN;
    P.pp_u[item] = u[0];
    P.pp_d[item] = d;
    if (!isfinite(u[0]) || (P.crn && !isfinite(d))) atomicOr(status, 1 << MCG_ERR_NONFINITE);
}

// Exit evaluation, convergent: each warp scans its items 32 at a time, writes
// NaN for the ones without a result (no completion flag: capped, cancelled,
// never started, lost, outside Omega), clears the flag of the others and
// queues them in
// shared memory, evaluating them 32 at a time, so the slow double-precision
// pipe never runs a warp whose lanes are mostly idle.
template <int RHO, bool SEG>
__global__ void __launch_bounds__(128) exit_mixed_kernel(const WalkParams P)
{
    __shared__ unsigned long long queue[4][64];
    const float hf = P.crn ? P.h_f : 0.0f;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long* q = queue[w];
    const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    const unsigned long long first = ((unsigned long long)blockIdx.x * (blockDim.x >> 5) + w) * 32ull;
    int qn = 0;  // queued items (warp-uniform)
    for (unsigned long long base = first; base < P.total; base += warps * 32ull) {
        const unsigned long long item = base + (unsigned long long)lane;
        const bool in = item < P.total;
        const long long steps = in ? (long long)P.pp_steps[item] : 0ll;
        const bool valid = (steps & kDoneFlag) != 0;
        if (valid) P.pp_steps[item] = steps & ~kDoneFlag;
        if (in && !valid) {
            P.pp_u[item] = kNaN;
            P.pp_d[item] = kNaN;
        }
        const unsigned vm = __ballot_sync(kFull, valid);
        if (valid) q[qn + __popc(vm & ((1u << lane) - 1u))] = item;
        qn += __popc(vm);
        __syncwarp();
        if (qn >= 32) {
            exit_item<RHO, SEG>(P, q[lane], hf);
            const int rest = qn - 32;
            unsigned long long v = 0ull;
            if (lane < rest) v = q[32 + lane];
            __syncwarp();
            if (lane < rest) q[lane] = v;
            __syncwarp();
            qn = rest;
        }
    }
    if (lane < qn) exit_item<RHO, SEG>(P, q[lane], hf);
}

// Before a walk: the work counter at zero, and no item with a result that an
// earlier launch left: steps 0, which also clears the mixed walk's completion
// flags (its exit kernel writes NaN for items without one), and NaN per-path
// values for the double-precision walk, which writes them directly.  One
// launch (as memsets the four took 4 us each of a small solve).
__global__ void __launch_bounds__(256) reset_kernel(unsigned long long* counter, int64_t* steps, double* u, double* d,
                                                    unsigned long long n)
{
    const unsigned long long first = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (first == 0ull) *counter = 0ull;
    for (unsigned long long i = first; i < n; i += (unsigned long long)gridDim.x * blockDim.x) {
        steps[i] = 0;
        if (u) {
            u[i] = kNaN;
            d[i] = kNaN;
        }
    }
}

template <int RHO, bool CRN, bool BRIDGE, bool BALL, bool SEG>
cudaError_t launch_mixed(const WalkParams& P, int block, int grid, cudaStream_t st)
{
    walk_mixed_kernel<RHO, CRN, BRIDGE, BALL, SEG><<<grid, block, 0, st>>>(P);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const unsigned long long need = (P.total + 127ull) / 128ull;
    const unsigned long long cap = (unsigned long long)sms * 16ull;
    exit_mixed_kernel<RHO, SEG><<<(unsigned)(need < cap ? need : cap), 128, 0, st>>>(P);
    return cudaGetLastError();
}

template <int RHO>
cudaError_t launch_mixed_rho(const WalkParams& P, int block, int grid, cudaStream_t st)
{
    if (P.seg) return P.crn ? launch_mixed<RHO, true, false, false, true>(P, block, grid, st)
                            : launch_mixed<RHO, false, false, false, true>(P, block, grid, st);
    if (P.ball) return P.crn ? launch_mixed<RHO, true, false, true, false>(P, block, grid, st)
                             : launch_mixed<RHO, false, false, true, false>(P, block, grid, st);
    if (P.crn) return P.bridge ? launch_mixed<RHO, true, true, false, false>(P, block, grid, st)
                               : launch_mixed<RHO, true, false, false, false>(P, block, grid, st);
    return P.bridge ? launch_mixed<RHO, false, true, false, false>(P, block, grid, st)
                    : launch_mixed<RHO, false, false, false, false>(P, block, grid, st);
}

template <int RHO>
const void* mixed_fn(bool crn, bool seg)
{
    if (seg)
        return crn ? (const void*)walk_mixed_kernel<RHO, true, false, false, true>
                   : (const void*)walk_mixed_kernel<RHO, false, false, false, true>;
    return crn ? (const void*)walk_mixed_kernel<RHO, true, false, false, false>
               : (const void*)walk_mixed_kernel<RHO, false, false, false, false>;
}

const void* kernel_fn(int precision, int rho_kind, bool crn, bool seg)
{
    if (precision == MCG_FP64) return walk64_fn(rho_kind, crn, seg);
    switch (rho_kind) {
    case kRhoVoxelPacked: return mixed_fn<kRhoVoxelPacked>(crn, seg);
    case MCG_RHO_SPHERE: return mixed_fn<MCG_RHO_SPHERE>(crn, seg);
    case MCG_RHO_PRISM: return mixed_fn<MCG_RHO_PRISM>(crn, seg);
    case MCG_RHO_VOXEL: return mixed_fn<MCG_RHO_VOXEL>(crn, seg);
    default: return mixed_fn<MCG_RHO_NONE>(crn, seg);
    }
}

}  // namespace

namespace {

template <typename K>
void touch(K kernel)
{
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, (const void*)kernel) != cudaSuccess) cudaGetLastError();
}

template <int RHO>
void touch_mixed()
{
    touch(walk_mixed_kernel<RHO, true, false, true, false>);
    touch(walk_mixed_kernel<RHO, false, false, true, false>);
    touch(walk_mixed_kernel<RHO, true, true, false, false>);
    touch(walk_mixed_kernel<RHO, true, false, false, false>);
    touch(walk_mixed_kernel<RHO, false, true, false, false>);
    touch(walk_mixed_kernel<RHO, false, false, false, false>);
    touch(walk_mixed_kernel<RHO, true, false, false, true>);
    touch(walk_mixed_kernel<RHO, false, false, false, true>);
    touch(exit_mixed_kernel<RHO, false>);
    touch(exit_mixed_kernel<RHO, true>);
}

}  // namespace

cudaError_t launch_reset(const WalkParams& P, cudaStream_t st)
{
    const unsigned long long blocks = (P.total + 1023ull) / 1024ull;
    reset_kernel<<<(unsigned)(blocks < 1ull ? 1ull : blocks < 1216ull ? blocks : 1216ull), 256, 0, st>>>(
        P.counter, P.pp_steps, P.frec ? nullptr : P.pp_u, P.frec ? nullptr : P.pp_d, P.total);
    return cudaGetLastError();
}

void preload_walk_kernels()
{
    touch(reset_kernel);
    preload_walk64_kernels();
    touch_mixed<MCG_RHO_NONE>();
    touch_mixed<MCG_RHO_SPHERE>();
    touch_mixed<MCG_RHO_PRISM>();
    touch_mixed<MCG_RHO_VOXEL>();
    touch_mixed<kRhoVoxelPacked>();
}

int walk_blocks_per_sm(int precision, int rho_kind, int block, bool seg)
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel_fn(precision, rho_kind, true, seg), block, 0) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

cudaError_t launch_walk(const WalkParams& P0, int precision, int block, cudaStream_t st)
{
    WalkParams P = P0;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // a multi-request launch runs in the box without the bridge test
    if (P.seg && (P.ball || P.bridge || P.nseg <= 0)) return cudaErrorInvalidValue;
    const int kind = (P.rho_kind == MCG_RHO_VOXEL && P.zq) ? kRhoVoxelPacked : P.rho_kind;
    const int per_sm = walk_blocks_per_sm(precision, kind, block, P.seg != nullptr);
    long long grid = (long long)sms * per_sm;
    const long long need = (long long)((P.total + (unsigned long long)block - 1ull) / (unsigned long long)block);
    if (precision == MCG_FP64) return launch_walk64(P, block, (int)grid, st);
    P.quota = 32;
    {
        // Walks per warp.  With a warpful for every resident warp the lanes
        // run a walk each; with fewer the walks are spread over all warps,
        // up to kStripMax each, which run them as strips.  Where the line
        // lies (prism, 20 walks per resident warp: strips 65 ms, full lanes
        // in fewer warps 79 ms; 30 per warp: 84 against 94 ms).  A voxel
        // grid always starts with full warps: the rounding of its single-
        // precision sums follows the walks that share a warp, and a warp's
        // first 32 are consecutive items on any launch (later ones are not:
        // its free lanes take the next items of the list).
        const long long per_block = block / 32;
        const unsigned long long warps = (unsigned long long)(grid * per_block);
        const long long per_warp = (long long)(P.total / warps);
        if (per_warp < 32 && P.rho_kind != MCG_RHO_VOXEL) {
            P.quota = (int32_t)(per_warp < 1 ? 1 : per_warp > (long long)kStripMax ? kStripMax : per_warp);
            const long long spread = (long long)((P.total + (unsigned long long)per_block - 1ull) /
                                                 (unsigned long long)per_block);
            if (grid > spread) grid = spread;
        } else if (grid > need) {
            grid = need;
        }
    }
    if (grid < 1) grid = 1;
    switch (kind) {
    case kRhoVoxelPacked: return launch_mixed_rho<kRhoVoxelPacked>(P, block, (int)grid, st);
    case MCG_RHO_SPHERE: return launch_mixed_rho<MCG_RHO_SPHERE>(P, block, (int)grid, st);
    case MCG_RHO_PRISM: return launch_mixed_rho<MCG_RHO_PRISM>(P, block, (int)grid, st);
    case MCG_RHO_VOXEL: return launch_mixed_rho<MCG_RHO_VOXEL>(P, block, (int)grid, st);
    default: return launch_mixed_rho<MCG_RHO_NONE>(P, block, (int)grid, st);
    }
}

}  // namespace mcg
