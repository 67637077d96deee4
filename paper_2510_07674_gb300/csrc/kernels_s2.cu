// Stage-2 kernels: the fused trajectory optimisation (a group of 8, 4 or 2 warps per particle,
// every iteration inside one launch).  The lift that initialises it is in kernels_lift.cu.
#include <algorithm>

#include <cuda_fp16.h>

#include "launch_s2.h"
#include "stage1.cuh"
#include "stage2.cuh"

namespace spasm {

// ================================================================================== trajopt
constexpr int kTWarps = 8;                // warps of a trajectory CTA
constexpr int kTThreads = 32 * kTWarps;
constexpr int kChunkGroups = 8;           // 32-chunk groups of the chunk lists (kMaxC configurations)
constexpr int kSlots = 2;   // sphere items per lane: up to 56 robot + 8 held-block spheres

constexpr int kChunk = 4;   // configurations whose kinematics one warp evaluates together

// A trajectory CTA of 8 warps runs 1, 2 or 4 particles at once: each on its own group of 8, 4 or
// 2 warps, with its own region of dynamic shared memory and its own named barrier 1 + group.
// With one particle the group is the whole CTA.  An evaluation has a serial chain of phases that
// keep one or two warps busy (grasp and place frames, placed poses, placement gradient) and a
// queue of a dozen coarse items, so the fewer warps a particle has the less they wait for one
// another; two CTAs per SM (the registers' limit) overlap 2, 4 or 8 particles' chains.  One
// particle of 8 warps finishes sooner, so it takes launches that would not fill the SMs
// otherwise; the rule is traj_auto_ppc's.
template <int kPpc>
constexpr int kGrpWarps = kTWarps / kPpc;
template <int kPpc>
constexpr int kGrpThreads = kTThreads / kPpc;
template <int kPpc>
__device__ __forceinline__ int grp_tid() { return kPpc == 1 ? (int)threadIdx.x : (int)(threadIdx.x & (kGrpThreads<kPpc> - 1)); }
template <int kPpc>
__device__ __forceinline__ int grp_index() { return kPpc == 1 ? 0 : (int)(threadIdx.x / kGrpThreads<kPpc>); }
template <int kPpc>
__device__ __forceinline__ void grp_sync() {
    if (kPpc == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + grp_index<kPpc>()), "n"(kGrpThreads<kPpc>) : "memory");
}

// Cached cull.  When no sphere of a chunk penetrates a static obstacle (the environment, blocks
// at their initial poses), its cull and tests also return the chunk's static clearance: the
// smallest separation (largest per-axis gap) between any of its link boxes and any static box
// that could touch it, and for the obstacles its spheres were tested against the smallest
// sphere-level gap of those tests.  The same for the placed blocks, which move: the top one (the
// highest block placed before the chunk's last block) on its own, the ones below it together.
// Later iterations skip the static half while the bound on how far the chunk's spheres moved
// since stays below the static clearance, and the moving half while that bound plus the top
// block's own motion since stays below the clearance to it, and plus a bound on how far any one
// of the blocks below the top one moved below the clearance to those: the skipped work is exactly
// work whose result is zero.  A chunk with both halves skipped needs no kinematics; one with one
// half evaluated again keeps the other's clearance less the motion so far.  (Most chunks that
// have to be looked at again have come due for the placed blocks' motion alone, which leaves one
// word of boxes to cull.)
// A chunk's state byte: how many of its configurations had a candidate when it was last evaluated,
// the halves that this evaluation may skip, the halves without a penetration.
constexpr int kStateCand = 7, kStateSkipStatic = 16, kStateSkipMoving = 32, kStateZeroStatic = 64, kStateZeroMoving = 128;
constexpr int kStateZero = kStateZeroStatic | kStateZeroMoving;
constexpr float kClearSlack = 1e-5f;   // FP32 rounding of the boxes, metres

// Work queue of an evaluation: its items (the chunks, the residual jobs, the slices of the
// placed tower's collisions) go to the warps in list order from a shared counter, the larger
// items first, so that the warps finish together.  What the items add up goes into fixed-point
// accumulators (integer sums are exact, hence independent of which warp took which item and
// when): a value v becomes round(v 2^40), |v| < 8e6.
constexpr float kFix = 1099511627776.f;   // 2^40
__device__ __forceinline__ void fx_add(long long* acc, float v) {
    atomicAdd(reinterpret_cast<unsigned long long*>(acc), (unsigned long long)__float2ll_rn(v * kFix));
}
__device__ __forceinline__ float fx_value(long long a) { return __ll2float_rn(a) * (1.f / kFix); }
constexpr int kPlaceUnits = (8 * kMaxB + 31) / 32;   // slices of 32 block spheres of the placed tower
constexpr int kResidualJobs = 1;                      // the placement residuals

// The obstacles of the cull, in words of 32 boxes (padded with empty ones): the environment's
// cuboids, its spheres, then one word of blocks, bit k the placed block k and bit 16 + k block k
// at its initial pose.
__host__ __device__ inline int t_cub_words(int n_cub) { return (n_cub + 31) >> 5; }
__host__ __device__ inline int t_words(int n_cub, int n_osph) { return t_cub_words(n_cub) + ((n_osph + 31) >> 5) + 1; }
constexpr int kMaxWords = kMaxCub / 32 + kMaxOSph / 32 + 1;
static_assert(2 * kMaxB == 32, "one word of blocks");

struct TWarp {
    float4 F[kChunk][8][3];  // frames 0..7 of each configuration of the chunk: rows (R_i0, R_i1, R_i2, o_i)
    float4 H[kChunk][3];     // held-block frame of each configuration (same row layout)
    uint32_t mask[kChunk][kMaxWords];   // obstacles that may touch configuration c of the chunk
    float4 edge[3][2];       // traj_step: the first and last rows of this warp's run, and the last of its previous 32
    float maxpen;            // this warp's largest penetration
    unsigned long long count[3];        // this warp's tests, configurations culled, and with a candidate
};

// What the epilogue needs of a grasp or place configuration's frames: row r of joint k's axis
// and origin, Z[k][r] = (z_r, o_r), and the held-block frame.
struct SpecialFrames {
    float4 H[3];
    float2 Z[7][3];
    float2 pad;
};

struct TShared {
    float4 blk[2 * kMaxB][4];   // block cuboids: k placed this iteration, 16 + k at the initial pose
    float4 bbox[2 * kMaxB][2];  // their axis-aligned boxes (lo, hi): the word of blocks
    float pose[4 * kMaxB];   // placed poses (x, y, z, yaw)
    float g4[4 * kMaxB];     // dL/d(placed pose)
    float h[kMaxNR], lam[kMaxNR], s[kMaxNR];
    float rpt[2 * kMaxB][6];           // (w_roll, w_pitch) of the block frame at special configuration e
                                       // (2 b: grasp of block b, 2 b + 1: place)
    float pg[kMaxB][4];                // dC_coll/d(placed pose j), sphere side (from the slice holding block j)
    float pgc[kPlaceUnits][kMaxB][4];  // dC_coll/d(placed pose i), cuboid side of block pairs, per slice
    float pcu[kPlaceUnits][2];         // per slice: sum and maximum of the tower's penetrations
    long long fx_wr[2][kMaxB][4];      // d/d(placed pose k) of the arm and block groups (fixed point)
    long long fx_tot[2];               // C_arm, C_block (fixed point)
    int next;                          // the work queue's counter
    StackScratch ps;
    float4 dh[8];            // joint j: cos alpha, sin alpha, a, d (per-lane reads in the kinematics)
    float th0[8];            // joint offsets
    float4 lbc[8], lbh[8];   // link-frame boxes of each link's spheres (centre, half extents)
    float mu, L, inv_S;
    float inv_above[kMaxB];       // 1 / (blocks above block k)
    float pose_prev[4 * kMaxB];   // placed poses of the previous evaluation
    // chunks to evaluate by tier (kChunk .. 1 configurations with candidates at the last cull, then the
    // candidate-free ones to cull again)
    union {
        unsigned char active[kChunk + 1][(kMaxC + kChunk - 1) / kChunk];
        float4 partial[2 * kMaxB][2];   // traj_step: the special configurations' gradients without their own rows
    };
    int n_tier[kChunk + 1];       // their counts
    unsigned hit[kMaxC / 32];     // bit t - 1: configuration t has gradient rows this evaluation
    float blk_cum[kMaxB];         // [k]: sum over the evaluations of the largest motion among the placed blocks 0..k
    float bown[kMaxB];            // [k]: sum over the evaluations of placed block k's own motion
    int pose_prev_ok;
    float c_arm, c_blk, maxpen, c_coll, c_stable, c_height, c_start;
    float max_start, max_tilt, pm_pen, pm_D, pm_dz, path, jl;
    float part[kTWarps][2];       // path length and joint-limit sums, a partial per 32 threads of 256
    int particle;                 // the particle the group works on
};

// The environment of a problem: barrier words, cuboids, spheres, their boxes.
__host__ __device__ inline size_t t_env_offset() { return 16; }
__host__ __device__ inline size_t t_aabb_offset(int n_cub, int n_osph) {
    return (16 + (size_t)n_cub * 64 + (size_t)n_osph * 16 + 15) & ~(size_t)15;
}
__host__ __device__ inline size_t t_env_bytes(int n_cub, int n_osph) {
    return (t_aabb_offset(n_cub, n_osph) + (size_t)(t_words(n_cub, n_osph) - 1) * 32 * 32 + 127) & ~(size_t)127;
}
// The region of a particle group.
__host__ __device__ inline size_t t_warp_offset() { return (sizeof(TShared) + 15) & ~(size_t)15; }
__host__ __device__ inline size_t t_q_offset(int warps) { return t_warp_offset() + (size_t)warps * sizeof(TWarp); }
__host__ __device__ inline size_t t_sp_offset(int C, int warps) { return t_q_offset(warps) + (size_t)C * 8 * sizeof(float); }
__host__ __device__ inline int t_n_chunks(int C) { return (C - 1 + kChunk - 1) / kChunk; }
// cached cull state: per configuration the motion bound since its chunk's last cull; per
// chunk, at that cull, the motion bound of the placed blocks below its top block and the top
// block's own motion, its (static, moving) clearances as an fp16 pair, its fp16 clearance to
// the top block and its state (kState*)
__host__ __device__ inline size_t t_cache_offset(int C, int B, int warps) {
    return (t_sp_offset(C, warps) + (size_t)2 * B * sizeof(SpecialFrames) + 15) & ~(size_t)15;
}
// Shared memory of one particle's group, rounded to 128 bytes.  The gradient rows of the collision groups are not in
// it: only the chunks with a penetration have any (4 of 155 per evaluation on the 10-block
// tower), so they go to the launch's scratch in global memory (TrajIO::rows), which stays in L2;
// two row buffers here would cost 40 of the region's then 95 KB.
static size_t t_region(int C, int B, int ppc) {
    return (t_cache_offset(C, B, kTWarps / ppc) + (size_t)C * sizeof(float) +
            (size_t)t_n_chunks(C) * (3 * sizeof(float) + sizeof(__half) + sizeof(unsigned char)) + 127) &
           ~(size_t)127;
}

// The collision gradient rows of one particle, as the tail of its region in a launch without scratch.
__host__ __device__ inline size_t t_rows_bytes(int C) { return ((size_t)C * 16 * sizeof(float) + 127) & ~(size_t)127; }

size_t traj_cta_smem_bytes(const TrajScalars& sc, int ppc, bool batched) {
    const size_t env = t_env_bytes(sc.n_cub, sc.n_osph);
    return (batched ? ppc : 1) * env + ppc * t_region(sc.C, sc.B, ppc);
}

int traj_slots(int B, int C, int n_cub, int n_osph) {
    return t_env_bytes(n_cub, n_osph) + 4 * t_region(C, B, 4) <= kHalfSmem ? 2 * kTrajSlots : kTrajSlots;
}

// Sphere item held in slot k by a lane: strided tiling, item lane + 32 k (the spheres of a link
// spread over neighbouring lanes), or blocked tiling, item kSlots lane + k (a lane's spheres are
// neighbours, mostly on one link).  Either covers 64 items; the choice reorders the per-lane
// sums only.
template <int kTile>
__device__ __forceinline__ int slot_item(int lane, int k) {
    return kTile ? kSlots * lane + k : lane + 32 * k;
}

// x / S for 0 <= x < 2 kMaxC by the reciprocal inv_S = 1 / S: exact, as x + 1/2 is at least 1/2 away
// from a multiple of S and the product's rounding is below 1e-3 of that distance.
__device__ __forceinline__ int div_steps(int x, float inv_S) { return (int)(((float)x + 0.5f) * inv_S); }

// The robot spheres a lane owns (slot_item), loaded once per kernel launch: link-frame centre,
// radius, link index.  Items beyond the robot spheres are the held block's.
struct LaneSpheres {
    float lx[kSlots], ly[kSlots], lz[kSlots], r[kSlots];
    int link[kSlots];
};

template <int kTile>
__device__ __forceinline__ LaneSpheres lane_spheres(const Scalars& sc) {
    const int lane = threadIdx.x & 31;
    LaneSpheres ls;
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
        const int it = slot_item<kTile>(lane, k);
        if (it < sc.n_rsph) {
            const float4 v = sc.rsph[it];
            ls.lx[k] = v.x; ls.ly[k] = v.y; ls.lz[k] = v.z; ls.r[k] = v.w;
            ls.link[k] = sc.rlink[it];
        } else {
            ls.lx[k] = ls.ly[k] = ls.lz[k] = ls.r[k] = 0.f;
            ls.link[k] = 7;
        }
    }
    return ls;
}

// Forward kinematics of four configurations by one warp: lane 8c + k holds link transform
// k of configuration t_c (k = 0: identity), and a 3-level inclusive scan of affine products
// inside each group of 8 lanes gives frame_k = T_1 ... T_k.  Group c writes its frames (rows
// (R_i0, R_i1, R_i2, o_i)) to F_c, or only the joints' axes and origins to Z_c when that is
// given, unless `write` is false for that group, and, when
// `want_h`, the frame of block b held by the tool to H_c.  With `box`,
// the lane also returns a world box (lo xyz, hi xyz) that holds every sphere of link k (and of
// the held block, at k = 7 with `want_h`): the link-frame box of those spheres carried by the
// frame, i.e. centre R c + o and half extents |R| h.
template <bool kP2P>
__device__ __forceinline__ void chunk_fk(const TrajScalars& sc, const TShared& sh, const float* __restrict__ q, int t_c, int b,
                                         bool write, bool want_h, float4 (*F_c)[3], float2 (*Z_c)[3], float4* H_c,
                                         float* box) {
    const int lane = threadIdx.x & 31;
    const int k = lane & 7;
    const int t = t_c;
    float A[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1}, bv[3] = {0, 0, 0};
    if (k > 0) {
        const int j = k - 1;
        float st, ct;
        sincosf(sh.th0[j] + q[t * 8 + j], &st, &ct);
        const float4 row = sh.dh[j];
        const float ca = row.x, sa = row.y;
        A[0] = ct;      A[1] = -st;     A[2] = 0.f;
        A[3] = ca * st; A[4] = ca * ct; A[5] = -sa;
        A[6] = sa * st; A[7] = sa * ct; A[8] = ca;
        bv[0] = row.z; bv[1] = -sa * row.w; bv[2] = ca * row.w;
    }
#pragma unroll(kP2P ? 3 : 1)
    for (int off = 1; off < 8; off <<= 1) {
        float L[9], lb[3];
#pragma unroll
        for (int i = 0; i < 9; ++i) L[i] = __shfl_up_sync(0xffffffffu, A[i], off, 8);
#pragma unroll
        for (int i = 0; i < 3; ++i) lb[i] = __shfl_up_sync(0xffffffffu, bv[i], off, 8);
        if (k >= off) {
            float nA[9], nb[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
#pragma unroll
                for (int cc = 0; cc < 3; ++cc)
                    nA[3 * r + cc] = L[3 * r] * A[cc] + L[3 * r + 1] * A[3 + cc] + L[3 * r + 2] * A[6 + cc];
                nb[r] = L[3 * r] * bv[0] + L[3 * r + 1] * bv[1] + L[3 * r + 2] * bv[2] + lb[r];
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) A[i] = nA[i];
#pragma unroll
            for (int i = 0; i < 3; ++i) bv[i] = nb[i];
        }
    }
    if (box) {
        const float4 lc = sh.lbc[k], lh = sh.lbh[k];
        const bool has = lh.x >= 0.f;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float w = A[3 * r] * lc.x + A[3 * r + 1] * lc.y + A[3 * r + 2] * lc.z + bv[r];
            const float e = fabsf(A[3 * r]) * lh.x + fabsf(A[3 * r + 1]) * lh.y + fabsf(A[3 * r + 2]) * lh.z;
            box[r] = has ? w - e : 3.4e38f;
            box[3 + r] = has ? w + e : -3.4e38f;
        }
    }
    if (!write) return;
    if (Z_c) {
        if (k > 0)
#pragma unroll
            for (int r = 0; r < 3; ++r) Z_c[k - 1][r] = make_float2(A[3 * r + 2], bv[r]);
    } else {
#pragma unroll
        for (int r = 0; r < 3; ++r) F_c[k][r] = make_float4(A[3 * r], A[3 * r + 1], A[3 * r + 2], bv[r]);
    }
    if (k == 7 && want_h) {
        float Rt[9], pt[3], Rb[9], pb[3];
        tool_frame<float>(sc, A, bv, Rt, pt);
        held_block<float>(sc, b, Rt, pt, Rb, pb);
#pragma unroll
        for (int r = 0; r < 3; ++r) H_c[r] = make_float4(Rb[3 * r], Rb[3 * r + 1], Rb[3 * r + 2], pb[r]);
        if (box) {
            // held-block spheres sit at (+-hx/2, +-hy/2, +-hz/2) with radius r_b in the block frame
            const float4 hb = sc.half[b];
            const float ex = 0.5f * hb.x + hb.w + 1e-5f, ey = 0.5f * hb.y + hb.w + 1e-5f, ez = 0.5f * hb.z + hb.w + 1e-5f;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const float e = fabsf(Rb[3 * r]) * ex + fabsf(Rb[3 * r + 1]) * ey + fabsf(Rb[3 * r + 2]) * ez;
                box[r] = fminf(box[r], pb[r] - e);
                box[3 + r] = fmaxf(box[3 + r], pb[r] + e);
            }
        }
    }
}

// World centres of the lane's sphere items for one configuration (frames F, held-block
// frame H); items beyond the robot spheres are the held block's (transfer interior only).
template <int kTile>
__device__ __forceinline__ void sphere_centres(const TrajScalars& sc, const LaneSpheres& ls, const float4 (*F)[3],
                                               const float4* H, int n_items, int b, float* cx, float* cy, float* cz,
                                               float* rr, bool* act, bool* isblk) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
        const int it = slot_item<kTile>(lane, k);
        act[k] = it < n_items;
        isblk[k] = act[k] && it >= sc.n_rsph;
        float x = ls.lx[k], y = ls.ly[k], z = ls.lz[k];
        float4 r0, r1, r2;
        if (isblk[k]) {
            block_sphere_local(sc.half[b], it - sc.n_rsph, x, y, z);
            r0 = H[0]; r1 = H[1]; r2 = H[2];
            rr[k] = sc.half[b].w;
        } else {
            const int l = ls.link[k];
            r0 = F[l][0]; r1 = F[l][1]; r2 = F[l][2];
            rr[k] = act[k] ? ls.r[k] : 0.f;
        }
        cx[k] = r0.x * x + r0.y * y + r0.z * z + r0.w;
        cy[k] = r1.x * x + r1.y * y + r1.z * z + r1.w;
        cz[k] = r2.x * x + r2.y * y + r2.z * z + r2.w;
    }
}

// Collision terms of the configurations t0 .. t0+nc-1 (kinematics in the warp's frames),
// evaluated by one warp: arm spheres and, on the transfer interior, the held block's spheres
// against the environment and the context blocks.  An exact cull first keeps the obstacles
// whose boxes overlap the box of all spheres of the chunk (consecutive waypoints are close);
// per configuration lanes own sphere items, screen both slots branch-free and evaluate the
// penetration only where the separation test fails.  With `grad`, writes the unscaled group
// gradients of configuration t to rows[16 t ..] (arm group, then block group, 8 floats each)
// where it penetrates something, marks those in sh.hit and accumulates placed-pose derivatives.
// seg_l: the segment of configuration t0 + lane / 8.
// skip (kStateSkip*): the half (static obstacles, placed blocks) known to be clear of the chunk.
// Returns the halves without a penetration (kStateZero*); for those evaluated, `clearance` /
// `clearance_top` / `clearance_moving` bound from below how far any of the chunk's spheres is
// from a static box / the top placed block it could touch (the block below the chunk's last
// block) / the other placed blocks: the gaps between link boxes and the boxes apart from them,
// and the sphere-level gaps of the tests that ran.
// The environment and the blocks share one cull loop and one test loop, and the kernel keeps
// its other loops rolled: with four particles per SM in different phases the instruction cache
// is what the warps compete for.
template <bool kP2P, int kTile>
__device__ __forceinline__ int chunk_collisions(const TrajScalars& sc, const LaneSpheres& ls,
                                                 const float4* __restrict__ cub, const float4* __restrict__ osph,
                                                 const float4* aabb, TShared& sh, TWarp& tw, float* rows, int t0,
                                                 int nc, int seg_l, int skip, bool grad, const float* lane_box, float& acc_arm,
                                                 float& acc_blk, float& acc_max, int& n_cand, float& clearance,
                                                 float& clearance_moving, float& clearance_top) {
    const int lane = threadIdx.x & 31;
    const int S = sc.S;
    float cx[kSlots], cy[kSlots], cz[kSlots], rr[kSlots];
    bool act[kSlots], isblk[kSlots];

    // pass 1: box of every sphere of the chunk (union of the lanes' link boxes), candidate
    // obstacles by warp ballots
    const float lo_x = warp_fmin(lane_box[0]), lo_y = warp_fmin(lane_box[1]), lo_z = warp_fmin(lane_box[2]);
    const float hi_x = warp_fmax(lane_box[3]), hi_y = warp_fmax(lane_box[4]), hi_z = warp_fmax(lane_box[5]);
    // second level: each candidate of the chunk box against the lanes' own link boxes (lane
    // 8c + k: link k of configuration c); configuration c keeps the candidate when one of its
    // link boxes overlaps the candidate's box.  Both levels are exact: no sphere inside the
    // boxes is dropped.  Every box apart from the chunk box, or from a lane's link box, that
    // the lane's configuration could touch lowers the lane's clearance to that separation
    // (largest per-axis gap, > 0 iff the boxes are apart).
    const float* lb = lane_box;
    // link 0 (lane k = 0) is the fixed base: its gaps to static boxes (the environment, blocks
    // at their initial poses) never shrink and do not bound the clearance
    const bool moving_link = (lane & 7) != 0;
    // a configuration of block b's segments can touch the placed blocks k < b and the blocks
    // k > b still at their initial poses (the chunk: any of its configurations)
    const int b_lane = seg_l >> 1, b_first = __shfl_sync(0xffffffffu, b_lane, 0);
    const int b_last = __shfl_sync(0xffffffffu, b_lane, 8 * (nc - 1));
    auto context = [](int below, int above) {   // placed blocks k < below, initial poses k > above
        return ((1u << below) - 1u) | (0xfffe0000u << above);
    };
    const unsigned halves = (skip & kStateSkipStatic ? 0u : 0xffff0000u) | (skip & kStateSkipMoving ? 0u : 0x0000ffffu);
    const unsigned ctx_l = context(b_lane, b_lane) & halves, ctx_chunk = context(b_last, b_first) & halves;
    // the highest placed block a configuration of the chunk can touch: it moves by its own motion,
    // the blocks below it by at most the largest motion among them
    const int top = b_last - 1;
    const int n_cw = t_cub_words(sc.n_cub), n_w = t_words(sc.n_cub, sc.n_osph);
    // the words to look at; point to point has no blocks
    const int wd0 = skip & kStateSkipStatic ? n_w - 1 : 0, wd1 = kP2P ? n_w - 1 : n_w;
    float clear = 3.4e38f, clear_m = 3.4e38f;
    uint32_t any = 0u;
#pragma unroll 1
    for (int wd = wd0; wd < wd1; ++wd) {
        const bool blocks = !kP2P && wd == n_w - 1;
        const float4* box = blocks ? sh.bbox[0] : aabb + 64 * wd;
        const float4 clo = box[2 * lane], chi = box[2 * lane + 1];
        const float s1 = fmaxf(fmaxf(fmaxf(clo.x - hi_x, lo_x - chi.x), fmaxf(clo.y - hi_y, lo_y - chi.y)),
                               fmaxf(clo.z - hi_z, lo_z - chi.z));
        const float g1 = s1 > 0.f ? s1 : 3.4e38f;
        unsigned m = __ballot_sync(0xffffffffu, s1 <= 0.f);
        if (blocks) {
            m &= ctx_chunk;
            if ((ctx_chunk >> lane) & 1u) {
                if (lane >= kMaxB) clear = fminf(clear, g1);
                else if (lane != top) clear_m = fminf(clear_m, g1);
            }
        } else {
            clear = fminf(clear, g1);
        }
        uint32_t mine = 0u;
#pragma unroll 1
        while (m) {
            const int bit = __ffs(m) - 1;
            m &= m - 1;
            const float4 blo = box[2 * bit], bhi = box[2 * bit + 1];
            const float s2 = fmaxf(fmaxf(fmaxf(blo.x - lb[3], lb[0] - bhi.x), fmaxf(blo.y - lb[4], lb[1] - bhi.y)),
                                   fmaxf(blo.z - lb[5], lb[2] - bhi.z));
            // a box that overlaps this link's box is tested against the spheres, which give the gap
            const float g2 = s2 > 0.f ? s2 : 3.4e38f;
            if (blocks && bit < kMaxB) {
                if (bit < b_lane && bit != top) clear_m = fminf(clear_m, g2);
            } else if (moving_link && (!blocks || bit - kMaxB > b_lane)) {
                clear = fminf(clear, g2);
            }
            mine |= s2 <= 0.f ? 1u << bit : 0u;
        }
        if (blocks) mine &= ctx_l;
        mine |= __shfl_xor_sync(0xffffffffu, mine, 1);
        mine |= __shfl_xor_sync(0xffffffffu, mine, 2);
        mine |= __shfl_xor_sync(0xffffffffu, mine, 4);
        any |= mine;
        if ((lane & 7) == 0) tw.mask[lane >> 3][wd] = mine;
    }
    const unsigned has = __ballot_sync(0xffffffffu, any != 0u);   // bit 8c: configuration c has a candidate
    clearance = warp_fmin(clear);
    clearance_moving = kP2P ? 3.4e38f : warp_fmin(clear_m);
    {
        // the top block: the gap from each link box of the configurations it concerns
        float ct = 3.4e38f;
        if (!kP2P && top >= 0 && top < b_lane) {
            const float4 blo = sh.bbox[top][0], bhi = sh.bbox[top][1];
            const float g = fmaxf(fmaxf(fmaxf(blo.x - lb[3], lb[0] - bhi.x), fmaxf(blo.y - lb[4], lb[1] - bhi.y)),
                                  fmaxf(blo.z - lb[5], lb[2] - bhi.z));
            if (g > 0.f) ct = g;   // an overlapping box is tested against the spheres, which give the gap
        }
        clearance_top = kP2P ? 3.4e38f : warp_fmin(ct);
    }
    __syncwarp();

    // pass 2: every configuration against its candidates (without any, its collision terms and
    // their gradient are zero and the sphere centres are not needed), in the order of the words.
    // gap_s / gap_m / gap_t: the lane's smallest sphere-level gap (lower bound) to a tested static
    // box / placed block below the top one / the top placed block; the fixed base's spheres do not
    // move relative to static boxes and are left out of gap_s.
    n_cand = 0;
    unsigned hits = 0u;   // bit c: configuration c penetrates something
    bool hit_s = false, hit_m = false;
    int visits = 0;
    float gap_s = 3.4e38f, gap_m = 3.4e38f, gap_t = 3.4e38f;
    unsigned tests = 0u;
#pragma unroll 1
    for (int ci = 0; ci < nc; ++ci) {
        if (!((has >> (8 * ci)) & 1u)) continue;
        const int t = t0 + ci;
        const int seg = __shfl_sync(0xffffffffu, seg_l, 8 * ci);
        const int b = seg >> 1;
        const bool held = (seg & 1) && t - seg * S < S;
        const int n_items = sc.n_rsph + (held ? 8 : 0);
        ++n_cand;
        sphere_centres<kTile>(sc, ls, tw.F[ci], tw.H[ci], n_items, b, cx, cy, cz, rr, act, isblk);
        bool fixed[kSlots];
#pragma unroll
        for (int sl = 0; sl < kSlots; ++sl) fixed[sl] = !isblk[sl] && ls.link[sl] == 0;
        float gx[kSlots], gy[kSlots], gz[kSlots], pen_sum[kSlots];
#pragma unroll
        for (int sl = 0; sl < kSlots; ++sl) gx[sl] = gy[sl] = gz[sl] = pen_sum[sl] = 0.f;
        bool any_hit = false;
        visits = 0;

#pragma unroll 1
        for (int wd = wd0; wd < wd1; ++wd) {
            const bool blocks = !kP2P && wd == n_w - 1;
            unsigned m = tw.mask[ci][wd];
            visits += __popc(m);
#pragma unroll 1
            while (m) {
                const int bit = __ffs(m) - 1;
                m &= m - 1;
                if (wd >= n_cw && !blocks) {
                    const float4 os = osph[32 * (wd - n_cw) + bit];
#pragma unroll
                    for (int sl = 0; sl < kSlots; ++sl) {
                        if (!act[sl]) continue;
                        if (!fixed[sl]) {
                            // the largest per-axis offset bounds the centre distance from below
                            const float dm = fmaxf(fmaxf(fabsf(cx[sl] - os.x), fabsf(cy[sl] - os.y)), fabsf(cz[sl] - os.z));
                            gap_s = fminf(gap_s, fmaxf(dm - rr[sl] - os.w, 0.f));
                        }
                        float ax, ay, az;
                        const float pen = pen_sphere<float>(cx[sl], cy[sl], cz[sl], rr[sl], os, ax, ay, az);
                        if (pen > 0.f) {
                            any_hit = hit_s = true;
                            pen_sum[sl] += pen;
                            acc_max = fmaxf(acc_max, pen);
                            gx[sl] += ax; gy[sl] += ay; gz[sl] += az;
                        }
                    }
                    continue;
                }
                const bool placed = blocks && bit < kMaxB;
                const float4* rec = blocks ? sh.blk[bit] : cub + 4 * (32 * wd + bit);
                const float4 o0 = rec[0], o1 = rec[1], o2 = rec[2], o3 = rec[3];
                float d8[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // d/d(placed pose): arm, then held-block spheres
                bool hit = false;
                float p0[kSlots], p1[kSlots], p2[kSlots], q0[kSlots], q1[kSlots], q2[kSlots], qm[kSlots];
#pragma unroll
                for (int sl = 0; sl < kSlots; ++sl)
                    qm[sl] = cub_local<float>(cx[sl], cy[sl], cz[sl], o0, o1, o2, o3, p0[sl], p1[sl], p2[sl], q0[sl],
                                              q1[sl], q2[sl]);
                // separated along a box axis by qm: the sphere is at least qm - r from the box
                float g = 3.4e38f;
#pragma unroll
                for (int sl = 0; sl < kSlots; ++sl)
                    if (act[sl] && (placed || !fixed[sl])) g = fminf(g, fmaxf(qm[sl] - rr[sl], 0.f));
                if (!placed) gap_s = fminf(gap_s, g);
                else if (bit == top) gap_t = fminf(gap_t, g);
                else gap_m = fminf(gap_m, g);
#pragma unroll
                for (int sl = 0; sl < kSlots; ++sl) {
                    if (!act[sl] || !(qm[sl] < rr[sl])) continue;
                    float ax, ay, az;
                    const float pen = pen_finish<float>(p0[sl], p1[sl], p2[sl], q0[sl], q1[sl], q2[sl], qm[sl], rr[sl],
                                                        o1, o2, o3, ax, ay, az);
                    if (pen > 0.f) {
                        hit = true;
                        pen_sum[sl] += pen;
                        acc_max = fmaxf(acc_max, pen);
                        gx[sl] += ax; gy[sl] += ay; gz[sl] += az;
                        // rigid motion of the cuboid: d/dP = -g, d/dyaw = -((c - P) x g)_z
                        const float dyaw = -((cx[sl] - o0.x) * ay - (cy[sl] - o0.y) * ax);
                        if (isblk[sl]) { d8[4] -= ax; d8[5] -= ay; d8[6] -= az; d8[7] += dyaw; }
                        else { d8[0] -= ax; d8[1] -= ay; d8[2] -= az; d8[3] += dyaw; }
                    }
                }
                any_hit |= hit;
                if (placed) hit_m |= hit;
                else hit_s |= hit;
                if (grad && placed && __any_sync(0xffffffffu, hit)) {
                    const float d = warp_sums<8>(d8);   // lane 4 i: value i
                    if ((lane & 3) == 0) fx_add(&sh.fx_wr[lane >> 4][bit][(lane >> 2) & 3], d);
                }
            }
        }
        tests += (unsigned)visits * (unsigned)n_items;
#pragma unroll
        for (int sl = 0; sl < kSlots; ++sl) {
            if (isblk[sl]) acc_blk += pen_sum[sl];
            else acc_arm += pen_sum[sl];
        }
        if (!__any_sync(0xffffffffu, any_hit)) continue;
        hits |= 1u << ci;
        if (!grad) continue;

        // backward: dC/dq_k = sum_s z_k . ((c_s - o_k) x g_s) over spheres on links >= k
        auto torque = [&](int k, float& arm, float& blk) {
            const float4* f = tw.F[ci][k + 1];
            const float4 f0 = f[0], f1 = f[1], f2 = f[2];
            const float ox = f0.w, oy = f1.w, oz = f2.w;
            const float zx = f0.z, zy = f1.z, zz = f2.z;
#pragma unroll
            for (int sl = 0; sl < kSlots; ++sl) {
                const int lk = isblk[sl] ? 7 : ls.link[sl];
                if (!any_hit || !act[sl] || lk < k + 1) continue;
                const float vx = cx[sl] - ox, vy = cy[sl] - oy, vz = cz[sl] - oz;
                const float mm = zx * (vy * gz[sl] - vz * gy[sl]) + zy * (vz * gx[sl] - vx * gz[sl]) +
                                 zz * (vx * gy[sl] - vy * gx[sl]);
                if (isblk[sl]) blk += mm; else arm += mm;
            }
        };
        if (kP2P) {
            // most configurations penetrate something and the rest of the code is small: all joints at
            // once, one chain of exchanges
            float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, none = 0.f;
#pragma unroll
            for (int k = 0; k < 7; ++k) torque(k, v[k], none);
            const float sum = warp_sums<8>(v);   // lane 4 i: value i
            if ((lane & 3) == 0) {
                rows[16 * t + (lane >> 2)] = sum;
                rows[16 * t + 8 + (lane >> 2)] = 0.f;
            }
        } else {
            // two joints (arm- and block-group torques of each) per round of a rolled loop: the seventh
            // joint's partner k = 7 has no axis and stays zero
#pragma unroll 1
            for (int k = 0; k < 8; k += 2) {
                float v[4] = {0.f, 0.f, 0.f, 0.f};   // arm k, arm k + 1, block k, block k + 1
                torque(k, v[0], v[2]);
                if (k < 6) torque(k + 1, v[1], v[3]);
                const float sum = warp_sums<4>(v);   // lane 8 i: value i
                if ((lane & 7) == 0) rows[16 * t + (lane >> 4) * 8 + k + ((lane >> 3) & 1)] = sum;
            }
        }
    }
    if (lane == 0) {
        tw.count[0] += tests;
        tw.count[1] += (unsigned)nc;
        tw.count[2] += (unsigned)n_cand;
    }
    if (has == 0u) return kStateZero;
    // the tests' gaps join the clearances of a half without a penetration
    if (hits && lane == 0) atomicOr(&sh.hit[(t0 - 1) >> 5], hits << ((t0 - 1) & 31));
    clearance = fminf(clearance, warp_fmin(gap_s));
    if (kP2P) return hits ? kStateZeroMoving : kStateZero;
    clearance_moving = fminf(clearance_moving, warp_fmin(gap_m));
    clearance_top = fminf(clearance_top, warp_fmin(gap_t));
    return (__any_sync(0xffffffffu, hit_s) ? 0 : kStateZeroStatic) | (__any_sync(0xffffffffu, hit_m) ? 0 : kStateZeroMoving);
}

// The scale dL/dh of residual r, (lambda_r + mu sqrt(w) h) sqrt(w).
__device__ __forceinline__ float residual_scale(const TShared& sh, int r, float sqw, float h) {
    const float hw = sqw * h;
    return (sh.lam[r] + sh.mu * hw) * sqw;
}

// C_coll of the placed tower: the fixed-order sum over the slices.
__device__ __forceinline__ float tower_collisions(const TShared& sh, int n_pu) {
    float c = 0.f;
#pragma unroll 1
    for (int u = 0; u < n_pu; ++u) c += sh.pcu[u][0];
    return c;
}

// Residuals of the start group at the grasp (place = false) or place configuration of block b
// from that configuration's frames: position error, roll and pitch, or roll and pitch, to sh.h
// from r on, their scales to sh.s; the roll and pitch torques to rpt.
__device__ __forceinline__ void start_residuals(const TrajScalars& sc, TShared& sh, int b, bool place,
                                                const SpecialFrames& sf, int r0, float rpt[6]) {
    float Rb[9], pb[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        Rb[3 * r] = sf.H[r].x; Rb[3 * r + 1] = sf.H[r].y; Rb[3 * r + 2] = sf.H[r].z; pb[r] = sf.H[r].w;
    }
    float roll, pitch;
    roll_pitch_torque<float>(Rb, roll, pitch, rpt, rpt + 3);
    const float h[5] = {roll, pitch, pb[0] - sc.init[b].x, pb[1] - sc.init[b].y, pb[2] - sc.init[b].z};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int r = r0 + (place ? i : (i + 3) % 5);   // grasp: x, y, z, roll, pitch
        if (place && i >= 2) continue;
        sh.h[r] = h[i];
        sh.s[r] = residual_scale(sh, r, sc.sqw[0], h[i]);
    }
}

// Joint k of their weighted gradient sum_r s_r dh_r/dq, plus at a place configuration the
// placed-pose gradient g4 through fk, from the torques the residual pass left in rpt.
__device__ __forceinline__ float start_gradient(bool place, const SpecialFrames& sf, const float* s_r, const float* g4,
                                                const float rpt[6], int k) {
    float Rb[9], pb[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        Rb[3 * r] = sf.H[r].x; Rb[3 * r + 1] = sf.H[r].y; Rb[3 * r + 2] = sf.H[r].z; pb[r] = sf.H[r].w;
    }
    const float wr[3] = {rpt[0], rpt[1], rpt[2]}, wp[3] = {rpt[3], rpt[4], rpt[5]};
    // wrench at the block frame: force F (on p_blk), torque M (about the world origin)
    const float* f = place ? g4 : s_r;
    const float s_roll = s_r[place ? 0 : 3], s_pitch = s_r[place ? 1 : 4];
    const float F[3] = {f[0], f[1], f[2]};
    float M[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) M[i] = s_roll * wr[i] + s_pitch * wp[i];
    if (place) {
        const float e[3] = {Rb[0], Rb[3], Rb[6]};
        float wy[3];
        yaw_torque(e, wy);
#pragma unroll
        for (int i = 0; i < 3; ++i) M[i] += g4[3] * wy[i];
    }
    // moment of F about the origin: p x F
    M[0] += pb[1] * F[2] - pb[2] * F[1];
    M[1] += pb[2] * F[0] - pb[0] * F[2];
    M[2] += pb[0] * F[1] - pb[1] * F[0];
    const float2 f0 = sf.Z[k][0], f1 = sf.Z[k][1], f2 = sf.Z[k][2];
    const float ok[3] = {f0.y, f1.y, f2.y};
    // z . (M - o x F)
    const float tx = M[0] - (ok[1] * F[2] - ok[2] * F[1]);
    const float ty = M[1] - (ok[2] * F[0] - ok[0] * F[2]);
    const float tz = M[2] - (ok[0] * F[1] - ok[1] * F[0]);
    return f0.x * tx + f1.x * ty + f2.x * tz;
}

// Collisions of the placed tower (the C_coll residual of the placement terms), slice u of its
// block spheres (items 32u .. 32u+31, item 8j + m: sphere m of block j) by one warp.  An exact
// cull first keeps the environment obstacles whose boxes overlap the tower's box (every block
// sphere lies inside its block's cuboid box); a box test screens each pair before the exact
// one; each sphere of block j is also tested against the cuboids of the blocks i < j below it.
// Writes the slice's sum and maximum of the penetrations (sh.pcu[u]); with `grad`, the
// unscaled pose gradient dC_coll/dx, sphere side in sh.pg[j] for the slice's blocks and
// cuboid side in sh.pgc[u][i] for every i < B - 1.
__device__ __forceinline__ void placed_slice(const TrajScalars& sc, const float4* __restrict__ cub,
                                             const float4* __restrict__ osph, const float4* __restrict__ aabb,
                                             TShared& sh, bool grad, int u) {
    const int lane = threadIdx.x & 31;
    const int B = sc.B, n_items = 8 * B;
    const int it = 32 * u + lane;
    const bool valid = it < n_items;
    const int j = valid ? it >> 3 : 0, m = it & 7;
    const float4 h = sc.half[j];
    float lx, ly, lz;
    block_sphere_local(h, m, lx, ly, lz);
    const float c = sh.blk[j][1].x, s = sh.blk[j][1].y;
    const float cx = sh.pose[4 * j] + c * lx - s * ly;
    const float cy = sh.pose[4 * j + 1] + s * lx + c * ly;
    const float cz = sh.pose[4 * j + 2] + lz;
    const float r = h.w;
    const int n_cw = t_cub_words(sc.n_cub), n_w = t_words(sc.n_cub, sc.n_osph);
    // the box of the slice's blocks
    const int bj = min(4 * u + (lane & 3), B - 1);
    const float4 mlo = sh.bbox[bj][0], mhi = sh.bbox[bj][1];
    const float tlx = warp_fmin(mlo.x), tly = warp_fmin(mlo.y), tlz = warp_fmin(mlo.z);
    const float thx = warp_fmax(mhi.x), thy = warp_fmax(mhi.y), thz = warp_fmax(mhi.z);
    float coll = 0.f, maxpen = 0.f;
    float ax = 0.f, ay = 0.f, az = 0.f;   // dC/dc of this item
    if (grad) {
        sh.pgc[u][lane >> 1][2 * (lane & 1)] = 0.f;
        sh.pgc[u][lane >> 1][2 * (lane & 1) + 1] = 0.f;
        __syncwarp();
    }
    // the environment's obstacles and the blocks below that box could touch: a sphere of j against
    // the cuboids of i < j (the slice's highest block bounds i)
    const int i_end = min(B - 1, (min(32 * u + 31, n_items - 1) >> 3));
#pragma unroll 1
    for (int wd = 0; wd < n_w; ++wd) {
        const bool blocks = wd == n_w - 1;
        const float4* box = blocks ? sh.bbox[0] : aabb + 64 * wd;
        const float4 clo = box[2 * lane], chi = box[2 * lane + 1];
        unsigned mk = __ballot_sync(
            0xffffffffu, !(clo.x > thx || chi.x < tlx || clo.y > thy || chi.y < tly || clo.z > thz || chi.z < tlz));
        if (blocks) mk &= (1u << i_end) - 1u;
#pragma unroll 1
        while (mk) {
            const int bit = __ffs(mk) - 1;
            mk &= mk - 1;
            const float4 lo = box[2 * bit], hi = box[2 * bit + 1];
            const bool apart =
                lo.x > cx + r || hi.x < cx - r || lo.y > cy + r || hi.y < cy - r || lo.z > cz + r || hi.z < cz - r;
            float gx = 0.f, gy = 0.f, gz = 0.f, pen = 0.f;
            if (wd >= n_cw && !blocks) {
                if (valid) pen = pen_sphere<float>(cx, cy, cz, r, osph[32 * (wd - n_cw) + bit], gx, gy, gz);
            } else if (valid && !apart && (!blocks || bit < j)) {
                const float4* rec = blocks ? sh.blk[bit] : cub + 4 * (32 * wd + bit);
                pen = pen_cuboid<float>(cx, cy, cz, r, rec[0], rec[1], rec[2], rec[3], gx, gy, gz);
            }
            const bool hit = pen > 0.f;
            float d4[4] = {0, 0, 0, 0};   // dC/d(pose of the block below) from this item
            if (hit) {
                coll += pen; maxpen = fmaxf(maxpen, pen);
                ax += gx; ay += gy; az += gz;
                // the cuboid moves rigidly: d/dP_i = -g, d/dyaw_i = -((c - P_i) x g)_z (the fused
                // product is spelt out so that the rounding does not depend on the compiler's choice)
                const float* pi = &sh.pose[4 * (bit & 15)];
                d4[0] = -gx; d4[1] = -gy; d4[2] = -gz;
                d4[3] = -__fmaf_rn(-(cy - pi[1]), gx, __fmul_rn(cx - pi[0], gy));
            }
            if (grad && blocks && __any_sync(0xffffffffu, hit)) {
                const float d = warp_sums<4>(d4);   // lane 8 i: value i
                if ((lane & 7) == 0) sh.pgc[u][bit][lane >> 3] = d;
            }
        }
    }
    if (grad) {
        float gyaw = ax * (-s * lx - c * ly) + ay * (c * lx - s * ly);   // dc/dyaw_j
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) {
            ax += __shfl_xor_sync(0xffffffffu, ax, off);
            ay += __shfl_xor_sync(0xffffffffu, ay, off);
            az += __shfl_xor_sync(0xffffffffu, az, off);
            gyaw += __shfl_xor_sync(0xffffffffu, gyaw, off);
        }
        // one writer per block j: the lane with m == 0
        if (valid && m == 0) { sh.pg[j][0] = ax; sh.pg[j][1] = ay; sh.pg[j][2] = az; sh.pg[j][3] = gyaw; }
    }
    coll = warp_sum(coll);
    maxpen = warp_fmax(maxpen);
    if (lane == 0) { sh.pcu[u][0] = coll; sh.pcu[u][1] = maxpen; }
}

// Modes of the trajectory kernel
enum TrajMode { kTrajEval = 0, kTrajDescend = 1 };

// Axis-aligned box of a cuboid record (centre, then R columns with half extents).
__device__ __forceinline__ void cuboid_aabb(const float4* c, float4* box) {
    const float ex = fabsf(c[1].x) * c[1].w + fabsf(c[2].x) * c[2].w + fabsf(c[3].x) * c[3].w;
    const float ey = fabsf(c[1].y) * c[1].w + fabsf(c[2].y) * c[2].w + fabsf(c[3].y) * c[3].w;
    const float ez = fabsf(c[1].z) * c[1].w + fabsf(c[2].z) * c[2].w + fabsf(c[3].z) * c[3].w;
    box[0] = make_float4(c[0].x - ex, c[0].y - ey, c[0].z - ez, 0.f);
    box[1] = make_float4(c[0].x + ex, c[0].y + ey, c[0].z + ez, 0.f);
}

// An empty box: never a candidate.
__device__ __forceinline__ void empty_box(float4* box) {
    box[0] = make_float4(3.4e38f, 3.4e38f, 3.4e38f, 0.f);
    box[1] = make_float4(-3.4e38f, -3.4e38f, -3.4e38f, 0.f);
}

// The run of configurations [t_lo, t_hi) that warp w of a group steps in traj_step, ascending with
// w: the first warp, busy with the placement gradient, takes none, or a third where there are but
// two; point to point has none and deals equal runs.
template <bool kP2P, int kPpc>
__device__ __forceinline__ void step_run(int C, int w, int& t_lo, int& t_hi) {
    constexpr int kWarps = kGrpWarps<kPpc>;
    const int first = kP2P ? (C + kWarps - 1) / kWarps : kWarps == 2 ? C / 3 : 0;
    const int run = (C - first + kWarps - 2) / (kWarps - 1);
    t_lo = w > 0 ? min(C, first + (w - 1) * run) : 0;
    t_hi = w > 0 ? min(C, t_lo + run) : first;
}

// Evaluate the whole particle: kinematics of the grasp/place configurations and the placed
// poses, the configuration loop, residuals and objective; with `grad`, the parts of dL/dq that
// traj_step adds up (the collision groups' rows and fixed-point sums, the residuals' scales and
// the placement gradient without its collision terms).
template <bool kP2P, int kTile, int kPpc>
__device__ void traj_evaluate(const TrajScalars& sc, const LaneSpheres& ls, const float4* cub, const float4* osph,
                              const float4* aabb, TShared& sh, TWarp* tws, SpecialFrames* sp, float* q, float* rows,
                              float* disp, float* cblk, __half2* cgap, unsigned char* state, float* ctopm,
                              __half* ctop, bool grad, bool last) {
    constexpr int kWarps = kGrpWarps<kPpc>;
    const int tid = grp_tid<kPpc>(), lane = tid & 31, w = tid >> 5;
    const int B = sc.B, S = sc.S, C = sc.C, NR = sc.NR;
    // point to point (kP2P): one segment ending at the target's grasp configuration; no placement
    constexpr bool p2p = kP2P;

    // The kinematics have one call site (their code is the larger part of a small phase): the warps
    // first run them over the 2B grasp / place configurations (4 per warp), kept for the epilogue,
    // then, once the placed poses are known, over the chunks of the evaluation's work queue.
    const int n_sp = p2p ? 1 : 2 * B, n_pu = p2p ? 0 : (8 * B + 31) / 32;
    const int n_chunks = (C - 1 + kChunk - 1) / kChunk, c = lane >> 3;
    const float inv_S = sh.inv_S;
    static_assert((kMaxC + kChunk - 1) / kChunk <= 256, "chunk indices fit the byte lists");
    static_assert((kMaxC + kChunk - 1) / kChunk <= 32 * kChunkGroups, "the groups hold every chunk");
    // bound on the motion of each block placed before block b (the only placed blocks the
    // configurations of a chunk whose last configuration belongs to block b's segments can
    // touch): its difference between two evaluations bounds any one block's motion between them
    auto blk_before = [&](int b) { return b > 0 ? sh.blk_cum[b - 1] : 0.f; };
    auto chunk_block = [&](int t0c) { return div_steps(min(t0c + kChunk - 1, C - 1) - 1, inv_S) >> 1; };
    // own motion of block k (the top block of a chunk of block k + 1's segments), 0 for none
    auto own_motion = [&](int k) { return k >= 0 ? sh.bown[k] : 0.f; };
#pragma unroll 1
    for (int i = tid; i < 2 * kMaxB * 4; i += kGrpThreads<kPpc>) (&sh.fx_wr[0][0][0])[i] = 0;
    if (tid < kMaxC / 32) sh.hit[tid] = 0u;
    if (tid <= kChunk) sh.n_tier[tid] = 0;
    if (tid == 0) { sh.fx_tot[0] = sh.fx_tot[1] = 0; sh.next = 0; }
    // start residuals: grasp configurations on lanes 0..15, place configurations on 16..31
    auto start_job = [&]() {
        const int b = lane & 15;
        const bool place = lane >= 16;
        if (b >= B) return;
        const int r = place ? 5 * B + 2 * b : 5 * b;
        if (!place || !p2p) start_residuals(sc, sh, b, place, sp[2 * b + place], r, sh.rpt[2 * b + place]);
        else sh.h[r] = sh.h[r + 1] = 0.f;
    };
    float acc_max = 0.f;
    bool special = true;
    int gi = w;
#pragma unroll 1
    for (;;) {
        int chk = 0, si = 0, t_c, b_c;
        bool write = true, want_h = true;
        if (special) {
            if (4 * gi >= n_sp) {
                special = false;
                grp_sync<kPpc>();
                // placed poses: the block frame at each place configuration, (x, y, z, yaw)
                if (w == 0) {
                    float moved = 0.f;
                    if (lane < B && !p2p) {
                        const float4* H = sp[2 * lane + 1].H;
                        const float pose[4] = {H[0].w, H[1].w, H[2].w, atan2f(H[1].x, H[0].x)};
                        // how far any point of the placed cuboid moved since the previous evaluation:
                        // |d position| + |d yaw| times its horizontal half diagonal
                        if (sh.pose_prev_ok) {
                            const float* pp = &sh.pose_prev[4 * lane];
                            const float dx = pose[0] - pp[0], dy = pose[1] - pp[1], dz = pose[2] - pp[2];
                            float dyaw = fabsf(pose[3] - pp[3]);
                            dyaw = fminf(dyaw, 2.f * kPi - dyaw);
                            const float4 h = sc.half[lane];
                            moved = (sqrtf(dx * dx + dy * dy + dz * dz) + dyaw * sqrtf(h.x * h.x + h.y * h.y)) * 1.0001f + 1e-6f;
                        }
                        for (int i = 0; i < 4; ++i) sh.pose[4 * lane + i] = sh.pose_prev[4 * lane + i] = pose[i];
                        block_cuboid(pose[0], pose[1], pose[2], pose[3], sc.half[lane], sh.blk[lane]);
                        cuboid_aabb(sh.blk[lane], sh.bbox[lane]);
                    } else if (lane < B) {   // point to point: the placed boxes stay empty
                        for (int i = 0; i < 4; ++i) sh.pose[4 * lane + i] = 0.f;
                    }
                    if (lane < B) sh.bown[lane] += moved;   // the block's own motion, before the scan
                    // inclusive max-scan over the blocks: blk_cum[k] accumulates, evaluation by evaluation, the
                    // largest motion among blocks 0..k.  Summed over the evaluations since a chunk's cull it
                    // bounds the motion of each of those blocks since then, which is all that a gap to any
                    // one of them needs (a sum over the blocks would bound their total motion instead)
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const float up = __shfl_up_sync(0xffffffffu, moved, off);
                        if (lane >= off) moved = fmaxf(moved, up);
                    }
                    if (lane < B) sh.blk_cum[lane] += moved;
                    if (lane == 0) sh.pose_prev_ok = 1;
                } else if (w == 1 && !p2p) {
                    start_job();   // beside the placed poses, which keep warp 0 about as long
                }
                grp_sync<kPpc>();
                // (2) the work queue, in order: the chunks to evaluate, which are those with a half that has no
                // valid cached cull (terms zero at its last cull, and the motion since below its clearances), by
                // tier (with a penetration: 4, 3, 2, 1 configurations with candidates; then the others); the
                // placement residuals (they need only the placed poses); the slices of the placed tower.  The
                // smaller items come last, so that the warps finish together.  Each warp appends the chunks
                // of its 32-chunk groups to the tiers' lists.
#pragma unroll 1
                for (int gr = w; gr < kChunkGroups; gr += kWarps) {
                    const int chk = 32 * gr + lane;
                    const int t0 = 1 + kChunk * chk, nc = min(kChunk, C - t0);
                    int tier = -1;
                    if (chk < n_chunks) {
                        float d = 0.f;
#pragma unroll 1
                        for (int i = 0; i < nc; ++i) d = fmaxf(d, disp[t0 + i]);
                        const __half2 cg = cgap[chk];
                        const int top = chunk_block(t0) - 1, st = state[chk];
                        const bool skip_s = (st & kStateZeroStatic) && d < __low2float(cg);
                        const bool skip_m = (st & kStateZeroMoving) && d + (blk_before(top) - cblk[chk]) < __high2float(cg) &&
                                            d + (own_motion(top) - ctopm[chk]) < __half2float(ctop[chk]);
                        if (!(skip_s && skip_m)) {
                            tier = (st & kStateZero) == kStateZero ? kChunk : kChunk - (st & kStateCand);
                            state[chk] = (unsigned char)((st & ~(kStateSkipStatic | kStateSkipMoving)) |
                                                         (skip_s ? kStateSkipStatic : 0) | (skip_m ? kStateSkipMoving : 0));
                        }
                    }
                    unsigned same = 0u;   // lane tr <= kChunk: the group's chunks in tier tr
#pragma unroll
                    for (int tr = 0; tr <= kChunk; ++tr) {
                        const unsigned bal = __ballot_sync(0xffffffffu, tier == tr);
                        if (lane == tr) same = bal;
                    }
                    const int base = lane <= kChunk ? atomicAdd(&sh.n_tier[lane], __popc(same)) : 0;
                    const int first = __shfl_sync(0xffffffffu, base, max(tier, 0));
                    const unsigned mates = __shfl_sync(0xffffffffu, same, max(tier, 0));
                    if (tier >= 0) sh.active[tier][first + __popc(mates & ((1u << lane) - 1u))] = (unsigned char)chk;
                }
                grp_sync<kPpc>();
                continue;
            }
            si = 4 * gi + c;
            write = si < n_sp;
            if (!write) si = 0;
            t_c = write ? (si + 1) * S : 1;
            b_c = si >> 1;
            gi += kWarps;
        } else {
            int idx = 0;
            if (lane == 0) idx = atomicAdd(&sh.next, 1);
            idx = __shfl_sync(0xffffffffu, idx, 0);
            int tier = 0;
#pragma unroll
            for (int tr = 0; tr <= kChunk; ++tr) {
                const int n = sh.n_tier[tr];
                if (tier == tr && idx >= n) { idx -= n; ++tier; }
            }
            if (tier > kChunk && idx >= kResidualJobs) {
                idx -= kResidualJobs;
                if (idx >= n_pu) break;
                placed_slice(sc, cub, osph, aabb, sh, grad, idx);
                continue;
            }
            if (tier > kChunk) {
                // placement residuals (tower terms) with their unit-coefficient support factors; point to
                // point, which has none, takes the start residuals here
                float my_D = 0.f, my_e = 0.f;
                if (p2p) start_job();
                else place_stack_warp(sc, sh.pose, kPlaceUnit, nullptr, sh.ps, sh.blk, my_D, my_e);
                const float c_stable = warp_sum(lane < B ? my_D : 0.f);
                const float c_height = warp_sum(lane < B ? my_e * my_e : 0.f);
                const float max_D = warp_fmax(lane < B ? my_D : 0.f);
                const float max_dz = warp_fmax(lane < B ? fabsf(my_e) : 0.f);
                if (lane < B) {
                    sh.h[7 * B + lane] = my_e;
                    sh.h[8 * B + lane] = my_D;
                    sh.s[7 * B + lane] = residual_scale(sh, 7 * B + lane, sc.sqw[1], my_e);
                    sh.s[8 * B + lane] = residual_scale(sh, 8 * B + lane, sc.sqw[2], my_D);
                }
                if (grad && !p2p) {   // their part of the placement gradient (the collisions' part follows the queue)
                    __syncwarp();
                    place_stack_grad(sc, sh.ps, &sh.s[8 * B], &sh.s[7 * B], sh.inv_above, sh.g4);
                }
                if (lane == 0) { sh.c_stable = c_stable; sh.c_height = c_height; sh.pm_D = max_D; sh.pm_dz = max_dz; }
                continue;
            }
            chk = sh.active[tier][idx];
            t_c = min(1 + kChunk * chk + c, C - 1);
            const int seg = div_steps(t_c - 1, inv_S);
            // the held block's frame matters on transfer-segment interiors only
            want_h = (seg & 1) && t_c - seg * S < S;
            b_c = seg >> 1;
        }
        float box[6];
        chunk_fk<kP2P>(sc, sh, q, t_c, b_c, write, want_h, tws[w].F[c], special ? sp[si].Z : nullptr,
                 special ? sp[si].H : tws[w].H[c], box);
        if (special) continue;
        __syncwarp();
        const int t0 = 1 + kChunk * chk, nc = min(kChunk, C - t0), seg_c = div_steps(t_c - 1, inv_S);
        float clearance, clearance_moving, clearance_top, c2[2] = {0.f, 0.f};
        int n_cand;
        const int skip = state[chk];
        const int zero = chunk_collisions<kP2P, kTile>(sc, ls, cub, osph, aabb, sh, tws[w], rows, t0, nc, seg_c, skip, grad, box,
                                                 c2[0], c2[1], acc_max, n_cand, clearance, clearance_moving,
                                                 clearance_top);
        if (zero != kStateZero) {
            const float v = warp_sums<2>(c2);   // lane 0: the arm's sum, lane 16: the held block's
            if ((lane & 15) == 0) fx_add(&sh.fx_tot[lane >> 4], v);
        }
        const float d = warp_fmax(lane < nc ? disp[t0 + lane] : 0.f);
        if (lane == 0) {
            state[chk] = (unsigned char)(n_cand | zero);
            const __half2 cg = cgap[chk];
            const int top = chunk_block(t0) - 1;
            // a skipped half keeps its clearance less the motion so far (disp starts at zero again) and the
            // blocks' motions it was taken at
            float cs = clearance - kClearSlack, cm = clearance_moving - kClearSlack, ct = clearance_top - kClearSlack;
            if (skip & kStateSkipStatic) cs = __fsub_rd(__low2float(cg), d);
            if (skip & kStateSkipMoving) {
                cm = __fsub_rd(__high2float(cg), d);
                ct = __fsub_rd(__half2float(ctop[chk]), d);
            } else {
                cblk[chk] = blk_before(top);
                ctopm[chk] = own_motion(top);
            }
            // fp16, rounded down: still lower bounds on the clearances
            cgap[chk] = __halves2half2(__float2half_rd(cs), __float2half_rd(cm));
            ctop[chk] = __float2half_rd(ct);
        }
        __syncwarp();
        if (lane < nc) disp[t0 + lane] = 0.f;
        __syncwarp();
    }
    acc_max = warp_fmax(acc_max);
    if (lane == 0) tws[w].maxpen = acc_max;
    int t_lo, t_hi;
    step_run<kP2P, kPpc>(C, w, t_lo, t_hi);
    if (lane < 4 && t_lo < t_hi)   // for the step: the run's first row, then its last
        tws[w].edge[lane >> 1][lane & 1] = reinterpret_cast<const float4*>(q + 8 * (lane < 2 ? t_lo : t_hi - 1))[lane & 1];
    grp_sync<kPpc>();

    if (!last) return;

    // (3) warp 0, after the last evaluation: the objective and the metrics
    if (w == 0) {
        const float tot_a = fx_value(sh.fx_tot[0]), tot_b = fx_value(sh.fx_tot[1]), c_coll = tower_collisions(sh, n_pu);
        if (lane == 0) {
            sh.h[9 * B] = c_coll;
            sh.h[9 * B + 1] = tot_a;
            sh.h[9 * B + 2] = tot_b;
        }
        __syncwarp();   // the group residuals before every lane reads sh.h[]
        float Lp = 0.f;
#pragma unroll 1
        for (int r = lane; r < NR; r += 32) {
            const float hw = residual_sqrt_weight(sc, r) * sh.h[r];
            Lp += sh.lam[r] * hw + 0.5f * sh.mu * hw * hw;
        }
        const float cm = warp_fmax(lane < kWarps ? tws[lane].maxpen : 0.f);
        const float pm = warp_fmax(lane < n_pu ? sh.pcu[lane][1] : 0.f);
        float v_start = 0.f, v_tilt = 0.f;
        if (lane < B) {
            const float* hg = &sh.h[5 * lane];
            const float* hp = &sh.h[5 * B + 2 * lane];
            v_start = hg[0] * hg[0] + hg[1] * hg[1] + hg[2] * hg[2] + hg[3] * hg[3] + hg[4] * hg[4];
            v_tilt = hp[0] * hp[0] + hp[1] * hp[1];
        }
        const float c_start = warp_sum(v_start + v_tilt);
        const float m_start = warp_fmax(v_start), m_tilt = warp_fmax(v_tilt);
        Lp = warp_sum(Lp);
        if (lane == 0) {
            sh.c_arm = tot_a; sh.c_blk = tot_b; sh.maxpen = cm;
            sh.c_coll = c_coll; sh.pm_pen = pm;
            sh.L = Lp; sh.c_start = c_start; sh.max_start = m_start; sh.max_tilt = m_tilt;
        }
    }
    grp_sync<kPpc>();
}

// One descent step, q <- clamp(q - eta g), and the bound on how far each configuration's spheres
// moved (disp); or, when grad_out is given, the gradient itself (8 floats per configuration, the
// last and the fixed first configuration's zero).  The gradient of configuration t: the path term
// from its neighbours, the joint limits, the collision groups' rows and, at the grasp and place
// configurations, their own row.
// Warp 0 first completes the placement gradient, which only the place configurations' rows need;
// the other warps step the configurations in between meanwhile and leave the special ones, whose
// gradient so far goes to sh.partial; after a barrier, a lane per joint adds the special rows
// and steps those.  (Rows first, then one pass over every configuration: 12 of an evaluation's
// 41 thousand cycles on the 10-block tower, with one warp at work for 8 of them.)
// In place, a configuration per lane (rows as float4 pairs): each warp takes a contiguous run of
// configurations, 32 at a time in ascending order; a row that its neighbour reads after the
// step is kept in TWarp::edge as it was (the run's first and last rows, kept by traj_evaluate,
// and the last row of the previous 32).
// `limits`: joints may lie outside their limits (a step clamps them, so only before the first).
template <bool kP2P, int kPpc>
__device__ __forceinline__ void traj_step(const TrajScalars& sc, TShared& sh, TWarp* tws, const SpecialFrames* sp, float* q,
                                          const float* rows, float* disp, float eta, bool limits, float* grad_out) {
    constexpr int kWarps = kGrpWarps<kPpc>;
    const int tid = grp_tid<kPpc>(), lane = tid & 31, w = tid >> 5;
    const int B = sc.B, C = sc.C, S = sc.S, n_pu = kP2P ? 0 : (8 * B + 31) / 32;
    int t_lo, t_hi;
    step_run<kP2P, kPpc>(C, w, t_lo, t_hi);
    const float tot_a = fx_value(sh.fx_tot[0]), tot_b = fx_value(sh.fx_tot[1]);
    const float s_arm = residual_scale(sh, 9 * B + 1, sc.sqw[4], tot_a);
    const float s_blk = residual_scale(sh, 9 * B + 2, sc.sqw[5], tot_b);
    if (w == 0) {
        const float c_coll = tower_collisions(sh, n_pu), s_coll = residual_scale(sh, 9 * B, sc.sqw[3], c_coll);
        if (lane == 0) { sh.h[9 * B] = c_coll; sh.h[9 * B + 1] = tot_a; sh.h[9 * B + 2] = tot_b; }
#pragma unroll 1
        for (int i = lane; i < (kP2P ? 0 : 4 * B); i += 32) {
            const int kb = i >> 2, c = i & 3;
            const float wa = fx_value(sh.fx_wr[0][kb][c]), wb = fx_value(sh.fx_wr[1][kb][c]);
            float gc = sh.pg[kb][c];
            if (kb + 1 < B)
#pragma unroll 1
                for (int u = 0; u < n_pu; ++u) gc += sh.pgc[u][kb][c];
            sh.g4[i] += s_coll * gc + s_arm * wa + s_blk * wb;
        }
    }
    const float inv_S = sh.inv_S, w2 = 2.f * sc.w_path;
    // a row without collision terms adds s_arm 0 + s_blk 0, which is zero unless a scale is not finite
    const bool all_rows = !(s_arm * 0.f + s_blk * 0.f == 0.f);
#pragma unroll 1
    for (int t0 = t_lo; t0 < t_hi; t0 += 32) {
        const int t = t0 + lane;
        const bool in = t < t_hi;
        const float4* qv = reinterpret_cast<const float4*>(q + 8 * min(t, t_hi - 1));
        const float4* pr = lane > 0 ? qv - 2 : t0 > t_lo ? tws[w].edge[2] : t0 > 0 ? tws[w - 1].edge[1] : qv;
        const float4* nx = t + 1 >= C ? qv : t + 1 < t_hi ? qv + 2 : tws[w + 1].edge[0];
        const float4 a0 = qv[0], a1 = qv[1], p0 = pr[0], p1 = pr[1], n0 = nx[0], n1 = nx[1];
        const float v[7] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z};
        const float pv[7] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z};
        const float nv[7] = {n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n1.z};
        __syncwarp();   // the last 32's rows, and tws[w].edge[2], have been read
        if (lane == 31) { tws[w].edge[2][0] = a0; tws[w].edge[2][1] = a1; }
        float g[7];
#pragma unroll
        for (int j = 0; j < 7; ++j) {
            g[j] = 0.f - w2 * (nv[j] - v[j]);
            g[j] += w2 * (v[j] - pv[j]);
        }
        if (limits) {
#pragma unroll
            for (int j = 0; j < 7; ++j) {
                const float over = fmaxf(v[j] - sc.qhi[j], 0.f), under = fmaxf(sc.qlo[j] - v[j], 0.f);
                g[j] += sc.w_jl * (2.f * over - 2.f * under);
            }
        }
        const bool hit = in && t > 0 && ((sh.hit[(t - 1) >> 5] >> ((t - 1) & 31)) & 1u);
        if (hit || all_rows) {
            float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0, r2 = r0, r3 = r0;
            if (hit) {
                const float4* rv = reinterpret_cast<const float4*>(rows + 16 * t);
                r0 = rv[0]; r1 = rv[1]; r2 = rv[2]; r3 = rv[3];
            }
            const float ga[7] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z};
            const float gb[7] = {r2.x, r2.y, r2.z, r2.w, r3.x, r3.y, r3.z};
#pragma unroll
            for (int j = 0; j < 7; ++j) g[j] += s_arm * ga[j] + s_blk * gb[j];
        }
        const int e = div_steps(t, inv_S) - 1;
        const bool special = e >= 0 && t == (e + 1) * S;
        if (in && special) {   // grasp of block e / 2 (e even) or place (e odd)
            sh.partial[e][0] = make_float4(g[0], g[1], g[2], g[3]);
            sh.partial[e][1] = make_float4(g[4], g[5], g[6], 0.f);
        } else if (grad_out) {
            float* go = grad_out + (size_t)t * 8;
            if (t == 0) {
#pragma unroll
                for (int j = 0; j < 7; ++j) g[j] = 0.f;
            }
            if (in && (reinterpret_cast<uintptr_t>(grad_out) & 15u) == 0) {
                reinterpret_cast<float4*>(go)[0] = make_float4(g[0], g[1], g[2], g[3]);
                reinterpret_cast<float4*>(go)[1] = make_float4(g[4], g[5], g[6], 0.f);
            } else if (in) {
#pragma unroll
                for (int j = 0; j < 7; ++j) go[j] = g[j];
                go[7] = 0.f;
            }
        } else if (in && t > 0) {
            float nw[7], moved = 0.f;
#pragma unroll
            for (int j = 0; j < 7; ++j) {
                const float x = v[j] - eta * g[j];
                nw[j] = fminf(fmaxf(x, sc.qlo[j]), sc.qhi[j]);
                moved += fabsf(nw[j] - v[j]) * sc.sweep[j];
            }
            float4* qw = reinterpret_cast<float4*>(q + 8 * t);
            qw[0] = make_float4(nw[0], nw[1], nw[2], nw[3]);
            qw[1] = make_float4(nw[4], nw[5], nw[6], a1.w);
            disp[t] += moved * 1.0001f + 1e-7f;
        }
        __syncwarp();   // tws[w].edge[2] before lane 0 reads it
    }
    grp_sync<kPpc>();
    // the special configurations, four per warp: lane 8 c + j, joint j
    const int n_sp = kP2P ? 1 : 2 * B, j = lane & 7, jj = min(j, 6);
#pragma unroll 1
    for (int e = 4 * w + (lane >> 3); e - (lane >> 3) < n_sp; e += 4 * kWarps) {
        const int b = e >> 1, t = (e + 1) * S;
        const bool in = e < n_sp && j < 7, place = e & 1;
        float g = 0.f, moved = 0.f;
        if (in) {
            g = reinterpret_cast<const float*>(sh.partial[e])[j];
            g += start_gradient(place, sp[e], &sh.s[place ? 5 * B + 2 * b : 5 * b], &sh.g4[4 * b], sh.rpt[e], j);
        }
        if (grad_out) {
            if (e < n_sp) grad_out[(size_t)t * 8 + j] = g;
            continue;
        }
        if (in) {
            const float v = q[8 * t + j], x = v - eta * g;
            const float nw = fminf(fmaxf(x, sc.qlo[jj]), sc.qhi[jj]);
            q[8 * t + j] = nw;
            moved = fabsf(nw - v) * sc.sweep[jj];
        }
        moved += __shfl_xor_sync(0xffffffffu, moved, 1);
        moved += __shfl_xor_sync(0xffffffffu, moved, 2);
        moved += __shfl_xor_sync(0xffffffffu, moved, 4);
        if (e < n_sp && j == 0) disp[t] += moved * 1.0001f + 1e-7f;
    }
}

// After the last evaluation: the path length and joint limits (sh.path, sh.jl, added to sh.L), a
// configuration per thread.
template <int kPpc>
__device__ __forceinline__ void traj_path(const TrajScalars& sc, TShared& sh, const float* q) {
    const int tid = grp_tid<kPpc>(), lane = tid & 31, w = tid >> 5;
    const int C = sc.C;
    // partial sums in the order of 256 threads, whatever the group: thread tid of kGrpThreads holds
    // those of threads tid, tid + kGrpThreads, ...
    float path[kPpc], jl[kPpc];
#pragma unroll
    for (int i = 0; i < kPpc; ++i) {
        float psum = 0.f, jsum = 0.f;
#pragma unroll 1
        for (int t = tid + i * kGrpThreads<kPpc>; t < C; t += kTThreads) {
#pragma unroll 1
            for (int j = 0; j < 7; ++j) {
                const float v = q[t * 8 + j];
                if (t + 1 < C) {
                    const float d = q[t * 8 + 8 + j] - v;
                    psum += d * d;
                }
                if (t > 0) {
                    const float over = fmaxf(v - sc.qhi[j], 0.f), under = fmaxf(sc.qlo[j] - v, 0.f);
                    jsum += over * over + under * under;
                }
            }
        }
        path[i] = psum;
        jl[i] = jsum;
    }
#pragma unroll
    for (int i = 0; i < kPpc; ++i) {
        const float ps = warp_sum(path[i]), js = warp_sum(jl[i]);
        if (lane == 0) { sh.part[w + i * kGrpWarps<kPpc>][0] = ps; sh.part[w + i * kGrpWarps<kPpc>][1] = js; }
    }
    grp_sync<kPpc>();
    if (tid == 0) {
        float p = 0.f, l = 0.f;
        for (int i = 0; i < kTWarps; ++i) { p += sh.part[i][0]; l += sh.part[i][1]; }
        sh.path = p;
        sh.jl = l;
        sh.L += sc.w_path * p + sc.w_jl * l;
    }
    // no barrier: only thread 0 reads sh.path, sh.jl and sh.L afterwards
}

// Boxes of a problem's environment by `threads` threads (tid of them); its tables are already in
// shared memory.  The caller's next barrier orders the writes.
__device__ __forceinline__ void env_setup(const TrajScalars& sc, unsigned char* env, int tid, int threads) {
    const float4* cub = reinterpret_cast<const float4*>(env + t_env_offset());
    const float4* osph = cub + 4 * sc.n_cub;
    float4* aabb = reinterpret_cast<float4*>(env + t_aabb_offset(sc.n_cub, sc.n_osph));
    const int n_cw = t_cub_words(sc.n_cub), n_w = t_words(sc.n_cub, sc.n_osph);
#pragma unroll 1
    for (int i = tid; i < 32 * (n_w - 1); i += threads) {
        const int o = i - 32 * n_cw;   // environment sphere
        float4* box = &aabb[2 * i];
        if (i < sc.n_cub) {
            cuboid_aabb(&cub[4 * i], box);
        } else if (o >= 0 && o < sc.n_osph) {
            const float4 sp = osph[o];
            box[0] = make_float4(sp.x - sp.w, sp.y - sp.w, sp.z - sp.w, 0.f);
            box[1] = make_float4(sp.x + sp.w, sp.y + sp.w, sp.z + sp.w, 0.f);
        } else {
            empty_box(box);
        }
    }
}

// Constants of a problem in its group's region that its particles share: the cuboids of the
// blocks at their initial poses (the placed ones empty), the kinematic rows.
template <int kPpc>
__device__ __forceinline__ void group_setup(const TrajScalars& sc, TShared& sh) {
    const int tid = grp_tid<kPpc>();
    if (tid < 2 * kMaxB) {
        const int k = tid - kMaxB;
        if (k >= 0 && k < sc.B) {
            block_cuboid(sc.init[k].x, sc.init[k].y, sc.init[k].z, sc.init[k].w, sc.half[k], sh.blk[tid]);
            cuboid_aabb(sh.blk[tid], sh.bbox[tid]);
        } else {
            empty_box(sh.bbox[tid]);
        }
    }
    if (tid == 0) sh.inv_S = 1.f / (float)sc.S;
    if (tid < kMaxB) sh.inv_above[tid] = tid + 1 < sc.B ? 1.f / (float)(sc.B - 1 - tid) : 0.f;
    if (tid < 8) {
        sh.dh[tid] = tid < 7 ? make_float4(sc.ca[tid], sc.sa[tid], sc.a[tid], sc.d[tid]) : make_float4(1.f, 0.f, 0.f, 0.f);
        sh.th0[tid] = tid < 7 ? sc.th0[tid] : 0.f;
        sh.lbc[tid] = sc.lbox_c[tid];
        sh.lbh[tid] = sc.lbox_h[tid];
    }
}

// One particle of the trajectory stage by a group: load its state, run the descent (or the
// single evaluation), write the outputs.  The problem's constants are already in shared memory
// (env_setup, group_setup).  rows: the group's slot of the collision gradient rows.
template <bool kP2P, int kTile, int kPpc>
__device__ __forceinline__ void traj_particle(const TrajScalars& sc, const LaneSpheres& ls, int p, int mode,
                                              const TrajIO& io, float* rows, const unsigned char* env,
                                              unsigned char* region) {
    constexpr int kThreads = kGrpThreads<kPpc>, kWarps = kGrpWarps<kPpc>;
    const float4* cub = reinterpret_cast<const float4*>(env + t_env_offset());
    const float4* osph = cub + 4 * sc.n_cub;
    const float4* aabb = reinterpret_cast<const float4*>(env + t_aabb_offset(sc.n_cub, sc.n_osph));
    TShared& sh = *reinterpret_cast<TShared*>(region);
    TWarp* tws = reinterpret_cast<TWarp*>(region + t_warp_offset());
    float* q = reinterpret_cast<float*>(region + t_q_offset(kWarps));
    SpecialFrames* sp = reinterpret_cast<SpecialFrames*>(region + t_sp_offset(sc.C, kWarps));
    float* disp = reinterpret_cast<float*>(region + t_cache_offset(sc.C, sc.B, kWarps));
    const int n_chunks = t_n_chunks(sc.C);
    float* cblk = disp + sc.C;
    __half2* cgap = reinterpret_cast<__half2*>(cblk + n_chunks);   // (static, moving) clearances
    float* ctopm = reinterpret_cast<float*>(cgap + n_chunks);    // the top block's own motion at the cull
    __half* ctop = reinterpret_cast<__half*>(ctopm + n_chunks);  // clearance to the top block
    unsigned char* state = reinterpret_cast<unsigned char*>(ctop + n_chunks);
    const int tid = grp_tid<kPpc>();
    const int C = sc.C, NR = sc.NR;
#pragma unroll 1
    for (int i = tid; i < C; i += kThreads) disp[i] = 0.f;
#pragma unroll 1
    for (int i = tid; i < n_chunks; i += kThreads) {
        cblk[i] = 0.f; cgap[i] = __float2half2_rn(0.f); state[i] = kChunk; ctopm[i] = 0.f; ctop[i] = __float2half_rn(0.f);
    }
    if (tid < kMaxB) { sh.blk_cum[tid] = 0.f; sh.bown[tid] = 0.f; }
    if (tid == 0) sh.pose_prev_ok = 0;

    // particle state -> shared memory (coalesced float4)
    const float4* qg = reinterpret_cast<const float4*>(io.q + (size_t)p * C * 8);
    float4* qs = reinterpret_cast<float4*>(q);
#pragma unroll 4
    for (int i = tid; i < C * 2; i += kThreads) qs[i] = qg[i];
    if (tid < 3 * kWarps) tws[tid / 3].count[tid % 3] = 0ull;
    const bool fresh = mode == kTrajDescend && io.init_multipliers;
#pragma unroll 1
    for (int r = tid; r < NR; r += kThreads) {
        sh.lam[r] = (fresh || !io.lam) ? 0.f : io.lam[(size_t)p * NR + r];
    }
    if (tid == 0) sh.mu = (fresh || !io.mu) ? sc.mu0 : io.mu[p];
    grp_sync<kPpc>();

    // K descent iterations (evaluation with gradient, update), then the final evaluation: one
    // call site of each, so that their code is inlined once
    const bool want_grad = mode == kTrajEval && io.grad != nullptr;
    float* grad_out = want_grad ? io.grad + (size_t)p * C * 8 : nullptr;
    const int K = mode == kTrajDescend ? io.k_steps : 0;
    for (int k = 1;; ++k) {
        const bool last = k > K;
        traj_evaluate<kP2P, kTile, kPpc>(sc, ls, cub, osph, aabb, sh, tws, sp, q, rows, disp, cblk, cgap, state, ctopm, ctop,
                                         last ? want_grad : true, last);
        if (!last || want_grad)
            traj_step<kP2P, kPpc>(sc, sh, tws, sp, q, rows, disp, sc.eta_traj * (1.f - (float)k / (float)K),
                            last || k == 1 || !(sc.w_jl * 0.f == 0.f), last ? grad_out : nullptr);
        if (last) break;
        if (sc.K_al > 0 && k % sc.K_al == 0) {
#pragma unroll 1
            for (int r = tid; r < NR; r += kThreads) sh.lam[r] += sh.mu * residual_sqrt_weight(sc, r) * sh.h[r];
            grp_sync<kPpc>();
            if (tid == 0) sh.mu = fminf(sh.mu * 2.f, sc.mu_max);
        }
        grp_sync<kPpc>();
    }
    traj_path<kPpc>(sc, sh, q);
    if (io.tests && tid < 3) {   // after the barrier in traj_path
        unsigned long long c = 0ull;
        for (int i = 0; i < kWarps; ++i) c += tws[i].count[tid];
        atomicAdd(io.tests + tid, c);
    }

    // outputs
    if (mode == kTrajDescend) {
        float4* qo = reinterpret_cast<float4*>(io.q + (size_t)p * C * 8);
#pragma unroll 1
        for (int i = tid; i < C * 2; i += kThreads) qo[i] = qs[i];
        if (io.lam)
#pragma unroll 1
            for (int r = tid; r < NR; r += kThreads) io.lam[(size_t)p * NR + r] = sh.lam[r];
        if (io.mu && tid == 0) io.mu[p] = sh.mu;
    }
    if (io.h)
#pragma unroll 1
        for (int r = tid; r < NR; r += kThreads) io.h[(size_t)p * NR + r] = sh.h[r];
    if (tid == 0) {
        if (io.L) io.L[p] = sh.L;
        if (io.groups) {
            float* g = io.groups + (size_t)p * 6;
            g[0] = sh.c_start; g[1] = sh.c_arm; g[2] = sh.c_blk; g[3] = sh.c_coll; g[4] = sh.c_stable; g[5] = sh.c_height;
        }
        const float rank = sc.w_path * sh.path + sc.w_stable * sh.c_stable + sc.w_height * sh.c_height +
                           sc.w_coll * sh.c_coll + sc.w_start * sh.c_start + sc.w_arm * sh.c_arm + sc.w_block * sh.c_blk;
        if (io.metrics) {
            float* m = io.metrics + (size_t)p * 8;
            m[0] = sh.maxpen; m[1] = sh.max_start; m[2] = sh.max_tilt; m[3] = sh.pm_pen; m[4] = sh.pm_D;
            m[5] = sh.pm_dz; m[6] = sh.path; m[7] = rank;
        }
        if (io.sat) {
            const bool ok = sh.maxpen <= sc.eps && sh.max_start <= sc.eps_start && sh.max_tilt <= sc.eps_start &&
                            sh.pm_pen <= sc.eps && sh.pm_D <= sc.eps && sh.pm_dz <= sc.eps && sh.jl == 0.f;
            io.sat[p] = ok ? 1 : 0;
        }
    }
}

// Bulk-copy staging of the environment tables into one group's region, with the group's own
// barrier: stage_tables for a group's threads (the bounded wait, the error word, a
// second bounded wait for copies in flight after a timeout).  `init`: first use of the
// group's mbarrier; `phase`: the parity this copy completes.
template <int kPpc>
__device__ __forceinline__ bool stage_tables_grp(void* dst0, const void* src0, uint32_t bytes0, void* dst1,
                                                 const void* src1, uint32_t bytes1, uint64_t* bar, int* err,
                                                 bool init = true, uint32_t phase = 0) {
    volatile uint32_t* okw = reinterpret_cast<volatile uint32_t*>(bar + 1);   // the region header's second word
    if (grp_tid<kPpc>() == 0) {
        if (init) {
            mbar_init(bar, 1);
            fence_mbar_init();
        }
        *okw = 1u;
    }
    // the copies write, through the async proxy, memory that the group has read and written before (the
    // last problem's tables, boxes and state): each thread's accesses are ordered before them
    fence_proxy_async();
    grp_sync<kPpc>();
    if (grp_tid<kPpc>() == 0) {
        mbar_expect_tx(bar, bytes0 + bytes1);
        if (bytes0) bulk_g2s(dst0, src0, bytes0, bar);
        if (bytes1) bulk_g2s(dst1, src1, bytes1, bar);
    }
    const bool done = mbar_wait_bounded(bar, phase, kTablePolls);
    if (!done) {
        set_error(err, kDevTimeout);
        mbar_wait_bounded(bar, phase, kTablePolls);
        *okw = 0u;
    }
    grp_sync<kPpc>();
    const bool all = *okw != 0u;
    grp_sync<kPpc>();   // every thread has read the flag before a later call resets it
    return all;
}

// Persistent grid over n particles, kPpc groups per CTA: a group starts with particle = its
// index and takes the next one from the work counter when it is done, so that particles of
// uneven length keep every group busy to the end; the group that finishes last leaves the
// counters at zero for the next launch.  The problem's tables are staged once per CTA, its
// constants once per group.  (kP2P: the point-to-point instantiation; kTile: the sphere tiling.)
// A launch without scratch (io.rows and io.work null) has a group per particle and its gradient
// rows in shared memory, so that nothing of it is shared with any other launch.
template <bool kP2P, int kTile, int kPpc>
__global__ void __launch_bounds__(kTThreads, 2) k_traj(const __grid_constant__ Scalars sc, DevTables tab, int n, int mode,
                                                       TrajIO io, int* err, int region_bytes) {
    extern __shared__ __align__(16) unsigned char smem_all[];
    if (io.active && *io.active <= 0) return;   // stage 1 of this problem found no placement
    // the environment, which the CTA's groups share, then their regions
    unsigned char* region = smem_all + t_env_bytes(sc.n_cub, sc.n_osph) + (size_t)grp_index<kPpc>() * region_bytes;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_all);
    float4* cub = reinterpret_cast<float4*>(smem_all + t_env_offset());
    float4* osph = cub + 4 * sc.n_cub;
    TShared& sh = *reinterpret_cast<TShared*>(region);
    const int groups = gridDim.x * kPpc, slot = blockIdx.x * kPpc + grp_index<kPpc>();
    if (stage_tables(cub, tab.cub, (uint32_t)sc.n_cub * 64u, osph, tab.osph, (uint32_t)sc.n_osph * 16u, bar, err)) {
        env_setup(sc, smem_all, threadIdx.x, kTThreads);
        group_setup<kPpc>(sc, sh);
        __syncthreads();
        const LaneSpheres ls = lane_spheres<kTile>(sc);
        float* rows = io.rows ? io.rows + (size_t)slot * sc.C * 16
                              : reinterpret_cast<float*>(region + region_bytes - t_rows_bytes(sc.C));
        for (int p = slot; p < n;) {
            traj_particle<kP2P, kTile, kPpc>(sc, ls, p, mode, io, rows, smem_all, region);
            if (!io.work) break;
            if (grp_tid<kPpc>() == 0) sh.particle = groups + atomicAdd(&io.work->next, 1);
            grp_sync<kPpc>();   // also: the outputs were read from the region before the next particle fills it
            p = sh.particle;
        }
    }
    if (io.work && grp_tid<kPpc>() == 0) {
        __threadfence();
        if (atomicAdd(&io.work->done, 1) == groups - 1) {
            __threadfence();
            io.work->next = 0;
            io.work->done = 0;
        }
    }
}

static_assert(sizeof(TrajScalars) % 16 == 0, "the batched kernel copies TrajScalars in 16-byte words");

// Batched form: a persistent grid over the particles of several problems.  Work items are
// runs of `per_fetch` consecutive particles of one problem, numbered problem after problem
// (jobs[j].first is the first item of problem j); each group (kPpc per CTA) takes the next
// item from *next until none is left.  On a change of problem the group stages that
// problem's constants and tables into its shared memory.  Every particle runs exactly the
// code of k_traj, so results equal the single-problem launches bit for bit, whatever the
// schedule.
template <int kTile, int kPpc>
__global__ void __launch_bounds__(kTThreads, 2) k_traj_batch(const TrajJob* __restrict__ jobs, int n_jobs, int n_items,
                                                             int per_fetch, int mode, int* next, int group_bytes) {
    extern __shared__ __align__(16) unsigned char smem_all[];
    __shared__ __align__(16) TrajScalars sc_arr[kPpc];
    __shared__ TrajIO io_arr[kPpc];
    __shared__ int s_item[kPpc], s_job[kPpc];
    const int g = grp_index<kPpc>(), tid = grp_tid<kPpc>();
    unsigned char* env = smem_all + (size_t)g * group_bytes;   // the group's environment, then its region
    unsigned char* region = env;
    TrajScalars& sc_s = sc_arr[g];
    TrajIO& io_s = io_arr[g];
    uint64_t* bar = reinterpret_cast<uint64_t*>(env);
    int cur = -1;
    uint32_t uses = 0;
    for (;;) {
        if (tid == 0) {
            const int it = atomicAdd(next, 1);
            int j = -1;
            if (it < n_items) {   // last job whose first item is <= it
                int lo = 0, hi = n_jobs - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (jobs[mid].first <= it) lo = mid; else hi = mid - 1;
                }
                j = lo;
            }
            s_item[g] = it;
            s_job[g] = j;
        }
        grp_sync<kPpc>();
        const int it = s_item[g], j = s_job[g];
        // every thread has the item before thread 0 takes the next one: an item of the same problem that
        // has no particle to run (a problem without a placement) meets no other barrier on its way there
        grp_sync<kPpc>();
        if (j < 0) break;
        const TrajJob& job = jobs[j];
        if (j != cur) {
            // stage the problem's constants (int4 words) and its tables
            const int4* src = reinterpret_cast<const int4*>(static_cast<const TrajScalars*>(job.sc));
            int4* dst = reinterpret_cast<int4*>(&sc_s);
            for (int i = tid; i < (int)(sizeof(TrajScalars) / 16); i += kGrpThreads<kPpc>) dst[i] = src[i];
            if (tid == 0) io_s = job.io;
            grp_sync<kPpc>();
            float4* cub = reinterpret_cast<float4*>(env + t_env_offset());
            float4* osph = cub + 4 * sc_s.n_cub;
            if (!stage_tables_grp<kPpc>(cub, job.tab.cub, (uint32_t)sc_s.n_cub * 64u, osph, job.tab.osph,
                                  (uint32_t)sc_s.n_osph * 16u, bar, job.err, uses == 0, uses & 1u))
                return;
            region = env + t_env_bytes(sc_s.n_cub, sc_s.n_osph);
            env_setup(sc_s, env, tid, kGrpThreads<kPpc>);   // ordered by the first barrier of traj_particle
            group_setup<kPpc>(sc_s, *reinterpret_cast<TShared*>(region));
            ++uses;
            cur = j;
        }
        const LaneSpheres ls = lane_spheres<kTile>(*job.sc);
        float* rows = io_s.rows + (size_t)(blockIdx.x * kPpc + g) * io_s.row_stride;
        const int p0 = (it - job.first) * per_fetch;
        // a problem whose stage 1 found no placement has nothing to optimise
        const int p1 = (io_s.active && *io_s.active <= 0) ? p0 : min(p0 + per_fetch, job.n);
        for (int p = p0; p < p1; ++p) {
            if (sc_s.kind == kKindP2P) traj_particle<true, kTile, kPpc>(sc_s, ls, p, mode, io_s, rows, env, region);
            else traj_particle<false, kTile, kPpc>(sc_s, ls, p, mode, io_s, rows, env, region);
            grp_sync<kPpc>();
        }
    }
}

// ================================================================================== launchers
// Two CTAs per SM share its shared memory; each has 1 KB of it reserved by the system.
static cudaError_t sm_limits(int* sms, size_t* half_smem) {
    int dev = 0, smem = 0, reserved = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    *half_smem = e == cudaSuccess ? (size_t)(smem / 2 - reserved) : 0;
    return e;
}

// Particles per CTA where the caller leaves the choice.  More than one when the launch has more
// particles than the SMs then hold (2 CTAs per SM) and two such CTAs fit an SM; otherwise
// fewer, on more warps each (fewer particles: each finishes sooner; larger regions: an SM would
// hold one CTA, 8 warps in place of 16).
// Towers of more than kAutoBlocks blocks keep one: their phases run through more of the kernel's
// code at a time, and four particles in different phases miss the instruction cache.  4096
// particles among 64 cuboids, 50 steps, one / two per CTA, ms: 2 blocks 4.1 / 2.8, 4 blocks
// 5.6 / 4.1, 6 blocks 7.6 / 6.7, 8 blocks 9.5 / 9.9, 10 blocks 13.8 / 17.7.
// Four take short trajectories (kShortC configurations; 1 block, 31 configurations, 700 / 4096
// particles, two / four per CTA: 0.56 / 0.35 and 1.94 / 1.30 ms), and longer ones up to kMidC when
// the launch has several rounds of them, as a particle on two warps runs long and the last ones
// run alone (3 blocks, 187 configurations, 4096 particles: 3.44 / 2.70 ms; at 2048, where the line
// keeps two, 1.91 / 1.55, but 2.86 / 3.33 where more of the chunks have candidates).
// cta_bytes_2, cta_bytes_4: the shared memory of a CTA with 2 or 4 particles (0: not to be used).
constexpr int kAutoBlocks = 6, kShortC = 48, kMidC = 192;
int traj_auto_ppc(size_t cta_bytes_2, size_t cta_bytes_4, long long particles, int blocks, int C) {
    int sms = 0;
    size_t half = 0;
    if (sm_limits(&sms, &half) != cudaSuccess || blocks > kAutoBlocks) return 1;
    const bool four = C <= kShortC ? particles > 4LL * sms : C <= kMidC && particles > 16LL * sms;
    if (cta_bytes_4 && four && cta_bytes_4 <= std::min(half, kHalfSmem)) return 4;
    return cta_bytes_2 && particles > 2LL * sms && cta_bytes_2 <= half ? 2 : 1;
}

template <int kTile, int kPpc>
static cudaError_t batch_kernel(const TrajJob* jobs, int n_jobs, int n_items, int per_fetch, int mode, int* next,
                                size_t dyn, int grid, cudaStream_t st) {
    cudaError_t e = allow_max_dynamic_smem(k_traj_batch<kTile, kPpc>, dyn);
    if (e != cudaSuccess) return e;
    k_traj_batch<kTile, kPpc><<<grid, kTThreads, dyn, st>>>(jobs, n_jobs, n_items, per_fetch, mode, next, (int)(dyn / kPpc));
    return cudaGetLastError();
}

cudaError_t launch_traj_batch(const TrajJob* jobs, int n_jobs, int n_items, int per_fetch, int mode, int* next,
                              size_t cta_bytes, int grid, cudaStream_t st, int tiling, int ppc) {
    if (n_items <= 0) return cudaSuccess;
    if (ppc == 2)
        return tiling ? batch_kernel<1, 2>(jobs, n_jobs, n_items, per_fetch, mode, next, cta_bytes, grid, st)
                      : batch_kernel<0, 2>(jobs, n_jobs, n_items, per_fetch, mode, next, cta_bytes, grid, st);
    return tiling ? batch_kernel<1, 1>(jobs, n_jobs, n_items, per_fetch, mode, next, cta_bytes, grid, st)
                  : batch_kernel<0, 1>(jobs, n_jobs, n_items, per_fetch, mode, next, cta_bytes, grid, st);
}

template <typename K>
static int occupancy(K kernel, size_t dyn) {
    int n = 0;
    if (allow_max_dynamic_smem(kernel, dyn) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kTThreads, dyn) != cudaSuccess) return 0;
    return n;
}

int traj_batch_ctas_per_sm(size_t cta_bytes, int tiling, int ppc) {
    if (ppc == 2) return tiling ? occupancy(k_traj_batch<1, 2>, cta_bytes) : occupancy(k_traj_batch<0, 2>, cta_bytes);
    return tiling ? occupancy(k_traj_batch<1, 1>, cta_bytes) : occupancy(k_traj_batch<0, 1>, cta_bytes);
}

int traj_ppc(const TrajScalars& sc, long long particles) {
    if (sc.particles_per_cta) return sc.particles_per_cta;
    // point to point keeps two: its chunks, all near obstacles, are long for two warps, unless they are
    // few (50 steps, 1024 / 4096 particles, two / four per CTA, ms: 32 configurations 1.57 / 1.80 and
    // 4.46 / 4.28, 64 configurations 2.73 / 2.91 and 8.27 / 7.93, 8 configurations 0.53 / 0.39 and
    // 1.59 / 1.03)
    const bool four = !sc.sphere_tiling && sc.kind != kKindP2P;
    return traj_auto_ppc(traj_cta_smem_bytes(sc, 2, false), four ? traj_cta_smem_bytes(sc, 4, false) : 0, particles, sc.B,
                         sc.C);
}

template <bool kP2P>
static int single_ctas(size_t dyn, int tiling, int ppc) {
    if constexpr (!kP2P)   // point to point never takes four (traj_ppc)
        if (ppc == 4) return occupancy(k_traj<false, 0, 4>, dyn);
    if (ppc == 2) return tiling ? occupancy(k_traj<kP2P, 1, 2>, dyn) : occupancy(k_traj<kP2P, 0, 2>, dyn);
    return tiling ? occupancy(k_traj<kP2P, 1, 1>, dyn) : occupancy(k_traj<kP2P, 0, 1>, dyn);
}

int traj_ctas_per_sm(const TrajScalars& sc) {
    const int ppc = traj_ppc(sc, sc.Q);
    const size_t dyn = traj_cta_smem_bytes(sc, ppc, false);
    return sc.kind == kKindP2P ? single_ctas<true>(dyn, sc.sphere_tiling, ppc)
                               : single_ctas<false>(dyn, sc.sphere_tiling, ppc);
}

template <bool kP2P, int kTile, int kPpc>
static cudaError_t traj_kernel(const Scalars& sc, DevTables t, int n, int mode, const TrajIO& io, int* err,
                               cudaStream_t st) {
    const size_t region = t_region(sc.C, sc.B, kPpc) + (io.rows ? 0 : t_rows_bytes(sc.C));
    const size_t dyn = t_env_bytes(sc.n_cub, sc.n_osph) + kPpc * region;
    int sms = 0;
    size_t half = 0;
    cudaError_t e = sm_limits(&sms, &half);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_traj<kP2P, kTile, kPpc>, dyn);
    if (e != cudaSuccess) return e;
    const int resident = std::min(sms * (dyn <= half ? 2 : 1), traj_slots(sc.B, sc.C, sc.n_cub, sc.n_osph) / kPpc);
    const int all = (n + kPpc - 1) / kPpc, grid = io.rows ? std::min(all, resident) : all;
    k_traj<kP2P, kTile, kPpc><<<grid, kTThreads, dyn, st>>>(sc, t, n, mode, io, err, (int)region);
    return cudaGetLastError();
}

template <bool kP2P>
static cudaError_t traj_dispatch(const Scalars& sc, DevTables t, int n, int mode, const TrajIO& io, int* err,
                                 cudaStream_t st) {
    int ppc = traj_ppc(sc, n);
    if (!io.rows) {   // with their rows in shared memory fewer particles share a CTA
        const size_t env = t_env_bytes(sc.n_cub, sc.n_osph), rows = t_rows_bytes(sc.C);
        while (ppc > 1 && env + ppc * (t_region(sc.C, sc.B, ppc) + rows) > kHalfSmem) ppc /= 2;
    }
    if constexpr (!kP2P)
        if (ppc == 4) return traj_kernel<false, 0, 4>(sc, t, n, mode, io, err, st);
    if (ppc == 2)
        return sc.sphere_tiling ? traj_kernel<kP2P, 1, 2>(sc, t, n, mode, io, err, st)
                                : traj_kernel<kP2P, 0, 2>(sc, t, n, mode, io, err, st);
    return sc.sphere_tiling ? traj_kernel<kP2P, 1, 1>(sc, t, n, mode, io, err, st)
                            : traj_kernel<kP2P, 0, 1>(sc, t, n, mode, io, err, st);
}

cudaError_t launch_traj(const Scalars& sc, DevTables t, int n, int mode, const TrajIO& io, int* err,
                        cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    return sc.kind == kKindP2P ? traj_dispatch<true>(sc, t, n, mode, io, err, st)
                               : traj_dispatch<false>(sc, t, n, mode, io, err, st);
}

}  // namespace spasm
