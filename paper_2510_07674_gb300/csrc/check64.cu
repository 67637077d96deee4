// FP64 feasibility check of returned trajectories (GetSatisfyingParticles applied to the
// final solutions, |f(x)| < eps of Sec. III), evaluated in double precision on the
// float32 joint values the optimiser returned.
//
// The verdict needs the largest arm / held-block penetration over every configuration, sphere
// and obstacle, and double precision runs at a sixty-fourth of the FP32 rate here (all of it in
// FP64: 790 us for 32 trajectories of the 10-block tower, with the FP64 pipe the limit).  So it
// is done in two passes:
//   k_check_screen  evaluates every configuration in FP32 (a warp takes four at a time) and keeps
//                   each configuration's largest value, signed: r - distance, positive inside.
//                   One more CTA per solution computes, in FP64, the placed poses and the grasp,
//                   tilt and placement metrics meanwhile.
//   k_check64       repeats in FP64 the configurations whose FP32 value is within twice the
//                   margin of the solution's largest (and above minus the margin: below, nothing
//                   is penetrated), a warp per configuration; usually one or two of 620.
// The margin bounds the FP32 evaluation's error (Scalars64::margin, some hundred rounding steps of
// the scene's extent, more where the joints have offsets), so the configuration that holds the FP64
// maximum is always among those repeated, and the metrics are those of the full FP64 evaluation:
// 85 us for the same 32 (the screen 55, beside the FP64 metrics' latency, the second pass 31).
// Configurations with a joint too large for an FP32 angle, or NaN, are repeated always, and so are
// those that can touch a placed block whose pose FP32 does not give to the margin: its place
// configuration has such a joint, or holds the block's x axis near the vertical, where the yaw
// amplifies the rotation's rounding without bound.
#include "check64.h"
#include "stage2.cuh"

namespace spasm {

__device__ __forceinline__ void held64(const Scalars64& s, int b, const double Rt[9], const double pt[3], double Rb[9],
                                       double pb[3]) {
    const double off = s.half[b][2] + s.grasp_off;
    for (int i = 0; i < 3; ++i) {
        Rb[3 * i] = Rt[3 * i];
        Rb[3 * i + 1] = -Rt[3 * i + 1];
        Rb[3 * i + 2] = -Rt[3 * i + 2];
        pb[i] = pt[i] + off * Rt[3 * i + 2];
    }
}

__device__ __forceinline__ void tool64(const Scalars64& s, const double R7[9], const double o7[3], double Rt[9], double pt[3]) {
    for (int i = 0; i < 3; ++i) {
        for (int j = 0; j < 3; ++j)
            Rt[3 * i + j] = R7[3 * i] * s.ee_R[j] + R7[3 * i + 1] * s.ee_R[3 + j] + R7[3 * i + 2] * s.ee_R[6 + j];
        pt[i] = o7[i] + R7[3 * i] * s.ee_p[0] + R7[3 * i + 1] * s.ee_p[1] + R7[3 * i + 2] * s.ee_p[2];
    }
}

struct D4 { double x, y, z, w; };

// Cuboid of a block placed at p (x, y, z) with the cosine and sine of its yaw.
__device__ __forceinline__ void block_cub64(const double* p, double cs, double sn, const double h[3], D4 c[4]) {
    c[0] = D4{p[0], p[1], p[2], 0.0};
    c[1] = D4{cs, sn, 0.0, h[0]};
    c[2] = D4{-sn, cs, 0.0, h[1]};
    c[3] = D4{0.0, 0.0, 1.0, h[2]};
}

__device__ __forceinline__ double pen_cub64(double cx, double cy, double cz, double r, const D4* c) {
    double gx, gy, gz;
    return pen_cuboid<double>(cx, cy, cz, r, c[0], c[1], c[2], c[3], gx, gy, gz);
}

// r minus the distance of (x, y, z) from the cuboid c in FP32, positive inside (r plus the depth).
__device__ __forceinline__ float value32(float x, float y, float z, float r, const float4* c) {
    const float4 o0 = c[0], o1 = c[1], o2 = c[2], o3 = c[3];
    float p0, p1, p2, q0, q1, q2;
    const float qm = cub_local<float>(x, y, z, o0, o1, o2, o3, p0, p1, p2, q0, q1, q2);
    const float m0 = fmaxf(q0, 0.f), m1 = fmaxf(q1, 0.f), m2 = fmaxf(q2, 0.f);
    return r - (qm > 0.f ? sqrtf(m0 * m0 + m1 * m1 + m2 * m2) : qm);
}

// Floats in an order that unsigned integers keep (for atomicMax); 0 is below every float.
__device__ __forceinline__ unsigned float_key(float v) {
    const unsigned u = __float_as_uint(v);
    return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float key_float(unsigned k) {
    return __uint_as_float(k & 0x80000000u ? k & 0x7fffffffu : ~k);
}

constexpr int kScrThreads = 256, kScrWarps = kScrThreads / 32;
constexpr int kScrCfgs = 4 * kScrWarps;   // configurations per CTA of the screen
constexpr int kChkThreads = 128, kChkWarps = kChkThreads / 32;
constexpr float kNone = -3.4e38f;         // no obstacle within the margin
constexpr float kMaxAngle = 8.f;          // largest joint value the FP32 evaluation takes

struct ScreenWarp {
    float4 F[4][8][3];   // frames 0..7 of the warp's configurations: rows (R_i0, R_i1, R_i2, o_i)
    float4 H[4][3];      // held-block frames
};
struct ScreenShared {
    ScreenWarp warp[kScrWarps];
    float4 blk[2 * kMaxB][4];   // block cuboids: k placed, 16 + k at the initial pose
    float4 box[kMaxCub + kMaxOSph + 2 * kMaxB][2];   // boxes: environment, then the blocks
    unsigned loose;             // bit k: FP32 does not give the pose of placed block k
};

__device__ __forceinline__ void cuboid_box(const float4* c, float4* box) {
    const float ex = fabsf(c[1].x) * c[1].w + fabsf(c[2].x) * c[2].w + fabsf(c[3].x) * c[3].w;
    const float ey = fabsf(c[1].y) * c[1].w + fabsf(c[2].y) * c[2].w + fabsf(c[3].y) * c[3].w;
    const float ez = fabsf(c[1].z) * c[1].w + fabsf(c[2].z) * c[2].w + fabsf(c[3].z) * c[3].w;
    box[0] = make_float4(c[0].x - ex, c[0].y - ey, c[0].z - ez, 0.f);
    box[1] = make_float4(c[0].x + ex, c[0].y + ey, c[0].z + ez, 0.f);
}

// Kinematics of four configurations by one warp: lane 8 c + k takes the sine and cosine of joint
// k - 1 of configuration c, every lane of the eight runs the chain, and lane 8 c + k keeps frame k
// (R, o).
template <typename T, typename SC>
__device__ __forceinline__ void fk_lanes(const SC& s, T sn, T cs, T R[9], T o[3]) {
    const int lane = threadIdx.x & 31, k = lane & 7, base = lane & ~7;
    T A[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1}, b[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < 9; ++i) R[i] = A[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) o[i] = b[i];
#pragma unroll 1
    for (int j = 0; j < 7; ++j) {
        const T sj = __shfl_sync(0xffffffffu, sn, base + j + 1), cj = __shfl_sync(0xffffffffu, cs, base + j + 1);
        dh_step<T>(A, b, (T)s.ca[j], (T)s.sa[j], (T)s.a[j], (T)s.d[j], cj, sj);
        if (k == j + 1) {
#pragma unroll
            for (int i = 0; i < 9; ++i) R[i] = A[i];
#pragma unroll
            for (int i = 0; i < 3; ++i) o[i] = b[i];
        }
    }
}

// FP64: the placed poses of solution r (for the second pass) and its grasp, tilt and placement
// metrics, by one CTA: eight lanes per grasp or place configuration, then a thread per sphere of
// the placed blocks.
__device__ void solution_metrics(const Scalars64& s, const D4* __restrict__ cub, const D4* __restrict__ osph,
                                 const float4* __restrict__ fcub, const float* __restrict__ qr, CheckAcc& A) {
    __shared__ double pose[kMaxB][5];   // x, y, z, cos yaw, sin yaw
    __shared__ double trig[2 * kMaxB][7][2];   // (sin, cos) of the joints of each grasp and place configuration
    __shared__ double vs[kMaxB], vt[kMaxB], vD[kMaxB], vz[kMaxB], pen[kScrWarps];
    const int tid = threadIdx.x, lane = tid & 31, B = s.B, S = s.S;
    static_assert(kScrThreads / 8 >= 2 * kMaxB, "a group of eight lanes per grasp and place configuration");
    // sines and cosines a thread per joint, then a lane per configuration: FP64 issues two lanes a
    // cycle whatever the mask, so a lane that repeats another's work costs as much as one of its own
    const int n_sp = s.p2p ? 1 : 2 * B;
    static_assert(kScrThreads >= 14 * kMaxB, "a thread per joint of the grasp and place configurations");
    if (tid < 7 * n_sp) {
        const int e = tid / 7, j = tid % 7;
        sincos(s.th0[j] + (double)qr[(e + 1) * S * 8 + j], &trig[e][j][0], &trig[e][j][1]);
    }
    __syncthreads();
    if (tid < n_sp) {
        const int b = tid >> 1;
        double R[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1}, o[3] = {0, 0, 0}, Rt[9], pt[3], Rb[9], pb[3];
#pragma unroll 1
        for (int j = 0; j < 7; ++j) dh_step<double>(R, o, s.ca[j], s.sa[j], s.a[j], s.d[j], trig[tid][j][1], trig[tid][j][0]);
        tool64(s, R, o, Rt, pt);
        held64(s, b, Rt, pt, Rb, pb);
        const double roll = atan2(Rb[7], Rb[8]), pitch = atan2(-Rb[6], sqrt(Rb[7] * Rb[7] + Rb[8] * Rb[8]));
        if (tid & 1) {
            double sy, cy;
            sincos(atan2(Rb[3], Rb[0]), &sy, &cy);
            pose[b][0] = pb[0]; pose[b][1] = pb[1]; pose[b][2] = pb[2]; pose[b][3] = cy; pose[b][4] = sy;
            vt[b] = roll * roll + pitch * pitch;
        } else {
            double e2 = 0.0;
            for (int i = 0; i < 3; ++i) { const double d = pb[i] - s.init[b][i]; e2 += d * d; }
            vs[b] = e2 + roll * roll + pitch * pitch;
        }
    }
    __syncthreads();
    if (tid < B) {
        const int b = tid;
        vD[b] = vz[b] = 0.0;
        if (s.p2p) {
            vt[b] = 0.0;
        } else {
            for (int i = 0; i < 5; ++i) A.pose[b][i] = pose[b][i];
            vz[b] = fabs(pose[b][2] - s.zt[b]);
            if (b + 1 < B) {
                double mx = 0.0, my = 0.0;
                for (int j = b + 1; j < B; ++j) { mx += pose[j][0]; my += pose[j][1]; }
                mx /= (double)(B - 1 - b);
                my /= (double)(B - 1 - b);
                const double cs = pose[b][3], sn = pose[b][4];
                const double vx = mx - pose[b][0], vy = my - pose[b][1];
                const double ux = cs * vx + sn * vy, uy = -sn * vx + cs * vy;
                const double ex = fmax(fabs(ux) - s.half[b][0], 0.0), ey = fmax(fabs(uy) - s.half[b][1], 0.0);
                vD[b] = sqrt(ex * ex + ey * ey);
            }
        }
    }
    // placement: spheres of block j vs the environment and the blocks below, the pairs that FP32 finds
    // within the margin
    double pp = 0.0;
    static_assert(kScrThreads >= 8 * kMaxB, "a thread per block sphere");
    if (!s.p2p && tid < 8 * B) {
        const int j = tid >> 3, m = tid & 7;
        const double lx = ((m & 1) ? 0.5 : -0.5) * s.half[j][0];
        const double ly = ((m & 2) ? 0.5 : -0.5) * s.half[j][1];
        const double lz = ((m & 4) ? 0.5 : -0.5) * s.half[j][2];
        const double cs = pose[j][3], sn = pose[j][4];
        const double cx = pose[j][0] + cs * lx - sn * ly, cy = pose[j][1] + sn * lx + cs * ly, cz = pose[j][2] + lz;
        const double rad = s.hmin[j] * 0.5;
        const float fx = (float)cx, fy = (float)cy, fz = (float)cz, fr = (float)rad;
#pragma unroll 1
        for (int ob = 0; ob < s.n_cub; ++ob)
            if (!(value32(fx, fy, fz, fr, fcub + 4 * ob) < -s.margin)) pp = fmax(pp, pen_cub64(cx, cy, cz, rad, &cub[4 * ob]));
#pragma unroll 1
        for (int ob = 0; ob < s.n_osph; ++ob) {
            double gx, gy, gz;
            pp = fmax(pp, pen_sphere<double>(cx, cy, cz, rad, osph[ob], gx, gy, gz));
        }
#pragma unroll 1
        for (int i = 0; i < j; ++i) {
            const float4 f[4] = {make_float4((float)pose[i][0], (float)pose[i][1], (float)pose[i][2], 0.f),
                                 make_float4((float)pose[i][3], (float)pose[i][4], 0.f, (float)s.half[i][0]),
                                 make_float4(-(float)pose[i][4], (float)pose[i][3], 0.f, (float)s.half[i][1]),
                                 make_float4(0.f, 0.f, 1.f, (float)s.half[i][2])};
            if (value32(fx, fy, fz, fr, f) < -s.margin) continue;
            D4 c[4];
            block_cub64(pose[i], pose[i][3], pose[i][4], s.half[i], c);
            pp = fmax(pp, pen_cub64(cx, cy, cz, rad, c));
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) pp = fmax(pp, __shfl_xor_sync(0xffffffffu, pp, off));
    if (lane == 0) pen[tid >> 5] = pp;
    __syncthreads();
    if (tid == 0) {
        double ms = 0.0, mt = 0.0, mD = 0.0, mz = 0.0;
        for (int b = 0; b < B; ++b) {
            ms = fmax(ms, vs[b]); mt = fmax(mt, vt[b]); mD = fmax(mD, vD[b]); mz = fmax(mz, vz[b]);
        }
        for (int w = 1; w < kScrWarps; ++w) pp = fmax(pp, pen[w]);
        A.pp = pp; A.ms = ms; A.mt = mt; A.mD = mD; A.mz = mz;
    }
}

// First pass: the first row of CTAs computes the solutions' metrics in FP64 (they take longest),
// the others screen their configurations in FP32.
__global__ void __launch_bounds__(kScrThreads) k_check_screen(const __grid_constant__ Scalars64 s,
                                                              const __grid_constant__ Scalars sc, DevTables tab,
                                                              const D4* __restrict__ cub, const D4* __restrict__ osph,
                                                              const float* __restrict__ q, const int* __restrict__ n_sol,
                                                              int P, float* __restrict__ val, CheckAcc* __restrict__ acc) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int r = blockIdx.x, slice = (int)blockIdx.y - 1;
    if (r >= (n_sol ? min(*n_sol, P) : P)) return;
    const int B = sc.B, S = sc.S, C = sc.C;
    const float* qr = q + (size_t)r * C * 8;
    if (slice < 0) {
        solution_metrics(s, cub, osph, tab.cub, qr, acc[r]);
        return;
    }
    ScreenShared& sh = *reinterpret_cast<ScreenShared*>(smem);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, k = lane & 7;
    ScreenWarp& W = sh.warp[w];
    const bool p2p = sc.kind == kKindP2P;
    const float margin = s.margin;
    const int n_env = sc.n_cub + sc.n_osph;

    // kinematics of configuration t (one per eight lanes): frame k of it, whether the lane's joint is
    // outside its limits, whether it is too large for FP32
    auto kinematics = [&](int t, float R[9], float o[3], bool& outside, bool& large) {
        float sn = 0.f, cs = 1.f;
        outside = large = false;
        if (k > 0) {
            const float v = qr[t * 8 + k - 1];
            outside = v < sc.qlo[k - 1] || v > sc.qhi[k - 1] || !isfinite(v);   // nothing else refuses a NaN
            large = !(fabsf(v) <= kMaxAngle);
            sincosf(sc.th0[k - 1] + v, &sn, &cs);
        }
        fk_lanes<float>(sc, sn, cs, R, o);
    };
    if (tid == 0) sh.loose = 0u;
    __syncthreads();
    // the blocks' cuboids and every obstacle's box
    if (!p2p) {
        for (int g = w; 4 * g < B; g += kScrWarps) {
            const int b = min(4 * g + (lane >> 3), B - 1);
            float R[9], o[3], Rt[9], pt[3], Rb[9], pb[3];
            bool outside, large;
            kinematics(t_place(S, b), R, o, outside, large);
            const unsigned joints = __ballot_sync(0xffffffffu, large) >> (lane & ~7) & 0xffu;
            if (k == 7) {
                tool_frame<float>(sc, R, o, Rt, pt);
                held_block<float>(sc, b, Rt, pt, Rb, pb);
                if (joints || !(Rb[0] * Rb[0] + Rb[3] * Rb[3] >= s.level2)) atomicOr(&sh.loose, 1u << b);
                block_cuboid(pb[0], pb[1], pb[2], atan2f(Rb[3], Rb[0]), sc.half[b], sh.blk[b]);
                cuboid_box(sh.blk[b], sh.box[n_env + b]);
            }
        }
        if (tid < B) {
            const float4 p = sc.init[tid];
            block_cuboid(p.x, p.y, p.z, p.w, sc.half[tid], sh.blk[kMaxB + tid]);
            cuboid_box(sh.blk[kMaxB + tid], sh.box[n_env + kMaxB + tid]);
        }
    }
    for (int i = tid; i < n_env; i += kScrThreads) {
        if (i < sc.n_cub) {
            cuboid_box(tab.cub + 4 * i, sh.box[i]);
        } else {
            const float4 v = tab.osph[i - sc.n_cub];
            sh.box[i][0] = make_float4(v.x - v.w, v.y - v.w, v.z - v.w, 0.f);
            sh.box[i][1] = make_float4(v.x + v.w, v.y + v.w, v.z + v.w, 0.f);
        }
    }
    __syncthreads();

    const int t0 = 1 + slice * kScrCfgs + 4 * w, nc = min(4, C - t0);
    if (nc <= 0) return;
    unsigned forced = 0u;
    {
        const int t = min(t0 + (lane >> 3), C - 1), seg = (t - 1) / S;
        float R[9], o[3];
        bool outside, large;
        kinematics(t, R, o, outside, large);
        if (__any_sync(0xffffffffu, outside) && lane == 0) atomicOr(&acc[r].viol, 1);
        forced = __ballot_sync(0xffffffffu, large);
#pragma unroll
        for (int i = 0; i < 3; ++i) W.F[lane >> 3][k][i] = make_float4(R[3 * i], R[3 * i + 1], R[3 * i + 2], o[i]);
        if (k == 7) {
            float Rt[9], pt[3], Rb[9], pb[3];
            tool_frame<float>(sc, R, o, Rt, pt);
            held_block<float>(sc, seg >> 1, Rt, pt, Rb, pb);
#pragma unroll
            for (int i = 0; i < 3; ++i) W.H[lane >> 3][i] = make_float4(Rb[3 * i], Rb[3 * i + 1], Rb[3 * i + 2], pb[i]);
        }
        __syncwarp();
    }
    const unsigned loose = sh.loose;
    float top = kNone;
#pragma unroll 1
    for (int ci = 0; ci < nc; ++ci) {
        const int t = t0 + ci, seg = (t - 1) / S, b = seg >> 1;
        const bool held = (seg & 1) && t - seg * S < S;
        const int n_items = sc.n_rsph + (held ? 8 : 0);
        // lanes own spheres: items lane and lane + 32 (the held block's after the robot's)
        float cx[2], cy[2], cz[2], rr[2];
        float lo[3] = {3.4e38f, 3.4e38f, 3.4e38f}, hi[3] = {-3.4e38f, -3.4e38f, -3.4e38f};
#pragma unroll
        for (int sl = 0; sl < 2; ++sl) {
            const int it = lane + 32 * sl;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4* f = W.H[ci];
            if (it < sc.n_rsph) {
                v = sc.rsph[it];
                f = W.F[ci][sc.rlink[it]];
            } else if (it < n_items) {
                block_sphere_local(sc.half[b], it - sc.n_rsph, v.x, v.y, v.z);
                v.w = sc.half[b].w;
            }
            const float4 r0 = f[0], r1 = f[1], r2 = f[2];
            cx[sl] = r0.x * v.x + r0.y * v.y + r0.z * v.z + r0.w;
            cy[sl] = r1.x * v.x + r1.y * v.y + r1.z * v.z + r1.w;
            cz[sl] = r2.x * v.x + r2.y * v.y + r2.z * v.z + r2.w;
            rr[sl] = it < n_items ? v.w : kNone;   // an idle slot's value stays at the bottom
            if (it < n_items) {
                const float e = v.w + margin;
                lo[0] = fminf(lo[0], cx[sl] - e); lo[1] = fminf(lo[1], cy[sl] - e); lo[2] = fminf(lo[2], cz[sl] - e);
                hi[0] = fmaxf(hi[0], cx[sl] + e); hi[1] = fmaxf(hi[1], cy[sl] + e); hi[2] = fmaxf(hi[2], cz[sl] + e);
            }
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) { lo[a] = warp_fmin(lo[a]); hi[a] = warp_fmax(hi[a]); }
        float v = kNone;
        const unsigned context = p2p ? 0u : ((1u << b) - 1u) | ((0xfffe0000u << b) & (((1u << B) - 1u) << kMaxB));
        const int n_ew = (n_env + 31) >> 5;
#pragma unroll 1
        for (int wd = 0; wd <= n_ew; ++wd) {
            const bool blocks = wd == n_ew;
            const int i = blocks ? n_env + lane : 32 * wd + lane;
            bool near = blocks ? (context >> lane) & 1u : i < n_env;
            if (near) {
                const float4 blo = sh.box[i][0], bhi = sh.box[i][1];
                near = blo.x <= hi[0] && bhi.x >= lo[0] && blo.y <= hi[1] && bhi.y >= lo[1] && blo.z <= hi[2] && bhi.z >= lo[2];
            }
            unsigned m = __ballot_sync(0xffffffffu, near);
#pragma unroll 1
            while (m) {
                const int bit = __ffs(m) - 1, o = 32 * wd + bit;
                m &= m - 1;
                if (!blocks && o >= sc.n_cub) {
                    const float4 sp = tab.osph[o - sc.n_cub];
#pragma unroll
                    for (int sl = 0; sl < 2; ++sl) {
                        const float dx = cx[sl] - sp.x, dy = cy[sl] - sp.y, dz = cz[sl] - sp.z;
                        v = fmaxf(v, rr[sl] + sp.w - sqrtf(dx * dx + dy * dy + dz * dz));
                    }
                    continue;
                }
                const float4* rec = blocks ? sh.blk[bit] : tab.cub + 4 * o;
#pragma unroll
                for (int sl = 0; sl < 2; ++sl) v = fmaxf(v, value32(cx[sl], cy[sl], cz[sl], rr[sl], rec));
            }
        }
        v = warp_fmax(v);
        const bool force = ((forced >> (8 * ci)) & 0xffu) || (loose & ((1u << b) - 1u));   // placed blocks k < b
        if (lane == 0) val[(size_t)r * C + t] = force ? INFINITY : v;
        if (!force) top = fmaxf(top, v);
    }
    if (lane == 0) atomicMax(&acc[r].top, float_key(top));
}

// Second pass: the configurations that can hold a solution's largest penetration, in FP64, a
// warp per configuration; `split` CTAs per solution share the configurations.  Each CTA folds
// its maximum into the solution's accumulator with an atomic, and the CTA that arrives last
// (counter after a fence; nothing waits) turns it into the metrics and the flag and clears the
// accumulator.
__global__ void __launch_bounds__(kChkThreads) k_check64(const __grid_constant__ Scalars64 s, const D4* __restrict__ cub,
                                                        const D4* __restrict__ osph, const float4* __restrict__ fcub,
                                                        const float* __restrict__ q, const int* __restrict__ n_sol, int P,
                                                        const float* __restrict__ val, double* __restrict__ metrics,
                                                        int* __restrict__ ok, CheckAcc* __restrict__ acc, int split) {
    const int r = blockIdx.x, slice = blockIdx.y, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int n = n_sol ? min(*n_sol, P) : P;
    if (r >= n) {
        if (tid == 0 && slice == 0) ok[r] = 0;
        return;
    }
    __shared__ double F[kChkWarps][9][12];   // per warp: frames 0..7 and the held block's, R then o
    __shared__ float4 blk[2 * kMaxB][4];     // FP32 cuboids of the blocks: k placed, 16 + k at the initial pose
    __shared__ int any;
    CheckAcc& A = acc[r];
    const int B = s.B, S = s.S, C = s.C;
    const float* qr = q + (size_t)r * C * 8;
    // nothing below it holds the maximum: neither a configuration (screened to within a margin) nor a
    // pair of one
    const float floor = fmaxf(key_float(A.top) - 2.f * s.margin, -s.margin);
    const int per = (C - 1 + split - 1) / split, t_end = min(C, 1 + (slice + 1) * per);
    double mp = 0.0;
    if (tid == 0) any = 0;
    __syncthreads();
    for (int t = 1 + slice * per + tid; t < t_end; t += kChkThreads)
        if (val[(size_t)r * C + t] >= floor) any = 1;
    __syncthreads();
    if (any && tid < 2 * kMaxB && (tid & 15) < B) {
        const bool placed = tid < kMaxB && !s.p2p;
        const int k = tid & 15;
        const double* p = placed ? A.pose[k] : s.init[k];
        float fs, fc;
        if (placed) { fc = (float)p[3]; fs = (float)p[4]; }
        else sincosf((float)p[3], &fs, &fc);
        blk[tid][0] = make_float4((float)p[0], (float)p[1], (float)p[2], 0.f);
        blk[tid][1] = make_float4(fc, fs, 0.f, (float)s.half[k][0]);
        blk[tid][2] = make_float4(-fs, fc, 0.f, (float)s.half[k][1]);
        blk[tid][3] = make_float4(0.f, 0.f, 1.f, (float)s.half[k][2]);
    }
    __syncthreads();
#pragma unroll 1
    for (int tb = 1 + slice * per; any && tb < t_end; tb += 32) {
        // the next 32 configurations: the warps share those to repeat
        unsigned todo = __ballot_sync(0xffffffffu, tb + lane < t_end && val[(size_t)r * C + tb + lane] >= floor);
#pragma unroll 1
        for (int turn = 0; todo; ++turn) {
            const int t = tb + __ffs(todo) - 1;
            todo &= todo - 1;
            if (turn % kChkWarps != w) continue;
            const int seg = (t - 1) / S, b = seg >> 1, k = lane & 7;
            const bool held = (seg & 1) && t - seg * S < S;
            double sn = 0.0, cs = 1.0, R[9], o[3];
            if (k > 0) sincos(s.th0[k - 1] + (double)qr[t * 8 + k - 1], &sn, &cs);
            fk_lanes<double>(s, sn, cs, R, o);
            __syncwarp();   // the previous configuration's frames have been read
            if (lane < 8) {
                for (int i = 0; i < 9; ++i) F[w][k][i] = R[i];
                for (int i = 0; i < 3; ++i) F[w][k][9 + i] = o[i];
                if (k == 7) {
                    double Rt[9], pt[3];
                    tool64(s, R, o, Rt, pt);
                    held64(s, b, Rt, pt, &F[w][8][0], &F[w][8][9]);
                }
            }
            __syncwarp();
            const int n_items = s.n_rsph + (held ? 8 : 0);
#pragma unroll 1
            for (int base = 0; base < n_items; base += 32) {
                const int it = base + lane;
                const bool valid = it < n_items;
                const double* f = F[w][8];
                double l[3] = {0.0, 0.0, 0.0}, rad = 0.0;
                if (it < s.n_rsph) {
                    f = F[w][s.rlink[it]];
                    for (int i = 0; i < 3; ++i) l[i] = s.rsph[it][i];
                    rad = s.rsph[it][3];
                } else if (valid) {
                    const int m = it - s.n_rsph;
                    for (int i = 0; i < 3; ++i) l[i] = ((m >> i) & 1 ? 0.5 : -0.5) * s.half[b][i];
                    rad = s.hmin[b] * 0.5;
                }
                const double cx = f[0] * l[0] + f[1] * l[1] + f[2] * l[2] + f[9];
                const double cy = f[3] * l[0] + f[4] * l[1] + f[5] * l[2] + f[10];
                const double cz = f[6] * l[0] + f[7] * l[1] + f[8] * l[2] + f[11];
                // the pairs that FP32 finds no lower than the floor: first the obstacles near any of the
                // warp's spheres (all of them when one is not finite), then sphere by sphere
                const float fx = (float)cx, fy = (float)cy, fz = (float)cz, fr = (float)rad, e = fr + s.margin;
                const bool finite = fabsf(fx) + fabsf(fy) + fabsf(fz) < 1e30f;
                const bool all = __any_sync(0xffffffffu, valid && !finite);
                const float lx = warp_fmin(valid ? fx - e : 3.4e38f), hx = warp_fmax(valid ? fx + e : -3.4e38f);
                const float ly = warp_fmin(valid ? fy - e : 3.4e38f), hy = warp_fmax(valid ? fy + e : -3.4e38f);
                const float lz = warp_fmin(valid ? fz - e : 3.4e38f), hz = warp_fmax(valid ? fz + e : -3.4e38f);
                auto near = [&](const float4* c) {
                    float4 box[2];
                    cuboid_box(c, box);
                    return all || (box[0].x <= hx && box[1].x >= lx && box[0].y <= hy && box[1].y >= ly && box[0].z <= hz &&
                                   box[1].z >= lz);
                };
#pragma unroll 1
                for (int wd = 0; 32 * wd < s.n_cub; ++wd) {
                    unsigned m = __ballot_sync(0xffffffffu, 32 * wd + lane < s.n_cub && near(fcub + 4 * (32 * wd + lane)));
#pragma unroll 1
                    while (m) {
                        const int ob = 32 * wd + __ffs(m) - 1;
                        m &= m - 1;
                        if (valid && !(value32(fx, fy, fz, fr, fcub + 4 * ob) < floor))
                            mp = fmax(mp, pen_cub64(cx, cy, cz, rad, &cub[4 * ob]));
                    }
                }
#pragma unroll 1
                for (int ob = 0; ob < s.n_osph; ++ob) {
                    double gx, gy, gz;
                    if (valid) mp = fmax(mp, pen_sphere<double>(cx, cy, cz, rad, osph[ob], gx, gy, gz));
                }
                // placed blocks below b, blocks above b at their initial poses
                unsigned m = __ballot_sync(0xffffffffu, (lane < kMaxB ? lane < b : lane - kMaxB > b && lane - kMaxB < B) &&
                                                            near(blk[lane]));
#pragma unroll 1
                while (m) {
                    const int bit = __ffs(m) - 1, i = bit & (kMaxB - 1);
                    m &= m - 1;
                    if (!valid || value32(fx, fy, fz, fr, blk[bit]) < floor) continue;
                    const double* pose = i < b ? A.pose[i] : s.init[i];
                    double yc = pose[3], ys = i < b ? pose[4] : 0.0;
                    if (i > b) sincos(s.init[i][3], &ys, &yc);
                    D4 c[4];
                    block_cub64(pose, yc, ys, s.half[i], c);
                    mp = fmax(mp, pen_cub64(cx, cy, cz, rad, c));
                }
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mp = fmax(mp, __shfl_xor_sync(0xffffffffu, mp, off));
    if (lane == 0 && mp > 0.0) atomicMax(&A.mp, (unsigned long long)__double_as_longlong(mp));   // non-negative: integer order
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(&A.count, 1) == split - 1) {   // the last slice of this solution
            __threadfence();
            const volatile CheckAcc& V = A;
            const double mpa = __longlong_as_double((long long)V.mp);
            const int lim_all = V.viol == 0;
            double* m = metrics + (size_t)r * 6;
            m[0] = mpa; m[1] = V.ms; m[2] = V.mt; m[3] = V.pp; m[4] = V.mD; m[5] = V.mz;
            ok[r] = (mpa <= s.eps && V.ms <= s.eps_start && V.mt <= s.eps_start && V.pp <= s.eps && V.mD <= s.eps &&
                     V.mz <= s.eps && lim_all) ? 1 : 0;
            A.mp = 0ull; A.top = 0u; A.viol = 0; A.count = 0;   // ready for the next check
        }
    }
}

cudaError_t launch_check64(const Scalars64& s, const Scalars& sc, DevTables tab, const void* cub, const void* osph,
                           const float* q, const int* n_sol, int P, double* metrics, int* ok, float* val, CheckAcc* acc,
                           cudaStream_t st) {
    if (P <= 0) return cudaSuccess;
    cudaError_t e = allow_max_dynamic_smem(k_check_screen, sizeof(ScreenShared));
    if (e != cudaSuccess) return e;
    const D4 *c64 = static_cast<const D4*>(cub), *o64 = static_cast<const D4*>(osph);
    const int split = (s.C - 1 + kScrCfgs - 1) / kScrCfgs;
    k_check_screen<<<dim3(P, split + 1), kScrThreads, sizeof(ScreenShared), st>>>(s, sc, tab, c64, o64, q, n_sol, P, val, acc);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_check64<<<dim3(P, split), kChkThreads, 0, st>>>(s, c64, o64, tab.cub, q, n_sol, P, val, metrics, ok, acc, split);
    return cudaGetLastError();
}

}  // namespace spasm
