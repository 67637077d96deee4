// Stage 1 of SPaSM (Alg. 1): tower placement cost and gradient, one warp per particle.
//
// Per particle the warp holds the B x 4 pose vector in shared memory.  Lanes own
// (block j, sphere m) items of the block sphere sets and test them against the
// environment tables (staged once per CTA in shared memory, read as broadcasts) and the
// cuboids of the blocks below j.  Gradients are reduced deterministically: groups of 8
// lanes (the 8 spheres of one block) by xor-shuffles, block-pair terms by whole-warp
// reductions taken only when a lane of the warp penetrates.
// Bound by instruction issue (79% of the cycles at 64 registers, 32 warps per SM), so work is left
// out where it cannot count: the 32 spheres of a pass (four blocks) meet the blocks below whose boxes
// they reach, about two of nine in a stacked 10-block tower, and no cost terms are summed where only
// the gradient is used.  What is left is summed in the same order.  Descending 4096 10-block towers:
// 471 -> 400 us; sampling and costing 16384: 41 -> 37 us.
#pragma once
#include "common.cuh"

namespace spasm {

struct PlaceOut {
    float c_stable, c_height, c_coll;    // sum D, sum e^2, sum pen (or pen^2)
    float maxpen, maxD, maxdz;           // satisfying metrics
};

// Per-warp shared scratch of the placement evaluation: the support factors, and in stage 1
// the block cuboids (stage 2 keeps its own).
struct StackScratch {
    float stab[kMaxB][4];    // a_i dD_i/dv (x, y), a_i dD_i/dyaw, D_i
};
struct PlaceScratch : StackScratch {
    float4 bc[kMaxB][4];     // block cuboids
};

// Coefficient modes of the gradient: none, stage-1 cost (a = w_stable, b = 2 w_height e), or the
// residuals with the unit-coefficient support factors (a = 1) left in ps.stab and no gradient
// written (stage 2 scales them by its multipliers once those are known).
enum PlaceMode { kPlaceForward = 0, kPlaceStage1 = 1, kPlaceUnit = 2 };

// Per-block terms of the tower (lane i < B owns block i): height residual e_i, support
// distance D_i and the block cuboids in ps.  With mode kPlaceStage1, sets
//   g = sum_i a_i dD_i/dx + sum_i b_i de_i/dx   (the collision part is added by the caller);
// with kPlaceUnit, leaves dD_i/d(centre of mass, yaw) in ps.stab for place_stack_grad.
// x, g: per-warp shared arrays of 4B floats.  Must be called by all 32 lanes of the warp.
// bc: the block cuboids, written here or, in mode kPlaceUnit, already those of x.
__device__ __forceinline__ void place_stack_warp(const TrajScalars& sc, const float* x, int mode, float* g,
                                                 StackScratch& ps, float4 (*bc)[4], float& my_D, float& my_e) {
    const int lane = threadIdx.x & 31;
    const int B = sc.B;
    const bool want_grad = mode != kPlaceForward;
    my_D = 0.f; my_e = 0.f;
    if (lane < B) {
        const int i = lane;
        my_e = x[4 * i + 2] - sc.zt[i];
        if (mode != kPlaceUnit)
            block_cuboid(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3], sc.half[i], bc[i]);
        float sx = 0.f, sy = 0.f, dvx = 0.f, dvy = 0.f, dyaw = 0.f;
        if (i + 1 < B) {
            const int n_above = B - 1 - i;
#pragma unroll 1
            for (int j = i + 1; j < B; ++j) { sx += x[4 * j]; sy += x[4 * j + 1]; }
            const float mx = sx / (float)n_above, my = sy / (float)n_above;
            const float c = bc[i][1].x, s = bc[i][1].y;   // of the yaw
            const float vx = mx - x[4 * i], vy = my - x[4 * i + 1];
            const float ux = c * vx + s * vy, uy = -s * vx + c * vy;       // Rz(-yaw) v
            const float ex = fmaxf(fabsf(ux) - sc.half[i].x, 0.f), ey = fmaxf(fabsf(uy) - sc.half[i].y, 0.f);
            my_D = sqrtf(ex * ex + ey * ey);
            if (want_grad && my_D > 0.f) {
                const float a = mode == kPlaceStage1 ? sc.w_stable : 1.f;
                const float du_x = (ux >= 0.f ? ex : -ex) / my_D, du_y = (uy >= 0.f ? ey : -ey) / my_D;
                dvx = a * (c * du_x - s * du_y);
                dvy = a * (s * du_x + c * du_y);
                dyaw = a * (du_x * uy - du_y * ux);
            }
        }
        ps.stab[i][0] = dvx; ps.stab[i][1] = dvy; ps.stab[i][2] = dyaw; ps.stab[i][3] = my_D;
    }
    __syncwarp();
    if (want_grad && mode != kPlaceUnit && lane < B) {
        const int i = lane;
        float gx = -ps.stab[i][0], gy = -ps.stab[i][1];
#pragma unroll 1
        for (int k = 0; k < i; ++k) {
            const float inv = 1.f / (float)(B - 1 - k);
            gx += ps.stab[k][0] * inv;
            gy += ps.stab[k][1] * inv;
        }
        const float b = 2.f * sc.w_height * my_e;
        g[4 * i] = gx; g[4 * i + 1] = gy; g[4 * i + 2] = b; g[4 * i + 3] = ps.stab[i][2];
    }
    __syncwarp();
}

// sum_i a_i dD_i/dx + sum_i b_i de_i/dx for coefficients a_in, b_in, from the unit factors that
// place_stack_warp's kPlaceUnit pass left in ps.
// inv_above[k] = 1 / (B - 1 - k), the blocks above block k < B - 1.
__device__ __forceinline__ void place_stack_grad(const TrajScalars& sc, const StackScratch& ps, const float* a_in,
                                                 const float* b_in, const float* inv_above, float* g) {
    const int lane = threadIdx.x & 31;
    const int B = sc.B;
    if (lane < B) {
        const int i = lane;
        float gx = -(a_in[i] * ps.stab[i][0]), gy = -(a_in[i] * ps.stab[i][1]);
#pragma unroll 1
        for (int k = 0; k < i; ++k) {
            const float inv = inv_above[k];
            gx += (a_in[k] * ps.stab[k][0]) * inv;
            gy += (a_in[k] * ps.stab[k][1]) * inv;
        }
        g[4 * i] = gx; g[4 * i + 1] = gy; g[4 * i + 2] = b_in[i]; g[4 * i + 3] = a_in[i] * ps.stab[i][2];
    }
    __syncwarp();
}

// Box of the warp's spheres (of its valid lanes), padded against the rounding of boxes and distances: a
// solid whose box lies apart from it penetrates none of them, so leaving it out changes no sum.
// A sphere that is not at a finite place (which a penetration test may count) makes every solid near.
struct SphereBox {
    float lo_x, lo_y, lo_z, hi_x, hi_y, hi_z;
    bool all;
    __device__ __forceinline__ bool near_box(float x, float y, float z, float ex, float ey, float ez) const {
        ex *= 1.000004f; ey *= 1.000004f; ez *= 1.000004f;
        return all || !(x - ex > hi_x || x + ex < lo_x || y - ey > hi_y || y + ey < lo_y || z - ez > hi_z ||
                        z + ez < lo_z);
    }
    __device__ __forceinline__ bool near_cuboid(const float4* c) const {
        const float4 c0 = c[0], c1 = c[1], c2 = c[2], c3 = c[3];
        return near_box(c0.x, c0.y, c0.z, fabsf(c1.x) * c1.w + fabsf(c2.x) * c2.w + fabsf(c3.x) * c3.w,
                        fabsf(c1.y) * c1.w + fabsf(c2.y) * c2.w + fabsf(c3.y) * c3.w,
                        fabsf(c1.z) * c1.w + fabsf(c2.z) * c2.w + fabsf(c3.z) * c3.w);
    }
};
__device__ __forceinline__ SphereBox warp_sphere_box(bool valid, float cx, float cy, float cz, float r) {
    const float away = fabsf(cx) + fabsf(cy) + fabsf(cz);
    const float e = r + 1e-5f + 1e-6f * away;
    SphereBox b;
    b.lo_x = warp_fmin(valid ? cx - e : 3.4e38f); b.hi_x = warp_fmax(valid ? cx + e : -3.4e38f);
    b.lo_y = warp_fmin(valid ? cy - e : 3.4e38f); b.hi_y = warp_fmax(valid ? cy + e : -3.4e38f);
    b.lo_z = warp_fmin(valid ? cz - e : 3.4e38f); b.hi_z = warp_fmax(valid ? cz + e : -3.4e38f);
    b.all = __any_sync(0xffffffffu, valid && !(away < 1e30f));
    return b;
}

// Sums over the groups of 8 lanes: lanes 2 n and 2 n + 1 of a group get the sum of value n.  The lanes of
// either half keep the values that they will own (4 shuffles, not 12), paired as a butterfly pairs them.
__device__ __forceinline__ float group_sums(float v0, float v1, float v2, float v3) {
    const bool up4 = threadIdx.x & 4, up2 = threadIdx.x & 2;
    float a = up4 ? v2 : v0, b = up4 ? v3 : v1;
    a += __shfl_xor_sync(0xffffffffu, up4 ? v0 : v2, 4);
    b += __shfl_xor_sync(0xffffffffu, up4 ? v1 : v3, 4);
    float r = up2 ? b : a;
    r += __shfl_xor_sync(0xffffffffu, up2 ? a : b, 2);
    return r + __shfl_xor_sync(0xffffffffu, r, 1);
}

// x, g: per-warp shared arrays of 4B floats.  With mode != kPlaceForward, writes
//   g = sum_i a_i dD_i/dx + sum_i b_i de_i/dx + s_coll dC_coll/dx.
// out (optional): the cost terms and metrics.  Must be called by all 32 lanes of the warp.
// cand: per-warp scratch of kMaxCub/32 + kMaxOSph/32 words (the candidate obstacles of the particle).
__device__ __forceinline__ void place_eval_warp(const Scalars& sc, const float4* __restrict__ cub, int n_cub,
                                                const float4* __restrict__ osph, int n_osph, const float* x,
                                                bool quad, int mode, float* g, PlaceScratch& ps, uint32_t* cand,
                                                PlaceOut* out) {
    const int lane = threadIdx.x & 31;
    const int B = sc.B;
    const bool want_grad = mode != kPlaceForward;
    float my_D, my_e;
    place_stack_warp(sc, x, mode, g, ps, ps.bc, my_D, my_e);

    // -- collisions: items (block j, sphere m)
    const float s_coll = sc.w_coll;
    float coll = 0.f, maxpen = 0.f;
    const int n_items = 8 * B;
    // exact cull: the box of every block sphere of the particle (padded by 1e-5 against the
    // rounding of the boxes) against each obstacle's box; only the obstacles that overlap it
    // can touch a sphere, and they are visited in the same order as without the cull
    const int n_cw = (n_cub + 31) >> 5, n_sw = (n_osph + 31) >> 5;
    {
        float lo_x = 3.4e38f, lo_y = 3.4e38f, lo_z = 3.4e38f, hi_x = -3.4e38f, hi_y = -3.4e38f, hi_z = -3.4e38f;
        for (int base = 0; base < n_items; base += 32) {
            const int it = base + lane;
            if (it < n_items) {
                const int j = it >> 3, m = it & 7;
                const float4 h = sc.half[j];
                float lx, ly, lz;
                block_sphere_local(h, m, lx, ly, lz);
                const float c = ps.bc[j][1].x, s = ps.bc[j][1].y;
                const float cx = x[4 * j] + c * lx - s * ly, cy = x[4 * j + 1] + s * lx + c * ly, cz = x[4 * j + 2] + lz;
                const float r = h.w + 1e-5f;
                lo_x = fminf(lo_x, cx - r); lo_y = fminf(lo_y, cy - r); lo_z = fminf(lo_z, cz - r);
                hi_x = fmaxf(hi_x, cx + r); hi_y = fmaxf(hi_y, cy + r); hi_z = fmaxf(hi_z, cz + r);
            }
        }
        lo_x = warp_fmin(lo_x); lo_y = warp_fmin(lo_y); lo_z = warp_fmin(lo_z);
        hi_x = warp_fmax(hi_x); hi_y = warp_fmax(hi_y); hi_z = warp_fmax(hi_z);
        for (int wd = 0; wd < n_cw; ++wd) {
            const int o = 32 * wd + lane;
            bool near = false;
            if (o < n_cub) {
                const float4 c0 = cub[4 * o], c1 = cub[4 * o + 1], c2 = cub[4 * o + 2], c3 = cub[4 * o + 3];
                const float ex = fabsf(c1.x) * c1.w + fabsf(c2.x) * c2.w + fabsf(c3.x) * c3.w;
                const float ey = fabsf(c1.y) * c1.w + fabsf(c2.y) * c2.w + fabsf(c3.y) * c3.w;
                const float ez = fabsf(c1.z) * c1.w + fabsf(c2.z) * c2.w + fabsf(c3.z) * c3.w;
                near = c0.x - ex <= hi_x && c0.x + ex >= lo_x && c0.y - ey <= hi_y && c0.y + ey >= lo_y &&
                       c0.z - ez <= hi_z && c0.z + ez >= lo_z;
            }
            const unsigned mk = __ballot_sync(0xffffffffu, near);
            if (lane == 0) cand[wd] = mk;
        }
        for (int wd = 0; wd < n_sw; ++wd) {
            const int o = 32 * wd + lane;
            bool near = false;
            if (o < n_osph) {
                const float4 sp = osph[o];
                near = sp.x - sp.w <= hi_x && sp.x + sp.w >= lo_x && sp.y - sp.w <= hi_y && sp.y + sp.w >= lo_y &&
                       sp.z - sp.w <= hi_z && sp.z + sp.w >= lo_z;
            }
            const unsigned mk = __ballot_sync(0xffffffffu, near);
            if (lane == 0) cand[kMaxCub / 32 + wd] = mk;
        }
        __syncwarp();
    }
    for (int base = 0; base < n_items; base += 32) {
        const int it = base + lane;
        const bool valid = it < n_items;
        const int j = valid ? it >> 3 : 0, m = it & 7;
        float cx = 0.f, cy = 0.f, cz = 0.f, r = 0.f, dcx = 0.f, dcy = 0.f;
        float pj0 = 0.f, pj1 = 0.f;
        if (valid) {
            const float4 h = sc.half[j];
            float lx, ly, lz;
            block_sphere_local(h, m, lx, ly, lz);
            const float c = ps.bc[j][1].x, s = ps.bc[j][1].y;
            pj0 = x[4 * j]; pj1 = x[4 * j + 1];
            cx = pj0 + c * lx - s * ly;
            cy = pj1 + s * lx + c * ly;
            cz = x[4 * j + 2] + lz;
            dcx = -s * lx - c * ly;   // dc/dyaw_j
            dcy = c * lx - s * ly;
            r = h.w;
        }
        float ax = 0.f, ay = 0.f, az = 0.f;   // dC/dc of this item (scaled by 2 pen in quad form)
        if (valid) {
            for (int wd = 0; wd < n_cw; ++wd) {
                unsigned mk = cand[wd];
                while (mk) {
                    const int o = 32 * wd + __ffs(mk) - 1;
                    mk &= mk - 1;
                    float gx, gy, gz;
                    const float pen = pen_cuboid<float>(cx, cy, cz, r, cub[4 * o], cub[4 * o + 1], cub[4 * o + 2],
                                                        cub[4 * o + 3], gx, gy, gz);
                    if (pen > 0.f) {
                        maxpen = fmaxf(maxpen, pen);
                        coll += quad ? pen * pen : pen;
                        const float sgrad = quad ? 2.f * pen : 1.f;
                        ax += sgrad * gx; ay += sgrad * gy; az += sgrad * gz;
                    }
                }
            }
            for (int wd = 0; wd < n_sw; ++wd) {
                unsigned mk = cand[kMaxCub / 32 + wd];
                while (mk) {
                    const int o = 32 * wd + __ffs(mk) - 1;
                    mk &= mk - 1;
                    float gx, gy, gz;
                    const float pen = pen_sphere<float>(cx, cy, cz, r, osph[o], gx, gy, gz);
                    if (pen > 0.f) {
                        maxpen = fmaxf(maxpen, pen);
                        coll += quad ? pen * pen : pen;
                        const float sgrad = quad ? 2.f * pen : 1.f;
                        ax += sgrad * gx; ay += sgrad * gy; az += sgrad * gz;
                    }
                }
            }
        }
        // blocks below in the stack: sphere of j vs cuboid of i < j, the blocks near the 32 spheres of this pass
        const int j_top = min(base + 31, n_items - 1) >> 3;
        unsigned below = 0u;
        if (j_top > 0) {
            const SphereBox sb = warp_sphere_box(valid, cx, cy, cz, r);
            bool near_block = false;
            if (lane < B) near_block = sb.near_cuboid(ps.bc[lane]);
            below = __ballot_sync(0xffffffffu, near_block) & ((1u << j_top) - 1u);
        }
        for (; below; below &= below - 1u) {
            const int i = __ffs(below) - 1;
            float bx = 0.f, by = 0.f, bz = 0.f, byaw = 0.f;   // dC/d pose_i from this item
            bool hit = false;
            if (valid && i < j) {
                float gx, gy, gz;
                const float pen = pen_cuboid<float>(cx, cy, cz, r, ps.bc[i][0], ps.bc[i][1], ps.bc[i][2], ps.bc[i][3],
                                                    gx, gy, gz);
                if (pen > 0.f) {
                    hit = true;
                    maxpen = fmaxf(maxpen, pen);
                    coll += quad ? pen * pen : pen;
                    const float sgrad = quad ? 2.f * pen : 1.f;
                    gx *= sgrad; gy *= sgrad; gz *= sgrad;
                    ax += gx; ay += gy; az += gz;
                    // the cuboid moves rigidly: d/dP_i = -g, d/dyaw_i = -((c - P_i) x g)_z
                    bx = -gx; by = -gy; bz = -gz;
                    byaw = -((cx - x[4 * i]) * gy - (cy - x[4 * i + 1]) * gx);
                }
            }
            if (want_grad && __any_sync(0xffffffffu, hit)) {
                float d4[4] = {bx, by, bz, byaw};
                const float d = warp_sums<4>(d4);   // lane 8 n: value n
                if ((lane & 7) == 0) g[4 * i + (lane >> 3)] += s_coll * d;
                __syncwarp();
            }
        }
        if (want_grad) {
            const float d = group_sums(ax, ay, az, ax * dcx + ay * dcy);
            // four writers per block j; groups of 8 lanes never share j
            if (valid && (m & 1) == 0) g[4 * j + (m >> 1)] += s_coll * d;
            __syncwarp();
        }
    }
    if (out) {
        out->c_coll = warp_sum(coll);
        out->maxpen = warp_max(maxpen);
        out->c_stable = warp_sum(lane < B ? my_D : 0.f);
        out->c_height = warp_sum(lane < B ? my_e * my_e : 0.f);
        out->maxD = warp_max(lane < B ? my_D : 0.f);
        out->maxdz = warp_max(lane < B ? fabsf(my_e) : 0.f);
    }
    __syncwarp();
}

__device__ __forceinline__ float place_cost_value(const Scalars& sc, const PlaceOut& o) {
    return sc.w_stable * o.c_stable + sc.w_height * o.c_height + sc.w_coll * o.c_coll;
}

// Projection onto the problem box (x, y in the goal box; z above the block's resting
// height; yaw wrapped to [-pi, pi)) of variable v = 4 i + k.
__device__ __forceinline__ float place_clamp(const Scalars& sc, int v, float val) {
    const int i = v >> 2, k = v & 3;
    if (k == 0) return fminf(fmaxf(val, sc.box_lo[0]), sc.box_hi[0]);
    if (k == 1) return fminf(fmaxf(val, sc.box_lo[1]), sc.box_hi[1]);
    if (k == 2) return fminf(fmaxf(val, sc.zlo[i]), sc.box_hi[2]);
    const float two_pi = 2.f * kPi;
    return val - two_pi * floorf((val + kPi) / two_pi);
}

}  // namespace spasm
