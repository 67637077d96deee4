// Stage 1 (Alg. 1) for the packing goal: the placement cost of the appendix's Tetris
// problem, one warp per particle.
//
//   C = w_coll (sum_{i<j} P(i, j) + sum_i sum_{w in walls} P(i, w)) + w_height sum_i |z_i - z*|
//
// Block i is a polyomino of unit cubes; each cube (edge u) carries 8 spheres of radius u/4
// at (+-u/4, +-u/4, +-u/4) from its centre (objects as sphere sets, Sec. III).  P(i, j) sums
// the penetration of every sphere of block j into every cube of block i < j, P(i, w) every
// sphere of block i into wall w (the environment cuboids).  Penetrations turn quadratic in
// the refinement phase; |z - z*| keeps its form.
//
// Lanes own (cell, sphere) items: the 8 spheres of a cube are 8 consecutive lanes, so a
// cube's sphere-side gradient is reduced inside its lane group and stored once per
// evaluation (gcell); lanes < B then add their cubes in order, so sums are deterministic.
// The cube side of a block pair is reduced over the warp once per lower block.
//
// Bound by instruction issue.  The 32 spheres of a pass (four cubes) meet the cubes below whose boxes
// they reach: one ballot per 32 cubes, in the order of the cubes, so the sums stay those of all of them.
// The cubes' boxes are laid out once per evaluation: 32 lanes that index the constant bank by cube in
// every pass cost more than the cull saves (4.88 -> 5.26 ms).  The walls' boxes (wall: centre, then half
// extents) are laid out once per CTA.  Descending 4096 packings of 8 blocks: 4.88 -> 3.99 ms.
#pragma once
#include "stage1.cuh"

namespace spasm {

__device__ __forceinline__ void place_eval_pack_warp(const Scalars& sc, const float4* __restrict__ cub,
                                                     const float4* __restrict__ wall, int n_cub,
                                                     const float4* __restrict__ osph, int n_osph, const float* x,
                                                     bool quad, int mode, float* g, PlaceScratch& ps, float4* gcell,
                                                     float4* cube, PlaceOut* out) {
    const int lane = threadIdx.x & 31;
    const int B = sc.B;
    const bool want_grad = mode != kPlaceForward;
    const float u = sc.cell_size, r = 0.25f * u;
    const float4 half = make_float4(0.5f * u, 0.5f * u, 0.5f * u, r);

    // -- per-block terms (lane i owns block i): height residual, the cube frame (cos, sin)
    float my_e = 0.f;
    if (lane < B) {
        const int i = lane;
        my_e = x[4 * i + 2] - sc.z_star;
        block_cuboid(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3], half, ps.bc[i]);
        if (want_grad) {
            const float b = sc.w_height * (my_e > 0.f ? 1.f : (my_e < 0.f ? -1.f : 0.f));
            g[4 * i] = 0.f; g[4 * i + 1] = 0.f; g[4 * i + 2] = b; g[4 * i + 3] = 0.f;
        }
    }
    __syncwarp();
    for (int k = lane; k < sc.n_cells; k += 32) {
        const int i = sc.cell_block[k];
        const float2 off = sc.cell[k];
        const float ci = ps.bc[i][1].x, si = ps.bc[i][1].y;
        cube[k] = make_float4(x[4 * i] + ci * off.x - si * off.y, x[4 * i + 1] + si * off.x + ci * off.y, x[4 * i + 2],
                              (fabsf(ci) + fabsf(si)) * half.x);
    }
    __syncwarp();

    const float s_coll = sc.w_coll;
    float coll = 0.f, maxpen = 0.f;
    const int n_items = 8 * sc.n_cells;
    for (int base = 0; base < n_items; base += 32) {
        const int it = base + lane;
        const bool valid = it < n_items;
        const int k = valid ? it >> 3 : 0, m = it & 7;
        const int j = sc.cell_block[k];
        const float c = ps.bc[j][1].x, s = ps.bc[j][1].y;
        const float lx = sc.cell[k].x + ((m & 1) ? 0.25f : -0.25f) * u;
        const float ly = sc.cell[k].y + ((m & 2) ? 0.25f : -0.25f) * u;
        const float lz = ((m & 4) ? 0.25f : -0.25f) * u;
        const float cx = x[4 * j] + c * lx - s * ly, cy = x[4 * j + 1] + s * lx + c * ly, cz = x[4 * j + 2] + lz;
        float ax = 0.f, ay = 0.f, az = 0.f;   // dC/dc of this sphere (scaled by 2 pen in the quadratic form)
        const SphereBox sb = warp_sphere_box(valid, cx, cy, cz, r);
        for (int first = 0; first < n_cub; first += 32) {
            bool near_wall = false;
            if (first + lane < n_cub) {
                const float4 q = wall[2 * (first + lane)], e = wall[2 * (first + lane) + 1];
                near_wall = sb.near_box(q.x, q.y, q.z, e.x, e.y, e.z);
            }
            unsigned walls = __ballot_sync(0xffffffffu, near_wall);
            for (; valid && walls; walls &= walls - 1u) {
                const int o = first + __ffs(walls) - 1;
                float gx, gy, gz;
                const float pen = pen_cuboid<float>(cx, cy, cz, r, cub[4 * o], cub[4 * o + 1], cub[4 * o + 2],
                                                    cub[4 * o + 3], gx, gy, gz);
                if (pen > 0.f) {
                    maxpen = fmaxf(maxpen, pen);
                    coll += quad ? pen * pen : pen;
                    const float sg = quad ? 2.f * pen : 1.f;
                    ax += sg * gx; ay += sg * gy; az += sg * gz;
                }
            }
        }
        if (valid) {
            for (int o = 0; o < n_osph; ++o) {
                float gx, gy, gz;
                const float pen = pen_sphere<float>(cx, cy, cz, r, osph[o], gx, gy, gz);
                if (pen > 0.f) {
                    maxpen = fmaxf(maxpen, pen);
                    coll += quad ? pen * pen : pen;
                    const float sg = quad ? 2.f * pen : 1.f;
                    ax += sg * gx; ay += sg * gy; az += sg * gz;
                }
            }
        }
        // cubes of the blocks below j in the skeleton order, those near the 32 spheres of this pass
        unsigned long long near_cubes = 0ull;
        for (int first = 0; first < sc.n_cells; first += 32) {
            bool near_cube = false;
            if (first + lane < sc.n_cells) {
                const float4 q = cube[first + lane];
                near_cube = sb.near_box(q.x, q.y, q.z, q.w, q.w, half.z);
            }
            near_cubes |= (unsigned long long)__ballot_sync(0xffffffffu, near_cube) << first;
        }
        const int j_top = sc.cell_block[min(base + 31, n_items - 1) >> 3];   // cells are in block order
        near_cubes &= (1ull << sc.cell_start[j_top]) - 1ull;                // cell_start[j_top] < kMaxCells
        while (near_cubes) {
            const int i = sc.cell_block[__ffsll((long long)near_cubes) - 1];
            unsigned long long cubes = near_cubes & ((1ull << sc.cell_start[i + 1]) - 1ull);   // of block i
            near_cubes ^= cubes;
            float bx = 0.f, by = 0.f, bz = 0.f, byaw = 0.f;   // dC/d(pose i) from this sphere
            bool hit = false;
            const float oxi = x[4 * i], oyi = x[4 * i + 1], ozi = x[4 * i + 2];
            const float dxo = cx - oxi, dyo = cy - oyi, dzo = cz - ozi, reach = sc.cell_reach[i] + r;
            if (valid && i < j && dxo * dxo + dyo * dyo + dzo * dzo < reach * reach) {
                const float ci = ps.bc[i][1].x, si = ps.bc[i][1].y;
                const float4 c0 = make_float4(ci, si, 0.f, half.x), c1 = make_float4(-si, ci, 0.f, half.y);
                const float4 c2 = make_float4(0.f, 0.f, 1.f, half.z);
                for (; cubes; cubes &= cubes - 1ull) {
                    const int kk = __ffsll((long long)cubes) - 1;
                    const float2 off = sc.cell[kk];
                    const float4 o = make_float4(oxi + ci * off.x - si * off.y, oyi + si * off.x + ci * off.y, ozi, 0.f);
                    float gx, gy, gz;
                    const float pen = pen_cuboid<float>(cx, cy, cz, r, o, c0, c1, c2, gx, gy, gz);
                    if (pen > 0.f) {
                        hit = true;
                        maxpen = fmaxf(maxpen, pen);
                        coll += quad ? pen * pen : pen;
                        const float sg = quad ? 2.f * pen : 1.f;
                        gx *= sg; gy *= sg; gz *= sg;
                        ax += gx; ay += gy; az += gz;
                        // the block moves rigidly about its origin: d/dO = -g, d/dyaw = -((c - O) x g)_z
                        bx -= gx; by -= gy; bz -= gz;
                        byaw -= dxo * gy - dyo * gx;
                    }
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
            const float gyaw = ax * (-s * lx - c * ly) + ay * (c * lx - s * ly);   // dc/dyaw_j
            const float d = group_sums(ax, ay, az, gyaw);
            if (valid && (m & 1) == 0) reinterpret_cast<float*>(gcell + k)[m >> 1] = d;
        }
    }
    __syncwarp();
    if (want_grad && lane < B) {
        const int i = lane;
        float sx = 0.f, sy = 0.f, sz = 0.f, syaw = 0.f;
        for (int k = sc.cell_start[i]; k < sc.cell_start[i + 1]; ++k) {
            const float4 v = gcell[k];
            sx += v.x; sy += v.y; sz += v.z; syaw += v.w;
        }
        g[4 * i] += s_coll * sx; g[4 * i + 1] += s_coll * sy; g[4 * i + 2] += s_coll * sz; g[4 * i + 3] += s_coll * syaw;
    }
    if (out) {
        out->c_coll = warp_sum(coll);
        out->maxpen = warp_max(maxpen);
        out->c_stable = 0.f;
        out->c_height = warp_sum(lane < B ? fabsf(my_e) : 0.f);
        out->maxD = 0.f;
        out->maxdz = warp_max(lane < B ? fabsf(my_e) : 0.f);
    }
    __syncwarp();
}

// The placement cost of the problem's goal (tower or packing; kTower: a tower).
template <bool kTower>
__device__ __forceinline__ void place_eval(const Scalars& sc, const float4* __restrict__ cub,
                                           const float4* __restrict__ wall, int n_cub,
                                           const float4* __restrict__ osph, int n_osph, const float* x, bool quad,
                                           int mode, float* g, PlaceScratch& ps, float4* gcell, float4* cube,
                                           uint32_t* cand, PlaceOut* out) {
    if (!kTower && sc.kind == kKindPack)
        place_eval_pack_warp(sc, cub, wall, n_cub, osph, n_osph, x, quad, mode, g, ps, gcell, cube, out);
    else
        place_eval_warp(sc, cub, n_cub, osph, n_osph, x, quad, mode, g, ps, cand, out);
}

}  // namespace spasm
