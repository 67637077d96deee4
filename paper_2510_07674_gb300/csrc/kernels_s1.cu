// Stage-1 kernels (Alg. 1): sampling + initial cost, evaluation, fused descent, and the
// selection kernel.
#include "launch.h"
#include "select.cuh"
#include "stage1.cuh"
#include "stage1_pack.cuh"

namespace spasm {

constexpr int kS1Warps = 8;
constexpr int kS1Threads = 32 * kS1Warps;

struct S1Warp {
    float x[4 * kMaxB];
    float g[4 * kMaxB];
    PlaceScratch ps;
    float4 gcell[kMaxCells];   // per-cube sphere-side gradients of the packing goal
    float4 cube[kMaxCells];    // packing: centre and horizontal half extent of each cube's box
    uint32_t cand[kMaxCub / 32 + kMaxOSph / 32];   // candidate obstacles of the particle (tower goal)
};

// dynamic shared memory: mbarrier | env cuboids | env spheres | boxes of the packing's walls | per-warp scratch
__host__ __device__ inline size_t s1_env_offset() { return 16; }
__host__ __device__ inline size_t s1_wall_offset(const Scalars& sc) {
    return 16 + (size_t)sc.n_cub * 64 + (size_t)sc.n_osph * 16;
}
__host__ __device__ inline size_t s1_warp_offset(const Scalars& sc) {
    return s1_wall_offset(sc) + (sc.kind == kKindPack ? (size_t)sc.n_cub * 32 : 0);
}
static size_t s1_smem_bytes(const Scalars& sc) { return s1_warp_offset(sc) + sizeof(S1Warp) * kS1Warps; }

struct S1Smem {
    uint64_t* bar;
    float4* cub;
    float4* osph;
    float4* wall;
    S1Warp* warp;
};

template <bool kTower>
__device__ __forceinline__ bool s1_setup(const Scalars& sc, DevTables t, S1Smem& s, int* err) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    s.bar = reinterpret_cast<uint64_t*>(smem_raw);
    s.cub = reinterpret_cast<float4*>(smem_raw + s1_env_offset());
    s.osph = s.cub + 4 * sc.n_cub;
    s.wall = reinterpret_cast<float4*>(smem_raw + s1_wall_offset(sc));
    s.warp = reinterpret_cast<S1Warp*>(smem_raw + s1_warp_offset(sc));
    const bool staged = stage_tables(s.cub, t.cub, (uint32_t)sc.n_cub * 64u, s.osph, t.osph, (uint32_t)sc.n_osph * 16u, s.bar, err);
    if (!kTower && staged && sc.kind == kKindPack) {
        for (int o = threadIdx.x; o < sc.n_cub; o += kS1Threads) {
            const float4 c0 = s.cub[4 * o], c1 = s.cub[4 * o + 1], c2 = s.cub[4 * o + 2], c3 = s.cub[4 * o + 3];
            s.wall[2 * o] = c0;
            s.wall[2 * o + 1] = make_float4(fabsf(c1.x) * c1.w + fabsf(c2.x) * c2.w + fabsf(c3.x) * c3.w,
                                            fabsf(c1.y) * c1.w + fabsf(c2.y) * c2.w + fabsf(c3.y) * c3.w,
                                            fabsf(c1.z) * c1.w + fabsf(c2.z) * c2.w + fabsf(c3.z) * c3.w, 0.f);
        }
        __syncthreads();
    }
    return staged;
}

template <bool kTower>
__global__ void __launch_bounds__(kS1Threads) k_place_sample_cost(const __grid_constant__ Scalars sc, DevTables t, int n,
                                                                   uint32_t attempt, float* __restrict__ x_out,
                                                                   float* __restrict__ cost_out, int* err,
                                                                   const LoopCtl* __restrict__ ctl) {
    uint64_t key = sc.seed;   // the Philox key
    if (ctl) { attempt = ctl->attempt; key = ctl->seed; }
    S1Smem s;
    if (!s1_setup<kTower>(sc, t, s, err)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int p = blockIdx.x * kS1Warps + w;
    if (p >= n) return;
    S1Warp& W = s.warp[w];
    if (lane < sc.B) {
        const int i = lane;
        const U4 u = philox4x32_10((uint32_t)i, (uint32_t)p, kTagSample, attempt, key);
        const float zlo = sc.zlo[i];
        W.x[4 * i + 0] = sc.box_lo[0] + u01(u.x) * (sc.box_hi[0] - sc.box_lo[0]);
        W.x[4 * i + 1] = sc.box_lo[1] + u01(u.y) * (sc.box_hi[1] - sc.box_lo[1]);
        W.x[4 * i + 2] = zlo + u01(u.z) * (sc.box_hi[2] - zlo);
        W.x[4 * i + 3] = -kPi + u01(u.w) * (2.f * kPi);
    }
    __syncwarp();
    PlaceOut o;
    place_eval<kTower>(sc, s.cub, s.wall, sc.n_cub, s.osph, sc.n_osph, W.x, false, kPlaceForward, nullptr, W.ps,
               W.gcell, W.cube, W.cand, &o);
    for (int v = lane; v < 4 * sc.B; v += 32) x_out[(size_t)v * n + p] = W.x[v];
    if (lane == 0) cost_out[p] = place_cost_value(sc, o);
}

template <bool kTower>
__global__ void __launch_bounds__(kS1Threads) k_place_eval(const __grid_constant__ Scalars sc, DevTables t, int n,
                                                            const float* __restrict__ x, int quad,
                                                            float* __restrict__ cost, float* __restrict__ grad,
                                                            float* __restrict__ metrics, float* __restrict__ terms,
                                                            int* err) {
    S1Smem s;
    if (!s1_setup<kTower>(sc, t, s, err)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int p = blockIdx.x * kS1Warps + w;
    if (p >= n) return;
    S1Warp& W = s.warp[w];
    for (int v = lane; v < 4 * sc.B; v += 32) W.x[v] = x[(size_t)v * n + p];
    __syncwarp();
    PlaceOut o;
    place_eval<kTower>(sc, s.cub, s.wall, sc.n_cub, s.osph, sc.n_osph, W.x, quad != 0, grad ? kPlaceStage1 : kPlaceForward, W.g, W.ps,
               W.gcell, W.cube, W.cand, &o);
    if (grad)
        for (int v = lane; v < 4 * sc.B; v += 32) grad[(size_t)v * n + p] = W.g[v];
    if (lane == 0) {
        if (cost) cost[p] = place_cost_value(sc, o);
        if (metrics) { metrics[3 * p] = o.maxpen; metrics[3 * p + 1] = o.maxD; metrics[3 * p + 2] = o.maxdz; }
        if (terms) { terms[3 * p] = o.c_stable; terms[3 * p + 1] = o.c_height; terms[3 * p + 2] = o.c_coll; }
    }
}

// Alg. 1, linear cost descent (eta = eta_init (1 - k/K_lin)) then quadratic refinement
// (fixed alpha), each followed by the box projection; then GetSatisfyingParticles and
// the final (quadratic-form) cost.  The whole loop runs inside one launch.
template <bool kTower>
__global__ void __launch_bounds__(kS1Threads, 4) k_place_descend(const __grid_constant__ Scalars sc, DevTables t, int m,
                                                               const float* __restrict__ x_src, int ld_src,
                                                               const int* __restrict__ idx, float* __restrict__ x_dst,
                                                               int k_lin, int k_quad, float* __restrict__ cost,
                                                               int* __restrict__ sat, float* __restrict__ metrics,
                                                               int* err) {
    S1Smem s;
    if (!s1_setup<kTower>(sc, t, s, err)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int p = blockIdx.x * kS1Warps + w;
    if (p >= m) return;
    S1Warp& W = s.warp[w];
    const int nv = 4 * sc.B;
    const int src = idx ? idx[p] : p;
    for (int v = lane; v < nv; v += 32) W.x[v] = x_src[(size_t)v * ld_src + src];
    __syncwarp();
    PlaceOut o;
    for (int k = 1; k <= k_lin; ++k) {
        const float eta = sc.eta_init * (1.f - (float)k / (float)k_lin);
        place_eval<kTower>(sc, s.cub, s.wall, sc.n_cub, s.osph, sc.n_osph, W.x, false, kPlaceStage1, W.g, W.ps,
               W.gcell, W.cube, W.cand, nullptr);
        for (int v = lane; v < nv; v += 32) W.x[v] = place_clamp(sc, v, W.x[v] - eta * W.g[v]);
        __syncwarp();
    }
    for (int k = 1; k <= k_quad; ++k) {
        place_eval<kTower>(sc, s.cub, s.wall, sc.n_cub, s.osph, sc.n_osph, W.x, true, kPlaceStage1, W.g, W.ps,
               W.gcell, W.cube, W.cand, nullptr);
        for (int v = lane; v < nv; v += 32) W.x[v] = place_clamp(sc, v, W.x[v] - sc.alpha * W.g[v]);
        __syncwarp();
    }
    place_eval<kTower>(sc, s.cub, s.wall, sc.n_cub, s.osph, sc.n_osph, W.x, true, kPlaceForward, nullptr, W.ps,
               W.gcell, W.cube, W.cand, &o);
    for (int v = lane; v < nv; v += 32) x_dst[(size_t)v * m + p] = W.x[v];
    if (lane == 0) {
        if (cost) cost[p] = place_cost_value(sc, o);
        if (sat) sat[p] = (o.maxpen <= sc.eps && o.maxD <= sc.eps && o.maxdz <= sc.eps) ? 1 : 0;
        if (metrics) { metrics[3 * p] = o.maxpen; metrics[3 * p + 1] = o.maxD; metrics[3 * p + 2] = o.maxdz; }
    }
}

__global__ void k_mask_costs(const float* __restrict__ cost, const int* __restrict__ sat, int n,
                             float* __restrict__ out, int* __restrict__ n_sat) {
    __shared__ int cnt;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    int mine = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const bool ok = sat[i] != 0;
        out[i] = ok ? cost[i] : __int_as_float(0x7fc00000);
        mine += ok;
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0) atomicAdd(&cnt, mine);
    __syncthreads();
    if (threadIdx.x == 0) *n_sat = cnt;
}

__global__ void k_gather_soa_to_aos(const float* __restrict__ src, int ld_src, int nv, const int* __restrict__ idx,
                                    int k, float* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= k * nv) return;
    const int r = i / nv, v = i % nv;
    out[i] = src[(size_t)v * ld_src + idx[r]];
}

// ------------------------------------------------------------------------------ launchers
// Towers run instantiations without the packing's evaluation, which takes registers from theirs (descending
// 4096 10-block towers: 412 us in the general kernel, 400 in the tower's; 64 one-block towers: 81 and 68 us).  The general
// one keeps both goals although packings alone come to it: compiled without the tower's evaluation, the
// packing's linear steps contract other products into FMAs, and a descent through contacts ends elsewhere.
template <typename Kernel, typename... Args>
static cudaError_t s1_launch(Kernel tower, Kernel any, const Scalars& sc, int n, cudaStream_t st, Args... args) {
    if (n <= 0) return cudaSuccess;
    const Kernel k = sc.kind == kKindPack ? any : tower;
    const size_t bytes = s1_smem_bytes(sc);
    cudaError_t e = allow_max_dynamic_smem(k, bytes);
    if (e != cudaSuccess) return e;
    k<<<(n + kS1Warps - 1) / kS1Warps, kS1Threads, bytes, st>>>(sc, args...);
    return cudaGetLastError();
}

cudaError_t launch_place_sample_cost(const Scalars& sc, DevTables t, int n, uint32_t attempt, float* x, float* cost,
                                     int* err, cudaStream_t st, const LoopCtl* ctl) {
    return s1_launch(k_place_sample_cost<true>, k_place_sample_cost<false>, sc, n, st, t, n, attempt, x, cost, err, ctl);
}

cudaError_t launch_place_eval(const Scalars& sc, DevTables t, int n, const float* x, int quad, float* cost, float* grad,
                              float* metrics, float* terms, int* err, cudaStream_t st) {
    return s1_launch(k_place_eval<true>, k_place_eval<false>, sc, n, st, t, n, x, quad, cost, grad, metrics, terms, err);
}

cudaError_t launch_place_descend(const Scalars& sc, DevTables t, int m, const float* x_src, int ld_src, const int* idx,
                                 float* x_dst, int k_lin, int k_quad, float* cost, int* sat, float* metrics, int* err,
                                 cudaStream_t st) {
    return s1_launch(k_place_descend<true>, k_place_descend<false>, sc, m, st, t, m, x_src, ld_src, idx, x_dst, k_lin,
                     k_quad, cost, sat, metrics, err);
}

static int next_pow2(int v) {
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

size_t topk_smem_bytes(int n, int k) {
    return (size_t)next_pow2(k < 1 ? 1 : k) * 8 + (size_t)n * 4;
}

cudaError_t launch_topk(const float* cost, int n, int k, int* idx, float* cost_out, cudaStream_t st) {
    if (n <= 0 || k <= 0) return cudaSuccess;
    if (k > n) k = n;
    const int kp2 = next_pow2(k);
    const size_t bytes = topk_smem_bytes(n, k);
    cudaError_t e = allow_max_dynamic_smem(k_topk, bytes);
    if (e != cudaSuccess) return e;
    k_topk<<<1, kSelectThreads, bytes, st>>>(cost, n, k, idx, cost_out, kp2);
    return cudaGetLastError();
}

cudaError_t launch_mask_costs(const float* cost, const int* sat, int n, float* cost_masked, int* n_sat,
                              cudaStream_t st) {
    k_mask_costs<<<1, 1024, 0, st>>>(cost, sat, n, cost_masked, n_sat);
    return cudaGetLastError();
}

cudaError_t launch_gather_soa_to_aos(const float* src, int ld_src, int nv, const int* idx, int k, float* out,
                                     cudaStream_t st) {
    if (k <= 0) return cudaSuccess;
    const int total = k * nv;
    k_gather_soa_to_aos<<<(total + 255) / 256, 256, 0, st>>>(src, ld_src, nv, idx, k, out);
    return cudaGetLastError();
}

}  // namespace spasm
