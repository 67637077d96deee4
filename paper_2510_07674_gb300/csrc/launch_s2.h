// Host-side launchers of the stage-2 kernels (internal to the library).
#pragma once
#include "launch.h"

namespace spasm {

// Work counters of a persistent trajectory launch, zero between launches: the particles handed
// out after each group's first, and the groups that are done.
struct TrajWork {
    int next, done;
};

// Buffers of one trajectory-kernel launch (device pointers; any may be null unless noted).
struct TrajIO {
    float* q;          // [n][C][8] joint configurations (required); updated by a descent
    float* lam;        // [n][NR] multipliers
    float* mu;         // [n] penalty parameters
    float* L;          // [n] augmented-Lagrangian objective
    float* grad;       // [n][C][8] dL/dq (evaluation mode)
    float* groups;     // [n][6] C_start, C_arm, C_block, C_coll, C_stable, C_height
    float* h;          // [n][NR] residual vector
    float* metrics;    // [n][8] max pen, max grasp error, max tilt, placement max pen / CoM / height, path, rank cost
    int* sat;          // [n] satisfying flag
    unsigned long long* tests;   // [0] sphere-obstacle tests executed (after the exact cull), [1]
                                 // configurations whose kinematics and cull ran, [2] of those, the
                                 // ones with a candidate obstacle (sphere-level work); accumulated
    int k_steps;       // descent steps
    int init_multipliers;   // descent starts from lambda = 0, mu = mu0
    const int* active;  // optional device word: when it holds 0 or less the launch does nothing (the
                        // trajectory stage of a problem whose stage 1 found no placement)
    // Scratch that no other launch in flight may have: the collision gradient rows of the particle each
    // resident group works on, [traj_slots][C][16], and launch_traj's work counters, zero between
    // launches.  launch_traj takes neither as well (both null): the rows then lie in shared memory.
    float* rows;
    TrajWork* work;
    int row_stride;   // batched launches: floats from one group's rows to the next one's
};
// Particle groups resident at once: two CTAs of two groups on each of 152 SMs, or of four where
// the problem is small enough (traj_slots); a launch on a part with more SMs keeps to as many.
constexpr int kTrajSlots = 608;
constexpr size_t kHalfSmem = 228 * 512 - 1024;   // shared memory of each of two CTAs on an SM
int traj_slots(int B, int C, int n_cub, int n_osph);
enum TrajModeHost { kTrajModeEval = 0, kTrajModeDescend = 1 };

// One problem of a batched trajectory launch (device array, sorted by `first`).
struct TrajJob {
    const Scalars* sc;   // device copy of the problem constants
    DevTables tab;
    TrajIO io;
    int* err;
    int n;               // particles
    int first;           // index of the problem's first work item
};

// Particles per CTA of a launch of that many particles: the problem's setting, or the
// launcher's choice (traj_auto_ppc, given the shared memory of a CTA with two and with four
// particles, 0 where that shape is not to be used, the blocks and the configurations).
int traj_ppc(const TrajScalars& sc, long long particles);
int traj_auto_ppc(size_t cta_bytes_2, size_t cta_bytes_4, long long particles, int blocks, int C);
// IK at grasp/place poses + interpolation; particle p lifts placement p % n_place.  With
// ctl != nullptr the attempt counter, the placement count and the Philox key are read on the
// device (ctl->t_attempt, ctl->n_place, ctl->seed) in place of `attempt`, `n_place` and
// sc.seed, and the launch writes nothing when ctl->n_place is 0.
cudaError_t launch_lift(const Scalars& sc, int n, const float* place, int n_place, uint32_t attempt, float* q,
                        cudaStream_t st, const LoopCtl* ctl = nullptr);
cudaError_t launch_traj(const Scalars& sc, DevTables t, int n, int mode, const TrajIO& io, int* err, cudaStream_t st);
// Persistent batched launch over jobs[0..n_jobs) (n_items work items of per_fetch particles;
// *next must be 0); cta_bytes = the largest traj_cta_smem_bytes of the jobs; grid x ppc <=
// kTrajSlots.  tiling, ppc: the sphere tiling (Scalars::sphere_tiling) and the particles per CTA
// (1 or 2) of the launch, the same for every job.
cudaError_t launch_traj_batch(const TrajJob* jobs, int n_jobs, int n_items, int per_fetch, int mode, int* next,
                              size_t cta_bytes, int grid, cudaStream_t st, int tiling, int ppc);
// Upper bound on the batched kernel's static shared memory (its copies of two problems' constants).
constexpr size_t kBatchStaticSmem = 2 * (sizeof(TrajScalars) + sizeof(TrajIO) + 8) + 64;
// Resident CTAs per SM of the batched kernel at that shared-memory size of a CTA (0 on error
// or when it does not fit).
int traj_batch_ctas_per_sm(size_t cta_bytes, int tiling, int ppc);
// Resident CTAs per SM of the per-problem trajectory kernel for this problem's sizes and launch
// shape (0 if it does not fit).
int traj_ctas_per_sm(const TrajScalars& sc);
// Dynamic shared memory of one trajectory CTA with ppc particles.
// (batched: each group has its own environment tables; otherwise the CTA's groups share them).
size_t traj_cta_smem_bytes(const TrajScalars& sc, int ppc, bool batched);

}  // namespace spasm
