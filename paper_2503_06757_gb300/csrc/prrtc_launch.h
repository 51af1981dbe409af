// prrtc_launch.h -- descriptors shared by the host runtime and the planner
// kernels, and the kernel launchers each .cu file exports.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cfloat>
#include <climits>
#include <cmath>
#include <utility>

#include "prrtc.h"
#include "prrtc_device.cuh"

namespace prrtc {

constexpr int kRootParent = -2;    // parent of a tree root
constexpr int kMixK = 8;           // learned mixture components
constexpr int kGmmStride = kMixK + 2 * kMixK * kMaxDof;  // logits | means [8][16] | log-sigmas [8][16]
constexpr int kUnsetParent = -1;   // parent slot not written yet (0xFF fill)
constexpr int kHeldMeta = 8;       // ints per lockstep worker record

// Launch-wide parameters and bookkeeping (one per planning launch).
struct PlanGlobals {
  int n_problems;
  int mode;              // PRRTC_MODE_*
  int max_iters;
  int n_full;            // ceil(range / resolution): states of a full-length step
  float range;
  float resolution;
  uint32_t bias_thr;     // goal bias as a threshold on the top 24 bits of a Philox word
  int path_cap;
  unsigned long long t0;             // launch start (min over blocks, %globaltimer ns)
  unsigned long long time_limit_ns;  // 0 = none
  int cursor;            // work-queue ticket counter
  int queue[3];          // the same, one per launch of the deterministic schedules
  int left[2];           // problems that the first and the second of those left to the next
  int closed;            // problems that have ended
  int error;             // device-side error code (PRRTC_ERR_*), 0 = none
  int error_info;
  uint32_t learned_thr;  // learned-vs-uniform draw as a threshold on the top 24 bits of a Philox word
  const int* active;     // problems of this launch as indices into the descriptors (null: 0..n-1)
  unsigned long long slice_ns;  // 0 = run problems to completion; else stop starting iterations
                                // this long after the launch start (problems resume next launch)
  int sampler;           // PRRTC_SAMPLER_*
  uint32_t halton_offset;
  float dd_radius;       // dynamic domain: 0 = off
  float dd_alpha;
  float dd_min_radius;
  int workers;           // lockstep mode: iterations per round (B)
  uint32_t debug_wait_polls;  // test hook: bounded wait on ProblemState::never_set before a path walk
  int expansions;        // async: iterations a worker claims per atomic on the problem's counter
  int obstacle_tile;     // primitives per type per first-stage round (32 or 64): picks the kernel instance
};

// Check of the sampler and dynamic-domain fields of a parameter block; null
// when they are usable, else the reason.
inline const char* sampling_params_problem(const prrtc_params& p) {
  if (p.sampler != PRRTC_SAMPLER_PHILOX && p.sampler != PRRTC_SAMPLER_HALTON) return "unknown sampler";
  if (!(p.dd_radius >= 0.f)) return "dd_radius must be >= 0";
  if (p.dd_radius > 0.f) {
    if (!(p.dd_alpha >= 0.f && p.dd_alpha < 1.f)) return "dd_alpha must be in [0, 1)";
    if (!(p.dd_min_radius >= 0.f) || !std::isfinite(p.dd_min_radius)) return "dd_min_radius must be >= 0";
  }
  return nullptr;
}

// The launch-wide fields that follow from a parameter block alone.
inline void globals_from_params(PlanGlobals& G, const prrtc_params& p) {
  G.mode = p.mode;
  G.max_iters = p.max_iters;
  G.n_full = (int)std::ceil((double)p.range / (double)p.resolution);
  if (G.n_full < 1) G.n_full = 1;
  G.range = p.range;
  G.resolution = p.resolution;
  G.bias_thr = (uint32_t)std::ceil((double)p.goal_bias * 16777216.0);
  G.learned_thr = (uint32_t)std::ceil((double)p.learned_ratio * 16777216.0);
  G.path_cap = p.path_capacity;
  G.sampler = p.sampler;
  G.halton_offset = p.halton_offset;
  G.dd_radius = p.dd_radius;
  G.dd_alpha = p.dd_alpha;
  G.dd_min_radius = p.dd_min_radius;
  G.workers = p.mode == PRRTC_MODE_LOCKSTEP ? p.workers : 1;
  G.debug_wait_polls = p.debug_wait_polls > 0 ? (uint32_t)p.debug_wait_polls : 0u;
  G.expansions = (p.mode == PRRTC_MODE_ASYNC && p.expansions > 1) ? p.expansions : 1;
  G.obstacle_tile = p.obstacle_tile == 64 ? 64 : 32;
}

// Per-problem inputs (uploaded every call).
struct ProblemDesc {
  const RobotDev* robot;
  EnvView env;
  float* nodes[2];       // [cap * dpad] per tree, rows NaN until written
  int* parent[2];        // [cap] per tree
  float* radius[2];      // [cap] per tree: dynamic-domain radius, NaN = unbounded
  float* path;           // [path_cap * dof]
  int* path_idx;         // [path_cap] scratch of (tree << 30 | node)
  int cap;
  int dpad;
  int dof;
  int n_spheres;         // distinct spheres (staging size)
  int n_pairs;
  uint32_t key_lo, key_hi;
  uint32_t pid;
  const float* gmm;      // learned mixture (kGmmStride floats, device) or null
  // serial and lockstep mode: the rows each virtual worker holds back, [workers][held_rows * dpad],
  // and per worker kHeldMeta ints (see LockstepHeld in prrtc_plan.cu); null otherwise
  float* held;
  int* held_meta;
  int held_rows;         // rows one iteration can add: 1 + the most connect steps
  float q_start[kMaxDof];
  float q_goal[kMaxDof];
};

// Per-problem device state.  The setup kernel resets everything but the
// arena bookkeeping (used[]), which tells it which rows to clear next time.
struct ProblemState {
  int iter;              // Alg. 1 iteration tickets handed out
  int count[2];          // tree sizes (may exceed cap after failed insertions)
  int solved;
  int done;
  int timed_out;
  int pre_status;        // start / goal in collision
  int s_tree;            // tree extended by the winning iteration
  int join_s, join_o;
  int path_n;
  int path_status;
  double cost;
  unsigned long long t_solve;
  unsigned long long edges, edge_states, sphere_tests, pair_tests, fk_states, nn_nodes, iterations, insert_fail;
  unsigned long long dd_rejected;
  unsigned long long prim_tests[4];
  unsigned long long verdict_states;
  // deterministic schedules: entry k of the lists of problems left to the second and third launch
  int left[2];
  int ahead;             // and how many rounds ran between two that changed a tree lately, x 16
  // arena bookkeeping, preserved across launches
  int used_rows[2];
  int used_dpad;
  int never_set;         // stays 0: the flag the bounded-wait test hook waits on
};

// Alg. 1 iterations a problem ran: the tickets handed out, or with batched
// claims (expansions > 1) the iteration bodies the workers counted.
inline int reported_iterations(const ProblemState& S, const prrtc_params& p) {
  const long long n = (p.mode == PRRTC_MODE_ASYNC && p.expansions > 1) ? (long long)S.iterations : (long long)S.iter;
  return (int)(n < p.max_iters ? n : p.max_iters);
}

// The check kernel lets a link skip the obstacles when its bounding sphere, its
// radius times kReachSlack, stays clear of a box around all of them.
constexpr float kReachSlack = 1.0012f;

// Box (lo, hi) that every sphere touching the obstacle (packed as in EnvView,
// kind 0..3) reaches with its radius times kReachSlack.  The kernels test a box
// in the coordinates A v of its rows as they were given: the box reaches as far
// as the rows of A^-1 say, and a sphere's radius grows by at most |A^-1|.  Rows
// that are not close to orthonormal (|A^-1| above 1.001, or a row longer than
// 1.1) get an unbounded box.  Cylinder axes may be off unit length by 1e-3.  The
// margin covers the kernels' own roundings.
inline void obstacle_bounds(int kind, const float4* e, float lo[3], float hi[3]) {
  const double c[3] = {e[0].x, e[0].y, e[0].z};
  double ext[3];
  if (kind == 0) {
    ext[0] = e[1].x; ext[1] = e[1].y; ext[2] = e[1].z;
  } else if (kind == 1) {
    double A[3][3], cross[3][3], longest = 0.0;
    for (int j = 0; j < 3; ++j) {
      A[j][0] = e[2 + j].x; A[j][1] = e[2 + j].y; A[j][2] = e[2 + j].z;
      longest = std::max(longest, std::sqrt(A[j][0] * A[j][0] + A[j][1] * A[j][1] + A[j][2] * A[j][2]));
    }
    for (int j = 0; j < 3; ++j) {  // column j of A^-1 times the determinant
      const double* u = A[(j + 1) % 3];
      const double* w = A[(j + 2) % 3];
      for (int a = 0; a < 3; ++a) cross[j][a] = u[(a + 1) % 3] * w[(a + 2) % 3] - u[(a + 2) % 3] * w[(a + 1) % 3];
    }
    const double det = A[0][0] * cross[0][0] + A[0][1] * cross[0][1] + A[0][2] * cross[0][2];
    const double h[3] = {e[1].x, e[1].y, e[1].z};
    double inv[3][3];
    for (int a = 0; a < 3; ++a) {
      ext[a] = 0.0;
      for (int j = 0; j < 3; ++j) {
        inv[a][j] = cross[j][a] / det;
        ext[a] += std::fabs(inv[a][j]) * h[j];
      }
    }
    bool bounded = longest < 1.1;
    for (int a = 0; a < 3; ++a) {  // |A^-1|^2 is at most the largest row sum of A^-1 A^-T
      double sum = 0.0;
      for (int b = 0; b < 3; ++b)
        sum += std::fabs(inv[a][0] * inv[b][0] + inv[a][1] * inv[b][1] + inv[a][2] * inv[b][2]);
      bounded = bounded && sum < 1.002;
    }
    if (!bounded) ext[0] = ext[1] = ext[2] = INFINITY;
  } else if (kind == 2) {
    const double ax[3] = {e[1].x, e[1].y, e[1].z};
    const double len = std::sqrt(ax[0] * ax[0] + ax[1] * ax[1] + ax[2] * ax[2]);
    for (int a = 0; a < 3; ++a) {
      const double u = std::fabs(ax[a]) / len;
      ext[a] = (double)e[0].w * std::sqrt(std::max(0.0, 1.0 - u * u)) + (double)e[1].w / len * u;
    }
  } else {
    ext[0] = ext[1] = ext[2] = e[0].w;
  }
  for (int a = 0; a < 3; ++a) {
    const double m = ext[a] + 1e-4 + 1e-5 * (std::fabs(c[a]) + ext[a]);
    lo[a] = (float)std::max(c[a] - m, -(double)FLT_MAX);
    hi[a] = (float)std::min(c[a] + m, (double)FLT_MAX);
  }
}

// Launchers (return cudaError_t of the launch).
// slots (nullable): a warp per state whatever n, and its counters (sphere
// passes, pair tests, the four second-stage counts, as 32-bit words) at
// slots[2 * state] instead of summed into counters[7].  All pointers may be
// pinned host memory.
// env.data holds two float4 more than its primitives: the lower and the upper
// corner of the box around all of them (obstacle_bounds).
cudaError_t launch_check_states(const RobotDev* robot, const RobotHeader& host_header, EnvView env, const float* q,
                                int n, uint8_t* valid, float* spheres, unsigned long long* counters, uint4* slots,
                                int* error, cudaStream_t stream);

// Philox4x32-10 of n counters (device arrays of 4n words each).
cudaError_t launch_philox(const uint32_t* ctr, int n, uint64_t key, uint32_t* out, cudaStream_t stream);

// FP32 FMA loop over 8 blocks of 256 threads per SM; *lane_ops receives the
// FMAs it issues (one lane-op each).  sink: one float per block (never written
// in practice).
cudaError_t launch_fma_loop(int sm_count, int iters, float* sink, cudaStream_t stream, long long* lane_ops);

// idx (nullable, device): the problems to set up, as indices into desc/state.
// error (nullable, device): receives PRRTC_ERR_TIMEOUT if a block's staging
// copies did not complete within the bounded wait.
cudaError_t launch_setup(const ProblemDesc* desc, ProblemState* state, int n, int max_spheres, int max_pairs,
                         int max_env_f4, cudaStream_t stream, const int* idx = nullptr, int* error = nullptr);

struct PlanLaunch {
  int grid;
  int warps;
  int smem;
  int robot_bytes;
  int env_bytes;
  int stage_bytes;
};

// Launches of the deterministic schedules (serial and lockstep mode): up to
// three in a row, with growing clusters of blocks per problem.
struct RoundsLaunch {
  int robot_bytes;
  int env_bytes;
  int stage_bytes;
  int workers;           // virtual workers of the largest cluster: slices of a problem's held rows
  int n_phases;
  struct Phase {
    int warps;           // per block
    int smem;
    int blocks;          // blocks of a cluster, which runs one problem
    int grid;
    int it_limit;        // from this many iterations on a problem is left to the next launch ...
    int open;            // ... once this many problems or fewer are open
  } ph[3];
};
// Easy problems are solved within a few rounds of 16 workers and rarely let a
// round of more of them count (one iteration in seven adds a row); the few
// hard ones, which set the batch's time, add a row in a hundred iterations or
// more and take all the workers they get.  So each launch gives what the one
// before left a larger cluster: from a number of iterations on, once no more
// problems are open than the next launch has clusters at once (Phase::open).
// Where many stay open they keep their clusters: 35 of 90 problems in clusters
// of 16, nine at a time, took twice as long as side by side in small ones, and
// a part of them sent on ran after the rest.  Kernel time (ms; limits of the
// first / second launch in iterations), sums over six sets of 200 shelf problems
// (serial, lockstep), then sets of 400, 100 and 40:
//   16 warps, clusters 1 / 4 / 16, 256 / 1024   16.7 13.8   3.64 2.69   1.62 1.24   0.89 0.70
//   ... no smaller blocks at first              16.3 13.3   3.81 2.66   1.62 1.24   0.88 0.70
//   ... 64 / 512                                16.2 13.9   3.63 2.74   1.59 1.21   0.97 0.77
//   ... 384 / 4096                              18.1 15.0   3.77 2.75   2.07 1.42   0.94 0.73
//   ... 768 / 8192                              20.2 17.6   4.20 3.30   2.11 1.86   0.94 0.73
//   clusters 1 / 2 / 16                         18.5 14.7   4.09 2.96   1.84 1.29   0.89 0.69
//   clusters 1 / 8 / 16                         18.0 16.0   3.81 2.98   1.44 1.09   0.88 0.70
//   clusters 1 / 4 / 8                          21.3 18.2   4.23 3.31   1.79 1.37   0.92 0.70
//   12 warps (6 at first)                       19.0 15.8   4.11 3.22   1.67 1.29   0.97 0.76
// (one warp a problem, one block a problem: 121 to 270 and 16 to 40 a set).  The
// smaller blocks of the first launch, two on an SM, are for batches of more
// problems than SMs that are over soon: 200 problems of eight iterations 156 ->
// 128 us with 8 workers a round, 50 of them waited for an SM before.
constexpr int kRoundsWarps = 16, kRoundsManyWarps = 8;
constexpr int kRoundsSmem = 226 * 1024;
constexpr int kRoundsMidCluster = 4, kRoundsMaxCluster = 16;
constexpr int kRoundsFirstIters = 256, kRoundsMidIters = 1024;

// base: the launch of plan_launch_config for the same arguments.  held_floats:
// floats of held rows per virtual worker, over all problems; held_limit: the
// most that may be allocated.  radii: dynamic domain is on.
RoundsLaunch rounds_launch_config(const PlanLaunch& base, int n_problems, int mode, int blocks, int warps, int workers,
                                  size_t held_floats, size_t held_limit, bool radii, int sm_count);

// The rule behind rounds_launch_config.  per_sm(warps, smem): resident blocks
// of that shape; max_cluster(warps, smem): its largest cluster.  The held rows
// of every launch stay within held_limit: fewer warps where those of a single
// block would exceed it, down to one round of `workers`, which the caller has
// checked.
template <class PerSm, class MaxCluster>
inline RoundsLaunch rounds_shape(const PlanLaunch& base, int n_problems, int mode, int blocks, int warps, int workers,
                                 size_t held_floats, size_t held_limit, bool radii, int sm_count, PerSm per_sm,
                                 MaxCluster max_cluster) {
  RoundsLaunch c{};
  c.robot_bytes = base.robot_bytes;
  c.env_bytes = base.env_bytes;
  c.stage_bytes = base.stage_bytes + (int)sizeof(WarpCount);  // a second counter block per warp
  const bool fixed = mode == PRRTC_MODE_LOCKSTEP && warps > 0;  // the caller's warps per block
  const int B = mode == PRRTC_MODE_LOCKSTEP ? workers : 1;
  auto smem = [&](int w) { return c.robot_bytes + c.env_bytes + w * c.stage_bytes; };
  // virtual workers of a cluster of C blocks of w warps
  auto virt = [&](int C, int w) { return std::max(C * w / B, 1) * B; };
  auto held = [&](int C, int w) { return held_floats * (size_t)virt(C, w); };
  int w = fixed ? base.warps : kRoundsWarps;
  while (w > 1 && smem(w) > kRoundsSmem) --w;
  while (w > B && held(1, w) > held_limit) --w;
  int most = (fixed || blocks > 0) ? 1 : max_cluster(w, smem(w));
  if (radii)  // one round at a time, as a rule: no larger cluster than it has work for
    for (int C = 1; C < most; C *= 2)
      if (C * w >= B) most = C;
  auto fits = [&](int C) { return C <= most && held(C, w) <= held_limit; };
  // the first launch: one wave of clusters
  int C = 1;
  while (n_problems * C * 2 <= sm_count && fits(2 * C)) C *= 2;
  for (;;) {
    RoundsLaunch::Phase& ph = c.ph[c.n_phases];
    // more problems than SMs: two smaller blocks on each at first
    const bool many = n_problems > sm_count && !fixed && c.n_phases == 0 && B <= kRoundsManyWarps;
    ph.warps = many ? std::min(w, kRoundsManyWarps) : w;
    ph.smem = smem(ph.warps);
    ph.blocks = C;
    ph.grid = (blocks > 0 ? blocks : std::min(n_problems, std::max(per_sm(ph.warps, ph.smem) * sm_count / C, 1))) * C;
    ph.it_limit = INT_MAX;
    ph.open = 0;
    if (c.n_phases++) {
      RoundsLaunch::Phase& prev = c.ph[c.n_phases - 2];
      // each problem at once, or as many times as a round of many workers gets shorter
      prev.open = ph.grid / C * std::max(1, std::min(C / prev.blocks, B / (prev.blocks * prev.warps)));
    }
    c.workers = std::max(c.workers, virt(C, ph.warps));
    const int next = std::min(C < kRoundsMidCluster ? kRoundsMidCluster : kRoundsMaxCluster, most);
    if (next <= C || !fits(next) || c.n_phases == 3) break;
    ph.it_limit = C == 1 ? kRoundsFirstIters : kRoundsMidIters;
    C = next;
  }
  return c;
}

// workers: the lockstep round size (PRRTC_MODE_LOCKSTEP), else ignored.
PlanLaunch plan_launch_config(int n_problems, int mode, int blocks, int warps, int max_spheres, int max_pairs,
                              int max_env_f4, int sm_count, int workers = 1);

// obstacle_tile: 64 launches the 64-obstacle-tile instance of the kernel,
// anything else the 32 one (launch_rounds always uses 32).  lean: the
// instance without the learned mixture draw, the Halton sampler, distance
// fields, oriented boxes and one-stage links; only for batches that use none of
// them
// (problem_is_lean).
cudaError_t launch_plan(const PlanGlobals* g, const ProblemDesc* desc, ProblemState* state, const PlanLaunch& cfg,
                        int obstacle_tile, bool lean, cudaStream_t stream);
cudaError_t launch_rounds(const PlanGlobals* g, const ProblemDesc* desc, ProblemState* state, const RoundsLaunch& cfg,
                          bool lean, cudaStream_t stream);

// Whether the lean planner instance serves a problem: no mixture, no distance
// field, at least one primitive and no oriented box, a bounding sphere on every
// robot link that has spheres (with the sphere hierarchy on), and revolute
// joints within +-3.2 rad.  The batch also needs Philox sampling and no dynamic
// domain.  The batch is lean when every
// problem is and the sampler is Philox.
inline bool problem_is_lean(const RobotHeader& H, const ProblemDesc& D) {
  if (D.gmm || D.env.esdf.v || D.env.n_float4() == 0 || D.env.n_obb || !H.two_stage) return false;
  for (int f = 0; f < H.dof; ++f) {
    if (H.sph_begin[f + 1] > H.sph_begin[f] && !(H.coarse[f].w > 0.f)) return false;
    // every joint value the planner forms lies between the limits, the start and
    // the goal: within +-3.2 rad the hardware sine/cosine is the one taken
    const bool revolute = H.jtype[f] == kRevZ || H.jtype[f] == kRevY || H.jtype[f] == kRevX;
    const float lo = std::min({H.lo[f], D.q_start[f], D.q_goal[f]});
    const float hi = std::max({H.lo[f] + H.span[f], D.q_start[f], D.q_goal[f]});
    if (revolute && !(lo >= -3.2f && hi <= 3.2f)) return false;
  }
  return true;
}

// Clear-list bookkeeping after a plan: rows each tree used, for the next setup.
cudaError_t launch_record_usage(const ProblemDesc* desc, ProblemState* state, int n, cudaStream_t stream,
                                const int* idx = nullptr);

// Copy every problem's path into one packed buffer; offsets[p]..offsets[p+1]
// is problem p's float range (n + 1 entries, device memory).
cudaError_t launch_gather_paths(const ProblemDesc* desc, const int* offsets, int n, float* out, cudaStream_t stream);

// The first `rows` rows of each solved problem's path (dof floats per row)
// into out + p * stride; stride >= rows * dof.
cudaError_t launch_gather_heads(const ProblemDesc* desc, const ProblemState* state, int n, int rows, int stride,
                                float* out, cudaStream_t stream);

// Distance fields (prrtc_esdf.cu): occupancy of voxel centres inside the
// environment's primitives, and the signed distance transform of an
// occupancy grid of V voxels (tmp: kEsdfTmpBytes * V bytes).
constexpr size_t kEsdfTmpBytes = sizeof(int) + sizeof(int16_t);
cudaError_t launch_voxelize(const EnvView& env, const float origin[3], float voxel, const int dims[3], uint8_t* occ,
                            cudaStream_t stream);
cudaError_t launch_esdf(const uint8_t* occ, const int dims[3], float voxel, void* tmp, float* out,
                        cudaStream_t stream);

// Runs set(), a kernel attribute of the current device `dev`, unless it has
// succeeded there before (`done`: one bit per device, one word per kernel).  An
// attribute belongs to a device: a process may use several, from several
// threads.
template <class F>
inline cudaError_t once_per_device(std::atomic<uint64_t>& done, int dev, F set) {
  const bool known = dev >= 0 && dev < 64;
  if (known && (done.load(std::memory_order_acquire) >> dev & 1u)) return cudaSuccess;
  const cudaError_t e = set();
  if (e == cudaSuccess && known) done.fetch_or((uint64_t)1 << dev, std::memory_order_release);
  return e;
}

// Launches of a chain of short kernels overlap: a kernel launched with
// launch_overlapped may start while the kernel before it in the stream still
// runs; it must call wait_before() ahead of its first access to global memory
// and may call let_next_start() once its own start-up is over.  A kernel that
// needs nothing of the one before it (and whose operands that one waited for
// ahead of its let_next_start()) may call wait_before() at its end instead: the
// two run side by side, and launches still end in order.
#ifdef __CUDACC__
__device__ __forceinline__ void wait_before() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_overlapped(void (*fn)(P...), int grid, int block, size_t smem, cudaStream_t stream, int cluster,
                              A&&... args) {
  cudaLaunchAttribute at[2]{};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3((unsigned)grid);
  lc.blockDim = dim3((unsigned)block);
  lc.dynamicSmemBytes = smem;
  lc.stream = stream;
  lc.attrs = at;
  lc.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&lc, fn, std::forward<A>(args)...);
}
#endif

// Tensor-core GEMM (prrtc_gemm.cu): C[M,N] = A[M,K] B[N,K]^T (+bias, ReLU).
int gemm_bf16(const void* a, const void* b, int M, int N, int K, const float* bias, int relu, float* c32, int ldc32,
              void* c16, int ldc16, cudaStream_t stream);
// The same with row strides lda / ldb (elements, multiples of 8, >= K) of the
// operands, e.g. a column range of a wider weight matrix; splits_hint 0 = auto.
// flags: operands stored the other way round, A as [K x M] rows of lda >= M,
// B as [K x N] rows of ldb >= N (a gradient's operands as the layers wrote
// them, without a transposed copy).  mask (nullable, BF16 [M x N], row stride
// ldm): outputs become 0 where it is not above 0 (a ReLU's gradient);
// PRRTC_ERR_UNSUPPORTED for products above one wave.  kNextMayStart: the next
// launch on the stream calls wait_before() ahead of its first access to memory
// (or is an ordinary one), so it may start up while this one still runs.
constexpr int kTransA = 1, kTransB = 2, kNextMayStart = 4;
int gemm_bf16_ld(const void* a, int lda, const void* b, int ldb, int M, int N, int K, const float* bias, int relu,
                 float* c32, int ldc32, void* c16, int ldc16, cudaStream_t stream, int splits_hint, int flags,
                 const void* mask, int ldm);
// Weight gradients of n layers, dW [out x in] = dZ [rows x out]^T H [rows x
// in], in as few launches as their sizes allow (all dimensions multiples of 8,
// all pointers 16-byte aligned).  ready: the operands are complete and visible
// before the launch ahead of this call on the stream lets the next one start --
// it has called wait_before() by then, and writes none of them.  The products
// then run beside it and each other without a wait of their own; with any other
// launch ahead (or false) they would read operands that are still being written.
// The launch after the call has to wait as usual.
struct GradientProduct {
  const void* dz;
  const void* h;
  float* dw;
  int out, in, rows;
};
int gemm_gradients(const GradientProduct* p, int n, bool ready, cudaStream_t stream);
int gemm_take_error();
// Copies the kernels' error word to *out on `stream` (does not clear it).
cudaError_t gemm_read_error(int* out, cudaStream_t stream);

}  // namespace prrtc
