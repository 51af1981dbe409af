// prrtc_check.cu -- batched collision verdicts of given configurations
// (Sec. III-A): sphere-model FK, sphere-vs-primitive and self-collision tests.
// A lane per configuration, or a warp for calls of few; robot tables and the
// obstacle set are staged in shared memory by TMA bulk copies.  Used for the
// per-state parity check against the oracle and as the FP32-roofline
// microbenchmark.
#include <algorithm>
#include <array>
#include <map>
#include <mutex>
#include <utility>

#include "prrtc.h"
#include "prrtc_launch.h"

namespace prrtc {

namespace {

constexpr int kMaxCheckWarps = 16;
// Lanes that make a link's or a link pair's tests pay at once instead of waiting
// for a full warp in the queue.
constexpr int kDirect = 24;

// Robot header, pair tables and the first env_f4 words of the environment into
// shared memory by bulk copies (one thread); 0 when they did not complete within
// the bounded wait.
__device__ int stage_tables(const RobotDev* robot, const EnvView& env, RobotHeader* R, uint32_t* pair, float* thr,
                            float4* senv, int env_f4, int np_pad, uint64_t* bar, int* error) {
  mbar_init(bar, 1);
  mbar_arrive_expect_tx(bar, (uint32_t)sizeof(RobotHeader) + 8u * (uint32_t)np_pad + 16u * (uint32_t)env_f4);
  bulk_g2s(R, &robot->h, sizeof(RobotHeader), bar);
  if (np_pad) {
    bulk_g2s(pair, robot->pair, 4u * np_pad, bar);
    bulk_g2s(thr, robot->thr, 4u * np_pad, bar);
  }
  if (env_f4) bulk_g2s(senv, env.data, 16u * env_f4, bar);
  if (mbar_wait(bar, 0, 1u << 26)) return 1;
  atomicExch(error, PRRTC_ERR_TIMEOUT);
  mbar_wait(bar, 0, 1u << 26);  // the block leaves: its copies first (bounded)
  return 0;
}

// A warp's queues, rings of 64 entries: links that may touch the environment
// and link pairs that may touch (index << 5 | state), and per primitive type
// what a link's bounding sphere touches (primitive << 9 | link << 5 | state).
// They take the place of the joint values, which have been used by then.
struct CheckQueues {
  uint32_t prim[4][64];
  uint16_t link[64];
};
static_assert(kMaxDof <= 16 && PRRTC_MAX_OBSTACLES <= 1 << 23 && kMaxPairBlocks < 1 << 11, "queue entries");

// What the warp knows of its 32 states while their links meet the environment.
struct CheckWarp {
  const RobotHeader* R;
  const float* stage;       // [slot][x, y, z][state]
  CheckQueues* Q;
  uint32_t* hit;            // states known to collide
  int lane;
  int queued[4], done[4];   // entries of the primitive queues
  uint32_t fine[4];         // lane-level tests
  __device__ __forceinline__ bool collides(uint32_t state) const { return (*hit >> state) & 1u; }
};

// The next (at most 32) entries of one primitive queue: one link of one state
// against one primitive per lane, all spheres of the link.
template <int K>
__device__ __forceinline__ void prim_round(CheckWarp& w, const float4* __restrict__ prims) {
  __syncwarp();  // the queue and the hits
  const bool mine = w.done[K] + w.lane < w.queued[K];
  const uint32_t code = w.Q->prim[K][(mine ? w.done[K] + w.lane : w.done[K]) & 63];
  w.done[K] = min(w.done[K] + 32, w.queued[K]);
  const int state = (int)(code & 31u), link = (int)(code >> 5 & 15u);
  const bool live = mine && !w.collides(state);
  if (!__any_sync(kFull, live)) return;
  const int s0 = w.R->sph_begin[link], cnt = w.R->sph_begin[link + 1] - s0;
  const int most = __reduce_max_sync(kFull, live ? cnt : 0);
  float4 e[Prim<K>::kStride];
#pragma unroll
  for (int k = 0; k < Prim<K>::kStride; ++k) e[k] = prims[Prim<K>::kStride * (code >> 9) + k];
  const float* st = w.stage + s0 * 96 + state;
  bool hit = false;
#pragma unroll 2
  for (int s = 0; s < most; ++s) {
    const int at = min(s, cnt - 1);  // a link with fewer spheres tests its last one again
    hit |= Prim<K>::hit(e, st[at * 96], st[at * 96 + 32], st[at * 96 + 64], w.R->sph[s0 + at].w);
  }
  w.fine[K] += __reduce_add_sync(kFull, live ? (uint32_t)cnt : 0u);
  if (live && hit) atomicOr(w.hit, 1u << state);
}

// The bounding sphere (b, br) of one link of one state per lane (code: link <<
// 5 | state) against the primitives of one type, 32 at a time; what it touches
// goes into the type's queue.
template <int K>
__device__ __forceinline__ void link_stage(CheckWarp& w, const float4* __restrict__ prims, int n, float3 b, float br,
                                           uint32_t code, bool& live) {
  for (int base = 0; base < n; base += 32) {
    const int m = min(32, n - base);
    uint32_t flags = 0;
#pragma unroll Prim<K>::kUnroll
    for (int k = 0; k < m; ++k)
      flags |= (uint32_t)Prim<K>::hit(prims + Prim<K>::kStride * (base + k), b.x, b.y, b.z, br) << k;
    if (!live) flags = 0u;
    for (uint32_t who; (who = __ballot_sync(kFull, flags != 0u)) != 0u;) {
      if (flags) {
        const int at = w.queued[K] + __popc(who & ((1u << w.lane) - 1u));
        w.Q->prim[K][at & 63] = (uint32_t)(base + __ffs(flags) - 1) << 9 | code;
        flags &= flags - 1;
      }
      w.queued[K] += __popc(who);
      if (w.queued[K] - w.done[K] >= 32) {
        prim_round<K>(w, prims);
        __syncwarp();
        live = live && !w.collides(code & 31u);
        if (!live) flags = 0u;
      }
    }
    if (!__any_sync(kFull, live)) return;
  }
}

// The sphere pairs of one link pair of one state per lane (col: the state's
// column of the staged centres).  Lanes that are not live repeat what they
// have.
__device__ __forceinline__ bool block_hits(const RobotHeader* __restrict__ R, const uint32_t* __restrict__ pair,
                                           const float* __restrict__ thr, const float* __restrict__ col, int blk,
                                           bool live) {
  const uint32_t rg = R->blk_range[blk], cross = R->blk_cross[blk];
  const int k0 = (int)(rg & 0xffffu), k1 = (int)(rg >> 16);
  bool hit = false;
  if (__all_sync(kFull, !live || cross != 0u)) {
    constexpr int kC = 5;
    // the side with more spheres in the registers (columns), the other one passes (rows)
    const int ni = (int)(cross >> 16 & 0xffu), nj = (int)(cross >> 24);
    const bool swap = nj < ni;
    const int nr = swap ? nj : ni, nc = swap ? ni : nj;
    const int row_thr = swap ? 1 : nj, col_thr = swap ? nj : 1;
    const float* r0 = col + (swap ? cross >> 8 & 0xffu : cross & 0xffu) * 96;
    const float* c0 = col + (swap ? cross & 0xffu : cross >> 8 & 0xffu) * 96;
    const int rows = __reduce_max_sync(kFull, live ? nr : 0), cols = __reduce_max_sync(kFull, live ? nc : 0);
    for (int first = 0; first < cols; first += kC) {
      float x[kC], y[kC], z[kC];
      int at[kC];
#pragma unroll
      for (int c = 0; c < kC; ++c) {
        const int k = max(min(first + c, nc - 1), 0);  // a smaller block tests its last ones again
        x[c] = c0[k * 96];
        y[c] = c0[k * 96 + 32];
        z[c] = c0[k * 96 + 64];
        at[c] = k * col_thr;
      }
      const float* sr = r0;
      const float* t = thr + k0;
      for (int r = 0; r < rows; ++r) {
        const float rx = sr[0], ry = sr[32], rz = sr[64];
#pragma unroll
        for (int c = 0; c < kC; ++c) {
          const float dx = rx - x[c], dy = ry - y[c], dz = rz - z[c];
          hit |= fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < t[at[c]];
        }
        if (r + 1 < nr) {
          sr += 96;
          t += row_thr;
        }
      }
    }
  } else {
    const int len = __reduce_max_sync(kFull, live ? k1 - k0 : 0);
    for (int t = 0; t < len; ++t) {
      const int k = min(k0 + t, k1 - 1);
      const uint32_t pr = pair[k];
      const float* si = col + (pr & 0xffffu) * 96;
      const float* sj = col + (pr >> 16) * 96;
      const float dx = si[0] - sj[0], dy = si[32] - sj[32], dz = si[64] - sj[64];
      hit |= fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < thr[k];
    }
  }
  return hit;
}

// Verdicts of given configurations.  A lane places the spheres of one state
// and stages them.  Then the links that come near the box around the obstacles
// queue up, distal ones first; every 32 of them meet the primitives with their
// bounding spheres, one link of one state per lane; what those touch queues up
// again, and every 32 of those entries test the link's spheres.  Link pairs
// whose group spheres overlap go the same way, unless most lanes have them.
// In a shelf scene four links in ten meet the primitives and touch two of
// fifty, other ones in every lane; in clutter most states collide at their
// first link, which empties the warp early.
//
// What bounds it is instruction issue and its latencies (63% of the slots; 10,100
// instructions per 32 states of the 7-DoF arm when every lane met every
// primitive link by link, 4,600 now), and with 14 joints the latency of the
// staged reads, because the centres of 32 states take 18 KB: the block takes
// as many warps as the shared memory holds.  A million states in a shelf scene
// of 50 obstacles: 500 -> 213 us (both arms 1711 -> 652); among 600 mixed ones
// 4220 -> 1520.
//
// kTwoStage = false: robots without bounding spheres, with the two-stage check
// off, distance fields and empty environments.  Spheres meet the obstacles one
// by one; the queues only cost there (a million states of a point robot between
// two boxes 43 -> 28 us, of the 7-DoF arm without obstacles 132 -> 93).
template <bool kTwoStage>
__global__ void __maxnreg__(128) check_states_kernel(
    const RobotDev* __restrict__ robot, EnvView env, const float* __restrict__ q, int n, uint8_t* __restrict__ valid,
    float* __restrict__ spheres, unsigned long long* __restrict__ counters, int* __restrict__ error, int np_pad,
    int warp_floats, int q_floats) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ int s_ok;
  __shared__ WarpCount s_count[kMaxCheckWarps];
  __shared__ int16_t s_raw[PRRTC_MAX_SPHERES];
  __shared__ uint32_t s_hit[kMaxCheckWarps];  // states of the warp known to collide
  __shared__ int16_t s_bslot[kMaxDof];        // stage slot of the link's bounding sphere (its only sphere's own)
  RobotHeader* R = reinterpret_cast<RobotHeader*>(smem);
  uint32_t* pair = reinterpret_cast<uint32_t*>(smem + sizeof(RobotHeader));
  float* thr = reinterpret_cast<float*>(pair + np_pad);
  const int env_f4 = env.n_float4();
  float4* senv = reinterpret_cast<float4*>(thr + np_pad);
  const int box_f4 = env_f4 ? kEnvBox : 0;  // corners of the box around the obstacles
  float* warp_all = reinterpret_cast<float*>(senv + env_f4 + kEnvBox);

  if (threadIdx.x == 0) s_ok = stage_tables(robot, env, R, pair, thr, senv, env_f4 + box_f4, np_pad, &bar, error);
  if (spheres)
    for (int r = threadIdx.x; r < PRRTC_MAX_SPHERES; r += blockDim.x) s_raw[r] = robot->raw_to_distinct[r];
  __syncthreads();
  if (!s_ok) return;  // block-uniform

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int dof = R->dof, n_raw = R->n_raw, n_blocks = R->n_blocks;
  const uint32_t below = (1u << lane) - 1u;
  float* qst = warp_all + warp * warp_floats;  // [joint][lane], then the queues
  float* stage = qst + q_floats;               // [sphere, then link][x, y, z][lane]
  float4 box_lo, box_hi;
  if (env_f4) box_lo = senv[env_f4], box_hi = senv[env_f4 + 1];
  if (warp == 0) {
    const uint32_t bounds = __ballot_sync(kFull, lane < dof && R->coarse[lane].w > 0.f);
    if (lane < dof)
      s_bslot[lane] = (int16_t)((bounds >> lane & 1u) ? R->n_spheres + __popc(bounds & below) : R->sph_begin[lane]);
  }
  __syncthreads();
  const int gw = blockIdx.x * warps + warp;
  const int nw = gridDim.x * warps;
  const bool has_grid = env.esdf.v != nullptr;
  const float4* e_obb = senv + 2 * env.n_aabb;
  const float4* e_cyl = e_obb + 5 * env.n_obb;
  const float4* e_sph = e_cyl + 2 * env.n_cyl;
  WarpCount* wc = &s_count[warp];
  warp_count_clear(wc, lane);
  CheckWarp w;
  w.R = R;
  w.stage = stage;
  w.Q = reinterpret_cast<CheckQueues*>(qst);
  w.hit = &s_hit[warp];
  w.lane = lane;
  uint16_t* queue = w.Q->link;
  for (int base = gw * 32; base < n; base += nw * 32) {
    const int idx = base + lane;
    const bool active = idx < n;
    const size_t src = (size_t)(active ? idx : n - 1) * dof;
    __syncwarp();  // the lanes have read each other's staged centres and queue entries
#pragma unroll 4
    for (int j = 0; j < dof; ++j) qst[j * 32 + lane] = q[src + j];
    uint32_t passes = 0, pairs = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) w.queued[k] = w.done[k] = 0, w.fine[k] = 0u;
    Frame T;
#pragma unroll 1
    for (int i = 0; i < dof; ++i) {
      const float qi = qst[i * 32 + lane];
      fk_joint(R, i, qi, [qi](float& sn, float& cs) { joint_sincos<false>(qi, sn, cs); }, T);
      const int s0 = R->sph_begin[i], s1 = R->sph_begin[i + 1];
      if (R->coarse[i].w > 0.f) {
        const float3 c = T.at(R->coarse[i]);
        float* st = stage + s_bslot[i] * 96 + lane;
        st[0] = c.x;
        st[32] = c.y;
        st[64] = c.z;
      }
#pragma unroll 2
      for (int s = s0; s < s1; ++s) {
        const float3 c = T.at(R->sph[s]);
        float* st = stage + s * 96 + lane;
        st[0] = c.x;
        st[32] = c.y;
        st[64] = c.z;
      }
    }
    bool open = active;  // no collision found so far
    const int n_active = min(32, n - base);
    if (lane == 0) *w.hit = 0u;
    __syncwarp();
    if (kTwoStage) {
      int queued = 0, done = 0;
      for (int i = dof - 1; i >= 0; --i) {
        int enough = 32;
        if (R->sph_begin[i] != R->sph_begin[i + 1]) {
          const float* st = stage + s_bslot[i] * 96 + lane;
          const float r = R->grp[i].w * kReachSlack;
          const float dx = fmaxf(fmaxf(box_lo.x - st[0], st[0] - box_hi.x), 0.f);
          const float dy = fmaxf(fmaxf(box_lo.y - st[32], st[32] - box_hi.y), 0.f);
          const float dz = fmaxf(fmaxf(box_lo.z - st[64], st[64] - box_hi.z), 0.f);
          const bool near = open && !(fmaf(dx, dx, fmaf(dy, dy, dz * dz)) > r * r);
          const uint32_t m = __ballot_sync(kFull, near);
          if (near) queue[(queued + __popc(m & below)) & 63] = (uint16_t)(i << 5 | lane);
          queued += __popc(m);
          // In clutter nearly every state has the link and most collide there: mixed
          // with the next links they would be tested for nothing (both arms among 600
          // obstacles, 100,000 states with centres 350 us when all wait, 320 so)
          if (__popc(m) >= kDirect) enough = kDirect;
        }
        while (queued - done >= enough || (i == 0 && done < queued)) {
          __syncwarp();  // the queue and the hits
          const bool mine = done + lane < queued;
          const uint32_t code = queue[(mine ? done + lane : done) & 63];
          done = min(done + 32, queued);
          const int link = (int)(code >> 5), state = (int)(code & 31u);
          bool live = mine && !w.collides(state);
          const uint32_t lives = __ballot_sync(kFull, live);
          if (!lives) continue;
          passes += (uint32_t)__popc(lives);
          const float* bs = stage + s_bslot[link] * 96 + state;
          const float3 b = make_float3(bs[0], bs[32], bs[64]);
          const float br = R->grp[link].w;
          link_stage<kAabb>(w, senv, env.n_aabb, b, br, code, live);
          link_stage<kObb>(w, e_obb, env.n_obb, b, br, code, live);
          link_stage<kCyl>(w, e_cyl, env.n_cyl, b, br, code, live);
          link_stage<kSph>(w, e_sph, env.n_sph, b, br, code, live);
        }
        __syncwarp();
        open = open && !w.collides(lane);
        if (!__any_sync(kFull, open)) break;
      }
      // what is left in the queues
      if (w.done[kAabb] < w.queued[kAabb]) prim_round<kAabb>(w, senv);
      if (w.done[kObb] < w.queued[kObb]) prim_round<kObb>(w, e_obb);
      if (w.done[kCyl] < w.queued[kCyl]) prim_round<kCyl>(w, e_cyl);
      if (w.done[kSph] < w.queued[kSph]) prim_round<kSph>(w, e_sph);
      __syncwarp();
      open = open && !w.collides(lane);
    } else if (has_grid || env_f4) {
      for (int i = dof - 1; i >= 0; --i) {
        for (int s = R->sph_begin[i]; s < R->sph_begin[i + 1]; ++s) {
          const float* st = stage + s * 96 + lane;
          const float r = R->sph[s].w;
          passes += (uint32_t)n_active;
          if (has_grid && open) open = !(esdf_read(env.esdf, st[0], st[32], st[64]) < r);
          if (env_f4 &&
              sphere_hits_env(st[0], st[32], st[64], r, senv, env.n_aabb, env.n_obb, env.n_cyl, env.n_sph))
            open = false;
        }
        if (!__any_sync(kFull, open)) break;
      }
    }
    if (__any_sync(kFull, open)) {
      int queued = 0, done = 0;
      for (int blk = 0; blk < n_blocks; ++blk) {
        const uint32_t fr = R->blk_frames[blk];
        const float bt = R->blk_thr[blk];
        bool near = open;
        if (bt < INFINITY) {
          const float* ga = stage + s_bslot[fr & 0xffffu] * 96 + lane;
          const float* gb = stage + s_bslot[fr >> 16] * 96 + lane;
          const float dx = ga[0] - gb[0], dy = ga[32] - gb[32], dz = ga[64] - gb[64];
          near = open && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < bt;
          pairs += (uint32_t)__popc(__ballot_sync(kFull, open));
        }
        const uint32_t m = __ballot_sync(kFull, near);
        const uint32_t rg = R->blk_range[blk];
        pairs += (uint32_t)__popc(m) * ((rg >> 16) - (rg & 0xffffu));
        if (__popc(m) >= kDirect) {  // most lanes: at once, each its own state
          if (block_hits(R, pair, thr, stage + lane, blk, near) && near) open = false;
        } else {
          if (near) queue[(queued + __popc(m & below)) & 63] = (uint16_t)(blk << 5 | lane);
          queued += __popc(m);
        }
        while (queued - done >= 32 || (blk == n_blocks - 1 && done < queued)) {
          __syncwarp();  // the queue and the hits
          const bool mine = done + lane < queued;
          const uint32_t code = queue[(mine ? done + lane : done) & 63];
          done = min(done + 32, queued);
          const uint32_t state = code & 31u;
          // states that a direct test above closed need no more
          const uint32_t closed = __ballot_sync(kFull, !open);
          const bool live = mine && !((closed >> state) & 1u);
          if (!__any_sync(kFull, live)) continue;
          const bool hit = block_hits(R, pair, thr, stage + state, (int)(code >> 5), live);
          if (live && hit) atomicOr(w.hit, 1u << state);
          __syncwarp();
          open = open && !w.collides(lane);
        }
        if (!__any_sync(kFull, open)) break;
      }
    }
    if (active) valid[idx] = open ? 1 : 0;
    if (spheres) {
      // four spheres of eight states per turn: 64 contiguous bytes a state
      __syncwarp();
      float4* out = reinterpret_cast<float4*>(spheres) + (size_t)base * n_raw;
      for (int r0 = 0; r0 < n_raw; r0 += 4) {
        const int r = r0 + (lane & 3);
        const int ds = s_raw[min(r, n_raw - 1)];
        const float radius = R->sph[ds].w;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int state = 8 * k + (lane >> 2);
          const float* st = stage + ds * 96 + state;
          if (r < n_raw && base + state < n)
            out[(size_t)state * n_raw + r] = make_float4(st[0], st[32], st[64], radius);
        }
      }
    }
    if (lane == 0) {
      wc->fk_states += (unsigned long long)n_active;
      wc->sphere_tests += passes;
      wc->pair_tests += pairs;
#pragma unroll
      for (int k = 0; k < 4; ++k) wc->prim[k] += w.fine[k];
    }
  }
  // the warp's work counters: sphere passes, pairs, FK states, second-stage tests
  __syncwarp();
  if (lane < 7 && counters) atomicAdd(counters + lane, reinterpret_cast<const unsigned long long*>(wc)[lane]);
}

// One primitive type against one link of one state by a whole warp, a
// primitive per lane: its bounding sphere first (filter), then its spheres.
// `st`: centres, 3 floats each.  Returns the lane's hit.
template <int K>
__device__ __forceinline__ bool warp_link_stage(const float4* __restrict__ prims, int n, float3 b, float br,
                                                bool filter, const float* __restrict__ st,
                                                const float4* __restrict__ sph, int cnt, int lane, uint32_t& fine) {
  bool hit = false;
  for (int base = 0; base < n; base += 32) {
    const float4* e = prims + Prim<K>::kStride * min(base + lane, n - 1);
    const bool touch = base + lane < n && (!filter || Prim<K>::hit(e, b.x, b.y, b.z, br));
    const uint32_t m = __ballot_sync(kFull, touch);
    if (!m) continue;
    if (filter) fine += (uint32_t)__popc(m) * (uint32_t)cnt;
    if (touch)
      for (int s = 0; s < cnt; ++s) hit |= Prim<K>::hit(e, st[3 * s], st[3 * s + 1], st[3 * s + 2], sph[s].w);
  }
  return hit;
}

// The same verdicts for few states: one state per warp.  A lane per joint
// takes its sine and cosine, every lane runs the chain, a lane per sphere
// places it, a lane per primitive tests the links and a lane per pair the
// pairs -- the arithmetic of the kernel above, so the verdicts and centres are
// the same.  A few states alone take a warp of the other kernel through every
// link, primitive and pair in turn, and most of its lanes or warps are idle.
constexpr int kStateWarps = 4;
constexpr int kStateFloats = 3 * (kMaxDistinctSpheres + kMaxDof);

__global__ void __launch_bounds__(kStateWarps * 32) check_state_warps_kernel(
    const RobotDev* __restrict__ robot, EnvView env, const float* __restrict__ q, int n, uint8_t* __restrict__ valid,
    float* __restrict__ spheres, unsigned long long* __restrict__ counters, uint4* __restrict__ slots,
    int* __restrict__ error, int np_pad, int dof) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ int s_ok;
  __shared__ float s_stage[kStateWarps][kStateFloats];
  RobotHeader* R = reinterpret_cast<RobotHeader*>(smem);
  uint32_t* pair = reinterpret_cast<uint32_t*>(smem + sizeof(RobotHeader));
  float* thr = reinterpret_cast<float*>(pair + np_pad);
  const int env_f4 = env.n_float4();
  float4* senv = reinterpret_cast<float4*>(thr + np_pad);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int idx = blockIdx.x * kStateWarps + warp;
  // on its way while the tables are staged (it may come from host memory)
  const float ql = idx < n && lane < dof ? q[(size_t)idx * dof + lane] : 0.f;
  if (threadIdx.x == 0) s_ok = stage_tables(robot, env, R, pair, thr, senv, env_f4, np_pad, &bar, error);
  __syncthreads();
  if (!s_ok || idx >= n) return;  // nothing below waits for another warp
  const int n_raw = R->n_raw, n_pairs = R->n_pairs;
  float* stage = s_stage[warp];                    // sphere centres, then the links' bounding spheres
  float* bounds = stage + 3 * kMaxDistinctSpheres;
  const bool has_grid = env.esdf.v != nullptr;
  const bool filter = R->two_stage && !has_grid;
  const float4* e_obb = senv + 2 * env.n_aabb;
  const float4* e_cyl = e_obb + 5 * env.n_obb;
  const float4* e_sph = e_cyl + 2 * env.n_cyl;
  uint32_t passes = 0, pairs = 0, fine[4] = {0, 0, 0, 0};
  float sl = 0.f, cl = 1.f;
  if (lane < dof && revolute(R->jtype[lane])) joint_sincos<false>(ql, sl, cl);
  Frame T;
  for (int i = 0; i < dof; ++i) {
    const float qi = __shfl_sync(kFull, ql, i), si = __shfl_sync(kFull, sl, i), ci = __shfl_sync(kFull, cl, i);
    fk_joint(R, i, qi, [si, ci](float& sn, float& cs) { sn = si, cs = ci; }, T);
    const int s0 = R->sph_begin[i], cnt = R->sph_begin[i + 1] - s0;
    for (int k = lane; k <= cnt; k += 32) {  // one more: the link's bounding sphere, or its only one
      const float3 c = T.at(k < cnt ? R->sph[s0 + k] : R->grp[i]);
      float* st = k < cnt ? stage + 3 * (s0 + k) : bounds + 3 * i;
      st[0] = c.x;
      st[1] = c.y;
      st[2] = c.z;
    }
  }
  __syncwarp();
  bool hit = false;
  for (int i = dof - 1; i >= 0 && env_f4; --i) {
    const int s0 = R->sph_begin[i], cnt = R->sph_begin[i + 1] - s0;
    if (!cnt) continue;
    const float3 b = make_float3(bounds[3 * i], bounds[3 * i + 1], bounds[3 * i + 2]);
    const float br = R->grp[i].w;
    const float* st = stage + 3 * s0;
    passes += filter ? 1u : (uint32_t)cnt;
    hit |= warp_link_stage<kAabb>(senv, env.n_aabb, b, br, filter, st, R->sph + s0, cnt, lane, fine[kAabb]);
    hit |= warp_link_stage<kObb>(e_obb, env.n_obb, b, br, filter, st, R->sph + s0, cnt, lane, fine[kObb]);
    hit |= warp_link_stage<kCyl>(e_cyl, env.n_cyl, b, br, filter, st, R->sph + s0, cnt, lane, fine[kCyl]);
    hit |= warp_link_stage<kSph>(e_sph, env.n_sph, b, br, filter, st, R->sph + s0, cnt, lane, fine[kSph]);
    if (__any_sync(kFull, hit)) break;
  }
  if (has_grid) {
    for (int s = lane; s < R->n_spheres; s += 32)
      hit |= esdf_read(env.esdf, stage[3 * s], stage[3 * s + 1], stage[3 * s + 2]) < R->sph[s].w;
    passes += (uint32_t)R->n_spheres;
  }
  if (!__any_sync(kFull, hit)) {
    for (int k = lane; k < n_pairs; k += 32) {
      const uint32_t pr = pair[k];
      const float* si = stage + 3 * (pr & 0xffffu);
      const float* sj = stage + 3 * (pr >> 16);
      const float dx = si[0] - sj[0], dy = si[1] - sj[1], dz = si[2] - sj[2];
      hit |= fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < thr[k];
    }
    pairs += (uint32_t)n_pairs;
  }
  hit = __any_sync(kFull, hit);
  if (lane == 0) valid[idx] = hit ? 0 : 1;
  if (spheres) {
    float4* out = reinterpret_cast<float4*>(spheres) + (size_t)idx * n_raw;
    for (int r = lane; r < n_raw; r += 32) {
      const int ds = robot->raw_to_distinct[r];
      out[r] = make_float4(stage[3 * ds], stage[3 * ds + 1], stage[3 * ds + 2], R->sph[ds].w);
    }
  }
  if (lane != 0) return;
  if (slots) {
    slots[2 * idx] = make_uint4(passes, pairs, fine[0], fine[1]);
    slots[2 * idx + 1] = make_uint4(fine[2], fine[3], 0u, 0u);
  } else if (counters) {
    atomicAdd(counters + 0, (unsigned long long)passes);
    atomicAdd(counters + 1, (unsigned long long)pairs);
    atomicAdd(counters + 2, 1ull);
    for (int k = 0; k < 4; ++k) atomicAdd(counters + 3 + k, (unsigned long long)fine[k]);
  }
}


// Shared memory of a block of `warps` warps.
struct CheckShape {
  int table_bytes;  // robot and environment
  int warp_floats;  // joint values or queues, sphere and bounding-sphere centres of 32 states
  int q_floats;     // the first part of them
  int np_pad;
  int bounds;       // links with a bounding sphere
  int smem(int warps) const { return table_bytes + warps * warp_floats * (int)sizeof(float); }
};

CheckShape check_shape(const RobotHeader& h, const EnvView& env) {
  CheckShape s;
  s.np_pad = (h.n_pairs + 3) & ~3;
  s.bounds = 0;
  for (int f = 0; f < h.dof; ++f) s.bounds += h.coarse[f].w > 0.f ? 1 : 0;
  s.table_bytes = (int)sizeof(RobotHeader) + 8 * s.np_pad + (env.n_float4() + kEnvBox) * 16;
  s.q_floats = std::max(h.dof * 32, (int)sizeof(CheckQueues) / 4);
  s.warp_floats = s.q_floats + (h.n_spheres + s.bounds) * 96;
  return s;
}

}  // namespace

// One Philox4x32-10 block per thread (the sampler's generator).
__global__ void philox_kernel(const uint4* __restrict__ ctr, int n, uint2 key, uint4* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = philox4x32_10(ctr[i], key);
}

cudaError_t launch_philox(const uint32_t* ctr, int n, uint64_t key, uint32_t* out, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int blocks = (int)std::min<long long>(((long long)n + 255) / 256, 152LL * 16);
  philox_kernel<<<blocks, 256, 0, stream>>>(reinterpret_cast<const uint4*>(ctr), n,
                                            make_uint2((uint32_t)(key & 0xffffffffu), (uint32_t)(key >> 32)),
                                            reinterpret_cast<uint4*>(out));
  return cudaGetLastError();
}

// The FP32 pipe at full rate: kChains independent FMA chains per thread, so
// that every warp scheduler always has an FMA ready.  One FMA counts one
// lane-op, the unit of the planner's ALU roofline.  The sum is stored only
// when it equals a value it never takes, which keeps the chains alive.
constexpr int kFmaChains = 8;
__global__ void fma_loop_kernel(int iters, float m, float* __restrict__ sink) {
  float a[kFmaChains];
#pragma unroll
  for (int k = 0; k < kFmaChains; ++k) a[k] = (float)(threadIdx.x + k) * 1e-3f;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int k = 0; k < kFmaChains; ++k) a[k] = fmaf(a[k], m, 1e-7f);
  }
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < kFmaChains; ++k) s += a[k];
  if (s == -1.f) sink[blockIdx.x] = s;
}

cudaError_t launch_fma_loop(int sm_count, int iters, float* sink, cudaStream_t stream, long long* lane_ops) {
  const int blocks = sm_count * 8, threads = 256;  // 64 warps per SM
  fma_loop_kernel<<<blocks, threads, 0, stream>>>(iters, 0.9999999f, sink);
  *lane_ops = (long long)blocks * threads * iters * kFmaChains;
  return cudaGetLastError();
}

// Warps per block and resident blocks of the check kernel on the current
// device for a robot and environment of these sizes, cached: the attribute,
// the device query and the occupancy queries took longer on the host than a
// small call takes on the device.
struct CheckWave {
  int warps, blocks;
};

static cudaError_t check_wave(const CheckShape& shape, bool two_stage, CheckWave* wave) {
  static std::mutex mu;
  static std::map<std::array<int, 4>, CheckWave> cache;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  const std::array<int, 4> key{dev, shape.table_bytes, shape.warp_floats, two_stage ? 1 : 0};
  const auto it = cache.find(key);
  if (it != cache.end()) {
    *wave = it->second;
    return cudaSuccess;
  }
  constexpr int kMost = 227 * 1024 - 8192;  // less the static arrays
  auto* fn = two_stage ? check_states_kernel<true> : check_states_kernel<false>;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
  int sms = 0;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // the block size that keeps the most warps on an SM; on a tie the smaller one
  CheckWave best{0, 0};
  for (int w = 1; w <= kMaxCheckWarps && shape.smem(w) <= kMost; ++w) {
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, w * 32, shape.smem(w));
    if (e != cudaSuccess) return e;
    if (w * per_sm > best.warps * best.blocks) best = CheckWave{w, per_sm};
  }
  if (best.warps < 1) return cudaErrorInvalidConfiguration;
  best.blocks *= sms;
  cache.emplace(key, best);
  *wave = best;
  return cudaSuccess;
}

// States up to which a warp each is faster than a lane each.  Either way at the
// line (us, 6000 states a warp each / 6100 a lane each): 7-DoF arm in a shelf
// 17.8 / 17.6, among eight boxes 15.6 / 14.9, among 600 obstacles 33 / 70; both
// arms in a shelf 30.5 / 34.0.  64 states a warp each take 10, 10, 17 and 14.5.
constexpr int kWarpPerState = 6000;

static cudaError_t state_warps_attribute() {
  static std::mutex mu;
  static bool set[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) return e;
  std::lock_guard<std::mutex> lk(mu);
  if (set[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(check_state_warps_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  set[dev] = e == cudaSuccess;
  return e;
}

cudaError_t launch_check_states(const RobotDev* robot, const RobotHeader& h, EnvView env, const float* q, int n,
                                uint8_t* valid, float* spheres, unsigned long long* counters, uint4* slots, int* error,
                                cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const CheckShape shape = check_shape(h, env);
  if (n <= kWarpPerState || slots) {
    const cudaError_t e = state_warps_attribute();
    if (e != cudaSuccess) return e;
    check_state_warps_kernel<<<(n - 1) / kStateWarps + 1, kStateWarps * 32, shape.table_bytes, stream>>>(
        robot, env, q, n, valid, spheres, counters, slots, error, shape.np_pad, h.dof);
    return cudaGetLastError();
  }
  CheckWave wave{};
  const bool two_stage = h.two_stage && shape.bounds > 0 && env.n_float4() > 0 && !env.esdf.v;
  const cudaError_t e = check_wave(shape, two_stage, &wave);
  if (e != cudaSuccess) return e;
  // a call below one wave spreads over the SMs, in blocks of as many warps as
  // that leaves (the same number in each quarter of an SM: 20,000 states of the
  // 7-DoF arm among eight boxes 16.5 -> 15.6 us)
  const int need = (n - 1) / 32 + 1;
  int warps = wave.warps;
  if (need < wave.warps * wave.blocks) {
    warps = (need - 1) / wave.blocks + 1;
    if (warps > 2) warps = std::min(wave.warps, (warps + 3) & ~3);
  }
  const int grid = std::min((need - 1) / warps + 1, wave.blocks);
  auto* fn = two_stage ? check_states_kernel<true> : check_states_kernel<false>;
  fn<<<grid, warps * 32, shape.smem(warps), stream>>>(robot, env, q, n, valid, spheres, counters, error, shape.np_pad,
                                                      shape.warp_floats, shape.q_floats);
  return cudaGetLastError();
}

}  // namespace prrtc
