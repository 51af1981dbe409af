// prrtc_gemm.cu -- BF16 GEMM on the 5th-generation tensor cores for the
// learned sampling proposal's dense layers:  C[M,N] = A[M,K] * B[N,K]^T with
// FP32 accumulation in tensor memory, optional bias + ReLU and FP32 / BF16
// outputs.
//
// Three kernels.  Products below one wave of tiles (every layer of the proposal
// up to a few thousand rows): gemm_cluster_kernel, K split over the blocks of a
// cluster, which add up their partial tiles through shared memory.  Larger ones:
// gemm_bf16_kernel, persistent, one CTA per SM or pair of CTAs per two SMs.  A
// work unit is one output tile of 128 x 256 (a pair: 256 x 256) over a range of
// K (a requested split that the clusters do not take: partial tiles go to a
// workspace and splitk_reduce_kernel adds them up in split order):
//   warp 0    -- one lane issues TMA loads of the 128 x 64 A and 256 x 64 B
//                tiles (a pair: each CTA its rows of A and half of B; 128-byte
//                swizzle) into a ring of 4 (6) stages;
//   warp 1    -- allocates all 512 TMEM columns (two 256-column
//                accumulators); one lane (a pair: of the first CTA) issues
//                tcgen05.mma (M=128 or 256, N=256, K=16, kind::f16) four times
//                per stage, commits each stage back to the producer and each
//                finished unit to the epilogue;
//   warps 2-5 -- read an accumulator with tcgen05.ld (each warp owns one
//                32-lane quarter of TMEM), run the epilogue, and hand the
//                accumulator back, so the epilogue of one unit overlaps the
//                main loop of the next.
// The epilogue stages each 32 x 32 chunk in a swizzled shared-memory tile and
// writes it with a TMA bulk tensor store (the TMA engine clips the matrix
// edges).
// Every mbarrier wait is bounded; a wait that gives up records an error, the
// roles stop, and the CTA still frees its tensor memory.
//
// What bounds the large products: 8192^3 (FP32 output, normal operands) took 714
// us with every lane of a warp at each wait, 669 with one lane running the MMA
// loop, 652 with one lane for the loads as well, and 580 (1.9 PFLOP/s) with that
// lane chosen by elect.sync, after which the compiler needs no loop over lanes
// around each instruction that takes uniform registers.  With operands of zeros
// it takes 490, the MMAs' time: the rest is the power limit.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <map>
#include <mutex>

#include "prrtc.h"
#include "prrtc_launch.h"

namespace prrtc {
namespace {

constexpr int BM = 128, BN = 256, BK = 64;
constexpr int A_BYTES = BM * BK * 2;
constexpr int EPI_TILE_BYTES = 32 * 128;   // one 32 x 32 FP32 chunk (or 32 x 32 BF16 in its first half)
constexpr int EPI_BUFS = 2;                 // staging tiles per epilogue warp (double buffered)
// One CTA per tile of 128 x 256, or a pair of CTAs per tile of 256 x 256: each
// holds its 128 rows of A and of the output, and its half of the tile's B.
template <int kCtas>
struct Tile {
  static constexpr int kM = BM * kCtas;             // rows of a tile
  static constexpr int kBRows = BN / kCtas;         // columns of the output whose B a CTA loads
  static constexpr int kStageBytes = A_BYTES + kBRows * BK * 2;
  static constexpr int kStages = kCtas == 2 ? 6 : 4;
  // ring | barriers (1 KB) | staging tiles, plus 1 KB for aligning the base
  static constexpr int kSmem = kStages * kStageBytes + 1024 + 1024 + 4 * EPI_BUFS * EPI_TILE_BYTES;
};
constexpr int THREADS = 192;
constexpr int EPI_WARPS = 4;
constexpr uint32_t TMEM_COLS = 2 * BN;  // two accumulators
constexpr uint32_t kPolls = 1u << 26;
constexpr int kMinKTilesPerSplit = 4;
constexpr int kMaxSplits = 16;

__device__ int g_gemm_error;

struct Epilogue {
  int M, N, K;
  const float* bias;
  int relu;
  int has_c32, has_c16;  // outputs written through the c32 / c16 tensor maps
  int splits;            // > 1: raw partials through the workspace map, rows split * m_pad + row
  int m_tiles, n_tiles, k_tiles;
  int m_pad;             // rows of one split's partial (M rounded up to the tile), so that the
                         // clipped-off rows of an edge tile never reach the next split's rows
};

// Output tensor maps of one launch: workspace (FP32, rows = splits * m_pad),
// FP32 output and BF16 output; boxes of 32 x 32 elements, 128- / 64-byte
// swizzle matching the staging layout below.
struct OutMaps {
  CUtensorMap ws, c32, c16;
};

// Shared-memory matrix descriptor of a K-major tile with 128-byte swizzle:
// start address, stride between 8-row groups (1024 B), descriptor version 1,
// swizzle mode 2 (128 B).
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;                 // leading byte offset (unused with 128 B swizzle, K-major)
  d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset
  d |= (uint64_t)1 << 46;                 // version
  d |= (uint64_t)2 << 61;                 // 128 B swizzle
  return d;
}

// The same for an MN-major tile (a transposed operand): 64 rows or columns of
// the operand are the 128 contiguous bytes, K runs over the tile's lines.
// Leading byte offset: from one group of 64 to the next (a box of BK lines);
// stride byte offset: from 8 lines of K to the next 8.
constexpr int MN_BOX_BYTES = BK * 128;
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(MN_BOX_BYTES >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B, K-major
// unless the transpose bits (15: A, 16: B) say MN-major, N >> 3 at bit 17,
// M >> 4 at bit 24.
__device__ __forceinline__ uint32_t idesc_bf16(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity) {
  if (mbar_wait(bar, parity, kPolls)) return true;
  atomicExch(&g_gemm_error, PRRTC_ERR_TIMEOUT);
  return false;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::
          "r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

// A load of one CTA of a pair that completes on the pair's first CTA's barrier
// (`bar`: its address in the cluster's shared memory).
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* tm, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], "
      "[%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar), "r"(x), "r"(y)
      : "memory");
}

// Address in the cluster's shared memory of block 0's copy of `p`.
__device__ __forceinline__ uint32_t of_first_block(const void* p) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
  return r;
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

template <int kCtas = 1>
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if (kCtas == 2) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
    return;
  }
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// Arrival on `bar` (a pair: in both CTAs) once the MMAs issued so far are done.
template <int kCtas = 1>
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  if (kCtas == 2) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
    return;
  }
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// True in one lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.b32 %0, 1, 0, p;\n}\n" : "=r"(r));
  return r != 0;
}

// Work unit -> tile and K range.  Tiles go in groups of kGroupRows rows:
// m fastest inside a group, then n, then the next group, so that the tiles in
// flight at once (one per SM) share a slab of A rows and a few B columns that
// stay in L2 instead of sweeping all of A for every column of B.
constexpr int kGroupRows = 16 * BM;
struct Unit {
  int m0, n0, split, kt0, kt1;
};

template <int kCtas>
__device__ __forceinline__ Unit unit_of(const Epilogue& ep, int u) {
  constexpr int kM = Tile<kCtas>::kM, kGroupM = kGroupRows / kM;
  Unit w;
  const int tile = u / ep.splits;
  w.split = u - tile * ep.splits;
  const int span = kGroupM * ep.n_tiles;
  const int first_m = (tile / span) * kGroupM;
  const int gm = min(ep.m_tiles - first_m, kGroupM);
  const int in = tile - (tile / span) * span;
  w.m0 = (first_m + in % gm) * kM;
  w.n0 = (in / gm) * BN;
  const int base = ep.k_tiles / ep.splits, rem = ep.k_tiles % ep.splits;
  w.kt0 = w.split * base + min(w.split, rem);
  w.kt1 = w.kt0 + base + (w.split < rem ? 1 : 0);
  return w;
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* tm, const void* src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(tm)),
               "r"(smem_u32(src)), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Wait until at most one committed bulk store still reads shared memory.
__device__ __forceinline__ void bulk_wait_read_le1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Stage one 32 x 32 chunk held one row per lane (lane = row, values v[0..31]
// = columns) into a shared-memory tile laid out as the TMA engine expects
// with the store map's swizzle, then let lane 0 store it with one bulk
// tensor copy.  FP32 rows are 128 bytes (128-byte swizzle: 16-byte unit u of
// row r sits at unit u ^ (r % 8)); BF16 rows are 64 bytes (64-byte swizzle:
// unit u ^ ((r / 2) % 4)).  Each store instruction of the warp touches every
// bank group once, and the TMA engine clips rows and columns outside the
// matrix.  `buf` alternates between the warp's two staging tiles.
__device__ __forceinline__ void stage_and_store(const CUtensorMap* map, unsigned char* tiles, int& buf, bool bf16,
                                                int x, int y, int lane, const float (&f)[32]) {
  unsigned char* tile = tiles + buf * EPI_TILE_BYTES;
  if (lane == 0) bulk_wait_read_le1();  // the store issued from this tile two rounds ago has read it
  __syncwarp();
  if (!bf16) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      float4* dst = reinterpret_cast<float4*>(tile + lane * 128 + ((u ^ (lane & 7)) << 4));
      *dst = make_float4(f[4 * u], f[4 * u + 1], f[4 * u + 2], f[4 * u + 3]);
    }
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      uint4 pk;
      __nv_bfloat162 h0 = __floats2bfloat162_rn(f[8 * u], f[8 * u + 1]);
      __nv_bfloat162 h1 = __floats2bfloat162_rn(f[8 * u + 2], f[8 * u + 3]);
      __nv_bfloat162 h2 = __floats2bfloat162_rn(f[8 * u + 4], f[8 * u + 5]);
      __nv_bfloat162 h3 = __floats2bfloat162_rn(f[8 * u + 6], f[8 * u + 7]);
      pk.x = *reinterpret_cast<uint32_t*>(&h0);
      pk.y = *reinterpret_cast<uint32_t*>(&h1);
      pk.z = *reinterpret_cast<uint32_t*>(&h2);
      pk.w = *reinterpret_cast<uint32_t*>(&h3);
      *reinterpret_cast<uint4*>(tile + lane * 64 + ((u ^ ((lane >> 1) & 3)) << 4)) = pk;
    }
  }
  fence_proxy_async_smem();  // make the generic-proxy writes visible to the TMA engine
  __syncwarp();
  if (lane == 0) {
    tma_store_2d(map, tile, x, y);
    bulk_commit();
  }
  buf ^= 1;
}

// Epilogue of one 32 x 32 chunk (rows row0.., columns col0..; lane = row).
__device__ __forceinline__ void store_chunk(const Epilogue& ep, const OutMaps& om, unsigned char* tiles, int& buf,
                                            int split, int row0, int col0, int lane, const uint32_t (&v)[32]) {
  float f[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) f[j] = __uint_as_float(v[j]);
  if (ep.splits > 1) {  // raw partial; the reduction kernel finishes it
    stage_and_store(&om.ws, tiles, buf, false, col0, split * ep.m_pad + row0, lane, f);
    return;
  }
  if (ep.bias) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (col0 + j < ep.N) f[j] += ep.bias[col0 + j];
  }
  if (ep.relu) {
#pragma unroll
    for (int j = 0; j < 32; ++j) f[j] = fmaxf(f[j], 0.f);
  }
  if (ep.has_c32) stage_and_store(&om.c32, tiles, buf, false, col0, row0, lane, f);
  if (ep.has_c16) stage_and_store(&om.c16, tiles, buf, true, col0, row0, lane, f);
}

// kTA, kTB: operand stored transposed.  kCtas = 2: the two blocks of a cluster
// share a tile; the first one's barriers and MMA warp drive both.
template <bool kTA, bool kTB, int kCtas>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_bf16_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const __grid_constant__ OutMaps om, Epilogue ep) {
  using T = Tile<kCtas>;
  constexpr int STAGES = T::kStages, STAGE_BYTES = T::kStageBytes;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* acc_full = empty + STAGES;   // [2] MMA -> epilogue
  uint64_t* acc_empty = acc_full + 2;    // [2] epilogue -> MMA
  uint64_t* roles_done = acc_empty + 2;  // every warp of the CTA -> TMEM release
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(roles_done + 1);
  unsigned char* epi_tiles = smem + STAGES * STAGE_BYTES + 256 + 768;  // 1024-aligned staging tiles
  __shared__ int s_abort;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_units = ep.m_tiles * ep.n_tiles * ep.splits;
  const int rank = kCtas == 2 ? (int)blockIdx.x & 1 : 0;  // place in the pair
  const int first = (int)blockIdx.x / kCtas, step = (int)gridDim.x / kCtas;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], kCtas * EPI_WARPS);
    }
    mbar_init(roles_done, THREADS / 32);
    s_abort = 0;
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
  }
  if (warp == 1) {
    if (kCtas == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  fence_before();
  __syncthreads();
  if (kCtas == 2) cluster_sync_all();  // the other block's barriers and tensor memory are set up
  fence_after();
  const uint32_t tmem = *tmem_slot;
  volatile int* abort_flag = &s_abort;

  // One elected lane runs the whole loop of the loads and of the MMAs: what a
  // warp does between two stages has to fit into the stage's MMAs (512 cycles).
  if (warp == 0) {
    if (elect_one()) {
      int s = 0, issued = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int u = first; u < n_units && ok; u += step) {
        const Unit w = unit_of<kCtas>(ep, u);
        const int m = w.m0 + rank * BM, n = w.n0 + rank * T::kBRows;
        for (int kt = w.kt0; kt < w.kt1; ++kt) {
          ok = !*abort_flag && wait_bar(&empty[s], ph ^ 1u);
          if (!ok) break;
          unsigned char* a = smem + s * STAGE_BYTES;
          if (rank == 0) mbar_arrive_expect_tx(&full[s], kCtas * STAGE_BYTES);
          const uint32_t pair_bar = kCtas == 2 ? of_first_block(&full[s]) : 0u;
          auto load = [&](unsigned char* dst, const CUtensorMap* tm, int x, int y) {
            if (kCtas == 2)
              tma_load_2d_pair(dst, tm, pair_bar, x, y);
            else
              tma_load_2d(dst, tm, &full[s], x, y);
          };
          if (kTA) {
#pragma unroll
            for (int j = 0; j < BM / 64; ++j) load(a + j * MN_BOX_BYTES, &tmA, m + 64 * j, kt * BK);
          } else {
            load(a, &tmA, kt * BK, m);
          }
          if (kTB) {
#pragma unroll
            for (int j = 0; j < T::kBRows / 64; ++j) load(a + A_BYTES + j * MN_BOX_BYTES, &tmB, n + 64 * j, kt * BK);
          } else {
            load(a + A_BYTES, &tmB, kt * BK, n);
          }
          issued = min(issued + 1, STAGES);
          if (++s == STAGES) s = 0, ph ^= 1u;
        }
      }
      if (!ok) {
        *abort_flag = 1;
        // the loads in flight land before the block ends
        for (; rank == 0 && issued > 0; --issued) {
          if (--s < 0) s = STAGES - 1, ph ^= 1u;
          wait_bar(&full[s], ph);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t idesc = idesc_bf16(T::kM, BN) | (kTA ? 1u << 15 : 0u) | (kTB ? 1u << 16 : 0u);
    // from one K step of 16 to the next: 32 bytes along K, or 16 lines of K
    constexpr uint32_t step_a = kTA ? 2048u : 32u, step_b = kTB ? 2048u : 32u;
    if (rank == 0 && elect_one()) {
      int s = 0, i = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int u = first; u < n_units && ok; u += step, ++i) {
        const Unit w = unit_of<kCtas>(ep, u);
        const int acc = i & 1;
        // wait until the epilogue has drained this accumulator (first use passes)
        ok = !*abort_flag && wait_bar(&acc_empty[acc], ((uint32_t)(i >> 1) & 1u) ^ 1u);
        if (!ok) break;
        fence_after();
        const uint32_t d = tmem + (uint32_t)(acc * BN);
        for (int kt = w.kt0; kt < w.kt1; ++kt) {
          ok = wait_bar(&full[s], ph);
          if (!ok) break;
          fence_after();
          const uint32_t a = smem_u32(smem + s * STAGE_BYTES);
          const uint32_t b = a + A_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            mma_bf16<kCtas>(d, kTA ? smem_desc_mn(a + step_a * k) : smem_desc(a + step_a * k),
                            kTB ? smem_desc_mn(b + step_b * k) : smem_desc(b + step_b * k), idesc,
                            (kt > w.kt0 || k > 0) ? 1u : 0u);
          mma_commit<kCtas>(&empty[s]);
          if (++s == STAGES) s = 0, ph ^= 1u;
        }
        if (ok) mma_commit<kCtas>(&acc_full[acc]);
      }
      if (!ok) *abort_flag = 1;
    }
    __syncwarp();
  } else {
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    unsigned char* tiles = epi_tiles + (warp - 2) * EPI_BUFS * EPI_TILE_BYTES;
    int buf = 0;
    int i = 0;
    for (int u = first; u < n_units; u += step, ++i) {
      const Unit w = unit_of<kCtas>(ep, u);
      const int acc = i & 1;
      int ok = 0;
      if (lane == 0) ok = wait_bar(&acc_full[acc], (uint32_t)(i >> 1) & 1u) ? 1 : 0;
      ok = __shfl_sync(kFull, ok, 0);
      if (!ok) {
        if (lane == 0) *abort_flag = 1;
        break;
      }
      fence_after();
      const int row0 = w.m0 + rank * BM + 32 * q;
      for (int c = 0; c < BN; c += 32) {
        uint32_t v[32];
        __syncwarp();
        tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * BN + c), v);
        const int col0 = w.n0 + c;
        if (row0 < ep.M && col0 < ep.N) store_chunk(ep, om, tiles, buf, w.split, row0, col0, lane, v);
      }
      fence_before();
      __syncwarp();
      if (lane == 0) {
        if (kCtas == 2)
          mbar_arrive_cluster(of_first_block(&acc_empty[acc]));
        else
          mbar_arrive(&acc_empty[acc]);
      }
    }
    if (lane == 0) bulk_wait_all();  // every bulk store of this warp has landed
    __syncwarp();
  }
  // Join: each warp signals that its role is over (its tensor-memory reads
  // have completed); the allocating warp frees tensor memory only after all
  // of them.  If the join times out the memory is still freed: the kernel is
  // ending and the error word is set.
  __syncwarp();
  fence_before();
  if (lane == 0) mbar_arrive(roles_done);
  if (warp == 1) {
    int joined = 0;
    if (lane == 0) joined = wait_bar(roles_done, 0) ? 1 : 0;
    joined = __shfl_sync(kFull, joined, 0);
    (void)joined;
    fence_after();
  }
  // A pair also ends together: the other block's barriers, shared and tensor
  // memory are in use until both are through.
  __syncwarp();
  if (kCtas == 2) cluster_sync_all();
  if (warp == 1) {
    if (kCtas == 2)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// Sum of the split-K partials (split s at rows s * m_pad ..) in split order,
// then bias, ReLU and outputs; four columns per thread (N is a multiple of 8).
__global__ void splitk_reduce_kernel(const float* __restrict__ ws, int splits, int M, int m_pad, int N,
                                     const float* __restrict__ bias, int relu, float* __restrict__ c32, int ldc32,
                                     __nv_bfloat16* __restrict__ c16, int ldc16) {
  const int n4 = N >> 2;
  const size_t total = (size_t)M * n4;
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
    const int row = (int)(t / n4), col = (int)(t % n4) * 4;
    float4 acc = *reinterpret_cast<const float4*>(ws + (size_t)row * N + col);
    for (int s = 1; s < splits; ++s) {
      const float4 p = *reinterpret_cast<const float4*>(ws + ((size_t)s * m_pad + row) * N + col);
      acc.x += p.x;
      acc.y += p.y;
      acc.z += p.z;
      acc.w += p.w;
    }
    if (bias) {
      acc.x += bias[col];
      acc.y += bias[col + 1];
      acc.z += bias[col + 2];
      acc.w += bias[col + 3];
    }
    if (relu) {
      acc.x = fmaxf(acc.x, 0.f);
      acc.y = fmaxf(acc.y, 0.f);
      acc.z = fmaxf(acc.z, 0.f);
      acc.w = fmaxf(acc.w, 0.f);
    }
    if (c32) *reinterpret_cast<float4*>(c32 + (size_t)row * ldc32 + col) = acc;
    if (c16) {
      __nv_bfloat162 h0 = __floats2bfloat162_rn(acc.x, acc.y), h1 = __floats2bfloat162_rn(acc.z, acc.w);
      uint2 pk;
      pk.x = *reinterpret_cast<uint32_t*>(&h0);
      pk.y = *reinterpret_cast<uint32_t*>(&h1);
      *reinterpret_cast<uint2*>(c16 + (size_t)row * ldc16 + col) = pk;
    }
  }
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// ------------------------------------------------------------ GEMMs below one wave
// The layers' products at training and inference batches fill less than one
// wave of 128 x 256 tiles even with K split, and are bound by what happens
// once per launch: the first loads, the tile's way out, the partials' round
// trip through memory and a second kernel.  Here a cluster of `splits` blocks
// owns one 128 x kBN output tile (kBN 64 or 128) and each block one range of
// K, the same ranges as above.  The blocks leave their FP32 partial tiles in
// shared memory; after a cluster barrier, block r adds up rows
// [128 r / splits, 128 (r + 1) / splits) over all blocks in split order (the
// sums of the second kernel, bit for bit) and writes the outputs.
//
// Launches in a row, bias, ReLU and BF16 output, in us: where the next one may
// start early (the proposal's) / where not (a caller's) (128 x 256 tiles and
// second kernel before): 512 x 512 x 1024 4.5 / 5.3 (9.6), 512 x 512 x 512 4.1 /
// 4.9 (9.2), 1024 x 4160 x 512 8.3 / 8.6 (15.5), 2048 x 1024 x 4160 17.6 / 18.7
// (23.5), 512 x 1024 x 4160 11.2 / 12.6 (12.5: there the eight partial tiles'
// exchange costs what the second kernel did).  About 1 us goes to the launch, 0.9
// to tensor memory and the first loads, 0.3 to each K tile, 1 to the cluster
// barriers.
//
// Roles as above: warp 0 loads, warp 1 issues the MMAs, warps 2-5 read the
// accumulator; all six add up.  The partial tile takes the ring's place: every
// load has landed and every MMA has read it by then.  Waits are bounded; a
// role that gives up records the error, and every thread still meets every
// barrier.
template <int kBN>
struct ClusterTile {
  static constexpr int kStages = kBN == 64 ? 4 : 3;  // two blocks per SM
  static constexpr int kBBytes = kBN * BK * 2;
  static constexpr int kStageBytes = A_BYTES + kBBytes;
  static constexpr int kSmem = kStages * kStageBytes + 1024 + 256;
  static_assert(BM * kBN * 4 <= kStages * kStageBytes, "the partial tile fits the ring");
};
constexpr int kMaxClusterSplits = 8;  // portable cluster size
constexpr int kClusterThreads = 256;

struct ClusterEpilogue {
  int M, N, k_tiles, m_tiles;
  const float* bias;
  int relu;
  const __nv_bfloat16* mask;  // nullable [M x N] of row stride ldm: outputs where mask <= 0 become 0
  int ldm;
  float* c32;
  int ldc32;
  __nv_bfloat16* c16;
  int ldc16;
};

// Up to four products of one launch (a layer's weight gradients, which wait
// for nothing but their operands): product g has the blocks from first[g] on.
constexpr int kMaxGroup = 4;
struct ClusterGroup {
  CUtensorMap a[kMaxGroup], b[kMaxGroup];
  ClusterEpilogue ep[kMaxGroup];
  int first[kMaxGroup];
  int n;
  // The operands are older than the launch before, which let this one start only
  // after its own wait: this launch waits for it at the end.  The weight
  // gradients run beside the bias gradients and each other so (a training step
  // 109 -> 106 us).
  int late;
  // The launch after this one may start before the outputs are written: only
  // where that one is known to wait for this (kNextMayStart).
  int early;
};

// Byte offset of 16-byte unit u of row i of a partial tile (rows of kBN
// floats): units of a 128-byte group are exchanged by the row, so that both
// the row-per-lane writes and the unit-per-thread reads touch every bank once.
template <int kBN>
__device__ __forceinline__ uint32_t part_off(int i, int u) {
  return (uint32_t)i * (kBN * 4) + (uint32_t)((u & ~7) | ((u ^ i) & 7)) * 16u;
}

template <int kBN, int kSplits, bool kTA, bool kTB>
__global__ void __launch_bounds__(kClusterThreads, 2)
    gemm_cluster_kernel(const __grid_constant__ ClusterGroup group) {
  using T = ClusterTile<kBN>;
  int which = 0;
  while (which + 1 < group.n && (int)blockIdx.x >= group.first[which + 1]) ++which;
  const ClusterEpilogue ep = group.ep[which];
  const CUtensorMap& tmA = group.a[which];
  const CUtensorMap& tmB = group.b[which];
  const int block = (int)blockIdx.x - group.first[which];
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + T::kStages * T::kStageBytes);
  uint64_t* empty = full + T::kStages;
  uint64_t* acc_full = empty + T::kStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = block % kSplits, tile = block / kSplits;
  const int m0 = tile % ep.m_tiles * BM, n0 = tile / ep.m_tiles * kBN;
  const int base = ep.k_tiles / kSplits, rem = ep.k_tiles % kSplits;
  const int kt0 = split * base + min(split, rem), kts = base + (split < rem ? 1 : 0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < T::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_full, 1);
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)kBN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  if (!group.late) wait_before();

  if (warp == 0) {
    if (elect_one()) {
      int it = 0;
      for (; it < kts; ++it) {
        const int s = it % T::kStages;
        if (!wait_bar(&empty[s], ((uint32_t)(it / T::kStages) & 1u) ^ 1u)) break;
        unsigned char* a = smem + s * T::kStageBytes;
        const int kt = kt0 + it;
        mbar_arrive_expect_tx(&full[s], T::kStageBytes);
        if (kTA) {
#pragma unroll
          for (int j = 0; j < BM / 64; ++j)
            tma_load_2d(a + j * MN_BOX_BYTES, &tmA, &full[s], m0 + 64 * j, kt * BK);
        } else {
          tma_load_2d(a, &tmA, &full[s], kt * BK, m0);
        }
        if (kTB) {
#pragma unroll
          for (int j = 0; j < kBN / 64; ++j)
            tma_load_2d(a + A_BYTES + j * MN_BOX_BYTES, &tmB, &full[s], n0 + 64 * j, kt * BK);
        } else {
          tma_load_2d(a + A_BYTES, &tmB, &full[s], kt * BK, n0);
        }
      }
      // the loads have landed before the block can leave, also after a give-up
      for (int s = 0; s < T::kStages && s < it; ++s) wait_bar(&full[s], (uint32_t)((it - 1 - s) / T::kStages) & 1u);
    }
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t idesc = idesc_bf16(BM, kBN) | (kTA ? 1u << 15 : 0u) | (kTB ? 1u << 16 : 0u);
    constexpr uint32_t step_a = kTA ? 2048u : 32u, step_b = kTB ? 2048u : 32u;
    if (elect_one()) {
      bool ok = true;
      for (int it = 0; it < kts && ok; ++it) {
        const int s = it % T::kStages;
        ok = wait_bar(&full[s], (uint32_t)(it / T::kStages) & 1u);
        if (!ok) break;
        fence_after();
        const uint32_t a = smem_u32(smem + s * T::kStageBytes), b = a + A_BYTES;
#pragma unroll
        for (int k = 0; k < BK / 16; ++k)
          mma_bf16(tmem, kTA ? smem_desc_mn(a + step_a * k) : smem_desc(a + step_a * k),
                   kTB ? smem_desc_mn(b + step_b * k) : smem_desc(b + step_b * k), idesc,
                   (it > 0 || k > 0) ? 1u : 0u);
        mma_commit(&empty[s]);
      }
      mma_commit(acc_full);  // completes once every MMA issued so far has
    }
    __syncwarp();
  } else if (warp < 6) {
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    int ok = 0;
    if (lane == 0) ok = wait_bar(acc_full, 0u) ? 1 : 0;
    ok = __shfl_sync(kFull, ok, 0);
    if (ok) {
      fence_after();
      const int i = 32 * q + lane;
#pragma unroll
      for (int c = 0; c < kBN; c += 32) {
        uint32_t v[32];
        tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c, v);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          *reinterpret_cast<uint4*>(smem + part_off<kBN>(i, c / 4 + u)) =
              make_uint4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
      }
    }
    fence_before();
  }
  if (group.early) let_next_start();
  if (kSplits > 1)
    cluster_sync_all();
  else
    __syncthreads();
  fence_after();
  if (warp == 1)  // every read of the accumulator is done
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)kBN) : "memory");

  // This block's rows, 16 bytes a thread and turn; the loads of kAhead turns
  // and all blocks are in flight together (one by one this part took as long
  // as the whole product).
  constexpr int kUnits = kBN / 4, kRows = BM / kSplits, kTurns = kRows * kUnits / kClusterThreads;
  constexpr int kAhead = kTurns < 8 / kSplits ? kTurns : (8 / kSplits > 0 ? 8 / kSplits : 1);
  static_assert(kTurns * kClusterThreads == kRows * kUnits && kTurns % kAhead == 0, "whole turns");
  const int u = threadIdx.x % kUnits, col = n0 + 4 * u;
  float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
  if (ep.bias && col < ep.N)  // any alignment
    bias = make_float4(__ldg(ep.bias + col), __ldg(ep.bias + col + 1), __ldg(ep.bias + col + 2), __ldg(ep.bias + col + 3));
  for (int turn = 0; turn < kTurns; turn += kAhead) {
    float4 part[kAhead][kSplits];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int i = split * kRows + ((turn + j) * kClusterThreads + (int)threadIdx.x) / kUnits;
      const uint32_t off = smem_u32(smem) + part_off<kBN>(i, u);
#pragma unroll
      for (int s = 0; s < kSplits; ++s) {
        float4& p = part[j][s];
        if (kSplits == 1) {
          asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(p.x), "=f"(p.y), "=f"(p.z), "=f"(p.w) : "r"(off));
        } else {
          uint32_t remote;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(off), "r"(s));
          asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                       : "=f"(p.x), "=f"(p.y), "=f"(p.z), "=f"(p.w)
                       : "r"(remote));
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int i = split * kRows + ((turn + j) * kClusterThreads + (int)threadIdx.x) / kUnits;
      const int row = m0 + i;
      float4 acc = part[j][0];
#pragma unroll
      for (int s = 1; s < kSplits; ++s) {
        acc.x += part[j][s].x;
        acc.y += part[j][s].y;
        acc.z += part[j][s].z;
        acc.w += part[j][s].w;
      }
      if (row >= ep.M || col >= ep.N) continue;
      if (ep.bias) {
        acc.x += bias.x;
        acc.y += bias.y;
        acc.z += bias.z;
        acc.w += bias.w;
      }
      if (ep.relu) {
        acc.x = fmaxf(acc.x, 0.f);
        acc.y = fmaxf(acc.y, 0.f);
        acc.z = fmaxf(acc.z, 0.f);
        acc.w = fmaxf(acc.w, 0.f);
      }
      if (ep.mask) {
        const uint2 h = *reinterpret_cast<const uint2*>(ep.mask + (size_t)row * ep.ldm + col);
        const __nv_bfloat162 h0 = *reinterpret_cast<const __nv_bfloat162*>(&h.x);
        const __nv_bfloat162 h1 = *reinterpret_cast<const __nv_bfloat162*>(&h.y);
        acc.x = __low2float(h0) > 0.f ? acc.x : 0.f;
        acc.y = __high2float(h0) > 0.f ? acc.y : 0.f;
        acc.z = __low2float(h1) > 0.f ? acc.z : 0.f;
        acc.w = __high2float(h1) > 0.f ? acc.w : 0.f;
      }
      if (ep.c32) *reinterpret_cast<float4*>(ep.c32 + (size_t)row * ep.ldc32 + col) = acc;
      if (ep.c16)
        *reinterpret_cast<uint2*>(ep.c16 + (size_t)row * ep.ldc16 + col) =
            make_uint2(pack_bf16x2(acc.x, acc.y), pack_bf16x2(acc.z, acc.w));
    }
  }
  if (kSplits > 1) cluster_sync_all();  // the other blocks have read this one's partial tile
  if (group.late) wait_before();        // this launch ends after the one before it
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::mutex g_encode_mu;

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  std::lock_guard<std::mutex> lk(g_encode_mu);
  if (!g_encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  return g_encode;
}

// Row-major [rows x K] BF16 matrix with row stride ld elements, K
// contiguous; boxes of 64 x box_rows (for a transposed operand the rows are K).
bool make_tmap(CUtensorMap* tm, const void* ptr, int rows, int K, int ld, int box_rows) {
  auto enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Output matrix [rows x cols] with row stride ld elements (FP32 or BF16),
// boxes of 32 x 32 with the swizzle of the epilogue's staging tiles.
bool make_out_tmap(CUtensorMap* tm, const void* ptr, int rows, int cols, int ld, bool bf16) {
  auto enc = encoder();
  if (!enc) return false;
  const int es_bytes = bf16 ? 2 : 4;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * es_bytes};
  cuuint32_t box[2] = {32, 32};
  cuuint32_t es[2] = {1, 1};
  return enc(tm, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(ptr),
             dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
             bf16 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Encoded tensor maps by (device, address, rows, inner extent, row stride,
// kind, box rows): the MLP calls the same few layouts every step, and encoding
// costs host time.  kind 0: BF16 operand (boxes of 64 x box rows), 2: FP32
// output, 3: BF16 output.
struct MapKey {
  int dev;
  const void* ptr;
  int rows, cols, ld, kind, box;
  bool operator<(const MapKey& o) const {
    if (dev != o.dev) return dev < o.dev;
    if (ptr != o.ptr) return ptr < o.ptr;
    if (rows != o.rows) return rows < o.rows;
    if (cols != o.cols) return cols < o.cols;
    if (ld != o.ld) return ld < o.ld;
    if (kind != o.kind) return kind < o.kind;
    return box < o.box;
  }
};
std::mutex g_map_mu;
std::map<MapKey, CUtensorMap> g_maps;
constexpr size_t kMaxCachedMaps = 256;

bool cached_map(CUtensorMap* tm, const void* ptr, int rows, int cols, int ld, int kind, int box = 0) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  const MapKey key{dev, ptr, rows, cols, ld, kind, box};
  std::lock_guard<std::mutex> lk(g_map_mu);
  auto it = g_maps.find(key);
  if (it != g_maps.end()) {
    *tm = it->second;
    return true;
  }
  const bool ok = kind == 0 ? make_tmap(tm, ptr, rows, cols, ld, box) : make_out_tmap(tm, ptr, rows, cols, ld, kind == 3);
  if (!ok) return false;
  if (g_maps.size() >= kMaxCachedMaps) g_maps.clear();
  g_maps.emplace(key, *tm);
  return true;
}

// Split-K workspace per (device, stream), grown on demand.
struct Workspace {
  float* ptr = nullptr;
  size_t floats = 0;
};
std::mutex g_ws_mu;
std::map<std::pair<int, cudaStream_t>, Workspace> g_ws;
std::atomic<uint64_t> g_ws_epoch{0};  // bumped whenever a workspace is (re)allocated

float* workspace(size_t floats, cudaStream_t stream) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  std::lock_guard<std::mutex> lk(g_ws_mu);
  Workspace& w = g_ws[{dev, stream}];
  if (w.floats >= floats && w.ptr) return w.ptr;
  if (w.ptr) {
    if (cudaStreamSynchronize(stream) != cudaSuccess) return nullptr;  // earlier launches may still read it
    cudaFree(w.ptr);
    w.ptr = nullptr;
    w.floats = 0;
  }
  g_ws_epoch.fetch_add(1);
  if (cudaMalloc(&w.ptr, floats * sizeof(float)) != cudaSuccess) {
    cudaGetLastError();
    w.ptr = nullptr;
    return nullptr;
  }
  w.floats = floats;
  return w.ptr;
}

}  // namespace

namespace {

// Dynamic shared memory of a kernel on the current device, set once (`done`).
template <class Fn>
cudaError_t smem_attribute(std::atomic<uint64_t>& done, Fn* fn, int bytes) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  return once_per_device(
      done, dev, [&] { return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
}

template <int kBN, int kSplits, bool kTA, bool kTB>
int launch_cluster_as(const ClusterGroup& group, int grid, cudaStream_t stream) {
  using T = ClusterTile<kBN>;
  auto* fn = gemm_cluster_kernel<kBN, kSplits, kTA, kTB>;
  static std::atomic<uint64_t> attr{0};
  if (smem_attribute(attr, fn, T::kSmem) != cudaSuccess) return PRRTC_ERR_CUDA;
  return launch_overlapped(fn, grid, kClusterThreads, T::kSmem, stream, kSplits, group) == cudaSuccess
             ? PRRTC_OK
             : PRRTC_ERR_CUDA;
}

template <int kBN, int kSplits>
int launch_cluster_split(bool ta, bool tb, const ClusterGroup& group, int grid, cudaStream_t stream) {
  if (ta) return tb ? launch_cluster_as<kBN, kSplits, true, true>(group, grid, stream) : PRRTC_ERR_UNSUPPORTED;
  return tb ? launch_cluster_as<kBN, kSplits, false, true>(group, grid, stream)
            : launch_cluster_as<kBN, kSplits, false, false>(group, grid, stream);
}

template <int kBN>
int launch_cluster_bn(int splits, bool ta, bool tb, const ClusterGroup& group, int grid, cudaStream_t stream) {
  switch (splits) {
    case 1: return launch_cluster_split<kBN, 1>(ta, tb, group, grid, stream);
    case 2: return launch_cluster_split<kBN, 2>(ta, tb, group, grid, stream);
    case 4: return launch_cluster_split<kBN, 4>(ta, tb, group, grid, stream);
    case 8: return launch_cluster_split<kBN, 8>(ta, tb, group, grid, stream);
    default: return PRRTC_ERR_UNSUPPORTED;
  }
}

int launch_cluster(int bn, int splits, bool ta, bool tb, const ClusterGroup& group, int grid, cudaStream_t stream) {
  return bn == 64 ? launch_cluster_bn<64>(splits, ta, tb, group, grid, stream)
                  : launch_cluster_bn<128>(splits, ta, tb, group, grid, stream);
}

// SMs of the current device.
int sm_count() {
  static std::atomic<int> known[64];
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  const bool keep = dev >= 0 && dev < 64;
  if (keep && (n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 1;
  if (keep) known[dev].store(n, std::memory_order_relaxed);
  return n;
}

// The library's split of K: doubled while the 128 x 256 tiles fill less than
// one wave and every range keeps kMinKTilesPerSplit K tiles.
int auto_splits(int M, int N, int K, int sms) {
  const int tiles = ((M + BM - 1) / BM) * ((N + BN - 1) / BN), k_tiles = (K + BK - 1) / BK;
  int splits = 1;
  while (splits < kMaxSplits && tiles * (splits * 2) <= sms && k_tiles / (splits * 2) >= kMinKTilesPerSplit)
    splits *= 2;
  return std::min(splits, k_tiles);
}

int cluster_blocks(int M, int N, int splits, int bn) {
  return ((M + BM - 1) / BM) * ((N + bn - 1) / bn) * splits;
}

// Tile width of the cluster kernel for a product, 0: not its size.  One wave:
// two blocks per SM.
int cluster_bn(int M, int N, int splits, int sms) {
  if (splits > kMaxClusterSplits || (splits & (splits - 1))) return 0;
  for (int bn : {64, 128})
    if (cluster_blocks(M, N, splits, bn) <= 2 * sms) return bn;
  return 0;
}

// Whether pairs of CTAs take the tiles (256 x 256) instead of single ones
// (128 x 256).  A pair loads a third less per MMA, which counts while the MMAs
// are the bound; with few K tiles the epilogue is, where the two kernels differ
// in the pairs' joint start and end.  Measured (us, single / pair), 4096^2:
// K 256 19.2 / 22.1, 512 21.8 / 24.4, 768 26.1 / 26.3, 1024 30.6 / 29.6, 2048
// 50.2 / 46.6, 4096 94.6 / 83.1; 8192^3 633 / 578; 9728 x 4096 K 512 35.3 /
// 40.3, 768 45.2 / 44.8, 1024 56.0 / 50.6.  The larger tiles may take more
// waves, each a tenth shorter for its work.
bool pair_pays(int M, int N, int k_tiles, int splits, int sms) {
  const int n = (N + BN - 1) / BN * splits;
  if (sms < 2 || k_tiles <= 12 * splits) return false;
  auto waves = [](int units, int at_once) { return (units + at_once - 1) / at_once; };
  return 10 * waves((M + 2 * BM - 1) / (2 * BM) * n, sms / 2) <= 11 * waves((M + BM - 1) / BM * n, sms);
}

// Adds one product to a group of clusters with tiles of bn columns.
int group_add(ClusterGroup& g, int& grid, int bn, int splits, const void* a, int lda, bool ta, const void* b, int ldb,
              bool tb, int M, int N, int K, const float* bias, int relu, const void* mask, int ldm, float* c32,
              int ldc32, void* c16, int ldc16) {
  const int k = g.n;
  if (!(ta ? cached_map(&g.a[k], a, K, M, lda, 0, BK) : cached_map(&g.a[k], a, M, K, lda, 0, BM)) ||
      !(tb ? cached_map(&g.b[k], b, K, N, ldb, 0, BK) : cached_map(&g.b[k], b, N, K, ldb, 0, bn)))
    return PRRTC_ERR_CUDA;
  g.ep[k] = ClusterEpilogue{M, N, (K + BK - 1) / BK, (M + BM - 1) / BM, bias, relu,
                            static_cast<const __nv_bfloat16*>(mask), ldm, c32, ldc32,
                            static_cast<__nv_bfloat16*>(c16), ldc16};
  g.first[k] = grid;
  g.n = k + 1;
  grid += cluster_blocks(M, N, splits, bn);
  return PRRTC_OK;
}

template <bool kTA, bool kTB, int kCtas>
int launch_gemm(const CUtensorMap& ma, const CUtensorMap& mb, const OutMaps& om, const Epilogue& ep, int grid,
                cudaStream_t stream) {
  constexpr int kSmem = Tile<kCtas>::kSmem;
  auto* fn = gemm_bf16_kernel<kTA, kTB, kCtas>;
  static std::atomic<uint64_t> attr{0};
  if (smem_attribute(attr, fn, kSmem) != cudaSuccess) return PRRTC_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kCtas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = kCtas > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, fn, ma, mb, om, ep) == cudaSuccess ? PRRTC_OK : PRRTC_ERR_CUDA;
}

}  // namespace

// Host launcher used by the MLP code and the C ABI entry point.  splits_hint:
// 0 = choose (split K while the tiles fill less than one wave), else forced.
int gemm_bf16_ld(const void* a, int lda, const void* b, int ldb, int M, int N, int K, const float* bias, int relu,
                 float* c32, int ldc32, void* c16, int ldc16, cudaStream_t stream, int splits_hint, int flags,
                 const void* mask, int ldm) {
  const int ta = flags & kTransA ? 1 : 0, tb = flags & kTransB ? 1 : 0;
  if (M <= 0 || N <= 0 || K <= 0 || !a || !b || (!c32 && !c16)) return PRRTC_ERR_INVALID_ARG;
  if (K % 8 || N % 8 || (c32 && ldc32 % 4) || (c16 && ldc16 % 8)) return PRRTC_ERR_UNSUPPORTED;
  if (lda < (ta ? M : K) || ldb < (tb ? N : K) || lda % 8 || ldb % 8) return PRRTC_ERR_UNSUPPORTED;
  if ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) return PRRTC_ERR_INVALID_ARG;
  if ((c32 && (reinterpret_cast<uintptr_t>(c32) & 15)) || (c16 && (reinterpret_cast<uintptr_t>(c16) & 15)))
    return PRRTC_ERR_INVALID_ARG;
  Epilogue ep{M, N, K, bias, relu, c32 ? 1 : 0, c16 ? 1 : 0, 1, 0, 0, 0, 0};
  ep.n_tiles = (N + BN - 1) / BN;
  ep.k_tiles = (K + BK - 1) / BK;
  ep.m_pad = (M + BM - 1) / BM * BM;
  const int sms = sm_count();
  int splits = splits_hint > 0 ? splits_hint : auto_splits(M, N, K, sms);
  splits = std::max(1, std::min(splits, std::min(kMaxSplits, ep.k_tiles)));
  if (const int bn = cluster_bn(M, N, splits, sms)) {
    ClusterGroup g;
    g.n = 0;
    g.late = 0;
    g.early = flags & kNextMayStart ? 1 : 0;
    int grid = 0;
    const int rc = group_add(g, grid, bn, splits, a, lda, ta, b, ldb, tb, M, N, K, bias, relu, mask, ldm, c32, ldc32,
                             c16, ldc16);
    return rc ? rc : launch_cluster(bn, splits, ta, tb, g, grid, stream);
  }
  if (mask || (ta && !tb)) return PRRTC_ERR_UNSUPPORTED;
  const bool pair = !ta && !tb && pair_pays(M, N, ep.k_tiles, splits, sms);
  const int ctas = pair ? 2 : 1;
  ep.m_tiles = (M + BM * ctas - 1) / (BM * ctas);
  CUtensorMap ma, mb;
  if (!(ta ? cached_map(&ma, a, K, M, lda, 0, BK) : cached_map(&ma, a, M, K, lda, 0, BM))) return PRRTC_ERR_CUDA;
  if (!(tb ? cached_map(&mb, b, K, N, ldb, 0, BK) : cached_map(&mb, b, N, K, ldb, 0, BN / ctas))) return PRRTC_ERR_CUDA;
  OutMaps om;
  std::memset(&om, 0, sizeof(om));
  if (c32 && !cached_map(&om.c32, c32, M, N, ldc32, 2)) return PRRTC_ERR_CUDA;
  if (c16 && !cached_map(&om.c16, c16, M, N, ldc16, 3)) return PRRTC_ERR_CUDA;
  ep.splits = splits;
  float* ws = nullptr;
  if (splits > 1) {
    ws = workspace((size_t)splits * ep.m_pad * N, stream);
    if (!ws) return PRRTC_ERR_OOM;
    if (!cached_map(&om.ws, ws, splits * ep.m_pad, N, N, 2)) return PRRTC_ERR_CUDA;
  }
  const int grid = ctas * std::min(ep.m_tiles * ep.n_tiles * splits, sms / ctas);
  const int rc = pair       ? launch_gemm<false, false, 2>(ma, mb, om, ep, grid, stream)
                 : ta && tb ? launch_gemm<true, true, 1>(ma, mb, om, ep, grid, stream)
                 : tb       ? launch_gemm<false, true, 1>(ma, mb, om, ep, grid, stream)
                            : launch_gemm<false, false, 1>(ma, mb, om, ep, grid, stream);
  if (rc) return rc;
  if (splits > 1) {
    const size_t work = (size_t)M * (N / 4);
    const int blocks = (int)std::min<size_t>((work + 255) / 256, (size_t)sms * 8);
    splitk_reduce_kernel<<<blocks, 256, 0, stream>>>(ws, splits, M, ep.m_pad, N, bias, relu, c32, ldc32,
                                                     static_cast<__nv_bfloat16*>(c16), ldc16);
    if (cudaGetLastError() != cudaSuccess) return PRRTC_ERR_CUDA;
  }
  return PRRTC_OK;
}

int gemm_gradients(const GradientProduct* p, int n, bool ready, cudaStream_t stream) {
  // products of one shape of cluster share a launch while it stays one wave
  ClusterGroup g;
  g.n = 0;
  g.late = ready ? 1 : 0;
  g.early = 1;
  int grid = 0, bn = 0, splits = 0;
  const int sms = sm_count();
  auto flush = [&]() {
    const int rc = g.n ? launch_cluster(bn, splits, true, true, g, grid, stream) : PRRTC_OK;
    g.n = 0;
    grid = 0;
    return rc;
  };
  int rc = PRRTC_OK;
  for (int i = 0; i < n && !rc; ++i) {
    const GradientProduct& q = p[i];
    const int s = auto_splits(q.out, q.in, q.rows, sms), w = cluster_bn(q.out, q.in, s, sms);
    if (!w) {  // from 4096 rows on: more splits than a cluster takes
      rc = gemm_bf16_ld(q.dz, q.out, q.h, q.in, q.out, q.in, q.rows, nullptr, 0, q.dw, q.in, nullptr, 0, stream, 0,
                        kTransA | kTransB, nullptr, 0);
      continue;
    }
    if (g.n && (g.n == kMaxGroup || w != bn || s != splits ||
                grid + cluster_blocks(q.out, q.in, s, w) > 2 * sms))
      rc = flush();
    bn = w;
    splits = s;
    if (!rc)
      rc = group_add(g, grid, bn, splits, q.dz, q.out, true, q.h, q.in, true, q.out, q.in, q.rows, nullptr, 0, nullptr,
                     0, q.dw, q.in, nullptr, 0);
  }
  return rc ? rc : flush();
}

int gemm_bf16(const void* a, const void* b, int M, int N, int K, const float* bias, int relu, float* c32, int ldc32,
              void* c16, int ldc16, cudaStream_t stream) {
  return gemm_bf16_ld(a, K, b, K, M, N, K, bias, relu, c32, ldc32, c16, ldc16, stream, 0, kNextMayStart, nullptr, 0);
}

// Changes whenever a split-K workspace is allocated or moved: work captured
// into a CUDA graph before the change may point at a freed workspace.
uint64_t gemm_workspace_epoch() { return g_ws_epoch.load(); }

// Reads and clears the kernel's error word (synchronous).
int gemm_take_error() {
  int e = 0, z = 0;
  if (cudaMemcpyFromSymbol(&e, g_gemm_error, sizeof(int)) != cudaSuccess) return PRRTC_ERR_CUDA;
  if (e) cudaMemcpyToSymbol(g_gemm_error, &z, sizeof(int));
  return e;
}

cudaError_t gemm_read_error(int* out, cudaStream_t stream) {
  return cudaMemcpyFromSymbolAsync(out, g_gemm_error, sizeof(int), 0, cudaMemcpyDeviceToHost, stream);
}

}  // namespace prrtc

// On the caller's stream nothing starts before the outputs are written, whatever
// launch attributes it has: the next launch there is not the library's own.
extern "C" int prrtc_gemm_bf16_splitk(const void* a, const void* b, int32_t M, int32_t N, int32_t K,
                                      const float* bias, int32_t relu, float* c32, void* c16, int32_t splits,
                                      void* stream) {
  if (splits < 0) return PRRTC_ERR_INVALID_ARG;
  return prrtc::gemm_bf16_ld(a, K, b, K, M, N, K, bias, relu, c32, N, c16, N, static_cast<cudaStream_t>(stream),
                             splits, 0, nullptr, 0);
}

extern "C" int prrtc_gemm_bf16(const void* a, const void* b, int32_t M, int32_t N, int32_t K, const float* bias,
                               int32_t relu, float* c32, void* c16, void* stream) {
  return prrtc_gemm_bf16_splitk(a, b, M, N, K, bias, relu, c32, c16, 0, stream);
}

extern "C" int prrtc_gemm_error(void) { return prrtc::gemm_take_error(); }
