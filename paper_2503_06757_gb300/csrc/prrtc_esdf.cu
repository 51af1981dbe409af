// prrtc_esdf.cu -- Euclidean signed distance fields on a voxel grid for the
// collision check against distance maps (the paper's ESDF setting, Sec. III-A
// and its real-world experiments): voxelisation of primitive obstacles and
// the signed distance transform of an occupancy grid.
//
// The transform is exact: squared distances between voxel centres are
// integers, and the squared Euclidean distance separates into three 1-D
// minimisations (along x, then y, then z) of f(t) + (i - t)^2.  A free voxel
// needs the distance to the nearest occupied one and is itself at distance 0
// from the free ones, an occupied voxel the other way round: one signed number
// per voxel (positive: free) carries the whole state between the passes.
//
// Voxels of the other kind are at distance 0, so along a line only the voxels
// of the same run of free (or occupied) voxels and the two voxels that bound
// the run can be nearest.
#include <algorithm>
#include <climits>

#include "prrtc.h"
#include "prrtc_launch.h"

namespace prrtc {
namespace {

constexpr int kInf = 1 << 29;  // "none on this line"; + n^2 cannot overflow

__global__ void voxelize_kernel(EnvView env, float ox, float oy, float oz, float voxel, int nx, int ny, int nz,
                                uint8_t* __restrict__ occ) {
  const size_t V = (size_t)nx * ny * nz;
  for (size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(v % nx), j = (int)((v / nx) % ny), k = (int)(v / ((size_t)nx * ny));
    const float px = ox + ((float)i + 0.5f) * voxel, py = oy + ((float)j + 0.5f) * voxel,
                pz = oz + ((float)k + 0.5f) * voxel;
    bool inside = false;
    const float4* e = env.data;
    for (int o = 0; o < env.n_aabb; ++o) {
      const float4 c = e[2 * o], h = e[2 * o + 1];
      inside |= fabsf(px - c.x) < h.x && fabsf(py - c.y) < h.y && fabsf(pz - c.z) < h.z;
    }
    e += 2 * env.n_aabb;
    for (int o = 0; o < env.n_obb; ++o) {
      const float4 c = e[5 * o], h = e[5 * o + 1], a = e[5 * o + 2], b = e[5 * o + 3], d = e[5 * o + 4];
      const float vx = px - c.x, vy = py - c.y, vz = pz - c.z;
      const float lx = fmaf(a.x, vx, fmaf(a.y, vy, a.z * vz));
      const float ly = fmaf(b.x, vx, fmaf(b.y, vy, b.z * vz));
      const float lz = fmaf(d.x, vx, fmaf(d.y, vy, d.z * vz));
      inside |= fabsf(lx) < h.x && fabsf(ly) < h.y && fabsf(lz) < h.z;
    }
    e += 5 * env.n_obb;
    for (int o = 0; o < env.n_cyl; ++o) {
      const float4 c = e[2 * o], a = e[2 * o + 1];
      const float vx = px - c.x, vy = py - c.y, vz = pz - c.z;
      const float z = fmaf(a.x, vx, fmaf(a.y, vy, a.z * vz));
      const float wx = fmaf(-z, a.x, vx), wy = fmaf(-z, a.y, vy), wz = fmaf(-z, a.z, vz);
      inside |= fabsf(z) < a.w && fmaf(wx, wx, fmaf(wy, wy, wz * wz)) < c.w * c.w;
    }
    e += 2 * env.n_cyl;
    for (int o = 0; o < env.n_sph; ++o) {
      const float4 s = e[o];
      const float dx = px - s.x, dy = py - s.y, dz = pz - s.z;
      inside |= fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < s.w * s.w;
    }
    occ[v] = inside ? 1 : 0;
  }
}

// Distance to the nearest voxel of the other kind along x, signed; kNoneX: none
// in the row (256^3: 41 us, a voxel scanning its row 903 us before).  A warp per row: the row as bit words (lane w holds word w, at
// most 1024 / 32 of them), the nearest set bit of the other kind within the
// voxel's word or, from two scans over the words, outside it.
constexpr int kNoneX = 0x7fff;

__global__ void edt_x_kernel(const uint8_t* __restrict__ occ, int nx, size_t rows, int16_t* __restrict__ out) {
  constexpr int kFar = 1 << 20;
  const int lane = threadIdx.x & 31, words = (nx + 31) >> 5;
  const size_t warps = (size_t)gridDim.x * (blockDim.x >> 5);
  for (size_t r = (size_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps) {
    const uint8_t* row = occ + r * nx;
    uint32_t mine = 0;  // occupied bits of word `lane`
#pragma unroll 4
    for (int w = 0; w < words; ++w) {
      const int i = w * 32 + lane;
      const uint32_t b = __ballot_sync(kFull, i < nx && row[i]);
      if (lane == w) mine = b;
    }
    const uint32_t in = lane < words ? (lane == words - 1 && (nx & 31) ? (1u << (nx & 31)) - 1u : kFull) : 0u;
    const uint32_t bits[2] = {~mine & in, mine};  // free, occupied
    int before[2], after[2];                      // nearest of each kind in the words before / after word `lane`
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      int last = bits[k] ? lane * 32 + 31 - __clz(bits[k]) : -kFar;
      int first = bits[k] ? lane * 32 + __ffs(bits[k]) - 1 : kFar;
      for (int off = 1; off < words; off <<= 1) {
        const int up = __shfl_up_sync(kFull, last, off), down = __shfl_down_sync(kFull, first, off);
        if (lane >= off) last = max(last, up);
        if (lane + off < 32) first = min(first, down);
      }
      before[k] = __shfl_up_sync(kFull, last, 1);
      after[k] = __shfl_down_sync(kFull, first, 1);
      if (lane == 0) before[k] = -kFar;
      if (lane == 31) after[k] = kFar;
    }
#pragma unroll 4
    for (int w = 0; w < words; ++w) {
      const int i = w * 32 + lane;
      const uint32_t f = __shfl_sync(kFull, bits[0], w), o = __shfl_sync(kFull, bits[1], w);
      const int bf = __shfl_sync(kFull, before[0], w), bo = __shfl_sync(kFull, before[1], w);
      const int af = __shfl_sync(kFull, after[0], w), ao = __shfl_sync(kFull, after[1], w);
      const bool is_occ = (o >> lane) & 1u;
      const uint32_t other = is_occ ? f : o;
      const uint32_t left = other & ((1u << lane) - 1u), right = other & ~((2u << lane) - 1u);
      const int lo = left ? w * 32 + 31 - __clz(left) : (is_occ ? bf : bo);
      const int hi = right ? w * 32 + __ffs(right) - 1 : (is_occ ? af : ao);
      const int d = min(min(i - lo, hi - i), kNoneX);
      if (i < nx) out[r * nx + i] = (int16_t)(is_occ ? -d : d);
    }
  }
}

// One number of the pass before as a signed squared distance (+-kInf: none).
__device__ __forceinline__ int load_sq(const int16_t* p) {
  const int d = __ldg(p), m = abs(d);
  const int q = m >= kNoneX ? kInf : m * m;
  return d < 0 ? -q : q;
}
__device__ __forceinline__ int load_sq(const int* p) { return __ldg(p); }

// What a pass writes: the signed squared distance, or (last pass) the field,
// voxel * distance, +- the grid diagonal where no voxel of the other kind exists.
__device__ __forceinline__ void store_sq(int* p, bool occ, int q, float, float) { *p = occ ? -q : q; }
__device__ __forceinline__ void store_sq(float* p, bool occ, int q, float voxel, float diag) {
  const float mag = q >= kInf ? diag : voxel * sqrtf((float)q);
  *p = occ ? -mag : mag;
}

// Squared distance that a voxel offers to the voxels of its own kind (v > 0),
// and 0 to those of the other; "none" stays at or above kInf.
__device__ __forceinline__ int own_sq(int v, int16_t) { return max(v, 0) * max(v, 0); }
__device__ __forceinline__ int own_sq(int v, int) { return max(v, 0); }

// Pass along an axis of length n and element stride `stride` (y: nx, z:
// nx*ny), small grids: a thread per voxel looks at its whole line, eight
// voxels in flight; neighbouring threads read neighbouring voxels.
template <class In, class Out>
__global__ void edt_scan_kernel(const In* __restrict__ in, int n, size_t stride, size_t V, Out* __restrict__ out,
                                float voxel, float diag) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;  // V < 2^31
  if (v >= V) return;
  const int pos = (int)(v / (uint32_t)stride % (uint32_t)n);
  const In* p = in + (v - (size_t)pos * stride);
  const bool occ = __ldg(in + v) < 0;
  const int kind = occ ? -1 : 1;
  int best = INT_MAX, d = pos, left = n;
  for (; left >= 8; left -= 8, p += 8 * stride, d -= 8) {
    int f[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) f[u] = __ldg(p + u * stride);
#pragma unroll
    for (int u = 0; u < 8; ++u) best = min(best, own_sq(f[u] * kind, In{}) + (d - u) * (d - u));
  }
  for (; left > 0; --left, p += stride, --d) best = min(best, own_sq(__ldg(p) * kind, In{}) + d * d);
  best = min(best, kInf);
  store_sq(out + v, occ, best, voxel, diag);
}

// The same pass for large grids.  For the voxels of one kind, the nearest place t*(i) minimises
// f(t) + (i - t)^2, with f = 0 at the voxels of the other kind, and the
// leftmost such t* never decreases with i.  So the place of the middle voxel
// splits the line: voxels left of it need look no further right than t*, those
// right of it no further left; log2(n) levels, each n steps a line, all voxels
// of a level at once.  A block takes 32 lines (lane = line, neighbours in
// memory) into shared memory; a warp takes one voxel of a level, in all 32
// lines.  The more frequent kind of the block's voxels goes this way; the
// others (as a rule the occupied ones: obstacles are thin) look outwards until
// the offset alone exceeds the best distance, at worst one step a voxel of
// their run.
//
// A candidate is one 32-bit key, (f(t) + (i - t)^2) << 10 | t (t below 1024,
// values below 2^22 with "none" at kNoneSq), so that a step is one minimum and
// ties go to the leftmost t.  The first levels have fewer voxels than the block
// has warps: the warps share a range.  What bounds the pass is instruction
// issue (75% of the slots), so the last two levels, three quarters of the
// voxels, go together: three voxels share the loads, the loop and the range,
// and store no place (256^3: 142 us a pass with every level by itself, 111 so;
// 80^3 14.5 and 9.5).
constexpr int kAxisWarps = 8;
constexpr int kNoneSq = 3140000;  // above 3 * 1023^2; with 1026^2 (padded positions) still below 2^22

constexpr int kAxisPad = 3;       // rows past the line that a step of four may touch

__host__ __device__ constexpr int axis_smem(int n) {
  return 32 * ((n + kAxisPad) * (int)sizeof(int) + n * (int)sizeof(uint16_t));
}

// Smallest key of voxel i over at least t = lo .. hi of the lane's column of
// 32-strided values (n of them, then kAxisPad rows of "none").  The lanes take
// as many steps as the longest range needs, four at a time, each from its own
// lo or, near the line's end, from farther left: positions outside the range
// lose against its leftmost minimum.
__device__ __forceinline__ uint32_t nearest_key(const int* __restrict__ col, int i, int lo, int hi, int n) {
  const int steps = (__reduce_max_sync(kFull, hi - lo) + 4) & ~3;
  int t = max(min(lo, n + kAxisPad - steps), 0);
  uint32_t k0 = ~0u, k1 = ~0u;
  const int* p = col + t * 32;
  for (int left = steps; left > 0; left -= 4, p += 128, t += 4) {
    int f[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) f[u] = max(p[u * 32], 0);
    const int d = i - t;
    k0 = min(k0, (uint32_t)(d * d + f[0]) << 10 | (uint32_t)t);
    k1 = min(k1, (uint32_t)((d - 1) * (d - 1) + f[1]) << 10 | (uint32_t)(t + 1));
    k0 = min(k0, (uint32_t)((d - 2) * (d - 2) + f[2]) << 10 | (uint32_t)(t + 2));
    k1 = min(k1, (uint32_t)((d - 3) * (d - 3) + f[3]) << 10 | (uint32_t)(t + 3));
  }
  return min(k0, k1);
}

// The same for voxels i, i + 1 and i + 2 over one range.
__device__ __forceinline__ void nearest_keys(const int* __restrict__ col, int i, int lo, int hi, int n,
                                             uint32_t (&key)[3]) {
  const int steps = (__reduce_max_sync(kFull, hi - lo) + 4) & ~3;
  int t = max(min(lo, n + kAxisPad - steps), 0);
  const int* p = col + t * 32;
  key[0] = key[1] = key[2] = ~0u;
  for (int left = steps; left > 0; left -= 4, p += 128) {
    int f[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) f[u] = max(p[u * 32], 0);
#pragma unroll
    for (int u = 0; u < 4; ++u, ++t) {
      const int d = i - t;
#pragma unroll
      for (int v = 0; v < 3; ++v) key[v] = min(key[v], (uint32_t)((d + v) * (d + v) + f[u]) << 10 | (uint32_t)t);
    }
  }
}

template <class In, class Out>
__global__ void __launch_bounds__(kAxisWarps * 32) edt_axis_kernel(const In* __restrict__ in, int n, size_t stride,
                                                                   size_t lines, Out* __restrict__ out, float voxel,
                                                                   float diag) {
  extern __shared__ int axis_smem_raw[];
  __shared__ int s_count[kAxisWarps];
  __shared__ uint32_t s_key[kAxisWarps][32];                    // shared voxels of the first levels
  int* s = axis_smem_raw;  // [n + kAxisPad][32], the more frequent kind positive
  uint16_t* nearest = reinterpret_cast<uint16_t*>(s + (n + kAxisPad) * 32);  // [n][32], t*
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const size_t line = (size_t)blockIdx.x * 32 + lane;
  const bool live = line < lines;
  const size_t at = live ? line : lines - 1;
  const size_t base = (at / stride) * (stride * (size_t)n) + at % stride;
  in += base;
  out += base;
  int count = 0;
#pragma unroll 8
  for (int i = warp; i < n; i += kAxisWarps) {
    const int v = load_sq(in + (size_t)i * stride);
    s[i * 32 + lane] = max(min(v, kNoneSq), -kNoneSq);
    count += v < 0 ? -1 : 1;
  }
  count = __reduce_add_sync(kFull, count);
  if (lane == 0) s_count[warp] = count;
  s_key[warp][lane] = ~0u;
  if (warp < kAxisPad) s[(n + warp) * 32 + lane] = kNoneSq;
  __syncthreads();
  count = 0;
#pragma unroll
  for (int w = 0; w < kAxisWarps; ++w) count += s_count[w];
  const bool flip = count < 0;  // more occupied voxels: they are the positive ones
  if (flip) {
    for (int i = warp; i < n; i += kAxisWarps) s[i * 32 + lane] = -s[i * 32 + lane];
    __syncthreads();
  }
  const int* col = s + lane;
  // voxel i's minimum: its place for the next levels, and the voxel's value
  auto write = [&](int i, uint32_t key) {
    const int q = (int)(key >> 10);
    if (live && col[i * 32] > 0) store_sq(out + (size_t)i * stride, flip, q >= kNoneSq ? kInf : q, voxel, diag);
  };
  auto finish = [&](int i, uint32_t key) {
    nearest[i * 32 + lane] = (uint16_t)(key & 1023u);
    write(i, key);
  };
  int half = 1;
  while (2 * half <= n) half *= 2;
  for (; half > 2; half >>= 1) {
    // voxels half - 1, 3 half - 1, ...; those at +-half are done
    const int nodes = (n - half) / (2 * half) + 1;
    const int parts = nodes >= kAxisWarps ? 1 : kAxisWarps / nodes;
    for (int k = parts > 1 ? warp / parts : warp; k < nodes; k += kAxisWarps) {
      const int i = half - 1 + 2 * half * k;
      const int lo = i - half >= 0 ? nearest[(i - half) * 32 + lane] : 0;
      const int hi = i + half < n ? nearest[(i + half) * 32 + lane] : n - 1;
      if (parts == 1) {
        finish(i, nearest_key(col, i, lo, hi, n));
      } else {
        const int len = (hi - lo + parts) / parts, first = min(lo + (warp % parts) * len, hi);
        atomicMin(&s_key[k][lane], nearest_key(col, i, first, min(first + len - 1, hi), n));
      }
    }
    __syncthreads();
    if (parts > 1) {
      if (warp < nodes) {
        finish(half - 1 + 2 * half * warp, s_key[warp][lane]);
        s_key[warp][lane] = ~0u;
      }
      __syncthreads();
    }
  }
  // The last two levels at once: voxels 4 k, 4 k + 1 and 4 k + 2 between the
  // places of 4 k - 1 and 4 k + 3.  Three quarters of the voxels share a range
  // by three and need no place of their own.
  for (int i = 4 * warp; i < n; i += 4 * kAxisWarps) {
    const int lo = i > 0 ? nearest[(i - 1) * 32 + lane] : 0;
    const int hi = i + 3 < n ? nearest[(i + 3) * 32 + lane] : n - 1;
    uint32_t key[3];
    nearest_keys(col, i, lo, hi, n, key);
#pragma unroll
    for (int v = 0; v < 3; ++v)
      if (i + v < n) write(i + v, key[v]);
  }
  if (abs(count) == n * 32) return;  // no voxel of the other kind
  // the other kind, outwards, four steps to each side at a time
  for (int i = warp; i < n; i += kAxisWarps) {
    int best = live ? -col[i * 32] : -1;
    const bool mine = best > 0;
    const int reach = max(i, n - 1 - i);
    for (int r = 1; r <= reach && r * r < best; r += 4) {
      int a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[u] = i - r - u >= 0 ? max(-col[(i - r - u) * 32], 0) : kNoneSq;
        b[u] = i + r + u < n ? max(-col[(i + r + u) * 32], 0) : kNoneSq;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) best = min(best, min(a[u], b[u]) + (r + u) * (r + u));
    }
    if (mine) store_sq(out + (size_t)i * stride, !flip, best >= kNoneSq ? kInf : best, voxel, diag);
  }
}

// Whether the pass scans whole lines.  It takes about V n / 2.4e6 us, the
// search by levels about 7 us + V / 1.5e5 us, so the line is V (n - 24) =
// 1.4e7.  Measured (us, scan / levels): 48^3 5 / 9, 64^3 8.7 / 9, 80^3 17 / 11,
// 100^3 33 / 16, 256^3 1225 / 111; n = 16 of 200 x 16 x 256 9 / 15; n = 256 of
// 16 x 16 x 256 14 / 14; n = 128 of 16 x 128 x 128 14 / 9.5.  Before, with both
// kinds scanned and two numbers per voxel: 64^3 10, 80^3 20, 100^3 42, 256^3
// 1540 (y) and 2350 (z).
bool scan_pays(int n, size_t V) { return n <= 24 || V * (size_t)(n - 24) < 14000000; }

int grid_for(size_t V) {
  const size_t blocks = (V + 255) / 256;
  return (int)(blocks < 65535 ? blocks : 65535);
}

template <class In, class Out>
cudaError_t launch_axis(const In* in, int n, size_t stride, size_t V, Out* out, float voxel, float diag,
                        cudaStream_t stream) {
  if (scan_pays(n, V)) {
    edt_scan_kernel<<<(int)((V + 255) / 256), 256, 0, stream>>>(in, n, stride, V, out, voxel, diag);
    return cudaGetLastError();
  }
  const cudaError_t e = cudaFuncSetAttribute(edt_axis_kernel<In, Out>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             axis_smem(PRRTC_ESDF_MAX_DIM));
  if (e != cudaSuccess) return e;
  const size_t lines = V / n;
  edt_axis_kernel<<<(int)((lines + 31) / 32), kAxisWarps * 32, axis_smem(n), stream>>>(in, n, stride, lines, out,
                                                                                       voxel, diag);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_voxelize(const EnvView& env, const float origin[3], float voxel, const int dims[3], uint8_t* occ,
                            cudaStream_t stream) {
  const size_t V = (size_t)dims[0] * dims[1] * dims[2];
  if (V == 0) return cudaSuccess;
  voxelize_kernel<<<grid_for(V), 256, 0, stream>>>(env, origin[0], origin[1], origin[2], voxel, dims[0], dims[1],
                                                   dims[2], occ);
  return cudaGetLastError();
}

cudaError_t launch_esdf(const uint8_t* occ, const int dims[3], float voxel, void* tmp, float* out,
                        cudaStream_t stream) {
  const size_t nx = dims[0], ny = dims[1], nz = dims[2], V = nx * ny * nz;
  if (V == 0) return cudaSuccess;
  int* sq = static_cast<int*>(tmp);
  int16_t* dx = reinterpret_cast<int16_t*>(sq + V);
  const size_t rows = ny * nz;
  edt_x_kernel<<<(int)std::min<size_t>((rows + 7) / 8, 65535), 256, 0, stream>>>(occ, dims[0], rows, dx);
  const float diag = voxel * sqrtf((float)dims[0] * dims[0] + (float)dims[1] * dims[1] + (float)dims[2] * dims[2]);
  cudaError_t e = launch_axis(dx, dims[1], nx, V, sq, voxel, diag, stream);
  if (e == cudaSuccess) e = launch_axis(sq, dims[2], nx * ny, V, out, voxel, diag, stream);
  return e;
}

}  // namespace prrtc
