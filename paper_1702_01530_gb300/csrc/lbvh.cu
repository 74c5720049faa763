// Linear BVH build on the GPU (sm_103a).
//
// Table 1 of the paper names BVH trees as the GPU-friendly acceleration
// structure; this is the linear BVH over Morton codes:
//   1. k_centroid_bounds : FP64 centroids (triangle ((v0+v1)+v2)/3, every
//      operation correctly rounded, no FMA), their per-axis min/max per block.
//      FP64 units are few, so triangles are compared by their sums (division
//      by 3 is monotonic) and as integers.
//   2. k_reduce_bounds     : the bounds of all blocks.
//   3. k_keys              : q_a = min(1023, floor((c_a - min_a) /
//      (max_a - min_a) * 1024)) (0 when the extent is 0), morton30 with x at
//      bit 3k+2, y at 3k+1, z at 3k; key = morton30 << 32 | primitive id. An
//      FP32 estimate decides the cell wherever its error bound keeps it clear
//      of a cell boundary; the FP64 definition decides the others.
//   4. radix sort          : stable LSD sort on the 30 Morton bits (8-bit
//      digits; per pass a histogram of every 2048-key tile (k_keys makes the
//      first), a scan of each digit's tile counts, a scatter). Keys start in
//      id order, so the result is sorted by the whole 64-bit key.
//   5. k_karras            : binary radix tree over the sorted keys, one
//      thread per internal node (direction, range end, split by binary
//      search on delta(i, j) = clz(key_i ^ key_j)).
//   6. k_refit             : leaf boxes (triangle min/max; sphere c -/+ r in
//      FP64 rounded outward to FP32) and bottom-up refit: the second thread to
//      arrive at a node merges both children and climbs on. A node whose
//      leaves all belong to one block (all but a few per block) is met in
//      shared memory; only the others pay for global arrival counters and
//      fences.
//
// Measured (GB300, 1,000,000 primitives in random order, the whole device-side
// build): 0.359 ms; 1.110 before, when one block scanned the tile counts
// (0.40), one thread reduced the bounds (0.12), every key was divided twice in
// FP64 (0.27 with the bounds) and every node had a global arrival counter
// (0.18). The kernels' shares now (alone, cold caches): refit 125 us, scatter
// 4 x 14, karras 38, bounds 38, keys 22, histograms 3 x 7, scans 4 x 4.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "rt_internal.cuh"

namespace rt {
namespace {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;                       // items per thread per tile
constexpr int kTile = kSortThreads * kSortItems;    // 2048 keys per block
constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 256;

struct Bounds6 { double lo[3], hi[3]; };

// triangle i of 10-word records; `wide`: the array is 8-byte aligned
__device__ __forceinline__ void load_tri(const float* t, uint32_t i, bool wide, float v[9]) {
  const float* p = t + 10ull * i;
  if (wide) {
    const float2* q = reinterpret_cast<const float2*>(p);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 x = __ldg(q + k);
      v[2 * k] = x.x;
      v[2 * k + 1] = x.y;
    }
    v[8] = __ldg(p + 8);
  } else {
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = __ldg(p + k);
  }
}

// (v0 + v1) + v2 of one axis, each addition correctly rounded
__device__ __forceinline__ double sum3(const float v[9], int k) {
  return __dadd_rn(__dadd_rn((double)v[k], (double)v[3 + k]), (double)v[6 + k]);
}

// order-preserving integer image of a double (no NaN)
__device__ __forceinline__ long long d2o(double d) {
  const long long b = __double_as_longlong(d);
  return b >= 0 ? b : b ^ 0x7FFFFFFFFFFFFFFFll;
}
__device__ __forceinline__ double o2d(long long o) {
  return __longlong_as_double(o >= 0 ? o : o ^ 0x7FFFFFFFFFFFFFFFll);
}

// per-block partial min/max of the centroids; spheres by their centres,
// triangles by the sums of their vertices, divided by 3 at the end
__global__ void k_centroid_bounds(const float* sph, const float* tri, uint32_t ns, uint32_t n, bool wide,
                                  Bounds6* partial) {
  __shared__ long long s[12][kRedThreads / 32];
  const long long kMost = 0x7FFFFFFFFFFFFFFFll;
  long long v[12];                 // sphere min, triangle min, sphere -max, triangle -max (x, y, z each)
#pragma unroll
  for (int k = 0; k < 12; ++k) v[k] = kMost;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (i < ns) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const long long o = d2o((double)__ldg(sph + 5ull * i + k));
        v[k] = min(v[k], o);
        v[6 + k] = min(v[6 + k], ~o);
      }
    } else {
      float t[9];
      load_tri(tri, i - ns, wide, t);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const long long o = d2o(sum3(t, k));
        v[3 + k] = min(v[3 + k], o);
        v[9 + k] = min(v[9 + k], ~o);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 12; ++k)
    for (int off = 16; off > 0; off >>= 1) v[k] = min(v[k], __shfl_xor_sync(0xFFFFFFFFu, v[k], off));
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int k = 0; k < 12; ++k) s[k][threadIdx.x >> 5] = v[k];
  __syncthreads();
  if (threadIdx.x >= 3) return;
  long long m[4] = {kMost, kMost, kMost, kMost};
  for (int q = 0; q < 4; ++q)
    for (int w = 0; w < kRedThreads / 32; ++w) m[q] = min(m[q], s[3 * q + threadIdx.x][w]);
  double lo = INFINITY, hi = -INFINITY;
  if (m[0] != kMost) { lo = o2d(m[0]); hi = o2d(~m[2]); }
  if (m[1] != kMost) {
    lo = fmin(lo, __ddiv_rn(o2d(m[1]), 3.0));
    hi = fmax(hi, __ddiv_rn(o2d(~m[3]), 3.0));
  }
  partial[blockIdx.x].lo[threadIdx.x] = lo;
  partial[blockIdx.x].hi[threadIdx.x] = hi;
}

// bounds of all blocks: warp q takes value q (lo x, y, z, hi x, y, z)
__global__ void k_reduce_bounds(Bounds6* partial, int nparts) {
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double m = q < 3 ? INFINITY : -INFINITY;
  for (int p = lane; p < nparts; p += 32) {
    const double x = q < 3 ? partial[p].lo[q] : partial[p].hi[q - 3];
    m = q < 3 ? fmin(m, x) : fmax(m, x);
  }
  for (int off = 16; off > 0; off >>= 1) {
    const double x = __shfl_xor_sync(0xFFFFFFFFu, m, off);
    m = q < 3 ? fmin(m, x) : fmax(m, x);
  }
  __syncthreads();               // every warp has read partial[0]
  if (lane == 0) { if (q < 3) partial[0].lo[q] = m; else partial[0].hi[q - 3] = m; }
}

__device__ __forceinline__ uint32_t quantise(double c, double lo, double hi) {
  double ext = __dsub_rn(hi, lo);
  if (ext == 0.0) return 0u;
  double f = floor(__dmul_rn(__ddiv_rn(__dsub_rn(c, lo), ext), 1024.0));
  f = fmin(1023.0, fmax(0.0, f));
  return (uint32_t)f;
}

__device__ __forceinline__ uint32_t spread10(uint32_t x) {  // bit k -> bit 3k
  x &= 0x3FFu;
  x = (x | (x << 16)) & 0x030000FFu;
  x = (x | (x << 8)) & 0x0300F00Fu;
  x = (x | (x << 4)) & 0x030C30C3u;
  x = (x | (x << 2)) & 0x09249249u;
  return x;
}

// FP32 view of one axis' quantisation: f = (c - lo) * scale, and the error of
// f = 1024 (c - lo) / (hi - lo) is at most err_m * (largest |coordinate|) + err_0
struct AxisEstimate { float lo, scale, err_m, err_0; };

__device__ __forceinline__ AxisEstimate axis_estimate(double lo, double hi) {
  AxisEstimate e;
  const float ext = (float)(hi - lo);
  e.lo = (float)lo;
  e.scale = 1024.f / ext;
  // sum of three (2 roundings of at most 3 |v|) and the product by 1/3: under
  // 4 |v| 2^-24; lo: |lo| 2^-24; difference, scale and product: under 6 f 2^-24
  // of f <= 1025. Twice that.
  e.err_m = e.scale * 8.f * 0x1p-24f;
  e.err_0 = e.scale * fabsf(e.lo) * 2.f * 0x1p-24f + 1025.f * 12.f * 0x1p-24f;
  return e;
}

// Keys of a tile of the sort, and the tile's histogram of the lowest digit
__global__ void __launch_bounds__(kSortThreads)
k_keys(const float* sph, const float* tri, uint32_t ns, uint32_t n, bool wide, const Bounds6* b,
       uint64_t* keys, uint32_t* ghist, int nblocks) {
  __shared__ uint32_t h[256];
  __shared__ AxisEstimate est[3];
  h[threadIdx.x] = 0;
  if (threadIdx.x < 3) est[threadIdx.x] = axis_estimate(b->lo[threadIdx.x], b->hi[threadIdx.x]);
  __syncthreads();
  const uint64_t base = (uint64_t)blockIdx.x * kTile;
  for (int r = 0; r < kSortItems; ++r) {
    const uint64_t i64 = base + (uint64_t)r * kSortThreads + threadIdx.x;
    if (i64 >= n) break;
    const uint32_t i = (uint32_t)i64;
    float v[9];
    const bool is_sphere = i < ns;
    if (is_sphere)
      for (int k = 0; k < 3; ++k) v[k] = v[3 + k] = v[6 + k] = __ldg(sph + 5ull * i + k);
    else
      load_tri(tri, i - ns, wide, v);
    uint32_t q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const AxisEstimate e = est[k];
      const float m = fmaxf(fabsf(v[k]), fmaxf(fabsf(v[3 + k]), fabsf(v[6 + k])));
      const float c = is_sphere ? v[k] : ((v[k] + v[3 + k]) + v[6 + k]) * (1.f / 3.f);
      const float f = (c - e.lo) * e.scale, fl = floorf(f), err = fmaf(e.err_m, m, e.err_0);
      // a comparison with a NaN or an infinity fails: the definition decides
      if (f - fl > err && fl + 1.f - f > err && fl >= 0.f && fl <= 1023.f)
        q[k] = (uint32_t)fl;
      else
        q[k] = quantise(is_sphere ? (double)v[k] : __ddiv_rn(sum3(v, k), 3.0), b->lo[k], b->hi[k]);
    }
    const uint32_t m = (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
    keys[i] = ((uint64_t)m << 32) | i;
    atomicAdd(&h[m & 0xFFu], 1u);
  }
  __syncthreads();
  ghist[(size_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// ---------------------------------------------------------------- radix sort
__global__ void k_hist(const uint64_t* keys, uint32_t n, int shift, uint32_t* ghist, int nblocks) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  uint64_t base = (uint64_t)blockIdx.x * kTile;
  for (int r = 0; r < kSortItems; ++r) {
    uint64_t i = base + (uint64_t)r * kSortThreads + threadIdx.x;
    if (i < n) atomicAdd(&h[(keys[i] >> shift) & 0xFF], 1u);
  }
  __syncthreads();
  ghist[(size_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// exclusive scan of each digit's tile counts (block d: row d of ghist), and
// the digit's total
__global__ void __launch_bounds__(256) k_scan(uint32_t* ghist, int nblocks, uint32_t* totals) {
  __shared__ uint32_t part[8];
  uint32_t* a = ghist + (size_t)blockIdx.x * nblocks;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t run = 0;
  for (int base = 0; base < nblocks; base += 256) {
    const int i = base + (int)threadIdx.x;
    const uint32_t v = i < nblocks ? a[i] : 0u;
    uint32_t incl = v;
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= (uint32_t)off) incl += x;
    }
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (uint32_t w = 0; w < 8; ++w) {
      if (w < warp) before += part[w];
      all += part[w];
    }
    if (i < nblocks) a[i] = run + before + incl - v;
    run += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = run;
}

// Stable scatter of one tile. Each warp ranks its 256 consecutive keys (8 per
// lane, in order) by match masks against its own digit counts, without waiting
// for the others; one block scan then turns the counts into positions, and the
// keys go through shared memory in digit order, so that neighbouring threads
// write neighbouring words of a digit's run.
__global__ void __launch_bounds__(kSortThreads)
k_scatter(const uint64_t* in, uint64_t* out, uint32_t n, int shift, const uint32_t* gscan, int nblocks,
          const uint32_t* totals) {
  constexpr int kWarps = kSortThreads / 32;
  __shared__ uint32_t wcnt[kWarps][256];
  __shared__ uint32_t to_global[256];          // global position of a digit's run minus its local one
  __shared__ uint32_t part[2][kWarps];
  __shared__ uint64_t sorted[kTile];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int w = 0; w < kWarps; ++w) wcnt[w][tid] = 0;
  const uint32_t total = totals[tid];
  const uint32_t run = gscan[(size_t)tid * nblocks + blockIdx.x];
  __syncthreads();
  const uint64_t first = (uint64_t)blockIdx.x * kTile + warp * (32u * kSortItems);
  uint64_t key[kSortItems];
  uint32_t rank[kSortItems];
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const uint64_t i = first + (uint64_t)r * 32 + lane;
    key[r] = i < n ? in[i] : ~0ull;
  }
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const bool valid = first + (uint64_t)r * 32 + lane < n;
    const uint32_t dig = valid ? (uint32_t)((key[r] >> shift) & 0xFF) : 256u;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, dig);
    const uint32_t before = valid ? wcnt[warp][dig] : 0u;
    rank[r] = before + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
    if (valid && (peers >> lane) == 1u) wcnt[warp][dig] = before + __popc(peers);   // the group's last lane
    __syncwarp();
  }
  __syncthreads();
  // thread d: counts of digit d per warp -> offsets; tile count and totals of
  // the digits below d by block scans
  uint32_t cnt = 0;
  for (int w = 0; w < kWarps; ++w) {
    const uint32_t c = wcnt[w][tid];
    wcnt[w][tid] = cnt;
    cnt += c;
  }
  uint32_t il = cnt, ig = total;
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, il, off), y = __shfl_up_sync(0xFFFFFFFFu, ig, off);
    if (lane >= (uint32_t)off) { il += x; ig += y; }
  }
  if (lane == 31) { part[0][warp] = il; part[1][warp] = ig; }
  __syncthreads();
  uint32_t local = il - cnt, global = ig - total;
  for (uint32_t w = 0; w < warp; ++w) { local += part[0][w]; global += part[1][w]; }
  to_global[tid] = global + run - local;
  for (int w = 0; w < kWarps; ++w) wcnt[w][tid] += local;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortItems; ++r)
    if (first + (uint64_t)r * 32 + lane < n)
      sorted[wcnt[warp][(uint32_t)((key[r] >> shift) & 0xFF)] + rank[r]] = key[r];
  __syncthreads();
  const uint64_t tile = (uint64_t)blockIdx.x * kTile;
  const uint32_t count = (uint32_t)(n - tile < (uint64_t)kTile ? n - tile : (uint64_t)kTile);
  for (uint32_t i = tid; i < count; i += kSortThreads) {
    const uint64_t k = sorted[i];
    out[to_global[(uint32_t)((k >> shift) & 0xFF)] + i] = k;
  }
}

// ------------------------------------------------------------ radix tree
__device__ __forceinline__ int delta(const uint64_t* k, int64_t n, int64_t i, int64_t j) {
  if (j < 0 || j >= n) return -1;
  return __clzll(k[i] ^ k[j]);
}

// also writes each node's range of leaves, [first, last]
__global__ void k_karras(const uint64_t* keys, uint32_t n, float4* nodes, int32_t* parent, uint2* range) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n - 1) return;
  int d = (delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1)) > 0 ? 1 : -1;
  int dmin = delta(keys, n, i, i - d);
  int64_t lmax = 2;
  while (delta(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
  int64_t l = 0;
  for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
    if (delta(keys, n, i, i + (l + t) * d) > dmin) l += t;
  int64_t j = i + l * d;
  int dnode = delta(keys, n, i, j);
  int64_t s = 0, t = l;
  do {
    t = (t + 1) >> 1;
    if (delta(keys, n, i, i + (s + t) * d) > dnode) s += t;
  } while (t > 1);
  int64_t g = i + s * d + min(d, 0);
  int32_t left = (min(i, j) == g) ? ~(int32_t)g : (int32_t)g;
  int32_t right = (max(i, j) == g + 1) ? ~(int32_t)(g + 1) : (int32_t)(g + 1);
  nodes[4 * i + 3] = make_float4(__int_as_float(left), __int_as_float(right), 0.f, 0.f);
  parent[left >= 0 ? left : (int64_t)n - 1 + ~left] = (int32_t)i;
  parent[right >= 0 ? right : (int64_t)n - 1 + ~right] = (int32_t)i;
  range[i] = make_uint2((uint32_t)min(i, j), (uint32_t)max(i, j));
  if (i == 0) parent[0] = -1;
}

// write box (lo, hi) into the child slot `slot` (0 left, 1 right) of node p
__device__ __forceinline__ void store_child_box(float4* nodes, int32_t p, int slot,
                                                const float lo[3], const float hi[3]) {
  float* f = reinterpret_cast<float*>(nodes + 4 * (int64_t)p);
  if (slot == 0) {
    f[0] = lo[0]; f[1] = hi[0]; f[2] = lo[1]; f[3] = hi[1];
    f[8] = lo[2]; f[9] = hi[2];
  } else {
    f[4] = lo[0]; f[5] = hi[0]; f[6] = lo[1]; f[7] = hi[1];
    f[10] = lo[2]; f[11] = hi[2];
  }
}

constexpr int kRefitThreads = 256;

__global__ void __launch_bounds__(kRefitThreads)
k_refit(const float* sph, const float* tri, uint32_t ns, uint32_t n, bool wide, const uint64_t* keys,
        float4* nodes, float4* prims, const int32_t* parent, const uint2* range, uint32_t* arrivals,
        uint32_t* err) {
  // a block's own nodes (all leaves in this block; node i lies in its own
  // range, so i - first leaf is a slot): arrival count and both children's boxes
  __shared__ uint32_t s_arrived[kRefitThreads];
  __shared__ float s_box[2][6][kRefitThreads];
  const uint32_t b0 = blockIdx.x * kRefitThreads, b1 = min(n, b0 + kRefitThreads) - 1;
  s_arrived[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t k = b0 + threadIdx.x;
  if (k >= n) return;
  const uint32_t id = (uint32_t)(keys[k] & 0xFFFFFFFFull);
  float lo[3], hi[3];
  if (id < ns) {
    const float* p = sph + 5ull * id;
    float r = p[3];
    uint32_t mat = __float_as_uint(p[4]);
    for (int a = 0; a < 3; ++a) {
      lo[a] = __double2float_rd(__dsub_rd((double)p[a], (double)r));
      hi[a] = __double2float_ru(__dadd_ru((double)p[a], (double)r));
    }
    prims[3ull * k + 0] = make_float4(p[0], p[1], p[2], __uint_as_float(id));
    prims[3ull * k + 1] = make_float4(r, 0.f, 0.f, __uint_as_float(mat));
    prims[3ull * k + 2] = make_float4(0.f, 0.f, 0.f, 0.f);
  } else {
    float v[9];
    load_tri(tri, id - ns, wide, v);
    uint32_t mat = __float_as_uint(tri[10ull * (id - ns) + 9]);
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(v[a], fminf(v[3 + a], v[6 + a]));
      hi[a] = fmaxf(v[a], fmaxf(v[3 + a], v[6 + a]));
    }
    prims[3ull * k + 0] = make_float4(v[0], v[1], v[2], __uint_as_float(id));
    prims[3ull * k + 1] = make_float4(v[3] - v[0], v[4] - v[1], v[5] - v[2], __uint_as_float(mat));
    prims[3ull * k + 2] = make_float4(v[6] - v[0], v[7] - v[1], v[8] - v[2], 0.f);
  }
  if (n == 1) {  // no internal node: keep the leaf box in the spare slot 0
    store_child_box(nodes, 0, 0, lo, hi);
    return;
  }
  int32_t child = ~(int32_t)k;
  int32_t p = parent[n - 1 + k];
  for (int step = 0; step < 130; ++step) {
    const float4 cd = __ldg(nodes + 4 * (int64_t)p + 3);      // written by k_karras
    const int slot = (__float_as_int(cd.x) == child) ? 0 : 1;
    const uint2 rg = __ldg(range + p);
    if (rg.x >= b0 && rg.y <= b1) {                  // this block's node
      const uint32_t s = (uint32_t)p - b0;
      for (int a = 0; a < 3; ++a) { s_box[slot][a][s] = lo[a]; s_box[slot][3 + a][s] = hi[a]; }
      __threadfence_block();
      if (atomicAdd(&s_arrived[s], 1u) == 0u) return;  // sibling not done yet
      __threadfence_block();
      float sl[3], sh[3];
      for (int a = 0; a < 3; ++a) { sl[a] = s_box[slot ^ 1][a][s]; sh[a] = s_box[slot ^ 1][3 + a][s]; }
      float4* o = nodes + 4 * (int64_t)p;
      if (slot == 0) {
        o[0] = make_float4(lo[0], hi[0], lo[1], hi[1]);
        o[1] = make_float4(sl[0], sh[0], sl[1], sh[1]);
        o[2] = make_float4(lo[2], hi[2], sl[2], sh[2]);
      } else {
        o[0] = make_float4(sl[0], sh[0], sl[1], sh[1]);
        o[1] = make_float4(lo[0], hi[0], lo[1], hi[1]);
        o[2] = make_float4(sl[2], sh[2], lo[2], hi[2]);
      }
      for (int a = 0; a < 3; ++a) { lo[a] = fminf(lo[a], sl[a]); hi[a] = fmaxf(hi[a], sh[a]); }
    } else {
      store_child_box(nodes, p, slot, lo, hi);
      __threadfence();
      if (atomicAdd(&arrivals[p], 1u) == 0u) return;   // sibling not done yet
      __threadfence();
      // both children are in: merge them into the box of p
      const float4 a = __ldcg(nodes + 4 * (int64_t)p + 0);
      const float4 b = __ldcg(nodes + 4 * (int64_t)p + 1);
      const float4 c = __ldcg(nodes + 4 * (int64_t)p + 2);
      lo[0] = fminf(a.x, b.x); hi[0] = fmaxf(a.y, b.y);
      lo[1] = fminf(a.z, b.z); hi[1] = fmaxf(a.w, b.w);
      lo[2] = fminf(c.x, c.z); hi[2] = fmaxf(c.y, c.w);
    }
    if (p == 0) return;                                // root reached
    child = p;
    p = parent[p];
  }
  atomicOr(err, ERR_BUILD);
}

// Raw primitive records word by word: spheres of 5 (centre, radius, material),
// triangles of 10 (vertices, material). Bound by the read.
__global__ void __launch_bounds__(256)
k_check_prims(const uint32_t* __restrict__ sph, const uint32_t* __restrict__ tri, uint64_t sph_words,
              uint64_t tri_words, uint32_t n_mats, uint32_t* __restrict__ bad) {
  const uint64_t step = (uint64_t)gridDim.x * blockDim.x, first = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool wrong = false;
  for (uint64_t i = first; i < sph_words; i += step) {
    const uint32_t v = sph[i], f = (uint32_t)(i % 5);
    if (f == 4) wrong |= v >= n_mats;
    else wrong |= (v & 0x7F800000u) == 0x7F800000u || (f == 3 && !(__uint_as_float(v) > 0.f));
  }
  for (uint64_t i = first; i < tri_words; i += step) {
    const uint32_t v = tri[i];
    wrong |= i % 10 == 9 ? v >= n_mats : (v & 0x7F800000u) == 0x7F800000u;
  }
  if (__any_sync(0xFFFFFFFFu, wrong) && (threadIdx.x & 31) == 0) *bad = 1;
}

}  // namespace

cudaError_t check_prims(const float4* d_sph_in, const float* d_tri_in, uint32_t ns, uint32_t nt, uint32_t n_mats,
                        uint32_t* bad, cudaStream_t st) {
  const uint64_t sph_words = 5ull * ns, tri_words = 10ull * nt;
  const uint64_t blocks = (std::max(sph_words, tri_words) + 255) / 256;
  k_check_prims<<<(int)std::min<uint64_t>(blocks, 8ull * (uint64_t)num_sms()), 256, 0, st>>>(
      reinterpret_cast<const uint32_t*>(d_sph_in), reinterpret_cast<const uint32_t*>(d_tri_in), sph_words,
      tri_words, n_mats, bad);
  return cudaGetLastError();
}

size_t lbvh_tmp_bytes(uint32_t n) {
  size_t nblocks = (n + kTile - 1) / kTile;
  size_t b = 0;
  b += kRedBlocks * sizeof(Bounds6);                         // bounds
  b += (size_t)n * 8 + 256;                                  // ping-pong keys, then the nodes' leaf ranges
  b += 256 * nblocks * 4 + 256;                              // histogram
  b += 256 * 4;                                              // digit totals
  b += (size_t)n * 4 + 256;                                  // arrival counters
  return b + 1024;
}

cudaError_t build_lbvh(const float4* d_sph_in, const float* d_tri_in, uint32_t ns, uint32_t nt,
                       float4* d_nodes, float4* d_prims, uint64_t* d_keys, int32_t* d_parent,
                       void* d_tmp, size_t tmp_bytes, uint32_t* d_err, cudaStream_t st) {
  const float* sph = reinterpret_cast<const float*>(d_sph_in);
  uint32_t n = ns + nt;
  if (tmp_bytes < lbvh_tmp_bytes(n)) return cudaErrorInvalidValue;
  int nblocks = (int)((n + kTile - 1) / kTile);
  char* t = reinterpret_cast<char*>(d_tmp);
  auto take = [&](size_t bytes) { char* p = t; t += (bytes + 255) & ~size_t(255); return p; };
  Bounds6* partial = reinterpret_cast<Bounds6*>(take(kRedBlocks * sizeof(Bounds6)));
  uint64_t* keys_b = reinterpret_cast<uint64_t*>(take((size_t)n * 8));
  uint32_t* hist = reinterpret_cast<uint32_t*>(take(256ull * nblocks * 4));
  uint32_t* totals = reinterpret_cast<uint32_t*>(take(256 * 4));
  uint32_t* arrivals = reinterpret_cast<uint32_t*>(take((size_t)n * 4));
  const bool wide = (reinterpret_cast<uintptr_t>(d_tri_in) & 7u) == 0;

  int red_grid = (int)std::min<uint32_t>((uint32_t)kRedBlocks, (n + kRedThreads - 1) / kRedThreads);
  k_centroid_bounds<<<red_grid, kRedThreads, 0, st>>>(sph, d_tri_in, ns, n, wide, partial);
  k_reduce_bounds<<<1, 192, 0, st>>>(partial, red_grid);
  k_keys<<<nblocks, kSortThreads, 0, st>>>(sph, d_tri_in, ns, n, wide, partial, d_keys, hist, nblocks);
  uint64_t* a = d_keys;
  uint64_t* b = keys_b;
  for (int shift = 32; shift < 64; shift += 8) {
    if (shift > 32) k_hist<<<nblocks, kSortThreads, 0, st>>>(a, n, shift, hist, nblocks);
    k_scan<<<256, 256, 0, st>>>(hist, nblocks, totals);
    k_scatter<<<nblocks, kSortThreads, 0, st>>>(a, b, n, shift, hist, nblocks, totals);
    uint64_t* x = a; a = b; b = x;
  }
  // four passes: the sorted keys are back in d_keys, and keys_b is free
  uint2* range = reinterpret_cast<uint2*>(keys_b);
  if (n > 1) {
    k_karras<<<(n - 1 + 255) / 256, 256, 0, st>>>(d_keys, n, d_nodes, d_parent, range);
    cudaMemsetAsync(arrivals, 0, (size_t)n * 4, st);
  } else {
    cudaMemsetAsync(d_parent, 0xFF, 4, st);
  }
  k_refit<<<(n + kRefitThreads - 1) / kRefitThreads, kRefitThreads, 0, st>>>(
      sph, d_tri_in, ns, n, wide, d_keys, d_nodes, d_prims, d_parent, range, arrivals, d_err);
  return cudaGetLastError();
}

}  // namespace rt
