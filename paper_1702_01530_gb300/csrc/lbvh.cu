// Linear BVH build on the GPU (sm_103a).
//
// Table 1 of the paper names BVH trees as the GPU-friendly acceleration
// structure; this is the linear BVH over Morton codes:
//   1. k_centroid_bounds : FP64 centroids (triangle ((v0+v1)+v2)/3, every
//      operation correctly rounded, no FMA), their per-axis min/max per block.
//      Triangles are compared by their sums (division by 3 is monotonic).
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
//   5. k_tree              : primitives in sorted order with their boxes
//      (triangle min/max; sphere c -/+ r in FP64 rounded outward to FP32) and
//      the binary radix tree with its boxes over every 256 of them, bottom-up in
//      shared memory.
//   6. k_tree_up           : the same over what 16 such blocks leave over, and so
//      on until one block is left.
//
// Measured (GB300, 1,000,000 primitives in random order, the whole device-side
// build): 0.267 ms (0.30 when each launch waited for the kernel before it to
// end). 1.110 when one block scanned the tile counts (0.40), one thread reduced
// the bounds (0.12), every key was divided twice in FP64 (0.27 with the bounds)
// and every node had a global arrival counter (0.18); 0.359 with a search per
// node (38 us) and a refit that read its parents, children and ranges from
// memory at every step (125 us). Its kernels' shares now: tree 77 us, upper
// levels 15 each, scatter 4 x 13, bounds 25, keys 23, histograms 3 x 5, scans
// 4 x 3. What is left in k_tree is the chain of a block's climb, seven to ten
// levels of shared-memory exchanges.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "rt_internal.cuh"

namespace rt {
namespace {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;                       // items per thread per tile
constexpr int kTile = kSortThreads * kSortItems;    // 2048 keys per block
constexpr int kRedThreads = 512;
constexpr int kRedBlocks = 256;

struct Bounds6 { double lo[3], hi[3]; };

// Words of the raw records. FIRST: the first kernel of a build, which may overlap
// the one that writes them, so ordinary loads; complete for the later ones.
template <bool FIRST, typename T>
__device__ __forceinline__ T raw(const T* p) {
  if (FIRST) return *p;
  return __ldg(p);
}

// triangle i of 10-word records; `wide`: the array is 8-byte aligned
template <bool FIRST = false>
__device__ __forceinline__ void load_tri(const float* t, uint32_t i, bool wide, float v[9]) {
  const float* p = t + 10ull * i;
  if (wide) {
    const float2* q = reinterpret_cast<const float2*>(p);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 x = raw<FIRST>(q + k);
      v[2 * k] = x.x;
      v[2 * k + 1] = x.y;
    }
    v[8] = raw<FIRST>(p + 8);
  } else {
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = raw<FIRST>(p + k);
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

// Per-block partial min/max of the centroids; spheres by their centres,
// triangles by the sums of their vertices, divided by 3 at the end. FP64 has few
// units, so FP32 sums with a bound of their error (two roundings, each at most
// 2^-24 of the vertices' magnitudes) first find which triangles can hold an
// extreme of the block's range; only their sums are formed in FP64 (1M triangles:
// 25 us; 38 with every sum in FP64).
__device__ __forceinline__ void sum_range(const float v[9], int k, float& least, float& most) {
  const float f = (v[k] + v[3 + k]) + v[6 + k];
  const float e = 0x1p-22f * (fabsf(v[k]) + fabsf(v[3 + k]) + fabsf(v[6 + k])) + 1e-44f;
  least = f - e;
  most = f + e;
}

__global__ void __launch_bounds__(kRedThreads)
k_centroid_bounds(const float* sph, const float* tri, uint32_t ns, uint32_t n, bool wide, Bounds6* partial) {
  after_previous();
  __shared__ float s_f[12][kRedThreads / 32];      // sphere min, -max; triangle: upper bound of the min, of -max
  __shared__ long long s_d[6][kRedThreads / 32];   // triangle min, ~max
  const long long kMost = 0x7FFFFFFFFFFFFFFFll;
  const uint32_t first = blockIdx.x * kRedThreads + threadIdx.x, step = gridDim.x * kRedThreads;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float f[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) f[k] = INFINITY;
  uint32_t i = first;
  for (; i < ns && i < n; i += step)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float c = raw<true>(sph + 5ull * i + k);
      f[k] = fminf(f[k], c);
      f[3 + k] = fminf(f[3 + k], -c);
    }
  const uint32_t first_tri = i;
  for (; i < n; i += step) {
    float t[9];
    load_tri<true>(tri, i - ns, wide, t);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float least, most;
      sum_range(t, k, least, most);
      f[6 + k] = fminf(f[6 + k], most);
      f[9 + k] = fminf(f[9 + k], -least);
    }
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    for (int off = 16; off > 0; off >>= 1) f[k] = fminf(f[k], __shfl_xor_sync(0xFFFFFFFFu, f[k], off));
    if (lane == 0) s_f[k][warp] = f[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 12; ++k)
    for (int w = 0; w < kRedThreads / 32; ++w) f[k] = fminf(f[k], s_f[k][w]);
  long long v[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) v[k] = kMost;
  for (i = first_tri; i < n; i += step) {
    float t[9];
    load_tri<true>(tri, i - ns, wide, t);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float least, most;
      sum_range(t, k, least, most);
      if (!(least > f[6 + k]) || !(-most > f[9 + k])) {      // also what overflows FP32
        const long long o = d2o(sum3(t, k));
        v[k] = min(v[k], o);
        v[3 + k] = min(v[3 + k], ~o);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    for (int off = 16; off > 0; off >>= 1) v[k] = min(v[k], __shfl_xor_sync(0xFFFFFFFFu, v[k], off));
    if (lane == 0) s_d[k][warp] = v[k];
  }
  __syncthreads();
  if (threadIdx.x >= 3) return;
  const int a = threadIdx.x;
  long long least = kMost, most = kMost;
  float c0 = INFINITY, c1 = INFINITY;
  for (int w = 0; w < kRedThreads / 32; ++w) {
    least = min(least, s_d[a][w]);
    most = min(most, s_d[3 + a][w]);
    c0 = fminf(c0, s_f[a][w]);
    c1 = fminf(c1, s_f[3 + a][w]);
  }
  double lo = (double)c0, hi = -(double)c1;
  if (least != kMost) {
    lo = fmin(lo, __ddiv_rn(o2d(least), 3.0));
    hi = fmax(hi, __ddiv_rn(o2d(~most), 3.0));
  }
  partial[blockIdx.x].lo[a] = lo;
  partial[blockIdx.x].hi[a] = hi;
}

// bounds of all blocks: warp q takes value q (lo x, y, z, hi x, y, z)
__global__ void k_reduce_bounds(Bounds6* partial, int nparts) {
  after_previous();
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
  after_previous();
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
      for (int k = 0; k < 3; ++k) v[k] = v[3 + k] = v[6 + k] = raw<false>(sph + 5ull * i + k);
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
  after_previous();
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
  after_previous();
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
  after_previous();
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

// box of the primitive with raw index id
__device__ __forceinline__ void prim_box(const float* sph, const float v[9], uint32_t ns, uint32_t id, float lo[3],
                                         float hi[3]) {
  if (id < ns) {
    const float* p = sph + 5ull * id;
    const float r = p[3];
    for (int a = 0; a < 3; ++a) {
      lo[a] = __double2float_rd(__dsub_rd((double)p[a], (double)r));
      hi[a] = __double2float_ru(__dadd_ru((double)p[a], (double)r));
    }
  } else {
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(v[a], fminf(v[3 + a], v[6 + a]));
      hi[a] = fmaxf(v[a], fmaxf(v[3 + a], v[6 + a]));
    }
  }
}

// The tree is found bottom-up, without searches (Apetrei 2014): of a range's two
// neighbours the one with the longer common prefix is its sibling's side; the
// second of two siblings to arrive at their split makes the parent, whose number
// is the end of its range that faces its own sibling (Karras' numbering; the root
// is 0). A block does this in shared memory for a run of items, which cover a
// range of leaves: first 256 leaves, then the subtrees that kUpGroup such runs
// leave over, and so on until one run is left. Prefix and suffix minima of the
// run's deltas tell whether a sibling's range ends inside the run; a subtree whose
// sibling's does not is left over. What a run leaves over hangs off the two paths
// of nodes that contain one of its ends, which are at most one per bit of the
// keys: at most 128.
template <int N>
struct Run {
  int delta[N + 1];                    // [j]: of the leaves on either side of boundary j, before item j
  int pre[N + 1], suf[N + 2];          // minima up to and from j
  uint32_t arrived[N + 1], far[2][N + 1];   // at a split: arrivals, and the sides' other ends
  float box[2][6][N + 1];              // and their boxes
};

// minima of r.delta[0 .. m] from either end, by the whole block
template <int N, int THREADS>
__device__ __forceinline__ void run_minima(Run<N>& r, int m, int (*s_warp)[THREADS / 32]) {
  constexpr int kPer = (N + 1 + THREADS - 1) / THREADS;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, j0 = tid * kPer;
  int pre = 64, suf = 64;
  for (int j = j0; j < j0 + kPer && j <= m; ++j) pre = min(pre, r.delta[j]);
  suf = pre;
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xFFFFFFFFu, pre, o), y = __shfl_down_sync(0xFFFFFFFFu, suf, o);
    if (lane >= o) pre = min(pre, x);
    if (lane + o < 32) suf = min(suf, y);
  }
  if (lane == 31) s_warp[0][warp] = pre;
  if (lane == 0) s_warp[1][warp] = suf;
  // of the threads before (after) this one alone
  pre = __shfl_up_sync(0xFFFFFFFFu, pre, 1);
  suf = __shfl_down_sync(0xFFFFFFFFu, suf, 1);
  if (lane == 0) pre = 64;
  if (lane == 31) suf = 64;
  __syncthreads();
  for (int w = 0; w < THREADS / 32; ++w) {
    if (w < warp) pre = min(pre, s_warp[0][w]);
    if (w > warp) suf = min(suf, s_warp[1][w]);
  }
  for (int j = j0; j < j0 + kPer && j <= m; ++j) r.pre[j] = pre = min(pre, r.delta[j]);
  for (int j = j0 + kPer - 1; j >= j0; --j)
    if (j <= m) r.suf[j] = suf = min(suf, r.delta[j]);
  if (tid == 0) r.suf[m + 1] = 64;     // past the last boundary: above every delta
}

// Climb from item i of a run of m items with box (lo, hi). first(j) is the
// first leaf of item j (first(m): past the run). Returns whether the climb ended
// at a subtree that is left over: then l is its first item and child its number.
template <int N, typename First>
__device__ __forceinline__ bool run_climb(Run<N>& run, const First& first, int i, int m, int32_t item, float lo[3],
                                          float hi[3], float4* nodes, int32_t* parent, uint32_t n, int& l,
                                          int32_t& child) {
  int r = i;
  l = i;
  child = item;
  for (int step = 0; step <= m; ++step) {
    const int dl = run.delta[l], dr = run.delta[r + 1];
    if (dl < 0 && dr < 0) {                            // all leaves: the root
      parent[0] = -1;
      return false;
    }
    const bool is_left = dr > dl;
    const int q = is_left ? r + 1 : l;                 // the split: a boundary inside the run if the parent is
    if (!(is_left ? run.suf[q + 1] < dr : q > 0 && run.pre[q - 1] < dl)) return true;
    const int side = is_left ? 0 : 1;
    for (int a = 0; a < 3; ++a) { run.box[side][a][q] = lo[a]; run.box[side][3 + a][q] = hi[a]; }
    run.far[side][q] = (uint32_t)(is_left ? l : r);
    __threadfence_block();
    if (atomicAdd(&run.arrived[q], 1u) == 0u) return false;   // sibling not done yet
    __threadfence_block();
    float sl[3], sh[3];
    for (int a = 0; a < 3; ++a) { sl[a] = run.box[side ^ 1][a][q]; sh[a] = run.box[side ^ 1][3 + a][q]; }
    if (is_left) r = (int)run.far[1][q]; else l = (int)run.far[0][q];
    const uint32_t begin = first(l), split = first(q), end = first(r + 1);   // leaves [begin, split) and [split, end)
    const int32_t left = split - begin == 1 ? ~(int32_t)begin : (int32_t)(split - 1);
    const int32_t right = end - split == 1 ? ~(int32_t)split : (int32_t)split;
    child = (int32_t)(run.delta[r + 1] > run.delta[l] ? end - 1 : begin);
    float4* o = nodes + 4 * (int64_t)child;
    o[0] = is_left ? make_float4(lo[0], hi[0], lo[1], hi[1]) : make_float4(sl[0], sh[0], sl[1], sh[1]);
    o[1] = is_left ? make_float4(sl[0], sh[0], sl[1], sh[1]) : make_float4(lo[0], hi[0], lo[1], hi[1]);
    o[2] = is_left ? make_float4(lo[2], hi[2], sl[2], sh[2]) : make_float4(sl[2], sh[2], lo[2], hi[2]);
    o[3] = make_float4(__int_as_float(left), __int_as_float(right), 0.f, 0.f);
    parent[left >= 0 ? left : (int64_t)n - 1 + ~left] = child;
    parent[right >= 0 ? right : (int64_t)n - 1 + ~right] = child;
    for (int a = 0; a < 3; ++a) { lo[a] = fminf(lo[a], sl[a]); hi[a] = fmaxf(hi[a], sh[a]); }
  }
  return false;
}

// the primitives in sorted order, and the trees over every 256 of them
constexpr int kTreeThreads = 256;
__global__ void __launch_bounds__(kTreeThreads, 6)
k_tree(const float* sph, const float* tri, uint32_t ns, uint32_t n, bool wide, const uint64_t* keys,
       float4* nodes, float4* prims, int32_t* parent, uint2* left_over, uint32_t* counts) {
  after_previous();
  __shared__ union {
    float4 prim[3 * kTreeThreads];
    Run<kTreeThreads> run;
  } u;
  __shared__ int s_warp[2][kTreeThreads / 32];
  __shared__ int32_t s_left[kTreeThreads];             // by first leaf: what is left over
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t b0 = blockIdx.x * kTreeThreads, m = min((uint32_t)kTreeThreads, n - b0), k = b0 + tid;
  const bool leaf = (uint32_t)tid < m;
  constexpr int32_t kNone = 0x7FFFFFFF;

  // primitives: gathered, then written whole lines at a time
  float lo[3] = {0.f, 0.f, 0.f}, hi[3] = {0.f, 0.f, 0.f};
  if (leaf) {
    const uint32_t id = (uint32_t)(keys[k] & 0xFFFFFFFFull);
    float v[9];
    if (id < ns) {
      const float* p = sph + 5ull * id;
      u.prim[3 * tid] = make_float4(p[0], p[1], p[2], __uint_as_float(id));
      u.prim[3 * tid + 1] = make_float4(p[3], 0.f, 0.f, p[4]);
      u.prim[3 * tid + 2] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      load_tri(tri, id - ns, wide, v);
      const float mat = tri[10ull * (id - ns) + 9];
      u.prim[3 * tid] = make_float4(v[0], v[1], v[2], __uint_as_float(id));
      u.prim[3 * tid + 1] = make_float4(v[3] - v[0], v[4] - v[1], v[5] - v[2], mat);
      u.prim[3 * tid + 2] = make_float4(v[6] - v[0], v[7] - v[1], v[8] - v[2], 0.f);
    }
    prim_box(sph, v, ns, id, lo, hi);
  }
  const int d = leaf ? delta(keys, n, (int64_t)k, (int64_t)k - 1) : -1;
  __syncthreads();
  for (uint32_t i = tid; i < 3 * m; i += kTreeThreads) prims[3ull * b0 + i] = u.prim[i];
  if (n == 1) {                                        // no internal node: keep the leaf box in the spare slot 0
    if (tid == 0) store_child_box(nodes, 0, 0, lo, hi);
    return;
  }
  __syncthreads();
  s_left[tid] = kNone;
  u.run.arrived[tid] = 0;
  if (leaf) u.run.delta[tid] = d;
  if (tid == 0) {
    u.run.arrived[kTreeThreads] = 0;
    u.run.delta[m] = delta(keys, n, (int64_t)b0 + m - 1, (int64_t)b0 + m);
  }
  __syncthreads();
  run_minima<kTreeThreads, kTreeThreads>(u.run, (int)m, s_warp);
  __syncthreads();
  if (leaf) {
    int l;
    int32_t child;
    if (run_climb(u.run, [&](int j) { return b0 + (uint32_t)j; }, tid, (int)m, ~(int32_t)k, lo, hi, nodes, parent, n,
                  l, child))
      s_left[l] = child;
  }
  __syncthreads();
  const int32_t mine = s_left[tid];
  const uint32_t ball = __ballot_sync(0xFFFFFFFFu, mine != kNone);
  if (lane == 0) s_warp[0][warp] = __popc(ball);
  __syncthreads();
  uint32_t at = __popc(ball & ((1u << lane) - 1u)), total = 0;
  for (int w = 0; w < kTreeThreads / 32; ++w) {
    if (w < warp) at += s_warp[0][w];
    total += s_warp[0][w];
  }
  if (mine != kNone) left_over[b0 + at] = make_uint2((uint32_t)mine, k);
  if (tid == 0) counts[blockIdx.x] = total;
}

// The trees over what kUpGroup runs left over (runs of `span` leaves each; run
// j's list begins at left_over[j span]); what these leave over begins at their
// first run's list.
constexpr int kUpThreads = 512, kUpGroup = 16, kUpItems = kUpGroup * 128;
struct UpShared {
  Run<kUpItems> run;
  uint32_t first[kUpItems + 1];
  int32_t num[kUpItems], left[kUpItems];   // items; by first item: what is left over
  int warp[2][kUpThreads / 32];
  uint32_t base[kUpGroup + 1];
};
__global__ void __launch_bounds__(kUpThreads)
k_tree_up(const float* sph, const float* tri, uint32_t ns, uint32_t n, bool wide, const uint64_t* keys,
          float4* nodes, int32_t* parent, uint2* left_over, const uint32_t* counts, uint32_t runs,
          uint64_t span, uint32_t* counts_out, uint32_t* err) {
  after_previous();
  extern __shared__ __align__(16) unsigned char up_smem[];
  UpShared& s = *reinterpret_cast<UpShared*>(up_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t r0 = blockIdx.x * kUpGroup, r1 = min(runs, r0 + kUpGroup);
  constexpr int32_t kNone = 0x7FFFFFFF;
  if (warp == 0) {
    const uint32_t c = r0 + lane < r1 ? counts[r0 + lane] : 0u;
    uint32_t sum = c;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, sum, o);
      if (lane >= o) sum += x;
    }
    if (lane <= kUpGroup) s.base[lane] = sum - c;
  }
  __syncthreads();
  const uint32_t m = s.base[kUpGroup];
  if (m > (uint32_t)kUpItems || m == 0) {              // cannot happen (see above)
    if (tid == 0) { atomicOr(err, ERR_BUILD); counts_out[blockIdx.x] = 0; }
    return;
  }
  const uint64_t begin = r0 * span, end = min((uint64_t)n, begin + kUpGroup * span);
  auto item = [&](uint32_t i) {                        // (number, first leaf) of item i
    uint32_t g = 0;
    while (g + 1 < kUpGroup && s.base[g + 1] <= i) ++g;
    return left_over[(r0 + g) * span + (i - s.base[g])];
  };
  for (uint32_t i = tid; i < m; i += kUpThreads) {
    const uint2 x = item(i);
    s.first[i] = x.y;
    s.num[i] = (int32_t)x.x;
    s.left[i] = kNone;
    s.run.delta[i] = delta(keys, n, (int64_t)x.y, (int64_t)x.y - 1);
    s.run.arrived[i] = 0;
  }
  if (tid == 0) {
    s.first[m] = (uint32_t)end;
    s.run.delta[m] = delta(keys, n, (int64_t)end - 1, (int64_t)end);
    s.run.arrived[m] = 0;
  }
  __syncthreads();
  run_minima<kUpItems, kUpThreads>(s.run, (int)m, s.warp);
  __syncthreads();
  for (uint32_t i = tid; i < m; i += kUpThreads) {
    const int32_t num = s.num[i];
    float lo[3], hi[3];
    if (num < 0) {
      const uint32_t id = (uint32_t)(keys[~num] & 0xFFFFFFFFull);
      float v[9];
      if (id >= ns) load_tri(tri, id - ns, wide, v);
      prim_box(sph, v, ns, id, lo, hi);
    } else {
      const float4 a = nodes[4 * (int64_t)num], b = nodes[4 * (int64_t)num + 1], c = nodes[4 * (int64_t)num + 2];
      lo[0] = fminf(a.x, b.x); hi[0] = fmaxf(a.y, b.y);
      lo[1] = fminf(a.z, b.z); hi[1] = fmaxf(a.w, b.w);
      lo[2] = fminf(c.x, c.z); hi[2] = fmaxf(c.y, c.w);
    }
    int l;
    int32_t child;
    if (run_climb(s.run, [&](int j) { return s.first[j]; }, (int)i, (int)m, num, lo, hi, nodes, parent, n, l, child))
      s.left[l] = child;
  }
  __syncthreads();
  uint32_t total = 0;
  for (uint32_t base = 0; base < m; base += kUpThreads) {
    const uint32_t i = base + tid;
    const int32_t mine = i < m ? s.left[i] : kNone;
    const uint32_t ball = __ballot_sync(0xFFFFFFFFu, mine != kNone);
    if (lane == 0) s.warp[0][warp] = __popc(ball);
    __syncthreads();
    uint32_t at = total + __popc(ball & ((1u << lane) - 1u));
    for (int w = 0; w < kUpThreads / 32; ++w) {
      if (w < warp) at += s.warp[0][w];
      total += s.warp[0][w];
    }
    if (mine != kNone) left_over[begin + at] = make_uint2((uint32_t)mine, s.first[i]);
    __syncthreads();
  }
  if (tid == 0) counts_out[blockIdx.x] = total;
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
  b += (size_t)n * 8 + 256;                                  // ping-pong keys, then what the runs leave over
  b += 256 * nblocks * 4 + 256;                              // histogram
  b += 256 * 4;                                              // digit totals
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
  const bool wide = (reinterpret_cast<uintptr_t>(d_tri_in) & 7u) == 0;

  int red_grid = (int)std::min<uint32_t>((uint32_t)kRedBlocks, (n + kRedThreads - 1) / kRedThreads);
  Chain chain{st};
  chain.then(k_centroid_bounds, red_grid, kRedThreads, 0, sph, d_tri_in, ns, n, wide, partial);
  chain.then(k_reduce_bounds, 1, 192, 0, partial, red_grid);
  chain.then(k_keys, nblocks, kSortThreads, 0, sph, d_tri_in, ns, n, wide, partial, d_keys, hist, nblocks);
  uint64_t* a = d_keys;
  uint64_t* b = keys_b;
  for (int shift = 32; shift < 64; shift += 8) {
    if (shift > 32) chain.then(k_hist, nblocks, kSortThreads, 0, a, n, shift, hist, nblocks);
    chain.then(k_scan, 256, 256, 0, hist, nblocks, totals);
    chain.then(k_scatter, nblocks, kSortThreads, 0, a, b, n, shift, hist, nblocks, totals);
    uint64_t* x = a; a = b; b = x;
  }
  // four passes: the sorted keys are back in d_keys; keys_b holds what the runs leave over, the
  // histograms their counts
  uint2* left_over = reinterpret_cast<uint2*>(keys_b);
  if (n == 1 && chain.error == cudaSuccess) chain.error = cudaMemsetAsync(d_parent, 0xFF, 4, st);
  uint32_t runs = (uint32_t)(((uint64_t)n + kTreeThreads - 1) / kTreeThreads);
  chain.then(k_tree, runs, kTreeThreads, 0, sph, d_tri_in, ns, n, wide, d_keys, d_nodes, d_prims, d_parent,
             left_over, hist);
  if (runs > 1) {
    // an attribute of the current device: set on every call
    const cudaError_t e = cudaFuncSetAttribute(k_tree_up, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(UpShared));
    if (chain.error == cudaSuccess) chain.error = e;
  }
  uint32_t* counts = hist;
  for (uint64_t span = kTreeThreads; runs > 1; span *= kUpGroup) {
    const uint32_t groups = (runs + kUpGroup - 1) / kUpGroup;
    chain.then(k_tree_up, groups, kUpThreads, sizeof(UpShared), sph, d_tri_in, ns, n, wide, d_keys, d_nodes,
               d_parent, left_over, counts, runs, span, counts + runs, d_err);
    counts += runs;
    runs = groups;
  }
  return chain.end();
}

}  // namespace rt
