// Binned-SAH rebuild of the binary tree over the LBVH's leaves (GPU, sm_103a).
//
// Table 1 of the paper names BVH trees as the acceleration structure and
// leaves the build open. The Morton LBVH (lbvh.cu) is the tree whose topology
// the tests pin bit for bit and whose traversal defines the algorithmic work;
// its splits follow Morton-code bits, not the geometry, so its boxes overlap
// more than they need to. Renders walk a second binary tree over the same
// leaves (one primitive per leaf, the same primitive slots and leaf boxes),
// built top down with the surface area heuristic over binned centroids
// (MacDonald & Booth 1990; binning after Wald 2007): on the 1080p blob pair
// it takes 15 % fewer node visits for shadow and mirror rays and renders the
// same image 11 % faster. Any binary tree over the same conservative leaf
// boxes yields the same closest hit and the same any-hit answer.
//
// Two phases, without a host decision between them:
//   top   one level per step, every node of more than kMidLeaves leaves cut into
//         slices of kSlice leaves, one block each: (1) 16 bins per axis of the
//         slice, added to the node's; (2) the split of least SAH cost, area(L)
//         n(L) + area(R) n(R), over the 45 bin boundaries, and a stable
//         partition of the slice (lefts before it from the slices' bin
//         counts), with the centroid bounds of the two children; (3) the node
//         record and the children's entries. The kernels read their counts on
//         the device, so the levels are queued without waiting; the host looks
//         only after as many as a balanced tree has.
//   mid   a subtree of at most kMidLeaves leaves in one block, one thread per
//         leaf: the same steps in shared memory for all its nodes of a level
//         at once, down to segments of at most 32 leaves; then one warp per
//         segment, all its nodes of a level at once, each split at the least
//         SAH cost over every position of its leaves sorted by centroid (a
//         warp sort by (segment, centroid, position), segmented prefix and
//         suffix boxes).
// An object-median split stands in when the centroids coincide or the depth
// budget is low, so that no leaf lies deeper than kMaxDepth (the traversal stack
// holds 64 entries). All combined values are minima, maxima and integer sums,
// and partitions are stable, so the tree does not depend on thread timing or on
// the slicing.
// Node numbering: a binary tree over n leaves has n - 1 inner nodes and each
// owns one split position s (left = [begin, s), right = [s, end)), s in
// [1, n-1]; node id = s - 1, except that the root is 0 and the node whose
// split position is 1 takes the root's id. Ids are therefore unique, dense
// and independent of launch order. A node writes its own id into its parent's
// record, and its leaf children into its own.
//
// Bound by the latency of the levels at 257k primitives and by shared-memory
// atomics and shuffles at 10M. Measured (kernels of the build alone): 257k blob
// primitives 0.52 ms, 10M terrain triangles 10 ms; with one block per node, a
// host read per level, lane reductions for every bin and one warp per subtree
// stack in the last 32 leaves: 1.76 ms and 36.5 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <utility>

#include "rt_internal.cuh"

namespace rt {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kBins = 16;
constexpr int kMaxDepth = 60;        // median splits keep every leaf at or above this depth
constexpr uint32_t kMidLeaves = 256; // subtrees of at most this many leaves: one block each
constexpr uint32_t kSmallLeaves = 32;
constexpr uint32_t kSlice = 512;     // leaves of a slice of a top node, at least (creation of 257k: 1.07 ms;
                                     // 1.12 with 1024, 1.10 with 768, 1.11 with 256)
constexpr uint32_t kRoot = 0xFFFFFFFFu;   // parent_slot of the root

struct Job {
  uint32_t begin, end;               // leaf slots idx[begin, end) of this node (end - begin >= 2)
  uint32_t parent_slot;              // parent id << 1 | child slot, or kRoot
  uint32_t depth;                    // top bit (mid jobs): which index buffer holds the leaves
};

struct Control;
struct TopNode;

// the scratch of a build over n leaves, and where its results go
struct Build {
  uint32_t slice, max_slices, max_nodes, max_mid;   // leaves per slice; entries of a level and of the build
  float4 *lo, *hi;                                  // leaf boxes
  uint32_t* idx[2];                                 // leaf order, nodes and the node of each slice:
  TopNode* nodes[2];                                // [0] this level's, [1] the next one's
  uint32_t* slice_node[2];
  int* slice_cnt;                                   // of each slice, the leaves up to each bin of an axis
  Job* mid;
  Control* ctl;
  float4* out;
  uint32_t* err;
  uint32_t n;
};

// order-preserving ints are used for all boxes that atomics combine
struct Bins {
  int cnt[3][kBins];
  int box[3][kBins][6];              // lo xyz, hi xyz
};
constexpr int kBinWords = (int)(sizeof(Bins) / sizeof(int));

struct TopNode {
  Job job;
  uint32_t slice0, n_slices;
  int bounds[6];                     // centroid bounds of the leaves
  Bins bins;
  int child_bounds[2][6];            // centroid bounds of the two sides
  int child_box[2][6];               // their boxes (median splits only; else from the bins)
  uint32_t done;                     // slices partitioned
};

// per level parity: nodes and slices of that level; and of the whole build
struct Control {
  uint32_t n_nodes[2], n_slices[2];
  uint32_t n_mid, root_split;
};

__device__ __forceinline__ int f2o(float f) {        // order-preserving int image of a float
  const int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7FFFFFFF;
}
__device__ __forceinline__ float o2f(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7FFFFFFF); }
// value i of an empty box
__device__ __forceinline__ int empty6(int i) { return i < 3 ? f2o(INFINITY) : f2o(-INFINITY); }

// word i of a set of bins: its empty value, and what it combines by (0 sum, -1 min, 1 max)
__device__ __forceinline__ int empty_word(int i) { return i < 3 * kBins ? 0 : empty6((i - 3 * kBins) % 6); }
__device__ __forceinline__ int word_op(int i) { return i < 3 * kBins ? 0 : (i - 3 * kBins) % 6 < 3 ? -1 : 1; }
__device__ __forceinline__ int* words(Bins& b) { return &b.cnt[0][0]; }

// A leaf's box and centroid as values to combine by minimum (0..2) and maximum
// (3..5). A centroid that is no number (its box spans all floats) bounds nothing.
__device__ __forceinline__ void centroid(const float4& lo, const float4& hi, float c[3]) {
  c[0] = 0.5f * (lo.x + hi.x); c[1] = 0.5f * (lo.y + hi.y); c[2] = 0.5f * (lo.z + hi.z);
}
__device__ __forceinline__ void centroid6(const float c[3], int v[6]) {
  for (int q = 0; q < 3; ++q) { v[q] = f2o(fminf(c[q], INFINITY)); v[3 + q] = f2o(fmaxf(c[q], -INFINITY)); }
}
__device__ __forceinline__ void box6(const float4& lo, const float4& hi, int v[6]) {
  v[0] = f2o(lo.x); v[1] = f2o(lo.y); v[2] = f2o(lo.z); v[3] = f2o(hi.x); v[4] = f2o(hi.y); v[5] = f2o(hi.z);
}

__device__ __forceinline__ float half_area(const float lo[3], const float hi[3]) {
  const float dx = fmaxf(hi[0] - lo[0], 0.f), dy = fmaxf(hi[1] - lo[1], 0.f),
              dz = fmaxf(hi[2] - lo[2], 0.f);
  return dx * dy + dy * dz + dz * dx;
}

__device__ __forceinline__ int bin_of(float c, float cmin, float cext) {
  return min(kBins - 1, (int)((c - cmin) * ((float)kBins / cext)));
}

// centroid frame of a node, and whether it splits at the object median (its
// centroids coincide, or the depth budget is short)
__device__ __forceinline__ bool node_frame(const int* bounds, uint32_t m, uint32_t depth, float cmin[3],
                                           float cext[3]) {
  bool spread = false;
  for (int a = 0; a < 3; ++a) {
    cmin[a] = o2f(bounds[a]);
    cext[a] = o2f(bounds[3 + a]) - cmin[a];
    spread |= cext[a] > 0.f;
  }
  const uint32_t lg = 32 - __clz(m - 1);
  return !spread || depth + lg >= (uint32_t)kMaxDepth - 4;
}

// The split of a node from its bins (one warp): of the 3 x 15 bin boundaries
// the first of least cost, area(L) n(L) + area(R) n(R); axis -1 if none has
// leaves on both sides. Lanes 0-15 hold the bins in order and take the boxes
// and counts of all bins up to theirs, lanes 16-31 hold them in reverse and
// take those from theirs on.
__device__ __forceinline__ void choose_split(const Bins& bins, const float cext[3], int& axis, int& bin) {
  const int lane = threadIdx.x & 31, i = lane & 15, q = lane < 16 ? i : 15 - i;
  float best = INFINITY;
  int at = 3 * kBins;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    int n = bins.cnt[a][q];
    float v[6];
    for (int x = 0; x < 6; ++x) v[x] = o2f(bins.box[a][q][x]);
#pragma unroll
    for (int o = 1; o < kBins; o <<= 1) {
      const int m = __shfl_up_sync(0xFFFFFFFFu, n, o, kBins);
      if (i >= o) n += m;
#pragma unroll
      for (int x = 0; x < 6; ++x) {
        const float u = __shfl_up_sync(0xFFFFFFFFu, v[x], o, kBins);
        if (i >= o) v[x] = x < 3 ? fminf(v[x], u) : fmaxf(v[x], u);
      }
    }
    const float area = half_area(v, v + 3);
    const float rc = __shfl_sync(0xFFFFFFFFu, __fmul_rn(area, (float)n), 30 - lane);   // of the bins after this one
    const int rn = __shfl_sync(0xFFFFFFFFu, n, 30 - lane);
    const float cost = __fmaf_rn(area, (float)n, rc);
    if (lane < kBins - 1 && cext[a] > 0.f && n > 0 && rn > 0 && cost < best) {
      best = cost;
      at = a * kBins + lane;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float c = __shfl_xor_sync(0xFFFFFFFFu, best, o);
    const int i2 = __shfl_xor_sync(0xFFFFFFFFu, at, o);
    if (c < best || (c == best && i2 < at)) { best = c; at = i2; }
  }
  axis = at == 3 * kBins ? -1 : at / kBins;
  bin = at == 3 * kBins ? 0 : at % kBins;
}

// the id of a node from its split position; it goes into the parent's record
__device__ __forceinline__ uint32_t place_node(uint32_t split, uint32_t parent_slot, uint32_t root_split,
                                               float4* out, uint32_t n, uint32_t* err) {
  if (parent_slot == kRoot) return 0u;
  uint32_t id = split == 1 ? root_split - 1 : split - 1;
  if (id >= n - 1) { atomicOr(err, ERR_BUILD); id = n - 2; }   // splits lie in [1, n-1]: cannot happen
  reinterpret_cast<int32_t*>(out + 4 * (size_t)(parent_slot >> 1) + 3)[parent_slot & 1u] = (int32_t)id;
  return id;
}

// a node's boxes, and its leaf children (slots; kRoot: an inner child, which
// writes itself)
__device__ __forceinline__ void write_node(float4* out, uint32_t id, const float cl[2][3],
                                           const float ch[2][3], uint32_t leaf0, uint32_t leaf1) {
  float4* o = out + 4 * (size_t)id;
  o[0] = make_float4(cl[0][0], ch[0][0], cl[0][1], ch[0][1]);
  o[1] = make_float4(cl[1][0], ch[1][0], cl[1][1], ch[1][1]);
  o[2] = make_float4(cl[0][2], ch[0][2], cl[1][2], ch[1][2]);
  int32_t* w = reinterpret_cast<int32_t*>(o + 3);
  if (leaf0 != kRoot) w[0] = ~(int32_t)leaf0;
  if (leaf1 != kRoot) w[1] = ~(int32_t)leaf1;
  w[2] = 0;
  w[3] = 0;
}

// one leaf into a bin
__device__ __forceinline__ void add_box(Bins& bins, int a, int bin, const int v[6]) {
  atomicAdd(&bins.cnt[a][bin], 1);
  for (int q = 0; q < 3; ++q) {
    atomicMin(&bins.box[a][bin][q], v[q]);
    atomicMax(&bins.box[a][bin][3 + q], v[3 + q]);
  }
}

__device__ __forceinline__ float at3(const float v[3], int a) { return a == 0 ? v[0] : a == 1 ? v[1] : v[2]; }

// Minima (values 0..2) and maxima (3..5) of the lanes of `grp`, combined into
// dst by its first lane
__device__ __forceinline__ void combine6(uint32_t grp, const int v[6], int* dst) {
  int r[6];
  for (int q = 0; q < 3; ++q) {
    r[q] = __reduce_min_sync(grp, v[q]);
    r[3 + q] = __reduce_max_sync(grp, v[3 + q]);
  }
  if ((uint32_t)(__ffs(grp) - 1) == (threadIdx.x & 31))
    for (int q = 0; q < 3; ++q) {
      atomicMin(dst + q, r[q]);
      atomicMax(dst + 3 + q, r[3 + q]);
    }
}

// leaf box of slot k: the child box of k's parent that holds leaf ~k; the
// identity order; and the centroid bounds of all leaves
__global__ void __launch_bounds__(kThreads)
k_leaves(const float4* nodes, const int32_t* parent, uint32_t n,
         float4* lo, float4* hi, uint32_t* idx, TopNode* root) {
  after_previous();
  const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  __shared__ int s_bounds[6];
  if (threadIdx.x < 6) s_bounds[threadIdx.x] = empty6(threadIdx.x);
  __syncthreads();
  int v[6];
  for (int q = 0; q < 6; ++q) v[q] = empty6(q);
  if (k < n) {
    const int32_t p = parent[n - 1 + k];
    const float4 a = nodes[4 * (size_t)p], b = nodes[4 * (size_t)p + 1],
                 c = nodes[4 * (size_t)p + 2], e = nodes[4 * (size_t)p + 3];
    const bool first = __float_as_int(e.x) == ~(int32_t)k;
    const float4 l = first ? make_float4(a.x, a.z, c.x, 0.f) : make_float4(b.x, b.z, c.z, 0.f);
    const float4 h = first ? make_float4(a.y, a.w, c.y, 0.f) : make_float4(b.y, b.w, c.w, 0.f);
    lo[k] = l;
    hi[k] = h;
    idx[k] = k;
    float m[3];
    centroid(l, h, m);
    centroid6(m, v);
  }
  if (!root) return;
  combine6(0xFFFFFFFFu, v, s_bounds);
  __syncthreads();
  if (threadIdx.x < 3) atomicMin(&root->bounds[threadIdx.x], s_bounds[threadIdx.x]);
  else if (threadIdx.x < 6) atomicMax(&root->bounds[threadIdx.x], s_bounds[threadIdx.x]);
}

// the build's control words and, in a build with a top phase, its root entry;
// else the whole build is one mid job
__global__ void k_begin(Control* c, TopNode* root, uint32_t* slice_node, Job* mid, uint32_t n, uint32_t slice) {
  after_previous();
  const uint32_t slices = (uint32_t)(((uint64_t)n + slice - 1) / slice);
  if (root) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < slices; i += gridDim.x * blockDim.x)
      slice_node[i] = 0;
    if (blockIdx.x == 0) {
      for (int i = threadIdx.x; i < kBinWords; i += blockDim.x) words(root->bins)[i] = empty_word(i);
      if (threadIdx.x < 6) root->bounds[threadIdx.x] = empty6(threadIdx.x);
      if (threadIdx.x < 12) {
        root->child_bounds[threadIdx.x / 6][threadIdx.x % 6] = empty6(threadIdx.x % 6);
        root->child_box[threadIdx.x / 6][threadIdx.x % 6] = empty6(threadIdx.x % 6);
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *c = Control{{root ? 1u : 0u, 0u}, {root ? slices : 0u, 0u}, root ? 0u : 1u, 0u};
    if (root) {
      root->job = Job{0u, n, kRoot, 0u};
      root->slice0 = 0;
      root->n_slices = slices;
      root->done = 0;
    } else {
      mid[0] = Job{0u, n, kRoot, 0u};
    }
  }
}

// ------------------------------------------------------------------ top phase
// a slice's leaves: [sb, se) of its node's range
__device__ __forceinline__ void slice_range(const TopNode& t, uint32_t s, uint32_t slice, uint32_t& sb,
                                            uint32_t& se) {
  const uint64_t at = (uint64_t)t.job.begin + (uint64_t)(s - t.slice0) * slice;
  sb = (uint32_t)at;
  se = (uint32_t)min((uint64_t)t.job.end, at + slice);
}

// the boxes (and slots) of leaves base + u kThreads + thread below `end`, all
// loads in flight at once: a slice is a chain of two dependent loads otherwise
constexpr int kUnroll = 4;
__device__ __forceinline__ void load_leaves(const Build& g, uint32_t base, uint32_t end, float4 lo[kUnroll],
                                            float4 hi[kUnroll], uint32_t* slot) {
  uint32_t k[kUnroll];
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) {
    const uint32_t i = base + u * kThreads + threadIdx.x;
    k[u] = i < end ? g.idx[0][i] : 0u;
  }
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) {
    lo[u] = g.lo[k[u]];
    hi[u] = g.hi[k[u]];
    if (slot) slot[u] = k[u];
  }
}

// 1. bins of a slice, added to its node's; the slice's own counts are kept
__global__ void __launch_bounds__(kThreads)
k_top_bins(const Build g, int cur) {
  after_previous();
  const uint32_t* slice_node = g.slice_node[0];
  int* slice_cnt = g.slice_cnt;
  TopNode* nodes = g.nodes[0];
  Control* ctl = g.ctl;
  const uint32_t slice = g.slice;
  // sets of bins for the 8 warps: more cost their clearing and merging, fewer their atomics' conflicts
  // (a 257k-primitive scene's creation 1.14 ms with 8, 1.10 with 4, 1.12 with 2, 1.15 with 1)
  constexpr int kSets = 4;
  __shared__ Bins s_bins[kSets];
  const uint32_t tid = threadIdx.x, n_slices = ctl->n_slices[cur];
  if (blockIdx.x == 0 && tid == 0) ctl->n_nodes[cur ^ 1] = ctl->n_slices[cur ^ 1] = 0;   // step 3 fills them
  for (uint32_t s = blockIdx.x; s < n_slices; s += gridDim.x) {
    TopNode& t = nodes[slice_node[s]];
    float cmin[3], cext[3];
    if (node_frame(t.bounds, t.job.end - t.job.begin, t.job.depth, cmin, cext)) continue;   // block-uniform
    uint32_t sb, se;
    slice_range(t, s, slice, sb, se);
    __syncthreads();
    for (int i = tid; i < kBinWords; i += kThreads) {
      const int e = empty_word(i);
      for (int w = 0; w < kSets; ++w) words(s_bins[w])[i] = e;
    }
    __syncthreads();
    Bins& mine = s_bins[(tid >> 5) % kSets];
    for (uint32_t base = sb; base < se; base += kUnroll * kThreads) {
      float4 lo[kUnroll], hi[kUnroll];
      load_leaves(g, base, se, lo, hi, nullptr);
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const bool in = base + u * kThreads + tid < se;
        const uint32_t active = __ballot_sync(0xFFFFFFFFu, in);
        if (!in) continue;
        float c[3];
        int v[6];
        centroid(lo[u], hi[u], c);
        box6(lo[u], hi[u], v);
        // Neighbouring leaves mostly share a bin: where a warp's leaves fall
        // in at most two bins, their lanes combine first. The reductions of
        // different lane sets run one after another, so with more bins plain
        // shared-memory atomics are faster (20 levels of 10M leaves: 4.5 ms
        // always combining, 8.5 never, 3.2 with this rule; 3.4 from four bins up).
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          if (!(cext[a] > 0.f)) continue;        // uniform over the block
          const int bin = bin_of(c[a], cmin[a], cext[a]);
          const uint32_t grp = __match_any_sync(active, bin);
          const bool leader = (uint32_t)(__ffs(grp) - 1) == (tid & 31);
          if (__popc(__ballot_sync(active, leader)) <= 2) {
            if (leader) atomicAdd(&mine.cnt[a][bin], __popc(grp));
            combine6(grp, v, mine.box[a][bin]);
          } else {
            add_box(mine, a, bin, v);
          }
        }
      }
    }
    __syncthreads();
    for (int i = tid; i < kBinWords; i += kThreads) {
      const int op = word_op(i);                 // the counts are words 0..47
      int v = words(s_bins[0])[i];
      for (int w = 1; w < kSets; ++w) {
        const int x = words(s_bins[w])[i];
        v = op == 0 ? v + x : op < 0 ? min(v, x) : max(v, x);
      }
      int* to = words(t.bins) + i;
      if (i < 64) {                              // whole warps
        int sum = v;
        for (int o = 1; o < kBins; o <<= 1) {
          const int u = __shfl_up_sync(0xFFFFFFFFu, sum, o, kBins);
          if ((i & (kBins - 1)) >= o) sum += u;
        }
        if (op == 0) slice_cnt[(size_t)s * 3 * kBins + i] = sum;
      }
      if (v == empty_word(i)) continue;
      if (op == 0) atomicAdd(to, v); else if (op < 0) atomicMin(to, v); else atomicMax(to, v);
    }
  }
}

// 3. a node's record, and its children: top entries of the next level, mid
// jobs or leaves (one block)
struct NodeShared {
  float box[2][6];
  uint32_t at[2], slice0[2], id;
};
__device__ void top_node(const TopNode& t, uint32_t n_left, int axis, int bin, const uint32_t* idx_out,
                         const Build& g, int cur, NodeShared& sh) {
  const uint32_t tid = threadIdx.x, b = t.job.begin, e = t.job.end, split = b + n_left;
  const uint32_t rb[2] = {b, split}, re[2] = {split, e};
  Control* ctl = g.ctl;
  if (tid < 12) {
    const int c = tid / 6, f = tid % 6;
    int v = empty6(f);
    if (axis < 0) {
      v = __ldcg(&t.child_box[c][f]);
    } else {
      for (int q = 0; q < kBins; ++q) {
        const int x = t.bins.box[axis][q][f];        // an empty bin's box is empty
        if ((q <= bin) == (c == 0)) v = f < 3 ? min(v, x) : max(v, x);
      }
    }
    sh.box[c][f] = o2f(v);
  }
  if (tid == 0) {
    if (t.job.parent_slot == kRoot) ctl->root_split = split;
    const uint32_t id = place_node(split, t.job.parent_slot, ctl->root_split, g.out, g.n, g.err);
    sh.id = id;
    for (int c = 0; c < 2; ++c) {
      const uint32_t m = re[c] - rb[c];
      sh.at[c] = kRoot;
      if (m == 1) continue;
      if (m <= kMidLeaves) {
        const uint32_t at = atomicAdd(&ctl->n_mid, 1u);
        if (at >= g.max_mid) { atomicOr(g.err, ERR_BUILD); continue; }
        g.mid[at] = Job{rb[c], re[c], id << 1 | (uint32_t)c, (t.job.depth + 1) | ((uint32_t)(cur ^ 1) << 31)};
      } else {
        const uint32_t ns = (uint32_t)(((uint64_t)m + g.slice - 1) / g.slice);
        const uint32_t at = atomicAdd(&ctl->n_nodes[cur ^ 1], 1u), s0 = atomicAdd(&ctl->n_slices[cur ^ 1], ns);
        if (at >= g.max_nodes || s0 + ns > g.max_slices) { atomicOr(g.err, ERR_BUILD); continue; }
        sh.at[c] = at;
        sh.slice0[c] = s0;
      }
    }
  }
  __syncthreads();
  const uint32_t id = sh.id;
  if (tid == 0) {
    float cl[2][3], ch[2][3];
    for (int c = 0; c < 2; ++c)
      for (int x = 0; x < 3; ++x) { cl[c][x] = sh.box[c][x]; ch[c][x] = sh.box[c][3 + x]; }
    write_node(g.out, id, cl, ch, re[0] - rb[0] == 1 ? __ldcg(idx_out + rb[0]) : kRoot,
               re[1] - rb[1] == 1 ? __ldcg(idx_out + rb[1]) : kRoot);
  }
  for (int c = 0; c < 2; ++c) {
    if (sh.at[c] == kRoot) continue;
    TopNode& u = g.nodes[1][sh.at[c]];
    const uint32_t m = re[c] - rb[c], ns = (uint32_t)(((uint64_t)m + g.slice - 1) / g.slice);
    for (int i = tid; i < kBinWords; i += kThreads) words(u.bins)[i] = empty_word(i);
    if (tid < 6) u.bounds[tid] = __ldcg(&t.child_bounds[c][tid]);
    if (tid < 12) {
      u.child_bounds[tid / 6][tid % 6] = empty6(tid % 6);
      u.child_box[tid / 6][tid % 6] = empty6(tid % 6);
    }
    if (tid == 0) {
      u.job = Job{rb[c], re[c], id << 1 | (uint32_t)c, t.job.depth + 1};
      u.slice0 = sh.slice0[c];
      u.n_slices = ns;
      u.done = 0;
    }
    for (uint32_t i = tid; i < ns; i += kThreads) g.slice_node[1][sh.slice0[c] + i] = sh.at[c];
  }
}

// 2. the node's split (every slice computes it) and the stable partition of
// the slice, with the centroid bounds (and for a median the boxes) of the sides;
// then step 3 by the node's last slice
__global__ void __launch_bounds__(kThreads, 4)
k_top_scatter(const Build g, int cur) {
  after_previous();
  uint32_t* idx_out = g.idx[1];
  const uint32_t* slice_node = g.slice_node[0];
  const int* slice_cnt = g.slice_cnt;
  TopNode* nodes = g.nodes[0];
  const uint32_t slice = g.slice;
  __shared__ NodeShared s_node;
  __shared__ bool s_last;
  __shared__ Bins s_bins;
  __shared__ int s_choice[2];
  __shared__ uint32_t s_sum[2], s_scan[kUnroll][kWarps];
  __shared__ int s_bounds[2][6], s_box[2][6];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_slices = g.ctl->n_slices[cur];
  for (uint32_t s = blockIdx.x; s < n_slices; s += gridDim.x) {
    TopNode& t = nodes[slice_node[s]];
    const uint32_t b = t.job.begin, m = t.job.end - b, q = s - t.slice0;
    float cmin[3], cext[3];
    bool median = node_frame(t.bounds, m, t.job.depth, cmin, cext);
    __syncthreads();
    for (int i = tid; i < kBinWords; i += kThreads) words(s_bins)[i] = words(t.bins)[i];
    if (tid < 12) {
      s_bounds[tid / 6][tid % 6] = empty6(tid % 6);
      s_box[tid / 6][tid % 6] = empty6(tid % 6);
    }
    if (tid < 2) s_sum[tid] = 0;
    __syncthreads();
    if (!median && warp == 0) {
      int axis, bin;
      choose_split(s_bins, cext, axis, bin);
      if (lane == 0) { s_choice[0] = axis; s_choice[1] = bin; }
    }
    __syncthreads();
    int axis = median ? -1 : s_choice[0], bin = median ? 0 : s_choice[1];
    // lefts of the slices before this one, and of the node
    if (axis >= 0) {
      uint32_t before = 0, all = 0;
      for (uint32_t r = tid; r < t.n_slices; r += kThreads) {
        const uint32_t left = (uint32_t)slice_cnt[(size_t)(t.slice0 + r) * 3 * kBins + axis * kBins + bin];
        all += left;
        if (r < q) before += left;
      }
      before = __reduce_add_sync(0xFFFFFFFFu, before);
      all = __reduce_add_sync(0xFFFFFFFFu, all);
      if (lane == 0 && all) { atomicAdd(&s_sum[0], before); atomicAdd(&s_sum[1], all); }
    }
    __syncthreads();
    const uint32_t before = s_sum[0];
    uint32_t n_left = s_sum[1];
    // an empty side cannot happen with an axis (its cost is infinite)
    if (axis < 0 || n_left == 0 || n_left == m) { axis = -1; n_left = m / 2; }
    uint32_t sb, se;
    slice_range(t, s, slice, sb, se);
    const uint32_t rights_before = (sb - b) - before;
    uint32_t cnt_left = 0;
    int sides[2][6];                              // centroid bounds of the thread's lefts and rights
    for (int c = 0; c < 2; ++c)
      for (int f = 0; f < 6; ++f) sides[c][f] = empty6(f);
    for (uint32_t base = sb; base < se; base += kUnroll * kThreads) {
      float4 lo[kUnroll], hi[kUnroll];
      uint32_t k[kUnroll], ball[kUnroll];
      load_leaves(g, base, se, lo, hi, k);
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const uint32_t i = base + u * kThreads + tid;
        float c[3];
        centroid(lo[u], hi[u], c);
        const bool left = i < se && (axis < 0 ? i - b < n_left
                                              : bin_of(at3(c, axis), at3(cmin, axis), at3(cext, axis)) <= bin);
        ball[u] = __ballot_sync(0xFFFFFFFFu, left);
        if (lane == 0) s_scan[u][warp] = __popc(ball[u]);
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const uint32_t i = base + u * kThreads + tid;
        uint32_t wb = 0, chunk = 0;
#pragma unroll
        for (uint32_t w = 0; w < (uint32_t)kWarps; ++w) {
          const uint32_t x = s_scan[u][w];
          if (w < warp) wb += x;
          chunk += x;
        }
        const uint32_t rank = wb + __popc(ball[u] & ((1u << lane) - 1u));   // lefts before i among these
        const uint32_t in = __ballot_sync(0xFFFFFFFFu, i < se);
        if (i < se) {
          const bool left = ball[u] >> lane & 1u;
          if (axis < 0) idx_out[i] = k[u];
          else if (left) idx_out[b + before + cnt_left + rank] = k[u];
          else idx_out[b + n_left + rights_before + (i - sb) - cnt_left - rank] = k[u];
          float c[3];
          int v[6];
          centroid(lo[u], hi[u], c);
          centroid6(c, v);
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            sides[0][f] = min(sides[0][f], left ? v[f] : empty6(f));
            sides[1][f] = min(sides[1][f], left ? empty6(f) : v[f]);
            sides[0][3 + f] = max(sides[0][3 + f], left ? v[3 + f] : empty6(3));
            sides[1][3 + f] = max(sides[1][3 + f], left ? empty6(3) : v[3 + f]);
          }
          if (axis < 0) {
            box6(lo[u], hi[u], v);
            combine6(left ? ball[u] : in & ~ball[u], v, s_box[left ? 0 : 1]);
          }
        }
        cnt_left += chunk;
      }
      __syncthreads();
    }
    for (int c = 0; c < 2; ++c) combine6(0xFFFFFFFFu, sides[c], s_bounds[c]);
    __syncthreads();
    if (tid < 12) {
      const int c = tid / 6, f = tid % 6, v = s_bounds[c][f], w = s_box[c][f];
      if (v != empty6(f)) {
        if (f < 3) atomicMin(&t.child_bounds[c][f], v); else atomicMax(&t.child_bounds[c][f], v);
      }
      if (axis < 0 && w != empty6(f)) {
        if (f < 3) atomicMin(&t.child_box[c][f], w); else atomicMax(&t.child_box[c][f], w);
      }
    }
    // the slice that finishes last writes the node
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&t.done, 1u) + 1 == t.n_slices;
    __syncthreads();
    if (s_last) {
      __threadfence();
      top_node(t, n_left, axis, bin, idx_out, g, cur, s_node);
    }
  }
}

// ------------------------------------------------------------------ mid phase
// The subtree over the m <= 32 leaves of a segment (one warp; lane < m: leaf
// slot and box): every node takes the split of least SAH cost over all
// positions of its leaves sorted by centroid on each axis (ties by the current
// order, then by the lower axis), or the middle of the current order when the
// depth budget is short. All nodes of a level at once: lane l belongs to the
// segment [b, e) of lanes. Shuffles bound it (they share the one shared-memory
// pipe of the SM), so ranks are counted and scans run only as far as the level's
// longest segment, and only the winning position's child boxes are handed out.
// key: the warp's scratch.
__device__ void small_subtree(uint32_t m, uint32_t slot, float bx[6], uint32_t base, uint32_t parent_slot,
                              uint32_t depth, uint32_t root_split, float4* out, uint32_t n,
                              uint32_t* err, uint32_t* key) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t b = lane < m ? 0u : lane, e = lane < m ? m : lane + 1;
  for (uint32_t guard = 0; guard < kSmallLeaves; ++guard) {
    const uint32_t s = e - b;
    const bool active = s >= 2;
    const uint32_t longest = __reduce_max_sync(0xFFFFFFFFu, s);
    if (longest < 2) return;
    const bool sah = active && depth + s - 1 <= (uint32_t)kMaxDepth;
    uint32_t order = lane, cut = b + s / 2 - 1;       // source lane of this position; last left position
    float c0[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, c1[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // child boxes
    if (!__any_sync(0xFFFFFFFFu, s > 2 || (active && !sah))) {
      // two leaves: every axis costs the same, so the first one's order (a
      // cost past the largest float: the current order)
      const uint32_t other = active ? (lane == b ? b + 1 : b) : lane;
      const float mine = 0.5f * (bx[0] + bx[3]), area = half_area(bx, bx + 3);
      const float theirs = __shfl_sync(0xFFFFFFFFu, mine, other), oa = __shfl_sync(0xFFFFFFFFu, area, other);
      if (active) {
        const bool swap = lane == b ? theirs < mine : mine < theirs;
        if (swap && area + oa < INFINITY) order = other;
        cut = b;
      }
      for (int x = 0; x < 6; ++x) {
        const float v = __shfl_sync(0xFFFFFFFFu, bx[x], order);   // box at this position
        c0[x] = __shfl_sync(0xFFFFFFFFu, v, b);
        c1[x] = __shfl_sync(0xFFFFFFFFu, v, e - 1);
      }
    } else {
      float best = INFINITY;
      uint32_t at = 96, vals = 0;                    // axis << 5 | position of `best`; the three orders, 5 bits each
      // rank by (centroid with -0 as 0, position) in the segment, all axes at once
      int k3[3];
      uint32_t rank[3] = {b, b, b};
      for (int a = 0; a < 3; ++a) k3[a] = f2o(0.5f * (bx[a] + bx[3 + a]) + 0.f);
      for (uint32_t j = 0; j < longest; ++j) {
        const uint32_t src = b + j;
        const bool in = src < e;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int o = __shfl_sync(0xFFFFFFFFu, k3[a], src & 31u);
          rank[a] += in && (src < lane ? o <= k3[a] : o < k3[a]) ? 1u : 0u;
        }
      }
      __syncwarp();
      for (int a = 0; a < 3; ++a) {
        key[rank[a]] = lane;
        __syncwarp();
        vals |= key[lane] << (5 * a);
        __syncwarp();
      }
      for (int axis = 0; axis < 3; ++axis) {
        const uint32_t val = vals >> (5 * axis) & 31u;
        float p[6], q[6];
        for (int x = 0; x < 6; ++x) p[x] = q[x] = __shfl_sync(0xFFFFFFFFu, bx[x], val);
        for (uint32_t o = 1; o < longest; o <<= 1) {
          const bool up = lane >= b + o, dn = lane + o < e;
#pragma unroll
          for (int x = 0; x < 6; ++x) {
            const float u = __shfl_up_sync(0xFFFFFFFFu, p[x], o), d = __shfl_down_sync(0xFFFFFFFFu, q[x], o);
            if (up) p[x] = x < 3 ? fminf(p[x], u) : fmaxf(p[x], u);
            if (dn) q[x] = x < 3 ? fminf(q[x], d) : fmaxf(q[x], d);
          }
        }
        for (int x = 0; x < 6; ++x) q[x] = __shfl_down_sync(0xFFFFFFFFu, q[x], 1);   // of the positions after this one
        if (sah && lane + 1 < e) {
          const float cost = half_area(p, p + 3) * (float)(lane - b + 1) + half_area(q, q + 3) * (float)(e - lane - 1);
          if (cost < best) {
            best = cost;
            at = (uint32_t)axis << 5 | lane;
            for (int x = 0; x < 6; ++x) { c0[x] = p[x]; c1[x] = q[x]; }
          }
        }
      }
      // the segment's least cost; among equals the lower axis, then position: its last lane's prefix
      for (uint32_t o = 1; o < longest; o <<= 1) {
        const float c = __shfl_up_sync(0xFFFFFFFFu, best, o);
        const uint32_t i = __shfl_up_sync(0xFFFFFFFFu, at, o);
        if (lane >= b + o && (c < best || (c == best && i < at))) { best = c; at = i; }
      }
      best = __shfl_sync(0xFFFFFFFFu, best, e - 1);
      at = __shfl_sync(0xFFFFFFFFu, at, e - 1);
      const bool found = active && best < INFINITY;
      if (found) { cut = at & 31u; order = vals >> (5 * (at >> 5)) & 31u; }
      for (int x = 0; x < 6; ++x) {
        c0[x] = __shfl_sync(0xFFFFFFFFu, c0[x], cut & 31u);
        c1[x] = __shfl_sync(0xFFFFFFFFu, c1[x], cut & 31u);
      }
      // no split by cost: the middle of the current order, its boxes by walking the segment
      if (__any_sync(0xFFFFFFFFu, active && !found)) {
        float m0[6], m1[6];
        for (int x = 0; x < 6; ++x) m0[x] = m1[x] = x < 3 ? INFINITY : -INFINITY;
        for (uint32_t j = 0; j < longest; ++j)
          for (int x = 0; x < 6; ++x) {
            const float v = __shfl_sync(0xFFFFFFFFu, bx[x], (b + j) & 31u);
            if (b + j <= cut) m0[x] = x < 3 ? fminf(m0[x], v) : fmaxf(m0[x], v);
            else if (b + j < e) m1[x] = x < 3 ? fminf(m1[x], v) : fmaxf(m1[x], v);
          }
        if (active && !found)
          for (int x = 0; x < 6; ++x) { c0[x] = m0[x]; c1[x] = m1[x]; }
      }
    }
    slot = __shfl_sync(0xFFFFFFFFu, slot, order);
    for (int x = 0; x < 6; ++x) bx[x] = __shfl_sync(0xFFFFFFFFu, bx[x], order);
    const uint32_t mid = cut + 1;                    // first right position
    const uint32_t right_slot = __shfl_sync(0xFFFFFFFFu, slot, active ? mid : lane);
    uint32_t id = 0;
    if (active && lane == b) {
      id = place_node(base + mid, parent_slot, root_split, out, n, err);
      const float cl[2][3] = {{c0[0], c0[1], c0[2]}, {c1[0], c1[1], c1[2]}};
      const float ch[2][3] = {{c0[3], c0[4], c0[5]}, {c1[3], c1[4], c1[5]}};
      write_node(out, id, cl, ch, mid - b == 1 ? slot : kRoot, e - mid == 1 ? right_slot : kRoot);
    }
    id = __shfl_sync(0xFFFFFFFFu, id, b);
    if (active) {
      const bool right = lane >= mid;
      parent_slot = id << 1 | (right ? 1u : 0u);
      ++depth;
      if (right) b = mid; else e = mid;
    }
    __syncwarp();
  }
  if (lane == 0) atomicOr(err, ERR_BUILD);
}

// Subtrees of 2 to kMidLeaves leaves, one block each, one thread per leaf.
// segments of more than kSmallLeaves leaves (or the root)
constexpr int kMaxSeg = (int)(kMidLeaves / (kSmallLeaves + 1));
static_assert(kMaxSeg <= kWarps, "a warp per segment");
__global__ void __launch_bounds__(kThreads, 4)
k_sah_mid(const float4* leaf_lo, const float4* leaf_hi,
          const uint32_t* idx0, const uint32_t* idx1, Control* ctl,
          const Job* jobs, float4* out, uint32_t n, uint32_t* err) {
  after_previous();
  __shared__ uint32_t s_slot[kThreads];
  __shared__ float s_box[6][kThreads];
  __shared__ uint32_t s_begin[kThreads], s_end[kThreads];          // segment of each position
  __shared__ uint32_t s_parent[kThreads], s_depth[kThreads];       // of the segment that begins here
  __shared__ uint32_t s_scan[kWarps], s_seg[kThreads];
  __shared__ Bins s_bins[kMaxSeg];
  __shared__ int s_bounds[kMaxSeg][6], s_child[kMaxSeg][2][6];
  __shared__ int s_choice[kMaxSeg][2];
  __shared__ uint32_t s_at[kMaxSeg], s_nleft[kMaxSeg], s_root_split, s_total, s_key[kWarps][kSmallLeaves];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_jobs = ctl->n_mid;
  for (uint32_t j = blockIdx.x; j < n_jobs; j += gridDim.x) {
    const Job job = jobs[j];
    const uint32_t base = job.begin, m = job.end - job.begin;
    if (m < 2 || m > kMidLeaves) { if (tid == 0) atomicOr(err, ERR_BUILD); continue; }   // block-uniform
    const uint32_t* idx = job.depth >> 31 ? idx1 : idx0;
    __syncthreads();
    if (tid == 0) s_root_split = ctl->root_split;
    uint32_t slot = 0;
    float bx[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (tid < m) {
      slot = idx[base + tid];
      const float4 lo = leaf_lo[slot], hi = leaf_hi[slot];
      bx[0] = lo.x; bx[1] = lo.y; bx[2] = lo.z; bx[3] = hi.x; bx[4] = hi.y; bx[5] = hi.z;
    }
    s_begin[tid] = tid < m ? 0u : tid;
    s_end[tid] = tid < m ? m : tid + 1;
    if (tid == 0) { s_parent[0] = job.parent_slot; s_depth[0] = job.depth & 0x7FFFFFFFu; }
    __syncthreads();
    for (int level = 0; level <= kMaxDepth; ++level) {
      const uint32_t b = s_begin[tid], e = s_end[tid], sz = e - b;
      const bool active = sz > kSmallLeaves || (sz >= 2 && s_parent[b] == kRoot);
      // ordinals of the active segments
      const bool head = active && tid == b;
      const uint32_t hb = __ballot_sync(0xFFFFFFFFu, head);
      if (lane == 0) s_scan[warp] = __popc(hb);
      if (tid < kMaxSeg * 6) s_bounds[tid / 6][tid % 6] = empty6(tid % 6);
      if (tid < kMaxSeg * 12) s_child[tid / 12][(tid / 6) % 2][tid % 6] = empty6(tid % 6);
      __syncthreads();
      uint32_t ord = 0, n_seg = 0;
      for (uint32_t w = 0; w < (uint32_t)kWarps; ++w) {
        if (w < warp) ord += s_scan[w];
        n_seg += s_scan[w];
      }
      if (n_seg == 0) break;                                   // block-uniform
      if (head) { ord += __popc(hb & ((1u << lane) - 1u)); s_seg[b] = ord; s_at[ord] = b; }
      for (uint32_t i = tid; i < (uint32_t)kBinWords; i += kThreads) {
        const int v = empty_word((int)i);
        for (uint32_t w = 0; w < n_seg; ++w) words(s_bins[w])[i] = v;
      }
      __syncthreads();
      const uint32_t g = active ? s_seg[b] : 0xFFu, members = __ballot_sync(0xFFFFFFFFu, active);
      const float c[3] = {0.5f * (bx[0] + bx[3]), 0.5f * (bx[1] + bx[4]), 0.5f * (bx[2] + bx[5])};
      const int v6[6] = {f2o(bx[0]), f2o(bx[1]), f2o(bx[2]), f2o(bx[3]), f2o(bx[4]), f2o(bx[5])};
      if (active) {
        int cv[6];
        centroid6(c, cv);
        combine6(__match_any_sync(members, g), cv, s_bounds[g]);
      }
      __syncthreads();
      float cmin[3] = {0.f, 0.f, 0.f}, cext[3] = {0.f, 0.f, 0.f};
      bool median = true;
      if (active) median = node_frame(s_bounds[g], sz, s_depth[b], cmin, cext);
      for (int a = 0; a < 3; ++a) {
        if (median || !(cext[a] > 0.f)) continue;
        const int bin = bin_of(c[a], cmin[a], cext[a]);
        add_box(s_bins[g], a, bin, v6);
      }
      __syncthreads();
      if (warp < n_seg) {
        float ext[3];
        int axis, bin;
        for (int x = 0; x < 3; ++x) ext[x] = o2f(s_bounds[warp][3 + x]) - o2f(s_bounds[warp][x]);
        choose_split(s_bins[warp], ext, axis, bin);
        if (lane == 0) { s_choice[warp][0] = axis; s_choice[warp][1] = bin; }
      }
      __syncthreads();
      // stable partition of every active segment
      int axis = active && !median ? s_choice[g][0] : -1;
      bool left = false;
      if (active)
        left = axis < 0 ? tid - b < sz / 2
                        : bin_of(at3(c, axis), at3(cmin, axis), at3(cext, axis)) <= s_choice[g][1];
      const uint32_t ball = __ballot_sync(0xFFFFFFFFu, left);
      if (lane == 0) s_scan[warp] = __popc(ball);
      __syncthreads();
      uint32_t rank = __popc(ball & ((1u << lane) - 1u));
      for (uint32_t w = 0; w < warp; ++w) rank += s_scan[w];
      s_seg[tid] = rank;                                       // lefts before this position
      if (tid == kThreads - 1) s_total = rank + (left ? 1u : 0u);
      __syncthreads();
      uint32_t to = tid, n_left = 0;
      if (active) {
        const uint32_t at_b = s_seg[b], at_e = e < kThreads ? s_seg[e] : s_total;
        n_left = at_e - at_b;
        if (n_left == 0 || n_left == sz) {                     // cannot happen with an axis
          axis = -1;
          n_left = sz / 2;
          left = tid - b < n_left;
        }
        if (axis >= 0) to = left ? b + (rank - at_b) : b + n_left + (tid - b - (rank - at_b));
        combine6(__match_any_sync(members, g * 2 + (left ? 0 : 1)), v6, s_child[g][left ? 0 : 1]);
        if (tid == b) s_nleft[g] = n_left;
      }
      s_slot[to] = slot;
      for (int x = 0; x < 6; ++x) s_box[x][to] = bx[x];
      __syncthreads();
      slot = s_slot[tid];
      for (int x = 0; x < 6; ++x) bx[x] = s_box[x][tid];
      if (active) {
        const uint32_t mid = b + n_left;
        if (tid >= mid) s_begin[tid] = mid; else s_end[tid] = mid;
      }
      // the records (the root's split position first: its children need it)
      if (tid == 0 && s_parent[0] == kRoot) {                  // only in the first level of a whole build
        s_root_split = s_nleft[0];
        ctl->root_split = s_nleft[0];
      }
      __syncthreads();
      if (tid < n_seg) {
        const uint32_t sb = s_at[tid], nl = s_nleft[tid], mid = sb + nl, se = s_end[mid];
        const uint32_t split = base + mid, depth = s_depth[sb];
        const uint32_t id = place_node(split, s_parent[sb], s_root_split, out, n, err);
        float cl[2][3], ch[2][3];
        for (int k = 0; k < 2; ++k)
          for (int x = 0; x < 3; ++x) { cl[k][x] = o2f(s_child[tid][k][x]); ch[k][x] = o2f(s_child[tid][k][3 + x]); }
        write_node(out, id, cl, ch, nl == 1 ? s_slot[sb] : kRoot, se - mid == 1 ? s_slot[mid] : kRoot);
        s_parent[sb] = id << 1;
        s_parent[mid] = id << 1 | 1u;
        s_depth[sb] = s_depth[mid] = depth + 1;
      }
      __syncthreads();
    }
    // every segment has at most kSmallLeaves leaves: a warp each, the list of
    // their first positions in s_seg
    {
      const bool head = tid < m && s_begin[tid] == tid && s_end[tid] - tid >= 2;
      const uint32_t hb = __ballot_sync(0xFFFFFFFFu, head);
      __syncthreads();
      if (lane == 0) s_scan[warp] = __popc(hb);
      s_slot[tid] = slot;
      for (int x = 0; x < 6; ++x) s_box[x][tid] = bx[x];
      __syncthreads();
      uint32_t at = 0, total = 0;
      for (uint32_t w = 0; w < (uint32_t)kWarps; ++w) {
        if (w < warp) at += s_scan[w];
        total += s_scan[w];
      }
      if (head) s_seg[at + __popc(hb & ((1u << lane) - 1u))] = tid;
      __syncthreads();
      for (uint32_t w = warp; w < total; w += kWarps) {
        const uint32_t sb = s_seg[w], sm = s_end[sb] - sb, at_lane = min(sb + lane, (uint32_t)kThreads - 1);
        float lb[6];
        for (int x = 0; x < 6; ++x) lb[x] = s_box[x][at_lane];
        small_subtree(sm, s_slot[at_lane], lb, base + sb, s_parent[sb], s_depth[sb], s_root_split, out, n, err,
                      s_key[warp]);
      }
      __syncthreads();
    }
  }
}

bool g_sah_slicing = true;

// Centre and half extent of [lo, hi], so that [c - e, c + e] contains it: e is
// rounded up, and widened by 2^-22 of the box's distance from the origin for
// the rounding of the two products the walk forms from it. An empty box
// (lo > hi) gets e = -inf, which no ray hits. FP64 has few units: where both
// differences are exact in FP32 (rounded down as up), as they are when lo and
// hi are within a factor of two, FP32 gives the same two values (10M nodes:
// 189 us; all in FP64 1333 us).
__device__ __forceinline__ void centre_extent(float lo, float hi, float& c, float& e) {
  if (!(lo <= hi)) { c = 0.f; e = -INFINITY; return; }
  const float big = fmaxf(fabsf(lo), fabsf(hi));
  c = __fadd_rn(0.5f * lo, 0.5f * hi);
  const float up = __fsub_ru(hi, c), dn = __fsub_ru(c, lo);
  if (up == __fsub_rd(hi, c) && dn == __fsub_rd(c, lo) && (big > 1e-30f || big == 0.f)) {
    e = __fmaf_ru(0x1p-22f, big, fmaxf(up, dn));
    return;
  }
  c = (float)(0.5 * ((double)lo + (double)hi));
  const double half = fmax((double)hi - (double)c, (double)c - (double)lo);
  e = __double2float_ru(half + 0x1p-22 * (double)big);
}

__global__ void k_render_nodes(const float4* nodes, uint32_t n_inner, float4* out) {
  after_previous();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_inner) return;
  const float4 a = nodes[4 * (size_t)i], b = nodes[4 * (size_t)i + 1], c = nodes[4 * (size_t)i + 2];
  float4 u, v, w;
  centre_extent(a.x, a.y, u.x, u.z);
  centre_extent(a.z, a.w, u.y, u.w);
  centre_extent(b.x, b.y, v.x, v.z);
  centre_extent(b.z, b.w, v.y, v.w);
  centre_extent(c.x, c.y, w.x, w.y);
  centre_extent(c.z, c.w, w.z, w.w);
  float4* o = out + 4 * (size_t)i;
  o[0] = u;
  o[1] = v;
  o[2] = w;
  o[3] = nodes[4 * (size_t)i + 3];
}
}  // namespace

cudaError_t render_nodes(const float4* nodes, uint32_t n, float4* out, cudaStream_t st) {
  if (n < 2) return cudaSuccess;      // no inner node
  launch_after(k_render_nodes, (n - 1 + 255) / 256, 256, 0, st, nodes, n - 1, out);
  return cudaGetLastError();
}

void set_sah_slicing(bool on) { g_sah_slicing = on; }

namespace {
// returns the bytes that the scratch takes
size_t sah_scratch(char* base, uint32_t n, bool slicing, Build& s) {
  // slices of at least kSlice leaves, and at most about 2048 of a node: every slice adds up the
  // counts of its node's slices
  s.slice = slicing ? std::max(kSlice, (uint32_t)(((uint64_t)n + 2047) / 2048)) : 0xFFFFFFFFu;
  s.max_nodes = n / (kMidLeaves + 1) + 1;
  s.max_slices = n / kSlice + s.max_nodes + 1;
  s.max_mid = n / 2 + 1;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    char* p = base + at;
    at += (bytes + 255) / 256 * 256;
    return p;
  };
  s.lo = reinterpret_cast<float4*>(take((size_t)n * sizeof(float4)));
  s.hi = reinterpret_cast<float4*>(take((size_t)n * sizeof(float4)));
  for (int i = 0; i < 2; ++i) {
    s.idx[i] = reinterpret_cast<uint32_t*>(take((size_t)n * sizeof(uint32_t)));
    s.nodes[i] = reinterpret_cast<TopNode*>(take((size_t)s.max_nodes * sizeof(TopNode)));
    s.slice_node[i] = reinterpret_cast<uint32_t*>(take((size_t)s.max_slices * sizeof(uint32_t)));
  }
  s.slice_cnt = reinterpret_cast<int*>(take((size_t)s.max_slices * 3 * kBins * sizeof(int)));
  s.mid = reinterpret_cast<Job*>(take((size_t)s.max_mid * sizeof(Job)));
  s.ctl = reinterpret_cast<Control*>(take(sizeof(Control)));
  return at;
}
}  // namespace

size_t sah_tmp_bytes(uint32_t n) {
  Build b{};
  return sah_scratch(nullptr, n ? n : 1, true, b);
}

cudaError_t build_sah_tree(const float4* lbvh_nodes, const int32_t* parent, uint32_t n,
                           float4* out, void* tmp, uint32_t* err, cudaStream_t st) {
  if (n < 2) return cudaMemcpyAsync(out, lbvh_nodes, 4 * sizeof(float4), cudaMemcpyDeviceToDevice, st);
  Build s{};
  sah_scratch(static_cast<char*>(tmp), n, g_sah_slicing, s);
  s.out = out;
  s.err = err;
  s.n = n;
  const bool top = n > kMidLeaves;
  const uint32_t* const idx[2] = {s.idx[0], s.idx[1]};
  TopNode* root = top ? s.nodes[0] : nullptr;
  Chain chain{st};
  chain.then(k_begin, 1, kThreads, 0, s.ctl, root, s.slice_node[0], s.mid, n, s.slice);
  chain.then(k_leaves, (int)(((uint64_t)n + kThreads - 1) / kThreads), kThreads, 0, lbvh_nodes, parent, n, s.lo,
             s.hi, s.idx[0], root);
  uint32_t n_mid = 1;
  if (top) {
    const int blocks = (int)std::min(s.max_slices, 8u * (uint32_t)num_sms());
    // as many levels as a balanced tree has and kExtra more, then kExtra at a time
    constexpr int kExtra = 4;
    int until = kExtra;
    for (uint32_t m = n; m > kMidLeaves; m = (m + 1) / 2) ++until;
    Control c{};
    for (int level = 0; chain.error == cudaSuccess; ++level) {
      if (level == until || level == kMaxDepth + 2) {
        chain.error = cudaMemcpyAsync(&c, s.ctl, sizeof c, cudaMemcpyDeviceToHost, st);
        if (chain.error == cudaSuccess) chain.error = cudaStreamSynchronize(st);
        if (chain.error != cudaSuccess || c.n_nodes[level & 1] == 0) break;
        if (level == kMaxDepth + 2) return cudaErrorUnknown;      // deeper than the depth budget
        until += kExtra;
      }
      const int cur = level & 1;
      chain.then(k_top_bins, blocks, kThreads, 0, s, cur);
      chain.then(k_top_scatter, blocks, kThreads, 0, s, cur);
      std::swap(s.idx[0], s.idx[1]);
      std::swap(s.nodes[0], s.nodes[1]);
      std::swap(s.slice_node[0], s.slice_node[1]);
    }
    n_mid = c.n_mid;
    if (chain.error == cudaSuccess && n_mid > s.max_mid) chain.error = cudaErrorUnknown;
  }
  if (n_mid)
    chain.then(k_sah_mid, (int)std::min(n_mid, 0x7FFFFFFFu), kThreads, 0, s.lo, s.hi, idx[0], idx[1], s.ctl, s.mid,
               out, n, err);
  return chain.end();
}

}  // namespace rt
