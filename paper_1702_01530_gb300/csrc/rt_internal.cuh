// Internal declarations of the GB300 stereo ray tracer (CUDA, sm_103a).
//
// Data layout in HBM (all 16-byte aligned, read with 16-byte vector loads):
//   nodes  : (n-1) BVH2 nodes of 64 B = 4 x float4, binary radix tree
//            numbering (root 0). Both children's boxes live in the parent:
//              [0] = (c0.lo.x, c0.hi.x, c0.lo.y, c0.hi.y)
//              [1] = (c1.lo.x, c1.hi.x, c1.lo.y, c1.hi.y)
//              [2] = (c0.lo.z, c0.hi.z, c1.lo.z, c1.hi.z)
//              [3] = (left, right, -, -) as int bits; >= 0 internal, < 0 leaf ~k
//   render nodes (the copy of a tree that renders walk, same numbering): each
//            child box as centre c and half extent e:
//              [0] = (c0.c.x, c0.c.y, c0.e.x, c0.e.y)
//              [1] = (c1.c.x, c1.c.y, c1.e.x, c1.e.y)
//              [2] = (c0.c.z, c0.e.z, c1.c.z, c1.e.z)
//              [3] = (left, right, -, -)
//   prims  : n leaf records of 48 B = 3 x float4 in leaf (sorted key) order:
//            triangle: (v0.xyz, id) (e1.xyz, material) (e2.xyz, 0)
//            sphere  : (c.xyz, id)  (r, 0, 0, material)  (0, 0, 0, 0)
//            (id and material stored as uint bits; id < n_spheres = sphere)
//   mats   : float4 (albedo rgb, reflectivity)
//   lights : float4 (position xyz, intensity)
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <utility>

#include "../../include/rt_stereo.h"

namespace rt {

// device error word bits
enum : uint32_t {
  ERR_STACK = 1u,      // traversal stack bound exceeded
  ERR_ITER = 2u,       // traversal iteration bound reached
  ERR_QUEUE = 4u,      // a wavefront queue would overflow
  ERR_INDEX = 8u,      // an index read from memory is out of range
  ERR_BUILD = 16u,     // BVH refit did not reach the root
};

// the tree a render walks
constexpr int kTreeBinary = 0, kTreeWide4 = 1;

constexpr int kStackSize = 64;   // >= the depth of the LBVH (64-bit keys) and of the SAH tree (60)
constexpr int32_t kEmptyChild = 0x7FFFFFFF;  // unused slot of a 4-wide node
constexpr float kAmbient = 0.1f;
constexpr float kBgR = 0.2f, kBgG = 0.3f, kBgB = 0.5f;

struct DeviceScene {
  const float4* nodes;    // render nodes
  const float4* nodes4;   // 4-wide nodes (7 float4 each), the top n_top first
  const float4* prims;
  const float4* mats;
  const float4* lights;
  uint32_t n_prims, n_spheres, n_mats, n_lights;
  uint32_t n4, n_top;     // 4-wide nodes, of which the first n_top are staged in shared memory
};

// host-computed camera basis (double -> float)
struct CameraParams {
  float eye[3], right[3], up[3], fwd[3];
  float tan_x, tan_y, zc, half_sep;
  float sx, sy;                // 2 tan_x / W and 2 tan_y / H (pixel step in window units)
  uint32_t W, H;              // the whole image (it fixes the rays)
  uint32_t tiles_x, tiles_y;  // 8x4-pixel tiles per eye (of the traced rows)
  uint32_t y0, rows;          // the rows traced: y0 .. y0 + rows - 1 (0 and H for a whole image)
};

// stages of one render, in launch order
enum Stage : int {
  ST_CLEAR = 0,     // counter and accumulator clears
  ST_TRACE = 1,     // all rays: primary, shadow and mirror (one persistent kernel)
  ST_RESOLVE = 2,   // fixed-point sums to float RGB
  ST_WARP = 3,      // reprojection: forward warp and features
  ST_NET = 4,       // reprojection: retrace network
  ST_MASK = 5,      // reprojection: retrace mask and compaction
  ST_RETRACE = 6,   // reprojection: tracing the masked right pixels
  ST_COMPOSE = 7,   // reprojection: right image composition
  ST_COUNT = 8
};
constexpr int kMaxEvents = 24;

// reprojection scratch of a scene (per right-eye pixel unless noted)
struct ReprojBuffers {
  void* base = nullptr;
  uint64_t cap = 0;              // pixels per eye the buffers hold
  float* depth_L = nullptr;      // left G-buffer: view depth, normal (3), hit id
  float* normal_L = nullptr;
  float* refl_L = nullptr;       // reflectivity of the left primary hit (0 on a miss)
  uint32_t* id_L = nullptr;
  unsigned long long* zbuf = nullptr;  // forward-warp z-test keys
  __nv_bfloat16* feat16 = nullptr;     // network input, 16 channels
  uint8_t* hole = nullptr;
  float* warped = nullptr;       // warped left RGB (3)
  uint8_t* mask = nullptr;       // retrace mask
  uint32_t* plist = nullptr;     // masked pixels (global indices)
  uint32_t* count = nullptr;     // number of masked pixels
  float* prob = nullptr;         // network output
};

// scratch of one render (scene-owned, grown on demand)
struct Workspace {
  size_t bytes = 0;
  void* base = nullptr;
  uint32_t* accum = nullptr;     // 2*P*3 fixed-point colour sums
  float4* wq = nullptr;          // warp queues: n_warps x (cap_s + cap_r) x 3 float4
  float4* pool = nullptr;        // drain pools: shadow then mirror, cap_p entries of 3 float4 each
  uint32_t* pool_flag = nullptr; // per pool entry: epoch of the render that wrote it
  uint32_t cap_p = 0;            // entries per drain pool
  uint32_t cap_p_limit = 0;      // test hook: renders use at most this many (0 = cap_p)
  uint32_t epoch = 0;            // renders issued on this workspace (pool flags hold it)
  uint32_t* counters = nullptr;  // see Counter enum
  uint32_t cap_s = 0, cap_r = 0; // shadow / mirror entries per warp
  uint64_t n_warps = 0;          // warps the queues are sized for
  uint64_t cap_pixels = 0;       // 2*P the accumulators are sized for
  float4* frame = nullptr;       // frame buffers for rt_render_stereo_host
  size_t frame_bytes = 0;
  // rt_render_stereo_sequence: two device frame slots (each both images),
  // a copy stream and per slot the events "rendered" and "copied"
  float* seq_frame = nullptr;
  size_t seq_frame_bytes = 0;    // bytes of one slot
  cudaStream_t seq_copy = nullptr;
  cudaEvent_t seq_rendered[2] = {}, seq_copied[2] = {};
  uint32_t L = 0;
  ReprojBuffers rp;
  // stage timing (CUDA events on the render stream), see Stage
  bool profile = false;
  cudaEvent_t ev[kMaxEvents] = {};
  int ev_stage[kMaxEvents] = {};  // stage that ends at event k
  int n_ev = 0;
};

// counters block layout (uint32 each)
// (one 128-byte line each: the tile counter that every warp hammers, a flag
// that changes once, and the drain-pool counters)
enum Counter : int {
  C_TILE = 0,       // next primary tile
  C_SHADOW = 1,     // shadow rays enqueued (all warps)
  C_REFL = 2,       // mirror rays enqueued (all warps)
  C_TILES_OUT = 32, // set once a warp has found every tile handed out
  C_S_AVAIL = 64,   // drain pools: published entries not yet taken (int32), shadow
  C_R_AVAIL = 65,   // ... mirror
  C_S_HEAD = 66,    // drain pools: next entry to take / next entry to reserve, shadow
  C_S_TAIL = 67,
  C_R_HEAD = 68,    // ... mirror
  C_R_TAIL = 69,
  C_TOTAL = 96
};

struct RenderArgs {
  DeviceScene sc;
  CameraParams cam;
  uint32_t max_depth;
  float color_scale;       // fixed-point scale of the colour accumulators
  float* out_L;
  float* out_R;
  uint32_t* hit_L;
  uint32_t* hit_R;
  float* depth_L;
  float* depth_R;
  float* normal_L;         // G-buffer: primary-hit normal (facing the ray), 3 floats/pixel
  float* refl_L;           // G-buffer: reflectivity of the left primary hit (0 on a miss)
  float* normal_R;
  uint64_t* ray_counts;
  uint64_t* work;          // non-null => instrumented traversal
  uint32_t* err;           // device error word
  uint32_t eyes;           // 1 = left only, 2 = right only, 3 = both
  const uint32_t* plist;   // optional list of pixels to trace (eye*P + y*W + x)
  uint32_t plist_n;        // its length, or
  const uint32_t* plist_n_dev;  // its length in device memory (read by the kernel)
  bool resolve;            // write out_L/out_R from the sums (false: caller composes)
  int trace_stage;         // stage the tracing kernel is timed as (ST_TRACE or ST_RETRACE)
  int tree;                // kTreeBinary (sc.nodes) or kTreeWide4 (sc.nodes4)
  // several frames in one launch (0 or 1: just cam): n_frames cameras of the
  // same image size in host memory (frames[0] is cam); pixel ids, sums,
  // images and G-buffers then run over all frames, eye-major:
  // eye * (n_frames P) + frame * P + pixel
  uint32_t n_frames;
  const CameraParams* frames;
};
constexpr int kMaxFrames = 8;

// entry points implemented in the .cu files
cudaError_t build_lbvh(const float4* d_sph_in, const float* d_tri_in, uint32_t ns, uint32_t nt,
                       float4* d_nodes, float4* d_prims, uint64_t* d_keys, int32_t* d_parent,
                       void* d_tmp, size_t tmp_bytes, uint32_t* d_err, cudaStream_t st);
size_t lbvh_tmp_bytes(uint32_t n);
// *bad = 1 if a record is invalid: a value that is not finite, a radius not
// above 0, a material not below n_mats (raw records; *bad is 0 before)
cudaError_t check_prims(const float4* d_sph_in, const float* d_tri_in, uint32_t ns, uint32_t nt, uint32_t n_mats,
                        uint32_t* bad, cudaStream_t st);
size_t sah_tmp_bytes(uint32_t n);
// binned-SAH binary tree over the leaves of the LBVH (nodes, parent): same
// node layout and leaf slots, root 0; synchronises st about once
cudaError_t build_sah_tree(const float4* lbvh_nodes, const int32_t* parent, uint32_t n,
                           float4* out, void* tmp, uint32_t* err, cudaStream_t st);
// the render nodes of a binary tree over n primitives
cudaError_t render_nodes(const float4* nodes, uint32_t n, float4* out, cudaStream_t st);
size_t bvh4_tmp_bytes(uint32_t n);
void set_sah_slicing(bool on);   // slice the top levels of the SAH build (default on)
cudaError_t inner_parents(const float4* nodes, uint32_t n, int32_t* parent, cudaStream_t st);
cudaError_t build_bvh4(const float4* nodes, const int32_t* parent, uint32_t n, int top_depth,
                       float4* nodes4, uint32_t* counts_dev, void* tmp, cudaStream_t st);
cudaError_t render(const RenderArgs& a, Workspace& ws, cudaStream_t st);
// stage timing: start a profiled call (resets the event list) / mark the end of a stage
void profile_begin(Workspace& ws, cudaStream_t st);
void profile_mark(Workspace& ws, int stage, cudaStream_t st);
// Launch of a kernel that calls after_previous(): it is put on the SMs as the
// kernel before it in the stream drains instead of after that has ended and
// waits there (programmatic dependent launch), which hides its launch: 1 to 2 us
// a kernel in the training step and the builds. Before that wait, which covers
// all earlier work of the stream, it touches no memory that the kernel before may
// write or read. A kernel that allocates TMEM does so before the call: the next
// kernel's blocks come only when every block of this one has its own.
// It overlaps the kernel before it and no earlier one. What an earlier kernel of
// its chain writes is therefore no constant of its run: it is read with ordinary
// (or ld.cg) loads through pointers without __restrict__, which stay behind the
// wait, never with __ldg or through const __restrict__, which promise a value that
// nobody writes while the kernel is resident and need not stay behind the wait.
// The first kernel of a chain reads the caller's data so too. The read-only path
// is for what was complete before the chain: a scene's trees and primitives in a
// render, the raw records from a build's second kernel on.
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                         A&&... args) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &attr;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
// Launches of launch_after one after another, none after one that failed: a later
// kernel would index by what the failed one did not write (its keys, jobs, counts).
struct Chain {
  cudaStream_t st;
  cudaError_t error = cudaSuccess;
  template <typename... P, typename... A>
  void then(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, A&&... args) {
    if (error == cudaSuccess) error = launch_after(kernel, grid, block, smem, st, std::forward<A>(args)...);
  }
  // the first error, which the runtime then no longer reports
  cudaError_t end() const {
    const cudaError_t last = cudaGetLastError();
    return error != cudaSuccess ? error : last;
  }
};
#ifdef __CUDACC__
// waits for all earlier work of the stream; lets the next kernel be put in place
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif
int num_sms();
int render_grid();      // persistent blocks of the render kernel
int render_threads();   // threads per block of the render kernel
int treelet_depth();    // 4-wide levels numbered first for shared-memory staging

// reprojection (reproj.cu)
cudaError_t reproj_warp(const float* depth_L, const float* normal_L, const uint32_t* id_L,
                        const float* rgb_L, const float* refl_L, uint32_t W, uint32_t H, float f_px, float eye_sep,
                        float convergence, unsigned long long* zbuf, __nv_bfloat16* feat16,
                        float* feat32, uint8_t* hole, float* warped, cudaStream_t st);
cudaError_t reproj_labels(const uint8_t* hole, const float* warped, const float* full_R, uint32_t P,
                          float thr, float* label, cudaStream_t st);
cudaError_t reproj_mask(const uint8_t* hole, const float* prob, uint32_t P, float threshold,
                        uint8_t* mask, uint32_t* plist, uint32_t* count, cudaStream_t st);
cudaError_t reproj_compose(const uint8_t* mask, const uint32_t* accum_R, const float* warped,
                           uint32_t P, float inv_scale, float* out_R, cudaStream_t st);

// retrace network (nn.cu)
namespace nn {
constexpr uint32_t kParams = 21697;
size_t packed_fwd_elems(int l);
size_t packed_bwd_elems(int l);
cudaError_t pack_weights(const float* params, __nv_bfloat16* const wf[4], __nv_bfloat16* const wb[4],
                         cudaStream_t st);
// forward / forward_fp8: n_img feature maps of W x H pixels each, stacked
// image after image, in one launch; act (or null): BF16 planar maps that
// receive the three hidden activations
cudaError_t forward(const __nv_bfloat16* feat16, const float* params, __nv_bfloat16* const wf[4],
                    __nv_bfloat16* const act[3], float* prob, uint32_t W, uint32_t H, uint32_t* err,
                    cudaStream_t st, uint32_t n_img = 1);
// buffers of a training step on maps of P pixels
struct TrainBuffers {
  float *params, *m, *v;             // kParams each
  __nv_bfloat16* wf[4];              // packed weights, updated with the parameters
  __nv_bfloat16* wb[4];
  __nv_bfloat16* act[3];             // hidden activations, planar
  __nv_bfloat16* dz[3];              // data gradients of layers 3, 2, 1, planar
  __nv_bfloat16* g8;                 // BCE gradient, 8 channels per pixel
  uint32_t* mask;                    // ReLU masks of the hidden layers, a word per pixel each
  float* wpart;                      // wgrad_part_floats partial sums
  float* loss_part;                  // loss_parts partial sums of the loss
  float* loss;                       // sum of the pixels' losses
};
size_t wgrad_part_floats(uint32_t W, uint32_t H);
int loss_parts();
// forward, backward and (lr > 0) the Adam update number `step`; grads (or
// null): kParams floats, device
cudaError_t train_step(const __nv_bfloat16* feat16, const float* label, const TrainBuffers& t, uint32_t W,
                       uint32_t H, float lr, uint32_t step, float* grads, uint32_t* err, cudaStream_t st);
size_t packed_fp8_bytes(int l);
cudaError_t pack_weights_fp8(const float* params, const float* const scale[3], uint8_t* const w8[3],
                             cudaStream_t st);
cudaError_t forward_fp8(const __nv_bfloat16* feat16, const float* params, __nv_bfloat16* const wf[4],
                        uint8_t* const w8[3], const float* const inv[3], const float act_scale[3],
                        float* prob, uint32_t W, uint32_t H, uint32_t* err, cudaStream_t st,
                        uint32_t n_img = 1);
cudaError_t activation_amax(const __nv_bfloat16* const act[3], uint64_t P, unsigned* amax3,
                            cudaStream_t st);
}  // namespace nn

}  // namespace rt

// the opaque scene of the C-ABI
struct rt_scene {
  int device = 0;
  uint32_t ns = 0, nt = 0, n = 0, nm = 0, nl = 0;
  void* block = nullptr;       // persistent device allocation
  float4* nodes = nullptr;
  float4* nodes_sah = nullptr; // binary tree rebuilt with the SAH over the same leaves (sah.cu)
  float4* render_sah = nullptr;   // render nodes of the SAH tree
  // allocated and made when first chosen (rt_scene_set_traversal):
  float4* render_lbvh = nullptr;  // render nodes of the LBVH
  float4* nodes4 = nullptr;       // the 4-wide tree
  uint32_t n4 = 0, n_top = 0;
  int tree = RT_TREE_SAH;      // the tree renders walk (rt_scene_set_traversal)
  float4* prims = nullptr;
  float4* mats = nullptr;
  float4* lights = nullptr;
  uint64_t* keys = nullptr;
  int32_t* parent = nullptr;
  uint32_t* err = nullptr;
  uint32_t* h_err = nullptr;   // pinned
  float color_scale = 1.f;
  rt::Workspace ws;
};

// error message plumbing and host helpers (rt_api.cu)
void rt_set_error(const std::string& msg);
namespace rt {
int fail(int code, const std::string& msg);
int cuda_fail(cudaError_t e, const char* what);
int ensure_workspace(const rt_scene* sc, uint32_t W, uint32_t H);
int make_render_args(const rt_scene* scene, const rt_camera* cam, float eye_sep, float convergence,
                     uint32_t W, uint32_t H, uint32_t max_depth, RenderArgs& a);
}  // namespace rt
