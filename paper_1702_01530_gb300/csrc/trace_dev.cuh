// Device-side tracing primitives shared by the single-pair renderer
// (trace.cu) and the batched renderer (batch.cu): compile-time knobs, vector
// helpers, the ray-sphere and Moller-Trumbore tests, the BVH traversals and
// the fixed-point colour accumulation. Everything sits in an anonymous
// namespace, so each translation unit owns its copy.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "rt_internal.cuh"

namespace rt {
namespace {

// Tuning knobs (compile-time; GB300, SAH tree, each knob's times from one run, so
// they compare with one another and not with another knob's):
// RT_MIN_BLOCKS = minimum resident blocks per SM requested from the register
// allocator (0 = no request). 9 measured best: the default walk fits 56 registers
// with 8 bytes spilled outside its loop, 36 warps per SM. Pair of 257k blob
// primitives at 1080p / of 10 primitives at 1080p / of a terrain of 2.1 M triangles
// at 4K, ms, with 6, 7, 8, 9, 10 blocks (48 registers, spills in the shading code):
// 1.057, 1.041, 1.036, 1.015, 1.045 / 0.175, 0.174, 0.174, 0.174, 0.199 / 14.67,
// 14.31, 14.19, 13.49, 13.91.
#ifndef RT_MIN_BLOCKS
#define RT_MIN_BLOCKS 9
#endif
constexpr int kStack4 = 100;   // 3 pushes per 4-wide level, <= 33 levels
// shared-memory treelet: 4-wide levels staged per block (RT_TREELET_DEPTH
// levels, at most 1 + 4 + 16 + 64 = 85 nodes for depth 4)
#ifndef RT_TREELET_DEPTH
#define RT_TREELET_DEPTH 2
#endif
constexpr int kMaxTopBytes = 85 * 7 * 16;
// 4-wide closest-hit traversal pushes the other hit children farthest first
#ifndef RT_ORDERED_PUSH
#define RT_ORDERED_PUSH 0
#endif
// RT_FAST_RCP = 1: ray reciprocals and the triangle determinant's reciprocal
// by the approximate hardware reciprocal (rcp.approx.f32, at most 1 ulp off)
// instead of the correctly rounded one (whose slow path also cost the render
// kernel 24 bytes of register spills), the robust slab factor widened to
// match, and pixel positions by multiplication with host-computed scales
// instead of two divisions per primary ray: 1.050 -> 1.020 ms per 1080p blob
// pair, 0.222 -> 0.214 ms for the 10-primitive scene; on by default
#ifndef RT_FAST_RCP
#define RT_FAST_RCP 1
#endif
// RT_PRIMARY_STORE = 1: a pixel's primary ray stores its contribution
// (store_first) and the colour sums are not cleared before a render; 0: every
// contribution is an atomic add onto sums cleared by a memset. Same images;
// 1.018 -> 1.012 ms per 1080p blob pair, 0.212 -> 0.182 ms for the
// 10-primitive scene at 1080p.
#ifndef RT_PRIMARY_STORE
#define RT_PRIMARY_STORE 1
#endif
constexpr int kThreads = 128;
// conservative slab exit (Ize 2013): 1 + 2 gamma_3 with correctly rounded
// reciprocals, 1 + 2 gamma_5 when each may be one ulp off
constexpr float kRobust = RT_FAST_RCP ? 1.0000006f : 1.00000036f;

__device__ __forceinline__ float fmin3(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

struct V3 { float x, y, z; };
__device__ __forceinline__ V3 v3(float x, float y, float z) { return {x, y, z}; }
__device__ __forceinline__ V3 operator+(V3 a, V3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ V3 operator-(V3 a, V3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ V3 operator*(V3 a, float s) { return {a.x * s, a.y * s, a.z * s}; }
__device__ __forceinline__ float dot(V3 a, V3 b) { return fmaf(a.x, b.x, fmaf(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ V3 cross(V3 a, V3 b) {
  return {fmaf(a.y, b.z, -a.z * b.y), fmaf(a.z, b.x, -a.x * b.z), fmaf(a.x, b.y, -a.y * b.x)};
}
__device__ __forceinline__ V3 normalize(V3 a) { return a * rsqrtf(dot(a, a)); }
__device__ __forceinline__ V3 xyz(float4 f) { return {f.x, f.y, f.z}; }

__device__ __forceinline__ float rcp_f(float x) {
#if RT_FAST_RCP
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return __frcp_rn(x);
#endif
}

__device__ __forceinline__ float safe_rcp(float x) {
  const float tiny = 8.271806e-25f;  // 2^-80
  return rcp_f(fabsf(x) > tiny ? x : copysignf(tiny, x));
}

struct WorkCount { uint32_t inner, sphere, tri; };

// two FP32 values in one 64-bit register, and fma on both in one instruction
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Ray-sphere (d unit length). Stable form: disc = r^2 - |oc - b d|^2 keeps
// precision when the ray passes far from the centre relative to r; the two
// roots are q and c/q with q = -b - sign(b) sqrt(disc).
__device__ __forceinline__ bool hit_sphere(float4 p0, float r, V3 o, V3 d, float& t) {
  V3 oc = o - xyz(p0);
  float b = dot(oc, d);
  V3 f = oc - d * b;
  float r2 = r * r;
  float disc = r2 - dot(f, f);
  float cc = dot(oc, oc) - r2;
  float sq = sqrtf(fmaxf(disc, 0.f));
  float q = -b - copysignf(sq, b);
  float t0 = __fdividef(cc, q), t1 = q;
  float tn = fminf(t0, t1), tf = fmaxf(t0, t1);
  t = tn > 0.f ? tn : tf;
  return disc >= 0.f && t > 0.f;
}

// Moller-Trumbore, two-sided, edges inclusive (branch-free acceptance). The
// barycentric bounds are widened by kEdge so that a ray through the shared
// edge of two triangles cannot slip between them when FP32 rounding puts it
// just outside both (the band lies far inside the oracle's near-tie margin).
constexpr float kEdge = 1e-6f;
__device__ __forceinline__ bool hit_tri(float4 p0, float4 p1, float4 p2, V3 o, V3 d, float& t) {
  V3 e1 = xyz(p1), e2 = xyz(p2);
  V3 pv = cross(d, e2);
  float det = dot(e1, pv);
  float inv = rcp_f(det);
  V3 tv = o - xyz(p0);
  float u = dot(tv, pv) * inv;
  V3 qv = cross(tv, e1);
  float v = dot(d, qv) * inv;
  t = dot(e2, qv) * inv;
  return det != 0.f && u >= -kEdge && v >= -kEdge && u + v <= 1.f + kEdge && t > 0.f;
}

// BVH traversal. ANY = any-hit with t < tmax (returns true if blocked);
// otherwise closest hit with t <= t_best (equal t -> lower id), returns
// whether anything was hit.
//
// Nodes hold each child box as centre c and half extent e (render_nodes): per
// axis t_c = (c - o) / d, and the ray is inside the slab from t_c - e |1/d| to
// t_c + e |1/d|, which needs no minimum and maximum to order the two planes;
// x and y of a child share one two-wide fma. A child takes 6 fma instructions
// (3 of them two-wide) and 4 three-input minima and maxima, against 6 fma and
// 10 minima and maxima with the box as two corners: 721 -> 656 M warp
// instructions for the 1080p blob pair, 0.987 -> 0.946 ms; 4K frame of a
// 2.1 M-triangle terrain 12.34 -> 11.25 ms. What bounds it now is the latency of
// the node loads (5.0 of 13 stalled warps per issue) and the L1 (72 % of its
// throughput): a node as two 32-byte loads (11.48 ms), 10 blocks of 48 registers
// (0.966 / 11.46 ms) and leaving the triangle test after its first failed bound
// (0.956 / 11.29 ms) were slower.
template <bool ANY, bool COUNT>
__device__ __forceinline__ bool traverse(const DeviceScene& sc, V3 o, V3 d, float tmax,
                                         float& t_best, uint32_t& id_best, uint32_t& k_best,
                                         WorkCount& wc, uint32_t* err) {
  const V3 idir = v3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
  const f32x2 id_xy = pack2(idir.x, idir.y), od_xy = pack2(-o.x * idir.x, -o.y * idir.y);
  const f32x2 ai_xy = pack2(fabsf(idir.x), fabsf(idir.y)), na_xy = pack2(-fabsf(idir.x), -fabsf(idir.y));
  const float od_z = -o.z * idir.z, ai_z = fabsf(idir.z);
  int32_t stack[kStackSize];
  int sp = 0;
  const uint32_t n = sc.n_prims;
  int32_t node = n == 1 ? ~0 : 0;
  const uint32_t it_max = 2u * n + 64u;
  float tcur = ANY ? tmax : t_best;
  bool any = false;
  for (uint32_t it = 0;; ++it) {
    if (node >= 0) {
      // the iteration bound is checked on node visits only: a leaf visit
      // pushes nothing, so a run of them ends with the (bounded) stack
      if (it >= it_max || (uint32_t)node >= n - 1) {
        atomicOr(err, it >= it_max ? ERR_ITER : ERR_INDEX);
        break;
      }
      const float4* np = sc.nodes + 4 * (size_t)node;
      const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2*>(np));       // (c.xy, e.xy) of child 0
      const ulonglong2 b = __ldg(reinterpret_cast<const ulonglong2*>(np + 1));   // ... of child 1
      const float4 c = __ldg(np + 2);                                            // c.z, e.z of both
      const int2 e = __ldg(reinterpret_cast<const int2*>(np + 3));               // the children
      if (COUNT) wc.inner++;
      const f32x2 t0 = fma2(a.x, id_xy, od_xy), t1 = fma2(b.x, id_xy, od_xy);
      const float z0 = fmaf(c.x, idir.z, od_z), z1 = fmaf(c.z, idir.z, od_z);
      float i0x, i0y, o0x, o0y, i1x, i1y, o1x, o1y;
      unpack2(fma2(a.y, na_xy, t0), i0x, i0y);
      unpack2(fma2(a.y, ai_xy, t0), o0x, o0y);
      unpack2(fma2(b.y, na_xy, t1), i1x, i1y);
      unpack2(fma2(b.y, ai_xy, t1), o1x, o1y);
      const float in0 = fmax3(i0x, i0y, fmaxf(fmaf(-c.y, ai_z, z0), 0.f));
      const float out0 = fmin3(o0x, o0y, fminf(fmaf(c.y, ai_z, z0), tcur));
      const float in1 = fmax3(i1x, i1y, fmaxf(fmaf(-c.w, ai_z, z1), 0.f));
      const float out1 = fmin3(o1x, o1y, fminf(fmaf(c.w, ai_z, z1), tcur));
      const bool hit0 = in0 <= out0 * kRobust;
      const bool hit1 = in1 <= out1 * kRobust;
      if (hit0 | hit1) {
        const bool second = hit1 && (!hit0 || in1 < in0);
        node = second ? e.y : e.x;
        if (hit0 & hit1) {
          if (sp >= kStackSize) { atomicOr(err, ERR_STACK); break; }
          stack[sp++] = second ? e.x : e.y;
        }
        continue;
      }
    } else {
      const uint32_t k = (uint32_t)~node;
      if (k >= n) { atomicOr(err, ERR_INDEX); break; }
      const float4* pp = sc.prims + 3 * (size_t)k;
      const float4 p0 = __ldg(pp), p1 = __ldg(pp + 1);
      const uint32_t id = __float_as_uint(p0.w);
      float t;
      bool h;
      if (id < sc.n_spheres) {
        if (COUNT) wc.sphere++;
        h = hit_sphere(p0, p1.x, o, d, t);
      } else {
        if (COUNT) wc.tri++;
        h = hit_tri(p0, p1, __ldg(pp + 2), o, d, t);
      }
      if (ANY) {
        if (h && t < tmax) { any = true; break; }
      } else if (h && (t < tcur || (t == tcur && id < id_best))) {
        tcur = t;
        id_best = id;
        k_best = k;
        any = true;
      }
    }
    if (sp == 0) break;
    node = stack[--sp];
  }
  if (!ANY) t_best = tcur;
  return any;
}

// 4-wide traversal: one fetch of 7 float4 tests four child boxes; the
// nearest hit child is visited next and the other hit children are pushed.
// The first sc.n_top nodes are read from the shared-memory copy `top`.
template <bool ANY>
__device__ __forceinline__ bool traverse4(const DeviceScene& sc, const float4* top, V3 o, V3 d,
                                          float tmax, float& t_best, uint32_t& id_best,
                                          uint32_t& k_best, uint32_t* err) {
  const V3 idir = v3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
  const V3 od = v3(-o.x * idir.x, -o.y * idir.y, -o.z * idir.z);
  const V3 ai = v3(fabsf(idir.x), fabsf(idir.y), fabsf(idir.z));
  int32_t stack[kStack4];
  int sp = 0;
  const uint32_t n = sc.n_prims;
  int32_t node = n == 1 ? ~0 : 0;
  const uint32_t it_max = 2u * n + 64u;
  float tcur = ANY ? tmax : t_best;
  bool any = false;
  for (uint32_t it = 0;; ++it) {
    if (it >= it_max) { atomicOr(err, ERR_ITER); break; }
    if (node >= 0) {
      if ((uint32_t)node >= sc.n4) { atomicOr(err, ERR_INDEX); break; }
      float4 cx, ex, cy, ey, cz, ez, cc;
      if ((uint32_t)node < sc.n_top) {             // shared-memory treelet
        const float4* np = top + 7 * node;
        cx = np[0]; ex = np[1]; cy = np[2]; ey = np[3]; cz = np[4]; ez = np[5]; cc = np[6];
      } else {                                     // read-only global path
        const float4* np = sc.nodes4 + 7 * (size_t)node;
        cx = __ldg(np); ex = __ldg(np + 1); cy = __ldg(np + 2); ey = __ldg(np + 3);
        cz = __ldg(np + 4); ez = __ldg(np + 5); cc = __ldg(np + 6);
      }
      float tin[4];
      bool hit[4];
      // the binary walk's box test, so that every tree takes the same leaves
#define RT_SLAB(c, F)                                                                         \
      {                                                                                       \
        const float tx = fmaf(cx.F, idir.x, od.x), ty = fmaf(cy.F, idir.y, od.y),             \
                    tz = fmaf(cz.F, idir.z, od.z);                                            \
        tin[c] = fmax3(fmaf(-ex.F, ai.x, tx), fmaf(-ey.F, ai.y, ty),                          \
                       fmaxf(fmaf(-ez.F, ai.z, tz), 0.f));                                    \
        const float tout = fmin3(fmaf(ex.F, ai.x, tx), fmaf(ey.F, ai.y, ty),                  \
                                 fminf(fmaf(ez.F, ai.z, tz), tcur));                          \
        hit[c] = tin[c] <= tout * kRobust;                                                    \
      }
      RT_SLAB(0, x)
      RT_SLAB(1, y)
      RT_SLAB(2, z)
      RT_SLAB(3, w)
#undef RT_SLAB
      const int32_t ch[4] = {__float_as_int(cc.x), __float_as_int(cc.y), __float_as_int(cc.z),
                             __float_as_int(cc.w)};
#pragma unroll
      for (int c = 0; c < 4; ++c) hit[c] = hit[c] && ch[c] != kEmptyChild;  // unused slots
      int bi = -1;
      float best = INFINITY;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (hit[c] && (ANY ? bi < 0 : tin[c] < best)) { best = tin[c]; bi = c; }
      if (bi >= 0) {
        // the other hit children, farthest pushed first (closest-hit rays)
        float t4[4];
        int32_t c4[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          t4[c] = (hit[c] && c != bi) ? tin[c] : -INFINITY;
          c4[c] = ch[c];
        }
        if (!ANY && RT_ORDERED_PUSH) {
#define RT_CAS(i, j)                                                              \
          if (t4[i] < t4[j]) {                                                    \
            const float tt = t4[i]; t4[i] = t4[j]; t4[j] = tt;                    \
            const int32_t cx = c4[i]; c4[i] = c4[j]; c4[j] = cx;                  \
          }
          RT_CAS(0, 1) RT_CAS(2, 3) RT_CAS(0, 2) RT_CAS(1, 3) RT_CAS(1, 2)
#undef RT_CAS
        }
        bool overflow = false;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (t4[c] > -INFINITY) {
            if (sp < kStack4) stack[sp++] = c4[c];
            else overflow = true;
          }
        if (overflow) { atomicOr(err, ERR_STACK); break; }
        node = ch[bi];
        continue;
      }
    } else {
      const uint32_t k = (uint32_t)~node;
      if (k >= n) { atomicOr(err, ERR_INDEX); break; }
      const float4* pp = sc.prims + 3 * (size_t)k;
      const float4 p0 = __ldg(pp), p1 = __ldg(pp + 1);
      const uint32_t id = __float_as_uint(p0.w);
      float t;
      bool h;
      if (id < sc.n_spheres) h = hit_sphere(p0, p1.x, o, d, t);
      else h = hit_tri(p0, p1, __ldg(pp + 2), o, d, t);
      if (ANY) {
        if (h && t < tmax) { any = true; break; }
      } else if (h && (t < tcur || (t == tcur && id < id_best))) {
        tcur = t;
        id_best = id;
        k_best = k;
        any = true;
      }
    }
    if (sp == 0) break;
    node = stack[--sp];
  }
  if (!ANY) t_best = tcur;
  return any;
}

// The instrumented (COUNT) walk and the binary renders use the binary tree
// in sc.nodes (the SAH tree, or the LBVH whose node visits define the
// algorithmic work); a 4-wide render walks the 4-wide tree (the same leaves,
// the same hits).
// TREE: kTreeBinary (sc.nodes) or kTreeWide4 (sc.nodes4 = the 4-wide tree)
template <bool ANY, bool COUNT, int TREE>
__device__ __forceinline__ bool trace_ray(const DeviceScene& sc, const float4* top, V3 o, V3 d,
                                          float tmax, float& t_best, uint32_t& id_best,
                                          uint32_t& k_best, WorkCount& wc, uint32_t* err) {
  if (TREE == kTreeWide4 && !COUNT) return traverse4<ANY>(sc, top, o, d, tmax, t_best, id_best, k_best, err);
  return traverse<ANY, COUNT>(sc, o, d, tmax, t_best, id_best, k_best, wc, err);
}

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31; }

// Primary ray of pixel (px, py) of one eye (0 = left, 1 = right): both eyes
// aim at the same point Q of the window on the convergence plane.
__device__ __forceinline__ void primary_ray(const CameraParams& cam, uint32_t px, uint32_t py,
                                            uint32_t eye, V3& o, V3& d) {
#if RT_FAST_RCP
  const float nx = fmaf((float)px + 0.5f, cam.sx, -cam.tan_x);
  const float ny = fmaf(-((float)py + 0.5f), cam.sy, cam.tan_y);
#else
  const float nx = (2.f * ((float)px + 0.5f) / (float)cam.W - 1.f) * cam.tan_x;
  const float ny = (1.f - 2.f * ((float)py + 0.5f) / (float)cam.H) * cam.tan_y;
#endif
  const V3 E = v3(cam.eye[0], cam.eye[1], cam.eye[2]);
  const V3 Rt = v3(cam.right[0], cam.right[1], cam.right[2]);
  const V3 U = v3(cam.up[0], cam.up[1], cam.up[2]);
  const V3 F = v3(cam.fwd[0], cam.fwd[1], cam.fwd[2]);
  const V3 Q = E + (F + Rt * nx + U * ny) * cam.zc;
  o = E + Rt * (eye ? cam.half_sep : -cam.half_sep);
  d = normalize(Q - o);
}

// Surface at the closest hit (primitive slot k, id): hit point, geometric
// normal turned against the ray, material, and the secondary-ray offset
// eps = 1e-4 max(1, |p|_inf).
__device__ __forceinline__ void hit_surface(const float4* prims, const float4* mats,
                                            uint32_t n_spheres, uint32_t n_mats, uint32_t k,
                                            uint32_t id, V3 o, V3 d, float t, uint32_t* err, V3& p,
                                            V3& nrm, float4& mat, float& eps) {
  const float4* pp = prims + 3 * (size_t)k;
  const float4 p0 = __ldg(pp), p1 = __ldg(pp + 1);
  p = o + d * t;
  uint32_t mid = __float_as_uint(p1.w);
  if (id < n_spheres) nrm = (p - xyz(p0)) * (1.f / p1.x);
  else nrm = normalize(cross(xyz(p1), xyz(__ldg(pp + 2))));
  if (dot(nrm, d) > 0.f) nrm = nrm * -1.f;
  if (mid >= n_mats) { atomicOr(err, ERR_INDEX); mid = 0; }
  mat = __ldg(mats + mid);
  eps = 1e-4f * fmaxf(1.f, fmax3(fabsf(p.x), fabsf(p.y), fabsf(p.z)));
}

// Shadow ray from o2 towards light lp: unit direction lh, distance ld, and
// n.l scaled by the light's intensity and (1 - reflectivity); returns
// whether the light faces the surface (n.l > 0).
__device__ __forceinline__ bool light_ray(float4 lp, V3 o2, V3 nrm, float refl, V3& lh, float& ld,
                                          float& ndl) {
  const V3 lv = xyz(lp) - o2;
  const float inv = rsqrtf(dot(lv, lv));
  ld = dot(lv, lv) * inv;
  lh = lv * inv;
  ndl = dot(nrm, lh);
  const bool emit = ndl > 0.f;
  ndl *= lp.w * (1.f - refl);
  return emit;
}

// Mirror direction of d about nrm, renormalised.
__device__ __forceinline__ V3 mirror_dir(V3 d, V3 nrm) {
  return normalize(d - nrm * (2.f * dot(d, nrm)));
}

__device__ __forceinline__ void accumulate(uint32_t* acc, uint32_t pix, float r, float g, float b,
                                           float scale) {
  uint32_t* p = acc + 3 * (size_t)pix;
  atomicAdd(p + 0, __float2uint_rn(r * scale));
  atomicAdd(p + 1, __float2uint_rn(g * scale));
  atomicAdd(p + 2, __float2uint_rn(b * scale));
}

// The first contribution to a pixel: its primary ray's, stored rather than
// added, so the sums need no clearing before the launch. Every later
// contribution (shadow and mirror rays, all spawned by this ray after this
// store, on this lane or handed on through a release store) is an atomic add
// that the hand-over orders after it.
__device__ __forceinline__ void store_first(uint32_t* acc, uint32_t pix, float r, float g, float b,
                                            float scale) {
  uint32_t* p = acc + 3 * (size_t)pix;
  p[0] = __float2uint_rn(r * scale);
  p[1] = __float2uint_rn(g * scale);
  p[2] = __float2uint_rn(b * scale);
}

}  // namespace
}  // namespace rt
