// rr_trace.cu -- wavefront ray tracing of a batch of polar scans.
//
// Per batch: raygen -> { trace -> shade } x max_bounces -> image
// A batch is one or more scans of the same scene, each with its own pose and
// sensor model (ScanDesc); every ray carries the index of its scan, so scans
// of uneven ray counts and bounce limits share every launch.
//   raygen  Sec. III-A, Eq. 2: N_s rays per azimuth beam from the D3 cone.
//   trace   closest hit through the LBVH (watertight ray/triangle test of
//           Woop, Benthin, Wald, JCGT 2013) and, for multipath, the
//           visibility test of the air-path return toward the sensor.
//   shade   Sec. III-A: Fresnel split E0 = E1 + E2, Snell refraction,
//           attenuation in lossy media, traveled-path and air-path returns
//           through the beam window of the material lobe (Eq. 3-5), and the
//           reflected / refracted children.  Children and return records are
//           compacted stably (single pass, decoupled look-back over tiles of
//           256 or 512 rays), so every queue and every bounce's record list stays
//           in (azimuth, ray) order.
//
// All kernels are persistent: the grid is a multiple of the SM count and
// reads the queue length from device memory, so a whole batch is a fixed
// sequence of launches with no host round trip between bounces.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "rr_host.h"

namespace rr {

constexpr int kShadeTile = 256;   // rays of the smallest shading tile

// ---------------------------------------------------------------------------
// beam axis angle 2 pi a / n with an exact quadrant reduction; returns (cos, sin)
__device__ __forceinline__ float2 beam_angle(uint32_t a, uint32_t n) {
  const uint32_t m = 4u * a;
  const uint32_t q = (m + n / 2u) / n;              // nearest quarter turn
  const int rem = (int)m - (int)(q * n);            // in [-n/2, n/2]
  float s, c;
  sincospif(0.5f * (float)rem / (float)n, &s, &c);
  switch (q & 3u) {
    case 0: return make_float2(c, s);
    case 1: return make_float2(-s, c);
    case 2: return make_float2(-c, -s);
    default: return make_float2(s, -c);
  }
}

// world direction of beam az's axis for a scan
__device__ __forceinline__ float3 beam_axis(const ScanDesc* sd, uint32_t az) {
  const float2 cs = beam_angle(az, __ldg(&sd->dims.x));
  float se, ce;
  sincosf(__ldg(&sd->beam.z), &se, &ce);
  return qrot(__ldg(&sd->quat), make_float3(ce * cs.x, ce * cs.y, se));
}

// Eq. 2: sigma = (b / 2) / (sqrt(2) erfinv(P))
__device__ __forceinline__ float d3_sigma(float b, float P) {
  return b > 0.0f ? 0.5f * b / (1.41421356237309515f * erfinvf(P)) : 0.0f;
}

// ---------------------------------------------------------------------------
// raygen: ray (az, k) of the D3 cone of its scan, energy 1 / N_s
__global__ void k_raygen(ScanArgs a) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    ScanCounters* c = a.ctr;
    for (int b = 0; b <= (int)RR_MAX_BOUNCES; ++b) {
      c->count[b] = 0;
      c->rec_start[b] = 0;
      c->seg_start[b] = 0;
    }
    for (int b = 0; b < (int)RR_MAX_BOUNCES; ++b) {
      c->trace_ticket[b] = 0;
      c->shade_ticket[b] = 0;
      c->vis_count[b] = 0;
      c->vis_ticket[b] = 0;
    }
    c->count[0] = a.n_rays0;
    c->stat_scans += (unsigned long long)a.n_scans;
  }
  if (i >= a.n_rays0) return;
  const uint32_t scan = owner_of(a.ray0, a.n_scans, i);
  const ScanDesc* sd = a.desc + scan;
  const uint32_t ns = __ldg(&sd->dims.y);
  const uint32_t local = i - __ldg(&a.ray0[scan]);
  const uint32_t az_l = local / ns, k = local - az_l * ns;
  const uint32_t az = __ldg(&sd->offs.w) + az_l;   // a scan may trace a range of the azimuths
  const float4 beam = __ldg(&sd->beam);
  const uint4 x = draw(__ldg(&sd->rng), az, k, 0u);
  const float u0 = u01(x.x), u1 = u01(x.y), u2 = u01(x.z);
  const float gauss = sqrtf(-2.0f * logf(u0)) * cospif(2.0f * u1);
  const float r = d3_sigma(beam.x, beam.y) * gauss;
  float sw, cw;
  sincospif(2.0f * u2 - 1.0f, &sw, &cw);      // omega = pi (2 u2 - 1)
  const float daz = r * cw, dinc = r * sw * __ldg(&sd->ext.x);   // elliptic beams: inclination stretched
  const float2 ph = beam_angle(az, __ldg(&sd->dims.x));
  float sd_, cd;
  sincosf(daz, &sd_, &cd);
  const float ca = ph.x * cd - ph.y * sd_, sa = ph.y * cd + ph.x * sd_;   // cos, sin of phi + daz
  float si, ci;
  sincosf(beam.z + dinc, &si, &ci);
  const float3 d = normalize(qrot(__ldg(&sd->quat), make_float3(ci * ca, ci * sa, si)));
  const bool masked = a.mask != nullptr && a.mask[i] != 0;
  const float4 pr = __ldg(&sd->pos_rmax);
  RayRec ray;
  ray.o_L = make_float4(pr.x, pr.y, pr.z, 0.0f);
  ray.d_E = make_float4(d.x, d.y, d.z, 1.0f / (float)ns);
  ray.meta = make_uint4(kNone, (az << 16) | k, masked ? 0x80000000u : 0u, (scan << 16) | kAir);
  a.rays[0][i] = ray;
}

// ---------------------------------------------------------------------------
// traversal
struct WoopRay {
  float3 o;            // origin in the frame (kx, ky, kz)
  float Sx, Sy, Sz;    // shear: d_kx / d_kz, d_ky / d_kz, 1 / d_kz
  uint32_t rot;        // the rotated triangle copy whose coordinates are in that frame
};

// The frame's third axis kz is the dominant axis of d; kx and ky follow it
// cyclically (kx = kz + 1, ky = kz + 2 mod 3), which is the triangle copy
// rotated by (kz + 1) mod 3.  Woop et al. swap kx and ky when d_kz < 0 to keep
// the winding; the test below accepts both windings, and swapping the two
// axes negates U, V, W, det and T exactly (each is a difference of the same
// rounded products, or a sum of such terms), so t and the decision are the
// same bit for bit without the swap.
__device__ __forceinline__ WoopRay make_woop(float3 o, float3 d) {
  WoopRay w;
  const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
  const uint32_t kz = (ax >= ay && ax >= az) ? 0u : (ay >= az ? 1u : 2u);
  w.rot = kz == 2u ? 0u : kz + 1u;
  const float3 dr = tri_rotate(d, w.rot);
  w.o = tri_rotate(o, w.rot);
  w.Sx = dr.x / dr.z;
  w.Sy = dr.y / dr.z;
  w.Sz = 1.0f / dr.z;
  return w;
}

// watertight test; returns t (or -1) -- products are kept unfused so that a
// shared edge evaluates to exactly opposite values in both triangles
// (the vertices in the ray's frame: the triangle copy w.rot)
// (edge: the hit lies within 2^-10 of the triangle's edges)
__device__ __forceinline__ float woop_hit(const WoopRay& w, float3 v0, float3 v1, float3 v2, bool& edge) {
  edge = false;
  const float3 A = v0 - w.o, B = v1 - w.o, C = v2 - w.o;
  const float Az_ = A.z, Bz_ = B.z, Cz_ = C.z;
  const float Ax = __fsub_rn(A.x, __fmul_rn(w.Sx, Az_));
  const float Ay = __fsub_rn(A.y, __fmul_rn(w.Sy, Az_));
  const float Bx = __fsub_rn(B.x, __fmul_rn(w.Sx, Bz_));
  const float By = __fsub_rn(B.y, __fmul_rn(w.Sy, Bz_));
  const float Cx = __fsub_rn(C.x, __fmul_rn(w.Sx, Cz_));
  const float Cy = __fsub_rn(C.y, __fmul_rn(w.Sy, Cz_));
  const float U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
  const float V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
  const float W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
  if ((U < 0.0f || V < 0.0f || W < 0.0f) && (U > 0.0f || V > 0.0f || W > 0.0f)) return -1.0f;
  const float det = U + V + W;
  if (det == 0.0f) return -1.0f;
  const float T = U * (w.Sz * Az_) + V * (w.Sz * Bz_) + W * (w.Sz * Cz_);
  edge = fminf(fminf(fabsf(U), fabsf(V)), fabsf(W)) <= 0x1p-10f * fabsf(det);
  return T / det;
}

// Where two triangles share an edge, the test above takes the ray that meets it
// for both, at distances that differ in their last bits.  Either is a right
// answer; nodes with float boxes report the one whose hit is found first
// unless the other's box begins before that hit, because the slab test culls
// it.  The coarser boxes of the grid would let the other one win, and a path
// at a building's corner turn the other way (one in some 10^8 queries).  So
// over the grid a hit next to an edge stands only if that slab test of the
// triangle's own float box (planes at fma(b, 1/d, -o/d) moved apart by 4 u
// |o/d|, far planes inflated by 1 + 2 gamma_3) accepts the ray up to the best
// hit so far.  That depends on the order of the visits, so it makes the two
// forms agree in nearly all of these cases, not in all; without the best hit
// in the test it would decide none of them.  4 % of a scan.  Apart from the
// loop, for its registers: inlined it costs 2 % more.  v, o and d in the frame
// of the triangle copy.
constexpr float kBoxInflate = 1.00000036f;   // 1 + 2 gamma_3 (Ize 2013)
__device__ __noinline__ bool edge_hit_stands(float3 v0, float3 v1, float3 v2, float3 o, float3 d, float t_min,
                                             float t_best) {
  float lo = -INFINITY, hi = INFINITY;
  const float b0[3] = {fminf(fminf(v0.x, v1.x), v2.x), fminf(fminf(v0.y, v1.y), v2.y), fminf(fminf(v0.z, v1.z), v2.z)};
  const float b1[3] = {fmaxf(fmaxf(v0.x, v1.x), v2.x), fmaxf(fmaxf(v0.y, v1.y), v2.y), fmaxf(fmaxf(v0.z, v1.z), v2.z)};
  const float oo[3] = {o.x, o.y, o.z}, dd[3] = {d.x, d.y, d.z};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float id = __fdiv_rn(1.0f, fabsf(dd[k]) > 1e-30f ? dd[k] : copysignf(1e-30f, dd[k]));
    const float od = __fmul_rn(oo[k], id), e = copysignf(0x1p-22f * fabsf(od), id);
    const float t0 = fmaf(b0[k], id, __fsub_rn(-od, e)), t1 = fmaf(b1[k], id, __fadd_rn(-od, e));
    lo = fmaxf(lo, fminf(t0, t1));
    hi = fminf(hi, fmaxf(t0, t1));
  }
  return fmaxf(lo, t_min) <= fminf(__fmul_rn(hi, kBoxInflate), t_best);
}

// Selectors of a binary node's box word: __byte_perm(word, 0x3F000000, sel)
// gives the float F of the lower / upper bound (kNodeWords); they differ in
// the bits kSelFlip.
constexpr uint32_t kSelLo = 0x7104u, kSelHi = 0x7324u, kSelFlip = 0x0220u;
__device__ __forceinline__ float grid_plane(uint32_t word, uint32_t sel) {
  return __uint_as_float(__byte_perm(word, 0x3F000000u, sel));
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// two fmas in one instruction: (a, b) * (m, m) + c, c a packed pair
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 fma2(float a, float b, float m, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a, b)), "l"(pack2(m, m)), "l"(c));
  float2 o;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
  return o;
}

// ---------------------------------------------------------------------------
// Resumable traversal.  A query (closest hit, or any hit for visibility) is
// advanced one step at a time -- one node visit or one triangle test -- so
// that a lane whose query has ended can take the next one while the other
// lanes of its warp go on.
//
// Closest hit: t_min < t < t_best on entry, (t, original id)
// lexicographically smallest of the triangles tested; of triangles whose t
// agree up to rounding (a shared edge, overlap in one plane) the boxes may
// leave out all but one, the node format and build decide which.  Any hit:
// the first t_min < t < t_best.  The leaf `skip` (the one the ray starts on) is never reported.
struct Trav {
  float3 c0, c1;        // slab offsets of the near / far planes (float boxes: the lower / upper ones; trav_begin)
  WoopRay w;            // the watertight-test frame
  float3 id;            // 1 / direction, zero components replaced by +-1e-30; binary nodes: times the grid scale
  uint3 sel;            // binary: byte selectors that decode the near plane of a box word, per axis
  float t_min, t_best;
  uint32_t skip;
  uint32_t node;        // binary: next node; both: kNone once the query has ended
  uint32_t best, best_id, visits;
  uint32_t oct;                               // wide: direction octant
  uint32_t g_base, g_bits;                    // wide: node group
  uint32_t t_base, t_bits, t_counts;          // wide: a node's first triangle, hit leaf slots still to test, slot counts
  int sp;                                     // next free stack entry (binary: its byte offset)
};

// exact: binary nodes with float boxes
__device__ __forceinline__ void trav_begin(Trav& s, const ScanArgs& a, float3 o, float3 d, float t_min, float t_best,
                                           uint32_t skip, bool wide, bool exact) {
  s.w = make_woop(o, d);
  const float3 dn = make_float3(fabsf(d.x) > 1e-30f ? d.x : copysignf(1e-30f, d.x),
                                fabsf(d.y) > 1e-30f ? d.y : copysignf(1e-30f, d.y),
                                fabsf(d.z) > 1e-30f ? d.z : copysignf(1e-30f, d.z));
  if (wide || exact) {
    s.id = make_float3(1.0f / dn.x, 1.0f / dn.y, 1.0f / dn.z);
    // Slab test with one fma per plane: plane b is reached at t = fma(b, id, c)
    // with c = -(o id) -+ eps, where the robust form (b - o) id needs two
    // operations.  The fma form errs against (b - o) id by at most u |o id|
    // (o id rounded) + u |c| (c rounded) + u |t| (the fma itself), u = 2^-24.
    // eps = 4 u |o id| moves every near plane down and every far plane up by
    // more than the first two; the last is relative, like the errors of the
    // robust form, and is covered with the far-plane inflation of the robust
    // slab test (1 + 2 gamma_3, Ize 2013) at the node.  So a box the robust
    // test accepts is accepted here too.
    const float ox = __fmul_rn(o.x, s.id.x), oy = __fmul_rn(o.y, s.id.y), oz = __fmul_rn(o.z, s.id.z);
    float ex = 0x1p-22f * fabsf(ox), ey = 0x1p-22f * fabsf(oy), ez = 0x1p-22f * fabsf(oz);
    if (exact) {   // the lower plane is the near one for a positive direction component
      ex = copysignf(ex, s.id.x);
      ey = copysignf(ey, s.id.y);
      ez = copysignf(ez, s.id.z);
    }
    s.c0 = make_float3(-ox - ex, -oy - ey, -oz - ez);
    s.c1 = make_float3(-ox + ex, -oy + ey, -oz + ez);
  } else {
    // The same over grid planes base + F scale, F in [0.5, 2): t = fma(F, g, c)
    // with g = scale id and c = (base - o) id, id the hardware's approximate
    // reciprocal (2 u relative).  Against the exact plane distance the rounded
    // g errs by 3 u |g| per unit of F, c by 4 u |c| and the fma by u |t|, and
    // |t| <= 2 |g| + |c|: together with the relative far-plane inflation of
    // the robust slab test (6 u |t|) less than eps = 24 u (2 |g| + |c|), which
    // moves every near plane down and every far plane up, so that no
    // inflation is left for the node visits.
    s.id = make_float3(rcp_approx(dn.x), rcp_approx(dn.y), rcp_approx(dn.z));
    const float4 base = __ldg(a.frame), scale = __ldg(a.frame + 1);
    const float cx = __fmul_rn(base.x - o.x, s.id.x), cy = __fmul_rn(base.y - o.y, s.id.y),
                cz = __fmul_rn(base.z - o.z, s.id.z);
    s.sel = make_uint3(s.id.x < 0.0f ? kSelHi : kSelLo, s.id.y < 0.0f ? kSelHi : kSelLo,
                       s.id.z < 0.0f ? kSelHi : kSelLo);
    s.id = make_float3(scale.x * s.id.x, scale.y * s.id.y, scale.z * s.id.z);
    const float ex = 0x1.8p-20f * (2.0f * fabsf(s.id.x) + fabsf(cx)),
                ey = 0x1.8p-20f * (2.0f * fabsf(s.id.y) + fabsf(cy)),
                ez = 0x1.8p-20f * (2.0f * fabsf(s.id.z) + fabsf(cz));
    s.c0 = make_float3(cx - ex, cy - ey, cz - ez);
    s.c1 = make_float3(cx + ex, cy + ey, cz + ez);
  }
  s.t_min = t_min;
  s.t_best = t_best;
  s.skip = skip;
  s.best = kNone;
  s.best_id = 0u;
  s.visits = 0u;
  s.sp = wide ? 1 : 4;   // above the lowest entry, which ends the query
  if (wide) {
    s.oct = (s.id.x < 0.0f ? 1u : 0u) | (s.id.y < 0.0f ? 2u : 0u) | (s.id.z < 0.0f ? 4u : 0u);
    s.g_base = 0u;
    s.g_bits = (1u << 8) | (1u << s.oct);   // the root: internal slot 0 of a virtual group
    s.t_base = 0u;
    s.t_bits = 0u;
    s.t_counts = 0u;
    s.node = a.n_tris ? 0u : kNone;
  } else {
    s.node = a.n_tris == 0 ? kNone : (a.n_tris == 1 ? kLeafBit : 0u);
  }
}

// Binary nodes: node visits per triangle test.  A lane that reaches a leaf
// waits until kNodeSteps visits of the others are over and the warp tests its
// waiting leaves together: a query tests a triangle every 10 to 20 visits, so
// testing each at once sent the whole warp through the triangle test in two of
// three steps for one or two lanes (the same scans: 2 / 3 / 4 / 6 / 8 visits
// 17.82 / 17.72 / 17.65 / 17.64 / 18.10 ms; one test per visit 22.53).
constexpr int kNodeSteps = 4;
// Traversal stack: the end mark, kStack entries, and room for the pushes of one group of
// kNodeSteps visits, after which the query loop checks the depth.  The check
// at every push and pop, with the divisions of trav_begin, was 6 % of a scan
// (campus scan 1,134 -> 1,061 us, city scan 24.9 -> 23.4 ms).
// Binary: the ray's direction follows (for edge_hit_stands, out of the registers).
constexpr int kQueryStack = 1 + kStack + kNodeSteps;

// triangle j against the query; returns true when an any-hit query is
// answered.  dir: the ray's direction (binary nodes), null: any edge hit stands
// (the wide nodes' boxes).
template <bool kAny>
__device__ __forceinline__ bool trav_tri(Trav& s, const ScanArgs& a, uint32_t j, uint32_t& n_tris, bool count,
                                         const uint32_t* dir) {
  if (j == s.skip) return false;
  if (count) ++n_tris;
  const float4* tp = a.tri + a.tri_copy * s.w.rot + 3 * (size_t)j;
  const float4 v0 = __ldg(tp), v1 = __ldg(tp + 1), v2 = __ldg(tp + 2);
  bool edge;
  const float t = woop_hit(s.w, f3(v0), f3(v1), f3(v2), edge);
  if (t > s.t_min) {
    if (dir != nullptr && edge && t <= s.t_best) {
      const float3 d = make_float3(__uint_as_float(dir[0]), __uint_as_float(dir[1]), __uint_as_float(dir[2]));
      if (!edge_hit_stands(f3(v0), f3(v1), f3(v2), s.w.o, tri_rotate(d, s.w.rot), s.t_min, s.t_best)) return false;
    }
    if (kAny) {
      if (t < s.t_best) {
        s.best = j;
        return true;
      }
    } else {
      const uint32_t tid = __float_as_uint(v0.w);
      if (t < s.t_best || (t == s.t_best && s.best != kNone && tid < s.best_id)) {
        s.t_best = t;
        s.best = j;
        s.best_id = tid;
      }
    }
  }
  return false;
}

// Stack entry at byte offset sp of a binary traversal
__device__ __forceinline__ uint32_t& bin_entry(uint32_t* stack, int sp) {
  return *reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(stack) + sp);
}

// Binary BVH: one inner node (both children tested, nearer first).
__device__ __forceinline__ void step_inner(Trav& s, uint32_t* stack, const ScanArgs& a, uint32_t& n_nodes,
                                           bool count) {
  if (count) ++n_nodes;
  ++s.visits;   // bounded where the query loop looks at its lanes
  // the stack's top is read beside the node, needed or not: it is in L1, its
  // latency hides behind the node's, and what follows needs no branch
  const uint32_t top = bin_entry(stack, s.sp - 4);
  const uint4* np = a.nodes + kNodeWords * (size_t)s.node;
  uint4 n0, n1;
  asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(n0.x), "=r"(n0.y), "=r"(n0.z), "=r"(n0.w), "=r"(n1.x), "=r"(n1.y), "=r"(n1.z), "=r"(n1.w)
      : "l"(np));
  const float3 g = s.id, cn = s.c0, cf = s.c1;
  const uint3 sn = s.sel, sf = make_uint3(sn.x ^ kSelFlip, sn.y ^ kSelFlip, sn.z ^ kSelFlip);
  const float lo0 = fmaxf(max3(fmaf(grid_plane(n0.x, sn.x), g.x, cn.x), fmaf(grid_plane(n0.y, sn.y), g.y, cn.y),
                               fmaf(grid_plane(n0.z, sn.z), g.z, cn.z)), s.t_min);
  const float hi0 = fminf(min3(fmaf(grid_plane(n0.x, sf.x), g.x, cf.x), fmaf(grid_plane(n0.y, sf.y), g.y, cf.y),
                               fmaf(grid_plane(n0.z, sf.z), g.z, cf.z)), s.t_best);
  const float lo1 = fmaxf(max3(fmaf(grid_plane(n0.w, sn.x), g.x, cn.x), fmaf(grid_plane(n1.x, sn.y), g.y, cn.y),
                               fmaf(grid_plane(n1.y, sn.z), g.z, cn.z)), s.t_min);
  const float hi1 = fminf(min3(fmaf(grid_plane(n0.w, sf.x), g.x, cf.x), fmaf(grid_plane(n1.x, sf.y), g.y, cf.y),
                               fmaf(grid_plane(n1.y, sf.z), g.z, cf.z)), s.t_best);
  const bool h0 = lo0 <= hi0, h1 = lo1 <= hi1;
  // the nearer hit child next, the farther one pushed when both are hit (a
  // predicated store: every local store costs an L2 sector), else the next
  // stack entry.  The lowest entry is kNone, so popping it ends the query
  // without a test, and a full stack is noticed by the query loop, not here.
  // Selects instead of branches: one over the push cost 5-7 % of a scan, one
  // over the pop 2-6 % (city scan 23.4 -> 22.8 ms, city step 27.5 -> 26.0,
  // campus scan 1,072 -> 1,053 us).
  const bool both = h0 && h1, any = h0 || h1;
  const bool first0 = !h1 || (h0 && lo0 <= lo1);
  const uint32_t near = first0 ? n1.z : n1.w, far = first0 ? n1.w : n1.z;
  if (both) bin_entry(stack, s.sp) = far;
  s.sp += both ? 4 : (any ? 0 : -4);
  s.node = any ? near : top;
}

// Binary BVH with float boxes (kNodeWords): the same visit
__device__ __forceinline__ void step_inner_exact(Trav& s, uint32_t* stack, const ScanArgs& a, uint32_t& n_nodes,
                                                 bool count) {
  if (count) ++n_nodes;
  ++s.visits;
  const uint32_t top = bin_entry(stack, s.sp - 4);
  const size_t at = kNodeWords * (size_t)s.node;
  const float4* n0 = reinterpret_cast<const float4*>(a.nodes + at);
  const float4* n1 = reinterpret_cast<const float4*>(a.far + at);
  const float4 x0 = __ldg(n0), x1 = __ldg(n1), z0 = __ldg(n0 + 1), z1 = __ldg(n1 + 1);
  const float3 id = s.id, cl = s.c0, ch = s.c1;
  float lo[2], hi[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float4 xy = k ? x1 : x0, z = k ? z1 : z0;
    const float tx0 = fmaf(xy.x, id.x, cl.x), tx1 = fmaf(xy.y, id.x, ch.x);
    const float ty0 = fmaf(xy.z, id.y, cl.y), ty1 = fmaf(xy.w, id.y, ch.y);
    const float tz0 = fmaf(z.x, id.z, cl.z), tz1 = fmaf(z.y, id.z, ch.z);
    lo[k] = fmaxf(max3(fminf(tx0, tx1), fminf(ty0, ty1), fminf(tz0, tz1)), s.t_min);
    hi[k] = fminf(min3(fmaxf(tx0, tx1), fmaxf(ty0, ty1), fmaxf(tz0, tz1)) * kBoxInflate, s.t_best);
  }
  const bool h0 = lo[0] <= hi[0], h1 = lo[1] <= hi[1], both = h0 && h1, any = h0 || h1;
  const bool first0 = !h1 || (h0 && lo[0] <= lo[1]);
  const uint32_t c0 = __float_as_uint(z0.z), c1 = __float_as_uint(z0.w);
  if (both) bin_entry(stack, s.sp) = first0 ? c1 : c0;
  s.sp += both ? 4 : (any ? 0 : -4);
  s.node = any ? (first0 ? c0 : c1) : top;
}

// Binary BVH: one leaf
template <bool kAny>
__device__ __forceinline__ void step_leaf(Trav& s, uint32_t* stack, const ScanArgs& a, uint32_t& n_tris, bool count) {
  if (trav_tri<kAny>(s, a, s.node & ~kLeafBit, n_tris, count, stack + kQueryStack)) {
    s.node = kNone;
  } else {
    s.sp -= 4;
    s.node = bin_entry(stack, s.sp);
  }
}

// The 8-wide quantised BVH.  A node visit takes the next child of the current
// node group, else of a group from the stack; the triangles of the leaf slots
// it hits are tested before the query visits another node.  A leaf slot holds
// 1..3 consecutive triangles (its count in two bits of the node's word w1.w).
// Children are visited in slot order k ^ octant (near first) through node
// groups as in Ylitie, Karras, Laine, "Efficient incoherent ray traversal on
// GPUs through compressed wide BVHs" (HPG 2017): a group is (first child,
// internal-slot mask << 8 | hit children still to visit, bit k for slot
// k ^ octant), so one stack entry stands for up to 7 pending children; the
// lowest entry is empty and ends the query.  Slot boxes (see kWideNodeWords)
// contain the box of the binary node they stand for, and both node formats
// take a conservative slab test, so a query reaches every triangle it can hit
// in either BVH and finds the same closest hit (up to rounding, see Trav).
//
// Slab test: byte q of a plane word becomes the float F = 1 + q 2^-15 (bits
// 0x3F80qq00), and the plane P + q s is reached at t = fma(F, g, c) with
// g = 2^15 s id and c = (P - 2^15 s) id - o id: one fma a plane where decoding
// the plane first took two.  P - 2^15 s is exact; the roundings of g, c and
// the fma err by less than 2^-23 (2 |g| + |c|), the far-plane inflation of the
// robust test (6 u |t|) by less than 2^-21 of it, and e = 2^-20 (|g| + |c|),
// 1/32 of a quantum and more, covers both: it moves near planes down and far
// planes up.
//
// The former step took a triangle, a node or a stack entry, whichever was
// next, so a warp ran all three for a few lanes each, decoded every plane
// before its slab fma and set the hit masks slot by slot behind branches:
// campus scan over the wide nodes 2,447 us, 1,567 now (batch server's burst of
// 24 requests 18.3 -> 12.1 ms); 1 / 3 visits per leaf test 1,590 / 1,658.
__device__ __forceinline__ void step_wide_node(Trav& s, uint2* stack, const ScanArgs& a, uint32_t& n_nodes,
                                               bool count) {
  const uint2 top = stack[s.sp - 1];
  const bool pop = !(s.g_bits & 0xFFu);
  const uint32_t base = pop ? top.x : s.g_base;
  uint32_t bits = pop ? top.y : s.g_bits;
  s.sp -= pop ? 1 : 0;
  if (!(bits & 0xFFu)) {   // the empty entry
    s.node = kNone;
    return;
  }
  const uint32_t oct = s.oct, slot = (__ffs(bits) - 1u) ^ oct;
  bits &= bits - 1u;   // the lowest bit is a pending child's
  const uint32_t at = base + __popc((bits >> 8) & ((1u << slot) - 1u)), node = min(at, a.node_cap - 1u);
  if (bits & 0xFFu) stack[s.sp] = make_uint2(base, bits);
  s.sp += (bits & 0xFFu) ? 1 : 0;
  if (count) ++n_nodes;
  ++s.visits;   // bounded where the query loop looks at its lanes
  const float3 id = s.id;
  const bool neg_x = id.x < 0.0f, neg_y = id.y < 0.0f, neg_z = id.z < 0.0f;
  const uint4* np = a.nodes + kWideNodeWords * (size_t)node;
  const uint4 w0 = __ldg(np), w1 = __ldg(np + 1), w2 = __ldg(np + 2), w3 = __ldg(np + 3), w4 = __ldg(np + 4);
  if (at >= a.node_cap) atomicOr(&a.ctr->error, kErrBvh);   // no build that reports success gets here
  const float sx = __uint_as_float((w0.w & 0xFFu) << 23), sy = __uint_as_float(((w0.w >> 8) & 0xFFu) << 23),
              sz = __uint_as_float(((w0.w >> 16) & 0xFFu) << 23);
  // the node holds P - 2^23 s
  const float px = fmaf(sx, 8355840.0f, __uint_as_float(w0.x)), py = fmaf(sy, 8355840.0f, __uint_as_float(w0.y)),
              pz = fmaf(sz, 8355840.0f, __uint_as_float(w0.z));
  const float3 g = make_float3(32768.0f * sx * id.x, 32768.0f * sy * id.y, 32768.0f * sz * id.z);
  const float3 cn = make_float3(fmaf(px, id.x, s.c0.x), fmaf(py, id.y, s.c0.y), fmaf(pz, id.z, s.c0.z));
  const float3 cf = make_float3(fmaf(px, id.x, s.c1.x), fmaf(py, id.y, s.c1.y), fmaf(pz, id.z, s.c1.z));
  const float3 e = make_float3(0x1p-20f * (fabsf(g.x) + fabsf(cn.x)), 0x1p-20f * (fabsf(g.y) + fabsf(cn.y)),
                               0x1p-20f * (fabsf(g.z) + fabsf(cn.z)));
  const unsigned long long cx = pack2(cn.x - e.x, cf.x + e.x), cy = pack2(cn.y - e.y, cf.y + e.y),
                           cz = pack2(cn.z - e.z, cf.z + e.z);
  // near and far plane bytes per axis: (lo, hi) for a positive direction, swapped otherwise
  const uint32_t nx0 = neg_x ? w3.z : w2.x, nx1 = neg_x ? w3.w : w2.y;
  const uint32_t fx0 = neg_x ? w2.x : w3.z, fx1 = neg_x ? w2.y : w3.w;
  const uint32_t ny0 = neg_y ? w4.x : w2.z, ny1 = neg_y ? w4.y : w2.w;
  const uint32_t fy0 = neg_y ? w2.z : w4.x, fy1 = neg_y ? w2.w : w4.y;
  const uint32_t nz0 = neg_z ? w4.z : w3.x, nz1 = neg_z ? w4.w : w3.y;
  const uint32_t fz0 = neg_z ? w3.x : w4.z, fz1 = neg_z ? w3.y : w4.w;
  uint32_t hit = 0u;   // slots whose boxes the query enters
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t sel = 0x7604u | (uint32_t)(j & 3) << 4;   // (0, q, 0x80, 0x3F) of the word and 0x3F800000
#define RR_WIDE_PLANE(w0_, w1_) __uint_as_float(__byte_perm(j < 4 ? w0_ : w1_, 0x3F800000u, sel))
    // (near, far) of an axis in one packed fma: 3 % of a scan over these nodes
    // (the binary step, with two boxes a visit, gets 2 % slower by it)
    const float2 vx = fma2(RR_WIDE_PLANE(nx0, nx1), RR_WIDE_PLANE(fx0, fx1), g.x, cx);
    const float2 vy = fma2(RR_WIDE_PLANE(ny0, ny1), RR_WIDE_PLANE(fy0, fy1), g.y, cy);
    const float2 vz = fma2(RR_WIDE_PLANE(nz0, nz1), RR_WIDE_PLANE(fz0, fz1), g.z, cz);
    const float lo = fmaxf(max3(vx.x, vy.x, vz.x), s.t_min), hi = fminf(min3(vx.y, vy.y, vz.y), s.t_best);
#undef RR_WIDE_PLANE
    hit |= lo <= hi ? 1u << j : 0u;
  }
  hit &= w1.z;   // valid slots
  const uint32_t imask = w0.w >> 24;
  // internal hits in visiting order: bit k for slot k ^ octant
  uint32_t in = hit & imask;
  in = (oct & 1u) ? (in & 0x55u) << 1 | (in >> 1 & 0x55u) : in;
  in = (oct & 2u) ? (in & 0x33u) << 2 | (in >> 2 & 0x33u) : in;
  in = (oct & 4u) ? (in & 0x0Fu) << 4 | in >> 4 : in;
  s.g_base = w1.x;
  s.g_bits = imask << 8 | in;
  s.t_base = w1.y;
  s.t_bits = hit & ~imask;
  s.t_counts = w1.w;
}

// the triangles of the next hit leaf slot
template <bool kAny>
__device__ __forceinline__ void step_wide_leaf(Trav& s, const ScanArgs& a, uint32_t& n_tris, bool count) {
  const uint32_t j = __ffs(s.t_bits) - 1u;
  s.t_bits &= s.t_bits - 1u;
  const uint32_t below = s.t_counts & ((1u << (2u * j)) - 1u), n = s.t_counts >> (2u * j) & 3u;
  const uint32_t first = s.t_base + __popc(below & 0x5555u) + 2u * __popc(below & 0xAAAAu);
  for (uint32_t r = 0; r < n; ++r)
    if (first + r < a.n_tris && trav_tri<kAny>(s, a, first + r, n_tris, count, nullptr)) {
      s.t_bits = 0u;
      s.node = kNone;
      break;
    }
}

// ---------------------------------------------------------------------------
// Queries of one bounce.  kAny = false: the closest hit of every queued ray.
// kAny = true: the visibility test of the air-path return (Sec. III-A) for the
// candidates the shading pass listed (deferred visibility, which then settles
// the visible ones), or, with a min_energy cut, for the jobs k_vis_prep listed
// ahead of the shading pass.  Persistent: a warp claims jobs in chunks and hands
// them to its idle lanes once at least `refill` lanes are idle (or all are),
// so the lanes stay busy however uneven the query lengths are.

// Receive-beam weight of a return from p (Sec. III-A air path): g =
// exp(-delta^2 / 2 sigma^2), delta the angle between p - sensor and the beam
// axis of azimuth az; an elliptic beam scales the spread along the offset's
// direction around the axis.
__device__ __forceinline__ float rx_weight(const ScanDesc* sd, uint32_t az, float3 p) {
  const float4 beam = __ldg(&sd->beam);
  const float sigma = d3_sigma(beam.x, beam.y);
  const float3 v = p - f3(__ldg(&sd->pos_rmax));
  const float delta = angle_between(v, beam_axis(sd, az));
  float q = (delta / sigma) * (delta / sigma);
  const float aspect = __ldg(&sd->ext.x);
  if (aspect != 1.0f) {
    const float2 cs = beam_angle(az, __ldg(&sd->dims.x));
    float se, ce;
    sincosf(beam.z, &se, &ce);
    const float4 qt = __ldg(&sd->quat);
    const float3 ea = qrot(qt, make_float3(-cs.y, cs.x, 0.0f));
    const float3 ee = qrot(qt, make_float3(-se * cs.x, -se * cs.y, ce));
    const float c_a = dot(v, ea), c_e = dot(v, ee);
    const float perp2 = c_a * c_a + c_e * c_e;
    if (perp2 > 0.0f) q *= (c_a * c_a + c_e * c_e / (aspect * aspect)) / perp2;
  }
  return sigma > 0.0f ? expf(-0.5f * q) : 0.0f;
}

// Deferred visibility: the sensor is visible from candidate i of a bounce,
// so its air-path return is taken (Sec. III-A; returns deplete the ray): the
// reserved record gets its energy and the child it depletes (or, when the
// child was not spawned, the terminated tally) loses it; the debug dump and
// tallies are patched like the shading pass would have written them.
__device__ __noinline__ void settle_air_path(const ScanArgs& a, uint32_t bounce, uint32_t i) {
  const VisJob* jp = reinterpret_cast<const VisJob*>(a.rays[bounce & 1]) + i;
  const uint4 ix = jp->idx;
  const float4 v = jp->val;
  const float e_child = fmaxf(v.x - v.y, 0.0f);
  if (ix.y != kNone) a.rays[(bounce + 1) & 1][ix.y].d_E.w = e_child;
  if (ix.z != kNone) a.recs[ix.z].y = __float_as_uint(v.z);
  if (ix.w != kNone && a.tallies != nullptr) {
    float* tp = a.tallies + 4 * (size_t)ix.w;
    atomicAdd(tp, v.y);
    if (ix.y == kNone) atomicAdd(tp + 3, e_child - fmaxf(v.x, 0.0f));
  }
  const uint32_t si = __float_as_uint(v.w);
  if (si != kNone && a.segs != nullptr && si < a.seg_cap) {
    a.segs[si].flags |= 2u;
    a.segs[si].ret_a = v.y;
  }
}

// Steps a busy lane takes between two looks at the warp's idle lanes.  The
// look (votes, the refill hand-out, the end-of-query test) costs about a
// fifth of a node visit's instructions when taken every step; taking it every
// kSteps steps lets a lane whose query ended idle for at most kSteps steps.
// Binary nodes: 32 (batch of 24 scans of the 1M-triangle campus: 17.24 ms,
// 17.65 at 16, 17.40 at 64); wide nodes: 16.
constexpr int kSteps = 32, kStepsWide = 16;
constexpr int kWideVisits = 2;   // wide nodes: visits per test of the waiting leaf slots
// Resident threads per SM that the binary query kernels are compiled for:
// 1,152 leaves 56 registers a thread.  Unbounded, the unrolled visits take 64
// to 76 registers and lose more to occupancy than the spill-free code gains
// (city scan 30.5 ms, 26.6 ms at 1,280 threads and 48 registers, 24.8 at 56).
constexpr int kQueryThreads = 1152;
// kCount: the traversal counters (RR_COUNT_TRAVERSAL) are compiled only into
// the kernels of the scans that ask for them
// kSpread: only a.lanes lanes of a warp take queries (small launch sequences);
// apart, because the whole-warp kernels lose 1 % to the extra operands.
// kExact: binary nodes with float boxes; a kernel of its own, because a choice
// inside costs the scans over the grid 2 to 3 % in registers.
template <bool kAny, int kBlock, bool kWide, bool kCount, bool kSpread, bool kExact>
__global__ void __launch_bounds__(kBlock, kWide ? 0 : kQueryThreads / kBlock) k_query(ScanArgs a, uint32_t bounce) {
  typedef typename std::conditional<kWide, uint2, uint32_t>::type StackEntry;
  ScanCounters* C = a.ctr;
  const uint32_t n = kAny ? C->vis_count[bounce] : C->count[bounce];
  uint32_t* ticket = kAny ? &C->vis_ticket[bounce] : &C->trace_ticket[bounce];
  const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x, gsz = gridDim.x * blockDim.x;
  if (!kAny) {
    const uint32_t tiles = (n + kShadeTile - 1) / kShadeTile;
    for (uint32_t t = gtid; t < tiles; t += gsz) a.tile_status[t] = 0ull;
    // the shading pass of this bounce counts the next bounce's rays per order bucket
    if (a.order_hist != nullptr && bounce + 1 <= RR_MAX_BOUNCES)
      for (uint32_t t = gtid; t < kOrderBuckets; t += gsz) a.order_hist[(bounce + 1) * kOrderBuckets + t] = 0u;
  }
  const uint32_t* __restrict__ perm = (!kAny && bounce > 0) ? a.order_perm : nullptr;
  const RayRec* __restrict__ q = a.rays[bounce & 1];
  const uint2* __restrict__ jobs = reinterpret_cast<const uint2*>(a.rays[(bounce + 1) & 1]);
  // after a failed build every query ends at once as a miss and the scan fails
  const bool bvh_ok = (a.bvh_status == nullptr || *a.bvh_status == 0u) &&
                      (a.build_status == nullptr || (*a.build_status & kErrTopBuild) == 0u);
  if (!bvh_ok && gtid == 0) atomicOr(&C->error, kErrBvh);
  constexpr bool count = kCount;
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t refill = a.refill;   // at most a.lanes
  // the other lanes leave, the votes and shuffles below go on among the rest
  // (lane 0 always stays)
  if (kSpread && (uint32_t)lane >= a.lanes) return;
  Trav s;
  s.node = kNone;
  StackEntry stack[kWide ? kQueryStack : kQueryStack + 3];
  uint32_t ray_i = kNone;   // ray of the lane's query (kNone: idle)
  float wa = 0.0f;          // any hit: W(omega_a) of the candidate
  uint32_t c_base = 0u, c_end = 0u;   // claimed, unassigned jobs (warp-uniform)
  bool exhausted = false;             // the job list is used up (warp-uniform)
  uint32_t n_done = 0, n_nodes = 0, n_tris = 0;
  while (true) {
    const bool idle = ray_i == kNone;
    const uint32_t im = __ballot_sync(0xFFFFFFFFu, idle);
    if (im != 0u && !exhausted && ((uint32_t)__popc(im) >= refill || im == 0xFFFFFFFFu)) {
      const uint32_t need = (uint32_t)__popc(im), rank = (uint32_t)__popc(im & lt);
      const uint32_t avail = c_end - c_base;
      uint32_t job = kNone;
      if (idle && rank < avail) job = c_base + rank;
      if (need <= avail) {
        c_base += need;
      } else {
        c_base = c_end;
        const uint32_t more = need - avail, chunk = max(more, kSpread ? a.lanes : 32u);
        uint32_t b = 0;
        if (lane == 0) b = atomicAdd(ticket, chunk);
        b = __shfl_sync(0xFFFFFFFFu, b, 0);
        if (b >= n) {
          exhausted = true;
        } else {
          const uint32_t e = (n - b > chunk) ? b + chunk : n;
          if (idle && rank >= avail && b + (rank - avail) < e) job = b + (rank - avail);
          c_base = min(b + more, e);
          c_end = e;
        }
      }
      if (job != kNone) {
        float3 dir;
        if (kAny && a.defer_vis) {
          ray_i = a.vis_list[job];
          const float4 pl = reinterpret_cast<const VisJob*>(q)[ray_i].p_leaf;
          const uint32_t scan = min(reinterpret_cast<const VisJob*>(q)[ray_i].idx.x, a.n_scans - 1u);
          const ScanDesc* sd = a.desc + scan;
          const float3 p = f3(pl);
          const float3 v = f3(__ldg(&sd->pos_rmax)) - p;
          const float dist = length(v);
          dir = (1.0f / dist) * v;
          trav_begin(s, a, p, dir, __ldg(&sd->phys.x), dist, __float_as_uint(pl.w), kWide, kExact);
        } else if (kAny) {
          const uint2 jb = jobs[job];
          ray_i = jb.x;
          wa = __uint_as_float(jb.y);
          const RayRec ray = q[ray_i];
          const HitRec h = a.hits[ray_i];
          const uint2 sm = ray_scan_medium(a, ray.meta.w);
          const ScanDesc* sd = a.desc + sm.x;
          const float3 o = f3(ray.o_L), d = f3(ray.d_E);
          const float3 p = o + h.t * d;
          const float3 v = f3(__ldg(&sd->pos_rmax)) - p;
          const float dist = length(v);
          dir = (1.0f / dist) * v;
          trav_begin(s, a, p, dir, __ldg(&sd->phys.x), dist, h.leaf, kWide, kExact);
        } else {
          ray_i = perm ? perm[job] : job;
          if (ray_i >= n) ray_i = job;   // only after a failed shading pass (the scan reports it)
          const RayRec ray = q[ray_i];
          const uint2 sm = ray_scan_medium(a, ray.meta.w);
          const float4 phys = __ldg(&a.desc[sm.x].phys);   // t_min, min_energy, freq, r_lim
          const float n_cur = sm.y == kAir ? 1.0f : __ldg(&a.mats[sm.y].n);
          // past t_lim no return can reach the image
          dir = f3(ray.d_E);
          trav_begin(s, a, f3(ray.o_L), dir, phys.x, (phys.w - ray.o_L.w) / n_cur, ray.meta.x, kWide, kExact);
        }
        if (kWide) {
          reinterpret_cast<uint2*>(stack)[0] = make_uint2(0u, 0u);
        } else {
          uint32_t* st = reinterpret_cast<uint32_t*>(stack);
          st[0] = kNone;
          st[kQueryStack] = __float_as_uint(dir.x);
          st[kQueryStack + 1] = __float_as_uint(dir.y);
          st[kQueryStack + 2] = __float_as_uint(dir.z);
        }
        if (!bvh_ok) s.node = kNone;
      }
    }
    const bool busy = ray_i != kNone;
    if (!__any_sync(0xFFFFFFFFu, busy)) {
      if (exhausted) break;
      continue;
    }
    if (busy) {
      if (kWide) {
        uint2* st = reinterpret_cast<uint2*>(stack);
#pragma unroll 1
        for (int u = 0; u < kStepsWide && s.node != kNone; u += kWideVisits) {
#pragma unroll
          for (int v = 0; v < kWideVisits; ++v)
            if (s.t_bits == 0u && s.node != kNone) step_wide_node(s, st, a, n_nodes, count);
          if (s.t_bits) step_wide_leaf<kAny>(s, a, n_tris, count);
          if (s.sp > 1 + kStack) {   // deeper than the stack: the scan reports it
            atomicOr(&a.ctr->error, kErrStack);
            s.node = kNone;
            s.t_bits = 0u;
          }
        }
      } else {
        uint32_t* st = reinterpret_cast<uint32_t*>(stack);
#pragma unroll 1
        for (int u = 0; u < kSteps && s.node != kNone; u += kNodeSteps) {
#pragma unroll
          for (int v = 0; v < kNodeSteps; ++v)
            if (!(s.node & kLeafBit)) {   // kNone carries the leaf bit
              if (kExact) step_inner_exact(s, st, a, n_nodes, count);
              else step_inner(s, st, a, n_nodes, count);
            }
          if ((s.node & kLeafBit) && s.node != kNone) step_leaf<kAny>(s, st, a, n_tris, count);
          if (s.sp > 4 * (1 + kStack)) {   // a tree deeper than the stack: the scan reports it
            atomicOr(&a.ctr->error, kErrStack);
            s.node = kNone;
            s.sp = 0;
          }
        }
      }
      // depth-first traversal of a tree visits each of its internal nodes
      // (fewer than n_tris, binary or wide) at most once: more visits mean a
      // malformed hierarchy (checked here, at most kSteps visits late)
      if (s.node != kNone && s.visits > a.n_tris) {
        atomicOr(&a.ctr->error, kErrBvh);
        s.node = kNone;
      }
      if (s.node == kNone) {   // the query has ended
        if (kAny && a.defer_vis) {
          if (s.best == kNone) settle_air_path(a, bounce, ray_i);
        } else if (kAny) {
          HitRec* hp = a.hits + ray_i;
          uint32_t fl = hp->flags | 1u;
          float wag = 0.0f;
          if (s.best == kNone) {   // the sensor is visible from the hit point: its window W
            fl |= 2u;               // (the receive weight g is applied where the return is made)
            wag = wa;
          }
          hp->flags = fl;
          hp->wa_g = wag;
        } else {
          HitRec h;
          h.t = s.best == kNone ? INFINITY : s.t_best;
          h.leaf = s.best;
          h.flags = min(s.visits, 0xFFFFFFu) << 8;   // bits 8..31: node visits (diagnostics)
          h.wa_g = 0.0f;
          a.hits[ray_i] = h;
        }
        ++n_done;
        ray_i = kNone;
      }
    }
  }
  // counters, one atomic per warp (per lane where the warp is not whole)
  constexpr bool whole = !kSpread;
  if (whole)
    for (int off = 16; off > 0; off >>= 1) n_done += __shfl_xor_sync(0xFFFFFFFFu, n_done, off);
  if ((lane == 0 || !whole) && n_done)
    atomicAdd(kAny ? &C->stat_anyhit : &C->stat_closest, (unsigned long long)n_done);
  if (count) {
    unsigned long long nn = n_nodes, nt = n_tris;
    if (whole)
      for (int off = 16; off > 0; off >>= 1) {
        nn += __shfl_xor_sync(0xFFFFFFFFu, nn, off);
        nt += __shfl_xor_sync(0xFFFFFFFFu, nt, off);
      }
    if (lane == 0 || !whole) {
      atomicAdd(kAny ? &C->stat_nodes_any : &C->stat_nodes, nn);
      atomicAdd(kAny ? &C->stat_tris_any : &C->stat_tris, nt);
    }
  }
}

// Candidates of the air-path return (Sec. III-A) at bounce >= 1: the mean
// reflection direction (or, leaving a medium into air, the refracted one)
// against the direction to the sensor, through the beam window of the lobe.
// Rays whose window is open become jobs (ray, W) of the visibility query,
// appended with one atomic per warp into the free ray buffer of the next
// bounce (order does not matter: each job names its ray).
__global__ void __launch_bounds__(256) k_vis_prep(ScanArgs a, uint32_t bounce) {
  ScanCounters* C = a.ctr;
  const uint32_t n = C->count[bounce];
  const RayRec* __restrict__ q = a.rays[bounce & 1];
  uint2* __restrict__ jobs = reinterpret_cast<uint2*>(a.rays[(bounce + 1) & 1]);
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t warp0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u, wstride = gridDim.x * blockDim.x;
  for (uint32_t base = warp0; base < n; base += wstride) {
    const uint32_t i = base + lane;
    bool want = false;
    float wa = 0.0f;
    if (i < n) {
      const HitRec h = a.hits[i];
      if (h.leaf != kNone && h.leaf < a.n_tris) {
        const RayRec ray = q[i];
        const uint2 sm = ray_scan_medium(a, ray.meta.w);
        const uint32_t medium = sm.y;
        const ScanDesc* sd = a.desc + sm.x;
        if (__ldg(&sd->rng.w) & RR_MULTIPATH) {
          const float3 o = f3(ray.o_L), d = f3(ray.d_E);
          const float n_cur = medium == kAir ? 1.0f : __ldg(&a.mats[medium].n);
          const float4 nr = __ldg(a.tri + (size_t)kTriCopies * a.tri_copy + h.leaf);   // unit normal, material
          const uint32_t mid = __float_as_uint(nr.w);
          const MatDev m = a.mats[mid];
          float3 nrm = f3(nr);
          float cos_i = -dot(d, nrm);
          const bool entering = cos_i > 0.0f;
          float n2 = m.n;
          if (!entering) {
            nrm = -nrm;
            cos_i = -cos_i;
            n2 = 1.0f;
          }
          const float3 p = o + h.t * d;
          const float3 v = f3(__ldg(&sd->pos_rmax)) - p;
          const float side = dot(v, nrm);
          float3 dir_out = make_float3(0.f, 0.f, 0.f);
          bool cand = false;
          if (entering && medium == kAir) {
            dir_out = normalize(d + (2.0f * cos_i) * nrm);
            cand = side > 0.0f;
          } else if (!entering && medium != kAir && !m.pec) {
            const float eta = n_cur / n2;
            const float sin2_t = eta * eta * (1.0f - cos_i * cos_i);
            if (sin2_t < 1.0f) {
              const float cos_t = sqrtf(1.0f - sin2_t);
              dir_out = normalize(eta * d + (eta * cos_i - cos_t) * nrm);
              cand = side < 0.0f;
            }
          }
          if (cand) {   // as the deferred candidates: W and the receive weight g both non-zero
            wa = brdf_window(m, a.lut + (size_t)mid * (kLutCells + 1), angle_between(dir_out, v),
                             __ldg(&sd->beam.x));
            want = wa > 0.0f && wa * rx_weight(sd, ray.meta.y >> 16, p) > 0.0f;
          }
        }
      }
    }
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, want);
    if (m) {
      uint32_t b = 0;
      if (lane == __ffs(m) - 1) b = atomicAdd(&C->vis_count[bounce], (uint32_t)__popc(m));
      b = __shfl_sync(0xFFFFFFFFu, b, __ffs(m) - 1);
      if (want) jobs[b + __popc(m & lt)] = make_uint2(i, __float_as_uint(wa));
    }
  }
}

// ---------------------------------------------------------------------------
// decoupled look-back over tiles: status word = flag << 62 | recs << 31 | kids
constexpr unsigned long long kFlagAgg = 1ull << 62, kFlagPre = 2ull << 62;
constexpr unsigned long long kMask31 = 0x7FFFFFFFull;

__device__ __forceinline__ unsigned long long ld_status(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_status(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// exclusive (kids, recs) prefix of tile `tile`, computed by one full warp
__device__ __forceinline__ uint2 look_back(const ScanArgs& a, uint32_t tile, uint32_t agg_kids, uint32_t agg_recs) {
  const int lane = threadIdx.x & 31;
  unsigned long long* st = a.tile_status;
  const unsigned long long mine = ((unsigned long long)agg_recs << 31) | agg_kids;
  if (tile == 0) {
    if (lane == 0) st_status(st, kFlagPre | mine);
    return make_uint2(0u, 0u);
  }
  if (lane == 0) st_status(st + tile, kFlagAgg | mine);
  uint32_t ex_k = 0, ex_r = 0;
  int j = (int)tile - 1;
  uint32_t spins = 0;
  while (true) {
    const int idx = j - lane;
    unsigned long long s = idx >= 0 ? ld_status(st + idx) : kFlagPre;
    while (__any_sync(0xFFFFFFFFu, (s >> 62) == 0ull)) {
      if (++spins > kSpinLimit) {
        if (lane == 0) atomicOr(&a.ctr->error, kErrTimeout);
        s = kFlagPre;   // give up: the scan is reported as failed
        break;
      }
      if ((s >> 62) == 0ull) s = ld_status(st + idx);
    }
    const uint32_t pre = __ballot_sync(0xFFFFFFFFu, (s >> 62) == 2ull);
    const int first = pre ? __ffs(pre) - 1 : 32;
    const uint32_t vk = lane <= first ? (uint32_t)(s & kMask31) : 0u;
    const uint32_t vr = lane <= first ? (uint32_t)((s >> 31) & kMask31) : 0u;
    ex_k += __reduce_add_sync(0xFFFFFFFFu, vk);
    ex_r += __reduce_add_sync(0xFFFFFFFFu, vr);
    if (pre) break;
    j -= 32;
  }
  if (lane == 0)
    st_status(st + tile, kFlagPre | ((unsigned long long)(agg_recs + ex_r) << 31) | (agg_kids + ex_k));
  return make_uint2(ex_k, ex_r);
}

// failure detection: one warp runs the look-back of tile 1 while tile 0
// never publishes (its status word stays 0), so the bounded wait gives up
__global__ void k_selftest_look_back(ScanArgs a) { look_back(a, 1u, 0u, 0u); }

// ---------------------------------------------------------------------------
// query order: bucket of a queued ray (direction octant, then a 4 x 64 grid of
// cells of its origin around the sensor: height in r_max / 16 steps from one
// below the sensor, horizontal r_max / 4 cells in Morton order)
__device__ __forceinline__ uint32_t order_key(const ScanArgs& a, const RayRec& r) {
  const ScanDesc* sd = a.desc + ray_scan_medium(a, r.meta.w).x;
  const float4 pr = __ldg(&sd->pos_rmax);
  const float inv = 4.0f / fmaxf(pr.w, 1e-3f);
  const int cx = min(max((int)floorf((r.o_L.x - pr.x) * inv) + 4, 0), 7);
  const int cy = min(max((int)floorf((r.o_L.y - pr.y) * inv) + 4, 0), 7);
  const int cz = min(max((int)floorf((r.o_L.z - pr.z) * (4.0f * inv)) + 1, 0), 3);
  uint32_t xy = 0;
#pragma unroll
  for (int b = 0; b < 3; ++b) xy |= (((uint32_t)cx >> b) & 1u) << (2 * b) | (((uint32_t)cy >> b) & 1u) << (2 * b + 1);
  const uint32_t oct = (r.d_E.x < 0.0f ? 1u : 0u) | (r.d_E.y < 0.0f ? 2u : 0u) | (r.d_E.z < 0.0f ? 4u : 0u);
  return oct << 8 | (uint32_t)cz << 6 | xy;
}

// exclusive prefix of the bucket counts of a bounce (one block of 1024 threads, two buckets each)
__global__ void __launch_bounds__(1024) k_order_scan(ScanArgs a, uint32_t bounce) {
  __shared__ uint32_t s_w[32];
  const uint32_t* h = a.order_hist + bounce * kOrderBuckets;
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  const uint32_t c0 = h[2 * t], c1 = h[2 * t + 1];
  uint32_t x = c0 + c1;
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, off);
    if ((int)lane >= off) x += y;
  }
  if (lane == 31u) s_w[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t v = s_w[lane];
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, v, off);
      if ((int)lane >= off) v += y;
    }
    s_w[lane] = v;
  }
  __syncthreads();
  const uint32_t excl = x - (c0 + c1) + (warp ? s_w[warp - 1] : 0u);
  a.order_off[2 * t] = excl;
  a.order_off[2 * t + 1] = excl + c0;
}

// the permutation: every queued ray of the bounce to a position of its
// bucket.  A block takes a contiguous chunk of the queue, counts its keys in
// shared memory, reserves each bucket's share with one atomic and places its
// rays (in any order within a bucket: every query's result is independent
// of the order)
__global__ void __launch_bounds__(256) k_order_place(ScanArgs a, uint32_t bounce) {
  __shared__ uint32_t s_cnt[kOrderBuckets];
  __shared__ uint32_t s_base[kOrderBuckets];
  const uint32_t n = min(a.ctr->count[bounce], a.ray_cap);
  const uint32_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const uint32_t i0 = blockIdx.x * chunk, i1 = min(i0 + chunk, n);
  for (uint32_t j = threadIdx.x; j < kOrderBuckets; j += blockDim.x) s_cnt[j] = 0u;
  __syncthreads();
  for (uint32_t i = i0 + threadIdx.x; i < i1; i += blockDim.x)
    atomicAdd(&s_cnt[a.order_key[i] & (kOrderBuckets - 1u)], 1u);
  __syncthreads();
  for (uint32_t j = threadIdx.x; j < kOrderBuckets; j += blockDim.x) {
    const uint32_t c = s_cnt[j];
    s_base[j] = c ? atomicAdd(&a.order_off[j], c) : 0u;
    s_cnt[j] = 0u;
  }
  __syncthreads();
  for (uint32_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const uint32_t key = a.order_key[i] & (kOrderBuckets - 1u);
    const uint32_t pos = s_base[key] + atomicAdd(&s_cnt[key], 1u);
    if (pos < a.ray_cap) a.order_perm[pos] = i;
  }
}

// ---------------------------------------------------------------------------
// shade

// optional range weight of a return at range r (metres): (1 / r)^k for
// r > 1 m, k = the scan's range_falloff (Eq. 1's power falloff; 0: off)
__device__ __forceinline__ float range_weight(const ScanDesc* sd, float r) {
  const float k = __ldg(&sd->ext.w);
  return (k != 0.0f && r > 1.0f) ? powf(r, -k) : 1.0f;
}

// The shading pass runs in tiles of 256 rays with 3 resident blocks per SM (80
// registers) or in tiles of 512 with 2 (64 registers, a few spilled).  Launch
// sequences with many rays take the latter: more warps hide more of the random
// triangle, material and lobe loads, and half as many tiles wait for their
// predecessors (city scan 21.3 ms with tiles of 256, 21.0 with 512, 21.6 with
// 128; 24 batched scans 14.4 / 14.2 / 14.7).  Small ones take the former:
// there the launch holds fewer tiles than the SMs have room for and each tile's
// chain of dependent loads sets the time (campus scan 1,008 us against 1,068).
// What bounds it: 1,790 warp instructions per 32 rays at 19 of 32 lanes, the
// barriers around the compaction first among the stalls (issue 40 %).  The
// children and records stay in named registers until their places are known,
// and the debug dump is compiled apart: indexed arrays of both kept 240 bytes
// a thread in local memory (city scan 22.0 -> 21.3 ms, campus scan 1,039 ->
// 1,017 us, 24 batched scans 15.0 -> 14.5 ms).
constexpr uint32_t kShadeManyRays = 1u << 16;   // initial rays of a launch sequence

template <int kBlock, int kMinBlocks, bool kDebug>
__global__ void __launch_bounds__(kBlock, kMinBlocks) k_shade(ScanArgs a, uint32_t bounce) {
  __shared__ uint32_t s_tile;
  __shared__ uint32_t s_wsum[kBlock / 32];
  __shared__ uint2 s_excl;
  extern __shared__ uint32_t s_hist[];   // [kOrderBuckets] children per order bucket (query order on only)
  const uint32_t n = a.ctr->count[bounce];
  const uint32_t tiles = (n + kBlock - 1) / kBlock;
  const uint32_t rec0 = a.ctr->rec_start[bounce];
  const uint32_t seg0 = a.ctr->seg_start[bounce];
  const RayRec* qin = a.rays[bounce & 1];   // not restrict: deferred visibility writes its jobs over it
  RayRec* __restrict__ qout = a.rays[(bounce + 1) & 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (n == 0) {
    // empty queue: no tile will publish the offsets of the next bounce
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      a.ctr->count[bounce + 1] = 0u;
      a.ctr->rec_start[bounce + 1] = rec0;
      a.ctr->seg_start[bounce + 1] = seg0;
    }
    return;
  }
  const bool counting = a.order_key != nullptr && bounce + 1 < a.max_bounces;
  if (counting)
    for (uint32_t j = threadIdx.x; j < kOrderBuckets; j += kBlock) s_hist[j] = 0u;
  while (true) {
    if (threadIdx.x == 0) s_tile = atomicAdd(&a.ctr->shade_ticket[bounce], 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile >= tiles) break;
    const uint32_t i = tile * kBlock + threadIdx.x;
    // the children (reflected, refracted) and return records (traveled, air path), written once their places are known
    bool sp_refl = false, sp_refr = false, rec_t = false, rec_a = false;
    float3 p = make_float3(0.f, 0.f, 0.f), d_refl = p, d_refr = p;
    float L1 = 0.f, e_refl = 0.f, e_refr = 0.f;
    uint4 kmeta = make_uint4(0u, 0u, 0u, 0u);   // the reflected child's words; w of the refracted one: kmed
    uint32_t kmed = 0u;
    uint2 rt = make_uint2(0u, 0u), ra = rt;
    bool cand = false;           // an air-path candidate left to the visibility query (deferred visibility)
    int vj_kid = -1, vj_rec = -1;   // its child and record among this ray's (-1: none)
    if (i < n) {
      const RayRec ray = qin[i];
      const HitRec h = a.hits[i];
      const uint32_t az = ray.meta.y >> 16, k = ray.meta.y & 0xFFFFu;
      const uint32_t path = ray.meta.z & 0x7FFFFFFFu;
      const bool masked = (ray.meta.z >> 31) != 0u;
      const uint2 sm = ray_scan_medium(a, ray.meta.w);
      const uint32_t scan = sm.x, medium = sm.y;
      const ScanDesc* sd = a.desc + scan;
      const uint4 dims = __ldg(&sd->dims);   // n_az, ns, max_bounces, n_bins
      const uint4 offs = __ldg(&sd->offs);   // first ray, first column
      const float E = ray.d_E.w;
      float tal[4] = {0.f, 0.f, 0.f, 0.f};
      float dbg_cos = 0.f, dbg_ret_t = 0.f, dbg_ret_a = 0.f;
      uint32_t orig = kNone;
      if (h.leaf == kNone || h.leaf >= a.n_tris) {
        tal[2] = E;   // escaped (or beyond the range limit); an index past the triangles only after a failed step
      } else {
        const float3 o = f3(ray.o_L), d = f3(ray.d_E);
        const float4 pr = __ldg(&sd->pos_rmax);
        const float4 beam = __ldg(&sd->beam);   // b, P, elevation, bin_size
        const float4 phys = __ldg(&sd->phys);   // t_min, min_energy, freq, r_lim
        const uint4 rng = __ldg(&sd->rng);
        const float3 s_pos = f3(pr);
        const bool deeper = bounce + 1 < dims.z;
        const float t = h.t;
        p = o + t * d;
        const float n_cur = medium == kAir ? 1.0f : a.mats[medium].n;
        L1 = ray.o_L.w + n_cur * t;
        float E1 = E;
        if (medium != kAir) {
          const float alpha = kPi * n_cur * a.mats[medium].tan_d * phys.z / kC0;
          E1 = E * expf(-2.0f * alpha * t);
          tal[1] = E - E1;
        }
        const float4 nrw = __ldg(a.tri + (size_t)kTriCopies * a.tri_copy + h.leaf);   // unit normal, material
        orig = __float_as_uint(__ldg(&a.tri[3 * (size_t)h.leaf].w));
        const uint32_t mid = __float_as_uint(nrw.w);
        const MatDev m = a.mats[mid];
        const float4* lut = a.lut + (size_t)mid * (kLutCells + 1);
        float3 nrm = f3(nrw);
        float cos_i = -dot(d, nrm);
        const bool entering = cos_i > 0.0f;
        float n2 = m.n;
        uint32_t next_med = mid;
        if (!entering) {
          nrm = -nrm;
          cos_i = -cos_i;
          n2 = 1.0f;
          next_med = kAir;
        }
        float R = 1.0f, T = 0.0f, cos_t = 0.0f;
        bool can_refract = false;
        const float eta = n_cur / n2;
        if (!m.pec) {
          const float sin2_t = eta * eta * (1.0f - cos_i * cos_i);
          if (sin2_t < 1.0f) {
            cos_t = sqrtf(1.0f - sin2_t);
            const float rs = (n_cur * cos_i - n2 * cos_t) / (n_cur * cos_i + n2 * cos_t);
            const float rp = (n_cur * cos_t - n2 * cos_i) / (n_cur * cos_t + n2 * cos_i);
            R = 0.5f * (rs * rs + rp * rp);
            T = 1.0f - R;
            can_refract = true;
          }
        }
        d_refl = normalize(d + (2.0f * cos_i) * nrm);
        // traveled-path return: omega = theta0 + theta1 = 2 theta0, range L1
        const float theta0 = angle_between(d, -nrm);
        const float E1R = E1 * R, E1T = E1 * T;
        const float ret_t = E1R * fminf(brdf_window(m, lut, 2.0f * theta0, beam.x), 1.0f);
        float ret_a = 0.0f, range_a = 0.0f, e_rec = 0.0f;
        bool air_T = false;
        // the air-path candidate (Sec. III-A): its window W is open toward the
        // sensor; with deferred visibility it is found here, else the
        // visibility query has run and left W in the hit record when visible
        float wag = 0.0f;
        if (a.defer_vis) {
          if (bounce >= 1u && (rng.w & RR_MULTIPATH)) {
            const float3 v = s_pos - p;
            const float side = dot(v, nrm);
            float3 dir_out = d_refl;
            bool c = false;
            if (entering && medium == kAir) {
              c = side > 0.0f;
            } else if (!entering && medium != kAir && can_refract) {
              dir_out = normalize(eta * d + (eta * cos_i - cos_t) * nrm);
              c = side < 0.0f;
            }
            if (c) {   // a window closed toward the sensor, or a receive weight that is 0, returns nothing
              const float wa = brdf_window(m, lut, angle_between(dir_out, v), beam.x);
              if (wa > 0.0f) {
                wag = wa * rx_weight(sd, az, p);
                cand = wag > 0.0f;
              }
            }
          }
        } else if (h.wa_g > 0.0f) {
          wag = h.wa_g * rx_weight(sd, az, p);
        }
        if (wag > 0.0f) {
          float base, cap;
          if (entering && medium == kAir) {
            base = E1R;
            cap = E1R - ret_t;
          } else {
            air_T = true;
            base = E1T;
            cap = E1T;
          }
          ret_a = fmaxf(fminf(base * wag, cap), 0.0f);
          range_a = 0.5f * (L1 + length(s_pos - p));
        }
        // a candidate's return is taken once its visibility is known: until
        // then the ray gives nothing to the air path
        const float ret_a_now = cand ? 0.0f : ret_a;
        tal[0] = ret_t + ret_a_now;
        dbg_cos = cos_i;
        dbg_ret_t = ret_t;
        dbg_ret_a = ret_a_now;
        if (!masked) {
          if (ret_t > 0.0f) {
            const float bin = floorf(L1 / beam.w);
            if (bin < (float)dims.w) {
              float e = ret_t;
              if (rng.w & RR_SPECKLE) e *= -logf(u01(draw(rng, az, k, 1u | (((path << 8) | bounce) << 8)).x));
              e *= range_weight(sd, L1);
              rec_t = true;
              rt = make_uint2(((offs.y + az - offs.w) << kBinBits) | (uint32_t)bin, __float_as_uint(e));
            }
          }
          if (ret_a > 0.0f) {
            const float bin = floorf(range_a / beam.w);
            if (bin < (float)dims.w) {
              float e = ret_a;
              if (rng.w & RR_SPECKLE) e *= -logf(u01(draw(rng, az, k, 1u | (((path << 8) | bounce) << 8)).y));
              e *= range_weight(sd, range_a);
              if (cand) {   // reserved with energy 0, written if the sensor is visible
                e_rec = e;
                vj_rec = rec_t ? 1 : 0;
              }
              rec_a = true;
              ra = make_uint2(((offs.y + az - offs.w) << kBinBits) | (uint32_t)bin, cand ? 0u : __float_as_uint(e));
            }
          }
        }
        e_refl = fmaxf(E1R - ret_t - (air_T ? 0.0f : ret_a_now), 0.0f);
        e_refr = fmaxf(E1T - (air_T ? ret_a_now : 0.0f), 0.0f);
        const bool in_range = L1 < pr.w;
        sp_refl = deeper && in_range && e_refl >= phys.y;
        sp_refr = deeper && in_range && can_refract && (rng.w & RR_REFRACTION) && e_refr >= phys.y;
        if (!sp_refl) tal[3] += e_refl;
        if (!sp_refr) tal[3] += e_refr;
        kmeta = make_uint4(h.leaf, ray.meta.y, (ray.meta.z & 0x80000000u) | (path << 1), (scan << 16) | medium);
        kmed = (scan << 16) | next_med;
        if (sp_refr) d_refr = normalize(eta * d + (eta * cos_i - cos_t) * nrm);
        if (cand) {   // the job, over this ray's record (read above, not read again)
          vj_kid = air_T ? (sp_refr ? (sp_refl ? 1 : 0) : -1) : (sp_refl ? 0 : -1);
          VisJob j;
          j.p_leaf = make_float4(p.x, p.y, p.z, __uint_as_float(h.leaf));
          j.idx = make_uint4(scan, kNone, kNone,
                             a.tallies != nullptr ? offs.x + (az - offs.w) * dims.y + k : kNone);
          j.val = make_float4(air_T ? E1T : E1R - ret_t, ret_a, e_rec,
                              __uint_as_float(a.segs != nullptr ? seg0 + i : kNone));
          reinterpret_cast<VisJob*>(a.rays[bounce & 1])[i] = j;
        }
      }
      if (kDebug && a.tallies != nullptr) {
        float* tp = a.tallies + 4 * ((size_t)offs.x + (size_t)(az - offs.w) * dims.y + k);
        for (int q = 0; q < 4; ++q)
          if (tal[q] != 0.0f) atomicAdd(tp + q, tal[q]);
      }
      if (kDebug && a.segs != nullptr) {
        const uint32_t si = seg0 + i;
        if (si < a.seg_cap) {
          rr_segment sg;
          sg.az = az;
          sg.k = k;
          sg.path = path;
          sg.bounce = bounce;
          sg.tri = orig;
          sg.t = h.leaf == kNone ? INFINITY : h.t;
          sg.E = E;
          sg.flags = (h.flags & 0xFFu) | (cand ? 1u : 0u);   // bit 0: visibility tested, bit 1: visible
          sg.cos_i = dbg_cos;
          sg.ret_t = dbg_ret_t;
          sg.ret_a = dbg_ret_a;
          sg.visits = (float)(h.flags >> 8);   // node visits of the closest-hit query
          a.segs[si] = sg;
        } else {
          atomicOr(&a.ctr->error, kErrCapacitySegs);
        }
      }
    }
    // block scan of (kids, recs)
    const uint32_t nk = (sp_refl ? 1u : 0u) + (sp_refr ? 1u : 0u), nr = (rec_t ? 1u : 0u) + (rec_a ? 1u : 0u);
    const uint32_t packed = nk | (nr << 16);
    uint32_t x = packed;
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, off);
      if (lane >= off) x += y;
    }
    if (lane == 31) s_wsum[warp] = x;
    __syncthreads();
    uint32_t wpre = 0, total = 0;
    for (int w2 = 0; w2 < kBlock / 32; ++w2) {
      const uint32_t v = s_wsum[w2];
      if (w2 < warp) wpre += v;
      total += v;
    }
    const uint32_t local = x - packed + wpre;
    if (warp == 0) {
      const uint2 ex = look_back(a, tile, total & 0xFFFFu, total >> 16);
      if (lane == 0) s_excl = ex;
    }
    __syncthreads();
    const uint2 ex = s_excl;
    const uint32_t kbase = ex.x + (local & 0xFFFFu), rbase = ex.y + (local >> 16);
    if (a.defer_vis) {
      // the candidates' child and record positions, and the list of jobs
      // (one atomic per warp; the order of the list does not matter)
      const uint32_t vm = __ballot_sync(0xFFFFFFFFu, cand);
      if (vm) {
        uint32_t b0 = 0;
        if (lane == __ffs(vm) - 1) b0 = atomicAdd(&a.ctr->vis_count[bounce], (uint32_t)__popc(vm));
        b0 = __shfl_sync(0xFFFFFFFFu, b0, __ffs(vm) - 1);
        if (cand) {
          uint32_t cpos = vj_kid >= 0 ? kbase + (uint32_t)vj_kid : kNone;
          uint32_t rpos = vj_rec >= 0 ? rec0 + rbase + (uint32_t)vj_rec : kNone;
          if (cpos != kNone && cpos >= a.ray_cap) cpos = kNone;   // not written: the scan reports the overflow
          if (rpos != kNone && rpos >= a.rec_cap) rpos = kNone;
          VisJob* jw = reinterpret_cast<VisJob*>(a.rays[bounce & 1]) + i;
          jw->idx.y = cpos;
          jw->idx.z = rpos;
          a.vis_list[b0 + (uint32_t)__popc(vm & ((1u << lane) - 1u))] = i;
        }
      }
    }
    RayRec kid[2];
    kid[0].o_L = kid[1].o_L = make_float4(p.x, p.y, p.z, L1);
    kid[0].d_E = make_float4(d_refl.x, d_refl.y, d_refl.z, e_refl);
    kid[1].d_E = make_float4(d_refr.x, d_refr.y, d_refr.z, e_refr);
    kid[0].meta = kmeta;
    kid[1].meta = make_uint4(kmeta.x, kmeta.y, kmeta.z | 1u, kmed);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const uint32_t pos = kbase + (c && sp_refl ? 1u : 0u);
      if ((c ? sp_refr : sp_refl) && pos < a.ray_cap) {
        qout[pos] = kid[c];
        if (counting) {   // order bucket of the child, counted in the block's histogram
          const uint32_t key = order_key(a, kid[c]);
          a.order_key[pos] = (uint16_t)key;
          atomicAdd(&s_hist[key], 1u);
        }
      }
    }
    {
      const uint32_t pos = rec0 + rbase;
      if (rec_t && pos < a.rec_cap) a.recs[pos] = rt;
      if (rec_a && pos + (rec_t ? 1u : 0u) < a.rec_cap) a.recs[pos + (rec_t ? 1u : 0u)] = ra;
    }
    if (tile == tiles - 1 && threadIdx.x == 0) {
      const uint32_t kids = ex.x + (total & 0xFFFFu), recs = ex.y + (total >> 16);
      ScanCounters* cn = a.ctr;
      uint32_t next = kids;
      if (kids > a.ray_cap) {
        atomicOr(&cn->error, kErrCapacityRays);
        atomicMax(&cn->need_rays, kids);
        next = a.ray_cap;
      }
      uint32_t rend = rec0 + recs;
      if (rend > a.rec_cap || rend < rec0) {
        atomicOr(&cn->error, kErrCapacityRecs);
        atomicMax(&cn->need_recs, rend);
        rend = a.rec_cap;
      }
      cn->count[bounce + 1] = next;   // rays past their scan's bounce limit spawn no children
      cn->rec_start[bounce + 1] = rend;
      cn->seg_start[bounce + 1] = seg0 + n;
      cn->stat_returns += (unsigned long long)recs;
    }
    __syncthreads();
  }
  // the block's bucket counts into the bounce's histogram (the loop ended
  // with a barrier, so every count is in)
  if (counting) {
    uint32_t* h = a.order_hist + (size_t)(bounce + 1) * kOrderBuckets;
    for (uint32_t j = threadIdx.x; j < kOrderBuckets; j += kBlock)
      if (s_hist[j]) atomicAdd(&h[j], s_hist[j]);
  }
}

}  // namespace rr

namespace rr_host {

using namespace rr;

static int g_num_sms = 0;
static int g_query_occ[2][2][3] = {{{0}}};   // [wide][any][block 64 / 128 / 256]
static int g_shade_occ[2] = {0, 0};   // resident blocks of the small and large shading tiles

static int block_index(uint32_t block) { return block <= 64u ? 0 : (block <= 128u ? 1 : 2); }

template <bool kAny, int kBlock, bool kWide>
static void occ_of(int* out) {
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_query<kAny, kBlock, kWide, false, false, false>, kBlock, 0);
  if (*out < 1) *out = 1;
}

template <bool kWide>
static void occ_all(int (*o)[3]) {
  occ_of<false, 64, kWide>(&o[0][0]);
  occ_of<false, 128, kWide>(&o[0][1]);
  occ_of<false, 256, kWide>(&o[0][2]);
  occ_of<true, 64, kWide>(&o[1][0]);
  occ_of<true, 128, kWide>(&o[1][1]);
  occ_of<true, 256, kWide>(&o[1][2]);
}

void init_dims() {
  if (g_num_sms) return;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  occ_all<false>(g_query_occ[0]);
  occ_all<true>(g_query_occ[1]);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_shade_occ[0], k_shade<kShadeTile, 3, false>, kShadeTile, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_shade_occ[1], k_shade<2 * kShadeTile, 2, false>,
                                                2 * kShadeTile, 0);
  for (int& o : g_shade_occ)
    if (o < 1) o = 1;
  g_num_sms = sms < 1 ? 1 : sms;
}

int num_sms() {
  init_dims();
  return g_num_sms;
}

int trace_max_blocks_per_sm(uint32_t block, bool wide) {
  init_dims();
  return g_query_occ[wide ? 1 : 0][0][block_index(block)];
}

cudaError_t launch_raygen(const ScanArgs& a, cudaStream_t st) {
  const uint32_t n = a.n_rays0;
  k_raygen<<<n ? (n + 255) / 256 : 1, 256, 0, st>>>(a);
  return cudaGetLastError();
}

template <bool kAny, bool kWide, bool kCount, bool kExact>
static void query_launch_c(const ScanArgs& a, uint32_t bounce, int bi, int grid, cudaStream_t st) {
  if (bi == 0) {
    if (a.lanes < 32u && !kCount) k_query<kAny, 64, kWide, false, true, kExact><<<grid, 64, 0, st>>>(a, bounce);
    else k_query<kAny, 64, kWide, kCount, false, kExact><<<grid, 64, 0, st>>>(a, bounce);
  } else if (bi == 1) {
    k_query<kAny, 128, kWide, kCount, false, kExact><<<grid, 128, 0, st>>>(a, bounce);
  } else {
    k_query<kAny, 256, kWide, kCount, false, kExact><<<grid, 256, 0, st>>>(a, bounce);
  }
}
template <bool kAny, bool kWide, bool kExact>
static void query_launch(const ScanArgs& a, uint32_t bounce, int bi, int grid, cudaStream_t st) {
  // a counting kernel may hold more registers: its blocks beyond the
  // residency start later and find no work left
  if (a.any_flags & RR_COUNT_TRAVERSAL) query_launch_c<kAny, kWide, true, kExact>(a, bounce, bi, grid, st);
  else query_launch_c<kAny, kWide, false, kExact>(a, bounce, bi, grid, st);
}

cudaError_t launch_query(const ScanArgs& a, uint32_t bounce, bool any, const LaunchCfg& c, cudaStream_t st) {
  init_dims();
  const bool wide = a.wide != 0u;
  const int bi = block_index(c.trace_block);
  int per_sm = g_query_occ[wide ? 1 : 0][any ? 1 : 0][bi];
  if (c.trace_blocks_per_sm > 0 && (int)c.trace_blocks_per_sm < per_sm) per_sm = (int)c.trace_blocks_per_sm;
  // no more blocks than the bounce can have queries (each ray has two children at most)
  const uint64_t warps = (((uint64_t)a.n_rays0 << bounce) + a.lanes - 1) / a.lanes, per_block = 2u << bi;
  const int grid = (int)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)g_num_sms * per_sm, (warps + per_block - 1) / per_block));
  if (wide) {
    if (any) query_launch<true, true, false>(a, bounce, bi, grid, st);
    else query_launch<false, true, false>(a, bounce, bi, grid, st);
  } else if (a.far) {
    if (any) query_launch<true, false, true>(a, bounce, bi, grid, st);
    else query_launch<false, false, true>(a, bounce, bi, grid, st);
  } else {
    if (any) query_launch<true, false, false>(a, bounce, bi, grid, st);
    else query_launch<false, false, false>(a, bounce, bi, grid, st);
  }
  return cudaGetLastError();
}

cudaError_t launch_vis_prep(const ScanArgs& a, uint32_t bounce, cudaStream_t st) {
  init_dims();
  k_vis_prep<<<g_num_sms * 8, 256, 0, st>>>(a, bounce);
  return cudaGetLastError();
}

cudaError_t launch_order(const ScanArgs& a, uint32_t bounce, cudaStream_t st) {
  init_dims();
  k_order_scan<<<1, 1024, 0, st>>>(a, bounce);
  k_order_place<<<g_num_sms * 4, 256, 0, st>>>(a, bounce);
  return cudaGetLastError();
}

cudaError_t launch_shade(const ScanArgs& a, uint32_t bounce, cudaStream_t st) {
  init_dims();
  const size_t smem = a.order_key ? kOrderBuckets * sizeof(uint32_t) : 0;
  const uint64_t most = (uint64_t)a.n_rays0 << bounce;   // rays of the bounce
  const int small = (int)std::max<uint64_t>(
      1, std::min<uint64_t>((uint64_t)g_num_sms * g_shade_occ[0], (most + kShadeTile - 1) / kShadeTile));
  if (a.tallies != nullptr || a.segs != nullptr)
    k_shade<kShadeTile, 3, true><<<small, kShadeTile, smem, st>>>(a, bounce);
  else if (a.n_rays0 >= kShadeManyRays)
    k_shade<2 * kShadeTile, 2, false><<<g_num_sms * g_shade_occ[1], 2 * kShadeTile, smem, st>>>(a, bounce);
  else
    k_shade<kShadeTile, 3, false><<<small, kShadeTile, smem, st>>>(a, bounce);
  return cudaGetLastError();
}

cudaError_t selftest_look_back_wait(void* scratch, cudaStream_t st, bool* gave_up) {
  // scratch: a zeroed ScanCounters, then two zeroed tile status words
  ScanArgs a;
  memset(&a, 0, sizeof a);
  a.ctr = static_cast<ScanCounters*>(scratch);
  a.tile_status = reinterpret_cast<unsigned long long*>(static_cast<char*>(scratch) + sizeof(ScanCounters));
  k_selftest_look_back<<<1, 32, 0, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  uint32_t err = 0;
  e = cudaMemcpyAsync(&err, &a.ctr->error, sizeof err, cudaMemcpyDeviceToHost, st);
  if (e != cudaSuccess) return e;
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  *gave_up = (err & kErrTimeout) != 0u;
  return cudaSuccess;
}

}  // namespace rr_host
