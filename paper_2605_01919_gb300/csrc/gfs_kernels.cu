// Device kernels of the consistent-SDF hot path.
//
//   P build   k_cull_test     -- candidate generation, coverage by the balls
//                                that covered their direction's neighbours
//             k_cull_walk     -- coverage walk of the candidates left open
//                                (Def. 1 discretised, Prop. 1 (ii))
//   query     k_query_spheres -- FP32 pass over the spheres (containment,
//                                tangent and far bounds), state per point
//             k_query_near    -- FP32 pass over the survivors
//             k_query_decide  -- certified decisions, value and flags
//             k_query_exact   -- FP64 evaluation, used for every decision the
//                                FP32 path cannot certify (and precision=1)
//   backward  k_query_grad    -- d s*/d(x, p_i, s_i) through the argmin
//
// FP32 filter.  Every predicate the FP32 path decides (is q inside a shrunk
// ball, which candidate is nearest, is a bound exceeded) is compared against
// a rigorous error bound of the FP32 evaluation relative to the exact value.
// Outside the bound the FP32 answer equals the FP64 answer; inside it the
// predicate is re-decided with the FP64 expression the definition uses, so
// every decision is that of an FP64 evaluation.
#include <cub/cub.cuh>
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "gfs_internal.cuh"
#include "gfs_kernels.h"
#include "gfs_warp.cuh"

namespace cg = cooperative_groups;

namespace gfs {

constexpr float kU = 5.9604644775390625e-8f;  // 2^-24, FP32 unit roundoff
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float sqf(float v) { return v * v; }

// ---------------------------------------------------------------------------
// build: bounds of the data, input copy, Morton keys
// ---------------------------------------------------------------------------
__global__ void k_copy_inputs(const double* __restrict__ p, const double* __restrict__ s, int64_t n,
                              D4* __restrict__ sph64) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    sph64[i] = D4{p[3 * i], p[3 * i + 1], p[3 * i + 2], s[i]};
}

// Morton keys of the sample centres and the data bounds (max |coordinate|,
// max |s|) used by the error model.
__global__ void k_keys_d4(const D4* __restrict__ sph64, int64_t n, uint32_t* __restrict__ keys,
                          int* __restrict__ vals, unsigned int* __restrict__ bound_bits) {
  float amax = 0.f, rmax = 0.f;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const D4 d = sph64[i];
    amax = fmaxf(amax, __double2float_ru(fmax(fabs(d.x), fmax(fabs(d.y), fabs(d.z)))));
    rmax = fmaxf(rmax, __double2float_ru(fabs(d.w)));
    keys[i] = morton3(float(d.x), float(d.y), float(d.z));
    vals[i] = int(i);
  }
  for (int o = 16; o > 0; o >>= 1) {
    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(bound_bits + 0, __float_as_uint(amax));  // non-negative floats order as integers
    atomicMax(bound_bits + 1, __float_as_uint(rmax));
  }
}

// Launch-wide error bounds from the data bounds (max |coordinate|, max |s|).
__device__ BuildConsts make_consts(unsigned int amax_bits, unsigned int rmax_bits) {
  float A = fmaxf(1.0f, __uint_as_float(amax_bits));
  float R = __uint_as_float(rmax_bits);
  const float u = kU;
  const float s3 = 1.7320508f;
  BuildConsts c;
  c.A = A;
  c.R = R;
  // candidate coordinate q32 = fma(r32, u32, p32) vs q64: u(|p| + 2r + |q|)
  c.eq = u * (2.f * A + 2.f * R + 0.01f) * 1.01f + 1e-12f;
  // |x-p| -+ r in FP32 for points in [-A,A]^3 (x rounded from FP64):
  // 2 sqrt3 u A + 4.25 u delta + 2 u r with delta <= 2 sqrt3 A, times 2
  c.ea = 2.f * u * (3.5f * A + 5.25f * 2.f * s3 * A + 2.f * R) + 1e-12f;
  // survivor distance^2: 2 sqrt3 (eq + uA) sqrt(D) + 5 u D, times 2
  c.ed_lin = 4.f * s3 * (c.eq + u * A);
  c.ed_quad = 10.f * u;
  // FP32 slack of a ball's distance to a candidate point (its FP32 error is eq)
  c.pad = 4.f * s3 * (c.eq + u * A) + 1e-7f;
  // linear node bounds against a reference sphere's value at another point of
  // the packet: about 130 u A + 6 u R of FP32 rounding (the record's box and
  // residuals, |x - c| and the unit vectors, the sums), plus the widest error
  // band 2 ea, so that whatever they discard also lies outside that band.  A
  // candidate outside the box lies up to A + R: about 8 u R more, which the R term
  // holds (and the cull adds 4 eq for the candidate's own rounding)
  c.elin = u * (300.f * A + 24.f * R) + 1e-11f;
  return c;
}

__global__ void k_consts(const unsigned int* __restrict__ bound_bits, BuildConsts* __restrict__ bc) {
  *bc = make_consts(bound_bits[0], bound_bits[1]);
}

// FP32 coverage thresholds on d^2 for the filter: d2 < lo => covered for
// certain; d2 > hi => uncovered for certain; else re-decide in FP64.
__device__ __forceinline__ void cov_thresholds(double s64, float r32, float tol32, double tol, float e, float A,
                                               float& lo, float& hi) {
  if (!(fabs(s64) > tol)) {
    lo = -1.f;
    hi = -1.f;
    return;
  }
  const float u = kU;
  float rt = r32 - tol32;
  float rr = rt * rt;
  float rp = r32 + 1e-3f;
  float E = 2.f * (2.f * 1.7320508f * (e + u * A) * rp + 12.f * u * rp * rp) + 4e-15f * sqf(r32 + 1.f) + 1e-30f;
  lo = rr - E;
  hi = rr + E;
}

__global__ void k_gather_spheres(const D4* __restrict__ sph64, const int* __restrict__ order, int64_t n,
                                 const BuildConsts* __restrict__ bc, float tol32, double tol,
                                 float4* __restrict__ sph, float4* __restrict__ thr, float4* __restrict__ cvl,
                                 int* __restrict__ sid) {
  int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  int o = order[t];
  D4 d = sph64[o];
  float w = float(d.w);
  if (w == 0.f && d.w != 0.0) w = copysignf(1.4e-45f, float(d.w > 0 ? 1 : -1));  // keep the sign class
  float4 S = make_float4(float(d.x), float(d.y), float(d.z), w);
  sph[t] = S;
  sid[t] = o;
  float A = bc->A;
  float lc, hc, lq, hq;
  cov_thresholds(d.w, fabsf(w), tol32, tol, bc->eq, A, lc, hc);
  cov_thresholds(d.w, fabsf(w), tol32, tol, kU * A, A, lq, hq);
  thr[t] = make_float4(lc, hc, lq, hq);
  cvl[t] = make_float4(S.x, S.y, S.z, lc);
}

// ---------------------------------------------------------------------------
// hierarchy build
// ---------------------------------------------------------------------------
__device__ void point_leaf_node(const float4* __restrict__ items, int64_t nitems, float4* __restrict__ lo,
                                float4* __restrict__ hi, int64_t L) {
  int64_t b = L * kLeaf, e = min(b + kLeaf, nitems);
  float3 mn = make_float3(INFINITY, INFINITY, INFINITY), mx = make_float3(-INFINITY, -INFINITY, -INFINITY);
  for (int64_t i = b; i < e; ++i) {
    float4 v = items[i];
    mn.x = fminf(mn.x, v.x); mn.y = fminf(mn.y, v.y); mn.z = fminf(mn.z, v.z);
    mx.x = fmaxf(mx.x, v.x); mx.y = fmaxf(mx.y, v.y); mx.z = fmaxf(mx.z, v.z);
  }
  // widen by one ulp: the box then holds the FP64 points the FP32 ones were
  // rounded from
  lo[L] = make_float4(nextafterf(mn.x, -INFINITY), nextafterf(mn.y, -INFINITY), nextafterf(mn.z, -INFINITY), 0.f);
  hi[L] = make_float4(nextafterf(mx.x, INFINITY), nextafterf(mx.y, INFINITY), nextafterf(mx.z, INFINITY), 0.f);
}

__device__ void point_level_node(float4* __restrict__ lo, float4* __restrict__ hi, int64_t child_off, int64_t nchild,
                                 int64_t off, int64_t j) {
  int64_t b = j * kFan, e = min(b + kFan, nchild);
  float4 L = make_float4(INFINITY, INFINITY, INFINITY, 0.f), H = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
  for (int64_t c = b; c < e; ++c) {
    float4 a = lo[child_off + c], z = hi[child_off + c];
    L.x = fminf(L.x, a.x); L.y = fminf(L.y, a.y); L.z = fminf(L.z, a.z);
    H.x = fmaxf(H.x, z.x); H.y = fmaxf(H.y, z.y); H.z = fmaxf(H.z, z.z);
  }
  lo[off + j] = L;
  hi[off + j] = H;
}

__global__ void k_leaves(const float4* __restrict__ items, int64_t nitems, float4* __restrict__ lo,
                         float4* __restrict__ hi, int64_t nleaves) {
  int64_t L = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (L < nleaves) point_leaf_node(items, nitems, lo, hi, L);
}

__global__ void k_level(float4* __restrict__ lo, float4* __restrict__ hi, int64_t child_off, int64_t nchild,
                        int64_t off, int64_t nnode) {
  int64_t j = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (j < nnode) point_level_node(lo, hi, child_off, nchild, off, j);
}

// Centre of a small ball around weighted centres (c_i, w_i): one that makes
// max_i (|c_i - c| + w_i) small, by subgradient steps from the better of two
// starts (the item of largest weight, the mean centre).  Any centre bounds the
// node (the radii are taken against it afterwards), but the exact-coverage walk
// enters the children in the order of |t - C| - w, and the ball it meets
// first decides what the certificates of touching spheres say; so the roots and
// quotients stay IEEE ones and the steps 23: with 12 fast steps the uncovered
// circles of a 64^3 CSG grid were 119,682 instead of 119,672.
// it: kFan items, the first k of them given (the rest has w = -inf), so that
// the loops unroll and the items stay in registers.
__device__ float4 bound_ball(const float4 (&it)[kFan], int k) {
  // value at a centre: the largest |c_i - c| + w_i; the first item that has it
  // (the first one of all if none is above -inf), and its distance
  auto eval = [&](float cx, float cy, float cz, float4& far) {
    float d[kFan], v[kFan];
#pragma unroll
    for (int i = 0; i < kFan; ++i) {
      const float dx = it[i].x - cx, dy = it[i].y - cy, dz = it[i].z - cz;
      d[i] = sqrtf(dx * dx + dy * dy + dz * dz);
      v[i] = d[i] + it[i].w;
    }
    const float best = fmaxf(fmaxf(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])),
                                   fmaxf(fmaxf(v[4], v[5]), fmaxf(v[6], v[7]))), -INFINITY);
    far = make_float4(it[0].x, it[0].y, it[0].z, d[0]);
    if (best > -INFINITY) {
#pragma unroll
      for (int i = kFan - 1; i >= 0; --i)
        if (v[i] == best) far = make_float4(it[i].x, it[i].y, it[i].z, d[i]);
    }
    return best;
  };
  static_assert(kFan == 8, "eval's maximum");
  float4 big = it[0];
  float mx = 0.f, my = 0.f, mz = 0.f;
#pragma unroll
  for (int i = 0; i < kFan; ++i) {
    if (i >= k) break;
    if (it[i].w > big.w) big = it[i];
    mx += it[i].x;
    my += it[i].y;
    mz += it[i].z;
  }
  mx /= float(k);
  my /= float(k);
  mz /= float(k);
  float4 far, far1;
  const float v0 = eval(big.x, big.y, big.z, far), v1 = eval(mx, my, mz, far1);
  const bool at_big = v0 <= v1;
  if (!at_big) far = far1;
  float cx = at_big ? big.x : mx, cy = at_big ? big.y : my, cz = at_big ? big.z : mz;
  float bx = cx, by = cy, bz = cz, best = fminf(v0, v1);
  for (int t = 0; t < 23 && far.w > 1e-12f; ++t) {
    // a step of d / (t + 2) towards the farthest item
    const float dx = far.x - cx, dy = far.y - cy, dz = far.z - cz;
    const float step = far.w / float(t + 2);
    cx += dx / far.w * step;
    cy += dy / far.w * step;
    cz += dz / far.w * step;
    const float v = eval(cx, cy, cz, far);
    if (v < best) {
      best = v;
      bx = cx;
      by = cy;
      bz = cz;
    }
  }
  return make_float4(bx, by, bz, 0.f);
}

// bound_ball by 8 lanes, an item each (the same operations on the same numbers
// in the same order, so the same centre): a step's roots run side by side.  All
// 32 lanes call it, for four centres; `mine` has w = -inf past the k-th item.
__device__ float4 bound_ball8(const float4& mine, int k) {
  const int lane = threadIdx.x & 31, first = lane & ~(kFan - 1);
  auto eval = [&](float cx, float cy, float cz, float4& far) {
    const float dx = mine.x - cx, dy = mine.y - cy, dz = mine.z - cz;
    const float d = sqrtf(dx * dx + dy * dy + dz * dz);
    const float v = d + mine.w;
    float best = fmaxf(v, -INFINITY);
#pragma unroll
    for (int o = 1; o < kFan; o <<= 1) best = fmaxf(best, __shfl_xor_sync(kFull, best, o));
    const unsigned at = (__ballot_sync(kFull, v == best && best > -INFINITY) >> first) & 0xffu;
    const int src = first + (at ? __ffs(at) - 1 : 0);
    far = make_float4(__shfl_sync(kFull, mine.x, src), __shfl_sync(kFull, mine.y, src),
                      __shfl_sync(kFull, mine.z, src), __shfl_sync(kFull, d, src));
    return best;
  };
  int big = first;
  float bw = __shfl_sync(kFull, mine.w, first), mx = 0.f, my = 0.f, mz = 0.f;
#pragma unroll
  for (int i = 0; i < kFan; ++i) {
    const float x = __shfl_sync(kFull, mine.x, first + i), y = __shfl_sync(kFull, mine.y, first + i),
                z = __shfl_sync(kFull, mine.z, first + i), w = __shfl_sync(kFull, mine.w, first + i);
    if (i >= k) continue;
    if (w > bw) {
      big = first + i;
      bw = w;
    }
    mx += x;
    my += y;
    mz += z;
  }
  mx /= float(k);
  my /= float(k);
  mz /= float(k);
  const float gx = __shfl_sync(kFull, mine.x, big), gy = __shfl_sync(kFull, mine.y, big),
              gz = __shfl_sync(kFull, mine.z, big);
  float4 far, far1;
  const float v0 = eval(gx, gy, gz, far), v1 = eval(mx, my, mz, far1);
  const bool at_big = v0 <= v1;
  if (!at_big) far = far1;
  float cx = at_big ? gx : mx, cy = at_big ? gy : my, cz = at_big ? gz : mz;
  float bx = cx, by = cy, bz = cz, best = fminf(v0, v1);
  bool moving = true;  // (of this centre; a centre that has stopped keeps its best)
  for (int t = 0; t < 23; ++t) {
    moving = moving && far.w > 1e-12f;
    if (!__any_sync(kFull, moving)) break;
    const float dx = far.x - cx, dy = far.y - cy, dz = far.z - cz;
    const float step = far.w / float(t + 2);
    cx += dx / far.w * step;
    cy += dy / far.w * step;
    cz += dz / far.w * step;
    float4 next;
    const float v = eval(cx, cy, cz, next);
    if (moving) {
      far = next;
      if (v < best) {
        best = v;
        bx = cx;
        by = cy;
        bz = cz;
      }
    }
  }
  return make_float4(bx, by, bz, 0.f);
}

// Upper bound of a node radius term d = dist (+-) r computed in FP32: the
// rounding of dist (<= 3.6 ulp relative) and of the sum (1 ulp), and the FP32
// copy of an FP64 sphere (sqrt3 ulp of |p| = pm, 1 ulp of r), each covered
// with ~10 ulp.
__device__ __forceinline__ float radius_up(float dist, float d, float r, float pm) {
  return d + (dist + 2.f * r + fabsf(d) + pm) * 6e-7f;
}
// final widening of a stored radius (absolute slack in the coordinate bound A)
__device__ __forceinline__ float radius_fin(float v, float A) {
  return v > -INFINITY ? v + (fabsf(v) + A) * 4.8e-7f : v;
}

// A sphere node is built by two threads, kNear (box, centre C and its radii)
// and kFar (centre F and its radius, the linear record), in different warps: a
// centre's steps are one serial chain, and small hierarchies wait for it
// (16^3 samples built and queried: 0.67 ms, 0.71 with both chains on one
// thread, 0.655 with 8 lanes a centre where nodes are few).
enum NodePart { kNear, kFar };
constexpr int kNodeBlock = 128;                  // threads, two per node (wide: two groups of 8)
constexpr int kNodesPerBlock = kNodeBlock / 2;
// Up to this many nodes of a level the centres' chains are what takes the time:
// the levels (leaves) of 16^3 samples 26 (16) us by 8 lanes, 39 (23) by one; of
// 49^3 55 us with the small levels wide, 77 with none, 78 with all; leaves of 96^3
// 243 us wide, 77 not.
constexpr int64_t kWideNodes = 1024;
__host__ __device__ inline bool wide_nodes(int64_t n) { return n <= kWideNodes; }
__host__ __device__ inline int nodes_per_block(bool wide) { return wide ? kNodesPerBlock / kFan : kNodesPerBlock; }
__device__ __forceinline__ NodePart node_part() { return int(threadIdx.x) < kNodesPerBlock ? kNear : kFar; }
template <bool kWide>
__device__ __forceinline__ int64_t node_of_thread() {
  const int t = threadIdx.x % kNodesPerBlock;
  return blockIdx.x * int64_t(nodes_per_block(kWide)) + (kWide ? t / kFan : t);
}
// centre of a node's items, item(c) = the c-th (w = -inf past the last): kWide,
// all lanes call it and the first of each group of 8 goes on
template <bool kWide, class Item>
__device__ __forceinline__ float4 node_centre(int k, Item item) {
  if constexpr (kWide) {
    return bound_ball8(item(int(threadIdx.x) & (kFan - 1)), k);
  } else {
    float4 W[kFan];
#pragma unroll
    for (int c = 0; c < kFan; ++c) W[c] = item(c);
    return bound_ball(W, k);
  }
}

__device__ __forceinline__ void store_near(const Tree& T, int64_t node, float4 C, float wp, float wn, float w0,
                                           float A) {
  wp = radius_fin(wp, A);
  wn = radius_fin(wn, A);
  w0 = radius_fin(w0, A);
  T.na[node] = make_float4(C.x, C.y, C.z, fmaxf(wp, wn));
  T.nb[node] = make_float4(wp, wn, w0, 0.f);
}

// box part of a linear record from the node's (ulp-widened) box
__device__ __forceinline__ void lin_box(Lin& r, const float4& lo, const float4& hi, float A) {
  r.cx = 0.5f * (lo.x + hi.x);
  r.cy = 0.5f * (lo.y + hi.y);
  r.cz = 0.5f * (lo.z + hi.z);
  r.hx = 0.5f * (hi.x - lo.x) * (1.f + 8.f * kU) + 4.f * kU * A;
  r.hy = 0.5f * (hi.y - lo.y) * (1.f + 8.f * kU) + 4.f * kU * A;
  r.hz = 0.5f * (hi.z - lo.z) * (1.f + 8.f * kU) + 4.f * kU * A;
  r.hip = r.hin = -INFINITY;
  r.lop = r.lon = INFINITY;
}

// Least-squares gradient of k values (it[i].w at it[i]), slightly
// regularised (planar or coincident points give 0 across them), at most 1 in
// norm (signed distances are 1-Lipschitz; noise may exceed it).  Any gradient
// is valid: the residual bounds are taken against it.
__device__ void lin_fit(const float4 (&it)[kFan], int k, Lin& r) {
  float mx = 0.f, my = 0.f, mz = 0.f, mw = 0.f;
#pragma unroll
  for (int i = 0; i < kFan; ++i) {
    if (i >= k) break;
    mx += it[i].x;
    my += it[i].y;
    mz += it[i].z;
    mw += it[i].w;
  }
  const float inv = 1.f / float(k);
  mx *= inv;
  my *= inv;
  mz *= inv;
  mw *= inv;
  float xx = 0.f, xy = 0.f, xz = 0.f, yy = 0.f, yz = 0.f, zz = 0.f, bx = 0.f, by = 0.f, bz = 0.f;
#pragma unroll
  for (int i = 0; i < kFan; ++i) {
    if (i >= k) break;
    const float dx = it[i].x - mx, dy = it[i].y - my, dz = it[i].z - mz, dw = it[i].w - mw;
    xx += dx * dx;
    xy += dx * dy;
    xz += dx * dz;
    yy += dy * dy;
    yz += dy * dz;
    zz += dz * dz;
    bx += dx * dw;
    by += dy * dw;
    bz += dz * dw;
  }
  const float tr = xx + yy + zz;
  r.gx = r.gy = r.gz = 0.f;
  if (!(tr > 0.f)) return;
  const float s = 1.f / tr;
  xx = xx * s + 1e-4f;
  yy = yy * s + 1e-4f;
  zz = zz * s + 1e-4f;
  xy *= s;
  xz *= s;
  yz *= s;
  bx *= s;
  by *= s;
  bz *= s;
  const float c0 = yy * zz - yz * yz, c1 = xz * yz - xy * zz, c2 = xy * yz - xz * yy;
  const float det = xx * c0 + xy * c1 + xz * c2;
  const float id = 1.f / det;
  float gx = (c0 * bx + c1 * by + c2 * bz) * id;
  float gy = (c1 * bx + (xx * zz - xz * xz) * by + (xy * xz - xx * yz) * bz) * id;
  float gz = (c2 * bx + (xy * xz - xx * yz) * by + (xx * yy - xy * xy) * bz) * id;
  const float n2 = gx * gx + gy * gy + gz * gz;
  if (!(n2 < 1e30f)) return;  // not finite: no gradient
  const float f = n2 > 1.f ? rsqrtf(n2) : 1.f;
  r.gx = gx * f;
  r.gy = gy * f;
  r.gz = gz * f;
}

// residual of one sphere against the record's gradient, and the widening of
// a residual bound for the rounding of its terms and of the FP32 copies
__device__ __forceinline__ float lin_res(const Lin& r, const float4& P) {
  return P.w - (r.gx * (P.x - r.cx) + r.gy * (P.y - r.cy) + r.gz * (P.z - r.cz));
}
__device__ __forceinline__ float lin_infl(float s, float A) { return 2e-6f * A + 4e-7f * fabsf(s); }

__device__ __forceinline__ void lin_add(Lin& r, const float4& P, float A) {
  const float v = lin_res(r, P), e = lin_infl(P.w, A);
  if (P.w > 0.f) r.hip = fmaxf(r.hip, v + e);
  if (P.w >= 0.f) r.lop = fminf(r.lop, v - e);
  if (P.w < 0.f) r.lon = fminf(r.lon, v - e);
  if (P.w <= 0.f) r.hin = fmaxf(r.hin, v + e);
}

// (kWide: every lane of the warp calls it; live: the node exists)
template <bool kWide>
__device__ void sphere_leaf_node(const float4* __restrict__ items, float A, const Tree& T, int64_t L, NodePart part,
                                 bool live = true) {
  if (kWide && !live) L = 0;
  const int64_t b = L * kLeaf, e = min(b + kLeaf, T.nitems);
  static_assert(kLeaf == kFan, "a centre takes kFan items");
  const int k = int(e - b);
  // of a small ball enclosing the balls, or for the far bound
  const float4 C = node_centre<kWide>(k, [&](int c) {
    float4 v = items[b + min(c, k - 1)];  // past the end: the last one again, with w = -inf
    v.w = c < k ? (part == kNear ? fabsf(v.w) : -fabsf(v.w)) : -INFINITY;
    return v;
  });
  if (kWide && (!live || (threadIdx.x & (kFan - 1)))) return;
  // (a repeated last item changes no maximum below)
  float4 It[kFan];
  float3 mn = make_float3(INFINITY, INFINITY, INFINITY), mx = make_float3(-INFINITY, -INFINITY, -INFINITY);
#pragma unroll
  for (int c = 0; c < kFan; ++c) {
    const float4 v = It[c] = items[b + min(c, k - 1)];
    mn.x = fminf(mn.x, v.x); mn.y = fminf(mn.y, v.y); mn.z = fminf(mn.z, v.z);
    mx.x = fmaxf(mx.x, v.x); mx.y = fmaxf(mx.y, v.y); mx.z = fmaxf(mx.z, v.z);
  }
  const float4 lo = make_float4(nextafterf(mn.x, -INFINITY), nextafterf(mn.y, -INFINITY), nextafterf(mn.z, -INFINITY), 0.f);
  const float4 hi = make_float4(nextafterf(mx.x, INFINITY), nextafterf(mx.y, INFINITY), nextafterf(mx.z, INFINITY), 0.f);
  if (part == kNear) {
    T.lo[L] = lo;
    T.hi[L] = hi;
    float wp = -INFINITY, wn = -INFINITY, w0 = -INFINITY;
#pragma unroll
    for (int c = 0; c < kFan; ++c) {
      const float4 v = It[c];
      const float r = fabsf(v.w);
      const float pm = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fabsf(v.z));
      const float dx = v.x - C.x, dy = v.y - C.y, dz = v.z - C.z;
      const float dist = sqrtf(dx * dx + dy * dy + dz * dz);
      w0 = fmaxf(w0, radius_up(dist, dist, r, pm));
      if (v.w > 0.f) wp = fmaxf(wp, radius_up(dist, dist + r, r, pm));
      if (v.w < 0.f) wn = fmaxf(wn, radius_up(dist, dist + r, r, pm));
    }
    store_near(T, L, C, wp, wn, w0, A);
    return;
  }
  float wf = -INFINITY;
#pragma unroll
  for (int c = 0; c < kFan; ++c) {
    const float4 v = It[c];
    const float r = fabsf(v.w);
    const float pm = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fabsf(v.z));
    const float dx = v.x - C.x, dy = v.y - C.y, dz = v.z - C.z;
    const float df = sqrtf(dx * dx + dy * dy + dz * dz);
    wf = fmaxf(wf, radius_up(df, df - r, r, pm));
  }
  T.nf[L] = make_float4(C.x, C.y, C.z, radius_fin(wf, A));
  Lin r;
  lin_box(r, lo, hi, A);
  lin_fit(It, k, r);
#pragma unroll
  for (int c = 0; c < kFan; ++c) lin_add(r, It[c], A);
  lin_store(T, L, r);
}

template <bool kWide>
__device__ void sphere_level_node(const Tree& T, float A, int level, int64_t j, NodePart part, bool live = true) {
  if (kWide && !live) j = 0;
  const int64_t child_off = T.offset[level - 1], nchild = T.count[level - 1], off = T.offset[level];
  const int64_t b = j * kFan, e = min(b + kFan, nchild);
  const int k = int(e - b);
  const float4 C = node_centre<kWide>(k, [&](int u) {
    // a ball around the child that holds all its spheres, or its far bound
    const int64_t c = child_off + b + min(u, k - 1);
    float4 v = part == kNear ? T.na[c] : T.nf[c];
    if (part == kNear) v.w = fmaxf(v.w, T.nb[c].z);
    if (u >= k) v.w = -INFINITY;
    return v;
  });
  if (kWide && (!live || (threadIdx.x & (kFan - 1)))) return;
  float4 L = make_float4(INFINITY, INFINITY, INFINITY, 0.f), H = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
  float4 W[kFan];
#pragma unroll
  for (int u = 0; u < kFan; ++u) {
    const int64_t c = child_off + b + min(u, k - 1);
    const float4 a = T.lo[c], z = T.hi[c];
    L.x = fminf(L.x, a.x); L.y = fminf(L.y, a.y); L.z = fminf(L.z, a.z);
    H.x = fmaxf(H.x, z.x); H.y = fmaxf(H.y, z.y); H.z = fmaxf(H.z, z.z);
    W[u] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // radii through the children (|p - C| <= |p - C_c| + |C_c - C|)
  if (part == kNear) {
    T.lo[off + j] = L;
    T.hi[off + j] = H;
    float wp = -INFINITY, wn = -INFINITY, w0 = -INFINITY;
    for (int64_t c = b; c < e; ++c) {
      const float4 ca = T.na[child_off + c], cb = T.nb[child_off + c];
      const float dx = ca.x - C.x, dy = ca.y - C.y, dz = ca.z - C.z;
      const float dist = sqrtf(dx * dx + dy * dy + dz * dz);
      if (cb.x > -INFINITY) wp = fmaxf(wp, radius_up(dist, dist + cb.x, 0.f, 0.f));
      if (cb.y > -INFINITY) wn = fmaxf(wn, radius_up(dist, dist + cb.y, 0.f, 0.f));
      w0 = fmaxf(w0, radius_up(dist, dist + cb.z, 0.f, 0.f));
    }
    store_near(T, off + j, C, wp, wn, w0, A);
    return;
  }
  float wf = -INFINITY;
  for (int64_t c = b; c < e; ++c) {
    const float4 cf = T.nf[child_off + c];
    const float dx = cf.x - C.x, dy = cf.y - C.y, dz = cf.z - C.z;
    const float df = sqrtf(dx * dx + dy * dy + dz * dz);
    wf = fmaxf(wf, radius_up(df, df + cf.w, 0.f, 0.f));
  }
  T.nf[off + j] = make_float4(C.x, C.y, C.z, radius_fin(wf, A));
  // linear record: the gradient from the children's mid values at their box
  // centres, the residual bounds through the children
  // (s - g.(p - c) = s - g_k.(p - c_k) - g.(c_k - c) + (g_k - g).(p - c_k))
  Lin r;
  lin_box(r, L, H, A);
#pragma unroll
  for (int u = 0; u < kFan; ++u) {
    if (u >= k) break;
    const Lin q = lin_load(T, child_off + b + u);
    const float hi_k = fmaxf(q.hip, q.hin), lo_k = fminf(q.lop, q.lon);
    const float v = hi_k > -INFINITY ? 0.5f * (hi_k + lo_k) : 0.f;
    W[u] = make_float4(q.cx, q.cy, q.cz, v);
  }
  lin_fit(W, k, r);
  for (int64_t c = b; c < e; ++c) {
    const Lin q = lin_load(T, child_off + c);
    const float sh = r.gx * (q.cx - r.cx) + r.gy * (q.cy - r.cy) + r.gz * (q.cz - r.cz);
    const float sp = fabsf(q.gx - r.gx) * q.hx + fabsf(q.gy - r.gy) * q.hy + fabsf(q.gz - r.gz) * q.hz;
    const float e2 = sp * 1.000001f + 2e-6f * A + 4e-7f * fabsf(sh);
    if (q.hip > -INFINITY) r.hip = fmaxf(r.hip, q.hip - sh + e2 + 4e-7f * fabsf(q.hip));
    if (q.hin > -INFINITY) r.hin = fmaxf(r.hin, q.hin - sh + e2 + 4e-7f * fabsf(q.hin));
    if (q.lop < INFINITY) r.lop = fminf(r.lop, q.lop - sh - e2 - 4e-7f * fabsf(q.lop));
    if (q.lon < INFINITY) r.lon = fminf(r.lon, q.lon - sh - e2 - 4e-7f * fabsf(q.lon));
  }
  lin_store(T, off + j, r);
}

template <bool kWide>
__global__ void __launch_bounds__(kNodeBlock) k_sphere_leaves(const float4* __restrict__ items, float A, Tree T) {
  const int64_t L = node_of_thread<kWide>();
  if (kWide || L < T.count[0]) sphere_leaf_node<kWide>(items, A, T, L, node_part(), L < T.count[0]);
}

// items of node j at `level`: [j * span, (j + 1) * span), span = kLeaf * kFan^level
__host__ __device__ inline int64_t level_span(int level) {
  int64_t span = kLeaf;
  for (int l = 0; l < level; ++l) span *= kFan;
  return span;
}

template <bool kWide>
__global__ void __launch_bounds__(kNodeBlock) k_sphere_level(float A, Tree T, int level) {
  const int64_t j = node_of_thread<kWide>();
  if (kWide || j < T.count[level]) sphere_level_node<kWide>(T, A, level, j, node_part(), j < T.count[level]);
}

// Tightening of the internal radii, pass 1: one thread per sphere; at every
// level >= 1 it evaluates its sphere against the node's centre (a node's
// spheres are a contiguous range of the Morton order) and raises the node's
// per-radius maximum (same rounding bounds as the leaves).
constexpr int kTight = 8;  // words per node: the four radii, then hip, -lop, -lon, hin
// (one warp: 32 aligned consecutive spheres of one tree; keys: of the tree's
// nodes above the leaves)
__device__ void tighten_items(const float4* __restrict__ items, const Tree& T, float A, unsigned* __restrict__ keys,
                              int64_t i) {
  const bool live = i < T.nitems;
  const int lane = threadIdx.x & 31;
  const float4 v = live ? items[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  const float r = fabsf(v.w);
  const float pm = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fabsf(v.z));
  for (int l = 1; l < T.nlevels; ++l) {
    // a level-l node spans >= 64 consecutive spheres, so the 32 threads of a
    // warp (32 aligned consecutive spheres) share it
    const int64_t node = T.offset[l] + (live ? i / level_span(l) : 0);
    float m[kTight];
#pragma unroll
    for (int q = 0; q < kTight; ++q) m[q] = -INFINITY;
    if (live) {
      const float4 C = T.na[node], Fc = T.nf[node];
      float dx = v.x - C.x, dy = v.y - C.y, dz = v.z - C.z;
      const float dist = sqrtf(dx * dx + dy * dy + dz * dz);
      if (v.w > 0.f) m[0] = radius_up(dist, dist + r, r, pm);
      if (v.w < 0.f) m[1] = radius_up(dist, dist + r, r, pm);
      m[2] = radius_up(dist, dist, r, pm);
      dx = v.x - Fc.x, dy = v.y - Fc.y, dz = v.z - Fc.z;
      const float df = sqrtf(dx * dx + dy * dy + dz * dz);
      m[3] = radius_up(df, df - r, r, pm);
      Lin L = lin_load(T, node);
      L.hip = L.hin = -INFINITY;
      L.lop = L.lon = INFINITY;
      lin_add(L, v, A);
      m[4] = L.hip;
      m[5] = -L.lop;
      m[6] = -L.lon;
      m[7] = L.hin;
    }
#pragma unroll
    for (int q = 0; q < kTight; ++q) {
      // (fmaxf drops a NaN)
      const unsigned w = __reduce_max_sync(0xffffffffu, ord_key(fmaxf(m[q], -INFINITY)));
      if (lane == 0 && live && w > ord_key(-INFINITY)) atomicMax(keys + kTight * (node - T.offset[1]) + q, w);
    }
  }
}

__global__ void k_tighten_items(const float4* __restrict__ items, Tree T, float A, unsigned* __restrict__ keys) {
  tighten_items(items, T, A, keys, blockIdx.x * int64_t(blockDim.x) + threadIdx.x);
}

// pass 2: each internal radius becomes the smaller of its bound through the
// children and the exact maximum over its own spheres (same centre)
__device__ void tighten_node(const Tree& T, const unsigned* __restrict__ keys, float A, int64_t t) {
  const int64_t node = T.offset[1] + t;
  const float4 B = T.nb[node];
  float4 Fc = T.nf[node];
  float w[4] = {B.x, B.y, B.z, Fc.w};
  for (int q = 0; q < 4; ++q) {
    const unsigned k = keys[kTight * t + q];
    if (k != 0u) w[q] = fminf(w[q], radius_fin(ord_val(k), A));
  }
  {
    Lin r = lin_load(T, node);
    const unsigned* k = keys + kTight * t + 4;
    if (k[0] != 0u) r.hip = fminf(r.hip, ord_val(k[0]));
    if (k[1] != 0u) r.lop = fmaxf(r.lop, -ord_val(k[1]));
    if (k[2] != 0u) r.lon = fmaxf(r.lon, -ord_val(k[2]));
    if (k[3] != 0u) r.hin = fminf(r.hin, ord_val(k[3]));
    lin_store(T, node, r);
  }
  T.nb[node] = make_float4(w[0], w[1], w[2], 0.f);
  Fc.w = w[3];
  T.nf[node] = Fc;
  float4 Ca = T.na[node];
  Ca.w = fmaxf(w[0], w[1]);
  T.na[node] = Ca;
}

__global__ void k_tighten_nodes(Tree T, const unsigned* __restrict__ keys, float A, int64_t nupper) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t < nupper) tighten_node(T, keys, A, t);
}

// Morton keys of query points (processing order of the packet kernel)
__global__ void k_query_keys(const double* __restrict__ x64, const float* __restrict__ x32, int64_t m,
                             uint32_t* __restrict__ keys, int* __restrict__ vals) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= m) return;
  float x, y, z;
  if (x32) {
    x = x32[3 * i]; y = x32[3 * i + 1]; z = x32[3 * i + 2];
  } else {
    x = float(x64[3 * i]); y = float(x64[3 * i + 1]); z = float(x64[3 * i + 2]);
  }
  keys[i] = morton3(x, y, z);
  vals[i] = int(i);
}

__global__ void k_point_keys(const float4* __restrict__ items, int64_t n, uint32_t* __restrict__ keys,
                             int* __restrict__ vals) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  float4 v = items[i];
  keys[i] = morton3(v.x, v.y, v.z);
  vals[i] = int(i);
}

__global__ void k_gather_points(const float4* __restrict__ src, const int* __restrict__ order, int64_t n,
                                float4* __restrict__ dst) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  dst[i] = src[order[i]];
}


// sum of v over the active lanes of the warp, added once to *dst
__device__ __forceinline__ void warp_count(unsigned long long* dst, unsigned long long v) {
  const unsigned mask = __activemask();
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  if ((threadIdx.x & 31) == __ffs(mask) - 1 && v) atomicAdd(dst, v);
}

// segment of v in a prefix array (prefix[0] = 0, prefix[ns] = total)
__device__ __forceinline__ int find_seg(const int64_t* __restrict__ prefix, int ns, int64_t v) {
  int lo = 0, hi = ns;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (prefix[mid] <= v) lo = mid;
    else hi = mid;
  }
  return lo;
}

// ---------------------------------------------------------------------------
// query: FP32 pass with certification
// ---------------------------------------------------------------------------
struct Top2 {
  float best, sec;
  int idx;
};
__device__ __forceinline__ void top2_init(Top2& t) {
  t.best = INFINITY;
  t.sec = INFINITY;
  t.idx = -1;
}
__device__ __forceinline__ void top2_push(Top2& t, float v, int j) {
  if (v < t.best) {
    t.sec = fminf(t.sec, t.best);  // sec may hold a seeded threshold before the first push
    t.best = v;
    t.idx = j;
  } else if (v < t.sec) {
    t.sec = v;
  }
}
__device__ __forceinline__ float top2_th(const Top2& t, float band) { return fminf(t.sec, t.best + band); }

__device__ __forceinline__ void load_query(const QueryArgs& a, int64_t q, double& x, double& y, double& z) {
  if (a.x32) {
    x = double(a.x32[3 * q]);
    y = double(a.x32[3 * q + 1]);
    z = double(a.x32[3 * q + 2]);
  } else {
    x = a.x64[3 * q];
    y = a.x64[3 * q + 1];
    z = a.x64[3 * q + 2];
  }
}

__device__ __forceinline__ void write_result(const QueryArgs& a, int64_t q, double v, int64_t arg, int flags) {
  if (a.s_out) a.s_out[q] = float(v);
  if (a.s64_out) a.s64_out[q] = v;
  if (a.arg_out) a.arg_out[q] = arg;
  if (a.fl_out) a.fl_out[q] = uint16_t(flags);
}

// FP64 position of a survivor from its id
__device__ __forceinline__ void surv_pos64(const QueryArgs& a, uint32_t g, double& qx, double& qy, double& qz) {
  const uint32_t i = g / uint32_t(a.KS), k = g % uint32_t(a.KS);
  const D4 pi = a.sph64[i];
  if (int(k) < a.K) {
    ex_cand(pi, a.U64[3 * k], a.U64[3 * k + 1], a.U64[3 * k + 2], qx, qy, qz);
  } else {
    const double* w = a.witness64 + 3 * int64_t(i);
    qx = w[0];
    qy = w[1];
    qz = w[2];
  }
}

__device__ void query_exact_one(const QueryArgs& a, int64_t q);

// Per-point state between the query's passes, 64 B per processing slot: the
// sphere pass's results (48 B), then the nearest survivor (see near_pass).
constexpr int kStateWords = 4;
__device__ __forceinline__ void store_qstate(uint4* st, int64_t slot, bool c0, bool c1, int sample, const Top2& A0,
                                             const Top2& A1, const Top2& F) {
  uint4* p = st + kStateWords * slot;
  p[0] = make_uint4(__float_as_uint(A0.best), __float_as_uint(A0.sec), unsigned(A0.idx), __float_as_uint(A1.best));
  p[1] = make_uint4(__float_as_uint(A1.sec), unsigned(A1.idx), __float_as_uint(F.best), __float_as_uint(F.sec));
  p[2] = make_uint4(unsigned(F.idx), unsigned(sample), (c0 ? 1u : 0u) | (c1 ? 2u : 0u), 0u);
}
__device__ __forceinline__ void load_qstate(const uint4* st, int64_t slot, bool& c0, bool& c1, int& sample, Top2& A0,
                                            Top2& A1, Top2& F) {
  const uint4* p = st + kStateWords * slot;
  const uint4 u0 = p[0], u1 = p[1], u2 = p[2];
  A0.best = __uint_as_float(u0.x);
  A0.sec = __uint_as_float(u0.y);
  A0.idx = int(u0.z);
  A1.best = __uint_as_float(u0.w);
  A1.sec = __uint_as_float(u1.x);
  A1.idx = int(u1.y);
  F.best = __uint_as_float(u1.z);
  F.sec = __uint_as_float(u1.w);
  F.idx = int(u2.x);
  sample = int(u2.y);
  c0 = (u2.z & 1u) != 0;
  c1 = (u2.z & 2u) != 0;
}

}  // namespace gfs
#include "gfs_sphere_pass.cuh"
#include "gfs_cull.cuh"
#include "gfs_finish_pass.cuh"
namespace gfs {

// The query as three kernels: the sphere pass and the survivor pass (results
// to a.state), then the decisions.  Each holds less live state and code than
// one kernel doing all would: with the last two in one, a quarter of the
// stalls were instruction fetches.
//
// One warp per block: packets differ widely in work, and a block of several
// warps would hold its slots until its slowest one is done.
// Points per packet.  A packet's nodes are tested once for all its points,
// but the wider it is against the spacing of the spheres the more of them
// matter to some point, and a heavy packet ends long after the rest, which
// shows when there are few.  Sphere pass in ms, warp per point / packets of
// 8 / 16 / 32 (the first without the point-by-point launch: 16 / 38.2 / 32.7):
//   16.2M points on 64^3 samples       101.4 / 29.3 / 21.6 / 36.5
//   2.1M random points, 96^3 samples    69.8 / 43.8 / 39.8 / 42.9
//   118k points on 13^3 samples         0.43 / 0.18 / 0.18
//   100k random points, 32^3 samples    0.42 / 0.35 / 0.40
//   30k random points, 32^3 samples     0.16 / 0.47 / 0.75
//   32k random points, 64^3 samples     0.53 / 1.04 / 1.26
// lim.rho: a packet of G points of a uniform set of m fills a cube of side
// 2 cbrt(G / m) of the box; a packet whose radius is three such sides holds a
// jump of the Morton order and goes point by point (sphere pass of the first
// two, at 1.5 / 2.5 / 4 sides and without the rule: 30.6 / 21.5 / 20.3 / 22.3 and
// 40.4 / 38.7 / 39.6 / 40.1 ms; at 1.5 a sixth of the first one's packets,
// those that straddle the grid's octants, went point by point).
// lim.spheres, lim.rest: the first two want 600 units a point in the sphere
// pass (at 300 / 150 the second takes 51 / 74 ms: its packets are heavy
// throughout) and about 100 in the others (600 / 128 / 64 / 32: 10.9 / 9.0 /
// 10.0 / 12.6 ms); few points want less, for the sake of the last packets (100k
// on 32^3, both passes after the spheres: 1.16 / 0.60 / 0.54 / 0.50 ms).
constexpr float kJump = 6.f;
// Fewer points than that table wants (m < n, m < 3 n) are sparse: a
// packet of uniform ones spans several spacings of the samples and is better
// taken point by point, but points in a cluster, on a slice or in one place are
// as close as dense ones.  So a packet whose radius is below kClose spacings of
// n uniform samples (2 / cbrt(n) each, in halves) goes as a packet, and the
// others are marked for launches by points.  ms at kClose 1 / 1.5 / 2, after a
// warp per point: a cluster of 200k points on 64^3 samples 2.48 | 0.72 / 0.73 /
// 0.75, of 1M on 128^3 20.4 | 4.1 / 3.9 / 3.9, a slice of 1M on 128^3 32.9 | 27.9 /
// 21.1 / 21.2, 300k points beside the surface of 128^3 7.26 | 7.34 / 7.35 / 8.44
// (packets that give up), 1M random points 29.0 | 29.2 / 29.2 / 29.3, 100k on
// 64^3 1.64 | 1.69 / 1.69 / 1.78.
constexpr float kClose = 1.5f;
struct Packets {
  int G;
  bool sparse;
  PkLimit lim;
};
static Packets packets_of(const QueryArgs& a) {
  Packets p{a.m >= 131072 ? kPacket : (a.m >= 24576 ? 8 : 1), false, no_jump()};
  if (p.G == 1) return p;
  p.lim = p.G == kPacket ? PkLimit{0.f, 600, 100} : PkLimit{0.f, 80, 32};
  p.sparse = a.m < (p.G == kPacket ? a.n : 3 * a.n);
  // very many points a sample (ms with 16 / 32, after 32 with a walk per point:
  // 1M points on 100 samples 0.85 | 0.95 / 0.79, 4M 2.66 | 3.30 / 2.22, 1M on 1,000
  // 1.79 | 1.35 / 1.20; but 1M on 4,096 2.37 | 1.55 / 1.70, 0.2M on 1,000 0.90 | 0.59 /
  // 0.68)
  if (a.m >= 524288 && a.m >= 512 * a.n) p.G = 32;
  p.lim.rho = p.sparse ? kClose * cbrtf(1.f / float(a.n)) : kJump * cbrtf(float(p.G) / float(a.m));
  return p;
}

// A packet that pass(slot) does not finish is listed (counter, for the split
// launch), or marked in a.split (by the packet's number; sparse points), and a
// packet marked by an earlier pass is left to the launch by points.
template <bool kSparse, class Pass>
__device__ __forceinline__ void try_packet(const QueryArgs& a, bool first, unsigned* listed, Pass pass) {
  if constexpr (kSparse) {
    if (!first && a.split[blockIdx.x]) return;
    const bool done = pass();
    if (threadIdx.x == 0 && (first || !done)) a.split[blockIdx.x] = done ? 0u : 1u;
  } else {
    if (!pass() && threadIdx.x == 0) a.split[atomicAdd(listed, 1u)] = blockIdx.x;
  }
}
// the listed packets' points, one at a time
template <int G, class Pass>
__device__ __forceinline__ void split_points(const QueryArgs& a, unsigned packets, unsigned* next, Pass pass) {
  const int64_t total = int64_t(packets) * G;
  for (;;) {
    unsigned t = 0;
    if (threadIdx.x == 0) t = atomicAdd(next, 1u);
    t = __shfl_sync(kFull, t, 0);
    if (int64_t(t) >= total) return;
    const int64_t slot = int64_t(a.split[t / G]) * G + t % G;
    __syncwarp();
    if (slot < a.m) pass(slot);
  }
}

template <int G, bool kSparse>
__global__ void __launch_bounds__(32, 28) k_query_spheres(QueryArgs a, PkLimit lim) {
  __shared__ SpWarp S;
  try_packet<kSparse>(a, true, &a.cnt->q_split, [&]() { return sphere_pass<G>(a, int64_t(blockIdx.x) * G, S, threadIdx.x, lim); });
}
// The points of the packets that k_query_spheres<G, false> listed, one at a time.
template <int G>
__global__ void __launch_bounds__(32, 28) k_query_spheres_split(QueryArgs a) {
  __shared__ SpWarp S;
  split_points<G>(a, a.cnt->q_split, &a.cnt->q_split_next, [&](int64_t slot) { sphere_pass<1>(a, slot, S, threadIdx.x, no_jump()); });
}
// The marked packets' points, a block each (with the cursor of the split launch
// the survivor pass takes twice as long when nearly all are marked).
template <int G>
__global__ void __launch_bounds__(32, 28) k_query_spheres_marked(QueryArgs a) {
  __shared__ SpWarp S;
  if (a.split[blockIdx.x / G]) sphere_pass<1>(a, blockIdx.x, S, threadIdx.x, no_jump());
}

// The survivor pass, split the same way.
template <int G, bool kSparse>
__global__ void __launch_bounds__(32, 28) k_query_near(QueryArgs a, PkLimit lim) {
  __shared__ SpWarp S;
  try_packet<kSparse>(a, false, &a.cnt->f_split, [&]() { return near_pass<G>(a, int64_t(blockIdx.x) * G, S, threadIdx.x, lim); });
}
template <int G>
__global__ void __launch_bounds__(32, 28) k_query_near_split(QueryArgs a) {
  __shared__ SpWarp S;
  split_points<G>(a, a.cnt->f_split, &a.cnt->f_split_next, [&](int64_t slot) { near_pass<1>(a, slot, S, threadIdx.x, no_jump()); });
}
template <int G>
__global__ void __launch_bounds__(32, 28) k_query_near_marked(QueryArgs a) {
  __shared__ SpWarp S;
  if (a.split[blockIdx.x / G]) near_pass<1>(a, blockIdx.x, S, threadIdx.x, no_jump());
}

// The decisions, split the same way (packets of 8 / 16 / 32 on 16.2M points,
// 64^3 samples: 18.3 / 14.9 / 15.9 ms; 2.1M random points, 96^3: 8.6 / 9.4 / 12.4).
template <int G, bool kSparse>
__global__ void __launch_bounds__(32, 24) k_query_decide(QueryArgs a, PkLimit lim) {
  __shared__ SpWarp S;
  try_packet<kSparse>(a, false, &a.cnt->d_split, [&]() { return decide_pass<G, false>(a, int64_t(blockIdx.x) * G, S, threadIdx.x, lim); });
}
template <int G>
__global__ void __launch_bounds__(32, 24) k_query_decide_split(QueryArgs a) {
  __shared__ SpWarp S;
  split_points<G>(a, a.cnt->d_split, &a.cnt->d_split_next, [&](int64_t slot) { decide_pass<1, false>(a, slot, S, threadIdx.x, no_jump()); });
}
template <int G>
__global__ void __launch_bounds__(32, 24) k_query_decide_marked(QueryArgs a) {
  __shared__ SpWarp S;
  if (a.split[blockIdx.x / G]) decide_pass<1, false>(a, blockIdx.x, S, threadIdx.x, no_jump());
}

// ---------------------------------------------------------------------------
// query: exact FP64 evaluation (deferred queries, or precision = 1)
// ---------------------------------------------------------------------------
__device__ void query_exact_one(const QueryArgs& a, int64_t q) {
  double x, y, z;
  load_query(a, q, x, y, z);
  const double tol = a.tol;
  bool cov[2] = {false, false};
  double bestA[2] = {INFINITY, INFINITY};
  int idxA[2] = {INT_MAX, INT_MAX};
  double bestF = INFINITY;
  int sample = INT_MAX;
  {
    const Tree& T = a.st;
    uint32_t stack[kStack];
    int sp = 0;
    const int top = T.nlevels - 1;
    for (int64_t j = 0; j < T.count[top]; ++j) stack[sp++] = pack_node(top, j);
    while (sp > 0) {
      const uint32_t nd = stack[--sp];
      const int lev = node_level(nd);
      const int64_t idx = node_index(nd);
      if (lev == 0) {
        const int64_t b = idx * kLeaf, e = min(b + kLeaf, a.n);
        for (int64_t j = b; j < e; ++j) {
          const int o = a.sid[j];
          const D4 P = a.sph64[o];
          if (P.x == x && P.y == y && P.z == z && o < sample) sample = o;
          const double d2 = ex_d2(x, y, z, P.x, P.y, P.z);
          const double dl = __dsqrt_rn(d2);
          const double r = fabs(P.w);
          if (P.w != 0.0) {
            const int c = P.w < 0.0;
            if (!cov[c] && r > tol) {
              const double rt = __dsub_rn(r, tol);
              if (d2 < __dmul_rn(rt, rt)) cov[c] = true;
            }
            const double av = __dsub_rn(dl, r);
            if (av < bestA[c] || (av == bestA[c] && o < idxA[c])) {
              bestA[c] = av;
              idxA[c] = o;
            }
          }
          const double f = __dadd_rn(dl, r);
          if (f < bestF) bestF = f;
        }
      } else {
        const int64_t cb = idx * kFan, ce = min(cb + kFan, T.count[lev - 1]);
        const int64_t off = T.offset[lev - 1];
        for (int64_t c = cb; c < ce; ++c) {
          const float4 L = T.lo[off + c], H = T.hi[off + c];
          bool need = x >= double(L.x) && x <= double(H.x) && y >= double(L.y) && y <= double(H.y) &&
                      z >= double(L.z) && z <= double(H.z);
          if (!need) {
            const float4 B = T.na[off + c], R = T.nb[off + c], Fb = T.nf[off + c];
            const double tf = (bestF + double(Fb.w)) * (1.0 + 1e-12) + 1e-12;
            need = tf > 0.0 && ball_d2_64(x, y, z, Fb) <= tf * tf;
            double v = -INFINITY;
            for (int cl = 0; cl < 2; ++cl) {
              const float w = cl == 0 ? R.x : R.y;
              if (!(w > -INFINITY)) continue;
              double th = bestA[cl];
              if (!cov[cl]) th = fmax(th, -tol);
              v = fmax(v, th + double(w));
            }
            const double t = v * (1.0 + 1e-12) + 1e-12;
            need = need || (t > 0.0 && ball_d2_64(x, y, z, B) <= t * t);
          }
          if (need) stack[sp++] = pack_node(lev - 1, c);
        }
      }
    }
  }
  if (sample != INT_MAX) {
    write_result(a, q, a.sph64[sample].w, sample, GFS_CODE_SAMPLE);
    return;
  }
  if (cov[0] && cov[1]) {
    write_result(a, q, __longlong_as_double(0x7ff8000000000000LL), -1, GFS_CODE_INVALID);
    return;
  }
  if (!cov[0] && !cov[1]) {
    write_result(a, q, 0.0, -1, GFS_CODE_OUTSIDE);
    return;
  }
  const int cs = cov[0] ? 0 : 1, co = 1 - cs;
  double bd = INFINITY;
  uint32_t gbest = 0xffffffffu;
  const float eqs = a.bc->eq;
  if (a.vt[cs].nlevels > 0) {
    const Tree& T = a.vt[cs];
    const float4* items = a.surv[cs];
    uint32_t stack[kStack];
    int sp = 0;
    const int top = T.nlevels - 1;
    for (int64_t j = 0; j < T.count[top]; ++j) stack[sp++] = pack_node(top, j);
    while (sp > 0) {
      const uint32_t nd = stack[--sp];
      const int lev = node_level(nd);
      const int64_t idx = node_index(nd);
      if (lev == 0) {
        const int64_t b = idx * kLeaf, e = min(b + kLeaf, T.nitems);
        for (int64_t j = b; j < e; ++j) {
          const uint32_t g = __float_as_uint(items[j].w);
          double qx, qy, qz;
          surv_pos64(a, g, qx, qy, qz);
          const double d2 = ex_d2(x, y, z, qx, qy, qz);
          if (d2 < bd || (d2 == bd && g < gbest)) {
            bd = d2;
            gbest = g;
          }
        }
      } else {
        const int64_t cb = idx * kFan, ce = min(cb + kFan, T.count[lev - 1]);
        const int64_t off = T.offset[lev - 1];
        // survivor boxes hold the FP32 positions; the FP64 position of a
        // candidate is within eq of its FP32 one in each coordinate
        const double t = sqrt(bd) * (1.0 + 1e-12) + 2.0 * 1.7320508075688772 * double(eqs) + 1e-12;
        for (int64_t c = cb; c < ce; ++c) {
          const double d2 = box_d2_64(x, y, z, T.lo[off + c], T.hi[off + c]);
          if (d2 <= t * t) stack[sp++] = pack_node(lev - 1, c);
        }
      }
    }
  }
  const bool have_s = gbest != 0xffffffffu, have_u = idxA[co] != INT_MAX;
  const double ds = have_s ? __dsqrt_rn(bd) : INFINITY;
  const double ub = have_u ? bestA[co] : INFINITY;
  const double lb = -bestA[cs];
  double m;
  int code;
  int64_t arg;
  if (have_s && (!a.clamp_opp || ds <= ub)) {
    code = GFS_CODE_SURVIVOR;
    m = ds;
    arg = int64_t(gbest);
  } else if (a.clamp_opp && have_u) {
    code = GFS_CODE_OPPOSITE;
    m = ub;
    arg = idxA[co];
  } else {
    code = GFS_CODE_LOWER;
    m = lb;
    arg = idxA[cs];
  }
  if (m < 0.0) m = 0.0;
  int flags = code;
  if (m < __dsub_rn(lb, tol)) flags |= GFS_FLAG_LB_VIOL;
  if (m > __dadd_rn(bestF, tol)) flags |= GFS_FLAG_FAR_VIOL;
  if (have_u && ub < __dsub_rn(m, tol)) flags |= GFS_FLAG_OPP_VIOL;
  write_result(a, q, cs == 0 ? m : -m, arg, flags);
}

__global__ void __launch_bounds__(128) k_query_exact_all(QueryArgs a) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q < a.m) query_exact_one(a, q);
}

__global__ void __launch_bounds__(128) k_query_exact_deferred(QueryArgs a) {
  const unsigned int nd = min(a.cnt->ndefer, a.defer_cap);
  for (unsigned int t = blockIdx.x * blockDim.x + threadIdx.x; t < nd; t += gridDim.x * blockDim.x)
    query_exact_one(a, int64_t(a.defer[t]));
}

// ---------------------------------------------------------------------------
// backward: analytic derivative through the argmin
// ---------------------------------------------------------------------------
constexpr double kFix = 1099511627776.0;  // 2^40: fixed-point scale of the per-sample sums

__device__ __forceinline__ void fix_add(long long* dst, double v) {
  atomicAdd(reinterpret_cast<unsigned long long*>(dst), (unsigned long long)(long long)llrint(v * kFix));
}

__global__ void k_query_grad(GradArgs a) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q >= a.m) return;
  double x, y, z;
  if (a.x32) {
    x = a.x32[3 * q]; y = a.x32[3 * q + 1]; z = a.x32[3 * q + 2];
  } else {
    x = a.x64[3 * q]; y = a.x64[3 * q + 1]; z = a.x64[3 * q + 2];
  }
  const int code = a.flags[q] & 15;
  const double g = a.grad_s[q];
  const float sv = a.s[q];
  const double sigma = sv > 0.f ? 1.0 : (sv < 0.f ? -1.0 : 0.0);
  double gx = 0, gy = 0, gz = 0;
  if (code == GFS_CODE_SAMPLE) {
    if (a.acc_s) fix_add(a.acc_s + a.arg[q], g);
  } else if (sigma != 0.0 && (code == GFS_CODE_SURVIVOR || code == GFS_CODE_OPPOSITE || code == GFS_CODE_LOWER)) {
    if (code == GFS_CODE_SURVIVOR) {
      const uint32_t gid = uint32_t(a.arg[q]);
      const uint32_t i = gid / uint32_t(a.KS), k = gid % uint32_t(a.KS);
      const D4 pi = a.sph64[i];
      double qx, qy, qz, ux = 0, uy = 0, uz = 0;
      if (int(k) < a.K) {
        ux = a.U64[3 * k]; uy = a.U64[3 * k + 1]; uz = a.U64[3 * k + 2];
        ex_cand(pi, ux, uy, uz, qx, qy, qz);
      } else {
        qx = a.witness64[3 * i]; qy = a.witness64[3 * i + 1]; qz = a.witness64[3 * i + 2];
      }
      double vx = x - qx, vy = y - qy, vz = z - qz;
      const double d = sqrt(vx * vx + vy * vy + vz * vz);
      if (d > 0.0) {
        vx /= d; vy /= d; vz /= d;
        gx = g * sigma * vx; gy = g * sigma * vy; gz = g * sigma * vz;
        if (int(k) < a.K) {
          if (a.acc_p) {
            fix_add(a.acc_p + 3 * int64_t(i), -gx);
            fix_add(a.acc_p + 3 * int64_t(i) + 1, -gy);
            fix_add(a.acc_p + 3 * int64_t(i) + 2, -gz);
          }
          const double si = pi.w > 0 ? 1.0 : (pi.w < 0 ? -1.0 : 0.0);
          if (a.acc_s) fix_add(a.acc_s + i, -g * sigma * si * (vx * ux + vy * uy + vz * uz));
        }
      }
    } else {
      const int64_t j = a.arg[q];
      const D4 pj = a.sph64[j];
      double wx = x - pj.x, wy = y - pj.y, wz = z - pj.z;
      const double d = sqrt(wx * wx + wy * wy + wz * wz);
      if (d > 0.0) {
        wx /= d; wy /= d; wz /= d;
        const double dir = code == GFS_CODE_OPPOSITE ? 1.0 : -1.0;
        gx = g * sigma * dir * wx; gy = g * sigma * dir * wy; gz = g * sigma * dir * wz;
        if (a.acc_p) {
          fix_add(a.acc_p + 3 * j, -gx);
          fix_add(a.acc_p + 3 * j + 1, -gy);
          fix_add(a.acc_p + 3 * j + 2, -gz);
        }
        const double sj = pj.w > 0 ? 1.0 : (pj.w < 0 ? -1.0 : 0.0);
        if (a.acc_s) fix_add(a.acc_s + j, -g * sigma * dir * sj);
      }
    }
  }
  if (a.grad_x) {
    a.grad_x[3 * q] = float(gx);
    a.grad_x[3 * q + 1] = float(gy);
    a.grad_x[3 * q + 2] = float(gz);
  }
}

__global__ void k_fix_to_float(const long long* __restrict__ acc, int64_t n, float* __restrict__ out) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) out[i] = float(double(acc[i]) / kFix);
}

// survivors: ids of both class lists (zero-class entries only from list 0)
__global__ void k_collect_ids(const float4* __restrict__ s0, unsigned int n0, const float4* __restrict__ s1,
                              unsigned int n1, const D4* __restrict__ sph64, int KS, uint32_t* __restrict__ out,
                              unsigned int* __restrict__ count) {
  unsigned int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n0) {
    out[atomicAdd(count, 1u)] = __float_as_uint(s0[t].w);
  } else if (t < n0 + n1) {
    uint32_t g = __float_as_uint(s1[t - n0].w);
    if (sph64[g / uint32_t(KS)].w != 0.0) out[atomicAdd(count, 1u)] = g;
  }
}

__global__ void k_widen_ids(const uint32_t* __restrict__ in, int64_t n, int64_t* __restrict__ out) {
  int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i < n) out[i] = int64_t(in[i]);
}

// ---------------------------------------------------------------------------
// host-side launch helpers
// ---------------------------------------------------------------------------
static inline unsigned int nblk(int64_t n, int b) { return (unsigned int)((n + b - 1) / b); }

// kernels this library launched (own kernels; sorts counted as calls)
static unsigned long long g_launches = 0, g_sort_calls = 0;
void launch_counts(unsigned long long* own, unsigned long long* sorts) {
  *own = g_launches;
  *sorts = g_sort_calls;
}

cudaError_t launch_copy_inputs(const double* p, const double* s, int64_t n, D4* sph64, cudaStream_t st) {
  unsigned int g = nblk(n, 256);
  if (g > 4096) g = 4096;
  k_copy_inputs<<<g, 256, 0, st>>>(p, s, n, sph64);
  ++g_launches;
  return cudaGetLastError();
}

cudaError_t launch_keys_d4(const D4* sph64, int64_t n, uint32_t* keys, int* vals, unsigned int* bound_bits,
                           BuildConsts* bc, cudaStream_t st) {
  unsigned int g = nblk(n, 256);
  if (g > 4096) g = 4096;
  k_keys_d4<<<g, 256, 0, st>>>(sph64, n, keys, vals, bound_bits);
  ++g_launches;
  k_consts<<<1, 1, 0, st>>>(bound_bits, bc);
  ++g_launches;
  return cudaGetLastError();
}

cudaError_t sort_pairs(void* temp, size_t& temp_bytes, const uint32_t* kin, uint32_t* kout, const int* vin,
                       int* vout, int64_t n, cudaStream_t st) {
  if (temp) ++g_sort_calls;
  return cub::DeviceRadixSort::SortPairs(temp, temp_bytes, kin, kout, vin, vout, n, 0, 30, st);
}

cudaError_t sort_keys_u32(void* temp, size_t& temp_bytes, const uint32_t* kin, uint32_t* kout, int64_t n,
                          cudaStream_t st) {
  if (temp) ++g_sort_calls;
  return cub::DeviceRadixSort::SortKeys(temp, temp_bytes, kin, kout, n, 0, 32, st);
}

cudaError_t launch_gather_spheres(const D4* sph64, const int* order, int64_t n, const BuildConsts* bc, float tol32,
                                  double tol, float4* sph, float4* thr, float4* cvl, int* sid, cudaStream_t st) {
  k_gather_spheres<<<nblk(n, 256), 256, 0, st>>>(sph64, order, n, bc, tol32, tol, sph, thr, cvl, sid);
  ++g_launches;
  return cudaGetLastError();
}

cudaError_t launch_build_tree(const float4* items, int is_sphere, float A, Tree& T, unsigned* scratch,
                              cudaStream_t st) {
  if (T.nlevels == 0) return cudaSuccess;
  if (is_sphere) {
    for (int l = 0; l < T.nlevels; ++l) {
      const bool wide = wide_nodes(T.count[l]);
      const unsigned g = nblk(T.count[l], nodes_per_block(wide));
      if (l == 0) {
        if (wide) k_sphere_leaves<true><<<g, kNodeBlock, 0, st>>>(items, A, T);
        else k_sphere_leaves<false><<<g, kNodeBlock, 0, st>>>(items, A, T);
      } else {
        if (wide) k_sphere_level<true><<<g, kNodeBlock, 0, st>>>(A, T, l);
        else k_sphere_level<false><<<g, kNodeBlock, 0, st>>>(A, T, l);
      }
      ++g_launches;
    }
    if (scratch && T.nlevels > 1) {
      const int64_t nupper = T.offset[T.nlevels - 1] + T.count[T.nlevels - 1] - T.offset[1];
      const cudaError_t e = cudaMemsetAsync(scratch, 0, size_t(nupper) * kTight * sizeof(unsigned), st);
      if (e != cudaSuccess) return e;
      k_tighten_items<<<nblk(T.nitems, 256), 256, 0, st>>>(items, T, A, scratch);
      k_tighten_nodes<<<nblk(nupper, 128), 128, 0, st>>>(T, scratch, A, nupper);
      g_launches += 2;
    }
  } else {
    k_leaves<<<nblk(T.count[0], 128), 128, 0, st>>>(items, T.nitems, T.lo, T.hi, T.count[0]);
    ++g_launches;
    for (int l = 1; l < T.nlevels; ++l) {
      k_level<<<nblk(T.count[l], 128), 128, 0, st>>>(T.lo, T.hi, T.offset[l - 1], T.count[l - 1], T.offset[l],
                                                     T.count[l]);
      ++g_launches;
    }
  }
  return cudaGetLastError();
}

cudaError_t launch_query_keys(const double* x64, const float* x32, int64_t m, uint32_t* keys, int* vals,
                              cudaStream_t st) {
  if (m == 0) return cudaSuccess;
  k_query_keys<<<nblk(m, 256), 256, 0, st>>>(x64, x32, m, keys, vals);
  ++g_launches;
  return cudaGetLastError();
}

cudaError_t launch_point_keys(const float4* items, int64_t n, uint32_t* keys, int* vals, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_point_keys<<<nblk(n, 256), 256, 0, st>>>(items, n, keys, vals);
  ++g_launches;
  return cudaGetLastError();
}

cudaError_t launch_gather_points(const float4* src, const int* order, int64_t n, float4* dst, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_gather_points<<<nblk(n, 256), 256, 0, st>>>(src, order, n, dst);
  ++g_launches;
  return cudaGetLastError();
}

// Level by level over chunks of tiles (the chunk bounds the covering-ball
// array and the lists; a level's list has room for every candidate).
cudaError_t launch_cull(const CullArgs& one, const CullArgs* views, const int64_t* prefix, int ns, int64_t tiles,
                        const CullWork& w, cudaStream_t st) {
  CullSource s;
  s.views = views;
  s.prefix = prefix;
  s.ns = ns;
  s.hint = w.hint;
  s.list = w.list;
  s.groups = w.groups;
  s.K = one.K;
  s.KH = cull_kept(one.KH, tiles);
  s.few = tiles <= kCullFewTiles;
  unsigned* count = w.count;
  cudaError_t e = cudaMemsetAsync(w.count, 0, size_t(cull_launches(s.KH, tiles, w.chunk)) * 2 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  for (s.t0 = 0; s.t0 < tiles; s.t0 += w.chunk) {
    s.tiles = std::min(w.chunk, tiles - s.t0);
    s.k0 = 0;
    s.gcount = count;
    count += 2;
    for (int k1 = 12;; k1 = 4 * k1 - 6) {  // levels hold 12, 42, 162, ... directions (10 * 4^l + 2)
      s.k1 = k1 > s.KH ? one.K : k1;       // past the kept levels the directions do not depend on one another
      s.count = count;
      count += 2;
      const int dirs = s.k1 - s.k0;
      // directions per warp: 16 spread a tile's loads and the list's atomics;
      // fewer while the launch has less than 16 warps per SM
      const int D = int(std::max<int64_t>(1, std::min<int64_t>(16, s.tiles * dirs / (152 * 16))));
      const int chunks = (dirs + D - 1) / D;
      k_cull_test<<<unsigned((s.tiles * chunks + 3) / 4), 128, 0, st>>>(one, s, D, chunks);
      ++g_launches;
      if (!s.few) {
        k_cull_walk<<<152 * 8, 128, 0, st>>>(one, s);
        ++g_launches;
      }
      if (s.k1 == one.K) break;
      s.k0 = s.k1;
    }
    if (s.few || one.K > 12) {  // (the first level lists no groups)
      k_cull_groups<<<152 * 8, 128, 0, st>>>(one, s);
      ++g_launches;
    }
  }
  return cudaGetLastError();
}

template <int G>
static void query_spheres(const QueryArgs& a, const Packets& p, cudaStream_t st) {
  constexpr bool kMaySparse = G == 8 || G == kPacket;
  if (kMaySparse && p.sparse) {
    if constexpr (kMaySparse) {
      k_query_spheres<G, true><<<nblk(a.m, G), 32, 0, st>>>(a, p.lim);
      k_query_spheres_marked<G><<<unsigned(a.m), 32, 0, st>>>(a);
    }
  } else {
    k_query_spheres<G, false><<<nblk(a.m, G), 32, 0, st>>>(a, p.lim);
    if constexpr (G > 1) k_query_spheres_split<G><<<152 * 28, 32, 0, st>>>(a);
  }
  g_launches += G > 1 ? 2 : 1;
}

template <int G>
static void query_rest(const QueryArgs& a, const Packets& p, cudaStream_t st) {
  constexpr bool kMaySparse = G == 8 || G == kPacket;
  if (kMaySparse && p.sparse) {
    if constexpr (kMaySparse) {
      k_query_near<G, true><<<nblk(a.m, G), 32, 0, st>>>(a, p.lim);
      k_query_near_marked<G><<<unsigned(a.m), 32, 0, st>>>(a);
      k_query_decide<G, true><<<nblk(a.m, G), 32, 0, st>>>(a, p.lim);
      k_query_decide_marked<G><<<unsigned(a.m), 32, 0, st>>>(a);
    }
  } else {
    k_query_near<G, false><<<nblk(a.m, G), 32, 0, st>>>(a, p.lim);
    if constexpr (G > 1) k_query_near_split<G><<<152 * 28, 32, 0, st>>>(a);
    k_query_decide<G, false><<<nblk(a.m, G), 32, 0, st>>>(a, p.lim);
    if constexpr (G > 1) k_query_decide_split<G><<<152 * 24, 32, 0, st>>>(a);
  }
  g_launches += G > 1 ? 4 : 2;
}

cudaError_t launch_query_spheres(const QueryArgs& a, cudaStream_t st) {
  if (a.m == 0) return cudaSuccess;
  const Packets p = packets_of(a);
  switch (p.G) {
    case 1: query_spheres<1>(a, p, st); break;
    case 8: query_spheres<8>(a, p, st); break;
    case 32: query_spheres<32>(a, p, st); break;
    default: query_spheres<kPacket>(a, p, st);
  }
  return cudaGetLastError();
}

cudaError_t launch_query_finish(const QueryArgs& a, cudaStream_t st) {
  if (a.m == 0) return cudaSuccess;
  const Packets p = packets_of(a);
  switch (p.G) {
    case 1: query_rest<1>(a, p, st); break;
    case 8: query_rest<8>(a, p, st); break;
    case 32: query_rest<32>(a, p, st); break;
    default: query_rest<kPacket>(a, p, st);
  }
  return cudaGetLastError();
}

cudaError_t launch_query_exact(const QueryArgs& a, int all, cudaStream_t st) {
  if (a.m == 0) return cudaSuccess;
  if (all) {
    k_query_exact_all<<<nblk(a.m, 128), 128, 0, st>>>(a);
    ++g_launches;
  } else {
    unsigned int g = nblk(a.m, 128);
    if (g > 152u * 16u) g = 152u * 16u;
    k_query_exact_deferred<<<g, 128, 0, st>>>(a);
    ++g_launches;
  }
  return cudaGetLastError();
}

cudaError_t launch_grad(const GradArgs& a, int64_t n, float* grad_p, float* grad_sv, cudaStream_t st) {
  if (a.m > 0) k_query_grad<<<nblk(a.m, 128), 128, 0, st>>>(a);
  if (grad_p) k_fix_to_float<<<nblk(3 * n, 256), 256, 0, st>>>(a.acc_p, 3 * n, grad_p);
  if (grad_sv) k_fix_to_float<<<nblk(n, 256), 256, 0, st>>>(a.acc_s, n, grad_sv);
  return cudaGetLastError();
}

cudaError_t launch_collect_ids(const float4* s0, unsigned int n0, const float4* s1, unsigned int n1, const D4* sph64,
                               int KS, uint32_t* out, unsigned int* count, cudaStream_t st) {
  if (n0 + n1 == 0) return cudaSuccess;
  k_collect_ids<<<nblk(int64_t(n0) + n1, 256), 256, 0, st>>>(s0, n0, s1, n1, sph64, KS, out, count);
  ++g_launches;
  return cudaGetLastError();
}

cudaError_t launch_widen_ids(const uint32_t* in, int64_t n, int64_t* out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_widen_ids<<<nblk(n, 256), 256, 0, st>>>(in, n, out);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace gfs

#include "gfs_batch.cuh"
