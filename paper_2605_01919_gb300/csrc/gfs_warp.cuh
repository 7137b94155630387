// Warp-cooperative hierarchy walk shared by the GPU kernels (device code
// only: it uses warp intrinsics).
#pragma once

#include "gfs_internal.cuh"

namespace gfs {

// A warp's walk over a hierarchy with one stack stk of cap (+ kFan)
// entries: each round refresh() runs on every lane (false ends the walk),
// then the lanes take up to 32 nodes off the stack (walk_take); a lane calls
// leaf(index) for a leaf and need_child(node) for each child of an inner
// node, and the children it needs are pushed in lane order.  The lanes must
// enter together.
template <class Refresh, class NeedChild, class Leaf>
__device__ void warp_walk_until(const Tree& T, uint32_t* stk, int cap, int lane, Refresh refresh, NeedChild need_child,
                                Leaf leaf) {
  const unsigned kWarpAll = 0xffffffffu;
  if (T.nlevels == 0) return;
  const int top = T.nlevels - 1;
  int sp = int(T.count[top]);
  if (lane < sp) stk[lane] = pack_node(top, lane);
  __syncwarp();
  while (sp > 0) {
    if (!refresh()) return;
    const int take = walk_take(sp, cap, 32);
    const uint32_t nd = lane < take ? stk[sp - 1 - lane] : 0xffffffffu;
    sp -= take;
    __syncwarp();
    unsigned mask = 0;
    int64_t cb = 0;
    int lev = -1;
    if (nd != 0xffffffffu) {
      lev = node_level(nd);
      const int64_t idx = node_index(nd);
      if (lev == 0) {
        leaf(idx);
      } else {
        cb = idx * kFan;
        const int64_t ce = min(cb + kFan, T.count[lev - 1]);
        const int64_t off = T.offset[lev - 1];
        for (int64_t c = cb; c < ce; ++c)
          if (need_child(off + c)) mask |= 1u << unsigned(c - cb);
      }
    }
    const int cnt = __popc(mask);
    int pre = cnt;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kWarpAll, pre, o);
      if (lane >= o) pre += v;
    }
    const int total = __shfl_sync(kWarpAll, pre, 31);
    pre -= cnt;
    int w = sp + pre;
    for (int c = 0; c < kFan; ++c)
      if ((mask >> c) & 1u) stk[w++] = pack_node(lev - 1, cb + c);
    sp += total;
    __syncwarp();
  }
}

__device__ __forceinline__ float sqrt_fast(float v) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// distance and unit direction of (x, y, z) (direction 0 at distance 0)
__device__ __forceinline__ float unit3(float& x, float& y, float& z) {
  const float q = fmaf(x, x, fmaf(y, y, z * z));
  const float inv = q > 1e-36f ? rsqrtf(q) : 0.f;
  x *= inv;
  y *= inv;
  z *= inv;
  return q * inv;
}

// order-preserving bits of a float, and back
__device__ __forceinline__ unsigned ord_key(float v) {
  const unsigned b = __float_as_uint(v);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float ord_val(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// A node's linear bounds (struct Lin) at a point: direction and distance from
// the centre of its box, the box's support against -g and g (sp, sm), and the
// least |x - p| - |s| over its positive and negative spheres and |x - p| + |s|
// over all (an absent class: inf).  They hold within BuildConsts::elin, for
// points up to A (or A + R, a candidate's range).
struct LinAt {
  float nx, ny, nz, d, sp, sm;
  float pos, neg, far;
};
__device__ __forceinline__ LinAt lin_at(const Lin& q, float x, float y, float z) {
  LinAt r;
  r.nx = x - q.cx;
  r.ny = y - q.cy;
  r.nz = z - q.cz;
  r.d = unit3(r.nx, r.ny, r.nz);
  r.sp = fmaf(fabsf(r.nx + q.gx), q.hx, fmaf(fabsf(r.ny + q.gy), q.hy, fabsf(r.nz + q.gz) * q.hz));
  r.sm = fmaf(fabsf(r.nx - q.gx), q.hx, fmaf(fabsf(r.ny - q.gy), q.hy, fabsf(r.nz - q.gz) * q.hz));
  r.pos = r.d - q.hip - r.sp;
  r.neg = r.d + q.lon - r.sm;
  r.far = fminf(r.d + q.lop - r.sm, r.d - q.hin - r.sp);
  return r;
}
// the bounds' margin for an FP64 point in range rounded to FP32 (8 u A)
__device__ __forceinline__ float lin_point_margin(const BuildConsts& bc) {
  return bc.elin + 8.f * 5.9604644775390625e-8f * bc.A;
}

// (first node, nodes) of each level, in shared memory: lanes index it by the
// level of the entry they hold
struct LevelTable {
  int2 lv[kMaxLevels];
};
__device__ __forceinline__ void load_levels(const Tree& T, LevelTable& L, int lane) {
  __syncwarp();
  if (lane < kMaxLevels) L.lv[lane] = make_int2(int(T.offset[lane]), int(T.count[lane]));
  __syncwarp();
}

constexpr int kCoverStack = 512;  // walk stack entries of warp_cover_walk

// A sphere whose shrunk ball contains a point q (FP32 (x, y, z), the same on
// every lane), as its sorted slot, or -1: the warp walks the sphere hierarchy
// for the one point, 32 children or spheres a round.  Node test: the linear
// bound of |q - p| - |s| over the node's spheres stays below lim (-tol and
// the margins of the bound and of q's rounding); test(slot, v) decides a
// sphere (v: how deep, the least goes first when several hold the point).  The
// child that reaches deepest is visited first.  stk: kCoverStack entries.
template <class Test>
__device__ int warp_cover_walk(const Tree& T, const LevelTable& C, uint32_t* stk, int lane, float qx, float qy,
                               float qz, float lim, unsigned& n_nodes, unsigned& n_items, Test test) {
  const unsigned kAllLanes = 0xffffffffu;
  const int top = T.nlevels - 1, grp = lane >> 3, sub = lane & 7;
  int sp = C.lv[top].y;
  __syncwarp();
  if (lane < sp) stk[lane] = pack_node(top, lane);
  __syncwarp();
  while (sp > 0) {
    const int take = walk_take(sp, kCoverStack - kFan, 4);
    const uint32_t nd = grp < take ? stk[sp - 1 - grp] : 0xffffffffu;
    sp -= take;
    const int lev = node_level(nd);
    const int c = int(node_index(nd)) * kFan + sub;
    bool pass = false, cov = false;
    float v = INFINITY;
    if (nd != 0xffffffffu) {
      if (lev == 0) {
        if (c < T.nitems) {
          ++n_items;
          cov = test(c, v);
        }
      } else {
        const int2 L = C.lv[lev - 1];
        if (c < L.y) {
          ++n_nodes;
          const LinAt r = lin_at(lin_load(T, L.x + c), qx, qy, qz);
          v = fminf(r.pos, r.neg);
          pass = v <= lim;
        }
      }
    }
    if (__any_sync(kAllLanes, cov)) {
      const unsigned key = cov ? ord_key(v) : 0xffffffffu;
      return __shfl_sync(kAllLanes, c, __ffs(__ballot_sync(kAllLanes, key == __reduce_min_sync(kAllLanes, key))) - 1);
    }
    // the child that reaches deepest around the point goes on top, below it
    // those that reach at least half as deep
    const unsigned key = pass ? ord_key(v) : 0xffffffffu;
    const unsigned low = __reduce_min_sync(kAllLanes, key);
    const float deep = ord_val(low);
    const unsigned bn = __ballot_sync(kAllLanes, pass);
    const unsigned bq = __ballot_sync(kAllLanes, pass && v < 0.5f * deep);
    if (pass) {
      const unsigned bb = __ballot_sync(bn, key == low);
      const unsigned best = bb & (0u - bb), rest = bn & ~bq & ~best, good = bq & ~best, me = 1u << lane;
      const int at = (me & best) ? __popc(bn) - 1
                                 : ((me & good) ? __popc(rest) + __popc(good & (me - 1u)) : __popc(rest & (me - 1u)));
      stk[sp + at] = pack_node(lev - 1, c);
    }
    sp += __popc(bn);
    __syncwarp();
  }
  return -1;
}

}  // namespace gfs
