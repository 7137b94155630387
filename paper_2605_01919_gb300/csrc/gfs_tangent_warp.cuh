// Same-sign tangent augmentation, one warp per point (device code only).
//
// The steps and every FP64 expression are those of tangent_one in
// gfs_tangent.cuh (the host build checks that routine against the oracle);
// here the 32 lanes of a warp walk the sphere hierarchy for one point
// together: each round they take up to 32 nodes off a shared stack
// (warp_walk_until), every lane screens and evaluates its own nodes and
// leaves, and between rounds the lanes merge what they found.  The results
// are minima with fixed tie rules (the class distance with the lowest
// index, the far bound, the tangent point with the lowest id) and a
// containment OR, so they do not depend on which lane found what or in
// which round; the thresholds a round prunes with are the merged results
// of the rounds before it, which only ever prunes what cannot change them.
#pragma once

#include "gfs_tangent.cuh"
#include "gfs_warp.cuh"

namespace gfs {
namespace tangent {

constexpr unsigned kLanes = 0xffffffffu;
constexpr int kWarpStack = 512 + kDepthReserve;  // per-warp walk stack entries (plus a reserve of kFan)

// lexicographic minimum of (v, i) over the warp, on every lane
__device__ __forceinline__ void warp_min_vi(double& v, int& i) {
  for (int o = 16; o > 0; o >>= 1) {
    const double v2 = __shfl_xor_sync(kLanes, v, o);
    const int i2 = __shfl_xor_sync(kLanes, i, o);
    if (v2 < v || (v2 == v && i2 < i)) {
      v = v2;
      i = i2;
    }
  }
}

__device__ __forceinline__ void warp_min_vl(double& v, int64_t& i) {
  for (int o = 16; o > 0; o >>= 1) {
    const double v2 = __shfl_xor_sync(kLanes, v, o);
    const long long i2 = __shfl_xor_sync(kLanes, (long long)i, o);
    // id -1 (nothing found) sorts last
    const bool better = v2 < v || (v2 == v && i2 >= 0 && (i < 0 || i2 < i));
    if (better) {
      v = v2;
      i = i2;
    }
  }
}

// sphere_bounds over the warp; every lane receives the result.  stk: the
// warp's stack (kWarpStack + kFan entries).
__device__ inline void warp_sphere_bounds(const QueryArgs& a, double x, double y, double z, uint32_t* stk, int lane,
                                          SphereBounds& R) {
  const double tol = a.tol;
  R.cov[0] = R.cov[1] = false;
  R.bestA[0] = R.bestA[1] = INFINITY;
  R.idxA[0] = R.idxA[1] = INT_MAX;
  R.bestF = INFINITY;
  const float x32 = float(x), y32 = float(y), z32 = float(z), ax = amax3(x32, y32, z32);
  float thF = INFINITY, thA[2] = {INFINITY, INFINITY};
  const Tree& T = a.st;
  if (T.nlevels == 0) return;
  auto item = [&](int64_t j) {
    const float4 S = a.sph[j];
    const float d32 = dist32(x32, y32, z32, S), r32 = fabsf(S.w);
    const float er = err32(ax, S, d32, r32);
    bool need = d32 + r32 - er <= thF;
    if (S.w != 0.f) need = need || d32 - r32 - er <= thA[S.w < 0.f];
    if (!need) return;
    const int o = a.sid[j];
    const D4 P = a.sph64[o];
    const double d2 = ex_d2(x, y, z, P.x, P.y, P.z);
    const double dl = __dsqrt_rn(d2);
    const double r = fabs(P.w);
    if (P.w != 0.0) {
      const int c = P.w < 0.0;
      if (!R.cov[c] && r > tol) {
        const double rt = __dsub_rn(r, tol);
        if (d2 < __dmul_rn(rt, rt)) R.cov[c] = true;
      }
      const double av = __dsub_rn(dl, r);
      if (av < R.bestA[c] || (av == R.bestA[c] && o < R.idxA[c])) {
        R.bestA[c] = av;
        R.idxA[c] = o;
      }
      // this lane's thresholds tighten at once, the warp's at the next merge
      thA[c] = fminf(thA[c], f_up(R.cov[c] ? R.bestA[c] : fmax(R.bestA[c], -tol)));
    }
    const double f = __dadd_rn(dl, r);
    if (f < R.bestF) {
      R.bestF = f;
      thF = fminf(thF, f_up(f));
    }
  };
  auto merge = [&]() {
    R.cov[0] = __any_sync(kLanes, R.cov[0]);
    R.cov[1] = __any_sync(kLanes, R.cov[1]);
    warp_min_vi(R.bestA[0], R.idxA[0]);
    warp_min_vi(R.bestA[1], R.idxA[1]);
    for (int o = 16; o > 0; o >>= 1) R.bestF = fmin(R.bestF, __shfl_xor_sync(kLanes, R.bestF, o));
    // FP32 copies (rounded up) of the thresholds a sphere must reach to
    // matter (per class at least -tol while the class has no containing ball)
    thF = f_up(R.bestF);
    for (int c = 0; c < 2; ++c) thA[c] = f_up(R.cov[c] ? R.bestA[c] : fmax(R.bestA[c], -tol));
  };
  // seed: the leaf whose balls reach nearest to x (the same greedy descent
  // on every lane), its items split over the lanes
  {
    const int top = T.nlevels - 1;
    int64_t best = 0;
    float bk = INFINITY;
    for (int64_t j = 0; j < T.count[top]; ++j) {
      const float4 B = T.na[T.offset[top] + j];
      const float k = dist32(x32, y32, z32, B) - B.w;
      if (k < bk) {
        bk = k;
        best = j;
      }
    }
    for (int lev = top; lev > 0; --lev) {
      const int64_t cb = best * kFan, ce = imin64(cb + kFan, T.count[lev - 1]);
      const int64_t off = T.offset[lev - 1];
      bk = INFINITY;
      for (int64_t c = cb; c < ce; ++c) {
        const float4 B = T.na[off + c];
        const float k = dist32(x32, y32, z32, B) - B.w;
        if (k < bk || c == cb) {
          bk = k;
          best = c;
        }
      }
    }
    const int64_t j = best * kLeaf + lane;
    if (lane < kLeaf && j < a.n) item(j);
    merge();
  }
  warp_walk_until(
      T, stk, kWarpStack, lane,
      [&]() {
        merge();
        return true;
      },
      [&](int64_t node) {
        const float4 B = T.na[node], W = T.nb[node], Fb = T.nf[node];
        const float dF = dist32(x32, y32, z32, Fb);
        if (dF - err32(ax, Fb, dF, Fb.w) - Fb.w <= thF) return true;
        const float dC = dist32(x32, y32, z32, B);
        for (int cl = 0; cl < 2; ++cl) {
          const float w = cl == 0 ? W.x : W.y;
          if (!(w > -INFINITY)) continue;
          if (dC - err32(ax, B, dC, w) - w <= thA[cl]) return true;
        }
        return false;
      },
      [&](int64_t idx) {
        const int64_t b = idx * kLeaf, e = imin64(b + kLeaf, a.n);
        for (int64_t j = b; j < e; ++j) item(j);
      });
  merge();
}

// tangent_search over the warp; every lane receives the result.
__device__ inline void warp_tangent_search(const QueryArgs& a, int box_cull, double x, double y, double z, int cs,
                                           int mode, double lim, double lo, uint32_t* stk, int lane, TanBest& B) {
  const Tree& T = a.st;
  const double lim_d = mode == kBelowSurvivor ? sqrt(lim) : (mode == kWithinOpposite ? lim : INFINITY);
  const float x32 = float(x), y32 = float(y), z32 = float(z), ax = amax3(x32, y32, z32);
  const float lo_f = f_dn(lo);
  float hi_f = INFINITY;
  int hint = -1;  // the ball that covered this lane's last tangent point
  auto merge = [&]() {
    warp_min_vl(B.d2, B.id);
    // distances beyond hi cannot change the result
    const double hi = (B.id >= 0 ? fmin(lim_d, sqrt(B.d2)) : lim_d) * kRel + kAbs;
    hi_f = f_up(hi);
  };
  merge();
  warp_walk_until(
      T, stk, kWarpStack, lane,
      [&]() {
        merge();
        return true;
      },
      [&](int64_t node) {
        const float4 W = T.nb[node];
        const float w = cs == 0 ? W.x : W.y;
        if (!(w > -INFINITY)) return false;
        const float4 Cb = T.na[node], Fb = T.nf[node];
        const float dc = dist32(x32, y32, z32, Cb), df = dist32(x32, y32, z32, Fb);
        const float ec = err32(ax, Cb, dc, w), ef = err32(ax, Fb, df, Fb.w);
        const float near_lo = dc - w - ec, near_hi = fmaxf(w - dc + ec, df + Fb.w + ef);
        const float far_lo = df - Fb.w - ef, far_hi = dc + w + ec;
        return (near_lo <= hi_f && near_hi >= lo_f) || (far_lo <= hi_f && far_hi >= lo_f);
      },
      [&](int64_t idx) {
        const int64_t b = idx * kLeaf, e = imin64(b + kLeaf, a.n);
        for (int64_t j = b; j < e; ++j) {
          const float4 S = a.sph[j];
          if (S.w == 0.f || int(S.w < 0.f) != cs) continue;
          const float d32 = dist32(x32, y32, z32, S), r32 = fabsf(S.w);
          const float er = err32(ax, S, d32, r32);
          const float an32 = fabsf(d32 - r32), af32 = d32 + r32;
          const bool try_near = an32 + er >= lo_f && an32 - er <= hi_f;
          const bool try_far = af32 + er >= lo_f && af32 - er <= hi_f;
          if (!try_near && !try_far) continue;
          const int o = a.sid[j];
          const D4 P = a.sph64[o];
          const double r = fabs(P.w);
          const double vx = __dsub_rn(x, P.x), vy = __dsub_rn(y, P.y), vz = __dsub_rn(z, P.z);
          const double dv =
              __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)), __dmul_rn(vz, vz)));
          if (!(dv > 0.0)) continue;
          const double ux = __ddiv_rn(vx, dv), uy = __ddiv_rn(vy, dv), uz = __ddiv_rn(vz, dv);
          for (int side = 0; side < 2; ++side) {
            if (!(side == 0 ? try_near : try_far)) continue;
            const double sr = side == 0 ? r : -r;
            const double tx = __dadd_rn(P.x, __dmul_rn(sr, ux));
            const double ty = __dadd_rn(P.y, __dmul_rn(sr, uy));
            const double tz = __dadd_rn(P.z, __dmul_rn(sr, uz));
            if (box_cull && !ex_inbox(tx, ty, tz)) continue;
            const double d2 = ex_d2(x, y, z, tx, ty, tz);
            const bool within =
                mode == kBelowSurvivor ? d2 < lim : (mode == kWithinOpposite ? __dsqrt_rn(d2) <= lim : true);
            if (!within) continue;
            const int64_t id = 2 * int64_t(o) + side;
            if (B.id >= 0 && (d2 > B.d2 || (d2 == B.d2 && id > B.id))) continue;
            if (hint >= 0 && hint != o && ex_cov(tx, ty, tz, a.sph64[hint], a.tol)) continue;
            const int k = covered_by_other(a, tx, ty, tz, o);
            if (k >= 0) {
              hint = k;
              continue;
            }
            B.d2 = d2;
            B.id = id;
          }
        }
      });
  merge();
}

// ---------------------------------------------------------------------------
// The same two walks for points in the coordinate range [-A, A]^3 of the FP32
// bounds: 4 entries a round, each lane tests one child or one sphere, and a
// node has to pass its linear bounds (struct Lin) instead of the balls around
// its spheres.  A tangent point that may win is tested against the balls that
// held the point's latest covered ones, then walked by the whole warp, the
// nearest first, so an uncovered one ends the search early.  Bound: the latency
// of those walks (dependent rounds of 4 entries).  31,607 points of a 64^3 union
// grid take 14 ms, with the lanes walking apart by ball bounds 30 ms, with one
// point a lane 53 ms.  Points outside the range take the walks above.
// ---------------------------------------------------------------------------

constexpr int kTanRecent = 8;

static_assert(kWarpStack + kFan >= kCoverStack, "warp_lin_walk's stack");
struct TanWarp {
  uint32_t stk[kWarpStack + kFan], cstk[kCoverStack];  // (the first serves both kinds of walk)
  float4 rec[kTanRecent];  // (centre, squared distance below which a point is held for sure)
  int rec_id[kTanRecent];  // sorted slot
};

__device__ __forceinline__ float warp_min_f(float v) { return ord_val(__reduce_min_sync(kLanes, ord_key(v))); }

// node(global node, lin, level) -> visit its children; items(slot or -1) runs
// on all lanes in rounds that reach leaves.  Stack bound as in warp_cover_walk.
template <class Node, class Items>
__device__ __forceinline__ void warp_lin_walk(const Tree& T, const LevelTable& C, uint32_t* stk, int lane, Node node,
                                              Items items) {
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
    const bool leaf = nd != 0xffffffffu && lev == 0;
    bool pass = false;
    if (nd != 0xffffffffu && lev > 0) {
      const int2 L = C.lv[lev - 1];
      if (c < L.y) pass = node(int64_t(L.x) + c);
    }
    const unsigned bn = __ballot_sync(kLanes, pass);
    // children of the deepest popped entry end up on top
    if (pass) stk[sp + __popc(bn >> lane >> 1)] = pack_node(lev - 1, c);
    sp += __popc(bn);
    if (__any_sync(kLanes, leaf)) items(leaf && c < T.nitems ? c : -1);
    __syncwarp();
  }
}

// warp_sphere_bounds by that walk.
__device__ inline void warp_sphere_bounds_lin(const QueryArgs& a, const LevelTable& C, double x, double y, double z,
                                              TanWarp& W, int lane, SphereBounds& R) {
  const double tol = a.tol;
  R.cov[0] = R.cov[1] = false;
  R.bestA[0] = R.bestA[1] = INFINITY;
  R.idxA[0] = R.idxA[1] = INT_MAX;
  R.bestF = INFINITY;
  const Tree& T = a.st;
  if (T.nlevels == 0) return;
  const float x32 = float(x), y32 = float(y), z32 = float(z), ax = amax3(x32, y32, z32);
  const float mg = lin_point_margin(*a.bc);
  float thF = INFINITY, thA[2] = {INFINITY, INFINITY};
  auto item = [&](int64_t j) -> bool {
    const float4 S = a.sph[j];
    const float d32 = dist32(x32, y32, z32, S), r32 = fabsf(S.w);
    const float er = err32(ax, S, d32, r32);
    bool need = d32 + r32 - er <= thF;
    if (S.w != 0.f) need = need || d32 - r32 - er <= (S.w < 0.f ? thA[1] : thA[0]);
    if (!need) return false;
    const int o = a.sid[j];
    const D4 P = a.sph64[o];
    const double d2 = ex_d2(x, y, z, P.x, P.y, P.z);
    const double dl = __dsqrt_rn(d2);
    const double r = fabs(P.w);
    if (P.w != 0.0) {
      const bool in = r > tol && d2 < __dmul_rn(__dsub_rn(r, tol), __dsub_rn(r, tol));
      const double av = __dsub_rn(dl, r);
#pragma unroll
      for (int c = 0; c < 2; ++c)
        if (c == int(P.w < 0.0)) {
          R.cov[c] = R.cov[c] || in;
          if (av < R.bestA[c] || (av == R.bestA[c] && o < R.idxA[c])) {
            R.bestA[c] = av;
            R.idxA[c] = o;
          }
          thA[c] = fminf(thA[c], f_up(R.cov[c] ? R.bestA[c] : fmax(R.bestA[c], -tol)));
        }
    }
    const double f = __dadd_rn(dl, r);
    if (f < R.bestF) {
      R.bestF = f;
      thF = fminf(thF, f_up(f));
    }
    return true;
  };
  // thresholds of all lanes (a lane's are sound for the warp: its class is
  // covered if the lane says so, and the least value is at most its own)
  auto items = [&](int64_t j) {
    const bool got = j >= 0 && item(j);
    if (!__any_sync(kLanes, got)) return;
    thF = warp_min_f(thF);
    thA[0] = warp_min_f(thA[0]);
    thA[1] = warp_min_f(thA[1]);
  };
  // seed: each group of 8 lanes descends for one quantity (class 0, class 1,
  // far bound, any ball), the child with the least bound at every level
  {
    const int grp = lane >> 3, sub = lane & 7;
    int lev = T.nlevels - 1;
    int64_t node = sub;
    bool valid = sub < C.lv[lev].y;
    for (;;) {
      float v = INFINITY;
      if (valid) {
        const int64_t nd = C.lv[lev].x + node;
        const float4 B = grp == 2 ? T.nf[nd] : T.na[nd];
        float w = B.w;
        if (grp < 2) w = grp == 0 ? T.nb[nd].x : T.nb[nd].y;
        v = dist32(x32, y32, z32, B) - w;
      }
      unsigned key = v < INFINITY ? (ord_key(v) & ~7u) | unsigned(sub) : 0xffffffffu;
      for (int o = 4; o > 0; o >>= 1) key = min(key, __shfl_xor_sync(kLanes, key, o));
      const int64_t next = __shfl_sync(kLanes, (long long)node, (lane & 24) | int(key & 7u)) * kFan + sub;
      valid = key != 0xffffffffu;
      node = next;
      if (lev == 0) break;
      --lev;
      valid = valid && node < C.lv[lev].y;
    }
    items(valid && node < T.nitems ? node : -1);
  }
  warp_lin_walk(
      T, C, W.stk, lane,
      [&](int64_t nd) {
        const LinAt b = lin_at(lin_load(T, nd), x32, y32, z32);
        // (an absent class: inf - inf compares false)
        return b.pos - thA[0] <= mg || b.neg - thA[1] <= mg || b.far - thF <= mg;
      },
      items);
  R.cov[0] = __any_sync(kLanes, R.cov[0]);
  R.cov[1] = __any_sync(kLanes, R.cov[1]);
  warp_min_vi(R.bestA[0], R.idxA[0]);
  warp_min_vi(R.bestA[1], R.idxA[1]);
  for (int o = 16; o > 0; o >>= 1) R.bestF = fmin(R.bestF, __shfl_xor_sync(kLanes, R.bestF, o));
}

// warp_tangent_search by that walk.
__device__ inline void warp_tangent_search_lin(const QueryArgs& a, const LevelTable& C, int box_cull, double x,
                                               double y, double z, int cs, int mode, double lim, double lo,
                                               TanWarp& W, int lane, TanBest& B) {
  const Tree& T = a.st;
  if (T.nlevels == 0) return;
  const float A = a.bc->A;
  const double lim_d = mode == kBelowSurvivor ? sqrt(lim) : (mode == kWithinOpposite ? lim : INFINITY);
  const float x32 = float(x), y32 = float(y), z32 = float(z), ax = amax3(x32, y32, z32);
  const float lo_f = f_dn(lo);
  const float mg = lin_point_margin(*a.bc);
  const float cover_lim = -a.tol32 + a.bc->elin;
  float hi_f = f_up(lim_d * kRel + kAbs);
  int nrec = 0, at = 0;
  unsigned n_nodes = 0, n_items = 0;
  auto tangent_point = [&](int o, int side, double t[3]) -> bool {
    const D4 P = a.sph64[o];
    const double r = fabs(P.w);
    const double vx = __dsub_rn(x, P.x), vy = __dsub_rn(y, P.y), vz = __dsub_rn(z, P.z);
    const double dv = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)), __dmul_rn(vz, vz)));
    if (!(dv > 0.0)) return false;
    const double sr = side == 0 ? r : -r;
    t[0] = __dadd_rn(P.x, __dmul_rn(sr, __ddiv_rn(vx, dv)));
    t[1] = __dadd_rn(P.y, __dmul_rn(sr, __ddiv_rn(vy, dv)));
    t[2] = __dadd_rn(P.z, __dmul_rn(sr, __ddiv_rn(vz, dv)));
    return true;
  };
  // one candidate per lane (sphere at sorted slot j, or -1): all are settled
  auto settle = [&](int j, int o, int side) {
    bool open = j >= 0;
    double t[3] = {0.0, 0.0, 0.0}, d2 = INFINITY;
    if (open) open = tangent_point(o, side, t);
    if (open && box_cull) open = ex_inbox(t[0], t[1], t[2]);
    if (open) {
      d2 = ex_d2(x, y, z, t[0], t[1], t[2]);
      open = mode == kBelowSurvivor ? d2 < lim : (mode == kWithinOpposite ? __dsqrt_rn(d2) <= lim : true);
    }
    const int64_t id = 2 * int64_t(o) + side;
    const float tx = float(t[0]), ty = float(t[1]), tz = float(t[2]);
    const bool in_range = fabs(t[0]) <= A && fabs(t[1]) <= A && fabs(t[2]) <= A;
    auto held = [&](const float4& P) {
      const float dx = tx - P.x, dy = ty - P.y, dz = tz - P.z;
      return fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < P.w;
    };
    if (open && in_range)
      for (int u = 0; u < nrec; ++u)
        if (W.rec_id[u] != j && held(W.rec[u])) open = false;
    for (;;) {
      if (open && B.id >= 0 && (d2 > B.d2 || (d2 == B.d2 && id > B.id))) open = false;
      const unsigned key = open ? __float_as_uint(float(d2)) : 0xffffffffu;
      const unsigned low = __reduce_min_sync(kLanes, key);
      const unsigned m = __ballot_sync(kLanes, open && key == low);
      if (!m) return;
      const int src = __ffs(m) - 1;
      const int cj = __shfl_sync(kLanes, j, src);
      bool covered;
      if (__shfl_sync(kLanes, int(in_range), src)) {
        const double qx = __shfl_sync(kLanes, t[0], src), qy = __shfl_sync(kLanes, t[1], src),
                     qz = __shfl_sync(kLanes, t[2], src);
        const float qxf = float(qx), qyf = float(qy), qzf = float(qz);
        const int s = warp_cover_walk(T, C, W.cstk, lane, qxf, qyf, qzf, cover_lim, n_nodes, n_items,
                                      [&](int c, float& v) {
                                        if (c == cj) return false;
                                        const float4 P = a.sph[c], Th = a.thr[c];
                                        const float dx = qxf - P.x, dy = qyf - P.y, dz = qzf - P.z;
                                        const float e2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                                        if (!(e2 <= Th.w)) return false;
                                        v = e2 - Th.z;
                                        return e2 < Th.z || ex_cov(qx, qy, qz, a.sph64[a.sid[c]], a.tol);
                                      });
        covered = s >= 0;
        if (covered) {
          float4 P = a.sph[s];
          P.w = a.thr[s].z;
          if (open && in_range && j != s && held(P)) open = false;
          __syncwarp();
          if (lane == 0) {
            W.rec[at] = P;
            W.rec_id[at] = s;
          }
          at = (at + 1) % kTanRecent;
          nrec = min(nrec + 1, kTanRecent);
          __syncwarp();
        }
      } else {
        covered = __shfl_sync(kLanes, lane == src ? int(covered_by_other(a, t[0], t[1], t[2], o) >= 0) : 0, src);
      }
      if (!covered) {
        B.d2 = __shfl_sync(kLanes, d2, src);
        B.id = __shfl_sync(kLanes, (long long)id, src);
        hi_f = f_up(fmin(lim_d, sqrt(B.d2)) * kRel + kAbs);
      }
      if (lane == src) open = false;
    }
  };
  warp_lin_walk(
      T, C, W.stk, lane,
      [&](int64_t nd) {
        // bounds over the node's spheres of the class, d = |x - p| and r = |s|:
        // linear from below; from above d - r <= D - res + S(n +- g) +
        // |h|^2 / (2 (D - |h|)) (the chord's excess over its projection on n),
        // res the least residual of r, or |x - F| + wf
        const Lin q = lin_load(T, nd);
        const LinAt b = lin_at(q, x32, y32, z32);
        const float near_lo = cs == 0 ? b.pos : b.neg;
        if (!(near_lo < INFINITY)) return false;  // none of the class
        const float far_lo = cs == 0 ? b.d + q.lop - b.sm : b.d - q.hin - b.sp;
        if (far_lo - hi_f <= mg) return true;
        if (!(near_lo - hi_f <= mg)) return false;
        if (-near_lo + mg >= lo_f) return true;
        const float h2 = fmaf(q.hx, q.hx, fmaf(q.hy, q.hy, q.hz * q.hz)), hn = sqrtf(h2);
        const float over = b.d > 2.f * hn ? 0.5f * h2 / (b.d - hn) * (1.f + 1e-5f) : INFINITY;
        const float up = (cs == 0 ? b.d - q.lop + b.sp : b.d + q.hin + b.sm) + over;
        if (!(up + mg >= lo_f)) return false;
        const float4 Fb = T.nf[nd];
        const float df = dist32(x32, y32, z32, Fb);
        return df + Fb.w + err32(ax, Fb, df, Fb.w) >= lo_f;
      },
      [&](int64_t j) {
        bool near = false, far = false;
        int o = 0;
        if (j >= 0) {
          const float4 S = a.sph[j];
          if (S.w != 0.f && int(S.w < 0.f) == cs) {
            // screen: |x - t| is |d - r| (near) or d + r (far)
            const float d32 = dist32(x32, y32, z32, S), r32 = fabsf(S.w);
            const float er = err32(ax, S, d32, r32);
            const float an32 = fabsf(d32 - r32), af32 = d32 + r32;
            near = an32 + er >= lo_f && an32 - er <= hi_f;
            far = af32 + er >= lo_f && af32 - er <= hi_f;
            if (near || far) o = a.sid[j];
          }
        }
        if (__any_sync(kLanes, near)) settle(near ? int(j) : -1, o, 0);
        if (__any_sync(kLanes, far)) settle(far ? int(j) : -1, o, 1);
      });
}

// tangent_one over the warp (lane 0 writes the outputs).
__device__ inline void warp_tangent_one(const QueryArgs& a, const LevelTable& C, int box_cull, int64_t q, TanWarp& W,
                                        int lane) {
  const int code = a.fl_out[q] & 15;
  if (code != GFS_CODE_SURVIVOR && code != GFS_CODE_OPPOSITE && code != GFS_CODE_LOWER) return;
  double x, y, z;
  load_point(a, q, x, y, z);
  SphereBounds S;
  const float A = a.bc->A;
  const bool lin = fabs(x) <= A && fabs(y) <= A && fabs(z) <= A;
  if (lin) warp_sphere_bounds_lin(a, C, x, y, z, W, lane, S);
  else warp_sphere_bounds(a, x, y, z, W.stk, lane, S);
  if (S.cov[0] == S.cov[1]) return;  // OUTSIDE / INVALID: not refined
  const int cs = S.cov[0] ? 0 : 1, co = 1 - cs;
  const bool have_u = S.idxA[co] != INT_MAX;
  const double ub = have_u ? S.bestA[co] : INFINITY;
  int mode = kUnlimited;
  double lim = INFINITY;
  if (code == GFS_CODE_SURVIVOR) {
    double qx, qy, qz;
    if (!survivor_pos(a, a.arg_out[q], qx, qy, qz)) return;  // not this state's query output
    mode = kBelowSurvivor;
    lim = ex_d2(x, y, z, qx, qy, qz);
  } else if (code == GFS_CODE_OPPOSITE) {
    mode = kWithinOpposite;
    lim = ub;
  }
  const double lbv = -S.bestA[cs];
  const double lo = lbv - a.tol - 1e-9 - 1e-12 * fabs(lbv);
  TanBest B;
  B.d2 = INFINITY;
  B.id = -1;
  __syncwarp();
  if (lin) warp_tangent_search_lin(a, C, box_cull, x, y, z, cs, mode, lim, lo, W, lane, B);
  else warp_tangent_search(a, box_cull, x, y, z, cs, mode, lim, lo, W.stk, lane, B);
  if (B.id < 0 || lane != 0) return;
  const double m = __dsqrt_rn(B.d2);
  if (a.clamp_opp && !(m <= ub)) return;  // the opposite tangent point stays the value
  const double lb = -S.bestA[cs];
  int flags = GFS_CODE_TANGENT;
  if (m < __dsub_rn(lb, a.tol)) flags |= GFS_FLAG_LB_VIOL;
  if (m > __dadd_rn(S.bestF, a.tol)) flags |= GFS_FLAG_FAR_VIOL;
  if (have_u && ub < __dsub_rn(m, a.tol)) flags |= GFS_FLAG_OPP_VIOL;
  const double v = cs == 0 ? m : -m;
  if (a.s_out) a.s_out[q] = float(v);
  if (a.s64_out) a.s64_out[q] = v;
  a.arg_out[q] = B.id;
  a.fl_out[q] = uint16_t(flags);
}

}  // namespace tangent
}  // namespace gfs
