// Scored value, one warp per point (device code only).
//
// The candidates, their order and every FP64 expression are those of
// scored_one in gfs_scored.cuh (the host build checks that routine against the
// oracle).  Here the 32 lanes walk the hierarchies for one point together: in
// the survivor walks (warp_walk_until) each lane screens and evaluates its own
// nodes and items and keeps its own best, shared between rounds; the tangent
// points come from the walk by linear bounds (warp_lin_walk), the best open one
// is settled first, its coverage walked by the whole warp.  The chosen candidate
// is the greatest valid one of a total order, so it does not depend on which
// lane met it or when: a candidate is only dropped when a better one is known
// or when it is not valid, and the two least farthest-survivor distances are
// minima over distinct spheres.
// Bound: latency, of the coverage walks and of the FP64 tests.  8,191 points of a
// 48^3 union grid take 10 ms; 27 ms with ball bounds and a coverage walk per
// lane, 145 ms with one point a lane.
#pragma once

#include "gfs_scored.cuh"
#include "gfs_tangent_warp.cuh"
#include "gfs_warp.cuh"

namespace gfs {
namespace scored {

constexpr unsigned kLanes = 0xffffffffu;

// the best of the warp's candidates, on every lane
__device__ __forceinline__ void warp_best(Best& B) {
  for (int o = 16; o > 0; o >>= 1) {
    Best c;
    c.cls = __shfl_xor_sync(kLanes, B.cls, o);
    c.sr = __shfl_xor_sync(kLanes, B.sr, o);
    c.key = __shfl_xor_sync(kLanes, (long long)B.key, o);
    c.sign = __shfl_xor_sync(kLanes, B.sign, o);
    c.r = __shfl_xor_sync(kLanes, B.r, o);
    if (c.cls >= 0 && better(c.cls, c.sr, c.key, c.sign, B)) B = c;
  }
}

// Walk of one survivor hierarchy: item(g) for every survivor whose FP32 screen
// allows an exact distance <= R.
template <class Refresh, class Item>
__device__ inline void warp_survivors(const QueryArgs& a, const Frame& F, int cls, double R, uint32_t* stk, int lane,
                                      Refresh refresh, Item item) {
  const Tree& T = a.vt[cls];
  const float R32 = f_up(R);
  const float4* items = a.surv[cls];
  const float eq4 = 4.f * a.bc->eq;
  warp_walk_until(
      T, stk, tangent::kWarpStack, lane, refresh,
      [&](int64_t node) {
        const float bd = sqrtf(box_d2(F.x32, F.y32, F.z32, T.lo[node], T.hi[node]));
        return bd * (1.f - 1e-6f) - eq4 <= R32;
      },
      [&](int64_t idx) {
        const int64_t b = idx * kLeaf, e = imin64(b + kLeaf, T.nitems);
        for (int64_t j = b; j < e; ++j) {
          const float4 S = items[j];
          const float d32 = dist32(F.x32, F.y32, F.z32, S);
          if (d32 - err32(F.ax, S, d32, 0.f) - eq4 > R32) continue;
          item(__float_as_uint(S.w));
        }
      });
}

__device__ inline void warp_scored_one(const QueryArgs& a, int box_cull, const uint32_t* __restrict__ csr_ids,
                                       const int64_t* __restrict__ csr_off, const LevelTable& C, int64_t q,
                                       tangent::TanWarp& W, int lane) {
  const int code = a.fl_out[q] & 15;
  if (code == GFS_CODE_SAMPLE || code == GFS_CODE_INVALID) return;
  const double tol = a.tol;
  Frame F;
  tangent::load_point(a, q, F.x, F.y, F.z);
  F.x32 = float(F.x);
  F.y32 = float(F.y);
  F.z32 = float(F.z);
  F.ax = amax3(F.x32, F.y32, F.z32);
  tangent::SphereBounds SB;
  uint32_t* const stk = W.stk;
  const float A = a.bc->A;
  const bool lin = fabs(F.x) <= A && fabs(F.y) <= A && fabs(F.z) <= A;  // the range of the linear bounds
  if (lin) tangent::warp_sphere_bounds_lin(a, C, F.x, F.y, F.z, W, lane, SB);
  else tangent::warp_sphere_bounds(a, F.x, F.y, F.z, stk, lane, SB);
  if (SB.cov[0] && SB.cov[1]) return;  // INVALID (the plain query says so too)
  F.sig = SB.cov[0] ? 1 : (SB.cov[1] ? -1 : 0);
  F.ub[0] = SB.bestA[1];
  F.ub[1] = SB.bestA[0];
  F.far = SB.bestF;
  const double R = __dadd_rn(F.far, tol);  // no valid radius exceeds it (V3)
  // (V2) per lane the two least of its spheres' farthest-survivor distances
  F.m1 = F.m2 = INFINITY;
  F.j1 = F.j2 = -1;
  int64_t seen[4] = {-1, -1, -1, -1};
  int seen_at = 0;
  auto v2_sphere = [&](uint32_t g) {
    const int64_t i = int64_t(g) / a.KS;
    if (i == F.j1 || i == F.j2 || i == seen[0] || i == seen[1] || i == seen[2] || i == seen[3]) return;
    seen[seen_at] = i;
    seen_at = (seen_at + 1) & 3;
    double md = -1.0;
    const int64_t u0 = csr_off[i], u1 = imin64(csr_off[i + 1], u0 + a.KS);  // at most KS per sphere
    for (int64_t u = u0; u < u1; ++u) {
      double qx, qy, qz;
      tangent::survivor_pos(a, int64_t(csr_ids[u]), qx, qy, qz);
      const double d2 = ex_d2(F.x, F.y, F.z, qx, qy, qz);
      if (d2 > md) md = d2;
      if (md >= F.m2) return;  // neither of the two least (both only fall)
    }
    if (md < 0.0) return;
    if (md < F.m1) {
      F.m2 = F.m1;
      F.j2 = F.j1;
      F.m1 = md;
      F.j1 = i;
    } else if (md < F.m2) {
      F.m2 = md;
      F.j2 = i;
    }
  };
  // two least over distinct spheres: a sphere that several lanes measured has
  // one distance
  auto v2_merge = [&]() {
    for (int o = 16; o > 0; o >>= 1) {
      const double a1 = __shfl_xor_sync(kLanes, F.m1, o), a2 = __shfl_xor_sync(kLanes, F.m2, o);
      const long long b1 = __shfl_xor_sync(kLanes, (long long)F.j1, o), b2 = __shfl_xor_sync(kLanes, (long long)F.j2, o);
      auto put = [&](double m, int64_t j) {
        if (j < 0 || j == F.j1 || j == F.j2) return;
        if (m < F.m1 || (m == F.m1 && j < F.j1)) {
          F.m2 = F.m1;
          F.j2 = F.j1;
          F.m1 = m;
          F.j1 = j;
        } else if (m < F.m2 || (m == F.m2 && j < F.j2)) {
          F.m2 = m;
          F.j2 = j;
        }
      };
      put(a1, b1);
      put(a2, b2);
    }
    return true;
  };
  warp_survivors(a, F, 0, R, stk, lane, v2_merge, v2_sphere);
  warp_survivors(a, F, 1, R, stk, lane, v2_merge, v2_sphere);
  v2_merge();
  Best B;
  B.cls = -1;
  B.sr = B.r = 0.0;
  B.key = 0;
  B.sign = 0;
  auto share = [&]() {
    warp_best(B);
    return true;
  };
  // survivors (intersection points)
  auto surv_cand = [&](uint32_t g) {
    double qx, qy, qz;
    tangent::survivor_pos(a, int64_t(g), qx, qy, qz);
    try_candidate(a, F, qx, qy, qz, int64_t(g) / a.KS, false, int64_t(g), B, []() { return true; });
  };
  warp_survivors(a, F, 0, R, stk, lane, share, surv_cand);
  warp_survivors(a, F, 1, R, stk, lane, share, [&](uint32_t g) {
    // a zero sample's survivors are in both lists: once is enough
    if (a.sph64[int64_t(g) / a.KS].w == 0.0) return;
    surv_cand(g);
  });
  share();
  // tangent points: spheres whose near or far tangent point may lie within R
  {
    const Tree& T = a.st;
    const float R32 = f_up(R);
    // balls that covered the latest tangent points (W.rec: centre in FP32,
    // radius - tol rounded down; W.rec_id: input index)
    int nrec = 0, at = 0;
    unsigned n_nodes = 0, n_items = 0;
    const float cover_lim = -a.tol32 + a.bc->elin, mg = lin_point_margin(*a.bc);
    // as in scored_one: is the tangent point surely inside one of the balls
    auto surely_covered = [&](const float4& S, float d32, float sr, int j) -> bool {
      const float ap = amax3(S.x, S.y, S.z), r = fabsf(sr);
      if (!(d32 > 1e-3f * (F.ax + ap + r))) return false;
      const float inv = 1.f / d32;
      const float tx = S.x + sr * ((F.x32 - S.x) * inv), ty = S.y + sr * ((F.y32 - S.y) * inv),
                  tz = S.z + sr * ((F.z32 - S.z) * inv);
      const float mt = 64.f * 5.9604645e-8f * (F.ax + ap + r) * (1.f + r * inv);
      const float at_ = amax3(tx, ty, tz);
      bool in = false;
      for (int u = 0; u < nrec; ++u) {
        if (W.rec_id[u] == j) continue;
        const float4 f = W.rec[u];
        const float dd = dist32(tx, ty, tz, f);
        in = in || dd + mt + err32(at_, f, dd, 0.f) < f.w;
      }
      return in;
    };
    // one tangent point per lane (sphere at sorted slot jj, input index j; jj < 0
    // for none): those that would beat the best so far are settled, the best
    // of them first, its coverage walked by the whole warp
    auto settle = [&](int jj, int j, int side) {
      bool open = jj >= 0;
      double p[3] = {0.0, 0.0, 0.0};
      Best K = B;
      auto rate = [&]() {  // the best value of this lane's point that beats B
        open = false;
        K = B;
        try_candidate(a, F, p[0], p[1], p[2], int64_t(j), true, kTanKey + 2 * int64_t(j) + side, K, [&]() {
          open = true;
          return true;
        });
      };
      if (open) {
        const D4 P = a.sph64[j];
        const double vx = __dsub_rn(F.x, P.x), vy = __dsub_rn(F.y, P.y), vz = __dsub_rn(F.z, P.z);
        const double dv = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)), __dmul_rn(vz, vz)));
        open = dv > 0.0;
        if (open) {
          const double sr = side == 0 ? fabs(P.w) : -fabs(P.w);
          p[0] = __dadd_rn(P.x, __dmul_rn(sr, __ddiv_rn(vx, dv)));
          p[1] = __dadd_rn(P.y, __dmul_rn(sr, __ddiv_rn(vy, dv)));
          p[2] = __dadd_rn(P.z, __dmul_rn(sr, __ddiv_rn(vz, dv)));
          open = !box_cull || ex_inbox(p[0], p[1], p[2]);
        }
        if (open) rate();
      }
      const bool in_range = fabs(p[0]) <= A && fabs(p[1]) <= A && fabs(p[2]) <= A;
      for (;;) {
        // 2 bits of class, the rest of the ranking value (which is >= 0)
        const unsigned key = open ? (unsigned(K.cls) << 30) | (__float_as_uint(float(K.sr)) >> 1) : 0u;
        const unsigned high = __reduce_max_sync(kLanes, key);
        const unsigned m = __ballot_sync(kLanes, open && key == high);
        if (!m) return;
        const int src = __ffs(m) - 1;
        int ball = -1;  // sorted slot or (out of range) input index of a ball that holds the point
        const bool ranged = __shfl_sync(kLanes, int(in_range), src) != 0;
        if (ranged) {
          const double qx = __shfl_sync(kLanes, p[0], src), qy = __shfl_sync(kLanes, p[1], src),
                       qz = __shfl_sync(kLanes, p[2], src);
          const float qxf = float(qx), qyf = float(qy), qzf = float(qz);
          const int cj = __shfl_sync(kLanes, jj, src);
          ball = warp_cover_walk(T, C, W.cstk, lane, qxf, qyf, qzf, cover_lim, n_nodes, n_items, [&](int c, float& v) {
            if (c == cj) return false;
            const float4 P = a.sph[c], Th = a.thr[c];
            const float dx = qxf - P.x, dy = qyf - P.y, dz = qzf - P.z;
            const float e2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            if (!(e2 <= Th.w)) return false;
            v = e2 - Th.z;
            return e2 < Th.z || ex_cov(qx, qy, qz, a.sph64[a.sid[c]], a.tol);
          });
          if (ball >= 0) ball = a.sid[ball];
        } else {
          if (lane == src) ball = tangent::covered_except(a, p[0], p[1], p[2], j, -1, -1);
          ball = __shfl_sync(kLanes, ball, src);
        }
        if (ball >= 0) {
          const D4 Q = a.sph64[ball];
          if (lane == src || (open && ball != j && ex_cov(p[0], p[1], p[2], Q, a.tol))) open = false;
          __syncwarp();
          if (lane == 0) {
            W.rec[at] = make_float4(float(Q.x), float(Q.y), float(Q.z), tangent::f_dn(__dsub_rn(fabs(Q.w), tol)));
            W.rec_id[at] = ball;
          }
          at = (at + 1) % tangent::kTanRecent;
          nrec = min(nrec + 1, tangent::kTanRecent);
          __syncwarp();
        } else {
          B.cls = __shfl_sync(kLanes, K.cls, src);
          B.sr = __shfl_sync(kLanes, K.sr, src);
          B.key = __shfl_sync(kLanes, (long long)K.key, src);
          B.sign = __shfl_sync(kLanes, K.sign, src);
          B.r = __shfl_sync(kLanes, K.r, src);
          if (lane == src) open = false;
          if (open) rate();
        }
      }
    };
    tangent::warp_lin_walk(
        T, C, stk, lane,
        [&](int64_t node) {
          if (!lin) {
            const float4 Bc = T.na[node], Fb = T.nf[node];
            const float dC = dist32(F.x32, F.y32, F.z32, Bc), dF = dist32(F.x32, F.y32, F.z32, Fb);
            return dC - err32(F.ax, Bc, dC, Bc.w) - Bc.w <= R32 || dF - err32(F.ax, Fb, dF, Fb.w) - Fb.w <= R32;
          }
          // the least d - r and d + r of the node's spheres, d = |x - p|
          const LinAt b = lin_at(lin_load(T, node), F.x32, F.y32, F.z32);
          return fminf(b.pos, b.neg) - R32 <= mg || b.far - R32 <= mg;
        },
        [&](int64_t jj) {
          bool near_ok = false, far_ok = false;
          int j = 0;
          if (jj >= 0) {
            const float4 S = a.sph[jj];
            if (S.w != 0.f) {
              const float d32 = dist32(F.x32, F.y32, F.z32, S), r32 = fabsf(S.w);
              const float er = err32(F.ax, S, d32, r32);
              near_ok = fabsf(d32 - r32) - er <= R32;
              far_ok = d32 + r32 - er <= R32;
              if (near_ok || far_ok) j = a.sid[jj];
              const int si = S.w > 0.f ? 1 : -1;
              // FP32 screen against the best so far and V1, as in scored_one
#pragma unroll
              for (int side = 0; side < 2; ++side) {
                bool& ok = side == 0 ? near_ok : far_ok;
                if (!ok) continue;
                const float rr = side == 0 ? fabsf(d32 - r32) : d32 + r32;
                const float r_hi = rr + er, r_lo = rr - er;
                const int dr = side == 1 ? 0 : (d32 - r32 > er ? 1 : (r32 - d32 > er ? -1 : 2));
                bool any = false;
                for (int sgi = 0; sgi < 2 && !any; ++sgi) {
                  const int sign = sgi == 0 ? 1 : -1;
                  if (F.sig != 0 && sign != F.sig) continue;
                  if (double(r_lo) - tol > F.ub[sgi]) continue;  // V1 fails for sure
                  if (B.cls < 0) {
                    any = true;
                    break;
                  }
                  int cls;
                  if (side == 1) cls = sign * si > 0 ? 3 : 0;
                  else if (dr == 2) cls = 3;  // undecided: the highest it could be
                  else cls = sign * si * dr < 0 ? 3 : 0;
                  const double sr_hi = double(r_hi) * (sign > 0 ? 1.0 : 2.0);
                  if (cls > B.cls || (cls == B.cls && sr_hi >= B.sr)) any = true;
                }
                if (!any || surely_covered(S, d32, side == 0 ? r32 : -r32, j)) ok = false;
              }
            }
          }
          if (__any_sync(kLanes, near_ok)) settle(near_ok ? int(jj) : -1, j, 0);
          if (__any_sync(kLanes, far_ok)) settle(far_ok ? int(jj) : -1, j, 1);
        });
  }
  if (lane != 0) return;
  if (B.cls < 0) {
    a.fl_out[q] = uint16_t(a.fl_out[q] | GFS_FLAG_SCORE_FALLBACK);
    return;
  }
  const bool tan = B.key >= kTanKey;
  const double v = B.sign > 0 ? B.r : -B.r;
  int flags = tan ? GFS_CODE_TANGENT : GFS_CODE_SURVIVOR;
  const int c = B.sign > 0 ? 0 : 1;
  if (SB.cov[c] && B.r < __dsub_rn(-SB.bestA[c], tol)) flags |= GFS_FLAG_LB_VIOL;
  if (a.s_out) a.s_out[q] = float(v);
  if (a.s64_out) a.s64_out[q] = v;
  a.arg_out[q] = tan ? B.key - kTanKey : B.key;
  a.fl_out[q] = uint16_t(flags);
}

}  // namespace scored
}  // namespace gfs
