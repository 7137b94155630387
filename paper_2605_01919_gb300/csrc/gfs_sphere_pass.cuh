// The query's pass over the spheres (device code; included by
// gfs_kernels.cu).
//
// For every point: containment per sign class, the least |x - p| - |s| per
// class, the least |x - p| + |s| over all spheres (best and second best, for
// the certification in the second kernel) and the sample at x, if any.
//
// One warp serves a packet of G neighbouring points (or one point, when the
// points are sparse: the launch says where the line lies) and tests nodes and spheres once per packet, one per
// lane: 4 stack entries give 32 children (or 32 spheres of 4 leaves) a round.
// A test compares the node's or sphere's bound at the packet centre c with a
// reference sphere w, found first by a beam descent: with rho the packet's
// radius, n and n_w the unit directions from the node's box centre (or the
// sphere's centre) and from p_w to c, every point x of the packet has
//   bound(x) - value_w(x) >= bound(c) - value_w(c)
//                            - min(|n - n_w| rho + rho^2 / (2 |c - p_w|), 2 rho)
// (|v + d| <= |v| + n.d + |d|^2 / (2 |v|); the bound is linear in x for fixed
// n), so what exceeds that by the FP32 margin elin is no minimum, no near tie
// and no containing ball of any point of the packet.  Only the spheres that
// pass are evaluated per point, from a queue in shared memory.
//
// What bounds it: instruction issue (72% of the slots on 253^3 points over a
// 64^3 union grid, 36% of the warps resident).  One node test costs the packet
// one lane instead of 32, and the reference makes the first test already sharp.
// The walk it replaces tested every node and sphere on every lane, with
// thresholds found on the way: 81.1 ms on that workload (104k warp
// instructions per 32 points) against 21.5 ms, 106 against 40 ms for 2.1M
// random points on a 96^3 torus grid, 2.86 ms against 0.028 ms for 257 random
// points on a 32^3 grid, where 32 scattered points shared one walk.
#pragma once

namespace gfs {

// (walk_take keeps within it; 4 popped and at most 32 pushed a round, the deepest
// level on top, it holds kFan + 28 entries a level)
constexpr int kSpStack = 448;
constexpr int kSpQueue = 64;
constexpr int kCand = 8;

struct SpWarp : LevelTable {
  uint32_t stk[kSpStack];
  float4 qp[kSpQueue];
  int qi[kSpQueue];
  int cand[kCand * 32]; // per lane: items awaiting their FP64 evaluation (second pass)
};

// reference sphere of one quantity at the packet centre
struct SpRef {
  float v, nx, ny, nz, quad;
};

__device__ __forceinline__ void top2_merge(Top2& t, int o) {
  const float b = __shfl_xor_sync(kFull, t.best, o), s = __shfl_xor_sync(kFull, t.sec, o);
  const int i = __shfl_xor_sync(kFull, t.idx, o);
  t.sec = fminf(fmaxf(t.best, b), fminf(t.sec, s));
  if (b < t.best) {
    t.best = b;
    t.idx = i;
  }
}

// Limits of a packet beyond which it is better served point by point: the
// radius (a jump of the Morton order), and the units a walk may spend per
// point (a round 6, an evaluation 1) in the sphere pass and in the others.
struct PkLimit {
  float rho;
  int spheres, rest;
};
__host__ __device__ inline PkLimit no_jump() { return PkLimit{INFINITY, 600, 100}; }

// Returns false (nothing stored) past the limits.
template <int G>
__device__ bool sphere_pass(const QueryArgs& a, int64_t first, SpWarp& S, int lane, const PkLimit& lim) {
  constexpr int kParts = 32 / G;
  const int part = lane / G;
  const int64_t slot = first + (lane & (G - 1));
  const bool active = slot < a.m;
  const BuildConsts bc = *a.bc;
  double x64 = 0.0, y64 = 0.0, z64 = 0.0;
  if (active) load_query(a, a.perm ? int64_t(a.perm[slot]) : slot, x64, y64, z64);
  const float x = float(x64), y = float(y64), z = float(z64);
  const bool live = active && fabs(x64) <= bc.A && fabs(y64) <= bc.A && fabs(z64) <= bc.A;
  const float grow = 1.f + 8.f * kU;
  const float ea2 = 2.f * bc.ea;
  const float negtol = -a.tol32 + ea2;
  unsigned rechecks = 0, n_nodes = 0, n_items = 0;
  bool cov0 = false, cov1 = false;
  Top2 A0, A1, F;
  top2_init(A0);
  top2_init(A1);
  top2_init(F);
  int sample = INT_MAX;
  if (__any_sync(kFull, live)) {
    const Tree& T = a.st;
    if (lane < kMaxLevels) S.lv[lane] = make_int2(int(T.offset[lane]), int(T.count[lane]));
    // packet centre and radius (over the FP64 points: 2 u A per rounding)
    float cx = live ? x : 0.f, cy = live ? y : 0.f, cz = live ? z : 0.f, cn = live ? 1.f : 0.f;
    for (int o = G / 2; o > 0; o >>= 1) {
      cx += __shfl_xor_sync(kFull, cx, o);
      cy += __shfl_xor_sync(kFull, cy, o);
      cz += __shfl_xor_sync(kFull, cz, o);
      cn += __shfl_xor_sync(kFull, cn, o);
    }
    cx /= cn;
    cy /= cn;
    cz /= cn;
    float rho = 0.f;
    if (live) {
      const float dx = x - cx, dy = y - cy, dz = z - cz;
      rho = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    }
    rho = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(rho))) * (1.f + 16.f * kU) + 4.f * kU * bc.A;
    if (G > 1 && rho > lim.rho * bc.A) return false;
    __syncwarp();
    const int top = T.nlevels - 1, grp = lane >> 3, sub = lane & 7;
    // ---- references: a beam of 4 nodes per quantity, down to 4 leaves ------
    float best[3] = {INFINITY, INFINITY, INFINITY};
    int at[3] = {-1, -1, -1};
#pragma unroll 1
    for (int crit = 0; crit < 3; ++crit) {
      int lev = top;
      int64_t node = lane;
      bool valid = lane < S.lv[top].y;
      for (;;) {
        float v = INFINITY;
        if (valid) {
          const int64_t nd = S.lv[lev].x + node;
          const float4 B = crit == 2 ? T.nf[nd] : T.na[nd];
          float w = B.w;
          if (crit < 2) {
            const float4 R = T.nb[nd];
            w = crit == 0 ? R.x : R.y;
          }
          v = sqrt_fast(ball_d2(cx, cy, cz, B)) - w;
        }
        unsigned key = v < INFINITY ? (ord_key(v) & ~31u) | unsigned(lane) : 0xffffffffu;
        unsigned mine = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const unsigned m = __reduce_min_sync(kFull, key);
          if (key == m) key = 0xffffffffu;
          if (grp == k) mine = m;
        }
        valid = mine != 0xffffffffu;
        node = __shfl_sync(kFull, (long long)node, int(mine & 31u)) * kFan + sub;
        if (lev == 0) break;
        --lev;
        valid = valid && node < S.lv[lev].y;
      }
      if (valid && node < a.n) {
        const float4 P = a.sph[node];
        const float d = sqrt_fast(ball_d2(cx, cy, cz, P)), r = fabsf(P.w);
        // the reference's own slack counts against it
        const float pen = fminf(__fdividef(0.5f * rho * rho, fmaxf(d, 1e-30f)), 2.f * rho);
        const int c = P.w > 0.f ? 0 : 1;
        if (P.w != 0.f && d - r + pen < best[c]) {
          if (c == 0) {
            best[0] = d - r + pen;
            at[0] = int(node);
          } else {
            best[1] = d - r + pen;
            at[1] = int(node);
          }
        }
        if (d + r + pen < best[2]) {
          best[2] = d + r + pen;
          at[2] = int(node);
        }
      }
    }
    SpRef R[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const unsigned key =
          __reduce_min_sync(kFull, best[k] < INFINITY ? (ord_key(best[k]) & ~31u) | unsigned(lane) : 0xffffffffu);
      const int j = __shfl_sync(kFull, at[k], int(key & 31u));
      R[k].v = INFINITY;  // no sphere of the class: inf - inf compares false, nothing passes
      R[k].nx = R[k].ny = R[k].nz = R[k].quad = 0.f;
      if (key == 0xffffffffu) continue;
      const float4 P = a.sph[j];
      const float r = fabsf(P.w);
      R[k].nx = cx - P.x;
      R[k].ny = cy - P.y;
      R[k].nz = cz - P.z;
      const float d = unit3(R[k].nx, R[k].ny, R[k].nz);
      R[k].v = k == 2 ? d + r : d - r;
      R[k].quad = d > 0.f ? 0.5f * rho * rho / d : INFINITY;
      if (!live) continue;
      // each point's threshold starts from the reference's value there
      const float dl = __fsqrt_rn(ball_d2(x, y, z, P));
      if (k == 0) A0.sec = dl - r + ea2;
      if (k == 1) A1.sec = dl - r + ea2;
      if (k == 2) F.sec = dl + r + ea2;
    }
    const float rho2 = 2.f * rho, margin = bc.elin;
    // may something with bound v at c and direction n matter for quantity k
    auto reach = [&](float v, float nx, float ny, float nz, const SpRef& r) {
      float sl = 0.f;
      if constexpr (G > 1) {
        const float ux = nx - r.nx, uy = ny - r.ny, uz = nz - r.nz;
        sl = fminf(fmaf(sqrt_fast(fmaf(ux, ux, fmaf(uy, uy, uz * uz))), rho, r.quad), rho2);
      } else {
        sl = rho2;  // the rounding of the point
      }
      return v - r.v <= sl + margin;
    };
    // ---- evaluation of the queued spheres at every point ---------------------
    // (the thresholds th0, th1, thf change only when a sphere enters a pair)
    float th0, th1, thf;
    auto thresholds = [&]() {
      th0 = top2_th(A0, ea2);
      th1 = top2_th(A1, ea2);
      if (!cov0) th0 = fmaxf(th0, negtol);
      if (!cov1) th1 = fmaxf(th1, negtol);
      thf = top2_th(F, ea2);
      if (!live) th0 = th1 = thf = -INFINITY;
    };
    thresholds();
    int qn = 0, spent = 0;
    auto flush = [&]() {
      __syncwarp();
      spent += qn / kParts;
      n_items += live ? unsigned((qn - part + kParts - 1) / kParts) : 0u;
#pragma unroll 1
      for (int t = part; t < qn; t += kParts) {
        const float4 P = S.qp[t];
        const float dx = x - P.x, dy = y - P.y, dz = z - P.z;
        const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const float r = fabsf(P.w);
        const float tc = r + (P.w > 0.f ? th0 : th1), tf = thf - r;
        const bool pc = (P.w != 0.f) & (tc > 0.f) & (d2 < tc * tc * grow);
        const bool pf = (tf > 0.f) & (d2 < tf * tf * grow);
        if (!(pc | pf | (d2 == 0.f))) continue;
        if (!live) continue;
        const int j = S.qi[t];
        if (d2 == 0.f) {
          const int o = a.sid[j];
          const D4 pj = a.sph64[o];
          if (pj.x == x64 && pj.y == y64 && pj.z == z64 && o < sample) sample = o;
        }
        const float d = __fsqrt_rn(d2);
        if (pc) {
          const bool neg = P.w < 0.f;
          const float v = d - r;
          if (neg) top2_push(A1, v, j);
          else top2_push(A0, v, j);
          if (!(neg ? cov1 : cov0) && v <= negtol) {
            const float4 Th = a.thr[j];
            bool cv = d2 < Th.z;
            if (!cv && d2 <= Th.w) {
              ++rechecks;
              cv = ex_cov(x64, y64, z64, a.sph64[a.sid[j]], a.tol);
            }
            if (neg) cov1 = cv;
            else cov0 = cv;
          }
        }
        if (pf) top2_push(F, d + r, j);
        thresholds();
      }
      __syncwarp();
      qn = 0;
    };
    // ---- the walk -----------------------------------------------------------
    int sp = S.lv[top].y;
    if (lane < sp) S.stk[lane] = pack_node(top, lane);
    __syncwarp();
    while (sp > 0) {
      if constexpr (G > 1) {
        if (spent > lim.spheres * G) return false;
        spent += 6;
      }
      const int take = walk_take(sp, kSpStack - kFan, 4);
      const uint32_t nd = grp < take ? S.stk[sp - 1 - grp] : 0xffffffffu;
      sp -= take;
      const int lev = node_level(nd);
      const int c = int(node_index(nd)) * kFan + sub;  // child or sphere
      bool pass_n = false, pass_i = false;
      float4 P = make_float4(0.f, 0.f, 0.f, 0.f);
      if (nd != 0xffffffffu) {
        if (lev == 0) {
          if (c < a.n) {
            ++n_items;
            P = a.sph[c];
            float nx = cx - P.x, ny = cy - P.y, nz = cz - P.z;
            const float d = unit3(nx, ny, nz);
            const float r = fabsf(P.w);
            // (a sample at a point of the packet; its class's value; the far bound)
            const SpRef C = P.w > 0.f ? R[0] : R[1];
            pass_i = (d <= rho + margin) | ((P.w != 0.f) & reach(d - r, nx, ny, nz, C)) |
                     reach(d + r, nx, ny, nz, R[2]);
          }
        } else {
          const int2 L = S.lv[lev - 1];
          if (c < L.y) {
            ++n_nodes;
            const Lin q = lin_load(T, L.x + c);
            const float lim = rho + margin;
            const bool at = (fabsf(cx - q.cx) <= q.hx + lim) & (fabsf(cy - q.cy) <= q.hy + lim) &
                            (fabsf(cz - q.cz) <= q.hz + lim);
            const LinAt b = lin_at(q, cx, cy, cz);
            pass_n = at | reach(b.pos, b.nx, b.ny, b.nz, R[0]) | reach(b.neg, b.nx, b.ny, b.nz, R[1]) |
                     reach(b.far, b.nx, b.ny, b.nz, R[2]);
          }
        }
      }
      const unsigned bn = __ballot_sync(kFull, pass_n), bi = __ballot_sync(kFull, pass_i);
      // children of the deepest popped entry (lowest level) end up on top
      if (pass_n) S.stk[sp + __popc(bn >> lane >> 1)] = pack_node(lev - 1, c);
      sp += __popc(bn);
      if (pass_i) {
        const int k = qn + __popc(bi & ((1u << lane) - 1u));
        S.qp[k] = P;
        S.qi[k] = c;
      }
      qn += __popc(bi);
      if (qn > kSpQueue - 32) flush();
      else __syncwarp();
    }
    if (qn > 0) flush();
    // the parts of a point's spheres back together
    for (int o = G; o < 32; o <<= 1) {
      cov0 = __shfl_xor_sync(kFull, int(cov0), o) || cov0;
      cov1 = __shfl_xor_sync(kFull, int(cov1), o) || cov1;
      sample = min(sample, __shfl_xor_sync(kFull, sample, o));
      top2_merge(A0, o);
      top2_merge(A1, o);
      top2_merge(F, o);
    }
  }
  if (active && part == 0) store_qstate(a.state, slot, cov0, cov1, sample, A0, A1, F);
  warp_count(&a.cnt->query_rechecks, rechecks);
  warp_count(&a.cnt->q_sphere_ntests, n_nodes);
  warp_count(&a.cnt->q_sphere_items, n_items);
  return true;
}

// Points per packet; where packets begin is said at the launch.
constexpr int kPacket = 16;

// A packet of G, point by point where it has to be.
template <int G>
__device__ void sphere_pass_any(const QueryArgs& a, int64_t first, SpWarp& S, int lane) {
  if constexpr (G > 1)
    if (sphere_pass<G>(a, first, S, lane, no_jump())) return;
#pragma unroll 1
  for (int k = 0; k < G && first + k < a.m; ++k) {
    __syncwarp();
    sphere_pass<1>(a, first + k, S, lane, no_jump());
  }
}

}  // namespace gfs
