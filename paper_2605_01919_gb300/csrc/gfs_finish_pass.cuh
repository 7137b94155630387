// The query's passes after the sphere pass (device code; included by
// gfs_kernels.cu): the nearest survivor of each point's class (near_pass),
// then the FP64 winners, the value, the flags and the outputs (decide_pass).
//
// As in the sphere pass one warp serves a packet of G neighbouring points (or
// one point) and tests nodes and items once per packet, 32 a round, against
// the packet's thresholds: with n_w a reference direction, c and rho the
// packet's centre and radius and T(x) the points' thresholds, a bound B with
// direction n at c can matter to some point only if
//   B - |n - n_w| rho <= max_x (T(x) - n_w . (x - c))  and  B - rho <= max_x T(x)
// (within the FP32 margins).  The thresholds start from the best of four
// leaves found by a beam descent and follow the best found so far.  Near ties
// (41% of the points of the 253^3 upsampling of a 64^3 union grid: the
// samples above a box face share their foot points) are settled in FP64 by a
// second walk of the same kind over the error band, whose items each lane
// gathers before all lanes evaluate theirs together.
//
// What bounds it: instruction issue in the walks, the FP64 units in the
// decisions (70% busy on the union grid).  Both together, against a walk per
// point with box and ball bounds: 22.3 against 48.6 ms (16.2M points, 64^3
// union), 10.8 against 55.4 (2.1M random points, 96^3 torus), 0.59 against 8.4
// (32k random points, 64^3), 0.055 against 1.85 (257 points, 32^3).
#pragma once

namespace gfs {

struct Pk {
  float cx, cy, cz, rho;
};

// thresholds of a packet about a reference direction
struct PkRef {
  float nx, ny, nz, tau, tm;
};

__device__ __forceinline__ float warp_max(float v) { return ord_val(__reduce_max_sync(kFull, ord_key(v))); }

// centre and radius of the points with use set (some lane must have it; the
// parts of a packet repeat the same points)
template <int G>
__device__ __forceinline__ Pk packet_of(bool use, float x, float y, float z, float A) {
  Pk k;
  float cn = use ? 1.f : 0.f;
  k.cx = use ? x : 0.f;
  k.cy = use ? y : 0.f;
  k.cz = use ? z : 0.f;
  for (int o = G / 2; o > 0; o >>= 1) {
    k.cx += __shfl_xor_sync(kFull, k.cx, o);
    k.cy += __shfl_xor_sync(kFull, k.cy, o);
    k.cz += __shfl_xor_sync(kFull, k.cz, o);
    cn += __shfl_xor_sync(kFull, cn, o);
  }
  k.cx /= cn;
  k.cy /= cn;
  k.cz /= cn;
  float d = 0.f;
  if (use) {
    const float dx = x - k.cx, dy = y - k.cy, dz = z - k.cz;
    d = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
  }
  k.rho = warp_max(d) * (1.f + 16.f * kU) + 4.f * kU * A;
  return k;
}

// reference direction towards P, thresholds T of the points with use set
__device__ __forceinline__ void ref_dir(PkRef& r, const Pk& k, const float4& P) {
  r.nx = k.cx - P.x;
  r.ny = k.cy - P.y;
  r.nz = k.cz - P.z;
  unit3(r.nx, r.ny, r.nz);
}
__device__ __forceinline__ void ref_thr(PkRef& r, const Pk& k, bool use, float T, float x, float y, float z) {
  r.tm = warp_max(use ? T : -INFINITY);
  r.tau = warp_max(use ? T - fmaf(r.nx, x - k.cx, fmaf(r.ny, y - k.cy, r.nz * (z - k.cz))) : -INFINITY);
}
__device__ __forceinline__ bool pk_reach(const PkRef& r, float rho, float margin, float v, float nx, float ny, float nz) {
  const float ux = nx - r.nx, uy = ny - r.ny, uz = nz - r.nz;
  const float sl = sqrt_fast(fmaf(ux, ux, fmaf(uy, uy, uz * uz)));
  return (fmaf(-rho, sl, v) <= r.tau + margin) & (v - rho <= r.tm + margin);
}

// distance from the packet's centre to a node box, and its direction
__device__ __forceinline__ float box_dir(const Pk& k, const float4& lo, const float4& hi, float& nx, float& ny,
                                         float& nz) {
  nx = k.cx - fminf(fmaxf(k.cx, lo.x), hi.x);
  ny = k.cy - fminf(fmaxf(k.cy, lo.y), hi.y);
  nz = k.cz - fminf(fmaxf(k.cz, lo.z), hi.z);
  return unit3(nx, ny, nz);
}

// The walk: node(index) and item(index, P) say whether a child or an item may
// matter (P: its record, queued); flush(n) evaluates the n queued items.
// Returns false when it has spent more than budget units (a round 6, an
// evaluation 1; budget < 0: no limit), with the queue dropped.
template <int G, class Node, class Item, class Flush>
__device__ bool packet_walk(const Tree& T, SpWarp& S, int lane, int budget, Node node, Item item, Flush flush) {
  constexpr int kParts = 32 / G;
  const int top = T.nlevels - 1, grp = lane >> 3, sub = lane & 7;
  int sp = S.lv[top].y, qn = 0, spent = 0;
  if (lane < sp) S.stk[lane] = pack_node(top, lane);
  __syncwarp();
  while (sp > 0) {
    if (budget >= 0 && spent > budget) return false;
    spent += 6;
    const int take = walk_take(sp, kSpStack - kFan, 4);
    const uint32_t nd = grp < take ? S.stk[sp - 1 - grp] : 0xffffffffu;
    sp -= take;
    const int lev = node_level(nd);
    const int c = int(node_index(nd)) * kFan + sub;
    bool pass_n = false, pass_i = false;
    float4 P = make_float4(0.f, 0.f, 0.f, 0.f);
    if (nd != 0xffffffffu) {
      if (lev == 0) {
        if (c < T.nitems) pass_i = item(c, P);
      } else {
        const int2 L = S.lv[lev - 1];
        if (c < L.y) pass_n = node(int64_t(L.x) + c);
      }
    }
    const unsigned bn = __ballot_sync(kFull, pass_n), bi = __ballot_sync(kFull, pass_i);
    if (pass_n) S.stk[sp + __popc(bn >> lane >> 1)] = pack_node(lev - 1, c);
    sp += __popc(bn);
    if (pass_i) {
      const int k = qn + __popc(bi & ((1u << lane) - 1u));
      S.qp[k] = P;
      S.qi[k] = c;
    }
    qn += __popc(bi);
    __syncwarp();
    if (qn > kSpQueue - 32) {
      spent += qn / kParts;
      flush(qn);
      __syncwarp();
      qn = 0;
    }
  }
  if (qn > 0) flush(qn);
  __syncwarp();
  return true;
}

// Exact FP64 minimum over the spheres whose FP32 value lies at or below the
// point's threshold thr, and its input index (ties to the lowest), for the
// points with band set (idx: the sorted slot of the FP32 minimum).  Returns
// false as packet_walk does, or when the points lie far apart.
// mode 0: |x-p| - r over sign class cls; mode 1: |x-p| + r over all spheres.
template <int G>
__device__ bool sphere_band(const QueryArgs& a, const BuildConsts& bc, SpWarp& S, int lane, bool band, int idx,
                            double x64, double y64, double z64, float x, float y, float z, int mode, int cls,
                            float thr, const PkLimit& lim, double& best, int& arg) {
  constexpr int kParts = 32 / G;
  const int part = lane / G;
  best = INFINITY;
  arg = INT_MAX;
  const unsigned bm = __ballot_sync(kFull, band);
  if (!bm) return true;
  const Pk k = packet_of<G>(band, x, y, z, bc.A);
  if (G > 1 && k.rho > lim.rho * bc.A) return false;
  const Tree& T = a.st;
  // the point's spheres within the band, evaluated in FP64 by all lanes
  // together: done where found they would run one lane at a time on an FP64
  // pipe that takes 16 cycles a warp instruction
  int nc = 0;
  auto drain = [&]() {
    for (int t = 0; __any_sync(kFull, t < nc); ++t) {
      if (t >= nc) continue;
      const int o = a.sid[S.cand[32 * t + lane]];
      const D4 pj = a.sph64[o];
      const double dl = __dsqrt_rn(ex_d2(x64, y64, z64, pj.x, pj.y, pj.z));
      const double v = mode == 0 ? __dsub_rn(dl, fabs(pj.w)) : __dadd_rn(dl, fabs(pj.w));
      if (v < best || (v == best && o < arg)) {
        best = v;
        arg = o;
      }
    }
    nc = 0;
  };
  load_levels(T, S, lane);
  PkRef r;
  ref_dir(r, k, a.sph[__shfl_sync(kFull, idx, __ffs(bm) - 1)]);
  ref_thr(r, k, band, thr, x, y, z);
  const bool done = packet_walk<G>(
      T, S, lane, G > 1 ? lim.rest * G : -1,
      [&](int64_t nd) {
        const LinAt b = lin_at(lin_load(T, nd), k.cx, k.cy, k.cz);
        return pk_reach(r, k.rho, bc.elin, mode == 1 ? b.far : (cls == 0 ? b.pos : b.neg), b.nx, b.ny, b.nz);
      },
      [&](int c, float4& P) {
        P = a.sph[c];
        if (mode == 0 && (P.w == 0.f || int(P.w < 0.f) != cls)) return false;
        float nx = k.cx - P.x, ny = k.cy - P.y, nz = k.cz - P.z;
        const float d = unit3(nx, ny, nz);
        return pk_reach(r, k.rho, bc.elin, mode == 1 ? d + fabsf(P.w) : d - fabsf(P.w), nx, ny, nz);
      },
      [&](int qn) {
        for (int b = 0; b < qn; b += kParts) {
          const int t = b + part;
          if (band && t < qn) {
            const float4 P = S.qp[t];
            const float dx = x - P.x, dy = y - P.y, dz = z - P.z;
            const float d = __fsqrt_rn(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
            if ((mode == 1 ? d + fabsf(P.w) : d - fabsf(P.w)) <= thr) S.cand[32 * nc++ + lane] = S.qi[t];
          }
          if (__any_sync(kFull, nc == kCand)) drain();
        }
      });
  if (!done) return false;
  drain();
  for (int o = G; o < 32; o <<= 1) {
    const double b = __shfl_xor_sync(kFull, best, o);
    const int i = __shfl_xor_sync(kFull, arg, o);
    if (b < best || (b == best && i < arg)) {
      best = b;
      arg = i;
    }
  }
  return true;
}

// one point's nearest survivor so far: least and second least squared FP32
// distance, sorted slot of the least
struct Near {
  float bd, sd;
  int j;
};

// Nearest survivor of class cls for the points with use set.  false: budget
// spent (nothing final).
template <int G>
__device__ bool near_survivor(const QueryArgs& a, const BuildConsts& bc, SpWarp& S, int lane, bool use, int cls,
                              float x, float y, float z, int budget, Near& N, unsigned& n_nodes, unsigned& n_items) {
  constexpr int kParts = 32 / G;
  const int part = lane / G, grp = lane >> 3, sub = lane & 7;
  const Tree& T = a.vt[cls];
  const float4* items = a.surv[cls];
  load_levels(T, S, lane);
  const Pk k = packet_of<G>(use, x, y, z, bc.A);
  auto band2 = [&](float D) { return 2.f * (bc.ed_lin * __fsqrt_rn(D) + bc.ed_quad * D + 1e-30f); };
  // reference: a beam of 4 nodes by box distance, down to 4 leaves
  int lev = T.nlevels - 1;
  int64_t node = lane;
  bool valid = lane < S.lv[lev].y;
  for (;;) {
    float v = INFINITY;
    if (valid) v = box_d2(k.cx, k.cy, k.cz, T.lo[S.lv[lev].x + node], T.hi[S.lv[lev].x + node]);
    unsigned key = v < INFINITY ? (__float_as_uint(v) & ~31u) | unsigned(lane) : 0xffffffffu;
    unsigned mine = 0xffffffffu;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned m = __reduce_min_sync(kFull, key);
      if (key == m) key = 0xffffffffu;
      if (grp == q) mine = m;
    }
    valid = mine != 0xffffffffu;
    node = __shfl_sync(kFull, (long long)node, int(mine & 31u)) * kFan + sub;
    if (lev == 0) break;
    --lev;
    valid = valid && node < S.lv[lev].y;
  }
  valid = valid && node < T.nitems;
  unsigned key = 0xffffffffu;
  if (valid) {
    const float d = sqrt_fast(ball_d2(k.cx, k.cy, k.cz, items[node]));
    const float pen = fminf(__fdividef(0.5f * k.rho * k.rho, fmaxf(d, 1e-30f)), 2.f * k.rho);
    key = (__float_as_uint(d + pen) & ~31u) | unsigned(lane);
  }
  key = __reduce_min_sync(kFull, key);
  const float4 P0 = items[__shfl_sync(kFull, (long long)node, int(key & 31u))];
  N.bd = INFINITY;
  N.j = -1;
  N.sd = -1.f;
  float T0 = 0.f;
  if (use) {
    const float d2 = ball_d2(x, y, z, P0);
    N.sd = d2 + band2(d2);  // starting threshold: the reference and its error band
    T0 = sqrtf(d2);
  }
  float th = N.sd;
  PkRef r;
  ref_dir(r, k, P0);
  ref_thr(r, k, use, T0, x, y, z);
  const float margin = bc.elin + 8.f * bc.eq;
  const bool done = packet_walk<G>(
      T, S, lane, budget,
      [&](int64_t nd) {
        ++n_nodes;
        float nx, ny, nz;
        const float d = box_dir(k, T.lo[nd], T.hi[nd], nx, ny, nz);
        return pk_reach(r, k.rho, margin, d, nx, ny, nz);
      },
      [&](int c, float4& P) {
        ++n_items;
        P = items[c];
        float nx = k.cx - P.x, ny = k.cy - P.y, nz = k.cz - P.z;
        const float d = unit3(nx, ny, nz);
        return pk_reach(r, k.rho, margin, d, nx, ny, nz);
      },
      [&](int qn) {
        n_items += use ? unsigned((qn - part + kParts - 1) / kParts) : 0u;
        bool moved = false;
#pragma unroll 1
        for (int t = part; t < qn; t += kParts) {
          const float4 P = S.qp[t];
          const float dx = x - P.x, dy = y - P.y, dz = z - P.z;
          const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          if (!(d2 < th)) continue;
          if (d2 < N.bd) {
            N.sd = fminf(N.sd, N.bd);
            N.bd = d2;
            N.j = S.qi[t];
            moved = true;
          } else {
            N.sd = d2;
          }
          th = fminf(N.sd, N.bd + band2(N.bd));
        }
        // the packet's thresholds and direction from the best so far
        if (__any_sync(kFull, moved)) {
          float b = N.bd;
          for (int o = G; o < 32; o <<= 1) b = fminf(b, __shfl_xor_sync(kFull, b, o));
          T0 = fminf(T0, sqrtf(b));
          const unsigned kb = N.j >= 0 ? (__float_as_uint(N.bd) & ~31u) | unsigned(lane) : 0xffffffffu;
          const int src = int(__reduce_min_sync(kFull, kb) & 31u);
          ref_dir(r, k, items[__shfl_sync(kFull, N.j, src)]);
          ref_thr(r, k, use, T0, x, y, z);
        }
      });
  if (!done) return false;
  for (int o = G; o < 32; o <<= 1) {
    const float b = __shfl_xor_sync(kFull, N.bd, o), s = __shfl_xor_sync(kFull, N.sd, o);
    const int i = __shfl_xor_sync(kFull, N.j, o);
    N.sd = fminf(fmaxf(N.bd, b), fminf(N.sd, s));
    if (b < N.bd) {
      N.bd = b;
      N.j = i;
    }
  }
  return true;
}

// Exact nearest survivor of class cls among those whose FP32 squared distance
// is at most thr, for the points with band set (j: the FP32 nearest's slot).
template <int G>
__device__ bool surv_band(const QueryArgs& a, const BuildConsts& bc, SpWarp& S, int lane, bool band, int cls, int j,
                          double x64, double y64, double z64, float x, float y, float z, float thr, const PkLimit& lim,
                          double& best, uint32_t& gbest) {
  constexpr int kParts = 32 / G;
  const int part = lane / G;
  best = INFINITY;
  gbest = 0xffffffffu;
  const unsigned bm = __ballot_sync(kFull, band);
  if (!bm) return true;
  const Pk k = packet_of<G>(band, x, y, z, bc.A);
  if (G > 1 && k.rho > lim.rho * bc.A) return false;
  const Tree& T = a.vt[cls];
  const float4* items = a.surv[cls];
  int nc = 0;  // as in sphere_band
  auto drain = [&]() {
    for (int t = 0; __any_sync(kFull, t < nc); ++t) {
      if (t >= nc) continue;
      const uint32_t g = uint32_t(S.cand[32 * t + lane]);
      double qx, qy, qz;
      surv_pos64(a, g, qx, qy, qz);
      const double e2 = ex_d2(x64, y64, z64, qx, qy, qz);
      if (e2 < best || (e2 == best && g < gbest)) {
        best = e2;
        gbest = g;
      }
    }
    nc = 0;
  };
  load_levels(T, S, lane);
  PkRef r;
  ref_dir(r, k, items[__shfl_sync(kFull, j, __ffs(bm) - 1)]);
  ref_thr(r, k, band, band ? sqrtf(thr) : 0.f, x, y, z);
  const float margin = bc.elin + 8.f * bc.eq;
  const bool done = packet_walk<G>(
      T, S, lane, G > 1 ? lim.rest * G : -1,
      [&](int64_t nd) {
        float nx, ny, nz;
        const float d = box_dir(k, T.lo[nd], T.hi[nd], nx, ny, nz);
        return pk_reach(r, k.rho, margin, d, nx, ny, nz);
      },
      [&](int c, float4& P) {
        P = items[c];
        float nx = k.cx - P.x, ny = k.cy - P.y, nz = k.cz - P.z;
        const float d = unit3(nx, ny, nz);
        return pk_reach(r, k.rho, margin, d, nx, ny, nz);
      },
      [&](int qn) {
        for (int b = 0; b < qn; b += kParts) {
          const int t = b + part;
          if (band && t < qn) {
            const float4 P = S.qp[t];
            const float dx = x - P.x, dy = y - P.y, dz = z - P.z;
            if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= thr) S.cand[32 * nc++ + lane] = int(__float_as_uint(P.w));
          }
          if (__any_sync(kFull, nc == kCand)) drain();
        }
      });
  if (!done) return false;
  drain();
  for (int o = G; o < 32; o <<= 1) {
    const double b = __shfl_xor_sync(kFull, best, o);
    const uint32_t i = __shfl_xor_sync(kFull, gbest, o);
    if (b < best || (b == best && i < gbest)) {
      best = b;
      gbest = i;
    }
  }
  return true;
}

// The nearest survivors of one packet, from the sphere pass's state into the
// state's fourth word.  false: nothing written, the packet's points go one by
// one (as in sphere_pass).
template <int G>
__device__ bool near_pass(const QueryArgs& a, int64_t first, SpWarp& S, int lane, const PkLimit& lim) {
  const int64_t slot = first + (lane & (G - 1));
  const bool active = slot < a.m;
  const int64_t q = active ? int64_t(a.perm ? a.perm[slot] : uint32_t(slot)) : 0;
  const BuildConsts bc = *a.bc;
  double x64 = 0.0, y64 = 0.0, z64 = 0.0;
  if (active) load_query(a, q, x64, y64, z64);
  const float x = float(x64), y = float(y64), z = float(z64);
  unsigned n_nodes = 0, n_items = 0;
  const bool live = active && fabs(x64) <= bc.A && fabs(y64) <= bc.A && fabs(z64) <= bc.A;
  bool cov0 = false, cov1 = false;
  int sample = INT_MAX;
  if (active) {
    const uint4 u = a.state[kStateWords * slot + 2];
    sample = int(u.y);
    cov0 = (u.z & 1u) != 0;
    cov1 = (u.z & 2u) != 0;
  }
  const bool open = live && sample == INT_MAX && cov0 != cov1;
  const int cs = cov0 ? 0 : 1;
  if constexpr (G > 1) {
    if (__any_sync(kFull, open) && packet_of<G>(open, x, y, z, bc.A).rho > lim.rho * bc.A) return false;
  }
  Near N;
  N.bd = N.sd = INFINITY;
  N.j = -1;
#pragma unroll 1
  for (int cl = 0; cl < 2; ++cl) {
    const bool mine = open && cs == cl;
    if (!__any_sync(kFull, mine) || a.vt[cl].nlevels == 0) continue;
    Near M;
    if (!near_survivor<G>(a, bc, S, lane, mine, cl, x, y, z, G > 1 ? lim.rest * G : -1, M, n_nodes, n_items))
      return false;
    if (mine) N = M;
  }
  if (active && lane < G)
    a.state[kStateWords * slot + 3] = make_uint4(__float_as_uint(N.bd), __float_as_uint(N.sd), unsigned(N.j), 0u);
  warp_count(&a.cnt->q_surv_ntests, n_nodes);
  warp_count(&a.cnt->q_surv_items, n_items);
  return true;
}

// The decisions of one packet (or one point), from the state of the two
// passes before it: FP64 winners, value, flags, outputs.  Points outside the
// coordinate range of the FP32 error model go to the FP64 kernel through
// a.defer, or (kInlineExact) are evaluated in place.  false: nothing written,
// the packet's points go one by one.
template <int G, bool kInlineExact>
__device__ bool decide_pass(const QueryArgs& a, int64_t first, SpWarp& S, int lane, const PkLimit& lim) {
  const int part = lane / G;
  const int64_t slot = first + (lane & (G - 1));
  const bool active = slot < a.m;
  const int64_t q = active ? int64_t(a.perm ? a.perm[slot] : uint32_t(slot)) : 0;
  const BuildConsts bc = *a.bc;
  double x64 = 0.0, y64 = 0.0, z64 = 0.0;
  if (active) load_query(a, q, x64, y64, z64);
  const float x = float(x64), y = float(y64), z = float(z64);
  unsigned n_band = 0;
  const bool live = active && fabs(x64) <= bc.A && fabs(y64) <= bc.A && fabs(z64) <= bc.A;
  const bool defer = active && !live;
  const float ea2 = 2.f * bc.ea;
  // per-class state as scalars (indexing a register array would push it to
  // local memory)
  bool cov0 = false, cov1 = false;
  Top2 A0, A1, F;
  top2_init(A0);
  top2_init(A1);
  top2_init(F);
  int sample = INT_MAX;
  Near N;
  N.bd = N.sd = INFINITY;
  N.j = -1;
  if (active) {
    load_qstate(a.state, slot, cov0, cov1, sample, A0, A1, F);
    const uint4 u = a.state[kStateWords * slot + 3];
    N.bd = __uint_as_float(u.x);
    N.sd = __uint_as_float(u.y);
    N.j = int(u.z);
  }
  int code = -1;
  double value = 0.0;
  int64_t arg = -1;
  int flags = 0;
  if (live) {
    if (sample != INT_MAX) {
      code = GFS_CODE_SAMPLE;
      value = a.sph64[sample].w;
      arg = sample;
    } else if (cov0 && cov1) {
      code = GFS_CODE_INVALID;
      value = __longlong_as_double(0x7ff8000000000000LL);
    } else if (!cov0 && !cov1) {
      code = GFS_CODE_OUTSIDE;
    }
    if (code >= 0) flags = code;
  }
  const bool open = live && code < 0;
  const int cs = cov0 ? 0 : 1, co = 1 - cs;
  const Top2 As = cs == 0 ? A0 : A1;   // x's own class
  const Top2 Ao = cs == 0 ? A1 : A0;   // the opposite class
  const bool have_s = open && N.j >= 0, have_u = open && Ao.idx >= 0;
  // exact nearest survivor: direct when no other survivor lies in the error
  // band, else an FP64 pass over the band
  double ds = INFINITY;
  uint32_t gbest = 0xffffffffu;
  const float sthr = N.bd + 2.f * (bc.ed_lin * __fsqrt_rn(N.bd) + bc.ed_quad * N.bd + 1e-30f);
  const bool sband = have_s && !(N.sd >= sthr);
  if (have_s && !sband) {
    gbest = __float_as_uint(a.surv[cs][N.j].w);
    double qx, qy, qz;
    surv_pos64(a, gbest, qx, qy, qz);
    ds = __dsqrt_rn(ex_d2(x64, y64, z64, qx, qy, qz));
  }
#pragma unroll 1
  for (int cl = 0; cl < 2; ++cl) {
    uint32_t g2;
    const bool mine = sband && cs == cl;
    double e2;
    if (!surv_band<G>(a, bc, S, lane, mine, cl, N.j, x64, y64, z64, x, y, z, mine ? sthr : -1.f, lim, e2, g2))
      return false;
    if (mine) {
      ++n_band;
      ds = __dsqrt_rn(e2);
      gbest = g2;
    }
  }
  // exact nearest opposite tangent point
  double ub = INFINITY;
  int uj = -1;
  const bool uband = have_u && !(Ao.sec >= Ao.best + ea2);
  if (have_u && !uband) {
    uj = a.sid[Ao.idx];
    const D4 pj = a.sph64[uj];
    ub = __dsub_rn(__dsqrt_rn(ex_d2(x64, y64, z64, pj.x, pj.y, pj.z)), fabs(pj.w));
  }
#pragma unroll 1
  for (int cl = 0; cl < 2; ++cl) {
    int j2;
    const bool mine = uband && co == cl;
    double v;
    if (!sphere_band<G>(a, bc, S, lane, mine, Ao.idx, x64, y64, z64, x, y, z, 0, cl,
                        mine ? Ao.best + ea2 : -1.f, lim, v, j2))
      return false;
    if (mine) {
      ++n_band;
      ub = v;
      uj = j2;
    }
  }
  // value and the result code
  double m = 0.0;
  bool need_lb = false;
  if (open) {
    if (have_s && (!a.clamp_opp || ds <= ub)) {
      code = GFS_CODE_SURVIVOR;
      m = ds;
      arg = int64_t(gbest);
    } else if (a.clamp_opp && have_u) {
      code = GFS_CODE_OPPOSITE;
      m = ub;
      arg = uj;
    } else {
      code = GFS_CODE_LOWER;
      need_lb = true;
    }
  }
  const double E = double(bc.ea) * 1.01 + 1e-15;
  const double lbt = -double(As.best) - a.tol;
  const double ft = double(F.best) + a.tol;
  if (open && code != GFS_CODE_LOWER) {
    const double mm = m < 0.0 ? 0.0 : m;
    need_lb = !(mm < lbt - E) && !(mm > lbt + E);
  }
  // exact lower bound LB (max over the point's class of r - |x-p|) if needed
  double lb = 0.0;
  int lj = -1;
  const bool lband = need_lb && !(As.sec >= As.best + ea2);
  if (need_lb && !lband) {
    lj = a.sid[As.idx];
    const D4 pl = a.sph64[lj];
    lb = __dsub_rn(fabs(pl.w), __dsqrt_rn(ex_d2(x64, y64, z64, pl.x, pl.y, pl.z)));
  }
#pragma unroll 1
  for (int cl = 0; cl < 2; ++cl) {
    int j2;
    const bool mine = lband && cs == cl;
    double v;
    if (!sphere_band<G>(a, bc, S, lane, mine, As.idx, x64, y64, z64, x, y, z, 0, cl,
                        mine ? As.best + ea2 : -1.f, lim, v, j2))
      return false;
    if (mine) {
      ++n_band;
      lb = -v;
      lj = j2;
    }
  }
  if (open && code == GFS_CODE_LOWER) {
    m = lb;
    arg = lj;
  }
  if (m < 0.0) m = 0.0;
  // exact far bound if the FP32 margin does not decide FAR_VIOL
  const bool need_far = open && !(m > ft + E) && !(m < ft - E);
  const bool fband = need_far && !(F.sec >= F.best + ea2);
  double far = INFINITY;
  if (need_far && !fband) {
    const D4 pf = a.sph64[a.sid[F.idx]];
    far = __dadd_rn(__dsqrt_rn(ex_d2(x64, y64, z64, pf.x, pf.y, pf.z)), fabs(pf.w));
  }
  {
    int j2;
    double v;
    if (!sphere_band<G>(a, bc, S, lane, fband, F.idx, x64, y64, z64, x, y, z, 1, 0,
                        fband ? F.best + ea2 : -1.f, lim, v, j2))
      return false;
    if (fband) {
      ++n_band;
      far = v;
    }
  }
  if (open) {
    flags = code;
    if (m < lbt - E) flags |= GFS_FLAG_LB_VIOL;
    else if (need_lb && m < __dsub_rn(lb, a.tol)) flags |= GFS_FLAG_LB_VIOL;
    if (m > ft + E) flags |= GFS_FLAG_FAR_VIOL;
    else if (need_far && m > __dadd_rn(far, a.tol)) flags |= GFS_FLAG_FAR_VIOL;
    if (have_u && ub < __dsub_rn(m, a.tol)) flags |= GFS_FLAG_OPP_VIOL;
    value = cs == 0 ? m : -m;
  }
  warp_count(&a.cnt->q_band_passes, part == 0 ? n_band : 0u);
  if (part == 0) {
    if (live) {
      write_result(a, q, value, arg, flags);
    } else if (defer) {
      // outside the coordinate range the error bounds assume: FP64 path
      const unsigned int s2 = atomicAdd(&a.cnt->ndefer, 1u);
      if constexpr (kInlineExact) {
        query_exact_one(a, q);
      } else {
        if (s2 < a.defer_cap) a.defer[s2] = uint32_t(q);
      }
    }
  }
  return true;
}

// A packet of G, point by point where it has to be.
template <int G>
__device__ void decide_pass_any(const QueryArgs& a, int64_t first, SpWarp& S, int lane) {
  if (decide_pass<G, true>(a, first, S, lane, no_jump())) return;
#pragma unroll 1
  for (int k = 0; k < G && first + k < a.m; ++k) {
    __syncwarp();
    decide_pass<1, true>(a, first + k, S, lane, no_jump());
  }
}

template <int G>
__device__ void near_pass_any(const QueryArgs& a, int64_t first, SpWarp& S, int lane) {
  if (near_pass<G>(a, first, S, lane, no_jump())) return;
#pragma unroll 1
  for (int k = 0; k < G && first + k < a.m; ++k) {
    __syncwarp();
    near_pass<1>(a, first + k, S, lane, no_jump());
  }
}

}  // namespace gfs
