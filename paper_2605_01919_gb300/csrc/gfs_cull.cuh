// P build: coverage culling of the candidates q_ik = p_i + |s_i| u_k (device
// code; included by gfs_kernels.cu).
//
// A tile holds 32 Morton-consecutive spheres, one per lane.  Directions go
// level by level of the icosphere, two launches each: a direction of level
// l > 0 is the midpoint of two directions of the levels before it, so
// k_cull_test tests the two balls that covered the same sphere's candidates
// there first; on the 64^3 union grid they settle 99% of the in-box
// candidates of level 3.  What stays open (0.8% to 1.7% of level 3 on grids,
// noisy grids and scattered samples) is listed, and k_cull_walk takes the
// list entry by entry from a cursor: a candidate is walked by a whole warp,
// 32 nodes or spheres a round, until a ball covers it or none can.  The
// cursor keeps the walks even: done where they arise, the tiles of small
// spheres beside the surface, whose candidates mostly survive, ran on for
// milliseconds after the rest (scattered samples: 30.2 ms for 1.5 ms of walks).
//
// A candidate neither of whose sources was covered survives as a rule, and
// small spheres apart from one another leave most candidates that way.  Where a
// tile and direction have kCullDense of them, all the open ones are set aside as
// a group, whose lanes walk together in one launch per chunk (k_cull_groups):
// a whole walk by one warp each is the slower way for what is not covered.
//
// What bounds it: the walks (instruction issue, and the latency of a walk's
// dependent rounds); the tests are a tenth to a third of the time.  All
// launches together, against the packet walk of every candidate that its
// Morton neighbours left open: 3.1 against 37.1 ms (64^3 union, 168M
// candidates), 4.4 against 52.6 ms (49^3 noisy pseudo-SDF, 76M), 16 against
// 428 ms (96^3 torus, 568M), 1.7 against 18.8 ms (50k scattered samples, 32M),
// 22 against 164 ms (batch of 16 shapes, 268M).  Builds of spheres apart (before
// that / with single walks only / now): 20k random ones of radius up to 0.005
// 16.1 / 29.6 / 14.3 ms, 20k points within 0.002 of a surface 10.9 / 23.9 / 10.1,
// 20k zero samples 4.0 / 10.8 / 3.1.
#pragma once

namespace gfs {

constexpr int kCullTile = kCullTileSpheres;

// Probable survivors of a tile and direction from which they form a group (of
// at most 32): at 24 the grids and scattered sets above keep their times, at 16
// a 49^3 noisy pseudo-SDF takes 6.0 instead of 5.9 ms and 50k scattered samples
// 8.0 instead of 6.1, at 8 13.2 and 13.6.
constexpr int kCullDense = 24;
// The tile (32 spheres) of one warp: its shape's arguments, first sphere and
// place in the covering-ball array.
struct CullTile {
  const CullArgs* a;
  int64_t base;
  int* hint;  // a->KH x 32 words
};

// Tiles of one shape, or of all shapes of a batch (views, prefix: first tile
// of each shape); t0: first tile of this chunk.
struct CullSource {
  const CullArgs* views;
  const int64_t* prefix;
  int ns;
  int64_t t0, tiles;  // the chunk's tiles [t0, t0 + tiles)
  int* hint;          // tiles x KH x 32 words
  uint32_t* list;     // open candidates: ((tile in the chunk) * (k1 - k0) + k - k0) * 32 + lane
  unsigned* count;    // entries of the list, and the walk's cursor
  unsigned long long* groups;  // dense groups: (tile in the chunk) * K + k, and below the mask of the lanes
  unsigned* gcount;   // their number, and the cursor
  int k0, k1, KH, K;
  bool few;           // few tiles: every open candidate goes to the groups
};

__device__ __forceinline__ CullTile cull_tile(const CullArgs& one, const CullSource& s, int64_t t) {
  const CullArgs* a = &one;
  int64_t local = s.t0 + t;
  if (s.views) {
    const int sh = find_seg(s.prefix, s.ns, local);
    a = s.views + sh;
    local -= s.prefix[sh];
  }
  return CullTile{a, local * kCullTile, s.hint + t * s.KH * 32};
}

// Candidates of directions [k0, k1), one warp per (tile, D directions): the
// box, the balls that covered the direction's two sources, the tile's other
// spheres (Morton neighbours, by shuffles).  What stays open is listed, or set
// aside as a group.
__global__ void __launch_bounds__(128) k_cull_test(const __grid_constant__ CullArgs one, const CullSource s, int D, int chunks) {
  const int lane = threadIdx.x & 31;
  const int64_t id = blockIdx.x * int64_t(4) + (threadIdx.x >> 5);
  const int64_t t = id / chunks;
  if (t >= s.tiles) return;
  const CullTile tile = cull_tile(one, s, t);
  const CullArgs& a = *tile.a;
  const int kb = s.k0 + int(id - t * chunks) * D, ke = min(kb + D, s.k1);
  const int64_t i = tile.base + lane;
  const bool active = i < a.n;
  const float4 S = active ? a.sph[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  const float lo_i = active ? a.cvl[i].w : -1.f;
  const float r = fabsf(S.w);
  const float eb = 2.f * a.bc->eq;
  const bool box = a.box_cull != 0;
  // lane d keeps the open mask of direction kb + d, and how many of them will probably survive
  unsigned rechecks = 0, mine = 0;
  int probable = 0;
  const int least = s.few ? 1 : kCullDense;
  for (int k = kb; k < ke; ++k) {
    const float4 u = a.U4[k];
    const float qx = fmaf(r, u.x, S.x), qy = fmaf(r, u.y, S.y), qz = fmaf(r, u.z, S.z);
    bool open = active;
    int found = -1;
    bool likely = false;
    if (box) {
      const float mq = fmaxf(fabsf(qx), fmaxf(fabsf(qy), fabsf(qz)));
      if (mq > 1.f + eb) {
        open = false;
      } else if (open && mq >= 1.f - eb) {
        double x, y, z;
        ex_cand(a.sph64[a.sid[i]], a.U64[3 * k], a.U64[3 * k + 1], a.U64[3 * k + 2], x, y, z);
        ++rechecks;
        open = ex_inbox(x, y, z);
      }
    }
    if (s.few) {
      likely = true;
    } else if (k >= 12) {
      // d2 < lo: covered for certain (what lies nearer the boundary is left to the walk)
      const int2 src = reinterpret_cast<const int2*>(a.hsrc)[k];
      const int h0 = tile.hint[src.x * 32 + lane], h1 = tile.hint[src.y * 32 + lane];
      likely = h0 < 0 && h1 < 0;
      if (open && h0 >= 0) {
        const float4 P = a.cvl[h0];
        const float dx = qx - P.x, dy = qy - P.y, dz = qz - P.z;
        if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < P.w) {
          open = false;
          found = h0;
        }
      }
      if (open && h1 >= 0 && h1 != h0) {
        const float4 P = a.cvl[h1];
        const float dx = qx - P.x, dy = qy - P.y, dz = qz - P.z;
        if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < P.w) {
          open = false;
          found = h1;
        }
      }
    }
    unsigned m = __ballot_sync(kFull, open);
    if (m) {
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float px = __shfl_xor_sync(kFull, S.x, o), py = __shfl_xor_sync(kFull, S.y, o),
                    pz = __shfl_xor_sync(kFull, S.z, o), lo = __shfl_xor_sync(kFull, lo_i, o);
        const float dx = qx - px, dy = qy - py, dz = qz - pz;
        if (open && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < lo) {
          open = false;
          found = int(tile.base) + (lane ^ o);
        }
      }
      m = __ballot_sync(kFull, open);
      if (__popc(m) >= least) {
        const int p = __popc(__ballot_sync(kFull, open && likely));
        if (lane == k - kb) probable = p;
      }
    }
    if (k < s.KH) tile.hint[k * 32 + lane] = found;
    if (lane == k - kb) mine = m;
  }
  if (__any_sync(kFull, mine != 0)) {
    const unsigned dense = __ballot_sync(kFull, probable >= least);
    if (dense) {
      unsigned at = 0;
      if (lane == 0) at = atomicAdd(s.gcount, unsigned(__popc(dense)));
      at = __shfl_sync(kFull, at, 0) + __popc(dense & ((1u << lane) - 1u));
      if ((dense >> lane) & 1u) {
        s.groups[at] = (unsigned long long)(uint32_t(t) * uint32_t(a.K) + uint32_t(kb + lane)) << 32 | mine;
        mine = 0;
      }
    }
    const int cnt = __popc(mine);
    int pre = cnt;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, pre, o);
      if (lane >= o) pre += v;
    }
    unsigned at = 0;
    if (lane == 31) at = atomicAdd(s.count, unsigned(pre));
    at = __shfl_sync(kFull, at, 31) + unsigned(pre - cnt);
    const uint32_t code = (uint32_t(t) * uint32_t(s.k1 - s.k0) + uint32_t(kb + lane - s.k0)) * 32u;
    for (; mine; mine &= mine - 1) s.list[at++] = code + uint32_t(__ffs(mine) - 1);
  }
  warp_count(&a.cnt->cull_rechecks, rechecks);
}

// survivors to their lists: direction k of the tile's sphere `src`, for the
// lanes with `mine` set
__device__ __forceinline__ void cull_emit(const CullArgs& one, const CullTile& tile, bool mine, int k, int src,
                                          Counters* cnt, int lane) {
  float4 item = make_float4(0.f, 0.f, 0.f, 0.f);
  float sw = 0.f;
  int shape = 0;
  const CullArgs* a = &one;
  if (mine) {
    a = tile.a;
    const int64_t i = tile.base + src;
    const float4 S = a->sph[i];
    const float r = fabsf(S.w);
    const float4 u = a->U4[k];
    sw = S.w;
    shape = a->shape;
    item = make_float4(fmaf(r, u.x, S.x), fmaf(r, u.y, S.y), fmaf(r, u.z, S.z),
                       __uint_as_float(uint32_t(a->sid[i]) * uint32_t(a->KS) + uint32_t(k)));
  }
  // to the list of the sphere's sign class (zero spheres: both)
  for (int c = 0; c < 2; ++c) {
    const bool put = mine && (c == 0 ? !(sw < 0.f) : !(sw > 0.f));
    const unsigned m = __ballot_sync(kFull, put);
    if (!m) continue;
    unsigned at = 0;
    if (lane == 0) at = atomicAdd(&cnt->nsurv[c], unsigned(__popc(m)));
    at = __shfl_sync(kFull, at, 0) + __popc(m & ((1u << lane) - 1u));
    if (put && at < a->cap) {
      a->surv[c][at] = item;
      if (a->surv_shape[c]) a->surv_shape[c][at] = uint16_t(shape);
    }
  }
}

// one candidate by the whole warp: a ball that covers it (sorted slot), or -1
__device__ __forceinline__ int cull_walk_one(const CullArgs& a, int64_t i, int k, const LevelTable& C, uint32_t* stk,
                                             int lane, unsigned& rechecks, unsigned& n_nodes, unsigned& n_items) {
  const float4 S = a.sph[i];
  const float r = fabsf(S.w);
  const float lim = -a.tol32 + a.bc->elin + 4.f * a.bc->eq;
  const float4 u = a.U4[k];
  const float qx = fmaf(r, u.x, S.x), qy = fmaf(r, u.y, S.y), qz = fmaf(r, u.z, S.z);
  return warp_cover_walk(a.tree, C, stk, lane, qx, qy, qz, lim, n_nodes, n_items, [&](int c, float& v) {
    const float4 P = a.cvl[c];
    const float hi = a.thr[c].y;
    const float dx = qx - P.x, dy = qy - P.y, dz = qz - P.z;
    const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    if (c == i || !(d2 <= hi)) return false;
    v = d2 - P.w;
    if (d2 < P.w) return true;
    ++rechecks;
    double x, y, z;
    ex_cand(a.sph64[a.sid[i]], a.U64[3 * k], a.U64[3 * k + 1], a.U64[3 * k + 2], x, y, z);
    return ex_cov(x, y, z, a.sph64[a.sid[c]], a.tol);
  });
}

// The dense groups of all levels, once per chunk (they keep no covering balls:
// few of their candidates are covered): the candidates of one tile and
// direction, one a lane, walk together; a node is entered when some lane's
// candidate lies in its ball.  (Inside k_cull_walk, inlined or called, this loop
// made the single candidates' walks 12% slower.)
__global__ void __launch_bounds__(128) k_cull_groups(const __grid_constant__ CullArgs one, const CullSource s) {
  __shared__ uint32_t s_stk[4][kCoverStack];
  __shared__ LevelTable s_lv[4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t* stk = s_stk[w];
  LevelTable& C = s_lv[w];
  const unsigned groups = s.gcount[0];
  if (!groups) return;
  const uint32_t K = uint32_t(s.K);
  unsigned rechecks = 0, n_nodes = 0, n_items = 0;
  const CullArgs* loaded = nullptr;
  Counters* cnt = nullptr;
  if (!s.few && groups < gridDim.x * 4u) {
    // fewer groups than warps: one long walk each would be the whole time (1,000
    // samples at tau 3: 0.66 ms, now 0.54)
    for (;;) {
      unsigned t = 0;
      if (lane == 0) t = atomicAdd(s.gcount + 1, 1u);
      t = __shfl_sync(kFull, t, 0);
      if (t >= 32u * groups) break;
      const unsigned long long g = s.groups[t >> 5];
      const int src = int(t & 31u), k = int(uint32_t(g >> 32) % K);
      if (!((uint32_t(g) >> src) & 1u)) continue;
      const CullTile tile = cull_tile(one, s, uint32_t(g >> 32) / K);
      cnt = tile.a->cnt;
      load_levels(tile.a->tree, C, lane);
      const int j = cull_walk_one(*tile.a, tile.base + src, k, C, stk, lane, rechecks, n_nodes, n_items);
      if (j < 0) cull_emit(one, tile, lane == 0, k, src, cnt, lane);
    }
  } else for (;;) {
    unsigned t = 0;
    if (lane == 0) t = atomicAdd(s.gcount + 1, 1u);
    t = __shfl_sync(kFull, t, 0);
    if (t >= groups) break;
    const unsigned long long g = s.groups[t];
    bool open = (uint32_t(g) >> lane) & 1u;
    const int k = int(uint32_t(g >> 32) % K);
    const CullTile tile = cull_tile(one, s, uint32_t(g >> 32) / K);
    const CullArgs& a = *tile.a;
    cnt = a.cnt;
    if (loaded != tile.a) {
      load_levels(a.tree, C, lane);
      loaded = tile.a;
    }
    const int64_t i = tile.base + lane;
    const float4 P0 = open ? a.sph[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float r = fabsf(P0.w);
    const float4 u = a.U4[k];
    const float qx = fmaf(r, u.x, P0.x), qy = fmaf(r, u.y, P0.y), qz = fmaf(r, u.z, P0.z);
    const Tree& T = a.tree;
    const float pad = a.bc->pad, grow = 1.f + 8.f * kU;
    int sp = C.lv[T.nlevels - 1].y;
    __syncwarp();
    if (lane < sp) stk[lane] = pack_node(T.nlevels - 1, lane);
    __syncwarp();
    // (one node a round: at most kFan - 1 entries a level are left behind)
    while (sp > 0 && __any_sync(kFull, open)) {
      const uint32_t nd = stk[--sp];
      const int lev = node_level(nd);
      const int b = int(node_index(nd)) * kFan;
      if (lev == 0) {
        const int items = int(min(int64_t(kLeaf), T.nitems - b));
        n_items += open ? unsigned(items) : 0u;
#pragma unroll
        for (int c = 0; c < kLeaf; ++c) {
          if (c >= items) break;
          const float4 P = a.cvl[b + c];
          const float hi = a.thr[b + c].y;
          if (!open || b + c == i) continue;
          const float dx = qx - P.x, dy = qy - P.y, dz = qz - P.z;
          const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          bool cov = d2 < P.w;
          if (!cov && d2 <= hi) {
            ++rechecks;
            double x, y, z;
            ex_cand(a.sph64[a.sid[i]], a.U64[3 * k], a.U64[3 * k + 1], a.U64[3 * k + 2], x, y, z);
            cov = ex_cov(x, y, z, a.sph64[a.sid[b + c]], a.tol);
          }
          open = !cov;
        }
      } else {
        const int2 L = C.lv[lev - 1];
        const int nc = min(kFan, L.y - b);
        n_nodes += open ? unsigned(nc) : 0u;
        unsigned need = 0;
#pragma unroll
        for (int c = 0; c < kFan; ++c) {
          if (c >= nc) break;
          const float4 B = T.na[int64_t(L.x) + b + c];
          const float t = fmaf(B.w - a.tol32, grow, pad);
          if (open && t > 0.f && ball_d2(qx, qy, qz, B) < t * t) need |= 1u << c;
        }
        need = __reduce_or_sync(kFull, need);
        if (lane < kFan && ((need >> lane) & 1u)) stk[sp + __popc(need & ((1u << lane) - 1u))] = pack_node(lev - 1, b + lane);
        sp += __popc(need);
      }
      __syncwarp();
    }
    if (__any_sync(kFull, open)) cull_emit(one, tile, open, k, lane, cnt, lane);
  }
  if (cnt) {  // one counter block serves all shapes
    warp_count(&cnt->cull_rechecks, rechecks);
    warp_count(&cnt->c_ntests, n_nodes);
    warp_count(&cnt->c_items, n_items);
  }
}


// The listed candidates, a warp each; survivors are gathered 32 at a time
// (lane l keeps the l-th) for one atomic per class and flush.
__global__ void __launch_bounds__(128) k_cull_walk(const __grid_constant__ CullArgs one, const CullSource s) {
  __shared__ uint32_t s_stk[4][kCoverStack];
  __shared__ LevelTable s_lv[4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t* stk = s_stk[w];
  LevelTable& C = s_lv[w];
  const unsigned n = s.count[0];
  const uint32_t dirs = uint32_t(s.k1 - s.k0);
  unsigned rechecks = 0, n_nodes = 0, n_items = 0;
  const CullArgs* loaded = nullptr;
  Counters* cnt = nullptr;
  uint32_t kept = 0;
  int nkept = 0;
  auto flush = [&]() {
    const uint32_t td = kept >> 5;
    const bool mine = lane < nkept;
    CullTile tile{nullptr, 0, nullptr};
    if (mine) tile = cull_tile(one, s, td / dirs);
    cull_emit(one, tile, mine, s.k0 + int(td % dirs), int(kept & 31u), cnt, lane);
    nkept = 0;
  };
  unsigned e = 0, end = 0;
  // far from the end of the list a warp takes 8 entries per atomic
  const unsigned near_end = gridDim.x * 4u * 32u;
  for (;; ++e) {
    if (e >= end) {
      const unsigned b = n - min(n, e) > near_end ? 8u : 1u;
      unsigned at = 0;
      if (lane == 0) at = atomicAdd(s.count + 1, b);
      e = __shfl_sync(kFull, at, 0);
      end = min(n, e + b);
      if (e >= n) break;
    }
    const uint32_t code = s.list[e], td = code >> 5;
    const int k = s.k0 + int(td % dirs), src = int(code & 31u);
    const CullTile tile = cull_tile(one, s, td / dirs);
    const CullArgs& a = *tile.a;
    cnt = a.cnt;
    if (loaded != tile.a) {
      load_levels(a.tree, C, lane);
      loaded = tile.a;
    }
    const int j = cull_walk_one(a, tile.base + src, k, C, stk, lane, rechecks, n_nodes, n_items);
    if (j >= 0) {
      if (k < s.KH && lane == 0) tile.hint[k * 32 + src] = j;
    } else {
      if (lane == nkept) kept = code;
      if (++nkept == 32) flush();
    }
  }
  if (nkept) flush();
  if (cnt) {  // one counter block serves all shapes
    warp_count(&cnt->cull_rechecks, rechecks);
    warp_count(&cnt->c_ntests, n_nodes);
    warp_count(&cnt->c_items, n_items);
  }
}

}  // namespace gfs
