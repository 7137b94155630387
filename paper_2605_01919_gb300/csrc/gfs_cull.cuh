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
// What bounds it: the walks (instruction issue, and the latency of a walk's
// dependent rounds); the tests are a tenth to a third of the time.  Both
// launches together, against the packet walk of every candidate that its
// Morton neighbours left open: 3.1 against 37.1 ms (64^3 union, 168M
// candidates), 4.3 against 52.6 ms (49^3 noisy pseudo-SDF, 76M), 16 against
// 428 ms (96^3 torus, 568M), 1.7 against 18.8 ms (50k scattered samples, 32M),
// 22 against 164 ms (batch of 16 shapes, 268M).
#pragma once

namespace gfs {

constexpr int kCullTile = kCullTileSpheres;
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
  int k0, k1, KH;
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
// spheres (Morton neighbours, by shuffles).  What stays open is listed.
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
  unsigned rechecks = 0, mine = 0;  // mine: lane d keeps the open mask of direction kb + d
  for (int k = kb; k < ke; ++k) {
    const float4 u = a.U4[k];
    const float qx = fmaf(r, u.x, S.x), qy = fmaf(r, u.y, S.y), qz = fmaf(r, u.z, S.z);
    bool open = active;
    int found = -1;
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
    if (k >= 12) {
      // d2 < lo: covered for certain (what lies nearer the boundary is left to the walk)
      const int2 src = reinterpret_cast<const int2*>(a.hsrc)[k];
      const int h0 = tile.hint[src.x * 32 + lane], h1 = tile.hint[src.y * 32 + lane];
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
    }
    if (k < s.KH) tile.hint[k * 32 + lane] = found;
    if (lane == k - kb) mine = m;
  }
  if (__any_sync(kFull, mine != 0)) {
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
    const bool mine = lane < nkept;
    float4 item = make_float4(0.f, 0.f, 0.f, 0.f);
    float sw = 0.f;
    int shape = 0;
    const CullArgs* a = &one;
    if (mine) {
      const uint32_t td = kept >> 5;
      const CullTile tile = cull_tile(one, s, td / dirs);
      a = tile.a;
      const int k = s.k0 + int(td % dirs);
      const int64_t i = tile.base + (kept & 31u);
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
    const int64_t i = tile.base + src;
    const float4 S = a.sph[i];
    const float r = fabsf(S.w);
    const float lim = -a.tol32 + a.bc->elin + 4.f * a.bc->eq;
    const float4 u = a.U4[k];
    const float qx = fmaf(r, u.x, S.x), qy = fmaf(r, u.y, S.y), qz = fmaf(r, u.z, S.z);
    const int j = warp_cover_walk(a.tree, C, stk, lane, qx, qy, qz, lim, n_nodes, n_items, [&](int c, float& v) {
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
