// Covered area ratio of grid cells for the refinement order (Sec. 4.2).
#include <cuda_runtime.h>

#include <type_traits>

#include "gfs_order.cuh"
#include "gfs_order.h"
#include "gfs_warp.cuh"

namespace gfs {

namespace {

constexpr int kRecent = 16, kMaxSub = 64;

// One block per cell.  Each warp takes 32 of its points at a time; the balls
// that held its latest covered points (kRecent of them, FP32, tested by every
// lane) settle nearly all, and a point they leave open is walked by the
// whole warp (warp_cover_walk), whose ball is tried on the other open points
// at once.  Bound: the latency of the walks (a point that no ball holds needs
// a whole one); 1,536 surface cells of a 40^3 grid at 8^3 points take 2.0 ms,
// 7.7 ms with one warp per cell, and 32.5 ms with a walk per lane (FP64
// positions, a stack in local memory).
// FP32 decides only what is certain: thr.z is the threshold below which a
// point rounded to FP32 lies in the ball for sure; points outside the
// coordinate range of that bound take the FP64 walk of gfs_tangent.cuh.
template <int kCellWarps>
__global__ void __launch_bounds__(32 * kCellWarps) k_cell_coverage(QueryArgs a, const int32_t* __restrict__ cells,
                                                                   double ox, double oy, double oz,
                                                                   double h, int sub, uint32_t* __restrict__ counts) {
  __shared__ uint32_t s_stk[kCellWarps][kCoverStack];
  __shared__ LevelTable s_lv;
  __shared__ float4 s_rec[kCellWarps][kRecent];
  __shared__ double s_off[kMaxSub];
  __shared__ unsigned s_cnt;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int t = threadIdx.x; t < sub; t += blockDim.x) s_off[t] = __ddiv_rn(__dadd_rn(double(t), 0.5), double(sub));
  if (threadIdx.x < kMaxLevels)
    s_lv.lv[threadIdx.x] = make_int2(int(a.st.offset[threadIdx.x]), int(a.st.count[threadIdx.x]));
  if (threadIdx.x == 0) s_cnt = 0;
  __syncthreads();
  const int64_t c = blockIdx.x;
  const float A = a.bc->A;
  const float lim = -a.tol32 + a.bc->elin;
  float4* rec = s_rec[w];
  int nrec = 0, at = 0;
  unsigned cnt = 0, n_nodes = 0, n_items = 0;
  const int total = sub * sub * sub;
  for (int base = 32 * w; base < total; base += 32 * kCellWarps) {
    const int t = base + lane;
    const int ia = t / (sub * sub), ib = (t / sub) % sub, ic = t % sub;
    double x = 0.0, y = 0.0, z = 0.0;
    bool open = t < total;
    if (open) {  // order::cell_coord with the offsets tabulated
      x = __dadd_rn(ox, __dmul_rn(h, __dadd_rn(double(cells[3 * c]), s_off[ia])));
      y = __dadd_rn(oy, __dmul_rn(h, __dadd_rn(double(cells[3 * c + 1]), s_off[ib])));
      z = __dadd_rn(oz, __dmul_rn(h, __dadd_rn(double(cells[3 * c + 2]), s_off[ic])));
      if (!(fabs(x) <= A && fabs(y) <= A && fabs(z) <= A)) {
        if (tangent::covered_by_other(a, x, y, z, -1) >= 0) ++cnt;
        open = false;
      }
    }
    const float xf = float(x), yf = float(y), zf = float(z);
    auto held = [&](const float4& P) {
      const float dx = xf - P.x, dy = yf - P.y, dz = zf - P.z;
      return fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < P.w;
    };
    __syncwarp();
    for (int u = 0; u < nrec && __any_sync(0xffffffffu, open); ++u)
      if (open && held(rec[u])) {
        ++cnt;
        open = false;
      }
    unsigned left = __ballot_sync(0xffffffffu, open);
    while (left) {
      const int src = __ffs(left) - 1;
      left &= left - 1;
      const float qx = __shfl_sync(0xffffffffu, xf, src), qy = __shfl_sync(0xffffffffu, yf, src),
                  qz = __shfl_sync(0xffffffffu, zf, src);
      const double qx64 = __shfl_sync(0xffffffffu, x, src), qy64 = __shfl_sync(0xffffffffu, y, src),
                   qz64 = __shfl_sync(0xffffffffu, z, src);
      const int j = warp_cover_walk(a.st, s_lv, s_stk[w], lane, qx, qy, qz, lim, n_nodes, n_items,
                                    [&](int s, float& v) {
                                      const float4 P = a.sph[s], Th = a.thr[s];
                                      const float dx = qx - P.x, dy = qy - P.y, dz = qz - P.z;
                                      const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                                      if (!(d2 <= Th.w)) return false;
                                      v = d2 - Th.z;
                                      return d2 < Th.z || ex_cov(qx64, qy64, qz64, a.sph64[a.sid[s]], a.tol);
                                    });
      if (j < 0) continue;
      float4 P = a.sph[j];
      P.w = a.thr[j].z;
      if (lane == src || (open && ((left >> lane) & 1u) && held(P))) {
        ++cnt;
        open = false;
      }
      left &= __ballot_sync(0xffffffffu, open);
      if (lane == 0) rec[at] = P;
      at = (at + 1) % kRecent;
      nrec = min(nrec + 1, kRecent);
      __syncwarp();
    }
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) atomicAdd(&s_cnt, cnt);
  __syncthreads();
  if (threadIdx.x == 0) counts[c] = s_cnt;
}

unsigned long long g_order_launches = 0;

}  // namespace

cudaError_t launch_cell_coverage(const QueryArgs& a, const int32_t* cells, int64_t ncells, const double* origin,
                                 double h, int sub, uint32_t* counts, cudaStream_t st) {
  if (ncells <= 0) return cudaSuccess;
  // As many warps as the points fill, at most 8: with 8 throughout the 59,319
  // cells of a 40^3 union grid took 0.53 / 0.74 / 1.28 / 1.84 / 2.22 ms at 1^3 to 5^3
  // points, now 0.17 / 0.39 / 0.86 / 1.34 / 1.99, and 237k cells outside the range
  // (walks per lane) 2.44 / 2.89 / 3.17 / 3.34 / 3.83, now 0.81 / 0.97 / 1.07 / 1.63 /
  // 2.78.
  auto run = [&](auto warps) {
    constexpr int W = decltype(warps)::value;
    for (int64_t c0 = 0; c0 < ncells; c0 += 1 << 30)  // (grid dimension below 2^31)
      k_cell_coverage<W><<<unsigned(ncells - c0 < (1 << 30) ? ncells - c0 : 1 << 30), 32 * W, 0, st>>>(
          a, cells + 3 * c0, origin[0], origin[1], origin[2], h, sub, counts + c0);
  };
  if (sub <= 3) run(std::integral_constant<int, 1>());
  else if (sub == 4) run(std::integral_constant<int, 2>());
  else if (sub == 5) run(std::integral_constant<int, 4>());
  else run(std::integral_constant<int, 8>());
  ++g_order_launches;
  return cudaGetLastError();
}

unsigned long long order_launch_count() { return g_order_launches; }

}  // namespace gfs
